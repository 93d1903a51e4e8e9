"""lre_project below d = 2048 without eig_mu: the Lanczos path from d = 64 on
(persistent steps, the run up to d steps) and the one-launch path for n <= 5,
against the oracle's Smolin projection.

Tolerances: eigenvalues of both paths are at FP64 rounding of a matrix of norm
at most 1, d eps = 2.3e-13 at d = 1024; the complex64 result is within the
rounding of its entries, far inside 1e-6 relative Frobenius."""
import ctypes

import numpy as np
import pytest

from oracle import project
from synth import counts as sc
from synth import states as st
from tests.gpu_util import ctx_and_lre, need_gpu, rel_fro
from tests.test_gpu_projection import _hermitian_with_spectrum

pytestmark = pytest.mark.gpu

EIG_ATOL = 2.5e-13


@pytest.fixture(scope="module")
def env():
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    yield torch, lre, ctx
    lre.lre_destroy(ctx)


def _run(env, m, n, eig=True, alias=False):
    torch, lre, ctx = env
    mu = torch.from_numpy(m).cuda()
    out = mu if alias else torch.full_like(mu, float("nan"))
    er = torch.full((2 ** n,), float("nan"), dtype=torch.float64, device="cuda") if eig else None
    lre.lre_profile(ctx, True)
    lre.lre_project(ctx, mu, n, out, eig_rho=er)
    lre.lre_sync(ctx)
    names = {k for k, _ in lre.lre_profile_records(ctx)}
    lre.lre_profile(ctx, False)
    ref, _, lam = project.smolin(m.astype(np.complex128))
    got = out.cpu().numpy()
    assert rel_fro(got, ref) <= 1e-6
    assert np.array_equal(got, got.conj().T)
    if eig:
        np.testing.assert_allclose(er.cpu().numpy(), lam, atol=EIG_ATOL)
    return names, lam


def _estimate(n, shots, rank, seed):
    from oracle import direct
    thr = sc.cdf_thresholds(st.born_probabilities(st.pauli_expectations(st.ginibre_state(n, rank, seed=seed)), n))
    return direct.mu(direct.estimate(sc.sample_cdf(thr, shots, seed=seed + 1), shots, n), n).astype(np.complex64)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("shots,rank", [(100, 1), (20000, 3)])
def test_estimates(env, n, shots, rank):
    names, _ = _run(env, _estimate(n, shots, rank, 60 + n), n)
    assert ("project_small" in names) == (n <= 5)
    assert ("kry_matvec" in names) == (n >= 6)
    assert "hetrd(cusolver)" not in names, names


@pytest.mark.parametrize("n", [2, 5, 6, 8, 10])
@pytest.mark.parametrize("eig", [True, False])
def test_dropped_form(env, n, eig):
    """Few negative eigenvalues: the rebuild is mu + sI and the dropped directions."""
    d = 2 ** n
    rng = np.random.default_rng(n)
    lam = rng.uniform(0.2, 1.0, d)
    k = max(1, d // 16)
    lam[:k] = -rng.uniform(0.02, 0.1, k) * lam.mean()
    lam /= lam.sum()
    _, out = _run(env, _hermitian_with_spectrum(lam, 3 + n), n, eig=eig, alias=True)
    assert (out > 0).sum() > d // 2


@pytest.mark.parametrize("n", [3, 5, 6, 9])
def test_clusters(env, n):
    """Kept eigenvalues equal before the complex64 rounding."""
    d = 2 ** n
    lam = -np.linspace(1e-4, 2e-4, d)
    lam[-2:] = 0.3
    lam[-4:-2] = 0.1
    lam /= lam.sum()
    _run(env, _hermitian_with_spectrum(lam, 17 + n), n)


@pytest.mark.parametrize("n", [1, 4, 6, 7])
def test_degenerate_and_physical_inputs(env, n):
    """Invariant subspaces after one or two steps (I/d, a pure state, a mixture of
    both): exact multiplicities, and a physical input comes back as it is."""
    torch, lre, ctx = env
    d = 2 ** n
    eye = np.eye(d, dtype=np.complex64) / np.float32(d)
    pure = np.zeros((d, d), np.complex64)
    pure[0, 0] = pure[0, -1] = pure[-1, 0] = pure[-1, -1] = 0.5
    for m in (eye, pure, (0.5 * eye + 0.5 * pure).astype(np.complex64), -eye + 2 * pure):
        _run(env, m, n)
    mu = torch.from_numpy(eye).cuda()
    out = torch.empty_like(mu)
    lre.lre_project(ctx, mu, n, out)
    lre.lre_sync(ctx)
    np.testing.assert_array_equal(out.cpu().numpy(), eye)


@pytest.mark.parametrize("n", [4, 7])
def test_only_the_upper_triangle_is_read(env, n):
    m = _estimate(n, 300, 2, 5)
    low = m.copy()
    low[np.tril_indices(2 ** n, -1)] = 7.0
    torch, lre, ctx = env
    outs = []
    for x in (m, low):
        mu = torch.from_numpy(x).cuda()
        out = torch.empty_like(mu)
        lre.lre_project(ctx, mu, n, out)
        lre.lre_sync(ctx)
        outs.append(out.cpu().numpy())
    np.testing.assert_array_equal(outs[0], outs[1])



@pytest.mark.parametrize("n,scale", [(7, 1e-9), (8, 1e12), (11, 1e-9), (11, 1e12)])
def test_scaled_inputs(env, n, scale):
    """Norms far from a density matrix' leave the persistent steps, whose squared
    norms are FP32 pairs; the projection scales with its input (trace kept)."""
    torch, lre, ctx = env
    d = 2 ** n
    rng = np.random.default_rng(n)
    lam = -rng.uniform(0, 2e-4, d)
    lam[-4:] = (0.1, 0.2, 0.3, 0.4)
    m = _hermitian_with_spectrum(lam / lam.sum(), 5 + n)
    scaled = (m * np.float32(scale)).astype(np.complex64)
    outs = []
    for x in (m, scaled):
        mu = torch.from_numpy(x).cuda()
        out = torch.full_like(mu, float("nan"))
        lre.lre_project(ctx, mu, n, out)
        lre.lre_sync(ctx)
        outs.append(out.cpu().numpy().astype(np.complex128))
    assert rel_fro(outs[1] / float(np.float32(scale)), outs[0]) <= 1e-6


@pytest.mark.parametrize("n", [7, 9, 10])
@pytest.mark.parametrize("gap", [1e-2, 1e-5])
def test_close_neighbours(env, n, gap):
    """Kept values close together above a dense bulk that does not converge: the
    residuals must tell the two apart (accepted too early, the eigenvalues are off;
    never accepted, the reduction would run)."""
    d = 2 ** n
    rng = np.random.default_rng(n)
    lam = -rng.uniform(0.0, 0.25 / d, d)
    lam[-12:] = 0.05 * (1.0 + gap * np.arange(12))
    lam[-24:-12] = 0.01 * (1.0 + gap * rng.uniform(0, 12, 12))
    names, out = _run(env, _hermitian_with_spectrum(lam / lam.sum(), 29 + n), n)
    assert "kry_residuals" in names and "hetrd(cusolver)" not in names, names
    assert (out > 0).sum() < d // 2


@pytest.mark.parametrize("n", [7, 8, 9])
def test_missed_copy_close_to_the_threshold(env, n):
    """A kept eigenvalue with an exact copy (a Krylov space sees one until rounding brings
    in the other, which the spread of the rest delays) 4e-11 above the threshold: the
    certification must find the copy and the reduction run."""
    d = 2 ** n
    b = 2.0 ** -10 * (1 + 2.0 ** -23)
    lam = np.empty(d)
    lam[:4] = 1 + 2.0 ** -10, b, b, 0.93 * b
    mean = (1.0 - lam[:4].sum()) / (d - 4)
    lam[4:] = mean + (0.86 * b - mean) * np.linspace(-1.0, 1.0, d - 4)
    lam[4:] = np.round(lam[4:] * 2.0 ** 33) / 2.0 ** 33
    lam[4 + (d - 4) // 2] += 1.0 - lam.sum()
    names, out = _run(env, np.diag(lam).astype(np.complex64), n)
    assert (out > 0).sum() == 3
    assert "hetrd(cusolver)" in names, names


@pytest.mark.parametrize("n", [6, 7, 8])
@pytest.mark.parametrize("mixed", [0.0, 0.1, -0.05])
def test_reduction_of_structured_states(env, n, mixed):
    """Few nonzero amplitudes of equal size: the reduction's trailing columns are rounding
    residue of residue, and the library's reflectors of those are not finite at n = 6."""
    torch, lre, ctx = env
    d = 2 ** n
    v = np.zeros(d, np.complex128)
    v[[8, 19, 33, 58]] = 0.5, 0.5j, 0.5, -0.5j
    m = ((1 - mixed) * np.outer(v, v.conj()) + mixed * np.eye(d) / d).astype(np.complex64)
    _run(env, m, n)
    mu = torch.from_numpy(m).cuda()
    out = torch.full_like(mu, float("nan"))
    em, er = [torch.empty(d, dtype=torch.float64, device="cuda") for _ in range(2)]
    lre.lre_project(ctx, mu, n, out, em, er)  # eig_mu: by the reduction
    lre.lre_sync(ctx)
    ref, lam_mu, lam = project.smolin(m.astype(np.complex128))
    assert rel_fro(out.cpu().numpy(), ref) <= 1e-6
    np.testing.assert_allclose(em.cpu().numpy(), lam_mu, atol=EIG_ATOL)
    np.testing.assert_allclose(er.cpu().numpy(), lam, atol=EIG_ATOL)


@pytest.mark.parametrize("n", [6, 8])
@pytest.mark.parametrize("eig_mu", [True, False])
def test_input_that_is_not_finite_is_reported(env, n, eig_mu):
    torch, lre, ctx = env
    m = (np.eye(2 ** n) / 2 ** n).astype(np.complex64)
    m[1, 5] = np.nan
    mu = torch.from_numpy(m).cuda()
    em = torch.empty(2 ** n, dtype=torch.float64, device="cuda") if eig_mu else None
    with pytest.raises(lre.LreError) as e:
        lre.lre_project(ctx, mu, n, torch.empty_like(mu), em)
    assert e.value.status == lre.LRE_ERR_EIG_FAILED


@pytest.mark.parametrize("scale", [1e-25, 1e25])
def test_norms_beyond_fp32(env, scale):
    """Entries whose squares leave FP32's range, d = 2048: the Lanczos path still decides
    (its breakdown threshold goes by the norm), and the result is right."""
    torch, lre, ctx = env
    test_scaled_inputs(env, 11, scale)
    lam = -np.random.default_rng(11).uniform(0, 2e-4, 2048)
    lam[-4:] = (0.1, 0.2, 0.3, 0.4)
    mu = torch.from_numpy((_hermitian_with_spectrum(lam / lam.sum(), 16) * np.float32(scale)).astype(np.complex64)).cuda()
    lre.lre_profile(ctx, True)
    lre.lre_project(ctx, mu, 11, torch.empty_like(mu))
    lre.lre_sync(ctx)
    names = {k for k, _ in lre.lre_profile_records(ctx)}
    lre.lre_profile(ctx, False)
    assert "hetrd(cusolver)" not in names, names


@pytest.mark.parametrize("n", [6, 10, 11])
def test_repeats_bit_for_bit(env, n):
    """With other work on the device, so that CTAs finish in varying order."""
    torch, lre, ctx = env
    d = 2 ** n
    lam = -np.random.default_rng(n).uniform(0, 0.5 / d, d)
    lam[-4:] = (0.1, 0.2, 0.3, 0.4)
    mu = torch.from_numpy(_hermitian_with_spectrum(lam / lam.sum(), 7)).cuda()
    side, a = torch.cuda.Stream(), torch.randn(512, 512, device="cuda")
    torch.cuda.synchronize()
    first = None
    for _ in range(60):
        with torch.cuda.stream(side):
            for _ in range(8):
                a @ a
        out, er = torch.empty_like(mu), torch.empty(d, dtype=torch.float64, device="cuda")
        lre.lre_project(ctx, mu, n, out, eig_rho=er)
        lre.lre_sync(ctx)
        first = first or (out, er)
        assert torch.equal(out, first[0]) and torch.equal(er, first[1])


@pytest.mark.parametrize("n", [6, 11])
def test_barrier_that_gives_up_is_reported(env, n):
    """Barriers that wait for arrivals that never come, 5 ms each: the call returns
    LRE_ERR_TIMEOUT, writes no result, and the context stays usable."""
    torch, lre, ctx = env
    f = lre.load().lre_debug_steps_fault
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int], ctypes.c_int
    d = 2 ** n
    lam = -np.random.default_rng(n).uniform(0, 0.5 / d, d)
    lam[-4:] = (0.1, 0.2, 0.3, 0.4)
    m = _hermitian_with_spectrum(lam / lam.sum(), 7)
    mu = torch.from_numpy(m).cuda()
    out = torch.full_like(mu, 3.0)
    assert f(ctx, 5) == 0
    try:
        with pytest.raises(lre.LreError) as e:
            lre.lre_project(ctx, mu, n, out)
        assert e.value.status == lre.LRE_ERR_TIMEOUT
        with pytest.raises(lre.LreError) as e:
            lre.lre_sync(ctx)  # latched by the kernel too
        assert e.value.status == lre.LRE_ERR_TIMEOUT
    finally:
        assert f(ctx, 0) == 0
    assert (out == 3.0).all()
    _run(env, m, n)


@pytest.mark.parametrize("seed", [1, 2, 3, 4, 5, 6, 7, 8])
def test_eigenvalues_at_d_2048(env, seed):
    """eig_rho of 120 kept values, one of them most of the trace: the Rayleigh quotients' double-float rows average out
    and their sums are FP64, so a few units of rounding of the norm are left (8 allowed).
    Reference: the quotients of complex128 eigenvectors, whose own error enters squared."""
    torch, lre, ctx = env
    n, d, k = 11, 2048, 120
    rng = np.random.default_rng(seed)
    lam = -rng.uniform(0.0, 0.5 / d, d)
    lam[-k:] = 0.0005 * 1.02 ** np.arange(k)
    lam[-1] = rng.uniform(0.6, 0.9)
    mu = torch.from_numpy(_hermitian_with_spectrum(lam / lam.sum(), 50 + seed)).cuda()
    out, er = torch.empty_like(mu), torch.empty(d, dtype=torch.float64, device="cuda")
    lre.lre_profile(ctx, True)
    lre.lre_project(ctx, mu, n, out, eig_rho=er)
    lre.lre_sync(ctx)
    names = {name for name, _ in lre.lre_profile_records(ctx)}
    lre.lre_profile(ctx, False)
    assert "kry_matvec" in names and "hetrd(cusolver)" not in names, names
    m = mu.to(torch.complex128)
    w, v = torch.linalg.eigh(m)
    w = w.cpu().numpy()
    a, j = 0.0, 0
    while w[j] + a / (d - j) < 0.0:
        a += w[j]
        j += 1
    v = v[:, j:]
    q = ((v.conj() * (m @ v)).sum(0).real / (v.conj() * v).sum(0).real).cpu().numpy()
    want = np.sort(q + (np.trace(mu.cpu().numpy().astype(np.complex128)).real - q.sum()) / len(q))[::-1]
    assert np.abs(er[:len(q)].cpu().numpy() - want).max() <= 8 * np.finfo(np.float64).eps * q.max()


@pytest.mark.parametrize("n", [8, 9, 10])
def test_dense_values_around_the_threshold(env, n):
    """An exact state's rounding: a few large eigenvalues and a bulk spaced by 1e-12 on both
    sides of the threshold.  Diagonal input, so the eigenvalues are known exactly; sixteen
    units of rounding of the norm are left to the Lanczos coefficients and quotients."""
    torch, lre, ctx = env
    d = 2 ** n
    for seed in range(1, 25):
        rng = np.random.default_rng(seed)
        lam = rng.normal(0.0, 3e-10, d)
        lam[:24] = 0.005 * (1 + 1e-4 * np.arange(24))
        lam[24] = 1.0 - lam[:24].sum() - lam[25:].sum()
        lam = lam.astype(np.float32)
        want = project.smolin_eigenvalues(np.sort(lam.astype(np.float64))[::-1])
        mu = torch.from_numpy(np.diag(lam).astype(np.complex64)).cuda()
        er = torch.empty(d, dtype=torch.float64, device="cuda")
        lre.lre_project(ctx, mu, n, torch.empty_like(mu), eig_rho=er)
        lre.lre_sync(ctx)
        tol = 16 * np.finfo(np.float64).eps * lam.max()
        np.testing.assert_allclose(er.cpu().numpy(), want, rtol=0, atol=tol, err_msg=str(seed))


@pytest.mark.parametrize("n", [6, 7, 8, 9, 10])
@pytest.mark.parametrize("kind", ["physical", "few negative", "half", "cluster"])
def test_spectrum_of_mostly_kept_values(env, n, kind):
    """eig_rho where the kept set is the larger one: all its values to a few units of
    rounding of the norm (8 allowed), from d Lanczos steps (a long cluster of equal values
    from the reduction).  Reference: quotients of complex128 eigenvectors."""
    torch, lre, ctx = env
    d = 2 ** n
    rng = np.random.default_rng(n)
    lam = rng.normal(1.0, 1.0, d) if kind == "half" else rng.uniform(0.1, 1.0, d)
    if kind == "few negative":
        lam[:d // 16] = -rng.uniform(0.0, 0.3, d // 16)
    if kind == "cluster":
        lam[:d - 20] = 0.5
    mu = torch.from_numpy(_hermitian_with_spectrum(lam / lam.sum(), 90 + n)).cuda()
    out, er = torch.empty_like(mu), torch.empty(d, dtype=torch.float64, device="cuda")
    lre.lre_profile(ctx, True)
    lre.lre_project(ctx, mu, n, out, eig_rho=er)
    lre.lre_sync(ctx)
    names = {name for name, _ in lre.lre_profile_records(ctx)}
    lre.lre_profile(ctx, False)
    assert ("hetrd(cusolver)" in names) == (kind == "cluster"), names
    m = mu.to(torch.complex128)
    _, v = torch.linalg.eigh(m)
    q = np.sort(((v.conj() * (m @ v)).sum(0).real / (v.conj() * v).sum(0).real).cpu().numpy())[::-1]
    want = project.smolin_eigenvalues(q)
    assert (want > 0).sum() > d // 2
    assert np.abs(er.cpu().numpy() - want).max() <= 8 * np.finfo(np.float64).eps * np.abs(q).max()
    ref = project.smolin(mu.cpu().numpy().astype(np.complex128))[0]
    assert rel_fro(out.cpu().numpy(), ref) <= 1e-6
