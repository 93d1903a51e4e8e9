"""lre_project for n <= 5 (one launch) on exact low-rank and structured input, whose
tridiagonal reduction runs into columns of rounding residue, on scaled input, and on
input that is not finite, against the oracle's Smolin projection.

Tolerances: eigenvalues at FP64 rounding of the input's norm (the bound of
test_gpu_projection_paths), the complex64 result within 1e-6 relative Frobenius."""
import numpy as np
import pytest

from oracle import project
from tests.gpu_util import ctx_and_lre, need_gpu, rel_fro

pytestmark = pytest.mark.gpu

EIG_RTOL = 2.5e-13


@pytest.fixture(scope="module")
def env():
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    yield torch, lre, ctx
    lre.lre_destroy(ctx)


def _kron(vs):
    out = np.ones(1, dtype=np.complex128)
    for v in vs:
        out = np.kron(out, np.asarray(v, dtype=np.complex128))
    return out


def _weight_state(n, k):
    v = np.array([1.0 if bin(i).count("1") == k else 0.0 for i in range(2 ** n)], dtype=np.complex128)
    return v / np.linalg.norm(v)


def _cluster(n):
    v = np.ones(2 ** n, dtype=np.complex128)
    for i in range(2 ** n):
        v[i] = (-1) ** bin(i & (i >> 1)).count("1")
    return v / np.linalg.norm(v)


def _vectors(n):
    s = np.sqrt(0.5)
    return {
        "plus": _kron([[s, s]] * n),
        "plus i": _kron([[s, 1j * s]] * n),
        "equal product": _kron([[np.cos(0.3), np.sin(0.3)]] * n),
        "0.8 0.6 product": _kron([[0.8, 0.6]] * n),
        "phased product": _kron([[np.cos(0.3), np.exp(0.7j) * np.sin(0.3)]] * n),
        "unequal product": _kron([[np.cos(0.2 + 0.3 * q), np.exp(0.4j * q) * np.sin(0.2 + 0.3 * q)] for q in range(n)]),
        "cluster": _cluster(n),
        "W": _weight_state(n, 1),
        "Dicke": _weight_state(n, min(2, n)),
    }


def _inputs(n):
    """Rank-one states, their mixtures with I/d, and (1 + e) P - e I/d."""
    d = 2 ** n
    eye = np.eye(d) / d
    for name, v in _vectors(n).items():
        p = np.outer(v, v.conj())
        yield name, p
        yield name + " + I", 0.9 * p + 0.1 * eye
        yield name + " - I", 1.05 * p - 0.05 * eye


def _check(env, m, n, name, eig=True):
    torch, lre, ctx = env
    mu = torch.from_numpy(m).cuda()
    out = torch.full_like(mu, float("nan"))
    em, er = [torch.full((2 ** n,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2)]
    lre.lre_project(ctx, mu, n, out, em if eig else None, er if eig else None)
    lre.lre_sync(ctx)
    ref, lam_mu, lam = project.smolin(m.astype(np.complex128))
    got = out.cpu().numpy()
    assert np.isfinite(got.view(np.float32)).all(), name
    assert rel_fro(got, ref) <= 1e-6, (name, rel_fro(got, ref))
    assert np.array_equal(got, got.conj().T), name
    if eig:
        tol = EIG_RTOL * np.abs(lam_mu).max()
        np.testing.assert_allclose(em.cpu().numpy(), lam_mu, rtol=0, atol=tol, err_msg=name)
        np.testing.assert_allclose(er.cpu().numpy(), lam, rtol=0, atol=tol, err_msg=name)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("eig", [True, False])
def test_structured_states(env, n, eig):
    for name, m in _inputs(n):
        _check(env, m.astype(np.complex64), n, name, eig)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("scale", [1e-30, 1e-20, 1e-9, 1e12, 1e30])
def test_scaled_inputs(env, n, scale):
    """The projection keeps the input's trace, so it scales with it."""
    rng = np.random.default_rng(n)
    g = rng.standard_normal((2 ** n, 2 ** n)) + 1j * rng.standard_normal((2 ** n, 2 ** n))
    noisy = _vectors(n)["W"]
    noisy = np.outer(noisy, noisy.conj()) + 0.05 * (g + g.conj().T) / 2 ** n
    for name, m in list(_inputs(n)) + [("noisy", noisy)]:
        _check(env, (m * scale).astype(np.complex64), n, "%s x %g" % (name, scale))


_PAULI = [np.eye(2), np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.diag([1, -1])]


def _stabilizer(n, k, rng):
    """The state of k commuting Pauli strings of value +-1: a projector of rank 2^(n-k), over its rank."""
    d = 2 ** n
    rho, done = np.eye(d, dtype=np.complex128), []
    while len(done) < k:
        p = np.ones((1, 1), dtype=np.complex128)
        for _ in range(n):
            p = np.kron(p, _PAULI[rng.integers(4)])
        t = rho @ (np.eye(d) + rng.choice([-1, 1]) * p) / 2
        if all(np.allclose(p @ g, g @ p) for g in done) and 0.4 < np.trace(t).real / np.trace(rho).real < 0.6:
            rho = t
            done.append(p)
    return rho / np.trace(rho).real


@pytest.mark.parametrize("n", [2, 3, 4, 5])
def test_projectors(env, n):
    """Eigenvalues of high multiplicity, T in many blocks: stabilizer projectors, sums of
    two, and (1 + e) P - e I/d."""
    rng = np.random.default_rng(n)
    eye = np.eye(2 ** n) / 2 ** n
    plus, minus = _vectors(n)["plus"], _kron([[np.sqrt(0.5), -np.sqrt(0.5)]] * n)
    _check(env, (0.5 * np.outer(plus, plus) + 0.5 * np.outer(minus, minus)).astype(np.complex64), n, "plus and minus")
    for it in range(150):
        m = _stabilizer(n, int(rng.integers(1, n + 1)), rng)
        if it % 3 == 2:
            w = rng.choice([0.5, rng.uniform(0.1, 0.9)])
            m = w * m + (1 - w) * _stabilizer(n, int(rng.integers(1, n + 1)), rng)
        e = rng.choice([0.0, 0.05, 0.3, -0.2])
        _check(env, ((1 + e) * m - e * eye).astype(np.complex64), n, "projector %d" % it, eig=it % 2 == 0)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
def test_diagonal_eigenvalues(env, n):
    """Diagonal input is its own tridiagonal form, and its counts are exact: what is left
    is half the last bracket, eps ||mu|| wide, and the rounding of its middle."""
    torch, lre, ctx = env
    rng = np.random.default_rng(n)
    for it in range(40):
        lam = rng.standard_normal(2 ** n).astype(np.float32)
        mu = torch.from_numpy(np.diag(lam).astype(np.complex64)).cuda()
        em = torch.empty(2 ** n, dtype=torch.float64, device="cuda")
        lre.lre_project(ctx, mu, n, torch.empty_like(mu), em)
        lre.lre_sync(ctx)
        want = np.sort(lam.astype(np.float64))[::-1]
        tol = np.finfo(np.float64).eps * np.abs(want).max()
        np.testing.assert_allclose(em.cpu().numpy(), want, rtol=0, atol=tol)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("value", [np.nan, np.inf, complex(0, np.nan)])
def test_input_that_is_not_finite_is_reported(env, n, value):
    torch, lre, ctx = env
    d = 2 ** n
    for r, c in ((0, 0), (0, d - 1), (d - 2, d - 1), (d - 1, d - 1)):
        if r == c and np.isfinite(np.real(value)):
            continue  # the diagonal's imaginary part is not read
        m = (np.eye(d) / d).astype(np.complex64)
        m[r, c] = value
        mu = torch.from_numpy(m).cuda()
        out = torch.full_like(mu, 3.0)
        with pytest.raises(lre.LreError) as e:
            lre.lre_project(ctx, mu, n, out)
        assert e.value.status == lre.LRE_ERR_EIG_FAILED
        lre.lre_sync(ctx)
        assert (out == 3.0).all()
    _check(env, (np.eye(d) / d).astype(np.complex64), n, "the next call")


@pytest.mark.parametrize("n", [1, 4])
def test_the_call_synchronises(env, n):
    torch, lre, ctx = env
    mu = (torch.eye(2 ** n, dtype=torch.complex64) / 2 ** n).cuda()
    out = torch.empty_like(mu)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        torch.cuda._sleep(20_000_000)
        lre.lre_project(ctx, mu, n, out, stream=stream)
        assert stream.query()
    assert torch.equal(out, mu)


def test_captured_in_a_graph(env):
    torch, lre, ctx = env
    n = 4
    g = torch.Generator().manual_seed(1)
    a, b = [torch.randn((16, 16), dtype=torch.complex64, generator=g) for _ in range(2)]
    a, b = [((x + x.conj().T) / 16).cuda() for x in (a, b)]
    want = torch.empty_like(b)
    lre.lre_project(ctx, b, n, want)
    mu, out = a.clone(), torch.empty_like(a)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        lre.lre_project(ctx, mu, n, out, stream=torch.cuda.current_stream())
    mu.copy_(b)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    mu[0, 0] = float("nan")
    graph.replay()
    with pytest.raises(lre.LreError) as e:
        lre.lre_sync(ctx)
    assert e.value.status == lre.LRE_ERR_EIG_FAILED
