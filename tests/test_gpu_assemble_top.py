"""The assembly that starts in the last fold pass (n >= 7, uniform shots): against
the oracle where its counts are drawn on the CPU, and bit for bit against the
passes over plain T (which the seven-qubit first pass still takes) beyond."""
import numpy as np
import pytest

from oracle import direct
from tests.gpu_util import ctx_and_lre, need_gpu, rel_fro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7, 8, 9])
@pytest.mark.parametrize("dtype,shots", [(np.int16, 900), (np.int16, 9000), (np.int32, 300000), (np.int32, 3000000)])
def test_matches_oracle(n, dtype, shots):
    """Split-plane, int32 and int64 sums into the last pass; rho exactly Hermitian."""
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    try:
        rng = np.random.default_rng(n)
        c = rng.multinomial(shots, rng.dirichlet(np.full(2 ** n, 0.3)), size=3 ** n).astype(dtype)
        theta = torch.empty(4 ** n, dtype=torch.float64, device="cuda")
        rho = torch.full((2 ** n, 2 ** n), float("nan"), dtype=torch.complex64, device="cuda")
        lre.lre_estimate(ctx, torch.from_numpy(c).cuda(), shots, n, theta, rho)
        lre.lre_sync(ctx)
        want = direct.estimate(c, shots, n)
        np.testing.assert_array_equal(theta.cpu().numpy(), want)
        got = rho.cpu().numpy()
        assert rel_fro(got, direct.mu(want, n)) <= 1e-6
        np.testing.assert_array_equal(got, got.conj().T)
    finally:
        lre.lre_destroy(ctx)


@pytest.mark.parametrize("n", [8, 9, 10, 11, 12, 13])
def test_same_bits_as_the_passes_over_plain_t(n):
    torch = need_gpu()
    import bench
    from synth import gen
    c = torch.empty((3 ** n, 2 ** n), dtype=torch.int16, device="cuda")
    gen.gen_ghz(n, 0.05, 1000, 40 + n, c)
    out = []
    for seven in (0, 1):
        lre, ctx = ctx_and_lre()
        try:
            bench.set_first7(lre, ctx, seven)
            theta = torch.empty(4 ** n, dtype=torch.float64, device="cuda")
            rho = torch.full((2 ** n, 2 ** n), float("nan"), dtype=torch.complex64, device="cuda")
            lre.lre_profile(ctx, True)
            lre.lre_estimate(ctx, c, 1000, n, theta, rho)
            lre.lre_sync(ctx)
            names = {k for k, _ in lre.lre_profile_records(ctx)}
            assert ("fold_first7_mma" in names) == (seven == 1), names
            out.append((theta, rho))
        finally:
            lre.lre_destroy(ctx)
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
