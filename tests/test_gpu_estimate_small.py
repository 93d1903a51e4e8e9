"""The one-launch estimate for n <= 6 (uniform shots) against the oracle: bits of
theta, rho within 1e-6, over both count types and the edges of its range (the
largest shots whose sums fit int32, counts off a 16-byte boundary, no rho)."""
import numpy as np
import pytest

from oracle import direct
from tests.gpu_util import ctx_and_lre, need_gpu, rel_fro

pytestmark = pytest.mark.gpu


def _counts(n, shots, dtype, seed):
    rng = np.random.default_rng(seed)
    p = rng.dirichlet(np.full(2 ** n, 0.3), size=3 ** n)
    return np.stack([rng.multinomial(shots, q) for q in p]).astype(dtype)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("dtype,shots", [(np.int16, 1), (np.int16, 32767), (np.int32, 1000), (np.int32, "most"),
                                         (np.int32, "over")])
@pytest.mark.parametrize("shift", [0, 1])
def test_matches_oracle(n, dtype, shots, shift):
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    most = (2 ** 31 - 2) // 3 ** n
    shots = {"most": most, "over": most + 1}.get(shots, shots)
    c = _counts(n, shots, dtype, 10 * n + shift)
    buf = torch.zeros(c.size + 8, dtype=torch.int16 if dtype == np.int16 else torch.int32, device="cuda")
    view = buf[shift:shift + c.size].view(c.shape)  # shift 1: off the vector loads' alignment
    view.copy_(torch.from_numpy(c))
    try:
        want = direct.estimate(c, shots, n)
        for with_rho in (True, False):
            theta = torch.full((4 ** n,), float("nan"), dtype=torch.float64, device="cuda")
            rho = torch.full((2 ** n, 2 ** n), float("nan"), dtype=torch.complex64, device="cuda") if with_rho else None
            lre.lre_profile(ctx, True)
            lre.lre_estimate(ctx, view, shots, n, theta, rho)
            lre.lre_sync(ctx)
            names = [k for k, _ in lre.lre_profile_records(ctx)]
            lre.lre_profile(ctx, False)
            assert (names == ["estimate_small"]) == (shift == 0 and shots <= most), names
            np.testing.assert_array_equal(theta.cpu().numpy(), want)
            if with_rho:
                assert rel_fro(rho.cpu().numpy(), direct.mu(want, n)) <= 1e-6
    finally:
        lre.lre_destroy(ctx)


@pytest.mark.parametrize("n", [1, 4, 6])
def test_total_mismatch_is_latched(n):
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    try:
        c = torch.from_numpy(_counts(n, 100, np.int32, n)).cuda()
        theta = torch.empty(4 ** n, dtype=torch.float64, device="cuda")
        lre.lre_estimate(ctx, c, 101, n, theta)
        with pytest.raises(lre.LreError) as e:
            lre.lre_sync(ctx)
        assert e.value.status == lre.LRE_ERR_SHOTS_MISMATCH
    finally:
        lre.lre_destroy(ctx)
