"""The six-qubit first pass of the per-basis-weighted estimate (n >= 7) against the
oracle: both count types, unequal shots, counts on both sides of the int32 / int64
switch of its parity transform, and counts off a 16-byte boundary (the two-qubit
passes).  |dtheta| <= 1e-12: at most 3^9 terms of magnitude 1 in FP64, as for the
passes it replaces; the rho bound is the rounding of its entries."""
import numpy as np
import pytest

from oracle import direct
from tests.gpu_util import ctx_and_lre, need_gpu, rel_fro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7, 8, 9])
@pytest.mark.parametrize("dtype,top,shift", [(np.int16, 9, 0), (np.int16, 500, 0), (np.int32, 500, 0),
                                             (np.int32, 2 ** 25 - 1, 0), (np.int32, 2 ** 25, 0),
                                             (np.int32, 2 ** 28, 0), (np.int32, 500, 1)])
def test_matches_oracle(n, dtype, top, shift):
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    rng = np.random.default_rng(n + top % 97)
    c = rng.integers(0, top, size=(3 ** n, 2 ** n), endpoint=True).astype(dtype)
    c[::7, 0] = top
    c[5] = 0
    c[5, 3] = 1  # a basis with a single shot
    N = c.sum(axis=1, dtype=np.int64)
    buf = torch.zeros(c.size + 8, dtype=torch.int16 if dtype == np.int16 else torch.int32, device="cuda")
    view = buf[shift:shift + c.size].view(c.shape)
    view.copy_(torch.from_numpy(c))
    try:
        theta = torch.full((4 ** n,), float("nan"), dtype=torch.float64, device="cuda")
        rho = torch.full((2 ** n, 2 ** n), float("nan"), dtype=torch.complex64, device="cuda")
        lre.lre_profile(ctx, True)
        lre.lre_estimate(ctx, view, torch.from_numpy(N).cuda(), n, theta, rho)
        lre.lre_sync(ctx)
        names = {k for k, _ in lre.lre_profile_records(ctx)}
        assert ("fold_first6_weighted" in names) == (shift == 0), names
        want = direct.estimate(c, N, n)
        np.testing.assert_allclose(theta.cpu().numpy(), want, atol=1e-12, rtol=0)
        assert rel_fro(rho.cpu().numpy(), direct.mu(want, n)) <= 1e-6
    finally:
        lre.lre_destroy(ctx)
