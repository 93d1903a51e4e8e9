"""Sturm counts by principal minors (tri_minor.cuh) where T falls into blocks and the
point is an eigenvalue of one of them: between the number of eigenvalues below the
point and the number of those not above it, in all three precisions.  Entries are
multiples of 1/8, exact in FP32."""
import ctypes

import numpy as np
import pytest

from tests.gpu_util import ctx_and_lre, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 4, 5, 8, 9, 17, 32, 63])
def test_split_matrices(n):
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    f = lre.load().lre_debug_minor_counts
    f.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    f.restype = ctypes.c_int
    rng = np.random.default_rng(n)
    try:
        for it in range(40):
            a = rng.integers(-8, 9, n) / 8.0
            b = rng.integers(1, 5, n) / 8.0 * (rng.random(n) < (0.0, 0.3, 0.7)[it % 3])
            if it == 0:
                a = np.arange(n) / 64.0  # a split T and a point on its first entry
            x = np.concatenate([a, [-2.0, 2.0]])
            w = np.linalg.eigvalsh(np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1))
            low = (w[None, :] < x[:, None] - 1e-9).sum(1)
            high = (w[None, :] <= x[:, None] + 1e-9).sum(1)
            da, db, dx = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (a, -b * b, x)]
            out = torch.empty((len(x), 3), dtype=torch.int32, device="cuda")
            assert f(ctx, da.data_ptr(), db.data_ptr(), n, dx.data_ptr(), len(x), out.data_ptr()) == 0
            got = out.cpu().numpy()
            for k, kind in enumerate(("FP64", "double-float", "FP32")):
                assert (low <= got[:, k]).all() and (got[:, k] <= high).all(), (it, kind, a, b, x, got[:, k], low, high)
    finally:
        lre.lre_destroy(ctx)
