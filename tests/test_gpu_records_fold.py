"""Device shot records folded without dense counts (9 <= n <= 12, rows of 16-byte
multiples, 27 shots a basis within 16 bits): the same bits as the dense counts of the
same records, also one step outside the rule, and a record outside the outcomes is
reported."""
import numpy as np
import pytest

from tests.gpu_util import ctx_and_lre, need_gpu

pytestmark = pytest.mark.gpu


def _records(torch, n, shots, seed, shift=0):
    """GHZ-like records: half the shots in two outcomes, the rest spread."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = torch.randint(0, 2 ** n, (3 ** n, shots), generator=g, device="cuda", dtype=torch.int32)
    e = torch.randint(0, 4, (3 ** n, shots), generator=g, device="cuda", dtype=torch.int32)
    r = torch.where(e < 2, e * (2 ** n - 1), r).to(torch.int16)
    buf = torch.zeros(r.numel() + 8, dtype=torch.int16, device="cuda")
    view = buf[shift:shift + r.numel()].view(r.shape)
    view.copy_(r)
    return view


@pytest.mark.parametrize("n,shots,shift,folded", [
    (8, 1000, 0, False), (9, 8, 0, True), (9, 1000, 0, True), (9, 1208, 0, True), (9, 1216, 0, False),
    (9, 1004, 0, False), (9, 800, 3, False), (10, 504, 0, True), (10, 512, 0, True), (10, 520, 8, True),
    (10, 1208, 0, True), (11, 1000, 0, True), (11, 1208, 0, True), (12, 504, 0, True), (12, 1208, 0, True)])
def test_same_bits_as_dense_counts(n, shots, shift, folded):
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    try:
        rec = _records(torch, n, shots, n + shots, shift)
        counts = torch.empty((3 ** n, 2 ** n), dtype=torch.int32, device="cuda")
        lre.lre_histogram(ctx, rec, n, counts)
        out = []
        for arg, kind in ((counts, None), (rec, lre.LRE_SHOTS_U16)):
            theta = torch.full((4 ** n,), float("nan"), dtype=torch.float64, device="cuda")
            rho = torch.full((2 ** n, 2 ** n), float("nan"), dtype=torch.complex64, device="cuda")
            lre.lre_profile(ctx, True)
            lre.lre_estimate(ctx, arg, shots, n, theta, rho, kind=kind)
            lre.lre_sync(ctx)
            names = {k for k, _ in lre.lre_profile_records(ctx)}
            lre.lre_profile(ctx, False)
            if kind is not None:
                assert ("records_fold3" in names, "histogram" in names) == (folded, not folded), names
            out.append((theta, rho))
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        theta = torch.empty(4 ** n, dtype=torch.float64, device="cuda")
        lre.lre_estimate(ctx, rec, shots, n, theta, kind=lre.LRE_SHOTS_U16)  # without rho
        lre.lre_sync(ctx)
        assert torch.equal(theta, out[0][0])
    finally:
        lre.lre_destroy(ctx)


@pytest.mark.parametrize("n", [9, 12])
def test_out_of_range_record_is_reported(n):
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    try:
        rec = _records(torch, n, 64, 1)
        rec[3 ** n - 1, 5] = 2 ** n
        theta = torch.empty(4 ** n, dtype=torch.float64, device="cuda")
        lre.lre_estimate(ctx, rec, 64, n, theta, kind=lre.LRE_SHOTS_U16)
        with pytest.raises(lre.LreError) as e:
            lre.lre_sync(ctx)
        assert e.value.status == lre.LRE_ERR_INVALID_ARG
    finally:
        lre.lre_destroy(ctx)
