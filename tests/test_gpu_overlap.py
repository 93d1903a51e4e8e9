"""The estimate's launches set up while the kernel before them ends: back-to-back
calls that share the workspace, inputs rewritten between calls on the same stream,
and capture in a CUDA graph give the results of separate, synchronised calls."""
import numpy as np
import pytest

from tests.gpu_util import ctx_and_lre, need_gpu

pytestmark = pytest.mark.gpu


def _counts(torch, n, dtype, seed):
    from synth import gen
    c = torch.empty((3 ** n, 2 ** n), dtype=dtype, device="cuda")
    gen.gen_ghz(n, 0.1, 900, seed, c)
    torch.cuda.synchronize()
    return c


def _out(torch, n):
    return (torch.empty(4 ** n, dtype=torch.float64, device="cuda"),
            torch.empty((2 ** n, 2 ** n), dtype=torch.complex64, device="cuda"))


@pytest.mark.parametrize("dtype", ["int16", "int32"])
def test_back_to_back_calls_of_several_sizes(dtype):
    torch = need_gpu()
    dt = getattr(torch, dtype)
    lre, ctx = ctx_and_lre()
    try:
        sizes = (4, 7, 10, 6, 8, 11, 9, 7, 4)
        data = [_counts(torch, n, dt, 50 + k) for k, n in enumerate(sizes)]
        want = []
        for n, c in zip(sizes, data):
            t, r = _out(torch, n)
            lre.lre_estimate(ctx, c, 900, n, t, r)
            lre.lre_sync(ctx)
            torch.cuda.synchronize()
            want.append((t, r))
        for _ in range(3):
            got = [_out(torch, n) for n in sizes]
            work = [torch.zeros_like(c) for c in data]
            for n, c, w, (t, r) in zip(sizes, data, work, got):
                w.copy_(c)                       # another kernel writes the counts just before
                lre.lre_estimate(ctx, w, 900, n, t, r)
                w.zero_()                        # and rewrites them just after
            lre.lre_sync(ctx)
            for a, b in zip(got, want):
                assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    finally:
        lre.lre_destroy(ctx)


@pytest.mark.parametrize("n", [4, 7, 10])
def test_captured_in_a_graph(n):
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    try:
        c = _counts(torch, n, torch.int16, 3)
        other = _counts(torch, n, torch.int16, 4)
        t, r = _out(torch, n)
        lre.lre_estimate(ctx, other, 900, n, t, r)  # sizes the workspace
        lre.lre_sync(ctx)
        want = t.clone(), r.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            lre.lre_estimate(ctx, c, 900, n, t, r, stream=torch.cuda.current_stream())
        c.copy_(other)
        t.fill_(float("nan"))
        r.zero_()
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(t, want[0]) and torch.equal(r, want[1])
    finally:
        lre.lre_destroy(ctx)


def test_per_basis_chain():
    """Per-basis shots (FP64 chain, and lre_assemble): the same bits back to back, with
    counts and totals rewritten around each call, and from a graph."""
    torch = need_gpu()
    lre, ctx = ctx_and_lre()
    try:
        sizes = (3, 6, 10, 7, 11, 9, 1, 8)
        data = [_counts(torch, n, torch.int32, 90 + n) for n in sizes]
        shots = [c.sum(dim=1, dtype=torch.int64) for c in data]
        want = []
        for n, c, sh in zip(sizes, data, shots):
            t, r = _out(torch, n)
            lre.lre_estimate(ctx, c, sh, n, t, r)
            lre.lre_sync(ctx)
            torch.cuda.synchronize()
            want.append((t, r))
        for _ in range(3):
            got = []
            for n, c, sh in zip(sizes, data, shots):
                w, ws, (t, r) = c.clone(), sh.clone(), _out(torch, n)
                lre.lre_estimate(ctx, w, ws, n, t, r)
                w.zero_()
                ws.fill_(1)
                again = torch.empty_like(r)
                lre.lre_assemble(ctx, t, n, again)
                got.append((t, r, again, w, ws))
            lre.lre_sync(ctx)
            for a, b in zip(got, want):
                assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(a[2], b[1])
        n, c, sh = 7, data[3], shots[3]
        t, r = _out(torch, n)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            lre.lre_estimate(ctx, c, sh, n, t, r, stream=torch.cuda.current_stream())
        for _ in range(3):
            t.fill_(float("nan"))
            r.zero_()
            graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(t, want[3][0]) and torch.equal(r, want[3][1])
    finally:
        lre.lre_destroy(ctx)
