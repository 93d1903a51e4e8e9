"""Two threads, each with a context and a stream of its own, on calls of different
sizes of the same kernels: a kernel's dynamic shared-memory limit is shared by all
threads, so the smaller size must not lower it under the other's launch."""
import threading

import numpy as np
import pytest

from tests.gpu_util import ctx_and_lre, need_gpu
from tests.test_gpu_projection import _hermitian_with_spectrum

pytestmark = pytest.mark.gpu


def _together(torch, small, large, rounds):
    """large() `rounds` times on one thread while the other repeats small()."""
    errors, stop = [], threading.Event()

    def run(f, more):
        lre, ctx = ctx_and_lre()
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                while more():
                    f(lre, ctx, stream)
                lre.lre_sync(ctx, stream)
        except Exception as e:  # noqa: BLE001 - reported by the test
            errors.append(e)
        finally:
            stop.set()
            lre.lre_destroy(ctx)

    left = iter(range(rounds))
    ts = [threading.Thread(target=run, args=(small, lambda: not stop.is_set())),
          threading.Thread(target=run, args=(large, lambda: next(left, None) is not None))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors


def test_projections():
    torch = need_gpu()

    def call(n):
        d = 2 ** n
        lam = -np.random.default_rng(n).uniform(0, 0.5 / d, d)
        lam[-4:] = (0.1, 0.2, 0.3, 0.4)
        # a rotation of the first 64 levels only: cheap to make at d = 4096
        m = np.diag(lam / lam.sum()).astype(np.complex64)
        u = _hermitian_with_spectrum(lam[-64:] / lam.sum(), n)
        m[-64:, -64:] = u
        mu = torch.from_numpy(m).cuda()
        out = torch.empty_like(mu)
        return lambda lre, ctx, s: lre.lre_project(ctx, mu, n, out, stream=s)

    small, large = call(6), call(12)
    torch.cuda.synchronize()
    _together(torch, small, large, 25)


def test_records():
    torch = need_gpu()

    def call(n, shots):
        rec = torch.randint(0, 2 ** n, (3 ** n, shots), device="cuda", dtype=torch.int32).to(torch.int16)
        theta = torch.empty(4 ** n, dtype=torch.float64, device="cuda")
        return lambda lre, ctx, s: lre.lre_estimate(ctx, rec, shots, n, theta, kind=lre.LRE_SHOTS_U16, stream=s)

    small, large = call(9, 8), call(12, 64)
    torch.cuda.synchronize()
    _together(torch, small, large, 400)
