"""The records' fold without dense counts refuses what its 16-bit bins and sums, or its
vector loads, cannot hold, whoever calls it (no device work: the arguments decide)."""
import ctypes

import pytest

from paper_1602_08604_gb300 import build, lre

UNSUPPORTED = 2


@pytest.mark.parametrize("n,shots,offset", [(8, 1000, 0), (13, 1000, 0), (9, 1216, 0), (12, 32760, 0), (11, 1 << 40, 0),
                                            (10, 1004, 0), (10, 0, 0), (10, -8, 0), (10, 1000, 2)])
def test_refused(n, shots, offset):
    build.build()
    f = lre.load()._ZN3lre16records_fold_runEP7lre_ctxPKtliPvS4_P11CUstream_st
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_int] + [ctypes.c_void_p] * 3
    f.restype = ctypes.c_int
    assert f(None, 4096 + offset, shots, n, None, None, None) == UNSUPPORTED
