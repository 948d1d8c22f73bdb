"""The derivative pass's workspace holds what its launch writes, on a device of any SM count (CPU).

The CTAs per block, and with them the rows of partial sums and the place of the reordered dL/dF
behind them, depend on the device's SMs: the workspace has to be sized from the same count.
"""
import ctypes as C

import numpy as np
import pytest

from paper_1305_4196_gb300 import build as B


@pytest.fixture(scope="module")
def shape():
    B.build()
    f = C.CDLL(B.LIB).mdgb_backward_shape
    f.argtypes = [C.c_void_p, C.c_int64, C.c_int32, C.c_int32, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p]

    def call(nc, n, nsp, fp64, sms):
        nc = np.array(nc, dtype=np.int32)
        split, at, size = C.c_int32(), C.c_int64(), C.c_int64()
        assert f(nc.ctypes.data, n, nsp, 0 if fp64 else 1, sms, C.byref(split), C.byref(at), C.byref(size)) == 0
        return split.value, at.value, size.value
    return call


@pytest.mark.parametrize("nc", [(4, 4, 4), (6, 6, 6), (8, 8, 8), (12, 8, 16), (34, 34, 34)])
@pytest.mark.parametrize("nsp", [1, 2, 3, 4])
@pytest.mark.parametrize("fp64", [False, True])
def test_workspace_holds_the_launch(shape, nc, nsp, fp64):
    blocks = nc[0] * nc[1] * nc[2] // 8
    for n in (1, 33, 2048, 641 * blocks, 700 * blocks + 1):
        for sms in (1, 16, 132, 148, 152, 160, 188, 264, 1024):
            split, at, size = shape(nc, n, nsp, fp64, sms)
            assert 1 <= split <= 8
            rows = blocks * split  # one row of partial sums per CTA, behind the totals
            assert at >= 2 * nsp * nsp * (1 + rows) and at % 4 == 0
            assert size >= at + n * (4 if fp64 else 2)


def test_the_split_follows_the_devices_sms(shape):
    """64 blocks of 641 and more atoms (the case in which a workspace sized for 152 SMs is too
    small for a launch on 188): five CTAs per block at 152 SMs, six at 188, in any order of calls."""
    n = 64 * 641
    for _ in range(2):
        assert shape((8, 8, 8), n, 2, False, 152)[0] == 5
        assert shape((8, 8, 8), n, 2, False, 188)[0] == 6
