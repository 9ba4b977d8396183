"""The plan that shares blocks and SMs out among the entanglement spectrum's streams
(host code): every block has a lane, the largest blocks the least loaded one, no
lane has fewer SMs than the one-launch panels of its blocks need, up to panels of
2,048 rows -- a panel keeps 135 float-float numbers of each of a CTA's rows and one
per column in 216 KB -- and the shares do not exceed the GPU."""
import ctypes
from math import comb

import numpy as np
import pytest

from paper_2605_07621_gb300 import _lib


def _plan(m, lanes, sms):
    lib = ctypes.CDLL(_lib.LIB_PATH)
    f = lib._ZN3edk15entangle_sharesEPKxiiiPiS2_
    f.restype, f.argtypes = None, [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_void_p,
                                   ctypes.c_void_p]
    m = np.asarray(m, np.int64)
    lane, share = np.full(len(m), -1, np.int32), np.full(lanes, -1, np.int32)
    f(m.ctypes.data, len(m), lanes, sms, lane.ctypes.data, share.ctypes.data)
    return lane, share


def _blocks(n, up):
    a = n // 2
    return [min(comb(a, s), comb(n - a, up - s)) for s in range(max(0, up - (n - a)), min(a, up) + 1)]


def _need(m):
    rows = min(m, 2048)
    g = 1
    while rows > 64 and (-(-rows // g) * 135 + rows + 1 + 4) * 8 > 216 * 1024:
        g += 1
    return g


@pytest.mark.parametrize("n,up", [(8, 4), (20, 10), (24, 12), (25, 12), (28, 14), (28, 11), (28, 9), (30, 15), (32, 16),
                                  (32, 12), (34, 9)])
@pytest.mark.parametrize("lanes", [1, 2, 3, 5])
@pytest.mark.parametrize("sms", [132, 152])
def test_shares(n, up, lanes, sms):
    m = _blocks(n, up)
    lane, share = _plan(m, lanes, sms)
    assert lane.min() >= 0 and lane.max() < lanes
    assert share.min() >= 0 and share.sum() <= sms
    for i, k in enumerate(lane):
        assert share[k] >= max(1, _need(m[i]))
    assert share.sum() >= 0.9 * sms - lanes  # nearly all of the GPU is given out


def test_one_block_takes_all():
    lane, share = _plan([924], 5, 152)
    assert share[lane[0]] == 152


def test_few_sms():
    lane, share = _plan(_blocks(32, 16), 5, 16)
    assert (share <= 16).all() and (share[np.unique(lane)] >= 1).all()
