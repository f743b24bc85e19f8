"""The list of near pairs (csrc/near.cu) on sets with more ties than it holds.

Points on two sites have every cross-site pair at one distance: N^2 / 4 near pairs,
which pass 2^31 from N = 92 682 on and whose 32-bit sums then wrap. Such a list
must come back empty with its overflow word set and nothing written; the same set
with room for its pairs must come back whole."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1105_2769_gb300 import _lib

pytestmark = pytest.mark.gpu


class Near(ctypes.Structure):
    _fields_ = [("tau", ctypes.c_void_p), ("pairs", ctypes.c_void_p), ("count", ctypes.c_void_p),
                ("rest", ctypes.c_void_p * 8)]


def _near_list(X):
    """(overflow word, number of pairs, what stands behind the list's memory)"""
    lib = ctypes.CDLL(_lib.LIB_PATH)
    size = lib._Z14mbm_near_bytesl
    size.restype, size.argtypes = ctypes.c_size_t, [ctypes.c_int64]
    fill = lib._Z16launch_near_listPK6float4S1_lPvPiS3_P7MbmNearP11CUstream_st
    fill.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p,
                     ctypes.c_void_p, ctypes.c_void_p, ctypes.POINTER(Near), ctypes.c_void_p]
    n = len(X)
    xh = torch.zeros(n, 4, device="cuda")
    xh[:, :3] = torch.from_numpy(X).cuda()
    xl = torch.zeros(n, 4, device="cuda")
    need = size(n)
    mem = torch.full((need + (1 << 20),), 0x5A, dtype=torch.uint8, device="cuda")
    words = torch.zeros(64, dtype=torch.int32, device="cuda")
    near = Near()
    stream = torch.cuda.current_stream().cuda_stream
    assert fill(xh.data_ptr(), xl.data_ptr(), n, mem.data_ptr(), words.data_ptr(),
                words.data_ptr() + 4, ctypes.byref(near), stream) == 0
    torch.cuda.synchronize()
    count = mem[near.count - mem.data_ptr():][:4].view(torch.int32).item()
    return words[0].item(), count, bool((mem[need:] == 0x5A).all())


@pytest.mark.parametrize("n", [40, 400, 92682, 92700, 131072])
def test_two_sites(n):
    X = np.zeros((n, 3), dtype=np.float32)
    X[n // 2:, 0] = 1.0
    overflow, count, untouched = _near_list(X)
    assert untouched
    fits = (n // 2) * (n - n // 2) <= 16 * n
    assert (overflow, count) == ((0, (n // 2) * (n - n // 2)) if fits else (1, 0))
