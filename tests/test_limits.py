"""Index sizes that are refused before any device work (no GPU needed)."""
import ctypes

import numpy as np

from paper_2112_10408_gb300 import tnn


def test_more_than_2_30_segments_are_refused_as_out_of_memory():
    # 201 trajectories of odd length in segments of two: (n + 201) / 2 segments
    n = (1 << 31) - 65
    off = np.append(np.arange(201), n).astype(np.int64)
    assert int(((np.diff(off) + 1) // 2).sum()) > 1 << 30
    L = tnn.load_library()
    p = tnn.tnn_build_params()
    p.seg_len = 2
    for i in range(4):
        p.sigma[i] = 1.0
    h = ctypes.c_void_p()
    st = L.tnn_build_segments(ctypes.c_void_p(16), n, ctypes.c_void_p(off.ctypes.data), 201, ctypes.byref(p), None,
                              ctypes.byref(h))
    assert st == 2 and b"2^30" in L.tnn_last_error() and not h.value
