"""Setting up an FP64 problem whose kernels store operators per element.

At N = 5 with the 25-point rule a problem of 8192 elements keeps some 350 MB of stored
operators.  Forming its host image takes less time than one thread takes to write as
many fresh bytes once: the pages come zeroed from the allocator and several threads
fill them.
"""

import ctypes
import os
import time

import numpy as np
import pytest

from paper_2005_02516_gb300 import esdg
from test_library_cpu import _build


@pytest.mark.skipif((os.cpu_count() or 1) < 4, reason="the set-up runs on several threads")
def test_stored_operators_are_formed_at_the_rate_of_memory():
    prepare, write = [], []
    for _ in range(4):
        lib, rc, h = _build(N=5, nx=64, ny=64, warp=0.05, rule=esdg.ESDG_RULE_SYMMETRIC)
        assert rc == 0
        K, Np, Nq, nb = ctypes.c_int(), ctypes.c_int(), ctypes.c_int(), ctypes.c_size_t()
        assert lib.esdg_sizes(h, ctypes.byref(K), ctypes.byref(Np), ctypes.byref(Nq), None, ctypes.byref(nb)) == 0
        q, b = np.ones((3, K.value, Nq.value)), np.zeros((K.value, Np.value))
        t0 = time.perf_counter()
        assert lib.esdg_prepare(h, b.ctypes.data, q.ctypes.data, esdg.ESDG_INIT_DEPTH) == 0
        prepare.append(time.perf_counter() - t0)
        lib.esdg_destroy(h)
        t0 = time.perf_counter()
        fresh = bytearray(nb.value)
        ctypes.memset((ctypes.c_char * nb.value).from_buffer(fresh), 1, nb.value)
        write.append(time.perf_counter() - t0)
        del fresh
    assert min(prepare) < min(write), (prepare, write)
