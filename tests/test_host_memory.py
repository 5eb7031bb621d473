"""Host set-up when threads or memory run out: every range of elements is done
once, started threads are joined, and the C entries return ESDG_ENOMEM instead of
letting an exception through.
"""

import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# a thread that cannot be started from the `limit`-th on
PROGRAM = r"""
#include "host_threads.hpp"
#include <atomic>
#include <cstdio>

static int started = 0, limit = 0;
static bool no_memory = false;

struct Thread {
    std::thread t;
    template <typename F>
    explicit Thread(F f) {
        if (started == limit) {
            if (no_memory) throw std::bad_alloc();
            throw std::system_error(std::make_error_code(std::errc::resource_unavailable_try_again));
        }
        ++started;
        t = std::thread(f);
    }
    void join() { t.join(); }
    static unsigned hardware_concurrency() { return 8; }
};

static int covered_once(int K, bool worker_fails) {
    std::vector<std::atomic<int>> hits(K);
    for (auto& h : hits) h = 0;
    std::atomic<bool> fail_next(worker_fails);
    const std::thread::id caller = std::this_thread::get_id();
    esdg::in_threads<Thread>(K, 4, 16, [&](int e0, int e1) {
        if (std::this_thread::get_id() != caller && fail_next.exchange(false)) throw std::bad_alloc();
        for (int e = e0; e < e1; ++e) ++hits[e];
    });
    for (auto& h : hits)
        if (h != 1) return 0;
    return 1;
}

int main() {
    for (int mem = 0; mem < 2; ++mem)
        for (int l = 0; l < 9; ++l)
            for (int K : {1, 3, 31, 32, 33, 1000})
                for (int fails = 0; fails < 2; ++fails) {
                    no_memory = mem;
                    limit = l;
                    started = 0;
                    if (!covered_once(K, fails)) return 1;
                }
    // what the calling thread's own range throws comes through, after the join
    limit = 8;
    started = 0;
    const std::thread::id caller = std::this_thread::get_id();
    std::atomic<int> others(0);
    try {
        esdg::in_threads<Thread>(64, 8, 16, [&](int, int) {
            if (std::this_thread::get_id() == caller) throw std::bad_alloc();
            ++others;
        });
        return 2;
    } catch (const std::bad_alloc&) {
    }
    return others == 7 ? 0 : 3;
}
"""


def test_ranges_whose_thread_cannot_start_are_done_by_the_caller(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_2005_02516_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0


# address space for all but the image of an N = 5 problem (about 400 MB), then for
# the mesh of a larger one
LIMITED = r"""
import ctypes, resource, sys
sys.path[:0] = [%(root)r, %(tests)r]
import numpy as np
from paper_2005_02516_gb300 import esdg
from test_library_cpu import _build, _cfg

def vm():
    return int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()

lib, rc, h = _build(N=5, nx=64, ny=64, warp=0.05, rule=esdg.ESDG_RULE_SYMMETRIC)
assert rc == 0
K, Np, Nq = ctypes.c_int(), ctypes.c_int(), ctypes.c_int()
lib.esdg_sizes(h, ctypes.byref(K), ctypes.byref(Np), ctypes.byref(Nq), None, None)
q, b = np.ones((3, K.value, Nq.value)), np.zeros((K.value, Np.value))
free = resource.getrlimit(resource.RLIMIT_AS)
resource.setrlimit(resource.RLIMIT_AS, (vm() + (200 << 20), free[1]))
assert lib.esdg_prepare(h, b.ctypes.data, q.ctypes.data, esdg.ESDG_INIT_DEPTH) == esdg.ESDG_ENOMEM
assert b"memory" in lib.esdg_last_error(h)
h2 = ctypes.c_void_p()
assert lib.esdg_build_operators(ctypes.byref(_cfg(N=5, nx=512, ny=256)), ctypes.byref(h2)) == esdg.ESDG_ENOMEM
assert not h2.value
resource.setrlimit(resource.RLIMIT_AS, free)
assert lib.esdg_prepare(h, b.ctypes.data, q.ctypes.data, esdg.ESDG_INIT_DEPTH) == 0
lib.esdg_destroy(h)
print("done")
"""


@pytest.mark.skipif(not sys.platform.startswith("linux"), reason="address-space limits")
def test_host_memory_that_runs_out_is_an_error_code():
    code = LIMITED % dict(root=ROOT, tests=os.path.join(ROOT, "tests"))
    env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1")
    p = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300, env=env)
    assert p.returncode == 0 and "done" in p.stdout, p.stderr[-2000:]
