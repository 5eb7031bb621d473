"""The pair operator that the FP64 stages read, decoded from its fixed-point limbs,
against the oracle's metric-averaged Q_skew on a curved and on a stretched mesh: every
unordered pair once, from the lane and step of the kernel's schedule, zeros elsewhere.

Tolerance: an entry is stored to 2^-60 of twice the largest row sum of its direction
(at most Nh of the largest entry); library and oracle evaluate the reference
operators, metrics and averages in FP64 on their own, a few hundred roundings.
"""

import ctypes

import numpy as np
import pytest

from oracle import Oracle
from oracle.sbp import SBPOracle
from paper_2005_02516_gb300 import esdg
from test_library_cpu import _cfg, _lib

RULES = [("modal", N, rule) for N in range(1, 6) for rule in ("symmetric", "collapsed") if (N, rule) != (5, "collapsed")
         ] + [("sbp", N, "symmetric") for N in range(1, 5)]


def _context(method, N, rule, dom):
    c = _cfg(N=N, nx=4, ny=3, warp=0.05, method=esdg.ESDG_METHOD_SBP if method == "sbp" else esdg.ESDG_METHOD_MODAL,
             rule=esdg.ESDG_RULE_SYMMETRIC if rule == "symmetric" else esdg.ESDG_RULE_COLLAPSED)
    c.x0, c.x1, c.y0, c.y1 = dom
    lib, h = _lib(), ctypes.c_void_p()
    assert lib.esdg_build_operators(ctypes.byref(c), ctypes.byref(h)) == 0
    return lib, h


def _order(lib, h, kind, o, okind, K, n):
    """Index in the oracle's points of each of the library's, the same in all elements."""
    x, y = np.zeros((K, n)), np.zeros((K, n))
    assert lib.esdg_get_points(h, kind, x.ctypes.data, y.ctypes.data) == 0
    xo, yo = o.points(okind)
    size = [np.ptp(xo), np.ptp(yo)]
    d = np.abs(x[0][:, None] - xo[0][None]) / size[0] + np.abs(y[0][:, None] - yo[0][None]) / size[1]
    p = d.argmin(axis=1)
    assert sorted(p) == list(range(n))
    assert np.abs(x - xo[:, p]).max() < 1e-12 * size[0] and np.abs(y - yo[:, p]).max() < 1e-12 * size[1]
    return p


@pytest.mark.parametrize("dom", [(-1.0, 1.0, -1.0, 1.0), (-100.0, 100.0, -1.0, 1.0)], ids=["square", "stretched"])
@pytest.mark.parametrize("method,N,rule", RULES)
def test_each_pair_is_stored_once_with_the_oracles_value(method, N, rule, dom):
    args = dict(x0=dom[0], x1=dom[1], y0=dom[2], y1=dom[3], ax=0.05, ay=0.05)
    o = SBPOracle(N, 4, 3, **args) if method == "sbp" else Oracle(N, 4, 3, rule=rule, **args)
    lib, h = _context(method, N, rule, dom)
    V, F = o.Nq, 0 if method == "sbp" else o.Nfq
    perm = _order(lib, h, esdg.ESDG_POINTS_VOLQ, o, "volq", o.K, V)
    if F:
        perm = np.concatenate([perm, V + _order(lib, h, esdg.ESDG_POINTS_FACEQ, o, "faceq", o.K, F)])
    steps = ctypes.c_int()
    assert lib.esdg_pair_operator(h, ctypes.byref(steps), None) == 0
    q = np.full((o.K, steps.value, 32, 2), np.nan)
    assert lib.esdg_pair_operator(h, ctypes.byref(steps), q.ctypes.data) == 0
    lib.esdg_destroy(h)
    ks = np.arange(o.K)
    if method == "sbp":
        Q = o.sbp_operators(ks)
    else:
        m, ref = o.mesh, o.ref
        Q = [0.5 * (ref.Qhr[None] * (a[:, :, None] + a[:, None, :]) + ref.Qhs[None] * (b[:, :, None] + b[:, None, :]))
             for a, b in ((m.rxJ, m.sxJ), (m.ryJ, m.syJ))]
    want = np.stack([(x - x.transpose(0, 2, 1))[:, perm][:, :, perm] / 4 for x in Q], axis=-1)
    L = max(V, F)
    groups = 2 if L <= 16 else 1
    vv, vf = -(-(V // 2) // groups), -(-L // groups) if F else 0
    assert steps.value == vv + vf
    got = np.zeros_like(want)
    seen = set()
    for st in range(steps.value):
        for lane in range(32):
            j, hf = (lane % 16, lane // 16) if groups == 2 else (lane, 0)
            pair = None
            if j < V and st < vv:
                d = 1 + st + vv * hf
                if d <= V // 2 and not (2 * d == V and j >= V // 2):
                    pair = j, (j + d) % V
            elif j < V:
                t = st - vv + vf * hf
                if t < L and (j + t) % L < F:
                    pair = j, V + (j + t) % L
            if pair is None:
                assert not q[:, st, lane].any()
                continue
            assert frozenset(pair) not in seen
            seen.add(frozenset(pair))
            got[:, pair[0], pair[1]] = q[:, st, lane]
            got[:, pair[1], pair[0]] = -q[:, st, lane]
    most = np.abs(want).max(axis=(1, 2), keepdims=True)
    assert np.all(np.abs(got - want) <= 1e-13 * most)
    # the pairs without an entry in the schedule: none but the diagonal and face by face
    missing = {(a, b) for a in range(V) for b in range(a + 1, V + F)} - {tuple(sorted(p)) for p in seen}
    assert not missing


@pytest.mark.parametrize("kw", [dict(N=5, rule=esdg.ESDG_RULE_COLLAPSED), dict(N=4, precision=esdg.ESDG_FP32),
                                dict(N=5, method=esdg.ESDG_METHOD_SBP)])
def test_configurations_without_it_say_so(kw):
    lib, h = _lib(), ctypes.c_void_p()
    assert lib.esdg_build_operators(ctypes.byref(_cfg(**kw)), ctypes.byref(h)) == 0
    steps = ctypes.c_int()
    assert lib.esdg_pair_operator(h, ctypes.byref(steps), None) == esdg.ESDG_EINVAL
    lib.esdg_destroy(h)
