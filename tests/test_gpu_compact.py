"""The compact form of the FP64 25-point rules (no operators stored per element):
right-hand sides, steps and diagnostics against the FP64 oracle with the tolerances of
the parity tests, and the ways a problem comes to it.
"""

import ctypes

import numpy as np
import pytest

from oracle import Oracle
from paper_2005_02516_gb300 import workloads as W
from _bounds import check_state

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FORMS = [(5, "symmetric", "exact"), (5, "symmetric", "weight_adjusted"), (4, "collapsed", "exact"),
         (4, "collapsed", "weight_adjusted")]


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("N,rule,mass", FORMS)
def test_compact_form_matches_the_oracle(N, rule, mass, walls):
    from paper_2005_02516_gb300 import esdg
    args = dict(warp=0.05, rule=rule, mass=mass, walls=walls)
    s = esdg.Solver(N, 5, 4, precision="fp64", compact=True, **args)
    full = esdg.Solver(N, 5, 4, precision="fp64", **args)
    assert s.device_bytes < full.device_bytes
    o = Oracle(N, 5, 4, ax=0.05, ay=0.05, rule=rule, mass=mass, walls=walls)
    b = W.LAKE_BUMP.bathymetry(*o.points("nodal"))
    u = W.random_modal_state(o.K, o.Np, seed=W.BASE_SEED + N)
    o.set_bathymetry(b)
    for x in (s, full):
        x.set_bathymetry(b)
        x.set_state(u)
    got, want = s.rhs(0.0).cpu().numpy(), o.rhs(u, 0.0)
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    assert np.allclose(s.entropy(0.0)[:2], full.entropy(0.0)[:2], rtol=1e-13, atol=0)
    s.step(2, o.dt(), 0.0)
    res, t = np.zeros_like(u), 0.0
    for _ in range(2):
        u, res, t = o.step(u, res, t, o.dt())
    check_state(s.get_state(), u, 2e-12)


@pytest.mark.parametrize("N,rule,mass", FORMS)
def test_compact_form_with_forcing_matches_the_stored_form(N, rule, mass):
    from paper_2005_02516_gb300 import esdg
    out = []
    for compact in (False, True):
        s = esdg.Solver(N, 5, 4, precision="fp64", warp=0.05, rule=rule, mass=mass, forcing="mms_sine", compact=compact)
        s.set_state(W.random_modal_state(s.K, s.Np, seed=W.BASE_SEED + N))
        out.append(s.rhs(0.7).cpu().numpy())
    assert np.abs(out[1] - out[0]).max() <= 1e-12 * np.abs(out[0]).max()


def test_a_prepared_context_keeps_its_state():
    from paper_2005_02516_gb300 import esdg
    states = []
    for compact in (False, True):
        p = esdg.Problem(5, 5, 4, precision="fp64", warp=0.05, rule="symmetric")
        xq, yq = p.points(esdg.ESDG_POINTS_VOLQ)
        xb, yb = p.points(esdg.ESDG_POINTS_NODAL)
        q = np.ascontiguousarray(np.stack([2 + 0.1 * np.sin(xq), 0.1 * xq, 0.1 * yq]))
        b = np.ascontiguousarray(0.1 * np.cos(xb) * np.cos(yb))
        assert p.lib.esdg_prepare(p.h, b.ctypes.data, q.ctypes.data, esdg.ESDG_INIT_SURFACE) == 0
        if compact:
            assert p.lib.esdg_prefer_compact(p.h) == 0
        assert p.lib.esdg_attach_device(p.h, None, 0, None) == 0
        assert p.lib.esdg_prefer_compact(p.h) == esdg.ESDG_ESTATE
        assert p.lib.esdg_step(p.h, 1, 0.001, None) == 0
        u = np.zeros((3, p.K, p.Np))
        assert p.lib.esdg_copy_state(p.h, u.ctypes.data, 0) == 0
        states.append(u)
    check_state(states[1], states[0], 2e-12)


def test_a_server_runs_the_form_that_fits_its_budget():
    from paper_2005_02516_gb300 import esdg
    p = esdg.Problem(5, 12, 12, precision="fp64", warp=0.05, rule="symmetric")
    xq, yq = p.points(esdg.ESDG_POINTS_VOLQ)
    q = np.stack([2 + 0.1 * np.sin(xq), 0 * xq, 0 * xq])
    b = np.zeros((p.K, p.Np))
    srv = esdg.Server(p.device_bytes // 3, 4)
    ticket = srv.submit(p, b, q, 3)
    srv.drain(60.0)
    assert srv.query(ticket)[0] == 2 and srv.stats()[3] == 1
    u = srv.result(ticket)
    assert np.all(np.isfinite(u)) and u[0].max() > 1.0
    srv.close()
