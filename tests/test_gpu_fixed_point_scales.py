"""The FP64 path's block fixed-point sums where the components of a field or of
an operator differ by orders of magnitude: each keeps the bits it has in FP64.

Tolerance: an entry of du/dt against the oracle within 2 c u of the largest sum
of absolute terms of its element and field, u = 2^-53 and c the first-order bound
of tests/_bounds.py for the chain of sums, once for the kernel and once for the
oracle, which evaluates the same sums in FP64.  (The DG-SBP scheme has no entropy
projection, whose H = v_1 / g + (u^2 + v^2) / (2 g) loses bits of the depth to a
fast flow in any arithmetic: the modal scheme is checked at speeds of about 10 with
g = 1, where the two squares are 100 times the depth, which the bound is scaled
with.)
"""

import numpy as np
import pytest

from oracle import Oracle
from oracle.sbp import SBPOracle
from paper_2005_02516_gb300 import workloads as W
from _bounds import c_modal, c_sbp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _check(got, want, mag, c):
    mag = mag.max(axis=2, keepdims=True)
    assert np.all(np.abs(got - want) <= 2 * c * 2.0 ** -53 * mag)


def _sbp_case(N, speeds, **dom):
    from paper_2005_02516_gb300 import esdg
    s = esdg.Solver(N, 5, 4, precision="fp64", method="sbp", rule="symmetric", **dom)
    o = SBPOracle(N, 5, 4, ax=dom["warp"], ay=dom["warp"], **{k: v for k, v in dom.items() if k != "warp"})
    xb, yb = o.points("nodal")
    b = 0.3 + 0.1 * np.cos(xb) * np.cos(yb)
    s.set_bathymetry(b)
    o.set_bathymetry(b)
    rng = np.random.default_rng(W.BASE_SEED + N)
    u = 1.0 + 0.1 * rng.standard_normal((3, o.K, o.Nq))
    u[0] = 2.0 + 0.05 * rng.standard_normal((o.K, o.Nq))
    u[1] *= 2.0 * speeds[0]
    u[2] *= 2.0 * speeds[1]
    return s, o, u


# velocities of a thin fast film (Froude numbers up to 700) along x or y
SPEEDS = [(20.0, 1e-3), (1e-3, 20.0), (1e3, 1e-3), (1e-3, 1e3)]


@pytest.mark.parametrize("speeds", SPEEDS)
@pytest.mark.parametrize("N", [1, 2, 3, 4])
def test_sbp_rhs_with_one_fast_component(N, speeds):
    s, o, u = _sbp_case(N, speeds, warp=0.05)
    s.set_state(u)
    _check(s.rhs(0.0).cpu().numpy(), o.rhs(u, 0.0), o.rhs_term_magnitude(u, 0.0), c_sbp(o.Nq))


@pytest.mark.parametrize("speeds", [(10.0, 1e-3), (1e-3, 10.0)])
@pytest.mark.parametrize("N,rule", [(N, rule) for N in range(1, 6) for rule in ("symmetric", "collapsed")])
def test_modal_rhs_with_one_fast_component(N, rule, speeds):
    from paper_2005_02516_gb300 import esdg
    s = esdg.Solver(N, 5, 4, precision="fp64", warp=0.05, rule=rule)
    o = Oracle(N, 5, 4, ax=0.05, ay=0.05, rule=rule)
    b = W.LAKE_BUMP.bathymetry(*o.points("nodal"))
    s.set_bathymetry(b)
    o.set_bathymetry(b)
    u = W.random_modal_state(o.K, o.Np, seed=W.BASE_SEED + N)
    u[1:, :, 0] += u[0, :, 0]
    u[1] *= speeds[0]
    u[2] *= speeds[1]
    s.set_state(u)
    _check(s.rhs(0.0).cpu().numpy(), o.rhs(u, 0.0), o.rhs_term_magnitude(u, 0.0),
           c_modal(o.Np, o.Nq, o.Nfq) * (1 + 100.0))


# domains stretched along x or y: one of Qx and Qy is the aspect ratio below the
# other.  Fluid at rest, and flow along the long side, for which both products
# of T = Qx HU + Qy HV are of one size
STRETCHED = [(ax, ay, flow) for ax, ay in [(100.0, 1.0), (1e4, 1.0), (1.0, 1e4)] for flow in (0.0, 0.1)]


@pytest.mark.parametrize("ax,ay,flow", STRETCHED)
@pytest.mark.parametrize("N", [1, 2, 3, 4])
def test_sbp_rhs_on_stretched_elements(N, ax, ay, flow):
    m = max(ax, ay)
    s, o, u = _sbp_case(N, (flow * ax / m, flow * ay / m), warp=0.05, x0=-ax, x1=ax, y0=-ay, y1=ay)
    s.set_state(u)
    _check(s.rhs(0.0).cpu().numpy(), o.rhs(u, 0.0), o.rhs_term_magnitude(u, 0.0), c_sbp(o.Nq))


@pytest.mark.parametrize("ax,ay,flow", STRETCHED)
@pytest.mark.parametrize("N,rule", [(N, rule) for N in range(1, 6) for rule in ("symmetric", "collapsed")])
def test_modal_rhs_on_stretched_elements(N, rule, ax, ay, flow):
    from paper_2005_02516_gb300 import esdg
    dom = dict(x0=-ax, x1=ax, y0=-ay, y1=ay)
    s = esdg.Solver(N, 5, 4, precision="fp64", warp=0.05, rule=rule, **dom)
    o = Oracle(N, 5, 4, ax=0.05, ay=0.05, rule=rule, **dom)
    b = 0.3 + 0.1 * np.cos(o.points("nodal")[0] / ax) * np.cos(o.points("nodal")[1] / ay)
    s.set_bathymetry(b)
    o.set_bathymetry(b)
    u = W.random_modal_state(o.K, o.Np, seed=W.BASE_SEED + N)
    u[1:, :, 0] += u[0, :, 0]
    u[1] *= flow * ax / max(ax, ay)
    u[2] *= flow * ay / max(ax, ay)
    s.set_state(u)
    _check(s.rhs(0.0).cpu().numpy(), o.rhs(u, 0.0), o.rhs_term_magnitude(u, 0.0), c_modal(o.Np, o.Nq, o.Nfq))


# With g = 1 and a = 4^k, h -> a h, b -> a b, (u, v) -> sqrt(a) (u, v) maps the
# equations into themselves and scales du/dt of the momenta by a^2: at k = -260 these
# are subnormal (multiples of 2^-1074).  A row of fluxes is off by at most 64
# roundings to such a multiple, the lift and the inverse mass sum rows of absolute
# values below 2^16 on this mesh.
SUBNORMAL = [(N, rule, mass, "modal") for N in range(1, 6) for rule in ("symmetric", "collapsed")
             for mass in ("exact", "weight_adjusted")] + [(N, "symmetric", "exact", "sbp") for N in range(1, 6)]


@pytest.mark.parametrize("N,rule,mass,method", SUBNORMAL)
def test_subnormal_values_keep_their_bits(N, rule, mass, method):
    from paper_2005_02516_gb300 import esdg
    got = []
    for k in (0, -260):
        a = 4.0 ** k
        s = esdg.Solver(N, 5, 4, precision="fp64", warp=0.05, rule=rule, mass=mass, method=method)
        s.set_bathymetry(a * W.LAKE_BUMP.bathymetry(*s.points(esdg.ESDG_POINTS_NODAL)))
        if method == "sbp":
            u = 0.05 * np.random.default_rng(W.BASE_SEED + N).standard_normal((3, s.K, s.ndof))
            u[0] += 2.0
        else:
            u = W.random_modal_state(s.K, s.Np, seed=W.BASE_SEED + N)
        s.set_state(u * np.array([a, a * 2.0 ** k, a * 2.0 ** k])[:, None, None])
        got.append(s.rhs(0.0).cpu().numpy())
    want, small = got[0][1:], got[1][1:]
    assert np.abs(want).max() > 0.01  # 2^-1047: far above the tolerance
    # (compared as integers in units of 2^-1074: factors of 2^537 twice, exact)
    units = small * 2.0 ** 537 * 2.0 ** 537
    assert np.all(np.abs(units - want * 2.0 ** (1074 - 1040)) <= 2.0 ** 22)
