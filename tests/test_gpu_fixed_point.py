"""The FP64 path's block fixed-point sums (esdg_fixed.cuh) where their scales
matter: every rule and inverse mass of the kernel, at rest, with velocities far
below the wave speed and of its order, and over the exponent range.

Scaling: for g = 1 the shallow water equations map h -> a h, b -> a b,
(u, v) -> sqrt(a) (u, v) into themselves, the right-hand side of h by a^(3/2) and
of the momenta by a^2.  With a = 4^k every factor is a power of two, under which
sums, products, quotients and roots of floating-point numbers and fixed-point
sums with run-time scales are unchanged: the right-hand sides must agree bit for
bit.  Accuracy: an entry of du/dt against the oracle within c u of the largest
sum of absolute terms of its element and field, u = 2^-53 and c the first-order
bound of tests/_bounds.py for the chain of sums (the fixed-point operands are
off by less, 2^-57 of the element's largest value).
"""

import numpy as np
import pytest

from oracle import Oracle
from paper_2005_02516_gb300 import workloads as W
from _bounds import c_modal

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

RULES = [(N, rule) for N in range(1, 6) for rule in ("symmetric", "collapsed")]


def _solver(N, rule, mass, b, method="modal"):
    from paper_2005_02516_gb300 import esdg
    s = esdg.Solver(N, 5, 4, precision="fp64", warp=0.05, rule=rule, mass=mass, method=method)
    s.set_bathymetry(b)
    return s


@pytest.mark.parametrize("mass,method", [("exact", "modal"), ("weight_adjusted", "modal"), ("exact", "sbp")])
@pytest.mark.parametrize("N,rule", RULES)
def test_rhs_is_exact_under_powers_of_two(N, rule, mass, method):
    from paper_2005_02516_gb300 import esdg
    if method == "sbp" and rule == "collapsed":
        pytest.skip("DG-SBP has its own rule")
    p = esdg.Problem(N, 5, 4, warp=0.05, rule=rule, method=method)
    xb, yb = p.points(esdg.ESDG_POINTS_NODAL)
    b = W.LAKE_BUMP.bathymetry(xb, yb)
    if method == "sbp":
        u = 0.05 * np.random.default_rng(W.BASE_SEED + N).standard_normal((3, p.K, p.Nq))
        u[0] += 2.0
    else:
        u = W.random_modal_state(p.K, p.Np, seed=W.BASE_SEED + N)
    want = _solver(N, rule, mass, b, method)
    want.set_state(u)
    want = want.rhs(0.0).cpu().numpy()
    for k in (-60, 1, 60):
        a, ra = 4.0 ** k, 2.0 ** k
        s = _solver(N, rule, mass, a * b, method)
        s.set_state(u * np.array([a, a * ra, a * ra])[:, None, None])
        got = s.rhs(0.0).cpu().numpy()
        assert np.array_equal(got, want * np.array([a * ra, a * a, a * a])[:, None, None])


@pytest.mark.parametrize("speed", [0.0, 1e-12, 1.0])
@pytest.mark.parametrize("N,rule", RULES)
def test_rhs_accuracy_over_velocity_scales(N, rule, speed):
    o = Oracle(N, 5, 4, ax=0.05, ay=0.05, rule=rule)
    xb, yb = o.points("nodal")
    b = W.LAKE_BUMP.bathymetry(xb, yb)
    o.set_bathymetry(b)
    u = W.random_modal_state(o.K, o.Np, seed=W.BASE_SEED + 7 * N)
    u[1:] *= speed
    s = _solver(N, rule, "exact", b)
    s.set_state(u)
    got, want = s.rhs(0.0).cpu().numpy(), o.rhs(u, 0.0)
    mag = o.rhs_term_magnitude(u, 0.0).max(axis=2, keepdims=True)
    assert np.all(np.abs(got - want) <= 2 * c_modal(o.Np, o.Nq, o.Nfq) * 2.0 ** -53 * mag)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_states_are_reported(bad):
    from paper_2005_02516_gb300 import esdg
    p = esdg.Problem(4, 5, 4, warp=0.05, rule="symmetric")
    u = W.random_modal_state(p.K, p.Np, seed=W.BASE_SEED)
    s = _solver(4, "symmetric", "exact", np.zeros((p.K, p.Np)))
    v = u.copy()
    v[1, 3, 2] = bad
    s.set_state(v)
    with pytest.raises(esdg.EsdgError) as ei:
        s.rhs(0.0)
    assert ei.value.code == esdg.ESDG_ENONFINITE
    s.set_state(u)
    assert np.all(np.isfinite(s.rhs(0.0).cpu().numpy()))
