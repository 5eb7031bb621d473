"""Stage launches at the sizes where their shape changes: fewer elements than
SMs, batches that just fill or overflow one warp a SM, the rounds of a full
chip, and last rounds of a few elements.  Two steps (ten dependent launches
and the projection) and one right-hand side against the FP64 oracle, with the
tolerances of the parity tests.
"""

import numpy as np
import pytest

from oracle import Oracle
from oracle.sbp import SBPOracle
from paper_2005_02516_gb300 import workloads as W
from _bounds import c_modal, c_sbp, check_fp32_rhs, check_state

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (N, nx, ny): K = 18, 608 and 612 (152 batches of 4 and one more), 1824 and
# 1850, 3648 and 3660 (the warps of 3 blocks on 152 SMs), 14596 (a second
# round of 24 warps); 2432, 2436 and 3698 (one round of 16 warps, just more, and
# one of 24, for the FP64 rules that take wider blocks above one round)
SHAPES = [(2, 3, 3), (2, 19, 16), (2, 17, 18), (1, 24, 38), (2, 25, 37), (1, 57, 32), (1, 61, 30), (1, 89, 82),
          (2, 32, 38), (2, 29, 42), (3, 29, 42), (2, 43, 43), (5, 29, 42)]


@pytest.mark.parametrize("N,nx,ny", SHAPES)
@pytest.mark.parametrize("method", ["modal", "sbp"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_steps_and_rhs_at_launch_boundaries(precision, method, N, nx, ny):
    from paper_2005_02516_gb300 import esdg
    if N == 5 and (method == "sbp" or precision == "fp32"):
        pytest.skip("N = 5: for the modal FP64 kernel's wider blocks only (the oracle takes minutes)")
    w = W.LAKE_BUMP
    s = esdg.Solver(N, nx, ny, precision=precision, warp=0.03, rule="symmetric", method=method)
    o = (SBPOracle(N, nx, ny, ax=0.03, ay=0.03) if method == "sbp"
         else Oracle(N, nx, ny, ax=0.03, ay=0.03, rule="symmetric"))
    xb, yb = s.points(esdg.ESDG_POINTS_NODAL)
    s.set_bathymetry(w.bathymetry(xb, yb))
    o.set_bathymetry(w.bathymetry(*o.points("nodal")))
    if method == "sbp":
        xq, yq = o.points("volq")
        u = o.init_state(w.initial(xq, yq), surface=True)
        u = u + 0.02 * np.random.default_rng(W.BASE_SEED).standard_normal(u.shape)
    else:
        u = W.random_modal_state(o.K, o.Np, seed=W.BASE_SEED + nx)
    s.set_state(u)
    got, want = s.rhs(0.0).cpu().numpy(), o.rhs(u, 0.0)
    if precision == "fp64":
        assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
        assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    else:
        mag = o.rhs_term_magnitude(u, 0.0)
        check_fp32_rhs(got, want, mag, c_sbp(o.Nq) if method == "sbp" else c_modal(o.Np, o.Nq, o.Nfq))
    s.step(2, o.dt(), 0.0)
    res, t = np.zeros_like(u), 0.0
    for _ in range(2):
        u, res, t = o.step(u, res, t, o.dt())
    check_state(s.get_state(), u, 2e-12 if precision == "fp64" else 1e-5)
