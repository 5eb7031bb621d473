"""The velocities of the FP64 diagnostics are quotients of one rounding.

With h = hu = hv at every node the velocities are exactly 1, and with a gravity
whose terms lie far below the last bit the entropy 1/2 h (u^2 + v^2) at a node is
exactly h: entropy and mass are then the same sums of the same terms in the same
order, equal bit for bit.  (A product with a rounded 1 / h gives 1 - 2^-53 for
many h.)
"""

import numpy as np
import pytest

from paper_2005_02516_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N,rule,method", [(2, "symmetric", "modal"), (4, "symmetric", "modal"),
                                           (3, "collapsed", "modal"), (4, "symmetric", "sbp")])
def test_entropy_of_unit_velocities_is_the_mass(N, rule, method, precision):
    from paper_2005_02516_gb300 import esdg
    s = esdg.Solver(N, 9, 7, precision=precision, warp=0.05, rule=rule, method=method, g=2.0 ** -1000 if
                    precision == "fp64" else 2.0 ** -100)
    s.set_bathymetry(np.zeros((s.K, s.Np)))
    for depth in 49.0 + 2.0 ** -40 * np.arange(16):  # one depth for all nodes: every term has the same rounding
        h = np.zeros((s.K, s.ndof))
        h[:, :s.ndof if method == "sbp" else 1] = depth
        s.set_state(np.stack([h, h, h]))
        entropy, mass, _ = s.entropy(0.0, rate=False)
        assert mass > 0 and entropy == mass
