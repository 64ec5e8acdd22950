"""The interpolating chart change where its point wrapping and its FP32 corner
sums can go wrong: points whole periods away (near and far wraps), on and next
to the ends of an axis, outside a wall, and an old Jacobian that varies
strongly from node to node, against the oracle at the bars of the chart-change
tests."""
import numpy as np
import pytest

import oracle
from paper_1803_07822_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-11, "fp32": 1e-5}


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("periods", [0, 1, -1, -2, 3])
@pytest.mark.parametrize("storage", ["fp64", "fp32"])
def test_points(storage, periods):
    from paper_1803_07822_gb300.lattice import CurvedLattice
    n = (13, 11, 7)
    N = int(np.prod(n))
    rng = np.random.default_rng(7)
    lo = (oracle.PERIODIC, oracle.PERIODIC, oracle.WALL)
    J0 = (np.eye(3).reshape(9, 1) + 0.2 * rng.uniform(-1, 1, (9, N)))  # rough: 20 % from node to node
    old = I.Chart(n, J0, np.zeros((27, N)))
    new = I.Chart(n, np.repeat((np.eye(3) + 0.05 * rng.standard_normal((3, 3))).reshape(9, 1), N, axis=1),
                  np.zeros((27, N)))
    psi = np.stack(I.grid(n)) + rng.uniform(-1, 1, (3, N))
    psi[:, :40] = np.round(psi[:, :40])          # on nodes
    psi[0, 40:44] = [0.0, n[0] - 1e-9, n[0], -1e-9]
    psi[2, 44:46] = [-3.0, n[2] + 5.0]           # outside the walls
    psi[:2] += periods * np.array([[n[0]], [n[1]]])
    rho, u = 1.0 + 0.01 * rng.standard_normal(N), 0.02 * rng.standard_normal((3, N))
    g = CurvedLattice(n, lo, lo, tau=0.8, storage=storage)
    o = oracle.Lattice(n, lo, lo, tau=0.8)
    g.set_chart(old)
    o.set_metric(old.g6, old.dg18)
    g.init_equilibrium(rho, u)
    o.init(rho, u)
    g.update_metric_interp(new.g6, new.dg18, new.J9, psi)
    o.transform_interp(new.g6, new.dg18, old.J9, new.J9, psi)
    (rg, vg), (ro, vo) = g.moments(cartesian=True), o.moments(new.J9)
    assert rel(rg, ro) < TOL[storage] and rel(vg, vo) < TOL[storage]
    assert g.check() in (True, False)  # the pending metric flag is clear
