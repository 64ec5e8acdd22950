"""Points a rounding error below a period of a periodic axis.  p + n rounds to n
there, which is node 0 and not the last node: an identity map with such points
leaves the fields as they were, in the oracle and in the library (bars: the
weights' and the recomposition's rounding, 1e-13 in FP64, 1e-6 in FP32)."""
import numpy as np
import pytest

import oracle
from paper_1803_07822_gb300 import inputs as I

N3 = (32, 6, 5)


def points(eps, periods):
    """The identity map with the points at 0 of axes 0 and 1 moved by eps and
    every point by whole periods; eps survives next to 0 only."""
    psi = np.stack(I.grid(N3)).astype(np.float64)
    for a in (0, 1):
        psi[a] = np.where(psi[a] == 0.0, eps, psi[a] + periods * N3[a])
    return psi


def state():
    rng = np.random.default_rng(3)
    N = int(np.prod(N3))
    flat = I.Chart(N3, np.repeat(np.eye(3).reshape(9, 1), N, axis=1), np.zeros((27, N)))
    return flat, 1.0 + 0.01 * rng.standard_normal(N), 0.02 * rng.standard_normal((3, N))


CASES = [(-1e-16, 0), (-1e-16, 1), (-1e-16, -2), (-3e-18, 0), (-5e-324, 0), (0.0, 0)]


@pytest.mark.parametrize("eps,periods", CASES)
def test_oracle(eps, periods):
    flat, rho, u = state()
    lo = (oracle.PERIODIC,) * 3
    o = oracle.Lattice(N3, lo, lo, tau=0.8)
    o.set_metric(flat.g6, flat.dg18)
    o.init(rho, u)
    r0, v0 = o.moments(flat.J9)
    o.transform_interp(flat.g6, flat.dg18, flat.J9, flat.J9, points(eps, periods))
    r1, v1 = o.moments(flat.J9)
    assert np.abs(r1 - r0).max() < 1e-13 and np.abs(v1 - v0).max() < 1e-13


@pytest.mark.gpu
@pytest.mark.parametrize("storage,bar", [("fp64", 1e-13), ("fp32", 1e-6)])
@pytest.mark.parametrize("eps,periods", CASES)
def test_library(eps, periods, storage, bar):
    from paper_1803_07822_gb300.lattice import CurvedLattice
    flat, rho, u = state()
    lat = CurvedLattice(N3, (0, 0, 0), tau=0.8, storage=storage)
    lat.set_chart(flat)
    lat.init_equilibrium(rho, u)
    r0, v0 = lat.moments(cartesian=True)
    lat.update_metric_interp(flat.g6, flat.dg18, flat.J9, points(eps, periods))
    r1, v1 = lat.moments(cartesian=True)
    assert np.abs(r1 - r0).max() < bar and np.abs(v1 - v0).max() < bar
