"""FP64 readouts with face nodes (the boundary rule) against the oracle: every
axis with faces, edges and corners, contravariant and Cartesian, at the bar of
the FP64 parity tests (1e-11)."""
import numpy as np
import pytest

import oracle
from paper_1803_07822_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P, W, IN, OUT = oracle.PERIODIC, oracle.WALL, oracle.INFLOW, oracle.OUTFLOW


@pytest.mark.parametrize("lo,hi", [((P, P, P), (P, P, P)), ((W, W, W), (W, W, W)), ((P, IN, W), (P, OUT, W)), ((OUT, P, P), (IN, P, P))])
@pytest.mark.parametrize("n", [(5, 4, 3), (19, 13, 11)])
def test_against_the_oracle(n, lo, hi):
    from paper_1803_07822_gb300.lattice import CurvedLattice
    ch = I.channel_chart(n, I.fourier_deformation(n, 2, 0.04, seed=4, flow_periodic=True, kmax=1, lmax=1))
    rng = np.random.default_rng(8)
    N = int(np.prod(n))
    rho, u = 1.0 + 0.01 * rng.standard_normal(N), 0.02 * rng.standard_normal((3, N))
    g = CurvedLattice(n, lo, hi, tau=0.8, storage="fp64")
    o = oracle.Lattice(n, lo, hi, tau=0.8)
    g.set_chart(ch)
    o.set_metric(ch.g6, ch.dg18)
    g.init_equilibrium(rho, u)
    o.init(rho, u)
    g.step(3)
    o.step(3)
    for J in (None, ch.J9):
        (rg, vg), (ro, vo) = g.moments(cartesian=J is not None), o.moments(J)
        assert np.linalg.norm(rg - ro) <= 1e-11 * np.linalg.norm(ro)
        assert np.linalg.norm(vg - vo) <= 1e-11 * np.linalg.norm(vo)
