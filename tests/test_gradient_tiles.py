"""The marching gradient kernels at the edges of their tiles (32 x 8 columns,
chunks of planes) and at the smallest extents, against the oracle at the bar
of the lattice-derivative tests (1e-12 of the largest entry)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
P, W = oracle.PERIODIC, oracle.WALL


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n,bc", [((2, 2, 2), (P, P, P)), ((5, 5, 5), (W, W, W)), ((32, 8, 32), (P, P, P)),
                                  ((33, 9, 37), (P, W, P)), ((31, 7, 70), (W, P, W)), ((30, 6, 5), (W, W, W)),
                                  ((65, 17, 6), (P, P, W))])
def test_against_the_oracle(n, bc, order):
    from paper_1803_07822_gb300.lattice import CurvedLattice
    f = np.random.default_rng(11).standard_normal((3, int(np.prod(n))))
    lat = CurvedLattice(n, bc)
    got = lat.lattice_gradient(f, order).cpu().numpy()
    ref = oracle.lattice_gradient(n, f, order, bc)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
