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


def test_second_order_keeps_the_fields_bits():
    """A field that varies by 1e-3 around one: its differences are exact, so
    the second-order gradient is off by the roundings of its own sums only,
    at most eight of 2^-53 of the largest entry and the factor's one (bar
    2e-15); a field scaled before the differences would be off by 4e-14."""
    from paper_1803_07822_gb300.lattice import CurvedLattice
    n = (33, 9, 37)
    z, y, x = np.meshgrid(*[2 * np.pi * np.arange(k) / k for k in n[::-1]], indexing="ij")
    f = 1 + 1e-3 * (np.sin(x) * np.cos(y) + np.cos(z + x) + np.sin(y - z))
    got = CurvedLattice(n, (P, P, P)).lattice_gradient(f.reshape(1, -1), 2).cpu().numpy().reshape(3, *f.shape)
    fl = f.astype(np.longdouble)
    ref = [0, 0, 0]
    for c in np.ndindex(3, 3, 3):
        c = np.array(c) - 1
        if np.abs(c).sum() not in (1, 2):
            continue
        s = np.roll(fl, tuple(-c[::-1]), (0, 1, 2)) / (6 if np.abs(c).sum() == 1 else 12)
        for i in range(3):
            ref[i] = ref[i] + c[i] * s
    ref = np.stack(ref)
    assert np.abs(got - ref).max() <= 2e-15 * np.abs(ref).max()
