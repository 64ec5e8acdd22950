"""The velocity of an FP32 lattice's readout is the FP64 quotient of its FP32
momentum and density, rounded: u rho is the momentum up to an ulp of FP64, so
its FP32 rounding is the momentum itself, whose quotient by rho u must be, bit
for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def lattice(dim):
    from paper_1803_07822_gb300.lattice import CurvedLattice, CurvedLattice2D
    n = (97, 53) if dim == 2 else (23, 17, 19)
    rng = np.random.default_rng(dim)
    N = int(np.prod(n))
    lat = CurvedLattice2D(n, (0, 1), tau=0.8) if dim == 2 else CurvedLattice(n, (0, 0, 1), tau=0.8)
    eye = np.eye(dim)[np.triu_indices(dim)]
    lat.set_metric(np.repeat(eye[:, None], N, axis=1), np.zeros((dim * len(eye), N)))
    lat.init_equilibrium(1.0 + 0.1 * rng.standard_normal(N), 0.03 * rng.standard_normal((dim, N)))
    lat.step(2)
    return lat


@pytest.mark.parametrize("dim", [2, 3])
def test_velocity_is_the_rounded_quotient(dim):
    rho, u = lattice(dim).moments(cartesian=False)
    rho, u = np.asarray(rho).ravel(), np.asarray(u).reshape(dim, -1)
    assert np.array_equal(rho, rho.astype(np.float32))
    j = (u * rho).astype(np.float32).astype(np.float64)
    assert np.array_equal(u, j / rho)
