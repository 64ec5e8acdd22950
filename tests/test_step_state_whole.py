"""A step between saved states writes the whole state that cslbm_step writes:
all 19 populations and all ten history values of every node, on lattices the
row passes do not take, faces across one, two and three axes."""
import numpy as np
import pytest

from paper_1803_07822_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
@pytest.mark.parametrize("lo,hi", [((0, 0, 0),) * 2, ((0, 0, 1),) * 2, ((0, 2, 1), (0, 3, 1)), ((1, 1, 1),) * 2])
@pytest.mark.parametrize("n", [(13, 7, 5), (21, 33, 17)])
def test_whole_state(n, lo, hi, storage):
    import torch
    from paper_1803_07822_gb300.lattice import CurvedLattice
    lat = CurvedLattice(n, lo, hi, tau=0.7, fext=(0.0, 1e-4, 0.0), storage=storage)
    lat.set_chart(I.channel_chart(n, I.fourier_deformation(n, 2, 0.04, seed=2, flow_periodic=True, kmax=1, lmax=1)))
    rng = np.random.default_rng(1)
    N = int(np.prod(n))
    lat.init_equilibrium(1 + 0.01 * rng.standard_normal(N), 0.02 * rng.standard_normal((3, N)))
    real = torch.float32 if storage == "fp32" else torch.float64
    a = lat.save_state()
    for _ in range(4):
        b = lat.step_state(a)
        assert torch.equal(lat.save_state(), a)
        lat.step(1)
        a = lat.save_state()
        assert torch.equal(a.view(real), b.view(real))
