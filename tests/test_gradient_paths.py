"""The lattice gradient's marching and per-site kernels: ragged tiles and chunks
of the marches (which small lattices do not take: many fields make their
blocks), continued values beyond the faces of every axis, and constant fields,
whose gradient is exactly zero where the continuation's integer weights leave
them exact.  Bar against the oracle: 1e-12 of the largest entry, as in the
lattice-derivative tests."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
P, W = oracle.PERIODIC, oracle.WALL


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("bc", [(P, P, P), (P, P, W), (P, W, W), (W, P, P), (W, W, W)])
@pytest.mark.parametrize("n,fields", [((95, 31, 70), 104), ((64, 16, 33), 160), ((127, 40, 37), 31),  # marches
                                      ((33, 17, 20), 3), ((9, 5, 40), 2)])                             # per site
def test_against_the_oracle(n, fields, bc, order):
    import torch
    from paper_1803_07822_gb300.lattice import CurvedLattice
    base = np.random.default_rng(5).standard_normal((2, int(np.prod(n))))
    pick = torch.arange(fields, device="cuda") % 2
    got = CurvedLattice(n, bc).lattice_gradient(torch.as_tensor(base, device="cuda")[pick], order)
    ref = oracle.lattice_gradient(n, base, order, bc)
    assert np.abs(got[:, :2].cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
    for c in range(2, fields):
        assert torch.equal(got[:, c], got[:, c % 2])


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("bc", [(P, P, P), (P, W, W), (W, P, P), (W, W, W)])
@pytest.mark.parametrize("n,fields", [((95, 31, 70), 104), ((33, 17, 20), 3)])
def test_constant_fields(n, fields, bc, order):
    import torch
    from paper_1803_07822_gb300.lattice import CurvedLattice
    lat = CurvedLattice(n, bc)
    for c in (1.0, -7.3e5, 0.375):
        f = torch.full((fields, int(np.prod(n))), c, dtype=torch.float64, device="cuda")
        assert not torch.count_nonzero(lat.lattice_gradient(f, order))
