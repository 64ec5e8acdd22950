"""The value of a wall-force objective keeps the rounding of its FP32 states.

The streamwise force on a deformed wall is a sum of pressure terms hundreds of
times larger than itself, so that another rounding of the states moves it by
several times its own error (the closed form of a face node's rho u in place of
the boundary rule's first moment: 22 x 101 x 29, 1.7e-7 of the value off FP64
became 5.5e-7).  VALUES are the library's before its passes staged their inputs
(nvcc 13.0).  Inputs are dyadic fractions, the same bits on any machine; the
force is summed in FP64 in any order, so equal states give the value to 1e-9."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (extents, steps): value.  Extents along axis 0 that the row passes do not take
# (odd, even but no multiple of 4, longer than a tile) and that they take.
VALUES = {
    ((21, 33, 17), 30): 0.16929141560097705,
    ((22, 101, 29), 30): 0.5655914998686455,
    ((37, 40, 19), 12): 0.17005036675505902,
    ((260, 16, 12), 12): 0.461287018299803,
    ((32, 48, 20), 30): 0.37994534031555816,
    ((64, 32, 24), 12): 0.23073459393204132,
}


def tri(k, n):
    """A triangle wave of period n in 0..1 at the integers k, in steps of 1/256."""
    t = np.minimum(k % n, (n - k) % n)
    return np.floor(512.0 * t / n) / 256.0


def fields(n):
    """Some smooth metric (g6, dg18) and Jacobian J9 close to that of a channel
    with a wall of slope 1/8 (derivatives by differences, all dyadic)."""
    z, y, x = np.meshgrid(*(np.arange(m) for m in n[::-1]), indexing="ij")
    d = (tri(x + 3, n[0]) * 0.25 + tri(y, n[1]) * 0.5 - 0.375) * 0.125
    dx = np.floor((np.roll(d, -1, 2) - np.roll(d, 1, 2)) * 2.0 ** 19) / 2.0 ** 20
    dy = np.floor((np.roll(d, -1, 1) - np.roll(d, 1, 1)) * 2.0 ** 19) / 2.0 ** 20
    J = np.zeros((9, *d.shape))
    J[0] = J[4] = 1.0
    J[6], J[7], J[8] = z * dx, z * dy, 1.0 + d
    g = np.stack([1.0 + J[6] * J[6], J[6] * J[7], J[6] * J[8], 1.0 + J[7] * J[7], J[7] * J[8], J[8] * J[8]])
    dg = np.zeros((18, *d.shape))
    for k, h in enumerate((dx, dy)):  # d_k J^2_2 = d_k d, d_2 J^2_k = d_k d
        dg[6 * k + 5] = 2.0 * h * J[8]
        dg[6 * k + 2] = h * J[6]
        dg[6 * k + 4] = h * J[7]
        dg[12 + (2 if k == 0 else 4)] = h * J[8]
        dg[12 + (0 if k == 0 else 3)] = 2.0 * h * J[6 + k]
    return g.reshape(6, -1), dg.reshape(18, -1), J.reshape(9, -1)


def objective(n, steps):
    import torch
    from paper_1803_07822_gb300.adjoint import wall_force_objective
    from paper_1803_07822_gb300.lattice import CurvedLattice
    lat = CurvedLattice(n, (0, 0, 1), tau=0.75, fext=(0.0, 2.0 ** -12, 0.0), storage="fp32")
    args = [torch.as_tensor(a, device="cuda") for a in fields(n)]
    return float(wall_force_objective(lat, *args, steps, 10, axis=2, side=1, e3=(0.0, 1.0, 0.0)))


@pytest.mark.parametrize("n,steps", list(VALUES))
def test_objective_keeps_its_value(n, steps):
    assert objective(n, steps) == pytest.approx(VALUES[n, steps], rel=1e-9)
