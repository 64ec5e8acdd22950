"""The readout's division-free velocity against FP64 division of the same FP32
(FP64) density and momentum, over values at the ends of their ranges: zeros,
subnormals, huge values, infinities and NaN take the division itself."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (rest population s_0, population s_+x) of a flat lattice at rest otherwise:
# rho = 1 + s_0 + s_+x, rho u_x = s_+x
ROWS = [(0.0, 0.0), (0.0, 0.01), (1e-3, -0.02), (-1.0, 0.0), (-1.0, 1e-3), (-2.0, 0.25), (1e30, 1.0), (3e38, 3e38),
        (0.0, 1e-40), (0.0, -1e-42), (1e-30, 1.2e-38), (np.inf, 0.5), (0.0, np.inf), (np.nan, 0.1), (0.0, -np.nan),
        (-0.999999, 1e-7)]


@pytest.mark.parametrize("cartesian", [False, True])
@pytest.mark.parametrize("storage", ["fp32", "fp64"])
def test_velocity_of_unusual_states(storage, cartesian):
    import torch
    from paper_1803_07822_gb300.lattice import CurvedLattice
    n = (5, 4, 4)
    N = 80
    dt = np.float32 if storage == "fp32" else np.float64
    lat = CurvedLattice(n, storage=storage)
    lat.init_equilibrium()
    s = np.zeros((29, N), dtype=dt)  # 19 populations, 10 history coefficients; planes 0, 1: rest, +x
    s0, s1 = (np.repeat(np.array([r[k] for r in ROWS], dtype=dt), n[0]) for k in (0, 1))
    s[0], s[1] = s0, s1
    lat.load_state(torch.from_numpy(s.view(np.uint8).reshape(-1)).cuda())
    with np.errstate(all="ignore"):
        rho = (dt(1) + (s0 + s1)).astype(np.float64)
        u = s1.astype(np.float64) / rho
    r, v = lat.moments(cartesian=cartesian)
    np.testing.assert_array_equal(r, rho)
    if cartesian:  # J = I: the off-diagonal zeros meet the other components (0 x inf = NaN)
        with np.errstate(all="ignore"):
            u = u + 0.0 * (0.0 / rho) + 0.0 * (0.0 / rho)
    # half an ulp of the division plus an ulp of the reciprocal and the product
    fine = np.isfinite(u)
    np.testing.assert_allclose(v[0][fine], u[fine], rtol=4e-16, atol=0.0)
    np.testing.assert_array_equal(v[0][~fine], u[~fine])
