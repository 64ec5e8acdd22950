"""The fused row pass at sizes where AUTO takes another: the test hook that
withholds a publication makes the next launch a fused one at any size, and with
an iteration that no block reaches it withholds none.  All forms of tiles
(ragged, one row, rows that straddle warps, walls across x, periodic flow) in
FP32, FP16 and BF16: the same bits as the gather pass that AUTO takes there
(one arithmetic per node), also after a launch whose waits ran out."""
import ctypes

import numpy as np
import pytest

from paper_1803_07822_gb300 import _abi
from test_gpu_parity import TILED, compare, make_pair, tiled_case, TOL

pytestmark = pytest.mark.gpu
CASES = [t for t in TILED if t[0] != "periodic everywhere"]  # axis 2 periodic: no fused form
IDS = [t[0] for t in CASES]
WAIT = 500_000_000


def fused(g, steps, iteration=1 << 28, wait=WAIT):
    lib = _abi.load()
    for _ in range(steps):
        assert lib.cslbm_test_withhold_publication(g.ctx, iteration, ctypes.c_longlong(wait)) == _abi.OK
        before = g.profile_read()[2]
        g.step(1)
        assert g.profile_read()[2] - before == 2  # k_step_fused, k_step_faces


def pair(w, storage):
    from paper_1803_07822_gb300.lattice import CurvedLattice
    out = []
    rng = np.random.default_rng(11)
    N = int(np.prod(w["n"]))
    rho, u = 1 + 0.005 * rng.standard_normal(N), 0.01 * rng.standard_normal((3, N))
    for _ in range(2):
        g = CurvedLattice(w["n"], w["bc_lo"], w["bc_hi"], tau=w["tau"], fext=w["fext"], storage=storage)
        g.set_chart(w["chart"])
        for (axis, side), v in w.get("faces", {}).items():
            g.set_boundary_velocity(axis, side, v)
        g.init_equilibrium(rho, u)
        g.profile()
        out.append(g)
    return out


def usable(n, storage):
    return storage == "fp32" or n[0] % 8 == 0


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("name,n,layout,kind", CASES, ids=IDS)
def test_same_bits_as_the_gather_pass(name, n, layout, kind, storage):
    if not usable(n, storage):
        pytest.skip("rows of 16-bit populations are no whole number of 16 bytes")
    g, twin = pair(tiled_case(n, layout, kind), storage)
    fused(g, 30)
    twin.step(30)
    assert g.check() and twin.check()
    # (slots that no node pulls are written by neither: compare what is read, then step on)
    for _ in range(2):
        for a, b in zip(g.moments(), twin.moments()):
            assert np.array_equal(a, b)
        g.step(3)
        fused(twin, 3)


@pytest.mark.parametrize("name,n,layout,kind", CASES, ids=IDS)
def test_against_the_oracle(name, n, layout, kind):
    w = tiled_case(n, layout, kind)
    g, o = make_pair(w, "fp32")
    rng = np.random.default_rng(11)
    N = int(np.prod(n))
    rho, u = 1 + 0.005 * rng.standard_normal(N), 0.01 * rng.standard_normal((3, N))
    g.init_equilibrium(rho, u)
    o.init(rho, u)
    g.profile()
    fused(g, 60)
    o.step(60)
    assert g.check()
    compare(g, o, w["chart"].J9, TOL["fp32"], name)


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_fused_steps_after_a_timeout(storage):
    """The waits of a launch run out, cslbm_check reports it and resets the
    publication counts: the fused steps that follow run clean and match a twin
    that took none."""
    lib = _abi.load()
    g, twin = pair(tiled_case(*CASES[IDS.index("periodic flow")][1:]), storage)
    fused(g, 5)
    twin.step(5)
    snap = g.save_state()
    assert lib.cslbm_test_withhold_publication(g.ctx, 0, ctypes.c_longlong(1_000_000)) == _abi.OK
    g.step(1)
    assert lib.cslbm_check(g.ctx) == _abi.ETIMEOUT
    g.load_state(snap)
    fused(g, 20)
    twin.step(20)
    assert lib.cslbm_check(g.ctx) == _abi.OK
    for a, b in zip(g.moments(), twin.moments()):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("kernel", ["fused", "rows", "flat", "auto"])
@pytest.mark.parametrize("name,n,layout,kind", CASES[:3], ids=IDS[:3])
def test_step_state_follows_every_pass(name, n, layout, kind, kernel):
    """A saved state stepped by cslbm_step_state (always the gather pass) is the
    state that cslbm_step reaches by whatever pass, all populations and all ten
    history values of every node: the adjoint's recomputed states are those of
    the forward run."""
    import torch
    from paper_1803_07822_gb300.lattice import CurvedLattice
    w = tiled_case(n, layout, kind)
    g = CurvedLattice(n, w["bc_lo"], w["bc_hi"], tau=w["tau"], fext=w["fext"], storage="fp32",
                      step_kernel="auto" if kernel == "fused" else kernel)
    g.set_chart(w["chart"])
    for (axis, side), v in w.get("faces", {}).items():
        g.set_boundary_velocity(axis, side, v)
    g.init_equilibrium()
    g.profile()
    a = g.save_state()
    for _ in range(4):
        b = g.step_state(a)
        fused(g, 1) if kernel == "fused" else g.step(1)
        a = g.save_state()
        assert torch.equal(a.view(torch.float32), b.view(torch.float32))
