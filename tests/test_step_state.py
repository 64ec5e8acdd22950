"""A step between saved states: the same state as save, step, save with the
gather pass, the lattice's own state untouched; the backward step from a saved
state the same as after loading it; refused buffers."""
import ctypes

import numpy as np
import pytest

from paper_1803_07822_gb300 import _abi
from paper_1803_07822_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def lattice(n, storage):
    from paper_1803_07822_gb300.lattice import CurvedLattice
    w = I.periodic_channel(n, 0.7, 0.05, 2, 0.05, 51, kmax=1, lmax=1)
    lat = CurvedLattice(w["n"], w["bc_lo"], w["bc_hi"], tau=w["tau"], fext=w["fext"], storage=storage,
                        step_kernel="flat")
    lat.set_chart(w["chart"])
    lat.init_equilibrium()
    lat.step(3)
    return lat, w


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [(16, 12, 9), (13, 7, 5)])
def test_step_between_saved_states(n, storage):
    import torch
    lat, _ = lattice(n, storage)
    a = lat.save_state()
    b = lat.step_state(a)
    assert torch.equal(lat.save_state(), a)
    lat.step(1)
    # (slots that no node pulls, past a wall, keep what the buffer held: compare what is read)
    want = lat.moments()
    lat.load_state(b)
    got = lat.moments()
    assert all(np.array_equal(u, v) for u, v in zip(want, got))


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
def test_backward_from_a_saved_state(storage):
    import torch
    from paper_1803_07822_gb300.adjoint import Adjoint
    lat, w = lattice((12, 16, 8), storage)
    st = lat.save_state()
    lat.step(1)
    g6 = torch.as_tensor(w["chart"].g6, device="cuda")
    dg18 = torch.as_tensor(w["chart"].dg18, device="cuda")
    final = lat.save_state()
    out = []
    for direct in (True, False):
        lat.load_state(final)
        adj = Adjoint(lat)
        adj.seed_wall_force(2, 1, (0.0, 1.0, 0.0))
        if direct:
            adj.step_backward(st)
        else:
            lat.load_state(st)
            adj.step_backward()
        adj.init_backward()
        out.append([t.clone() for t in adj.metric_grad(g6, dg18)])
    tol = {"fp32": 1e-6, "fp64": 1e-14}[storage]  # the face nodes' atomics add in any order
    for u, v in zip(*out):
        assert float((u - v).norm()) <= tol * float(v.norm())


def test_refused_buffers():
    lib = _abi.load()
    lat, _ = lattice((12, 8, 6), "fp32")
    a = lat.save_state()
    n = a.numel()
    host = np.zeros(n, dtype=np.uint8)
    f = lib.cslbm_step_state
    assert f(lat.ctx, a.data_ptr(), a.data_ptr(), n) == _abi.EINVAL      # in place
    assert f(lat.ctx, a.data_ptr(), None, n) == _abi.EINVAL
    assert f(lat.ctx, a.data_ptr(), host.ctypes.data, n) == _abi.EINVAL
    assert f(lat.ctx, a.data_ptr(), lat.save_state().data_ptr(), n - 4) == _abi.EINVAL
    from paper_1803_07822_gb300.lattice import CurvedLattice
    half = CurvedLattice((12, 8, 6), (0, 0, 1), storage="fp16")
    half.init_equilibrium()
    s, t = half.save_state(), half.save_state()
    assert f(half.ctx, s.data_ptr(), t.data_ptr(), s.numel()) == _abi.EINVAL
    assert ctypes.c_int(f(None, None, None, 0)).value == _abi.EINVAL
