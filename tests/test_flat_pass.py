"""The gather pass where its blocks, face list and index arithmetic can go
wrong: lattices smaller than a block, ragged last blocks, one- and two-node
periodic axes, walls on every axis, faces that meet at edges and corners.
And, on the CPU, its division by multiplication."""
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1803_07822_gb300 import inputs as I

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
P, W, IN, OUT = oracle.PERIODIC, oracle.WALL, oracle.INFLOW, oracle.OUTFLOW


def test_division_by_multiplication(tmp_path):
    exe = str(tmp_path / "div")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1803_07822_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "fast_div_check.cpp"), "-o", exe])
    divisors = [1, 2, 3, 5, 7, 13, 91, 127, 128, 129, 256, 1000, 4095, 4096, 65521, 65536, 65537, 7007, (1 << 27) - 1,
                1 << 27, (1 << 27) + 1, 171798691]
    subprocess.check_call([exe, *map(str, divisors)])


CASES = [((3, 3, 3), (W, W, W), (W, W, W)), ((1, 5, 4), (P, P, W), (P, P, W)), ((2, 2, 7), (P, P, P), (P, P, P)),
         ((130, 3, 5), (W, P, OUT), (W, P, IN)), ((33, 17, 3), (P, IN, W), (P, OUT, W)), ((5, 4, 33), (IN, W, P), (OUT, W, P)),
         ((43, 1, 3), (P, P, W), (P, P, W))]


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["fp32", "fp64"])
@pytest.mark.parametrize("n,lo,hi", CASES)
def test_against_the_oracle(n, lo, hi, storage):
    from paper_1803_07822_gb300.lattice import CurvedLattice
    # a constant sheared metric (J = I + a small constant matrix): no derivative, every term of the metric present
    N = int(np.prod(n))
    J = np.eye(3) + 0.05 * np.random.default_rng(3).standard_normal((3, 3))
    ch = I.Chart(n, np.repeat(J.reshape(9, 1), N, axis=1), np.zeros((27, N)))
    kw = dict(tau=0.8, fext=(1e-4, 2e-4, -1e-4))
    g = CurvedLattice(n, lo, hi, storage=storage, step_kernel="flat", **kw)
    o = oracle.Lattice(n, lo, hi, **kw)
    g.set_chart(ch)
    o.set_metric(ch.g6, ch.dg18)
    rng = np.random.default_rng(4)
    for a in range(3):
        for s, rule in ((0, lo[a]), (1, hi[a])):
            if rule in (W, IN):
                u = 0.01 * rng.standard_normal((3, g.face_nodes(a)))
                g.set_boundary_velocity(a, s, u)
                o.set_face_velocity(a, s, u)
    rho, u = 1.0 + 0.01 * rng.standard_normal(N), 0.02 * rng.standard_normal((3, N))
    g.init_equilibrium(rho, u)
    o.init(rho, u)
    g.step(7)
    o.step(7)
    tol = {"fp32": 1e-5, "fp64": 1e-11}[storage]  # the bars of the parity tests
    (rg, vg), (ro, vo) = g.moments(cartesian=True), o.moments(ch.J9)
    assert np.linalg.norm(rg - ro) < tol * np.linalg.norm(ro)
    assert np.linalg.norm(vg - vo) < tol * np.linalg.norm(vo)
