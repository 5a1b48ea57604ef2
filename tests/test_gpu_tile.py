"""Several time steps per launch on small lattices against one-step launches, bit for
bit: grids smaller than a halo, one column or row more than a tiling, odd widths,
both wall kinds per axis, every coefficient family, a source or none, per-node
tensors (FP64), and step counts that are no multiple of a launch's."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from paper_1603_09577_gb300 import Solver

pytestmark = pytest.mark.gpu

BCN = {0: "periodic", 1: "abb"}
# nx, ny, walls, conv, u, diff, r1
CASES = [(2, 2, (0, 0), 0, (0.05, -0.03), 0, 0.0), (3, 5, (1, 1), 1, (0.08, 0.05), 1, -0.01),
         (5, 40, (1, 0), 0, (0.0, 0.0), 2, -0.01), (37, 3, (0, 1), 1, (0.08, -0.05), 2, 0.0),
         (64, 64, (0, 0), 0, (0.05, 0.02), 1, -0.01), (131, 65, (1, 1), 1, (0.04, 0.05), 0, -0.01),
         (128, 128, (0, 0), 0, (0.05, 0.04), 0, 0.0), (199, 201, (0, 1), 0, (0.0, 0.0), 0, 0.0),
         (401, 300, (1, 0), 0, (0.0, 0.0), 1, 0.0), (2000, 7, (1, 1), 1, (0.05, 0.05), 2, 0.0),
         (400, 400, (0, 0), 1, (0.05, 0.05), 1, 0.0), (33, 1500, (0, 0), 0, (0.02, 0.05), 2, -0.01),
         (2, 900, (0, 1), 0, (0.02, 0.05), 1, 0.0), (900, 2, (1, 0), 1, (0.02, 0.05), 1, 0.0),
         (4, 1500, (0, 0), 1, (0.05, 0.05), 0, 0.0)]
IDS = [f"{c[0]}x{c[1]}-bc{c[2][0]}{c[2][1]}-c{c[3]}d{c[5]}" for c in CASES]


def solver(prec, nx, ny, bc, conv, u, diff, r1, K=None, **kw):
    s = Solver(nx, ny, prec=prec, bc=(BCN[bc[0]], BCN[bc[1]]), phi_wall=(0.2, 0.6, 0.1, 0.4),
               per_cell_K=K is not None, **kw)
    s.set_coeffs(s=W.s9(), conv=conv, u=u, diff=diff, K=(0.02, 0.006, 0.015), r1=r1)
    if K is not None:
        s.set_K_field(K)
    return s


def field(nx, ny):
    return torch.from_numpy(np.random.default_rng(nx * 7 + ny).uniform(0.1, 0.9, (ny, nx))).cuda()


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("case", CASES, ids=IDS)
def test_small_lattices_equal_single_steps(prec, case):
    phi0 = field(case[0], case[1])
    ref = solver(prec, *case, kernel_variant=1).set_phi(phi0)
    auto = [solver(prec, *case).set_phi(phi0)]
    if prec == "f32":
        auto += [solver(prec, *case, steps_per_pass=2).set_phi(phi0),
                 solver(prec, *case, steps_per_pass=2, kernel_variant=5, block_rows=4).set_phi(phi0)]
    for n in (1, 2, 3, 8, 23):
        ref.step(n)
        for s in auto:
            assert torch.equal(s.step(n).phi(), ref.phi()), (n, s.desc.steps_per_pass)


@pytest.mark.parametrize("case", CASES[4:7], ids=IDS[4:7])
def test_small_lattices_with_a_tensor_field(case):
    nx, ny = case[0], case[1]
    K = torch.from_numpy(W.adjoint_inputs(nx, seed=3, ny=ny)[0]).cuda()
    ref = solver("f64", *case, K=K, kernel_variant=1).set_phi(field(nx, ny)).step(11).phi()
    assert torch.equal(solver("f64", *case, K=K).set_phi(field(nx, ny)).step(11).phi(), ref)
    # FP32: with two steps per pass, against the node tiles (an even count)
    ref = solver("f32", *case, K=K, steps_per_pass=2, block_rows=4).set_phi(field(nx, ny)).step(10).phi()
    assert torch.equal(solver("f32", *case, K=K, steps_per_pass=2).set_phi(field(nx, ny)).step(10).phi(), ref)


@pytest.mark.parametrize("prec,spp,n", [("f32", 1, 2), ("f32", 1, 30), ("f32", 2, 4), ("f32", 2, 100), ("f64", 1, 10)])
def test_captured_calls_replay(prec, spp, n):
    case = (90, 64, (0, 1), 0, (0.05, 0.02), 1, -0.01)
    s = solver(prec, *case, steps_per_pass=spp).set_phi(field(90, 64)).capture(n)
    for _ in range(3):
        s.replay()
    ref = solver(prec, *case, kernel_variant=1).set_phi(field(90, 64)).step(3 * n)
    assert torch.equal(s.phi(), ref.phi())


@pytest.mark.parametrize("prec,tol", [("f64", 1e-12), ("f32", 1e-5)])
def test_small_lattice_matches_the_oracle(prec, tol):
    nx, ny = 71, 58
    phi0 = W.phi0_aniso(nx, seed=8, ny=ny)
    s = solver(prec, nx, ny, (1, 1), 1, (0.08, -0.05), 2, -0.01).set_phi(torch.from_numpy(phi0).cuda()).step(50)
    ref = O.run(O.Spec(nx=nx, ny=ny, bc_x=1, bc_y=1, phi_wall=(0.2, 0.6, 0.1, 0.4), s=W.s9(), conv=1, u=(0.08, -0.05),
                       diff=2, K=(0.02, 0.006, 0.015), r0=0.0, r1=-0.01), phi0, 50)
    assert np.linalg.norm(s.phi().cpu().numpy() - ref) / np.linalg.norm(ref) <= tol      # the parity tests' bars
