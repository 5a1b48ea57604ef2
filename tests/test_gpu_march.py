"""Sweeps of four time steps (the marching kernel) against one-step launches of the
one-node kernel, bit for bit, where the strips and chunks can go wrong: widths
around multiples of the 120 output columns, odd and unaligned widths (the wrapped
and the wall columns), both wall kinds per axis, heights that leave a short last
chunk, every coefficient family, a source or none, and a per-node tensor field."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from paper_1603_09577_gb300 import Solver

pytestmark = pytest.mark.gpu

BCN = {0: "periodic", 1: "abb"}
# nx, ny, walls, conv, u, diff, r1
CASES = [(1200, 300, (0, 0), 0, (0.05, -0.03), 0, 0.0), (1201, 260, (0, 0), 1, (0.08, 0.05), 1, -0.01),
         (1199, 240, (1, 1), 0, (0.0, 0.0), 2, -0.01), (1198, 261, (1, 0), 1, (0.08, -0.05), 2, 0.0),
         (1083, 301, (0, 1), 0, (0.05, 0.02), 1, -0.01), (130, 2100, (1, 1), 1, (0.04, 0.05), 0, -0.01),
         (129, 2101, (0, 0), 0, (0.05, 0.04), 2, 0.0), (128, 2050, (0, 1), 0, (0.0, 0.0), 0, 0.0),
         (4099, 65, (1, 0), 0, (0.0, 0.0), 1, 0.0), (2402, 120, (1, 1), 1, (0.05, 0.05), 1, 0.0)]


def solver(nx, ny, bc, conv, u, diff, r1, K=None, **kw):
    s = Solver(nx, ny, prec="f32", bc=(BCN[bc[0]], BCN[bc[1]]), phi_wall=(0.2, 0.6, 0.1, 0.4),
               per_cell_K=K is not None, **kw)
    s.set_coeffs(s=W.s9(), conv=conv, u=u, diff=diff, K=(0.02, 0.006, 0.015), r1=r1)
    if K is not None:
        s.set_K_field(K)
    return s


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-bc{c[2][0]}{c[2][1]}-c{c[3]}d{c[5]}" for c in CASES])
def test_sweeps_of_four_equal_single_steps(case):
    phi0 = torch.from_numpy(W.phi0_aniso(case[0], seed=case[0], ny=case[1])).cuda()
    ref = solver(*case, kernel_variant=1).set_phi(phi0).step(21).phi()
    for kw in (dict(), dict(steps_per_pass=2), dict(steps_per_pass=2, kernel_variant=5, block_rows=4)):
        s = solver(*case, **kw).set_phi(phi0).step(21)
        assert torch.equal(s.phi(), ref), kw
        f = ctypes.c_int()
        assert s.lib.lbm_debug_flags(s.h, ctypes.byref(f), None) == 0 and f.value == 0


@pytest.mark.parametrize("case", CASES[::3], ids=[f"{c[0]}x{c[1]}" for c in CASES[::3]])
def test_sweeps_of_four_with_a_tensor_field_equal_node_tiles(case):
    nx, ny = case[0], case[1]
    phi0 = torch.from_numpy(W.phi0_aniso(nx, seed=nx, ny=ny)).cuda()
    K = torch.from_numpy(W.adjoint_inputs(nx, seed=3, ny=ny)[0]).cuda()
    ref = solver(*case, K=K, steps_per_pass=2, block_rows=4).set_phi(phi0).step(20).phi()
    s = solver(*case, K=K, steps_per_pass=2).set_phi(phi0).step(20)
    assert torch.equal(s.phi(), ref)


@pytest.mark.parametrize("spp", [1, 2])
@pytest.mark.parametrize("n", [4, 8, 20, 22])
def test_captured_calls_end_on_the_buffer_they_started_from(spp, n):
    """Every call that could be captured still can: replays equal direct steps."""
    if n % (2 * spp):
        pytest.skip("an odd number of launches was never replayable")
    case = (700, 400, (0, 1), 0, (0.05, 0.02), 1, -0.01)
    phi0 = torch.from_numpy(W.phi0_aniso(700, seed=5, ny=400)).cuda()
    s = solver(*case, steps_per_pass=spp).set_phi(phi0).capture(n)
    for _ in range(3):
        s.replay()
    d = solver(*case, kernel_variant=1).set_phi(phi0).step(3 * n)
    assert torch.equal(s.phi(), d.phi())


def test_sweeps_of_four_match_the_oracle():
    nx, ny = 523, 517
    phi0 = W.phi0_aniso(nx, seed=8, ny=ny)
    s = solver(nx, ny, (1, 1), 1, (0.08, -0.05), 2, -0.01).set_phi(torch.from_numpy(phi0).cuda()).step(40)
    ref = O.run(O.Spec(nx=nx, ny=ny, bc_x=1, bc_y=1, phi_wall=(0.2, 0.6, 0.1, 0.4), s=W.s9(), conv=1, u=(0.08, -0.05),
                       diff=2, K=(0.02, 0.006, 0.015), r0=0.0, r1=-0.01), phi0, 40)
    got = s.phi().cpu().numpy()
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5          # the FP32 bar of the parity tests
