"""The marching kernel (sweeps of four time steps) where it runs: every case asserts that the
library takes it, for 148 and 152 SMs, and compares it with one-step launches bit for bit.
Widths around multiples of the strips' 120 columns, odd and unaligned ones (wrapped columns,
wall columns, copies column by column), every pair of walls with both parities of the width,
short last chunks, every coefficient family with and without a source, tensor fields, graphs."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from paper_1603_09577_gb300 import Solver

pytestmark = pytest.mark.gpu

BCN = {0: "periodic", 1: "abb"}
SIZES = [(1031, 1001), (1199, 997), (1200, 1003), (1201, 1100), (1320, 801), (4099, 300), (239, 5003), (2402, 500),
         (6001, 130), (238, 20001)]
# nx, ny, walls, conv, u, diff, r1: every pair of walls with odd and even widths, every family
CASES = [(*SIZES[i % len(SIZES)], (i // 2 % 2, i // 4 % 2), i // 3 % 3 == 0, (0.0, 0.0) if i % 3 == 1 else (0.06, -0.04),
          i % 3, -0.01 if i % 2 else 0.0) for i in range(24)]


def solver(nx, ny, bc, conv, u, diff, r1, K=None, **kw):
    s = Solver(nx, ny, prec="f32", bc=(BCN[bc[0]], BCN[bc[1]]), phi_wall=(0.2, 0.6, 0.1, 0.4),
               per_cell_K=K is not None, **kw)
    s.set_coeffs(s=W.s9(), conv=int(conv), u=u, diff=diff, K=(0.02, 0.006, 0.015), r1=r1)
    return s.set_K_field(K) if K is not None else s


def field(nx, ny):
    return torch.from_numpy(np.random.default_rng(nx * 7 + ny).uniform(0.1, 0.9, (ny, nx))).cuda()


def marches(s, n):
    return all(s.route(n, sms)["fours"] >= 2 for sms in (148, 152, 0))


def flags(s):
    f = ctypes.c_int()
    assert s.lib.lbm_debug_flags(s.h, ctypes.byref(f), None) == 0
    return f.value


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-bc{c[2][0]}{c[2][1]}-c{int(c[3])}d{c[5]}r{int(c[6] != 0)}"
                                             for c in CASES])
def test_sweeps_of_four_equal_single_steps(case):
    phi0 = field(case[0], case[1])
    ref = solver(*case, kernel_variant=1).set_phi(phi0).step(41).phi()
    for kw in (dict(), dict(steps_per_pass=2), dict(steps_per_pass=2, kernel_variant=5, block_rows=4)):
        s = solver(*case, **kw).set_phi(phi0)
        assert marches(s, 41), s.route(41)
        assert torch.equal(s.step(41).phi(), ref) and flags(s) == 0, kw


@pytest.mark.parametrize("i", range(8))
def test_tensor_fields(i):
    nx, ny = SIZES[i]
    case = (nx, ny, (i % 2, i // 2 % 2), i % 2, (0.03, 0.01), i % 3, -0.01 * (i % 2))
    K = torch.from_numpy(W.adjoint_inputs(nx, seed=3, ny=ny)[0]).cuda()
    phi0 = field(nx, ny)
    s = solver(*case, K=K, steps_per_pass=2).set_phi(phi0)
    assert marches(s, 41)
    ref = solver(*case, K=K, steps_per_pass=2, block_rows=4, fixed_launch=True).set_phi(phi0).step(41).phi()
    assert torch.equal(s.step(41).phi(), ref) and flags(s) == 0


@pytest.mark.parametrize("spp,n", [(1, 20), (1, 44), (2, 20), (2, 24)])
@pytest.mark.parametrize("bc", [(0, 0), (1, 0), (1, 1)])
def test_captured_calls_replay(spp, n, bc):
    case = (1201, 1100, bc, 0, (0.05, 0.02), 1, -0.01)
    phi0 = field(1201, 1100)
    s = solver(*case, steps_per_pass=spp).set_phi(phi0)
    assert marches(s, n)
    s.capture(n)
    for _ in range(3):
        s.replay()
    assert torch.equal(s.phi(), solver(*case, kernel_variant=1).set_phi(phi0).step(3 * n).phi())


def test_sweeps_of_four_match_the_oracle():
    nx, ny = 1031, 523
    phi0 = W.phi0_aniso(nx, seed=8, ny=ny)
    s = solver(nx, ny, (1, 1), 1, (0.08, -0.05), 2, -0.01).set_phi(torch.from_numpy(phi0).cuda())
    assert marches(s, 40)
    got = s.step(40).phi().cpu().numpy()
    ref = O.run(O.Spec(nx=nx, ny=ny, bc_x=1, bc_y=1, phi_wall=(0.2, 0.6, 0.1, 0.4), s=W.s9(), conv=1, u=(0.08, -0.05),
                       diff=2, K=(0.02, 0.006, 0.015), r0=0.0, r1=-0.01), phi0, 40)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5          # the FP32 bar of the parity tests
