"""D3Q19, FP32: two steps per sweep against the one-step kernel, bit for bit, on the
smallest lattices that take the sweeps: widths of a whole number of 30-column tiles
and one more, odd widths (split pairs), short last tiles and chunks, every family."""
import numpy as np
import pytest
import torch

from paper_1603_09577_gb300 import Solver3

pytestmark = pytest.mark.gpu

K = (0.02, 0.006, 0.004, 0.015, 0.003, 0.01)
CASES = [(240, 210, 96, 0, 0, 0.0), (241, 141, 130, 1, 1, -0.01), (242, 155, 113, 0, 2, -0.01),
         (2100, 45, 49, 1, 0, 0.0), (31, 300, 467, 0, 1, 0.0), (96, 15, 3000, 1, 2, -0.01)]


def solver(nx, ny, nz, conv, diff, r1, **kw):
    return Solver3(nx, ny, nz, prec="f32", **kw).set_coeffs(conv=conv, u=(0.05, -0.03, 0.02), diff=diff, K=K, se=1.1, r1=r1)


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}x{c[2]}-c{c[3]}d{c[4]}" for c in CASES])
def test_two_step_sweeps_equal_single_steps(case):
    nx, ny, nz = case[:3]
    assert nx * ny * nz >= 1 << 22
    phi0 = torch.from_numpy(np.random.default_rng(nx).uniform(0.2, 0.8, (nz, ny, nx)).astype(np.float32)).cuda()
    ref = solver(*case, block_rows=8).set_phi(phi0)
    s = solver(*case).set_phi(phi0)
    for n in (4, 1, 6):
        assert torch.equal(s.step(n).phi(torch.float32), ref.step(n).phi(torch.float32)), n


def test_captured_sweeps_replay():
    case = CASES[0]
    phi0 = torch.rand((96, 210, 240), device="cuda")
    s = solver(*case).set_phi(phi0).capture(6)
    for _ in range(2):
        s.replay()
    assert torch.equal(s.phi(torch.float32), solver(*case, block_rows=8).set_phi(phi0).step(12).phi(torch.float32))
