"""D3Q19 FP32 lattices whose shape decides between two-step sweeps and single steps: the
sweeps of narrow, flat and odd lattices (one row more than a tile, rows of a few nodes,
chunks of two planes) against the one-step kernel bit for bit, and flat lattices, which
take single steps."""
import numpy as np
import pytest
import torch

from paper_1603_09577_gb300 import Solver3

pytestmark = pytest.mark.gpu

CASES = [(240, 15, 1200, True), (241, 29, 601, True), (31, 31, 4400, True), (8, 9, 65535, True), (513, 511, 17, True),
         (4096, 512, 2, True), (96, 15, 3000, False), (4096, 2, 512, False)]


@pytest.mark.parametrize("nx,ny,nz,sweeps", CASES)
def test_narrow_and_flat_lattices(nx, ny, nz, sweeps):
    def solver(**kw):
        return Solver3(nx, ny, nz, prec="f32", **kw).set_coeffs(
            conv=nx % 2, u=(0.05, -0.03, 0.02), diff=ny % 3, K=(0.02, 0.006, 0.004, 0.015, 0.003, 0.01), se=1.1, r1=-0.01)

    phi0 = torch.from_numpy(np.random.default_rng(nx).uniform(0.2, 0.8, (nz, ny, nx)).astype(np.float32)).cuda()
    s, ref = solver().set_phi(phi0), solver(block_rows=8).set_phi(phi0)
    assert (s.route(4)["sweeps"] > 0) == sweeps
    for n in (4, 3, 6):
        assert torch.equal(s.step(n).phi(torch.float32), ref.step(n).phi(torch.float32)), n
