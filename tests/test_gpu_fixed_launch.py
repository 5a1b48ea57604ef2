"""The FP32 two-step kernels on their own (fixed launches): the 62 x 14 pair tiles, which
the library otherwise runs as the remainder of longer sweeps and the tiles of sizes in
between, and the 30 x 62 node tiles, each against the one-step kernel bit for bit on small,
ragged and odd grids, walls of every kind, every coefficient family, a tensor field."""
import numpy as np
import pytest
import torch

import workloads as W
from paper_1603_09577_gb300 import Solver

pytestmark = pytest.mark.gpu

BCN = {0: "periodic", 1: "abb"}
CASES = [(300, 250, (1, 1)), (257, 131, (0, 0)), (190, 64, (1, 0)), (129, 200, (0, 1)), (64, 17, (1, 1)), (131, 19, (0, 0)),
         (62, 14, (1, 1)), (63, 15, (0, 0)), (2, 3, (0, 0)), (3, 2, (1, 1)), (125, 29, (0, 1)), (61, 13, (1, 0))]
KERNELS = [("pairs", dict(kernel_variant=5, block_rows=4)), ("twos", dict(kernel_variant=0, block_rows=0))]


def solver(nx, ny, bc, conv=0, diff=0, K=None, **kw):
    s = Solver(nx, ny, prec="f32", bc=(BCN[bc[0]], BCN[bc[1]]), phi_wall=(0.2, 0.6, 0.1, 0.4), per_cell_K=K is not None,
               fixed_launch=True, **kw)
    s.set_coeffs(s=W.s9(), conv=conv, u=(0.05, -0.03), diff=diff, K=(0.02, 0.006, 0.015), r1=-0.05 if K is None else 0.0)
    return s.set_K_field(K) if K is not None else s


@pytest.mark.parametrize("kernel,kw", KERNELS, ids=[k for k, _ in KERNELS])
@pytest.mark.parametrize("i", range(len(CASES)), ids=[f"{c[0]}x{c[1]}-bc{c[2][0]}{c[2][1]}" for c in CASES])
def test_two_step_kernels_equal_single_steps(i, kernel, kw):
    nx, ny, bc = CASES[i]
    phi0 = torch.from_numpy(np.random.default_rng(i).uniform(0.2, 0.8, (ny, nx))).cuda()
    for conv in (0, 1):
        fam = dict(conv=conv, diff=i % 3)
        ref = solver(nx, ny, bc, kernel_variant=1, **fam).set_phi(phi0).step(21).phi()
        s = solver(nx, ny, bc, steps_per_pass=2, **fam, **kw).set_phi(phi0)
        assert s.route(21)[kernel] == 10
        assert torch.equal(s.step(21).phi(), ref), fam


@pytest.mark.parametrize("nx,ny", [(260, 150), (131, 19), (62, 15)])
def test_pair_tiles_with_a_tensor_field_equal_node_tiles(nx, ny):
    K = torch.from_numpy(W.adjoint_inputs(nx, seed=9, ny=ny)[0]).cuda()
    phi0 = torch.from_numpy(W.phi0_aniso(nx, seed=9, ny=ny)).cuda()
    a, b, c = (solver(nx, ny, (0, 0), K=K, steps_per_pass=2, **kw).set_phi(phi0).step(20).phi()
               for kw in (dict(kernel_variant=5, block_rows=4), dict(), dict(block_rows=4)))
    assert torch.equal(a, b) and torch.equal(b, c)
