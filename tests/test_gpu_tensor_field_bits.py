"""FP32 with a per-node tensor: with two steps per pass a run has the same bits however it
is split into calls (whole sweeps of several steps, or remainders of one step, on small
lattices and on large ones); with one step per pass the four-node kernel agrees with the
one-node kernel, which recomputes the adjoint's states, in the adjoint's family."""
import pytest
import torch

import workloads as W
from paper_1603_09577_gb300 import Solver

pytestmark = pytest.mark.gpu


def solver(nx, ny, bc="periodic", conv=0, diff=0, r1=0.0, **kw):
    s = Solver(nx, ny, prec="f32", bc=(bc, bc), phi_wall=(0.2, 0.6, 0.1, 0.4), per_cell_K=True, **kw)
    s.set_coeffs(s=W.s9(), conv=conv, u=(0.03, 0.01), diff=diff, r1=r1)
    K, phi0, _ = W.adjoint_inputs(nx, seed=9, ny=ny)
    return s.set_K_field(torch.from_numpy(K).cuda()).set_phi(torch.from_numpy(phi0).cuda())


@pytest.mark.parametrize("nx,ny", [(64, 48), (129, 70), (1024, 700), (1031, 1001)])
@pytest.mark.parametrize("fam", [dict(), dict(bc="abb", conv=1, diff=2, r1=-0.05)], ids=["linear", "walls"])
@pytest.mark.parametrize("launch", [dict(), dict(kernel_variant=5, block_rows=4), dict(fixed_launch=True),
                                    dict(kernel_variant=5, block_rows=4, fixed_launch=True)],
                         ids=["auto", "auto5", "tiles", "pairs"])
def test_splits_of_a_run_agree(nx, ny, fam, launch):
    whole = solver(nx, ny, steps_per_pass=2, **fam, **launch).step(24).phi()
    parts = solver(nx, ny, steps_per_pass=2, **fam, **launch)
    for n in (1, 2, 3, 1, 8, 9):
        parts.step(n)
    assert torch.equal(parts.phi(), whole)


@pytest.mark.parametrize("nx,ny", [(64, 48), (1024, 700)])
def test_four_node_kernel_has_the_bits_of_the_recomputed_states(nx, ny):
    a, b = (solver(nx, ny, kernel_variant=v).step(12).phi() for v in (1, 2))
    assert torch.equal(a, b)
    # with two steps per pass its remainder has the other kernels' bits
    if nx % 4 == 0:
        c, d = (solver(nx, ny, kernel_variant=v, steps_per_pass=2).step(11).phi() for v in (0, 2))
        assert torch.equal(c, d)
