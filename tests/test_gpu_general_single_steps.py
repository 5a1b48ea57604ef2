"""Single steps of the general path's small lattices run over tiles of their own (32 x 4,
or the lattice where it is smaller; the last one of an axis overlaps its neighbour): runs
of single steps equal whole calls bit for bit around multiples of the tile, down to the
smallest lattices, for every wall kind and both schemes."""
import numpy as np
import pytest
import torch

import workloads as W
from paper_1603_09577_gb300 import Solver

pytestmark = pytest.mark.gpu

BCN = {0: "periodic", 1: "abb", 2: "nee"}
SIZES = [(3, 3), (31, 4), (32, 8), (33, 9), (64, 48), (65, 33), (3, 200), (200, 3), (301, 130), (350, 350)]


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("scheme", ["A", "B"])
@pytest.mark.parametrize("bc", [(2, 2), (0, 2), (1, 1), (0, 0)])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_single_steps_equal_whole_calls(prec, scheme, bc, nx, ny):
    rng = np.random.default_rng(nx * 7 + ny)
    phi0 = torch.from_numpy(rng.uniform(0.2, 0.8, (ny, nx))).cuda()
    rec = torch.from_numpy(rng.uniform(0.3, 0.7, (6, 2 * (nx + ny)))).cuda()

    def solver():
        s = Solver(nx, ny, prec=prec, bc=(BCN[bc[0]], BCN[bc[1]]), phi_wall=(0.1, 0.2, 0.3, 0.4), scheme=scheme)
        s.set_coeffs(s=W.s9(), conv=2, power=2, u=(0.06, -0.03), diff=1, K=(0.02, 0.008, 0.01),
                     **(dict(src_family=1, b=0.02) if scheme == "A" else dict(r1=-0.01)))
        return (s.set_dirichlet(rec) if 2 in bc else s).set_phi(phi0)

    whole, parts = solver().step(9), solver()
    for _ in range(9):
        parts.step(1)
    assert torch.equal(parts.phi(), whole.phi())
