"""Routes of narrow, flat and in-between FP32 and FP64 lattices against one-step launches,
bit for bit, in calls of one to many steps: single steps, 30 x 30 node tiles, pair tiles
and small lattices' tiles meet there, whichever the estimates choose."""
import numpy as np
import pytest
import torch

import workloads as W
from paper_1603_09577_gb300 import Solver

pytestmark = pytest.mark.gpu

BCN = {0: "periodic", 1: "abb"}
SIZES = [(64, 5000), (33, 9000), (2, 30000), (30000, 3), (121, 6001), (91, 5000), (5000, 33), (600, 600), (520, 777)]


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("bc", [(0, 0), (1, 1), (0, 1), (1, 0)])
def test_routes_equal_single_steps(prec, nx, ny, bc):
    def solver(**kw):
        s = Solver(nx, ny, prec=prec, bc=(BCN[bc[0]], BCN[bc[1]]), phi_wall=(0.2, 0.6, 0.1, 0.4), **kw)
        return s.set_coeffs(s=W.s9(), conv=1, u=(0.05, -0.03), diff=nx % 3, K=(0.02, 0.006, 0.015), r1=-0.01)

    phi0 = torch.from_numpy(np.random.default_rng(nx).uniform(0.2, 0.8, (ny, nx))).cuda()
    ref = solver(kernel_variant=1).set_phi(phi0)
    runs = [solver(**kw).set_phi(phi0) for kw in ([dict()] if prec == "f64" else [dict(), dict(steps_per_pass=2)])]
    for n in (1, 2, 3, 4, 7, 16):
        ref.step(n)
        for s in runs:
            assert torch.equal(s.step(n).phi(), ref.phi()), (n, s.route(n))
