"""Several time steps per launch on the general path's small lattices against one-step
launches of the general kernel: extrapolated axes down to three nodes, widths and
heights one more than a tiling, time-dependent Dirichlet records, every wall kind and
scheme, step counts that are no multiple of a launch's, and splits of a call."""
import numpy as np
import pytest
import torch

import workloads as W
from paper_1603_09577_gb300 import Solver

pytestmark = pytest.mark.gpu

BCN = {0: "periodic", 1: "abb", 2: "nee"}
# rounding differs between the kernels in the last bit only: 30 steps of a stable scheme
# carry it at most linearly, a few hundred units of rounding at the field's scale
TOL = {"f64": 30 * 16 * 2.0 ** -53, "f32": 30 * 16 * 2.0 ** -24}
CASES = [(3, 3, (2, 2)), (3, 40, (2, 0)), (61, 5, (0, 2)), (64, 64, (2, 2)), (133, 71, (2, 2)), (97, 130, (1, 1)),
         (301, 301, (2, 2)), (160, 33, (2, 0)), (50, 50, (0, 0)),
         (3, 5, (2, 2)), (2, 2, (0, 0)), (2, 3, (1, 0)), (2, 900, (0, 1)), (900, 3, (0, 2))]
COEF = dict(conv=2, power=2, u=(0.06, -0.03), diff=1, K=(0.02, 0.008, 0.01))


def solver(prec, nx, ny, bc, scheme, rec, **kw):
    s = Solver(nx, ny, prec=prec, bc=(BCN[bc[0]], BCN[bc[1]]), phi_wall=(0.1, 0.2, 0.3, 0.4), scheme=scheme, **kw)
    src = dict(src_family=1, b=0.02) if scheme == "A" else dict(r1=-0.01)
    s.set_coeffs(s=W.s9(), **COEF, **src)
    if 2 in bc:
        s.set_dirichlet(rec)
    return s


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("scheme", ["A", "B"])
@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-bc{c[2][0]}{c[2][1]}" for c in CASES])
def test_small_general_lattices(prec, scheme, case):
    nx, ny, bc = case
    rng = np.random.default_rng(nx * 7 + ny)
    phi0 = torch.from_numpy(W.jacobi_smooth(rng.uniform(0.2, 0.8, (ny, nx)), 1)).cuda()
    rec = torch.from_numpy(rng.uniform(0.3, 0.7, (25, 2 * (nx + ny)))).cuda()
    ref = solver(prec, nx, ny, bc, scheme, rec, kernel_variant=1).set_phi(phi0).step(30).phi()
    whole = solver(prec, nx, ny, bc, scheme, rec).set_phi(phi0).step(30).phi()
    assert ((whole - ref).norm() / ref.norm()).item() <= TOL[prec]
    parts = solver(prec, nx, ny, bc, scheme, rec).set_phi(phi0)
    for n in (1, 2, 7, 20):
        parts.step(n)
    assert torch.equal(parts.phi(), whole)
