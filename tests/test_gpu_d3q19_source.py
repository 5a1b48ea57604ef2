"""D3Q19 with the linear flux and an affine source, whose constant and linear parts join
the collision's other terms in phi on the host: every diffusion function, a source of
either part alone and both, periodic axes and walls, against the oracle at the bars of
the parity tests."""
import numpy as np
import pytest
import torch

from oracle import d3q19 as D
from paper_1603_09577_gb300 import Solver3

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5}


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 0, 1)])
@pytest.mark.parametrize("diff", [0, 1, 2])
@pytest.mark.parametrize("r", [(0.02, 0.0), (0.0, -0.05), (0.01, 0.03), (-0.03, 0.5)])
def test_linear_flux_with_an_affine_source(prec, bc, diff, r):
    nx, ny, nz = 33, 9, 6
    kw = dict(conv=0, u=(0.05, -0.03, 0.02), diff=diff, K=(0.02, 0.004, -0.003, 0.015, 0.002, 0.012), se=1.2, r0=r[0], r1=r[1])
    pw = (0.1, 0.2, 0.3, 0.4, 0.5, 0.6)
    phi0 = np.random.default_rng(diff).uniform(0.2, 0.8, (nz, ny, nx))
    steps = 3 if r[1] > 0.1 else 20                  # the fast growth stays at O(1)
    ref = D.run(D.Spec3(nx=nx, ny=ny, nz=nz, bc=bc, phi_wall=pw, **kw), phi0, steps)
    s = Solver3(nx, ny, nz, prec=prec, bc=["abb" if b else "periodic" for b in bc], phi_wall=pw).set_coeffs(**kw)
    got = s.set_phi(torch.from_numpy(phi0).cuda()).step(steps).phi().cpu().numpy()
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= TOL[prec]
