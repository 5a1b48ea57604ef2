"""The stored initial state (Eq. 40 and the first collision) against the oracle's,
population by population, for every coefficient family with and without a source.
Values are O(1) and some 45 rounded operations deep: 64 units of the last place."""
import numpy as np
import pytest
import torch

import oracle as O
import oracle.d3q19 as D
import workloads as W
from paper_1603_09577_gb300 import Solver, Solver3

pytestmark = pytest.mark.gpu

FAMILIES = [(c, d, r) for c in (0, 1) for d in (0, 1, 2) for r in ((0.0, 0.0), (0.02, -0.03))]
U2, K2 = (0.06, -0.04), (0.02, 0.006, 0.015)
U3, K3 = (0.05, -0.03, 0.02), (0.02, 0.006, 0.004, 0.015, 0.003, 0.01)


@pytest.mark.parametrize("conv,diff,r", FAMILIES)
@pytest.mark.parametrize("u", [U2, (0.0, 0.0)])
def test_initial_state_f64(conv, diff, r, u):
    nx, ny = 33, 9
    phi0 = np.random.default_rng(5).uniform(-0.9, 0.9, (ny, nx))
    kw = dict(conv=conv, u=u, diff=diff, K=K2, r0=r[0], r1=r[1])
    s = Solver(nx, ny, prec="f64").set_coeffs(s=W.s9(), **kw).set_phi(torch.from_numpy(phi0).cuda())
    st = s.save().view(torch.float64)
    pitch = (nx + 63) // 64 * 64
    got = st[:9 * pitch * ny].view(9, ny, pitch)[:, :, :nx].cpu().numpy()
    ref = O.init(O.Spec(nx=nx, ny=ny, s=W.s9(), **kw), phi0)
    assert np.abs(got - ref).max() <= 64 * 2.0 ** -53
    assert np.abs(s.phi().cpu().numpy() - phi0).max() <= 64 * 2.0 ** -53


@pytest.mark.parametrize("conv,diff,r", FAMILIES)
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_initial_state_d3q19(prec, conv, diff, r):
    nx, ny, nz = 33, 5, 4
    phi0 = np.random.default_rng(6).uniform(-0.9, 0.9, (nz, ny, nx))
    kw = dict(conv=conv, u=U3, diff=diff, K=K3, se=1.1, r0=r[0], r1=r[1])
    s = Solver3(nx, ny, nz, prec=prec).set_coeffs(**kw).set_phi(torch.from_numpy(phi0).cuda())
    pitch = (nx + 63) // 64 * 64
    st = s.save().view(torch.float64 if prec == "f64" else torch.float32)
    got = st[:19 * nz * ny * pitch].view(19, nz, ny, pitch)[..., :nx].cpu().numpy()
    ref = D.init(D.Spec3(nx=nx, ny=ny, nz=nz, **kw), phi0)
    assert np.abs(got - ref).max() <= 64 * (2.0 ** -53 if prec == "f64" else 2.0 ** -24)
