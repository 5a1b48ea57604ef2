"""Long FP32 runs against the FP64 path: the error stays at the rounding of the stored
populations (one unit of the last place, 2^-23, in relative L2) and has no drift of the
mean (a fifth of that), whichever family, source or launch. A step whose roundings lean
one way adds up over thousands of steps."""
import math

import pytest
import torch

import workloads as W
from paper_1603_09577_gb300 import Solver

pytestmark = pytest.mark.gpu

# n, steps, conv, u, diff, K, r1, mean of the field
CASES = [(256, 3000, 1, (math.sqrt(0.5),) * 2, 0, (0.32, 0.0, 0.32), 0.0, 0.0),
         (256, 3000, 1, (math.sqrt(0.5),) * 2, 0, (0.32, 0.0, 0.32), 0.0, 0.35),
         (128, 2000, 0, (0.0, 0.0), 2, (0.02, 0.008, 0.02), -5e-5, 0.3),
         (128, 1500, 0, (0.0, 0.0), 2, (0.02, 0.0, 0.02), 0.0, 0.35),
         (128, 1500, 1, (0.05, -0.03), 0, (0.02, 0.0, 0.02), -5e-5, 0.35),
         (128, 1500, 0, (0.05, -0.03), 0, (0.02, 0.0, 0.02), -5e-5, 0.35)]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}-c{c[2]}d{c[4]}r{int(c[6] != 0)}m{c[7]}" for c in CASES])
def test_error_of_long_runs_stays_at_rounding(case):
    n, steps, conv, u, diff, K, r1, mean = case
    x = torch.arange(n, dtype=torch.float64, device="cuda") * (2 * math.pi / n)
    gen = torch.Generator(device="cuda").manual_seed(1)
    noise = 1e-3 * (2 * torch.rand((n, n), generator=gen, device="cuda", dtype=torch.float64) - 1)
    phi0 = (mean + (0.5 if mean < 0.31 else 0.3) * torch.sin(x)[None, :] * torch.sin(x)[:, None] + noise).float()

    def run(prec):
        dtype, pitch = torch.float64 if prec == "f64" else torch.float32, (n + 63) // 64 * 64
        s = Solver(n, n, prec=prec).set_coeffs(s=W.s9(), conv=conv, u=u, diff=diff, K=K, r1=r1)
        state = s.set_phi(phi0.to(dtype)).step(steps).save().view(dtype)
        # phi from the stored populations in 64 bits: the read-out's own constant, rounded
        # to FP32, would scale the field by up to 2^-24
        return state[:9 * n * pitch].view(9, n, pitch)[:, :, :n].double().sum(0) / (1.0 + 0.5 * r1)

    ref, got = run("f64"), run("f32")
    assert ((got - ref).norm() / ref.norm()).item() <= 2.0 ** -23
    assert abs((got - ref).sum().item()) / ref.abs().sum().item() <= 0.2 * 2.0 ** -23
