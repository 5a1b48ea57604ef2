"""Host time of the calls that a time loop makes: the constants of a launch are made
once per set of coefficients, so a launch of a D3Q19 step costs the host about what
one of a D2Q9 step does (made at every launch they doubled it)."""
import time

import pytest
import torch

from paper_1603_09577_gb300 import Solver, Solver3

pytestmark = pytest.mark.gpu


def per_launch(step, launches=40, reps=60):
    """Least host time of one launch over many calls that enqueue `launches` of them."""
    step(launches)
    best = float("inf")
    for _ in range(reps):
        torch.cuda.synchronize()
        t = time.perf_counter()
        step(launches)
        best = min(best, time.perf_counter() - t)
    return best / launches


@pytest.mark.parametrize("prec", ["f32", "f64", "bf16s"])
@pytest.mark.parametrize("bc", ["periodic", "abb"])
def test_d3q19_launches_cost_the_host_no_more_than_d2q9(prec, bc):
    s2 = Solver(32, 32, prec=prec, bc=(bc, bc), kernel_variant=1)
    s2.set_coeffs(u=(0.03, 0.01), K=(0.02, 0.004, 0.015)).set_phi(torch.rand((32, 32), device="cuda"))
    s3 = Solver3(8, 8, 8, prec=prec, bc=(bc,) * 3)
    s3.set_coeffs(u=(0.05, 0.02, 0.01), K=(0.02, 0.004, 0.002, 0.015, 0.003, 0.01), se=1.1)
    s3.set_phi(torch.rand((8, 8, 8), device="cuda"))
    assert per_launch(s3.step) <= 1.5 * per_launch(s2.step)
