"""A four-step sweep that takes a copy of its input rows for late (after it has arrived: no
wait runs out here): the sweep ends, leaves NaN and not numbers made from missing input,
the call that checks a run reports it, and the handle works again afterwards."""
import ctypes

import pytest
import torch

import workloads as W
from paper_1603_09577_gb300 import Solver
from paper_1603_09577_gb300 import _lib as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", ["periodic", "abb"])
@pytest.mark.parametrize("nx,ny", [(1031, 1001), (2048, 1024)])
def test_a_late_copy_is_reported(nx, ny, bc):
    s = Solver(nx, ny, prec="f32", bc=(bc, bc), phi_wall=(0.2, 0.6, 0.1, 0.4), steps_per_pass=2)
    s.set_coeffs(s=W.s9(), conv=0, u=(0.05, 0.02), diff=1, K=(0.02, 0.006, 0.015))
    phi0 = torch.rand((ny, nx), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    assert s.route(8)["fours"] == 2
    want = s.set_phi(phi0).step(8).phi()
    s.check_finite()
    assert C.lib().lbm_debug_late_copies(s.h, 2) == C.LBM_EINVAL
    C.check(C.lib().lbm_debug_late_copies(s.h, 1))
    s.set_phi(phi0).step(8)
    assert torch.isnan(s.phi()).all()
    with pytest.raises(C.LBMError) as e:
        s.check_finite()
    assert e.value.code == C.LBM_ETIMEOUT
    f = ctypes.c_int()
    assert C.lib().lbm_debug_flags(s.h, ctypes.byref(f), None) == 0 and f.value == 16
    C.check(C.lib().lbm_debug_late_copies(s.h, 0))
    assert torch.equal(s.set_phi(phi0).step(8).phi(), want)
    s.check_finite()
