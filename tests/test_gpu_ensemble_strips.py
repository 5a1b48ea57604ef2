"""The four-step strips of an ensemble against the two-step pair tiles and single steps,
bit for bit, as the header promises: odd and rectangular instances from 16 nodes a side to
over a thousand, widths around multiples of the strips' 120 columns, heights that leave
short last chunks, every coefficient family, step counts that are no multiple of a sweep
pair's, and replayed graphs. The ensembles are large enough to take strips."""
import ctypes

import numpy as np
import pytest
import torch

import workloads as W
from paper_1603_09577_gb300.ensemble import Ensemble

pytestmark = pytest.mark.gpu

SIDES = [(119, 311), (120, 64), (121, 129), (239, 1000), (240, 33), (241, 517), (16, 16), (17, 640), (640, 17), (359, 31),
         (361, 999), (1023, 16), (1000, 1001), (123, 20), (482, 479)]


def instances():
    rng = np.random.default_rng(11)
    out = []
    for nx, ny in SIDES * 3:
        d0 = rng.uniform(0.005, 0.05)
        out.append(dict(nx=nx, ny=ny, u=tuple(rng.uniform(-0.06, 0.06, 2)), K=(d0, 0.2 * d0, 0.8 * d0)))
    return out


def flags(e):
    f = ctypes.c_int()
    assert e.lib.lbm_ensemble_debug_flags(e.h, ctypes.byref(f), None) == 0
    return f.value


@pytest.mark.parametrize("conv", [0, 1])
@pytest.mark.parametrize("diff", [0, 1, 2])
def test_strips_equal_pair_tiles_and_single_steps(conv, diff):
    inst = instances()
    kw = dict(conv=conv, diff=diff, s=W.s9())
    e = Ensemble(inst, steps_per_pass=2, **kw)
    phi = torch.rand(e.nodes, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda") * 0.5 + 0.2
    assert e.route(61) == dict(fours=14, twos=2, ones=1)
    want = Ensemble(inst, steps_per_pass=1, **kw).set_phi(phi).step(61).phi()
    assert torch.equal(e.set_phi(phi).step(61).phi(), want) and flags(e) == 0
    assert torch.equal(Ensemble(inst, steps_per_pass=2, pair_tiles=True, **kw).set_phi(phi).step(61).phi(), want)


def test_captured_strips_replay():
    inst = instances()
    e = Ensemble(inst, steps_per_pass=2)
    phi = torch.rand(e.nodes, device="cuda") * 0.5 + 0.2
    want = Ensemble(inst, steps_per_pass=1).set_phi(phi).step(61).phi()
    e.set_phi(phi)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        e.capture(20)
        for _ in range(3):
            e.replay()
        e.step(1)
    torch.cuda.current_stream().wait_stream(side)
    assert torch.equal(e.phi(), want) and flags(e) == 0
