"""Runs the kernels that serve large lattices only, of liblbm_checked.so, on the smallest
lattices that take them, and the ones that a fixed launch selects: one JSON line with the
index-fault words, what was reached, and the largest difference from the one-step kernels.
Started by test_gpu_checked_large.py with LBM_LIBRARY=checked in a fresh process."""
import ctypes
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
sys.path.insert(0, ROOT)

import torch  # noqa: E402

import workloads as W  # noqa: E402
from paper_1603_09577_gb300 import Ensemble, Solver, Solver3  # noqa: E402
from paper_1603_09577_gb300 import _lib as C  # noqa: E402

BCN = {0: "periodic", 1: "abb", 2: "nee"}


def main():
    out = {"checked": C.lib().lbm_build_checked(), "faults": [], "max_diff": 0.0, "reached": {}}
    gen = torch.Generator(device="cuda").manual_seed(1)

    def note(name, reached, fn, h, got, ref):
        f = ctypes.c_int()
        C.check(fn(h, ctypes.byref(f), None))
        out["faults"].append(f.value)
        out["reached"][name] = out["reached"].get(name, 0) + int(reached)
        out["max_diff"] = max(out["max_diff"], float((got - ref).abs().max()))

    def run2(name, kernel, nx, ny, bc, steps, K=None, conv=1, **kw):
        def make(**launch):
            s = Solver(nx, ny, prec="f32", bc=(BCN[bc[0]], BCN[bc[1]]), phi_wall=(0.1, 0.2, 0.3, 0.4),
                       per_cell_K=K is not None, **launch)
            s.set_coeffs(s=W.s9(), conv=conv, u=(0.06, -0.03), diff=2, K=(0.02, 0.008, 0.01), r1=-0.05)
            return s if K is None else s.set_K_field(K)
        phi0 = torch.rand((ny, nx), generator=gen, device="cuda") * 0.5 + 0.2
        s = make(**kw).set_phi(phi0)
        ref = make(**(dict(kernel_variant=1) if K is None else dict(steps_per_pass=2, fixed_launch=True, block_rows=4)))
        reached = s.route(steps)[kernel]
        note(name, reached, s.lib.lbm_debug_flags, s.h, s.step(steps).phi(), ref.set_phi(phi0).step(steps).phi())

    for nx, ny in ((1031, 701), (1200, 997), (1199, 1003)):
        for bc in ((0, 0), (0, 1), (1, 0), (1, 1)):
            run2("march", "fours", nx, ny, bc, 20)
    run2("march", "fours", 1031, 1001, (1, 1), 20, conv=0)
    run2("march_kfield", "fours", 1031, 1001, (1, 0), 20, K=torch.from_numpy(W.adjoint_inputs(1031, seed=3, ny=1001)[0]).cuda(),
         steps_per_pass=2)
    for nx, ny, bc in ((37, 29, (1, 1)), (132, 35, (1, 0)), (201, 90, (0, 0)), (190, 77, (0, 1))):
        run2("pairs", "pairs", nx, ny, bc, 10, steps_per_pass=2, kernel_variant=5, block_rows=4, fixed_launch=True)
        run2("nodes", "twos", nx, ny, bc, 10, steps_per_pass=2, fixed_launch=True)
        run2("tiles", "tiles", nx, ny, bc, 10)
    # D3Q19 sweeps
    for nx, ny, nz in ((240, 15, 1200), (161, 161, 163), (31, 31, 4400)):
        def make3(**kw):
            return Solver3(nx, ny, nz, prec="f32", **kw).set_coeffs(
                conv=1, u=(0.05, -0.03, 0.02), diff=1, K=(0.02, 0.004, -0.003, 0.015, 0.002, 0.012), se=1.2, r1=-0.01)
        phi0 = torch.rand((nz, ny, nx), generator=gen, device="cuda") * 0.5 + 0.2
        s3 = make3().set_phi(phi0)
        note("sweep3", s3.route(6)["sweeps"], s3.lib.lbm3_debug_flags, s3.h, s3.step(6).phi(),
             make3(block_rows=8).set_phi(phi0).step(6).phi())
    # ensemble strips
    inst = [dict(nx=a, ny=b, u=(0.05, -0.03), K=(0.02, 0.004, 0.015))
            for a, b in [(119, 311), (121, 129), (239, 1000), (241, 517), (16, 16), (640, 17), (359, 31), (1000, 1001),
                         (17, 640), (482, 479)] * 3]
    e = Ensemble(inst, steps_per_pass=2)
    phi = torch.rand(e.nodes, generator=gen, device="cuda") * 0.5 + 0.2
    note("strips", e.route(13)["fours"], e.lib.lbm_ensemble_debug_flags, e.h, e.set_phi(phi).step(13).phi(),
         Ensemble(inst, steps_per_pass=1).set_phi(phi).step(13).phi())
    # general path: single steps in small tiles, tiles of several
    for nx, ny, bc in ((37, 29, (2, 2)), (33, 41, (0, 2)), (35, 22, (1, 0)), (3, 5, (2, 2))):
        def makeg():
            s = Solver(nx, ny, prec="f32", bc=(BCN[bc[0]], BCN[bc[1]]), phi_wall=(0.1, 0.2, 0.3, 0.4), scheme="A")
            s.set_coeffs(s=W.s9(), conv=2, power=1, u=(0.06, -0.03), diff=1, K=(0.02, 0.008, 0.01), src_family=1, b=0.02)
            return s.set_dirichlet(torch.full((1, 2 * (nx + ny)), 0.5, dtype=torch.float64, device="cuda")) if 2 in bc else s
        phi0 = torch.rand((ny, nx), generator=gen, device="cuda") * 0.5 + 0.2
        s, whole = makeg().set_phi(phi0), makeg().set_phi(phi0).step(7).phi()
        for _ in range(7):
            s.step(1)
        note("general_single", s.route(1)["tiles"], s.lib.lbm_debug_flags, s.h, s.phi(), whole)
    print(json.dumps(out))


if __name__ == "__main__":
    main()
