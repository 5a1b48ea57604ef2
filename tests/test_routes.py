"""Which kernels serve a call, asked of the library on the CPU (lbm_step_route,
lbm3_step_route): every route adds up to the steps asked for, keeps the number of
launches odd or even as steps_per_pass has it (captured calls then end on the buffer
they started from), and is what the benchmark's records name."""
import ctypes
import time

import pytest

import bench
from paper_1603_09577_gb300 import _lib as C
from paper_1603_09577_gb300.solver import BC, ROUTE_KEYS, SCHEME

SMS = (148, 152)


class Lattice:
    """A handle on a host stand-in for the workspace: routes need no device."""

    def __init__(self, nx, ny, prec="f32", bc=("periodic", "periodic"), steps_per_pass=1, per_cell_K=False,
                 kernel_variant=0, block_rows=0, scheme="B", conv=0, u=(0.05, 0.02), diff=0, power=1, b=0.0, r1=0.0):
        self.lib, self.nx, self.ny, self.prec = C.lib(), nx, ny, prec
        d = C.Desc()
        d.nx, d.ny, d.prec, d.bc_x, d.bc_y = nx, ny, C.PREC[prec], BC[bc[0]], BC[bc[1]]
        d.steps_per_pass, d.per_cell_K = steps_per_pass, int(per_cell_K)
        d.kernel_variant, d.block_rows, d.scheme = kernel_variant, block_rows, SCHEME[scheme]
        self.desc = d
        n = ctypes.c_size_t()
        C.check(self.lib.lbm_workspace_size(ctypes.byref(d), ctypes.byref(n)))
        self.h = ctypes.c_void_p()
        # the address is only recorded: nothing below touches the workspace
        C.check(self.lib.lbm_create(ctypes.byref(self.h), ctypes.byref(d), ctypes.c_void_p(1 << 20), n.value))
        self.set_coeffs(conv=conv, u=u, diff=diff, power=power, b=b, r1=r1, src_family=int(b != 0.0))

    def set_coeffs(self, conv=0, u=(0.05, 0.02), diff=0, power=1, b=0.0, r1=0.0, src_family=0):
        c = C.Coeffs()
        c.conv, c.diff, c.power, c.b, c.r1, c.src_family = conv, diff, power, b, r1, src_family
        c.u[:], c.K[:] = u, (0.02, 0.004, 0.015)
        c.s[:] = (1.0, 1.2, 1.2, 0.0, 1.0, 0.0, 1.0, 1.1, 1.1)
        c.Dm[:] = (1.0, 0.0, 1.0)
        C.check(self.lib.lbm_set_coeffs(self.h, ctypes.byref(c)))

    def route(self, n, sms=152):
        v = (ctypes.c_int * 5)()
        C.check(self.lib.lbm_step_route(self.h, n, sms, v))
        return dict(zip(ROUTE_KEYS, v))

    def __del__(self):
        if getattr(self, "h", None):
            self.lib.lbm_destroy(self.h)


SIZES = [(2, 2), (64, 64), (128, 128), (400, 400), (512, 512), (600, 600), (700, 1000), (1023, 777), (64, 16384),
         (2, 300000), (300000, 5), (128, 16384), (121, 20000), (130, 32768), (4096, 64), (2048, 2048), (4096, 4096)]
KINDS = [dict(prec="f64"), dict(prec="f32"), dict(prec="f32", steps_per_pass=2),
         dict(prec="f32", steps_per_pass=2, kernel_variant=5, block_rows=4), dict(prec="f32", kernel_variant=1),
         dict(prec="f32", per_cell_K=True), dict(prec="f32", per_cell_K=True, steps_per_pass=2), dict(prec="bf16s"),
         dict(prec="bf16s", steps_per_pass=2, kernel_variant=5, block_rows=4),
         dict(prec="f32", scheme="A", bc=("nee", "nee"), conv=2, b=0.02),
         dict(prec="f64", scheme="A", conv=2, b=0.02), dict(prec="f32", diff=3, steps_per_pass=2)]


@pytest.mark.parametrize("kind", KINDS, ids=lambda k: "-".join(f"{a}={b}" for a, b in k.items()))
@pytest.mark.parametrize("walls", [False, True])
def test_routes_add_up_and_keep_the_parity(kind, walls):
    for nx, ny in SIZES:
        kw = dict(kind)
        if "nee" in kw.get("bc", ()) and min(nx, ny) < 3:
            continue
        if walls and "bc" not in kw:
            kw["bc"] = ("abb", "abb")
        s = Lattice(nx, ny, **kw)
        spp = kw.get("steps_per_pass", 1)
        for sms in SMS:
            for n in (0, 1, 2, 3, 4, 5, 6, 7, 8, 12, 20, 23, 100):
                r = s.route(n, sms)
                assert min(r.values()) >= 0, (nx, ny, n, r)
                fixed = 4 * r["fours"] + 2 * (r["pairs"] + r["twos"]) + r["ones"]
                if r["tiles"]:
                    assert fixed == r["ones"] <= 2 and r["tiles"] <= n - r["ones"] <= 8 * r["tiles"], (nx, ny, n, r)
                else:
                    assert fixed == n, (nx, ny, n, r)
                wanted = n // 2 + n % 2 if spp == 2 else n
                assert sum(r.values()) % 2 == wanted % 2, (nx, ny, n, r)


@pytest.mark.parametrize("kw", [dict(nx=20000, ny=12), dict(nx=20000, ny=12, prec="f64"),
                                dict(nx=20000, ny=12, conv=2)], ids=["f32", "f64", "general"])
def test_changed_coefficients_do_not_search_the_tiling_again(kw):
    def least(fn):
        best = float("inf")
        for _ in range(50):
            t = time.perf_counter()
            fn()
            best = min(best, time.perf_counter() - t)
        return best

    s = Lattice(**kw)
    conv = kw.get("conv", 0)
    s.route(10)

    def change():
        s.set_coeffs(conv=conv, u=(0.01, 0.02))
        s.route(10)

    search = least(lambda: Lattice(**kw).route(10)) - least(lambda: Lattice(**kw))
    assert search > 10e-6                                     # what a repeated search would cost
    assert least(change) - least(lambda: s.set_coeffs(conv=conv, u=(0.01, 0.02))) < 0.2 * search


def test_the_benchmark_names_the_kernel_that_runs():
    def name(*a, steps=100, **kw):
        n, kernel, _ = bench.step_kernel(Lattice152(*a, **kw), steps)
        assert n == sum(Lattice(*a, **kw).route(steps).values())
        return kernel.split()[0]

    class Lattice152(Lattice):
        def route(self, n, sms=152):
            return super().route(n, sms)

    assert name(512, 512) == "k_tile"
    assert name(512, 512, per_cell_K=True) == "k_step"
    assert name(4096, 4096, prec="f64") == "k_tile"
    assert name(4096, 4096) == "k_march"
    assert name(4096, 4096, prec="bf16s", steps_per_pass=2, kernel_variant=5, block_rows=4) == "k_step2p"
    assert name(4096, 4096, prec="bf16s") == "k_step_v4"
    assert name(1002, 517, prec="bf16s") == "k_step"


@pytest.mark.parametrize("nx,ny", SIZES)
def test_a_fixed_launch_runs_what_the_descriptor_names(nx, ny):
    named = [(dict(steps_per_pass=2, kernel_variant=5, block_rows=4), "pairs"), (dict(steps_per_pass=2), "twos"),
             (dict(), "ones"), (dict(prec="f64"), "ones"), (dict(conv=2), "ones"), (dict(diff=3, steps_per_pass=2), "twos")]
    for kw, kernel in named:
        s = Lattice(nx, ny, **kw)
        C.check(s.lib.lbm_set_launch_fixed(s.h, 1))
        per = 1 if kernel == "ones" else 2
        assert s.route(20) == dict(dict.fromkeys(ROUTE_KEYS, 0), **{kernel: 20 // per}), kw


# (lattice, descriptor, steps): the kernels that measurements put first (route.cu), and
# what a rule on the node count alone had put in their place
W2 = dict(bc=("abb", "abb"))
P2 = dict(steps_per_pass=2)
MEASURED = [
    (600, 600, {}, 1, "ones"), (64, 64, dict(W2, **P2), 3, "tiles"), (512, 512, {}, 1, "ones"), (64, 64, P2, 1, "ones"),          # not tiles of one step
    (300000, 5, {}, 20, "ones"), (300000, 5, W2, 20, "ones"), (121, 20000, W2, 20, "twos"),  # not pair tiles
    (64, 16384, P2, 2, "twos"), (2, 300000, P2, 20, "twos"),
    (128, 16384, W2, 4, "twos"), (121, 20000, P2, 20, "pairs"), (128, 16384, W2, 400, "fours"),
    (4096, 4096, W2, 400, "fours"), (4096, 4096, P2, 2, "pairs"), (1023, 777, {}, 250, "fours"),
    (450, 450, dict(conv=2, **P2), 20, "twos"), (500, 500, dict(conv=2, **P2), 2, "twos"),
    (350, 350, dict(conv=2, **P2), 20, "tiles"), (450, 450, dict(conv=2), 20, "tiles"),
    (250, 250, dict(conv=2, prec="f64"), 20, "ones"), (200, 200, dict(conv=2, prec="f64"), 20, "tiles"),
    (400, 400, {}, 1000, "tiles"), (128, 128, dict(prec="f64"), 1000, "tiles"), (4096, 4096, dict(prec="f64"), 20, "tiles"),
    (16384, 8192, dict(prec="f64"), 20, "ones")]


@pytest.mark.parametrize("nx,ny,kw,steps,kernel", MEASURED)
@pytest.mark.parametrize("sms", SMS)
def test_the_route_is_the_measured_one(nx, ny, kw, steps, kernel, sms):
    r = Lattice(nx, ny, **kw).route(steps, sms)
    per = dict(tiles=1, fours=4, pairs=2, twos=2, ones=1)
    assert max(r, key=lambda k: r[k] * per[k]) == kernel, r


@pytest.mark.parametrize("sizes,strips", [
    ([(16, 16)] * 4000, False), ([(40, 40)] * 3000, False), ([(20, 1000)] * 300, False),
    ([(16 + i % 49, 16 + (7 * i) % 49) for i in range(3000)], False), ([(2000, 15), (2000, 2000)], False),
    ([(64, 64)] * 1000, True), ([(100, 100)] * 600, True), ([(1000, 20)] * 300, True), ([(500, 500)] * 40, True),
    ([(4096, 4096)], True), ([(1000, 1000)], False)])
def test_ensembles_take_strips_where_they_are_faster(sizes, strips):
    n = len(sizes)
    nx, ny = (ctypes.c_int * n)(*[a for a, _ in sizes]), (ctypes.c_int * n)(*[b for _, b in sizes])
    v = ctypes.c_int(-1)
    assert C.lib().lbm_ensemble_strips(n, nx, ny, ctypes.byref(v)) == C.LBM_OK
    assert (v.value > 0) == strips, v.value
    assert C.lib().lbm_ensemble_strips(n, nx, ny, None) == C.LBM_EINVAL


@pytest.mark.parametrize("size,sweeps", [
    ((256, 256, 256), True), ((64, 64, 1024), True), ((31, 31, 4400), True), ((61, 29, 2400), True), ((240, 210, 96), True),
    ((4096, 512, 2), True), ((96, 15, 3000), False), ((32, 15, 8800), False), ((4096, 2, 512), False), ((128, 128, 128), False)])
def test_d3q19_sweeps_where_they_are_faster(size, sweeps):
    L = C.lib()
    d, n, h, v = C.Desc3(), ctypes.c_size_t(), ctypes.c_void_p(), (ctypes.c_int * 2)()
    d.nx, d.ny, d.nz, d.prec = *size, C.LBM_F32
    C.check(L.lbm3_workspace_size(ctypes.byref(d), ctypes.byref(n)))
    C.check(L.lbm3_create(ctypes.byref(h), ctypes.byref(d), ctypes.c_void_p(1 << 20), n.value))
    for steps in (0, 1, 3, 4, 7, 40):
        C.check(L.lbm3_step_route(h, steps, v))
        assert list(v) == ([steps // 4 * 2, steps % 4] if sweeps else [0, steps])
    L.lbm3_destroy(h)


def test_route_arguments_are_checked():
    s = Lattice(64, 64)
    v = (ctypes.c_int * 5)()
    assert s.lib.lbm_set_launch_fixed(s.h, 2) == C.LBM_EINVAL
    assert s.lib.lbm_set_launch_fixed(None, 1) == C.LBM_EINVAL
    assert s.lib.lbm_step_route(None, 1, 152, v) == C.LBM_EINVAL
    assert s.lib.lbm_step_route(s.h, -1, 152, v) == C.LBM_EINVAL
    assert s.lib.lbm_step_route(s.h, 1, -1, v) == C.LBM_EINVAL
    assert s.lib.lbm_step_route(s.h, 1, 152, None) == C.LBM_EINVAL
    v2, v3 = (ctypes.c_int * 2)(), (ctypes.c_int * 3)()
    assert s.lib.lbm3_step_route(None, 1, v2) == C.LBM_EINVAL
    assert s.lib.lbm_ensemble_step_route(None, 1, 0, v3) == C.LBM_EINVAL
