"""Which passes a complex64 matvec runs, and what launch tracing says of them."""
import ctypes

import numpy as np
import pytest

from dda_inputs import random_complex, sphere_grid

pytestmark = pytest.mark.gpu

SEPARATE = {"x_fwd_c64", "y_fwd_c64", "z_conv_c64", "y_inv_c64", "x_inv_c64"}
SLAB = {"x_fwd_c64", "slab_c64", "x_inv_c64"}
K1, E1 = np.array([[0.6, 0.0, 0.8]]), np.array([[0.0, 1.0, 0.0]], dtype=complex)


@pytest.fixture(scope="module")
def lib():
    import paper_1202_3424_gb300 as dda
    dda.load_library()
    return dda


class Stat(ctypes.Structure):
    _fields_ = [("name", ctypes.c_char * 24), ("launches", ctypes.c_int64), ("total_ms", ctypes.c_double),
                ("units", ctypes.c_double)]


def _read(lib, ctx, name):
    """{kind: (launches, ms, units)} by dda_profile_read or dda_profile_kernels."""
    f = getattr(lib.load_library(), name)
    f.argtypes = [ctypes.c_void_p, ctypes.POINTER(Stat), ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    arr, n = (Stat * 64)(), ctypes.c_int()
    assert f(ctx.handle, arr, 64, ctypes.byref(n)) == 0
    return {arr[i].name.decode(): (arr[i].launches, arr[i].total_ms, arr[i].units) for i in range(n.value)}


class traced:
    def __init__(self, lib, ctx):
        self.lib, self.ctx = lib, ctx

    def __enter__(self):
        assert self.lib.load_library().dda_profile_enable(self.ctx.handle, 1) == 0
        return self

    def __exit__(self, *exc):
        self.kernels = _read(self.lib, self.ctx, "dda_profile_kernels")
        self.passes = _read(self.lib, self.ctx, "dda_profile_read")
        self.lib.load_library().dda_profile_enable(self.ctx.handle, 0)


def _ctx(lib, grid, m=1.5 + 0.1j, x=1.0):
    ctx = lib.Context(0)
    ctx.set_target(grid)
    ctx.set_materials([m])
    ctx.prepare_size_parameter(x, lib.Precision.FP32_REFINED)
    return ctx


def _rhs(R):
    return np.tile(K1, (R, 1)), np.tile(E1, (R, 1))


def test_tracing_by_kernel_and_by_pass(lib):
    """A product through the slab pass and one through the separate passes in
    one trace: each kernel once under its own name, each pass once per product,
    the same total time both ways."""
    ctx = _ctx(lib, sphere_grid(12))
    k, e = _rhs(2)
    X = random_complex((2, 3, ctx.info()["ndipoles"]), 3)
    with traced(lib, ctx) as t:
        ctx.matvec(2, k, e, X)
    assert {n: v[0] for n, v in t.kernels.items() if n.endswith("c64")} == dict.fromkeys(SLAB, 1)
    assert {n: v[0] for n, v in t.passes.items() if n.endswith("c64")} == dict.fromkeys(SEPARATE, 1)
    slab_ms = t.kernels["slab_c64"][1]
    assert slab_ms > 0 and t.passes["z_conv_c64"][1] == slab_ms
    assert t.passes["y_fwd_c64"][1] == t.passes["y_inv_c64"][1] == 0
    with traced(lib, ctx) as t:
        ctx.matvec(2, k, e, X)
        ctx.set_schedule(0)
        ctx.matvec(2, k, e, X)
    for name in SEPARATE | SLAB:
        once = 2 if name in SEPARATE & SLAB else 1
        assert t.kernels[name][0] == once and t.kernels[name][2] == 2 * once, name
    for name in SEPARATE:
        assert t.passes[name][0] == 2 and t.passes[name][2] == 4, name
    assert "slab_c64" not in t.passes
    total = [sum(v[1] for v in s.values()) for s in (t.kernels, t.passes)]
    assert total[0] == pytest.approx(total[1], rel=1e-12)
    ctx.close()


def _runs_slab(lib, ctx, R):
    """Whether the kernels of a product of R right-hand sides are the slab pass's; the query has to agree."""
    k, e = _rhs(R)
    X = random_complex((R, 3, ctx.info()["ndipoles"]), 3)
    with traced(lib, ctx) as t:
        ctx.matvec(2, k, e, X)
    ran = {n for n in t.kernels if n.endswith("c64")}
    assert ran in (SLAB, SEPARATE)
    assert ctx.get_slab_pass(R) == (ran == SLAB)
    return ran == SLAB


def test_slab_pass_is_asked_for_refused_and_queried(lib):
    """The setter against every other setter, and back to the rule; what the
    query reports pins the automatic choice, bit for bit."""
    ctx = _ctx(lib, sphere_grid(12))
    k, e = _rhs(2)
    X = random_complex((2, 3, ctx.info()["ndipoles"]), 3)
    assert _runs_slab(lib, ctx, 2)
    auto = ctx.matvec(2, k, e, X)
    ctx.set_slab_pass(0)
    assert not _runs_slab(lib, ctx, 2)
    ctx.set_slab_pass(-1)
    for setter, value, default in ((ctx.set_schedule, 0, -1), (ctx.set_xpass, 0, -1), (ctx.set_ypass, 0, -1),
                                   (ctx.set_slice_passes, -1, 0)):
        setter(value)
        assert not ctx.get_slab_pass(2)
        ctx.set_slab_pass(1)
        assert _runs_slab(lib, ctx, 2)
        ctx.set_slab_pass(-1)
        setter(default)
        assert ctx.get_slab_pass(2)
    # pinned, with the separate passes' schedules pinned after it
    ctx.set_slab_pass(ctx.get_slab_pass(2))
    ctx.set_schedule(ctx.get_schedule(2))
    ctx.set_xpass(ctx.get_xpass(2))
    ctx.set_ypass(ctx.get_ypass(2))
    assert np.array_equal(ctx.matvec(2, k, e, X), auto)
    for bad in (-2, 2):
        with pytest.raises(lib.DdaError):
            ctx.set_slab_pass(bad)
    ctx.close()


def test_slab_pass_where_it_is_not_built(lib):
    """Asked for, it still leaves long axes, tilted crystals and the other
    arithmetics to the separate passes."""
    ctx = _ctx(lib, np.ones((2, 70, 2), np.uint8))     # Ly = 192
    ctx.set_slab_pass(1)
    assert not _runs_slab(lib, ctx, 2)
    ctx.set_target(sphere_grid(12))
    ctx.set_anisotropic_materials([[1.5, 1.6, 1.4]], [(0.4, 1.1, -0.6)])
    ctx.prepare_size_parameter(1.0, lib.Precision.FP32_REFINED)
    assert not _runs_slab(lib, ctx, 2)
    ctx.set_materials([1.5 + 0.1j])
    with pytest.raises(lib.DdaError):
        ctx.get_slab_pass(2)                            # not prepared
    ctx.prepare_size_parameter(1.0, lib.Precision.FP64)
    with pytest.raises(lib.DdaError):
        ctx.get_slab_pass(2)                            # no complex64 tensor
    ctx.close()


def test_refined_solves_stop_alike_on_either_passes(lib):
    """Inner solves stop at a third of the tolerance (QMR, where it makes no
    progress, at half), whichever passes run: the true residual exceeds that by
    the drift of the FP32 recurrence alone (some sixty products, 2^-24 each, of
    a solution of the incident field's size: 4e-6)."""
    ctx = _ctx(lib, sphere_grid(24), 1.5 + 0.02j, 3.0)
    rng = np.random.default_rng(2)
    k = rng.standard_normal((16, 3))
    k /= np.linalg.norm(k, axis=1)[:, None]
    e = np.cross(k, [0.0, 0.0, 1.0])
    e = (e / np.linalg.norm(e, axis=1)[:, None]).astype(complex)
    tol = 1e-4
    for on in (0, 1):
        ctx.set_slab_pass(on)
        for solver in ("bicgstab", "bicgstab2", "qmr"):
            res, _, st = ctx.solve(lib.Precision.FP32_REFINED, k, e, want_P=False, tol=tol, maxit=400, solver=solver)
            assert st == 0
            share = 1 / 2 if solver == "qmr" else 1 / 3
            assert max(r["resid_rel"] for r in res) <= share * tol + 4e-6, (on, solver)
    ctx.close()


def test_qmr_does_not_stall_below_half_the_tolerance(lib):
    """QMR's residual levels out above the third of the tolerance that inner
    solves aim at, for one direction in four here.  Below the half, waiting 40
    iterations for a new minimum buys nothing: what is left are the few that
    level out above it (iterations of an unhindered solve: 51 to 63)."""
    u = ((np.arange(64) - 31.5) / 64) ** 2
    ctx = _ctx(lib, (u[:, None, None] + u[None, :, None] + u[None, None, :] <= 0.25).astype(np.uint8), 1.5 + 0.02j, 5.0)
    rng = np.random.default_rng(1)
    iters = []
    for _ in range(40):
        k = rng.standard_normal(3)
        k /= np.linalg.norm(k)
        a = np.cross([0.0, 0.0, 1.0], k)
        a /= np.linalg.norm(a)
        res, _, st = ctx.solve(lib.Precision.FP32_REFINED, np.stack([k, k]), np.stack([a, np.cross(k, a)]).astype(complex),
                               want_P=False, tol=1e-5, maxit=2000, solver="qmr")
        assert st == 0
        iters.append(max(r["iters"] for r in res))
    assert sum(i > 80 for i in iters) <= 4, sorted(iters)
    ctx.close()


# (lattice, R, plain products, solves): both sides of every line of the rule
RULE = [
    ((16, 24, 24), 1, True, True),       # 32 slabs of 48 x 48
    ((16, 48, 24), 1, True, False),      # of 96 x 48: a solve's lost 5 %
    ((16, 48, 24), 2, True, True),
    ((16, 64, 48), 1, False, False),     # of 128 x 96
    ((16, 64, 48), 2, True, True),
    ((24, 48, 48), 1, True, False),      # 48 slabs of 96 x 96: a solve's lost 10 %
    ((24, 48, 24), 1, True, True),
    ((24, 48, 48), 2, True, True),
    ((64, 16, 24), 8, False, False),     # 1024 slabs of 32 x 48
    ((64, 16, 24), 7, True, True),
    ((64, 24, 24), 8, True, True),
    ((48, 16, 16), 12, True, True),      # 96 points along x
]


@pytest.mark.parametrize("n,R,plain,solve", RULE, ids=["x".join(map(str, c[0])) + f"_R{c[1]}" for c in RULE])
def test_rule_decides_which_passes_run(lib, n, R, plain, solve):
    """The kernels that run are those the rule names, in a product and in a
    solve, and agree with the other passes' to the complex64 tolerance."""
    grid = np.zeros(n[::-1], np.uint8)
    grid[:3, :3, :3] = grid[-3:, -3:, -3:] = 1
    ctx = _ctx(lib, grid, 1.5 + 0.05j)
    assert (ctx.get_slab_pass(R), ctx.get_slab_pass(R, solve=True)) == (plain, solve)
    assert _runs_slab(lib, ctx, R) == plain
    k, e = _rhs(R)
    X = random_complex((R, 3, ctx.info()["ndipoles"]), 3)
    auto = ctx.matvec(2, k, e, X)
    for solver in ("bicgstab", "bicgstab2", "qmr"):
        with traced(lib, ctx) as t:
            _, P, st = ctx.solve(lib.Precision.FP32_REFINED, k, e, tol=1e-6, solver=solver)
        assert st == 0
        assert ("slab_c64" in t.kernels, "z_conv_c64" in t.kernels) == (solve, not solve)
    ctx.set_slab_pass(int(not plain))
    other = ctx.matvec(2, k, e, X)
    assert np.abs(auto - other).max() < 1e-5 * np.abs(other).max()
    ctx.close()


def _device_bytes(f):
    import torch
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    f()
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0]


def test_slab_tensor_is_kept_only_where_it_can_be_used(lib):
    """The slab pass's copy of the Green tensor (26 MB for a 64^3 lattice) is
    made for targets and schedules that can take the pass, and at the first
    product where a setter makes a place for it later."""
    grid = sphere_grid(64)
    size = (65 * 64 * 128 * 3 + 65 * 128 * 3) * 16

    def prepared(aniso, schedule):
        ctx = lib.Context(0)
        ctx.set_target(grid)
        if aniso:
            ctx.set_anisotropic_materials([[1.5, 1.6, 1.4]], [(0.4, 1.1, -0.6)])
        else:
            ctx.set_materials([1.5 + 0.1j])
        ctx.set_schedule(schedule)
        return ctx, _device_bytes(lambda: ctx.prepare_size_parameter(1.0, lib.Precision.FP32_REFINED))

    prepared(False, -1)[0].close()                       # (modules loaded)
    (iso, b_iso), (crystal, b_crystal), (forced, b_forced) = (prepared(*a) for a in ((False, -1), (True, -1), (False, 0)))
    slack = 4 << 20                                      # the allocator's granularity
    assert b_iso - b_crystal > size - slack and b_iso - b_forced > size - slack
    k, e = _rhs(1)
    X = random_complex((1, 3, iso.info()["ndipoles"]), 3)
    before = forced.matvec(2, k, e, X)
    forced.set_schedule(-1)
    assert _runs_slab(lib, forced, 1)
    after = forced.matvec(2, k, e, X)
    assert np.array_equal(after, iso.matvec(2, k, e, X)) and not np.array_equal(after, before)
    # another wavelength: the copy is the new one's
    for ctx in (forced, iso):
        ctx.prepare_size_parameter(2.0, lib.Precision.FP32_REFINED)
    forced.set_slab_pass(0)
    want = forced.matvec(2, k, e, X)
    assert np.abs(iso.matvec(2, k, e, X) - want).max() < 1e-5 * np.abs(want).max()
    for ctx in (iso, crystal, forced):
        ctx.close()


def test_no_allocation_product_after_a_schedule_was_forced(lib):
    """A product that may not allocate takes the slab pass once its copy of the
    tensor is there, and the separate passes until then."""
    import torch
    ctx = lib.Context(0)
    ctx.set_target(sphere_grid(12))
    ctx.set_materials([1.5 + 0.1j])
    ctx.set_schedule(0)
    ctx.prepare_size_parameter(1.0, lib.Precision.FP32_REFINED)
    ctx.set_schedule(-1)
    k, e = _rhs(2)
    x = torch.from_numpy(random_complex((2, 3, ctx.info()["ndipoles"]), 3).astype(np.complex64)).cuda()
    y0, y1, slab = (torch.empty_like(x) for _ in range(3))
    torch.cuda.synchronize()
    lib.dda_matvec_device_noalloc(ctx.handle, 2, k, e, x, y0)
    assert ctx.get_slab_pass(2)                         # makes the copy
    lib.dda_matvec_device_noalloc(ctx.handle, 2, k, e, x, y1)
    lib.dda_matvec_device(ctx.handle, 2, k, e, x, slab)
    y0, y1, slab = (y.cpu().numpy() for y in (y0, y1, slab))
    assert np.array_equal(y1, slab) and not np.array_equal(y0, slab)
    assert np.abs(y0 - y1).max() < 1e-5 * np.abs(y0).max()
    ctx.close()
