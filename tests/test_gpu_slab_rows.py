"""The x passes of the slab matvec (kx-major tiles) at every padded row length:
plain products against the pairwise oracle, and refined solves, whose gathers
and scatters carry the Krylov updates, against FP64 solves.  Tile stride,
launch bounds and radix plan differ per length.  The lattices' rows with sites
fill no whole tile of the x-inverse, and some rows hold no site."""
import numpy as np
import pytest

from dda_inputs import random_complex
from oracle import dda as oracle, pairwise
from test_gpu_pass_choice import SLAB, traced

pytestmark = pytest.mark.gpu

F32_TOL = 1e-5      # complex64 against the oracle, the tolerance of the other matvec tests
Q_TOL = 1e-5        # efficiencies of a solve to 1e-6 against FP64, that of the other refined solves
LX = {16: 7, 32: 13, 48: 22, 64: 31, 96: 47, 128: 61, 192: 95, 256: 120, 384: 181, 512: 250}
M = np.array([1.6 + 0.1j, 1.3 + 0.02j])


@pytest.fixture(scope="module")
def lib():
    import paper_1202_3424_gb300 as dda
    dda.load_library()
    return dda


def _grid(nx):
    """A 5x3-row bar of two materials, one site in eight left out and two rows empty."""
    rng = np.random.default_rng(nx)
    g = rng.integers(1, 3, (3, 5, nx)).astype(np.uint8)
    g[rng.random(g.shape) < 0.125] = 0
    g[1, 2] = g[2, 4] = 0
    g[0, 0, 0] = g[2, 3, -1] = 1
    return g


def _prepared(lib, nx, site):
    grid = _grid(nx)
    ctx = lib.Context(0)
    ctx.set_target(grid)
    if site:
        ctx.set_site_materials(M[grid[grid > 0].astype(int) - 1])
    else:
        ctx.set_materials(M)
    ctx.prepare_size_parameter(1.5, lib.Precision.FP32_REFINED)
    ctx.set_slab_pass(1)
    return grid, ctx


def _waves(R):
    rng = np.random.default_rng(R)
    k = rng.standard_normal((R, 3))
    k /= np.linalg.norm(k, axis=1)[:, None]
    e = np.cross(k, [0.0, 0.0, 1.0])
    return k, (e / np.linalg.norm(e, axis=1)[:, None]).astype(complex)


@pytest.mark.parametrize("site", [False, True], ids=["compositions", "sites"])
@pytest.mark.parametrize("Lx", sorted(LX))
def test_slab_rows_match_oracle(lib, Lx, site):
    grid, ctx = _prepared(lib, LX[Lx], site)
    info = ctx.info()
    assert (info["Lx"], info["Ly"], info["Lz"]) == (Lx, 16, 16)
    R = 5
    k, e = _waves(R)
    X = random_complex((R, 3, info["ndipoles"]), 3)
    with traced(lib, ctx) as t:
        Y = ctx.matvec(2, k, e, X)
    assert SLAB <= set(t.kernels)
    rr, comp = oracle.site_positions(grid)
    for r in range(R):
        beta = oracle.ldr_inverse_polarizability(M[comp - 1] ** 2, info["kd"], k[r], e[r])
        want = pairwise.matvec(rr, info["kd"], beta, X[r].T)[0]
        assert np.abs(Y[r].T - want).max() < F32_TOL * np.abs(want).max(), r
    ctx.close()


@pytest.mark.parametrize("site", [False, True], ids=["compositions", "sites"])
@pytest.mark.parametrize("solver", ["bicgstab", "bicgstab2", "qmr"])
@pytest.mark.parametrize("Lx", sorted(LX))
def test_refined_solve_through_slab_rows(lib, Lx, solver, site):
    _, ctx = _prepared(lib, LX[Lx], site)
    k, e = _waves(3)
    ref, P0, st = ctx.solve(lib.Precision.FP64, k, e, tol=1e-10, maxit=2000)
    assert st == 0
    with traced(lib, ctx) as t:
        res, P, st = ctx.solve(lib.Precision.FP32_REFINED, k, e, tol=1e-6, maxit=2000, solver=solver)
    assert st == 0 and max(r["resid_rel"] for r in res) <= 1e-6
    assert SLAB <= set(t.kernels) and "z_conv_c64" not in t.kernels
    q, q0 = (np.array([[r["qext"], r["qabs"], r["qsca"]] for r in s]) for s in (res, ref))
    assert np.abs(q - q0).max() < Q_TOL * np.abs(q0).max()
    ctx.close()
