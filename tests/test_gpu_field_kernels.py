"""Edges of the far-field sums and of the per-site tables, which other tests reach at one size each."""
import math

import numpy as np
import pytest

from dda_inputs import block_bernoulli_grid, random_complex
from oracle import dda as odda

pytestmark = pytest.mark.gpu

F64_TOL, F32_TOL = 1e-10, 1e-5     # the far field's tolerances against the oracle
TABLE_TOL = 1e-13                  # two ways to the same FP64 1/alpha: a few ulps of a few operations


@pytest.fixture(scope="module")
def lib():
    import paper_1202_3424_gb300 as dda
    dda.load_library()
    return dda


@pytest.mark.parametrize("prec,tol", [(0, F64_TOL), (2, F32_TOL)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("paired", [True, False], ids=["both_polarizations", "single"])
@pytest.mark.parametrize("nx,ny,nz,ndir", [(1, 1, 1, 1), (33, 5, 3, 63), (97, 3, 2, 129), (120, 2, 2, 65)],
                         ids=["one_site", "row33", "row97", "row120"])
def test_farfield_tiles_match_oracle(lib, nx, ny, nz, ndir, paired, prec, tol):
    """Rows longer than a warp's staging, two and four directions a lane (the
    switch lies between 97 and 120 sites a row), a direction past a tile's end,
    and right-hand sides that share their directions or do not."""
    rng = np.random.default_rng(nx + ndir)
    grid = (rng.random((nz, ny, nx)) < 0.7).astype(np.uint8)
    grid[0, 0, 0] = grid[-1, -1, -1] = 1
    ctx = lib.Context(0)
    ctx.set_target(grid)
    ctx.set_materials([1.5 + 0.1j])
    ctx.prepare_size_parameter(1.5, lib.Precision.FP32_REFINED)
    kd, n = ctx.info()["kd"], ctx.info()["ndipoles"]
    khat = np.array([[0.36, 0.48, 0.8], [0.36, 0.48, 0.8] if paired else [1.0, 0.0, 0.0]])
    P = random_complex((2, 3, n), 31)
    theta, phi = rng.uniform(0, math.pi, ndir), rng.uniform(0, 2 * math.pi, ndir)
    F = ctx.farfield(prec, khat, P, theta, phi)
    r, _ = odda.site_positions(grid)
    for q in range(2):
        want = odda.far_field(r, P[q].T, kd, odda.directions(khat[q], theta, phi))
        # the sums of the two right-hand sides are of one size: a tolerance relative to the larger
        assert np.abs(F[q] - want).max() < tol * kd ** 2 * np.abs(P[q]).sum(), (q,)
    ctx.close()


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (5, 51, 1), (4, 8, 8)], ids=["1", "255", "256"])
def test_site_tables_match_composition_tables(lib, nx, ny, nz):
    """1/alpha formed on the device, one entry per site, against the host's
    table of two compositions, in all three arithmetics."""
    grid = block_bernoulli_grid(nx, ny, nz, seed=5)
    m = np.array([1.5 + 0.1j, 2.0 + 1.5j])
    n = int(np.count_nonzero(grid))
    k = np.array([[0.36, 0.48, 0.8]] * 3)
    e = np.array([[0.8, -0.6, 0.0], [0.48, 0.64, -0.6], [0.8, -0.6, 0.0]], dtype=complex)
    X = random_complex((3, 3, n), 9)
    out = []
    for site in (False, True):
        ctx = lib.Context(0)
        ctx.set_target(grid)
        if site:
            ctx.set_site_materials(m[grid[grid > 0].astype(int) - 1], 1.1)
        else:
            ctx.set_materials(m, 1.1)
        ctx.prepare_size_parameter(0.7, lib.Precision.FP32_REFINED)
        out.append([ctx.matvec(p, k, e, X) for p in (0, 2, 3)])
        ctx.close()
    for a, b, tol in zip(*out, (TABLE_TOL, F32_TOL, TABLE_TOL)):
        assert np.abs(a - b).max() <= tol * np.abs(a).max()
