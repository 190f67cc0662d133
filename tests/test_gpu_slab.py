"""The slab pass (y and z transforms in one kernel) against the pairwise oracle.

It runs whenever no schedule of the separate passes is forced and both padded
lengths are at most 128 points.  Every pair of a y and a z length, on lattices
of few clustered sites (the oracle's cost) that reach the first and last row,
column and plane; one RHS (a block per SM) and enough for the small blocks.
"""
import numpy as np
import pytest

from dda_inputs import random_complex
from oracle import dda as oracle, pairwise

pytestmark = pytest.mark.gpu

F32_TOL = 1e-5      # complex64 against the oracle, the tolerance of the other matvec tests
HALF = {16: 7, 32: 15, 48: 23, 64: 31, 96: 47, 128: 63}   # odd sides just inside each padded length


@pytest.fixture(scope="module")
def lib():
    import paper_1202_3424_gb300 as dda
    dda.load_library()
    return dda


def _clusters(nx, ny, nz, seed):
    """3x3x3 clusters (neighbours' terms as large as the diagonal) at the corners and at random places."""
    rng = np.random.default_rng(seed)
    g = np.zeros((nz, ny, nx), np.uint8)
    at = [(0, 0, 0), (nx - 3, ny - 3, nz - 3), (0, ny - 3, 0), (nx - 3, 0, nz - 3)]
    at += [tuple(int(rng.integers(0, n - 2)) for n in (nx, ny, nz)) for _ in range(6)]
    for x, y, z in at:
        g[z:z + 3, y:y + 3, x:x + 3] = 1
    return g


@pytest.mark.parametrize("Lz", sorted(HALF))
@pytest.mark.parametrize("Ly", sorted(HALF))
def test_slab_matvec_matches_oracle(lib, Ly, Lz):
    grid = _clusters(20, HALF[Ly], HALF[Lz], 7 * Ly + Lz)
    ctx = lib.Context(0)
    ctx.set_target(grid)
    ctx.set_materials([2.0 + 0.5j])
    ctx.prepare_size_parameter(1.0, lib.Precision.FP32_REFINED)
    info = ctx.info()
    assert (info["Ly"], info["Lz"]) == (Ly, Lz)
    kd = info["kd"]
    k, e = np.array([[0.6, 0.0, 0.8]]), np.array([[0.0, 1.0, 0.0]], dtype=complex)
    rr, comp = oracle.site_positions(grid)
    beta = oracle.ldr_inverse_polarizability(np.full(comp.shape, (2.0 + 0.5j) ** 2), kd, k[0], e[0])
    X = random_complex((12, 3, info["ndipoles"]), 3)
    one = ctx.matvec(2, k, e, X[:1])                       # 48 slabs: one block per SM
    many = ctx.matvec(2, np.tile(k, (12, 1)), np.tile(e, (12, 1)), X)
    want = pairwise.matvec(rr, kd, beta, X[0].T)[0]
    scale = np.abs(want).max()
    assert np.abs(one[0].T - want).max() < F32_TOL * scale
    assert np.abs(many[0].T - want).max() < F32_TOL * scale
    # the other right-hand sides against the separate passes
    ctx.set_schedule(0)
    rest = ctx.matvec(2, np.tile(k, (12, 1)), np.tile(e, (12, 1)), X)
    assert np.abs(many - rest).max() < F32_TOL * np.abs(rest).max()
    ctx.close()
