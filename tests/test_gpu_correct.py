"""Coarse-grid correction with several parents per block (2D boxes of 4 and 8
cells per side): refined parents on a level in numbers below, at and beyond a
block's share, and not a multiple of it.

Tolerances: FP64 after the same cycles 1e-12, mixed solutions 1e-8.  Boundary
data of 1e-3 keep the FP64 round-off of the residual (4 |u| eps / h^2, h = 1/256)
two decades below the mixed solve's 1e-10."""
import numpy as np
import pytest

from oracle.oracle import OracleTree
from paper_1701_04329_gb300 import afgpu
from tests.gpu_helpers import load, rel_diff
from tests.test_gpu_parity import cycles_parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def pair_with_parents(N, level, parents):
    """Uniform to `level`, then `parents` separate boxes of that level refined."""
    a, b = OracleTree(2, N, level + 1), afgpu.Tree(2, N, level + 1)
    for t in (a, b):
        t.refine_uniform(level)
    flags = np.zeros(a.n_leaf_cells, dtype=np.int8)
    boxes = a.n_leaf_cells // (N * N)
    pick = np.linspace(0, boxes - 1, parents).astype(int)
    inner = (N // 2) * N + N // 2  # away from the sides, so that no neighbour is refined with it
    flags[pick * N * N + inner] = 1
    for t in (a, b):
        t.adapt(flags, 0)
    assert a.n_leaf_cells == b.n_leaf_cells
    x = a.cell_centers()
    return a, b, np.sin(9 * x[:, 0]) * np.cos(7 * x[:, 1]), 1e-3 * np.linspace(-1, 1, b.n_bfaces)


@pytest.mark.parametrize("N", [4, 8])
@pytest.mark.parametrize("parents", [1, 3, 4, 5, 9, 17])
def test_parents_per_block(N, parents):
    a, b, rho, bv = pair_with_parents(N, 5, parents)
    load(a, b, rho, bv)
    cycles_parity(a, b, 2)
    load(a, b, rho, bv)
    a.solve(1e-12, 60)
    st = b.solve(afgpu.default_opts(rel_tol=1e-10, precision=afgpu.AFG_MIXED))
    assert st["rel_residual"] <= 1e-10
    assert rel_diff(b.get_solution(), a.get_solution()) <= 1e-8


@pytest.mark.parametrize("parents", [304, 305, 307, 330])
def test_levels_of_many_boxes(parents):
    """Levels of 1216 boxes (a warp per box in the restriction) and just above
    (two boxes per warp), also in numbers that leave blocks of 16 partly empty."""
    a, b, rho, bv = pair_with_parents(8, 6, parents)
    load(a, b, rho, bv)
    cycles_parity(a, b, 2)
    load(a, b, rho, bv)
    a.solve(1e-12, 60)
    st = b.solve(afgpu.default_opts(rel_tol=1e-10, precision=afgpu.AFG_MIXED))
    assert st["rel_residual"] <= 1e-10
    assert rel_diff(b.get_solution(), a.get_solution()) <= 1e-8
