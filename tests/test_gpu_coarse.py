"""The coarse launch against the oracle: levels that cover the domain, from
the root box alone to grids spread over a cluster's blocks, with every kind
of side, blocks of root boxes, leaves on the launch's top level, and forests.

Tolerances: FP64 after the same cycles 1e-12, mixed solutions 1e-8 (the bars
of the other parity tests)."""
import numpy as np
import pytest

from oracle.oracle import OracleTree
from paper_1701_04329_gb300 import afgpu
from tests.gpu_helpers import load, rel_diff
from tests.test_gpu_parity import cycles_parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def pair(D, N, uniform, types=None, roots=None, extra=0, seed=0):
    rng = np.random.default_rng(seed)
    a = OracleTree(D, N, uniform + extra, roots=roots) if roots else OracleTree(D, N, uniform + extra)
    b = afgpu.Tree(D, N, uniform + extra, roots=roots)
    for t in (a, b):
        if types:
            t.set_boundary_types(types)
        t.refine_uniform(uniform)
    for _ in range(extra):  # some boxes of the top level stay leaves
        flags = np.repeat((rng.random(a.nleaf) < 0.3).astype(np.int8), N ** D)
        a.adapt(flags, 1)
        b.adapt(flags, 1)
    x = a.cell_centers()
    rho = np.sin(5 * x[:, 0] + 1) * np.cos(3 * x[:, 1]) + rng.normal(scale=0.1, size=len(x))
    return a, b, rho, rng.normal(size=a.n_bfaces)


@pytest.mark.parametrize("D,N,uniform,extra,types,roots", [
    (2, 4, 1, 0, None, None), (2, 4, 5, 0, None, None), (2, 8, 4, 0, [0, 1, 2, 2], None), (2, 8, 5, 1, None, None),
    (2, 16, 3, 1, [1, 0, 0, 1], None), (3, 4, 3, 0, [2, 2, 0, 1, 0, 0], None), (3, 8, 2, 1, None, None),
    (3, 16, 1, 0, [0, 0, 1, 0, 2, 2], None), (3, 16, 1, 1, None, None), (2, 8, 3, 1, None, (3, 2)),
    (2, 8, 4, 0, [0, 0, 2, 2], (1, 3)), (3, 8, 2, 0, [0, 0, 2, 2, 0, 1], (2, 1, 1))])
def test_cycle_by_cycle(D, N, uniform, extra, types, roots):
    a, b, rho, bv = pair(D, N, uniform, types, roots, extra)
    load(a, b, rho, bv)
    cycles_parity(a, b, 2)


@pytest.mark.parametrize("D,N,uniform,extra", [(2, 8, 6, 1), (3, 8, 3, 1), (3, 4, 4, 0), (2, 16, 1, 0)])
def test_mixed(D, N, uniform, extra):
    a, b, rho, bv = pair(D, N, uniform, extra=extra, seed=3)
    load(a, b, rho, bv)
    a.solve(1e-12, 60)
    # the FP64 residual cannot be told from its own rounding below about 2D |u| / h^2 times 2^-53
    h = 1.0 / (N * 2.0 ** (uniform + extra - 1))
    floor = 4 * 2 * D * np.abs(a.get_solution()).max() / h ** 2 * 2.0 ** -53 / np.abs(rho).max()
    tol = max(1e-11, floor)
    st = b.solve(afgpu.default_opts(rel_tol=tol, precision=afgpu.AFG_MIXED))
    assert st["rel_residual"] <= tol
    assert rel_diff(b.get_solution(), a.get_solution()) <= 1e-8


def test_boundary_data_changes_reach_the_coarse_levels():
    a, b, rho, bv = pair(2, 8, 4, seed=5)
    load(a, b, rho, bv)
    cycles_parity(a, b, 1)
    for scale in (0.0, -2.5):  # new data on the same tree, the cycles' graphs standing
        load(a, b, rho, scale * bv)
        cycles_parity(a, b, 1)


def test_forest_of_uneven_trees():
    specs = [(2, 2), (2, 0), (2, 1)]
    pairs = [pair(2, 8, u, [0, 0, 2, 2] if k == 1 else None, None, e, seed=10 + k) for k, (u, e) in enumerate(specs)]
    f = afgpu.Forest([p[1] for p in pairs])
    f.set_rhs(torch.tensor(np.concatenate([p[2] for p in pairs]), device="cuda"))
    f.set_dirichlet(torch.tensor(np.concatenate([p[3] for p in pairs]), device="cuda"))
    st = f.solve(afgpu.default_opts(rel_tol=1e-10))
    u, off = f.get_solution().cpu().numpy(), 0
    for k, (a, _, rho, bv) in enumerate(pairs):
        a.set_rhs(rho)
        a.set_dirichlet(bv)
        a.zero_solution()
        assert st[k]["cycles"] == a.solve(1e-10, 60)
        n = a.n_leaf_cells
        assert rel_diff(u[off:off + n], a.get_solution()) <= 1e-12
        off += n
