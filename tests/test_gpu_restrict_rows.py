"""FP32 residual + restriction by rows (3D boxes of 8 and 16 cells per side:
one and two vectors per half-row) inside mixed solves, on uniform and refined
trees.

The solution is within 1e-8 of the oracle's FP64 solution.  The restriction
carries the defect down, so a wrong one shows in the count of steps: two V-cycles
(a factor of 10 each, at least, with Dirichlet sides) reduce the residual
100-fold per step, so 1e-10 is reached within six steps (the first is an FMG cycle)."""
import pytest

from paper_1701_04329_gb300 import afgpu
from tests.gpu_helpers import load, pair_random, rel_diff

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,uni,extra", [(8, 3, 0), (8, 2, 2), (8, 4, 0), (16, 2, 0), (16, 2, 1)])
def test_mixed_3d(N, uni, extra):
    a, b, rho, bv = pair_random(3, N, uni, extra, 91 + N)
    load(a, b, rho, 1e-3 * bv)
    a.solve(1e-12, 60)
    st = b.solve(afgpu.default_opts(rel_tol=1e-10, precision=afgpu.AFG_MIXED))
    assert st["rel_residual"] <= 1e-10
    assert st["cycles"] <= 6
    assert rel_diff(b.get_solution(), a.get_solution()) <= 1e-8
