"""Variable-coefficient kernels with stored face coefficients against the
oracle, where their tiles change: every box size in both dimensions (FP32
boxes of 4 cells per side stay on the kernels that form the coefficients),
coefficients changed on a standing tree, and a jump of 1e6.

Tolerances: FP64 after the same cycles 1e-12, mixed solutions 1e-8."""
import numpy as np
import pytest

from paper_1701_04329_gb300 import afgpu
from tests.gpu_helpers import load, rel_diff
from tests.test_gpu_parity import cycles_parity
from tests.test_gpu_varcoef import var_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,N,uni,extra,op", [(2, 4, 1, 1, 2), (2, 8, 1, 0, 1), (2, 16, 2, 1, 2), (3, 4, 1, 1, 1),
                                              (3, 8, 2, 0, 1), (3, 16, 1, 1, 1),
                                              # levels in the coarse launch, up to grids spread over its blocks
                                              (2, 8, 4, 1, 1), (2, 8, 5, 0, 2), (2, 16, 3, 0, 2), (2, 4, 4, 1, 1),
                                              (3, 4, 3, 0, 1), (3, 8, 3, 0, 1), (2, 8, 1, 0, 2)])
def test_cycles(D, N, uni, extra, op):
    a, b, rho, bv, _ = var_pair(D, N, uni, extra, 900 + N + D, op)
    load(a, b, rho, bv)
    cycles_parity(a, b, 2)


def test_new_coefficients_and_a_large_jump():
    a, b, rho, bv, eps = var_pair(2, 8, 2, 1, 930, 1)
    load(a, b, rho, bv)
    cycles_parity(a, b, 1)
    x = a.cell_centers()
    for e in (eps[::-1].copy(), np.where((x < 0.5).all(1), 1e6, 1.0)):
        a.set_eps(e)
        b.set_eps(torch.tensor(e, device="cuda"))
        load(a, b, rho, bv)
        cycles_parity(a, b, 1)


@pytest.mark.parametrize("D,N,uni,extra,op", [(2, 4, 2, 1, 1), (3, 4, 2, 1, 1), (2, 16, 1, 1, 2), (3, 16, 1, 0, 1),
                                              (2, 8, 5, 0, 2), (3, 8, 2, 1, 1)])
def test_mixed(D, N, uni, extra, op):
    a, b, rho, bv, _ = var_pair(D, N, uni, extra, 940 + N + D, op, cells=2, lo=0.5, hi=4.0)
    load(a, b, rho, 1e-3 * bv)
    a.solve(1e-12, 80)
    st = b.solve(afgpu.default_opts(rel_tol=1e-10, precision=afgpu.AFG_MIXED, max_cycles=60))
    assert st["rel_residual"] <= 1e-10
    assert rel_diff(b.get_solution(), a.get_solution()) <= 1e-8
