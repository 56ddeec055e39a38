"""FP64 kernels on aligned images (3D, and the 2D residual of mixed solves)
where the alignment can go wrong: boxes of 4, 8 and 16 cells per side, scales
near both ends of the exponent range (boxes fall back to FP64 additions past
them), boxes whose values span far more than the aligned window, zero fields.

Tolerances: FP64 after the same cycles 1e-12, mixed solutions 1e-8."""
import numpy as np
import pytest

from paper_1701_04329_gb300 import afgpu
from tests.gpu_helpers import load, pair_random, rel_diff
from tests.test_gpu_parity import cycles_parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,uni,extra", [(4, 2, 1), (8, 3, 1), (8, 1, 2), (16, 2, 0), (16, 1, 1)])
def test_box_sizes(N, uni, extra):
    a, b, rho, bv = pair_random(3, N, uni, extra, 70 + N)
    load(a, b, rho, bv)
    cycles_parity(a, b, 2)


@pytest.mark.parametrize("scale", [1e-285, 1e-250, 1e-30, 1e30, 1e200])
def test_scales(scale):
    a, b, rho, bv = pair_random(3, 8, 2, 1, 81)
    load(a, b, scale * rho, scale * bv)
    a.fmg()
    b.fmg()
    assert rel_diff(b.get_solution(), a.get_solution()) <= 1e-12
    a.vcycle()
    b.vcycle()
    assert rel_diff(b.get_solution(), a.get_solution()) <= 1e-12


def test_values_of_very_different_size_in_one_box():
    """A source in a few cells and data on one side only: values from 1 down to
    1e-12 and zero within boxes, and of either sign."""
    a, b, rho, bv = pair_random(3, 8, 3, 0, 83)
    x = a.cell_centers()
    rho = np.where(np.abs(x - 0.3).max(1) < 0.02, 1e6, 0.0) * np.sign(np.sin(40 * x[:, 0]))
    load(a, b, rho, np.where(np.arange(len(bv)) % 97 == 0, bv, 1e-12 * bv))
    cycles_parity(a, b, 2)


def test_zero_fields():
    a, b, rho, bv = pair_random(3, 8, 3, 0, 84)
    load(a, b, 0 * rho, 0 * bv)
    b.fmg()
    assert float(b.get_solution().abs().max()) == 0.0
    load(a, b, 0 * rho, bv)  # u from the boundary alone (no relative residual: rho is zero)
    a.fmg()
    b.fmg()
    assert rel_diff(b.get_solution(), a.get_solution()) <= 1e-12


@pytest.mark.parametrize("N,uni,extra", [(4, 3, 1), (8, 3, 2), (16, 2, 1)])
def test_mixed_2d(N, uni, extra):
    a, b, rho, bv = pair_random(2, N, uni, extra, 85 + N)
    load(a, b, rho, 1e-3 * bv)
    a.solve(1e-12, 60)
    st = b.solve(afgpu.default_opts(rel_tol=1e-10, precision=afgpu.AFG_MIXED))
    assert st["rel_residual"] <= 1e-10
    assert rel_diff(b.get_solution(), a.get_solution()) <= 1e-8
