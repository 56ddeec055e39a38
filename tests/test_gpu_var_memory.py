"""Variable-coefficient solves where the stored face coefficients do not fit:
the kernels that form them from eps run instead, and nothing is refused that
ran without them.  The allocator callbacks stand in for a full device: they
refuse every large request, or hold a budget that leaves too little room at
different points of the run.

Tolerances: FP64 after the same cycles 1e-12, mixed solutions 1e-8."""
import numpy as np
import pytest

from paper_1701_04329_gb300 import afgpu
from tests.gpu_helpers import load, pair_random, rel_diff
from tests.test_gpu_parity import cycles_parity
from tests.test_gpu_varcoef import var_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Device:
    """PyTorch's allocator with a largest request and a budget (bytes)."""

    def __init__(self, largest=1 << 60, budget=1 << 60):
        self.largest, self.budget, self.live, self.peak, self.size = largest, budget, 0, 0, {}
        self.asked, self.refused = 0, 0

    def alloc(self, n):
        self.asked = max(self.asked, n)
        if n > self.largest or self.live + n > self.budget:
            self.refused += 1
            return None
        p = torch.cuda.caching_allocator_alloc(n)
        self.size[p] = n
        self.live += n
        self.peak = max(self.peak, self.live)
        return p

    def free(self, p):
        self.live -= self.size.pop(p)
        torch.cuda.caching_allocator_delete(p)

    def __enter__(self):
        afgpu.set_allocator(self.alloc, self.free)
        return self

    def __exit__(self, *exc):
        afgpu.set_allocator(None, None)


def mixed(a, b, rho, bv, eps):
    b.set_eps(torch.tensor(eps, device="cuda"))
    load(a, b, rho, 1e-3 * bv)
    st = b.solve(afgpu.default_opts(rel_tol=1e-10, precision=afgpu.AFG_MIXED, max_cycles=60))
    assert st["rel_residual"] <= 1e-10
    return b.get_solution()


def plain_largest(D, N, uni, extra, seed):
    """The largest request of the same tree's Laplacian: a field or a table.  The
    coefficients are three to eight fields; the trees here are large enough for
    that to be more than any table."""
    with Device() as dev:
        _, t, rho, _ = pair_random(D, N, uni, extra, seed, frac=0.3)
        t.set_rhs(torch.tensor(rho, device="cuda"))
        t.close()
    return dev.asked


CASES = [(2, 8, 4, 1, 1), (2, 4, 5, 1, 2), (2, 16, 3, 1, 2), (3, 8, 2, 1, 1), (3, 4, 3, 1, 1), (3, 16, 1, 1, 1)]


@pytest.mark.parametrize("D,N,uni,extra,op", CASES)
def test_without_room_for_coefficients(D, N, uni, extra, op):
    with Device(largest=plain_largest(D, N, uni, extra, 960 + N + D)) as dev:
        a, b, rho, bv, eps = var_pair(D, N, uni, extra, 960 + N + D, op, cells=2, lo=0.5, hi=4.0)
        load(a, b, rho, bv)
        cycles_parity(a, b, 2)
        a.set_eps(eps[::-1].copy())  # new coefficients on the standing tree
        b.set_eps(torch.tensor(eps[::-1].copy(), device="cuda"))
        load(a, b, rho, bv)
        cycles_parity(a, b, 1)
        a.set_eps(eps)
        u = mixed(a, b, rho, bv, eps)
        a.solve(1e-12, 80)
        assert rel_diff(u, a.get_solution()) <= 1e-8
        b.close()
    assert dev.refused == 2  # both precisions' coefficients, asked for once each


@pytest.mark.parametrize("D,N,uni,extra,op", [(2, 8, 4, 1, 1), (3, 8, 2, 1, 1)])
def test_budgets_between_none_and_all(D, N, uni, extra, op):
    """FP64 cycles, then a mixed solve, with room for none of the coefficients, for
    the FP64 ones until the FP32 fields are wanted, for those of one precision."""
    a, b, rho, bv, eps = var_pair(D, N, uni, extra, 980, op, cells=2, lo=0.5, hi=4.0)
    load(a, b, rho, 1e-3 * bv)
    a.solve(1e-12, 80)
    ref = a.get_solution()
    b.close()

    def once(dev):
        with dev:
            c, b, _, _, _ = var_pair(D, N, uni, extra, 980, op, cells=2, lo=0.5, hi=4.0)
            load(c, b, rho, bv)
            cycles_parity(c, b, 1)
            assert rel_diff(mixed(c, b, rho, bv, eps), ref) <= 1e-8
            b.close()
        return dev.peak

    none, all_of_it = once(Device(largest=plain_largest(D, N, uni, extra, 980))), once(Device())
    assert all_of_it > none + 8 * (2 * D + 2) * len(rho)
    for part in (0.0, 0.2, 0.5, 0.62, 0.68, 0.8, 0.95):
        once(Device(budget=int(none + part * (all_of_it - none))))


def test_fp64_runs_hold_no_fp32_coefficients():
    with Device() as dev:
        a, b, rho, bv, eps = var_pair(3, 8, 2, 1, 981, 1)
        load(a, b, rho, bv)
        b.fmg()
        fp64 = dev.peak
        b.set_eps(torch.tensor(eps, device="cuda"))
        b.vcycle()
        assert dev.peak == fp64
        b.solve(afgpu.default_opts(rel_tol=1e-6, precision=afgpu.AFG_MIXED), allow_not_converged=True)
        assert dev.peak >= fp64 + 4 * (2 * 3 + 2 + 3) * b.n_leaf_cells
        b.close()


def test_adapting_with_coefficients_needs_room_for_the_fields_only():
    """afg_adapt_transfer holds the old and the new fields; the old grid's coefficients go first."""
    with Device() as dev:
        a, b, rho, bv, eps = var_pair(3, 8, 2, 0, 982, 1)
        load(a, b, rho, bv)
        b.fmg()
        coef = 8 * 8 * b.n_leaf_cells
        before = dev.live
        b.adapt_transfer(np.zeros(b.n_leaf_cells, np.int8), 1)
        assert dev.peak <= max(before, 2 * (before - coef))
        b.close()


def test_the_laplacian_again_gives_the_coefficients_back():
    with Device() as dev:
        a, b, rho, bv, eps = var_pair(2, 8, 4, 1, 983, 1)
        load(a, b, rho, bv)
        cycles_parity(a, b, 1)
        with_coef = dev.live
        b.set_operator(afgpu.AFG_OP_LAPLACE)
        assert dev.live <= with_coef - 8 * 6 * b.n_leaf_cells
        a.set_operator(0)
        load(a, b, rho, bv)
        cycles_parity(a, b, 1)
        for t, e in ((a, eps), (b, torch.tensor(eps, device="cuda"))):
            t.set_operator(afgpu.AFG_OP_VAR)
            t.set_eps(e)
        load(a, b, rho, bv)
        cycles_parity(a, b, 1)
        assert dev.live == with_coef
        b.close()
