"""A request that the allocator refuses in the middle of a call leaves the tree
as it was before the call: the call reports AFG_ERR_NOMEM, and the next one,
with memory to be had, gives the solution.  Every request of the first mixed
solve and of the first adjoint solve is refused in turn."""
import pytest

from paper_1701_04329_gb300 import afgpu
from paper_1701_04329_gb300 import workloads as W
from tests.gpu_helpers import load, pair_from_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class RefuseNth:
    def __init__(self):
        self.left = None  # requests granted before one is refused

    def __call__(self, n):
        if self.left is not None:
            self.left -= 1
            if self.left < 0:
                return None
        return torch.cuda.caching_allocator_alloc(n)


@pytest.mark.parametrize("precision", [afgpu.AFG_FP64, afgpu.AFG_MIXED])
@pytest.mark.parametrize("call", ["solve", "adjoint"])
def test_refused_in_turn(precision, call):
    opts = afgpu.default_opts(precision=precision)

    def run(t, rho):
        if call == "solve":
            t.solve(opts)
            return t.get_solution()
        return t.adjoint(torch.tensor(rho, device="cuda"), opts)[0]

    alloc = RefuseNth()
    afgpu.set_allocator(alloc, torch.cuda.caching_allocator_delete)
    try:
        want, refused = None, 0
        for k in range(40):
            a, t, rho, bv = pair_from_problem(W.gauss2d(max_level=5))
            load(a, t, rho, bv)
            if want is None:
                want = run(t, rho)
                t.close()
                a, t, rho, bv = pair_from_problem(W.gauss2d(max_level=5))
                load(a, t, rho, bv)
            alloc.left = k
            try:
                run(t, rho)
                t.close()
                break
            except afgpu.AfgError as e:
                assert e.code == afgpu.AFG_ERR_NOMEM
                refused += 1
            alloc.left = None
            assert torch.equal(run(t, rho), want)
            t.close()
        expected = (3 if precision == afgpu.AFG_MIXED else 0) if call == "solve" else 14 + (3 if precision == afgpu.AFG_MIXED else 0)
        assert refused == expected
    finally:
        alloc.left = None
        afgpu.set_allocator(None, None)
