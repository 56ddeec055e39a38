"""A tree's first calls on a stream that does not wait for the default one: the
fields are zeroed before a call can write them.  The same bits as on the default
stream."""
import pytest

from paper_1701_04329_gb300 import afgpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [afgpu.AFG_FP64, afgpu.AFG_MIXED])
def test_first_calls(precision):
    def run():
        t = afgpu.Tree(3, 8, 6)
        t.refine_uniform(6)
        n = t.n_leaf_cells
        rho = torch.linspace(-1.0, 2.0, n, dtype=torch.float64, device="cuda")
        b = torch.linspace(0.0, 1.0, t.n_bfaces, dtype=torch.float64, device="cuda")
        torch.cuda.current_stream().synchronize()
        opts = afgpu.default_opts(rel_tol=1e-8, precision=precision, max_cycles=60)
        t.set_rhs(rho)
        t.set_dirichlet(b)
        t.solve(opts)
        lam, db, _ = t.adjoint(rho, opts)
        out = t.get_solution(), lam, db
        torch.cuda.current_stream().synchronize()
        t.close()
        return out

    want = run()
    side = torch.cuda.Stream()
    for _ in range(3):
        with torch.cuda.stream(side):
            got = run()
        assert all(torch.equal(x, y) for x, y in zip(got, want))
