"""A gradient that is not finite is not reported as a converged adjoint solve:
the max norms that decide keep a NaN, in both precisions of the
preconditioner, whatever cell holds it; and the tree solves the next gradient
as if nothing had been."""
import numpy as np
import pytest

from paper_1701_04329_gb300 import afgpu
from tests.gpu_helpers import pair_random

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,N,uni,extra", [(2, 8, 2, 1), (3, 4, 2, 1), (3, 8, 1, 1)])
@pytest.mark.parametrize("precision", [afgpu.AFG_FP64, afgpu.AFG_MIXED])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_not_finite(D, N, uni, extra, precision, value):
    _, b, _, _ = pair_random(D, N, uni, extra, 60 + N)
    opts = afgpu.default_opts(rel_tol=1e-10, max_cycles=60, precision=precision)
    g = np.random.default_rng(61).normal(size=b.n_leaf_cells)
    good = torch.tensor(g, device="cuda")
    lam0, _, st0 = b.adjoint(good, opts)
    for at in (0, len(g) // 2 + 1, len(g) - 1):
        bad = good.clone()
        bad[at] = value
        with pytest.raises(afgpu.AfgError) as e:
            b.adjoint(bad, opts)
        assert e.value.code == afgpu.AFG_ERR_NOT_CONVERGED
    lam1, _, st1 = b.adjoint(good, opts)
    assert st1["cycles"] == st0["cycles"] and torch.equal(lam0, lam1)
