"""A Gauss-Seidel wait that runs out is reported: with a limit of one poll, rows of a chain give up on the rows before
them, the V-cycle finishes with NaN, and the next call that reads the hierarchy's mark returns the error once.  With the
limit back at its default the same calls give what they gave before.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2010_11130_gb300 as air  # noqa: E402
from paper_2010_11130_gb300.air import gmres_solve_noalloc  # noqa: E402

TIMEOUT = -6


@pytest.fixture(scope="module", autouse=True)
def _built():
    air.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def _chain(precision):
    """20,000 rows, each coupled to the one before it: a depth of 20,000 groups of one row."""
    import scipy.sparse as sp
    n = 20000
    M = sp.diags([np.full(n - 1, -1.0), np.full(n, 2.0)], [-1, 0], format="csr")
    M.sort_indices()
    A = air.CSR.from_host(M.indptr, M.indices, M.data)
    b = torch.from_numpy(np.random.default_rng(1).standard_normal(n)).cuda()
    return A, air.setup(A, theta=0.25, relax="a", max_coarse=200, precision=precision, max_iter=20), b


def _fails(call):
    with pytest.raises(air.AirError) as e:
        call()
    assert e.value.status == TIMEOUT


@pytest.mark.parametrize("precision", [0, 1])
def test_a_wait_that_runs_out_is_reported(precision):
    A, H, b = _chain(precision)
    x = H.vcycle(b)
    H.check()
    assert torch.isfinite(x).all()
    H.set_wait_limit(1)
    assert torch.isnan(H.vcycle(b)).any()
    _fails(H.check)
    H.check()                                        # read once
    H.vcycle(b)
    torch.cuda.synchronize()
    H.set_wait_limit(1 << 20)
    _fails(lambda: air.gmres_solve(A, H, b))         # the mark of the V-cycle before
    assert torch.equal(H.vcycle(b), x)
    H.check()


@pytest.mark.parametrize("solve", [air.gmres_solve, air.bicgstab_solve, gmres_solve_noalloc])
def test_solves_report_it(solve):
    A, H, b = _chain(0)
    call = (lambda: solve(A, H, b, torch.empty_like(b))) if solve is gmres_solve_noalloc else (lambda: solve(A, H, b))
    x, info = call()
    assert info.status == 0
    H.set_wait_limit(1)
    _fails(call)
    H.set_wait_limit(1 << 20)
    y, again = call()
    assert again.status == 0 and torch.equal(x, y)


def test_the_batch_reports_it_for_the_problem_it_met():
    A, H, b = _chain(0)
    B, G, c = _chain(0)
    G.set_wait_limit(1)
    xs, infos, status = air.gmres_solve_batch([A, B], [H, G], [b, c])
    assert status == [0, TIMEOUT]
    H.check()
    G.check()
