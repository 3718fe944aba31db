"""Gauss-Seidel sweeps where rows wait for one another most: groups of independent rows wider than the warps in flight
(a ticket then stands for several rows), rows of more entries than lanes, and right-hand sides that carry the NaN whose
bits mark a value as not yet written.  FP64 V-cycles agree with the oracle's sequential sweeps to 1e-10, the bound of
test_gpu_gauss_seidel (only the order of a row's sum differs).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2010_11130_gb300 as air  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    air.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def _layered(width, layers, degree):
    """Lower triangular, unit diagonal: every row couples to `degree` rows of the layer before."""
    import scipy.sparse as sp
    rng = np.random.default_rng(3)
    n = width * layers
    r = np.repeat(np.arange(width, n), degree)
    c = (r // width - 1) * width + rng.integers(0, width, len(r))
    A = sp.coo_matrix((-rng.uniform(0.2, 0.3, len(r)), (r, c)), shape=(n, n)).tocsr() + sp.identity(n, format="csr")
    A.sort_indices()
    return A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data


@pytest.mark.parametrize("relax", ["a", "fa"])
@pytest.mark.parametrize("width,degree", [(12000, 12), (300, 70)])
def test_wide_groups_and_long_rows(width, degree, relax):
    rp, ci, v = _layered(width, 3, degree)
    n = len(rp) - 1
    H = air.setup(air.CSR.from_host(rp, ci, v), theta=0.25, relax=relax, max_coarse=200)
    O = oracle.setup(rp, ci, v, theta=0.25, relax=relax, max_coarse=200)
    b = np.random.default_rng(5).standard_normal(n)
    x = H.vcycle(torch.from_numpy(b).cuda()).cpu().numpy()
    xo = O.vcycle(b)
    assert np.linalg.norm(x - xo) <= 1e-10 * np.linalg.norm(xo)


def test_nan_of_the_pending_pattern():
    rp, ci, v = _layered(300, 3, 4)
    H = air.setup(air.CSR.from_host(rp, ci, v), theta=0.25, relax="a", max_coarse=200)
    b = torch.ones(900, dtype=torch.float64, device="cuda")
    b.view(torch.int64)[0] = -1
    x = H.vcycle(b)
    assert torch.isnan(x[0]) and not torch.isnan(x).all()
