"""The setup kernels where their forms change: blocks of the Falgout-style splitting whose graph fits in shared memory
and ones where it does not, l-AIR systems around the size that lanes solve on their own, Galerkin rows of every table
size.  Hierarchies are the oracle's bit for bit (C/F points, R and A patterns and values), as in test_gpu_parity.
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


def _banded(n, degree, reach, seed):
    """Rows of `degree` off-diagonal entries of like size within `reach` of the diagonal: all strong at theta 0.25."""
    import scipy.sparse as sp
    rng = np.random.default_rng(seed)
    r = np.repeat(np.arange(n), degree)
    c = (r + rng.integers(1, reach, len(r)) * rng.choice([-1, 1], len(r))) % n
    A = sp.coo_matrix((rng.uniform(0.5, 1.0, len(r)) * rng.choice([-1, 1], len(r)), (r, c)), shape=(n, n)).tocsr()
    A.sum_duplicates()
    A.setdiag(0.0)
    A.eliminate_zeros()
    A = A + sp.diags(np.asarray(abs(A).sum(1)).ravel() + 1.0)
    A = sp.csr_matrix(A)
    A.sort_indices()
    return A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data


def _compare(rp, ci, v, **kw):
    H = air.setup(air.CSR.from_host(rp, ci, v), **kw)
    O = oracle.setup(rp, ci, v, **kw)
    assert H.levels() == len(O.levels)
    for l, L in enumerate(O.levels):
        assert np.array_equal(H.export(l, "A.row_ptr"), L.A[0]) and np.array_equal(H.export(l, "A.col"), L.A[1])
        assert np.array_equal(H.export(l, "A.val"), L.A[2])
        if l + 1 < len(O.levels):
            assert np.array_equal(H.export(l, "cf"), L.cf)
            assert np.array_equal(H.export(l, "R.col"), L.R[1]) and np.array_equal(H.export(l, "R.val"), L.R[2])
    return H


@pytest.mark.parametrize("block", [1024, 2048])
@pytest.mark.parametrize("degree,reach", [(3, 40), (16, 100), (9, 3000)])
def test_falgout_blocks_inside_and_outside_shared_memory(degree, reach, block):
    rp, ci, v = _banded(5000, degree, reach, degree)
    _compare(rp, ci, v, theta=0.25, falgout_block=block, max_coarse=300, max_levels=3, max_dense=4096)


@pytest.mark.parametrize("degree", [1, 2, 6, 7, 9, 14])
def test_local_systems_and_galerkin_rows(degree):
    rp, ci, v = _banded(3001, degree, 60, 10 + degree)
    H = _compare(rp, ci, v, theta=0.25, max_coarse=200, max_levels=4, max_dense=4096)
    assert H.info(0).max_m >= min(degree, 2) - 1
