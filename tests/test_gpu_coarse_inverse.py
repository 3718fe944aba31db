"""The dense inverse of the coarsest operator at the edges of its panels, tiles, clusters and threads, through one-level
hierarchies, whose V-cycle is the inverse itself: one row, a panel more or less than full, more rows than one block or
one cluster holds a thread for, zero and tiny diagonals that force row swaps, and a singular matrix.

Bound: the inverse's residual is a few n eps cond; the matrices below have condition numbers under 1e4, so A x = b holds
to 1e-10 of |b| at n <= 4200.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2010_11130_gb300 as air  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    air.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def _setup(A, **kw):
    import scipy.sparse as sp
    A = sp.csr_matrix(A)
    A.sort_indices()
    n = A.shape[0]
    return air.setup(air.CSR.from_host(A.indptr, A.indices, A.data), max_coarse=n, max_dense=n, **kw)


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 33, 128, 255, 991, 4096, 4097])
def test_inverse_with_row_swaps(n):
    import scipy.sparse as sp
    rng = np.random.default_rng(n)
    # large entries on a random permutation, a tiny diagonal: nearly every column swaps rows
    p = rng.permutation(n)
    A = sp.random(n, n, density=min(1.0, 8.0 / n), random_state=rng, format="csr") * 0.1
    A = A + sp.csr_matrix((rng.choice([-2.0, 2.0], n), (np.arange(n), p)), shape=(n, n)) + 1e-3 * sp.identity(n)
    H = _setup(A)
    assert H.levels() == 1
    b = rng.standard_normal(n)
    x = H.vcycle(torch.from_numpy(b).cuda()).cpu().numpy()
    assert np.linalg.norm(A @ x - b) <= 1e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("n", [3, 40, 600])
def test_singular_matrix_is_reported(n):
    import scipy.sparse as sp
    A = sp.identity(n, format="lil")
    A[n - 1, n - 2] = 1.0
    A[n - 2, n - 1] = 1.0                       # the last two rows are equal
    with pytest.raises(air.AirError) as e:
        _setup(A)
    assert e.value.status == -5
