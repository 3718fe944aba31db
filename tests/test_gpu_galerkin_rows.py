"""Galerkin rows at the edges of their tables and of the lengths from which they are sorted, and l-AIR systems on both
sides of the size that lanes solve on their own.  Hierarchies are the oracle's bit for bit (C/F points, R and A patterns
and values), as in test_gpu_parity; what each matrix reaches is counted from the oracle's hierarchy and asserted.
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


def _matrix(n, rows, cols, vals):
    """A chain of strong couplings plus the given entries."""
    import scipy.sparse as sp
    rng = np.random.default_rng(n)
    A = sp.diags([-rng.uniform(0.9, 1.0, n - 1), rng.uniform(2.5, 3.0, n), -rng.uniform(0.9, 1.0, n - 1)], [-1, 0, 1],
                 format="csr")
    A = sp.csr_matrix(A + sp.coo_matrix((vals, (rows, cols)), shape=(n, n)))
    A.sort_indices()
    return A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data


def _compare(A, **kw):
    H = air.setup(air.CSR.from_host(*A), **kw)
    O = oracle.setup(*A, **kw)
    assert H.levels() == len(O.levels)
    for l, L in enumerate(O.levels):
        assert np.array_equal(H.export(l, "A.row_ptr"), L.A[0]) and np.array_equal(H.export(l, "A.col"), L.A[1])
        assert np.array_equal(H.export(l, "A.val"), L.A[2])
        if l + 1 < len(O.levels):
            assert np.array_equal(H.export(l, "cf"), L.cf)
            assert np.array_equal(H.export(l, "R.col"), L.R[1]) and np.array_equal(H.export(l, "R.val"), L.R[2])
    return O.levels


def _terms(L):
    """Terms r_ik a_kj of every row of R A."""
    return np.add.reduceat(np.diff(L.A[0])[L.R[1]], L.R[0][:-1])


def test_rows_around_every_table_size():
    n, rng = 12000, np.random.default_rng(0)
    bounds = (256, 512, 1024, 2048, 4096)
    lengths = [d for b in bounds for d in (b - 14, b + 2)] + [9000]
    heavy = 100 + 1000 * np.arange(len(lengths))
    rows = np.repeat(heavy, lengths)
    cols = np.concatenate([rng.choice(n, d, replace=False) for d in lengths])
    far = np.abs(rows - cols) > 1                                   # weak: the strength graph stays the chain's
    rows, cols = rows[far], cols[far]
    L = _compare(_matrix(n, rows, cols, rng.uniform(-1e-4, 1e-4, len(rows))), theta=0.25, max_coarse=500)
    T = _terms(L[0])
    for b in bounds:
        assert np.any((T <= b) & (T > 0.9 * b)) and np.any((T > b) & (T < 1.1 * b)), b
    assert T.max() > 8192


def test_rows_of_as_many_columns_as_are_ranked_or_sorted():
    n, rng = 12000, np.random.default_rng(1)
    lengths = [d for d in range(240, 272)] + [3000]
    heavy = 100 + 300 * np.arange(len(lengths))
    rows = np.repeat(heavy, lengths)
    cols = np.concatenate([2 * rng.choice(n // 2, d, replace=False) for d in lengths])     # about one coarse column each
    far = np.abs(rows - cols) > 1
    rows, cols = rows[far], cols[far]
    L = _compare(_matrix(n, rows, cols, rng.uniform(-1e-4, 1e-4, len(rows))), theta=0.25, max_coarse=500)
    nj = set(np.diff(L[1].A[0]).tolist())
    assert {255, 256, 257, 258} <= nj and max(nj) > 1500


def test_columns_of_as_many_places_as_are_counted_or_sorted():
    """Stars: every spoke depends on its hub alone, which becomes the one C point they interpolate from."""
    import scipy.sparse as sp
    counts = list(range(250, 262)) + [5000]
    n, rng = sum(counts) + len(counts) + 1, np.random.default_rng(2)
    hub = np.concatenate([[0], np.cumsum(np.add(counts, 1))[:-1]])
    spokes = np.concatenate([h + 1 + np.arange(c) for h, c in zip(hub, counts)])
    of = np.repeat(hub, counts)
    A = (sp.identity(n) * 3.0 + sp.coo_matrix((-rng.uniform(0.9, 1.0, len(of)), (spokes, of)), shape=(n, n)) +
         sp.coo_matrix((-rng.uniform(1e-4, 1e-3, len(of)), (of, spokes)), shape=(n, n)))
    # what the hubs' rows hold strongly is the last point
    A = sp.csr_matrix(A + sp.coo_matrix((-np.ones(len(hub)), (hub, np.full(len(hub), n - 1))), shape=(n, n)))
    A.sort_indices()
    A = A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data
    L = _compare(A, theta=0.25, max_coarse=5)
    RA = (sp.csr_matrix((np.ones(len(L[0].R[1])), L[0].R[1], L[0].R[0]), shape=(L[0].nc, n)) @
          sp.csr_matrix((np.ones(len(A[1])), A[1], A[0]), shape=(n, n))).tocsr()
    places = set()
    for i in range(L[0].nc):
        J = L[0].pcol[RA.indices[RA.indptr[i]:RA.indptr[i + 1]]]
        places |= set(np.bincount(J[J >= 0]).tolist())
    assert {255, 256, 257, 258} <= places and max(places) > 4096


@pytest.mark.parametrize("degree", [4, 12])
def test_local_systems_on_both_sides_of_the_lane_size(degree):
    import scipy.sparse as sp
    n, rng = 3000, np.random.default_rng(degree)
    r = np.repeat(np.arange(n), degree)
    c = (r + rng.integers(1, 60, len(r)) * rng.choice([-1, 1], len(r))) % n
    A = sp.csr_matrix(sp.coo_matrix((rng.uniform(0.5, 1.0, len(r)), (r, c)), shape=(n, n)))
    A.setdiag(0.0)
    A.eliminate_zeros()
    A = sp.csr_matrix(A + sp.diags(np.asarray(A.sum(1)).ravel() + 1.0))
    A.sort_indices()
    L = _compare((A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data), theta=0.25, max_coarse=200)
    m = np.concatenate([np.diff(q.R[0]) - 1 for q in L[:-1]])
    assert np.any((m > 0) & (m <= 6)) and np.any(m == 6) and np.any(m == 7) and m.max() > 7
