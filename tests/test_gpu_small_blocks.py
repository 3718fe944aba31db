"""Block-diagonal products and solves, transpose and scaled transpose at the sizes where a warp's batches are ragged:
one block, one block more or less than 32, the smallest and largest block size, rows longer than the register sort
holds, block rows of more blocks than one chunk.

Bounds: the blocks are diagonally dominant (condition below 10), so a product or solve of at most 11 terms is within
1e-13 of its largest entry; the scaled transpose takes two such products and one inverse: 1e-12.  The plain transpose
moves values bit for bit.
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


def _blocks(rng, k, b):
    return rng.standard_normal((k, b, b)) / b + 2.0 * np.eye(b)


@pytest.mark.parametrize("op", [0, 1, 2, 3])
@pytest.mark.parametrize("k,b", [(1, 1), (31, 2), (32, 6), (33, 7), (65, 10), (5, 11)])
def test_block_apply_in_place(k, b, op):
    rng = np.random.default_rng(k * 100 + b)
    Dk, x = _blocks(rng, k, b), rng.standard_normal((k, b))
    M = np.swapaxes(Dk, 1, 2) if op in (1, 3) else Dk
    want = np.linalg.solve(M, x[..., None])[..., 0] if op >= 2 else np.einsum("kij,kj->ki", M, x)
    y = torch.from_numpy(x.reshape(-1).copy()).cuda()
    air.block_diag_apply(b, torch.from_numpy(Dk).cuda(), op, y, y)
    assert np.max(np.abs(y.cpu().numpy().reshape(k, b) - want)) <= 1e-13 * np.max(np.abs(want))


def test_singular_block_is_reported():
    d = torch.from_numpy(np.stack([np.eye(3)] * 40)).cuda()
    d[37, 1] = 0.0
    with pytest.raises(air.AirError):
        air.block_diag_apply(3, d, 2, torch.ones(120, dtype=torch.float64, device="cuda"))


@pytest.mark.parametrize("n", [1, 33, 128, 129, 300])
def test_transpose_of_long_rows(n):
    import scipy.sparse as sp
    rng = np.random.default_rng(n)
    A = sp.random(n, n, density=0.1, random_state=rng, format="lil")
    A[:, 0] = rng.standard_normal((n, 1)) + 3.0          # column 0 is full: a row of n entries in the transpose
    A.setdiag(2.0)
    A = sp.csr_matrix(A)
    A.sort_indices()
    T = sp.csr_matrix(A.T)
    T.sort_indices()
    t = air.transpose(air.CSR.from_host(A.indptr, A.indices, A.data))
    assert np.array_equal(t.row_ptr.cpu().numpy(), T.indptr)
    assert np.array_equal(t.col.cpu().numpy(), T.indices)
    assert np.array_equal(t.val.cpu().numpy(), T.data)


@pytest.mark.parametrize("k,b", [(2, 1), (9, 3), (14, 4)])
def test_scaled_transpose_of_many_blocks(k, b):
    rng = np.random.default_rng(k)
    n = k * b
    full = np.einsum("fg,ij->figj", np.ones((k, k)), np.ones((b, b))).astype(bool)
    for f in range(k):
        full[f, :, f, :] = np.eye(b, dtype=bool)
    mask = full.reshape(n, n)
    A = np.where(mask, rng.standard_normal((n, n)), 0.0)
    A[np.arange(n), np.arange(n)] = 1.0
    rp = np.concatenate([[0], np.cumsum(mask.sum(1))])
    D = _blocks(rng, k, b)
    big = np.zeros((n, n))
    for f in range(k):
        big[f * b:(f + 1) * b, f * b:(f + 1) * b] = D[f]
    want = np.linalg.solve(big.T, A.T) @ big.T
    t = air.transpose_scaled(air.CSR.from_host(rp, np.nonzero(mask)[1], A[mask]), b, torch.from_numpy(D).cuda())
    assert np.array_equal(t.row_ptr.cpu().numpy(), rp) and np.array_equal(t.col.cpu().numpy(), np.nonzero(mask)[1])
    assert np.max(np.abs(t.val.cpu().numpy() - want[mask])) <= 1e-12 * np.max(np.abs(want))
