"""Block-diagonal products and solves by groups of b lanes: every block size, counts that fill a warp, a thread block
and one block more, in place, and a singular block reported wherever in a warp it sits.  The blocks are diagonally
dominant (condition below 10): a product or solve of at most 11 terms is within 1e-13 of its largest entry.
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


@pytest.mark.parametrize("op", [0, 1, 2, 3])
@pytest.mark.parametrize("b", range(1, 12))
def test_every_block_size(b, op):
    per = 32 // b
    for k in (1, per, per + 1, 4 * per, 4 * per + 1, 1000):
        rng = np.random.default_rng(100 * b + k)
        D = rng.standard_normal((k, b, b)) / b + 2.0 * np.eye(b)
        D = D[:, rng.permutation(b)]                        # pivots off the diagonal
        x = rng.standard_normal((k, b))
        M = np.swapaxes(D, 1, 2) if op in (1, 3) else D
        want = np.linalg.solve(M, x[..., None])[..., 0] if op >= 2 else np.einsum("kij,kj->ki", M, x)
        y = torch.from_numpy(x.reshape(-1).copy()).cuda()
        air.block_diag_apply(b, torch.from_numpy(np.ascontiguousarray(D)).cuda(), op, y, y)
        assert np.max(np.abs(y.cpu().numpy().reshape(k, b) - want)) <= 1e-13 * np.max(np.abs(want)), k


@pytest.mark.parametrize("b", [1, 3, 6, 11])
def test_singular_blocks_are_reported(b):
    per = 32 // b
    k = 8 * per + 1
    for at in (0, per - 1, per, 4 * per, k - 1):
        d = torch.eye(b, dtype=torch.float64, device="cuda").repeat(k, 1, 1)
        d[at, b - 1] = 0.0
        x = torch.ones(k * b, dtype=torch.float64, device="cuda")
        with pytest.raises(air.AirError):
            air.block_diag_apply(b, d, 2, x)
        air.block_diag_apply(b, d, 0, x)
