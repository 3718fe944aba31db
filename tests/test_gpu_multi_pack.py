"""V-cycles for many right-hand sides over every packing of the systems into lanes: k whose rows hold 16-byte, 8-byte
and single values, vectors on and off those boundaries, and sweep patterns of even and odd length, against the
single V-cycle with the tolerances of the other many-right-hand-side tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2010_11130_gb300 as air  # noqa: E402
from sthdg import assemble  # noqa: E402
from sthdg.problems import manufactured_2d  # noqa: E402


@pytest.fixture(scope="module")
def system():
    air.build()
    return assemble(manufactured_2d(6, 2, 1e-6))


@pytest.mark.parametrize("relax", ["F", "FC", "FFC"])
@pytest.mark.parametrize("precision", [0, 1])
def test_packings_match_single_vcycles(system, precision, relax):
    s = system
    H = air.setup(air.CSR.from_host(s.row_ptr, s.col, s.val), theta=0.25, max_coarse=100, precision=precision,
                  relax=relax)
    dtype, tol = (torch.float32, 1e-5) if precision else (torch.float64, 1e-13)
    rng = np.random.default_rng(5)
    B = rng.standard_normal((s.n, 32))
    single = [H.vcycle(torch.from_numpy(np.ascontiguousarray(B[:, j])).cuda()).cpu().numpy() for j in range(32)]
    for k in (1, 2, 3, 4, 6, 7, 12, 16, 17, 18, 31, 32):
        for off in (0, 1, 2):
            b = torch.zeros(off + s.n * k, dtype=dtype, device="cuda")[off:].view(s.n, k)
            b.copy_(torch.from_numpy(B[:, :k]))
            x = torch.empty(off + s.n * k, dtype=dtype, device="cuda")[off:].view(s.n, k)
            X = air.vcycle_multi(H, b, x).double().cpu().numpy()
            for j in range(k):
                assert np.linalg.norm(X[:, j] - single[j]) <= tol * np.linalg.norm(single[j]), (k, off, j)
