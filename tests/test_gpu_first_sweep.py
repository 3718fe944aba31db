"""The V-cycle whose first sweep reads the coarse correction through P, against the many-right-hand-side V-cycle, which
interpolates first, with the tolerances of the many-right-hand-side tests: first sweeps over F and over C, one to three
sweeps, systems whose sets fill slices of 32 rows and do not."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2010_11130_gb300 as air  # noqa: E402
from sthdg import assemble  # noqa: E402
from sthdg.problems import manufactured_1d, manufactured_2d  # noqa: E402


@pytest.mark.parametrize("relax", ["F", "C", "FC", "CF", "CCF", "FFC"])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("problem", [(manufactured_1d, 17, 1, 1e-4), (manufactured_1d, 32, 2, 1e-6),
                                     (manufactured_2d, 5, 2, 1e-6)])
def test_first_sweep_through_interpolation(problem, precision, relax):
    air.build()
    make, n, p, nu = problem
    s = assemble(make(n, p, nu))
    H = air.setup(air.CSR.from_host(s.row_ptr, s.col, s.val), theta=0.25, max_coarse=40, precision=precision,
                  relax=relax)
    dtype, tol = (torch.float32, 1e-5) if precision else (torch.float64, 1e-13)
    B = np.random.default_rng(9).standard_normal((s.n, 3))
    X = air.vcycle_multi(H, torch.from_numpy(B).to(dtype).cuda()).double().cpu().numpy()
    for j in range(3):
        x = H.vcycle(torch.from_numpy(np.ascontiguousarray(B[:, j])).cuda()).cpu().numpy()
        assert np.linalg.norm(X[:, j] - x) <= tol * np.linalg.norm(x)
