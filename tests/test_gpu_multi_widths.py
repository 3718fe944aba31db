"""Every width of the many-right-hand-side V-cycle gives a column the same bits: a row is summed in its entry order
whichever kernel takes it (packs of systems per lane, or a warp per row for more than 16 systems in FP64 or without
16-byte packs).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2010_11130_gb300 as air  # noqa: E402
from sthdg import assemble  # noqa: E402
from sthdg.problems import manufactured_2d  # noqa: E402


@pytest.mark.parametrize("relax", ["FCF", "C"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_columns_do_not_depend_on_the_width(dtype, relax):
    air.build()
    s = assemble(manufactured_2d(5, 2, 1e-6))
    A = air.CSR.from_host(s.row_ptr, s.col, s.val)
    H = air.setup(A, theta=0.25, max_coarse=100, precision=int(dtype == torch.float32), relax=relax)
    B = torch.from_numpy(np.random.default_rng(7).standard_normal((s.n, 32))).to("cuda", dtype)
    X = air.vcycle_multi(H, B)
    assert torch.isfinite(X).all()
    for k in range(1, 32):
        b = B[:, :k].contiguous()
        assert torch.equal(air.vcycle_multi(H, b), X[:, :k].contiguous()), k
        if k in (16, 17, 18, 31):                    # rows that start off a pack's boundary
            odd = torch.empty(s.n * k + 1, dtype=dtype, device="cuda")[1:].view(s.n, k)
            odd.copy_(b)
            assert torch.equal(air.vcycle_multi(H, odd), X[:, :k].contiguous()), k
