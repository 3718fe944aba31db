"""The assembly and velocity-gradient kernels for every space-time dimension and degree, with and without diffusion, on
meshes whose element count leaves a last block ragged, against the host assembly of sthdg.

Values: 1e-11 of a row's largest entry, as in test_gpu_hdg_assembly (the conditioning of A_K times a few roundoffs).
Gradient: phi(a) = mu^T (H(a) - S(a) Lam) of the unscaled host system along a random direction d, central difference
with h = 1e-5.  phi carries a relative rounding error of about 1e4 eps of its terms' size, divided by h: 2e-7; the
truncation is of order h^2.  Bound: 2e-6 of sum |mu| (|H| + |S| |Lam|).
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2010_11130_gb300 as air  # noqa: E402
from paper_2010_11130_gb300 import hdg  # noqa: E402
from sthdg import assemble  # noqa: E402
from sthdg.mesh import build_mesh  # noqa: E402
from sthdg.problems import manufactured_1d, manufactured_2d  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    air.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def _sparse(s):
    import scipy.sparse as sp
    return sp.csr_matrix((s.val, s.col, s.row_ptr), shape=(s.n, s.n))


@pytest.mark.parametrize("nu", [0.0, 1e-2])
@pytest.mark.parametrize("D,p,n", [(2, 1, 3), (2, 2, 3), (2, 3, 1), (3, 1, 3), (3, 2, 1), (3, 3, 1)])
def test_assembly_and_gradient(D, p, n, nu):
    base = manufactured_1d(n, p, nu) if D == 2 else manufactured_2d(n, p, nu, velocity="constant")
    mesh = build_mesh(D, n, reflect=base.reflect)
    rng = np.random.default_rng(7)
    mean = np.array([1.0]) if D == 2 else np.array([0.7, 0.3])
    ev = mean + 0.1 * rng.standard_normal((mesh.n_elems, D - 1))
    prob = dataclasses.replace(base, elem_velocity=ev)
    ref = assemble(prob, mesh=mesh, keep_diag=True)
    tab = hdg.HdgTables(D, p)
    hm = hdg.HdgMesh.from_mesh(mesh)
    xv, xf, xF = (x.cpu().numpy() for x in hdg.points(hm, tab))

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()

    data = hdg.HdgData(nu, 10.0 * p * p, dev(np.broadcast_to(ev[:, None], xv.shape[:2] + (D - 1,))),
                       dev(np.broadcast_to(ev[:, None, None], xf.shape[:3] + (D - 1,))), dev(prob.source(xv)),
                       dev(prob.u_initial(xf)), dev(prob.g_dirichlet(xF)))
    y = hdg.assemble(hm, tab, data)
    assert np.array_equal(y.A.row_ptr.cpu().numpy(), ref.row_ptr)
    assert np.array_equal(y.A.col.cpu().numpy(), ref.col)
    rows = np.repeat(np.arange(ref.n), np.diff(ref.row_ptr))
    top, err = np.zeros(ref.n), np.zeros(ref.n)
    np.maximum.at(top, rows, np.abs(ref.val))
    np.maximum.at(err, rows, np.abs(y.A.val.cpu().numpy() - ref.val))
    assert np.max(err / top) <= 1e-11
    assert np.max(np.abs(y.rhs.cpu().numpy() - ref.rhs)) <= 1e-11 * np.max(np.abs(ref.rhs))
    assert np.max(np.abs(y.diag.cpu().numpy() - ref.S_diag)) <= 1e-11 * np.max(np.abs(ref.S_diag))

    lam, adj, d = rng.standard_normal(ref.n), rng.standard_normal(ref.n), rng.standard_normal(ev.shape)
    grad = hdg.velocity_gradient(hm, tab, data, y, dev(lam), dev(adj)).cpu().numpy()
    b = tab.b
    mu = np.linalg.solve(np.swapaxes(ref.S_diag, 1, 2), adj.reshape(-1, b, 1)).reshape(-1)

    def phi(e):
        s = assemble(dataclasses.replace(prob, elem_velocity=e), mesh=mesh, scale=False)
        return mu @ (s.rhs - _sparse(s) @ lam), np.abs(mu) @ (np.abs(s.rhs) + np.abs(_sparse(s)) @ np.abs(lam))

    h = 1e-5
    (up, size), (down, _) = phi(ev + h * d), phi(ev - h * d)
    assert abs((up - down) / (2 * h) - np.sum(grad * d)) <= 2e-6 * size
