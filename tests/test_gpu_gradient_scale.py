"""The velocity gradient where the pivots of an element matrix have no finite reciprocal.

With the quadrature weights times s = 2^-1022 every element matrix is s times the ordinary one, its pivots are subnormal
(below 2^-1024 the reciprocal overflows), and the gradient is s times the ordinary gradient.  An entry of A is rounded to
a multiple of 2^-1074; the sums of about 30 such terms of size s / 100 give a relative error below 30 * 100 * 2^-52 =
7e-13, times the condition of an element matrix (below 1e3): bound 1e-8 of the largest component.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2010_11130_gb300 as air  # noqa: E402
from paper_2010_11130_gb300 import hdg  # noqa: E402
from sthdg.mesh import build_mesh  # noqa: E402


@pytest.mark.parametrize("D", [2, 3])
def test_gradient_with_subnormal_pivots(D):
    air.build()
    mesh = hdg.HdgMesh.from_mesh(build_mesh(D, 2))
    tab, small = hdg.HdgTables(D, 1), hdg.HdgTables(D, 1)
    s = 2.0 ** -1022
    for name in ("wq", "wf"):
        small._t[name] *= s
    rng = np.random.default_rng(3)

    def field(*shape, mean=0.0):
        return torch.from_numpy(mean + 0.1 * rng.standard_normal(shape)).cuda()

    E = mesh.n_elems
    data = hdg.HdgData(0.0, 10.0, field(E, tab.nq, D - 1, mean=0.6), field(E, D + 1, tab.nqf, D - 1, mean=0.6),
                       field(E, tab.nq), field(E, D + 1, tab.nqf), field(mesh.n_facets, tab.nqf))
    y = hdg.assemble(mesh, tab, data)
    lam, adj = field(y.A.n), field(y.A.n)
    ref = hdg.velocity_gradient(mesh, tab, data, y, lam, adj)
    got = hdg.velocity_gradient(mesh, small, data, y, lam, adj) * 2.0 ** 511 * 2.0 ** 511
    assert torch.isfinite(got).all()
    assert float((got - ref).abs().max()) <= 1e-8 * float(ref.abs().max())
