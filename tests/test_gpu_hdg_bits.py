"""The assembled system keeps its bits, those of the expressions evaluated entry by entry before the assembly kernel
shared products between entries.  Which products of an entry are fused was found by comparing outputs with that form,
for each D, p and with or without diffusion; nothing else holds those choices, so the digests below do.

Meshes, velocities and data are integers over a power of two, and the reference tables are rounded to multiples of
2^-20, so that the inputs do not depend on the host's library functions.  The digest is over the bytes of the scaled
values, the right-hand side and the diagonal blocks.
"""
import hashlib

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2010_11130_gb300 as air  # noqa: E402
from paper_2010_11130_gb300 import hdg  # noqa: E402
from sthdg.mesh import build_mesh  # noqa: E402

DIGESTS = {
    (2, 1, 0.0): "b4a69e886792d2eb",
    (2, 1, 0.01): "a6e7f8cb37d20f6f",
    (2, 2, 0.0): "57dbcdd29a4592e0",
    (2, 2, 0.01): "ee8f313fd98f7ba8",
    (2, 3, 0.0): "4a44b2b66a26681c",
    (2, 3, 0.01): "720fe1cce543a413",
    (3, 1, 0.0): "d6387bcbef217f2c",
    (3, 1, 0.01): "99d78503d83baf30",
    (3, 2, 0.0): "f8c3cca95eda86b7",
    (3, 2, 0.01): "18cd98bdb6031a50",
    (3, 3, 0.0): "94cb49563c8db0ce",
    (3, 3, 0.01): "f6d418fb86a2be11",
}


def digest(D, p, nu):
    rng = np.random.default_rng([D, p])

    def grid(shape, top):
        return rng.integers(-top, top + 1, shape) / 2.0 ** 20

    mesh = hdg.HdgMesh.from_mesh(build_mesh(D, 2, vertex_map=lambda X: X + grid(X.shape, 2 ** 15)))
    tab = hdg.HdgTables(D, p)
    for name in ("wq", "phi", "gphi", "wf", "psi", "phi_f", "gphi_f", "dir_proj"):
        tab._t[name].copy_(torch.round(tab._t[name] * 2.0 ** 20) / 2.0 ** 20)
    E, F = mesh.n_elems, mesh.n_facets
    shapes = (E, tab.nq, D - 1), (E, D + 1, tab.nqf, D - 1), (E, tab.nq), (E, D + 1, tab.nqf), (F, tab.nqf)
    fields = [grid(s, 2 ** 16) for s in shapes]
    for v in fields[0], fields[1]:
        v += np.array([1.0] if D == 2 else [0.6875, 0.3125])
    data = hdg.HdgData(nu, 10.0 * p * p, *[torch.from_numpy(f).cuda() for f in fields])
    y = hdg.assemble(mesh, tab, data)
    assert torch.isfinite(y.A.val).all()
    h = hashlib.sha256()
    for t in (y.A.val, y.rhs, y.diag):
        h.update(t.cpu().numpy().tobytes())
    return h.hexdigest()[:16]


@pytest.mark.parametrize("nu", [0.0, 1e-2])
@pytest.mark.parametrize("D,p", [(2, 1), (2, 2), (2, 3), (3, 1), (3, 2), (3, 3)])
def test_bits_of_the_assembled_system(D, p, nu):
    air.build()
    assert digest(D, p, nu) == DIGESTS[D, p, nu]
