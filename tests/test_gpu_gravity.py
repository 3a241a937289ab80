"""Reference gravity by direct summation on a mesh large enough for the
double-float sums (16,384 tets), against the oracle's FP64 sums.

Tolerance: the oracle's and the library's sums each round once per source in
FP64 at worst (44k sources: 1e-14 of |g|), so 1e-12 of the largest entry, as
for the smaller meshes of test_gpu_parity.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.model import layered_planet  # noqa: E402
from oracle import fem  # noqa: E402
from tests.helpers import rel_err  # noqa: E402


@pytest.mark.parametrize("shift,scale", [(0.0, 1.0), (0.75, 6371.0)])
def test_double_float_gravity(shift, scale):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1906_11082_gb300 import nm
    mesh, model = layered_planet(h=0.12, seed=3)
    mesh.xyz[:] = (mesh.xyz + shift) * scale       # off-centre, other units
    assert mesh.nt >= 16384
    P = nm.Problem(nm.Context(0), mesh, model)
    g = P.gravity()
    p2 = P.unodes()[1]
    pick = np.random.default_rng(0).choice(len(p2), 500, replace=False)
    tet = mesh.tet.astype(np.int64)
    nv = len(mesh.xyz)
    pair = np.sort(np.stack([tet[:, list(e)] for e in ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))], 1), -1)
    key = np.unique(pair[..., 0] * nv + pair[..., 1])
    pos = np.concatenate([mesh.xyz, 0.5 * (mesh.xyz[key // nv] + mesh.xyz[key % nv])])[p2[pick]]
    ref = fem.gravity_direct(pos, mesh.xyz, tet, model.rho, model.G)
    assert rel_err(g[pick], ref) <= 1e-12
