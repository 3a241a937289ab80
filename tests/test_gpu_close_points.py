"""Direct sums on meshes with a sliver, whose points come closer to each other
than the float triples of the double-float sums resolve: the sums run in FP64.

The sliver is a separate solid tet with coordinates on a fine binary grid, so
that its barycentres and mid-edge nodes are exact and the distance of two of
its points (2^-32 and a low part near 2^-46) is known to every bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.model import layered_planet  # noqa: E402
from oracle import fem  # noqa: E402


@pytest.fixture(scope="module")
def nm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1906_11082_gb300 import nm as mod
    return mod


def _with_tet(h, vertices):
    mesh, model = layered_planet(h=h, seed=3)
    nv = len(mesh.xyz)
    mesh.xyz = np.concatenate([mesh.xyz, vertices])
    mesh.tet = np.concatenate([mesh.tet, np.arange(nv, nv + 4, dtype=mesh.tet.dtype)[None]])
    mesh.region = np.concatenate([mesh.region, np.zeros(1, mesh.region.dtype)])
    solid = int(np.flatnonzero(mesh.region[:-1] == 0)[0])
    for name in ("rho", "lam", "mu", "N2"):
        a = getattr(model, name)
        setattr(model, name, np.concatenate([a, a[solid:solid + 1]]))
    return mesh, model


def test_mixed_self_gravitation_of_a_sliver(nm):
    """Apex t = 2^-30 + 2^-44 + 2^-45 above the barycentre of a face: the two
    charge points are t / 4 apart. The mixed form has to agree with its sums in
    double (1e-12 of the largest entry: the double-float K_eff product). Float
    triples would err by 2^-29 of that pair."""
    t = 2.0 ** -30 + 2.0 ** -44 + 2.0 ** -45
    c = np.array([0.5, 0.25, 0.25])
    a = 0.25
    v = np.array([c + [a, 0, 0], c + [0, a, 0], c - [a, a, 0], c + [0, 0, t]])
    mesh, model = _with_tet(0.25, v)
    P = nm.Problem(nm.Context(0), mesh, model, self_gravity=True)
    X = torch.randn((P.n, 8), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(1))
    Y, Z = torch.empty_like(X), torch.empty_like(X)
    P.apply_K(X, Y, k_P=40, prec=nm.NM_MIXED)
    P.set_option("double_float", 0)
    P.apply_K(X, Z, k_P=40, prec=nm.NM_MIXED)
    assert bool(torch.isfinite(Z).all())
    assert float((Y - Z).abs().max() / Z.abs().max()) <= 1e-12
    P.free()


def test_reference_gravity_near_a_sliver(nm):
    """Four points whose diagonals pass each other at t = 2^-28 + 2^-44 + 2^-46:
    the barycentre is t / 2 from two mid-edge nodes, although no edge is short,
    and rules the field there. Float triples would err by 2^-35 of it, with
    18,000 other tets; FP64 sums agree to 1e-12, as for other meshes."""
    t = 2.0 ** -28 + 2.0 ** -44 + 2.0 ** -46
    c = np.array([0.5, 0.25, 0.25])
    u, v = np.array([0.125, 0, 0]), np.array([0, 0.125, 0])
    up = np.array([0, 0, t])
    mesh, model = _with_tet(0.12, np.array([c + u, c - u, c + v + up, c - v + up]))
    assert mesh.nt >= 16384
    P = nm.Problem(nm.Context(0), mesh, model)
    g = P.gravity()
    tet, nv = mesh.tet.astype(np.int64), len(mesh.xyz)
    pair = np.sort(np.stack([tet[:, list(e)] for e in ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))], 1), -1)
    key = np.unique(pair[..., 0] * nv + pair[..., 1])
    pos = np.concatenate([mesh.xyz, 0.5 * (mesh.xyz[key // nv] + mesh.xyz[key % nv])])[P.unodes()[1]]
    near = np.flatnonzero(np.abs(pos - c).max(1) < 2.0 ** -20)
    assert len(near) == 2
    ref = fem.gravity_direct(pos[near], mesh.xyz, tet, model.rho, model.G)
    assert np.abs(g[near] - ref).max() <= 1e-12 * np.abs(ref).max()
    P.free()
