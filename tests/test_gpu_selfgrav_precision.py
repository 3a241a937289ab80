"""Error of the self-gravitation term against extended precision, at the size
its time is quoted at (layered planet h = 0.15, 36,160 charge points).

The block lives on mantle nodes of one hemisphere and the rows compared on the
other: no stored entry and no fluid couples them, so that K_eff gives exact
zeros there and the product is the term alone. The reference sums the oracle's
charges in long double.

Tolerances, from a model of both forms on the CPU at these points: C^T takes
differences of a smooth potential, which lifts a relative error of 2e-15 (FP64
sums, one rounding of the running sum per source) to 6e-13 of the result's
root mean square, and one of 1e-14 per term (float pairs) to 2.3e-12. The FP64
form has to stay below the middle of the two, 1.2e-12, the double-float form
below twice its own, 4.6e-12."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.model import layered_planet  # noqa: E402
from oracle import fem, selfgrav  # noqa: E402
from tests.helpers import to_internal, to_canonical  # noqa: E402

EDGES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))
COLS = 3


@pytest.fixture(scope="module")
def case():
    mesh, model = layered_planet(h=0.15, seed=7)
    pts, inv_r, C = selfgrav.charges(mesh, model)
    dm = fem.dof_map(mesh.tet, mesh.region, len(mesh.xyz))
    pos = np.zeros((dm.n_p2, 3))
    pos[:len(mesh.xyz)] = mesh.xyz
    for k, (a, c) in enumerate(EDGES):
        pos[dm.tet10[:, 4 + k]] = 0.5 * (mesh.xyz[mesh.tet[:, a]] + mesh.xyz[mesh.tet[:, c]])
    node = np.zeros((dm.Nu, 3))
    for copy in (dm.unode_solid, dm.unode_fluid):
        node[copy[copy >= 0]] = pos[copy >= 0]
    mantle = np.linalg.norm(node, axis=1) > 0.75
    rng = np.random.default_rng(0)
    on = mantle & (node[:, 2] > 0.1)
    X = np.zeros((dm.Nu, 3, COLS))
    X[on] = rng.standard_normal((on.sum(), 3, COLS))
    X = X.reshape(-1, COLS)
    rows = rng.choice(np.flatnonzero(np.repeat(mantle & (node[:, 2] < -0.35), 3)), 30, replace=False)
    Cc = C.tocsc()
    P, Q = pts.astype(np.longdouble), (C @ X).astype(np.longdouble)
    phi = {}
    ref = np.zeros((len(rows), COLS), np.longdouble)
    for k, r in enumerate(rows):
        for e in range(Cc.indptr[r], Cc.indptr[r + 1]):
            i = Cc.indices[e]
            if i not in phi:
                d = P - P[i]
                r2 = (d * d).sum(1)
                r2[i] = 1
                w = 1 / np.sqrt(r2)
                w[i] = inv_r[i]
                phi[i] = (w[:, None] * Q).sum(0)
            ref[k] -= model.G * Cc.data[e].astype(np.longdouble) * phi[i]
    return mesh, model, X, rows, ref


@pytest.fixture(scope="module")
def problem(case):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1906_11082_gb300 import nm
    P = nm.Problem(nm.Context(0), case[0], case[1], self_gravity=True)
    assert P.info["n_charges"] == 36160
    return nm, P


# widths of one, two and four column groups of 8, 16 and 32
@pytest.mark.parametrize("b", [3, 16, 32, 40])
@pytest.mark.parametrize("form", ["f64", "mixed", "mixed_in_double"])
def test_error_of_the_term(case, problem, form, b):
    _, _, X, rows, ref = case
    nm, P = problem
    Xw = np.zeros((len(X), b))
    Xw[:, b - COLS:] = X
    Y = torch.empty((len(X), b), dtype=torch.float64, device="cuda")
    if form == "mixed_in_double":
        P.set_option("double_float", 0)
    try:
        P.apply_K(torch.tensor(to_internal(P, Xw), device="cuda"), Y, k_P=20,
                  prec=nm.NM_F64 if form == "f64" else nm.NM_MIXED)
        got = to_canonical(P, Y.cpu().numpy())[rows][:, b - COLS:]
    finally:
        P.set_option("double_float", 1)
    err = (got - ref).astype(float)
    rel = np.sqrt((err ** 2).mean() / (ref.astype(float) ** 2).mean())
    assert rel <= (4.6e-12 if form == "mixed" else 1.2e-12), rel


@pytest.mark.parametrize("power", [70, -70])
def test_double_form_in_any_units(power):
    """Lengths in units of 2^power, G scaled so that every term of K_eff keeps
    its share: the product is 2^power times that in plain units (a power of two
    scales every step exactly; 1e-11 as for the product against the oracle).
    Squared distances leave the float range."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_1906_11082_gb300 import nm
    from synth.model import homogeneous_ball
    out = []
    for p in (0, power):
        mesh, model = homogeneous_ball(h=0.45, seed=1)
        mesh.xyz = mesh.xyz * 2.0 ** p
        model.G = 2.0 ** (-2 * p) / np.pi
        P = nm.Problem(nm.Context(0), mesh, model, self_gravity=True)
        X = torch.randn((P.n, 5), dtype=torch.float64, device="cuda",
                        generator=torch.Generator(device="cuda").manual_seed(2))
        T, K = torch.empty_like(X), torch.empty_like(X)
        P.apply_K(X, T)
        nm.Problem(nm.Context(0), mesh, model).apply_K(X, K)
        torch.cuda.synchronize()
        out.append(((K - T) * 2.0 ** -p, K * 2.0 ** -p))
    (t0, k0), (t1, k1) = out
    assert float((k1 - k0).abs().max() / k0.abs().max()) <= 1e-11
    assert float((t1 - t0).abs().max() / k0.abs().max()) <= 1e-11
    assert float(t0.abs().max() / k0.abs().max()) > 1e-4   # the term counts
