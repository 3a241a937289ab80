"""Combinations of the dispatch rules that the single-path tests leave out:
graph replay, the second stream and per-slice gamma tables on padded and
two-group widths; two lane groups per cluster at every lane count; three and
four single columns per lane of the double rows.

Graph replay and overlap run the same kernels on the same data: the same bits.
A refined mixed solve at k = 28 agrees with the same solve put together from
FP64 pieces to 1e-11, double rows with the oracle to 1e-11 and 1e-12, as in
test_gpu_widths.py; slices to 1e-8 as in test_gpu_parity.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.model import config_ball, layered_planet  # noqa: E402
from oracle import fem, filtlan, eig  # noqa: E402
from tests.helpers import to_internal, to_canonical, rel_err  # noqa: E402

DEV = "cuda:0"


@pytest.fixture(scope="module")
def nm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1906_11082_gb300 import nm as mod
    return mod


@pytest.fixture(scope="module")
def ctx(nm):
    return nm.Context(0)


@pytest.fixture(scope="module")
def planet(nm, ctx):
    mesh, model = layered_planet(h=0.25, seed=7)
    return fem.assemble(mesh, model), nm.Problem(ctx, mesh, model)


@pytest.fixture(scope="module")
def large(nm, ctx):
    """66k rows: the float steps fill the chip and take two lane groups."""
    return nm.Problem(ctx, *layered_planet(h=0.1, seed=2))


@pytest.mark.parametrize("option", ["graphs", "overlap"])
@pytest.mark.parametrize("b", [5, 21, 40, 61])
def test_padded_and_two_group_widths(nm, planet, option, b):
    S, P = planet
    lo, hi = P.spectrum_bounds(k_M=20)
    gam, c, e = nm.filter_design(lo, hi, 0.5, 9.0, 7)
    Y = torch.randn((S.n, b), dtype=torch.float64, device=DEV)
    Z = [torch.empty_like(Y), torch.empty_like(Y)]
    torch.cuda.synchronize()
    st = torch.cuda.Stream()   # capture needs a stream other than the legacy default
    for on in (0, 1):
        P.set_option(option, on)
        try:
            P.filter_apply(gam, c, e, 20, Y, Z[on], prec=nm.NM_MIXED, stream=st)
        finally:
            P.set_option(option, 0)
    st.synchronize()
    if option == "graphs":
        assert torch.equal(Z[0], Z[1])
    else:   # E_G S is added after the A_G product instead of inside it
        assert float((Z[0] - Z[1]).abs().max() / Z[0].abs().max()) <= 1e-11


@pytest.mark.parametrize("graphs", [0, 1])
def test_gamma_table_across_a_group_boundary(nm, ctx, graphs):
    """Five slices of eight columns are filtered as two groups of twenty: the
    third slice's columns lie in both."""
    w = config_ball()
    P = nm.Problem(ctx, w.mesh, w.model)
    K, M = eig.pencil_dense(fem.assemble(w.mesh, w.model))
    lam = eig.all_eigs(K, M)[0]
    slices = [(0.0, 2.7), (2.7, 3.0), (3.0, 3.8), (3.8, 4.3), (4.3, 4.8)]
    P.set_option("graphs", graphs)
    res = P.lanczos_multi(slices, block=8, degree=100, k_M=20, k_P=20, max_blocks=24, prec=nm.NM_MIXED, seed=4)
    assert len(res) == 5
    for (lo, hi), r in zip(slices, res):
        ref = lam[(lam >= (-1e-8 * lam[-1] if lo == 0 else lo * lo)) & (lam <= hi * hi)]
        big = np.abs(ref) > 1e-10 * lam[-1]
        assert len(r.lam) == len(ref)
        assert np.allclose(r.lam[big], ref[big], rtol=1e-8) and r.resid.max() <= 1e-6
        r.free()
    P.free()


@pytest.mark.parametrize("b", [20, 24, 28, 32, 40, 56, 64])
def test_two_lane_groups_per_cluster(nm, large, b):
    P, k = large, 28
    W = torch.randn((P.n, b), dtype=torch.float64, device=DEV)
    X, x, r, e = (torch.empty_like(W) for _ in range(4))
    P.solve_M(W, X, k, prec=nm.NM_MIXED)
    P.solve_M(W, x, k)
    P.apply_M(x, r)
    P.solve_M(W - r, e, k)
    ref = x + e
    assert float((X - ref).abs().max() / ref.abs().max()) <= 1e-11


@pytest.mark.parametrize("b,ld", [(21, 21), (21, 23), (33, 35), (27, 27), (9, 9), (15, 16)])
def test_single_columns_per_lane(planet, b, ld):
    """Odd widths: three and four columns per lane without paired accesses."""
    S, P = planet
    X = torch.zeros((S.n, ld), dtype=torch.float64, device=DEV)
    Xc = np.random.default_rng(b).standard_normal((S.n, b))
    X[:, :b] = torch.tensor(to_internal(P, Xc), device=DEV)
    op = filtlan.Operator(S, k_M=8, k_P=8)
    lo, hi = filtlan.spectrum_bounds(op, S.n)
    gam, c, e = filtlan.filter_coeffs(lo, hi, 0.5, 9.0, 2)
    Y = torch.full_like(X, 7.0)
    host = lambda: Y[:, :b].cpu().numpy()  # noqa: E731
    P.filter_apply(gam, c, e, 8, X[:, :b], Y[:, :b], k_P=8)
    assert rel_err(to_canonical(P, host()), filtlan.filter_apply(op, gam, c, e, Xc)) <= 1e-11
    P.apply_K(X[:, :b], Y[:, :b], k_P=8)
    assert rel_err(to_canonical(P, host()), op.K(Xc)) <= 1e-11
    P.apply_M(X[:, :b], Y[:, :b])
    assert rel_err(to_canonical(P, host()), S.M @ Xc) <= 1e-12
    assert bool((Y[:, b:] == 7.0).all())
