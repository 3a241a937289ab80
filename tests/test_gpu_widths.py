"""Sparse kernels over the block widths and sizes their rules distinguish,
against the CPU oracle.

Widths: every lane count of a column group (4 .. 32 columns), widths that are
no multiple of four (padded groups), widths of two groups. Tolerances as in
test_gpu_parity.py: 1e-11 relative for a refined mixed solve at k = 28, 2e-5
for a float solve.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.model import config_ball, layered_planet  # noqa: E402
from oracle import fem, filtlan  # noqa: E402
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


def _dev(a, dtype=torch.float64):
    return torch.tensor(a, dtype=dtype, device=DEV)


def _host(t):
    torch.cuda.synchronize()
    return t.double().cpu().numpy()


@pytest.mark.parametrize("b", [1, 3, 4, 8, 12, 16, 20, 21, 24, 28, 30, 33, 36, 44, 48, 52, 61, 64])
def test_mixed_solve_every_width(nm, planet, b):
    S, P = planet
    Wc = np.random.default_rng(b).standard_normal((S.n, b))
    X = torch.empty((S.n, b), dtype=torch.float64, device=DEV)
    P.solve_M(_dev(to_internal(P, Wc)), X, k_M=28, prec=nm.NM_MIXED)
    assert rel_err(to_canonical(P, _host(X)), filtlan.refined_solve(S.M, 1.0 / S.M.diagonal(), Wc, 28)) <= 1e-11


@pytest.mark.parametrize("b,ld", [(1, 1), (2, 2), (3, 4), (8, 8), (16, 17), (31, 31), (34, 34), (63, 63), (64, 66)])
def test_double_rows_every_width(planet, b, ld):
    """Row-by-row kernels: one and two columns per lane, one and two column
    chunks, every split of a row's entries; the outer update and the pressure
    chain inside a filter of degree 2; M, R and K products."""
    S, P = planet
    X = torch.zeros((S.n, ld), dtype=torch.float64, device=DEV)
    Xc = np.random.default_rng(b).standard_normal((S.n, b))
    X[:, :b] = _dev(to_internal(P, Xc))
    op = filtlan.Operator(S, k_M=8, k_P=8)
    lo, hi = filtlan.spectrum_bounds(op, S.n)
    gam, c, e = filtlan.filter_coeffs(lo, hi, 0.5, 9.0, 2)
    Y = torch.full_like(X, 7.0)
    P.filter_apply(gam, c, e, 8, X[:, :b], Y[:, :b], k_P=8)
    assert rel_err(to_canonical(P, _host(Y[:, :b])), filtlan.filter_apply(op, gam, c, e, Xc)) <= 1e-11
    P.apply_K(X[:, :b], Y[:, :b], k_P=8)
    assert rel_err(to_canonical(P, _host(Y[:, :b])), op.K(Xc)) <= 1e-11
    P.apply_M(X[:, :b], Y[:, :b])
    assert rel_err(to_canonical(P, _host(Y[:, :b])), S.M @ Xc) <= 1e-12
    P.apply_R(X[:, :b], Y[:, :b])
    assert rel_err(to_canonical(P, _host(Y[:, :b])), S.R @ Xc) <= 1e-12
    assert bool((Y[:, b:] == 7.0).all())


@pytest.mark.parametrize("b", [4, 21, 40, 64])
def test_float_filter_widths(nm, planet, b):
    """The last float step carries the outer Chebyshev update; two column
    groups of a block with its own leading dimension."""
    S, P = planet
    op = filtlan.Operator(S, k_M=12, k_P=12)
    lo, hi = filtlan.spectrum_bounds(op, S.n)
    gam, c, e = filtlan.filter_coeffs(lo, hi, 0.5, 9.0, 3)
    Yc = np.random.default_rng(b).standard_normal((S.n, b))
    Z = torch.empty((S.n, b), dtype=torch.float32, device=DEV)
    P.filter_apply(gam, c, e, 12, _dev(to_internal(P, Yc), torch.float32), Z, k_P=12)
    assert rel_err(to_canonical(P, _host(Z)), filtlan.filter_apply(op, gam, c, e, Yc)) <= 2e-5


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_float_solve_keeps_non_finite_values_local(nm, planet, bad):
    """One non-finite dof reaches its node's neighbours in two steps and no
    other row, although rows are gathered four at a time. (A row of a hit
    cluster sums its entries in another order: the float tolerance.)"""
    S, P = planet
    W = np.random.default_rng(3).standard_normal((S.n, 8))
    W[3 * 40, 2] = 0.0
    clean = torch.empty((S.n, 8), dtype=torch.float32, device=DEV)
    P.solve_M(_dev(W, torch.float32), clean, k_M=2)
    W[3 * 40, 2] = bad
    got = torch.empty_like(clean)
    P.solve_M(_dev(W, torch.float32), got, k_M=2)
    rp, col, _ = P.export(1)
    hit = torch.zeros((S.n, 8), dtype=torch.bool)
    hit[3 * col[rp[40]:rp[41]].astype(np.int64), 2] = True
    fin = torch.isfinite(got.cpu())
    assert bool((fin == ~hit).all())
    assert rel_err(got.cpu()[~hit], clean.cpu()[~hit]) <= 2e-5


def test_mixed_solve_on_the_ball(nm, ctx):
    """633 rows: the last cluster holds a single row, fewer clusters than warps."""
    w = config_ball()
    S, P = fem.assemble(w.mesh, w.model), nm.Problem(ctx, w.mesh, w.model)
    Wc = np.random.default_rng(1).standard_normal((S.n, 24))
    X = torch.empty((S.n, 24), dtype=torch.float64, device=DEV)
    P.solve_M(_dev(to_internal(P, Wc)), X, k_M=28, prec=nm.NM_MIXED)
    assert rel_err(to_canonical(P, _host(X)), filtlan.refined_solve(S.M, 1.0 / S.M.diagonal(), Wc, 28)) <= 1e-11


@pytest.mark.parametrize("I,J,K,pad", [(1, 1, 1, 0), (130, 9, 130, 1), (127, 33, 64, 1), (129, 16, 65, 2), (16, 8, 1000, 3)])
def test_split_products_odd_strides(nm, ctx, I, J, K, pad):
    """Dense products at the edges of their tiles (128 rows, 8 / 16 / 32
    columns, 64 terms), with strides and bases that rule out 16-byte copies,
    rows spread over 40 binades. Each kept or dropped piece errs by at most
    2^-50 of the product of the largest entries of its row and column."""
    rng = np.random.default_rng(I + J)
    X, Y = rng.standard_normal((K, I + pad)), rng.standard_normal((K, J + pad))
    X *= 2.0 ** rng.integers(-20, 20, (1, I + pad))
    C = torch.zeros((J, I + pad), dtype=torch.float64, device=DEV)
    dX, dY = _dev(X)[:, pad:], _dev(Y)[:, pad:]
    ctx.gemm_tn(dX, dY, C)
    bound = K * 2.0 ** -50 * np.outer(np.abs(X[:, pad:]).max(0), np.abs(Y[:, pad:]).max(0))
    assert (np.abs(_host(C)[:, :I].T - X[:, pad:].T @ Y[:, pad:]) <= bound).all()
    A, B = rng.standard_normal((I, K + pad)), rng.standard_normal((J, K + pad))
    A *= 2.0 ** rng.integers(-20, 20, (I, 1))
    D = torch.full((I, J + pad), 3.0, dtype=torch.float64, device=DEV)
    ctx.gemm_nn(_dev(A)[:, pad:], _dev(B)[:, pad:], D[:, :J], beta=1.0)
    bound = K * 2.0 ** -50 * np.outer(np.abs(A).max(1), np.abs(B).max(1)) + 2.0 ** -50
    assert (np.abs(_host(D)[:, :J] - (A[:, pad:] @ B[:, pad:].T + 3.0)) <= bound).all()
    assert bool((D[:, J:] == 3.0).all())


@pytest.mark.parametrize("b", [1, 5, 12, 16, 20, 24, 28, 32, 33, 48, 64])
def test_mixed_product_every_width(nm, planet, b):
    """Double-float K_eff product and residuals at every lane count, padded
    and two-group widths; fluid rows take E_G S in double. Tolerance as for
    the refined pressure solve at k = 28."""
    S, P = planet
    Xc = np.random.default_rng(b).standard_normal((S.n, b))
    Xc[::7] *= 1e-30                     # conversions outside their fast range
    Xc[5] = 0.0
    Y = torch.empty((S.n, b), dtype=torch.float64, device=DEV)
    P.apply_K(_dev(to_internal(P, Xc)), Y, k_P=28, prec=nm.NM_MIXED)
    op = filtlan.Operator(S, k_M=28, k_P=28, refine=True)
    assert rel_err(to_canonical(P, _host(Y)), op.K(Xc)) <= 1e-11
