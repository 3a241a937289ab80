"""Products that are the first call on a new problem: the float values they
read are made by that call.

Tolerances as for the same products in test_gpu_parity.py (1e-4 for a float
K_eff product at k_P = 40, 2e-5 for a float mass product)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.model import layered_planet  # noqa: E402
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
def planet():
    mesh, model = layered_planet(h=0.25, seed=7)
    return mesh, model, fem.assemble(mesh, model)


@pytest.mark.parametrize("first", ["K", "M"])
def test_first_float_product(nm, planet, first):
    """The pressure chain's E_G^T product loads its values before it waits for
    the kernel launched before it: the conversion that makes them must be over.
    The second call comes on a stream of its own."""
    mesh, model, S = planet
    Xc = np.random.default_rng(4).standard_normal((S.n, 8))
    ref = {"K": filtlan.Operator(S, k_M=10, k_P=40).K(Xc), "M": S.M @ Xc}
    tol = {"K": 1e-4, "M": 2e-5}
    P = nm.Problem(nm.Context(0), mesh, model)
    X = torch.tensor(to_internal(P, Xc), dtype=torch.float32, device=DEV)
    Y, Z = torch.empty_like(X), torch.empty_like(X)
    torch.cuda.synchronize()
    other = torch.cuda.Stream()

    def call(which, out, stream=None):
        if which == "K":
            P.apply_K(X, out, k_P=40, stream=stream)
        else:
            P.apply_M(X, out, stream=stream)

    second = "M" if first == "K" else "K"
    call(first, Y)
    call(second, Z, other)
    torch.cuda.synchronize()
    assert rel_err(to_canonical(P, Y.double().cpu().numpy()), ref[first]) <= tol[first]
    assert rel_err(to_canonical(P, Z.double().cpu().numpy()), ref[second]) <= tol[second]
    P.free()


@pytest.mark.parametrize("b", [30, 57, 64])
def test_staged_step_leaves_other_widths_alone(nm, planet, b):
    """Option tma is for blocks of 32 columns. Blocks that are padded to groups
    of 32 give the same bits before and after a call that built its tiles."""
    mesh, model, S = planet
    P = nm.Problem(nm.Context(0), mesh, model)
    P.set_option("tma", 1)
    W = torch.randn((S.n, b), dtype=torch.float64, device=DEV)
    W32 = torch.randn((S.n, 32), dtype=torch.float64, device=DEV)
    X, Y, Y32 = torch.empty_like(W), torch.empty_like(W), torch.empty_like(W32)
    P.solve_M(W, X, k_M=12, prec=nm.NM_MIXED)
    P.solve_M(W32, Y32, k_M=12, prec=nm.NM_MIXED)
    P.solve_M(W, Y, k_M=12, prec=nm.NM_MIXED)
    assert bool((X == Y).all())
    P.free()
