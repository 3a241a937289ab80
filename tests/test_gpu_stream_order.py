"""Calls on the library's own stream read a basis or a start block only once the
work queued on the current stream has made it, and the vectors they return are
there for work on any stream: the same values as with everything complete."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.model import config_ball  # noqa: E402

KW = dict(block=8, degree=100, k_M=40, k_P=40, max_blocks=16, seed=5)


@pytest.fixture(scope="module")
def problem():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1906_11082_gb300 import nm
    w = config_ball()
    P = nm.Problem(nm.Context(0), w.mesh, w.model)
    P.set_interval(0.0, 3.0)
    return P


def _late(value, out):
    """Queue value into out behind about 50 ms of work on the current stream."""
    torch.cuda._sleep(100_000_000)
    out.copy_(value)


@pytest.mark.parametrize("side", [False, True])
@pytest.mark.parametrize("call", ["ritz", "slice", "begin", "add"])
def test_inputs_still_being_made(problem, call, side):
    P = problem
    g = torch.Generator(device="cuda").manual_seed(3)
    src = torch.randn((P.n, 40 if call == "ritz" else 8), dtype=torch.float64, device="cuda", generator=g)

    def solve(t):
        if call == "ritz":
            P.set_interval(-1.0, 1e4, unit=1)   # the whole spectrum: every Ritz value of the basis
            try:
                return P.ritz(t)
            finally:
                P.set_interval(0.0, 3.0)
        if call == "slice":
            return P.lanczos_slice(start=t, **KW)
        run = P.lanczos_begin(None, start=t, **KW) if call == "begin" else P.lanczos_begin([(0.0, 3.0)], **KW)
        if call == "add":
            run.add(0.0, 3.0, start=t)
        while run.step():
            pass
        return run.finish()[-1]

    torch.cuda.synchronize()
    ref = solve(src)
    t = torch.zeros_like(src)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.default_stream()):
        _late(src, t)
        r = solve(t)
        X = r.vectors()
        norm = (X * X).sum(0)
    torch.cuda.synchronize()
    assert np.array_equal(r.lam, ref.lam) and len(r.lam) > 0
    assert torch.equal(norm, (ref.vectors() ** 2).sum(0))
    r.free()
    ref.free()
