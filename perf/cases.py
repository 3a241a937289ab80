"""What the solver's time is measured on: the calls its users make, over the sizes they make them at.

Meshes run from the 400-tet ball of the smoke run to the 264k-tet planet of
the benchmark (h = 0.45 .. 0.05), block widths over 1 .. 64 (8 in the tests
and the smoke run, 16 per served request, up to four requests or 64 columns
in one recurrence, 32 in the benchmark), inner steps 18 .. 40, and the three
arithmetics a caller can choose. A problem is assembled once per process and
kept, as a program that solves many slices of one planet keeps it; the
blocks, start vectors and meshes to assemble come from the seed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1906_11082_gb300 import nm
from synth.model import homogeneous_ball, layered_planet

PREC = {"f64": nm.NM_F64, "f32": nm.NM_F32, "mixed": nm.NM_MIXED}
L2_BYTES = 126e6
# Extreme eigenvalues of the Jacobi-scaled P2 element mass matrix: the bounds
# the mass and pressure solves use when the caller gives none.
MASS_LO, MASS_HI = 0.25, (19.0 + math.sqrt(249.0)) / 8.0


def listed():
    return [
        # The benchmark's filter: 1.15M dof, 32 columns, 18 inner steps (a slice runs it at degree 600 per block).
        {"name": "filter_bench", "kind": "filter", "body": "planet", "h": 0.05, "b": 32, "prec": "mixed", "k": 18, "degree": 8},
        # One served request alone on its mesh: 16 columns.
        {"name": "filter_request", "kind": "filter", "body": "planet", "h": 0.1, "b": 16, "prec": "mixed", "k": 20, "degree": 10},
        # Four requests that joined one batch: 64 columns.
        {"name": "filter_batch", "kind": "filter", "body": "planet", "h": 0.1, "b": 64, "prec": "mixed", "k": 20, "degree": 6},
        # A batch of seven 3-column slices on a small planet: a width that is no multiple of anything, launches that are short.
        {"name": "filter_ragged", "kind": "filter", "body": "planet", "h": 0.25, "b": 21, "prec": "mixed", "k": 20, "degree": 16},
        # The float filter.
        {"name": "filter_f32", "kind": "filter", "body": "planet", "h": 0.1, "b": 32, "prec": "f32", "k": 28, "degree": 8},
        # The plain double filter at the tests' block width.
        {"name": "filter_f64", "kind": "filter", "body": "planet", "h": 0.15, "b": 8, "prec": "f64", "k": 38, "degree": 6},
        # The smallest call in use: one mass solve on the smoke run's ball.
        {"name": "solve_ball", "kind": "solve", "body": "ball", "h": 0.45, "b": 8, "prec": "f64", "k": 40},
        # One Gram-Schmidt projection of a block against the benchmark's basis after 18 blocks.
        {"name": "project_bench", "kind": "project", "n": 1152807, "m": 576, "b": 32},
        # Rayleigh-Ritz of a served request's basis after 12 blocks.
        {"name": "ritz_request", "kind": "ritz", "body": "planet", "h": 0.1, "m": 192},
        # A whole slice: the ball's two lowest elastic multiplets, filtered block Lanczos in double.
        {"name": "slice_ball", "kind": "slice", "body": "ball", "h": 0.45, "b": 8, "k": 40, "degree": 100, "lo": 2.0, "hi": 3.0},
        # A new mesh arrives: assembly with its reference gravity, and the first products.
        {"name": "assemble", "kind": "assemble", "body": "planet", "h": 0.1, "b": 8},
        # The full operator (self-gravitation) applied to a block.
        {"name": "selfgrav", "kind": "apply", "body": "planet_sg", "h": 0.15, "b": 32, "prec": "mixed", "k": 20},
    ]


def draw(rng):
    """One more case of the same ranges. Largest cost: below the listed benchmark filter and projection."""
    def loguniform(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["filter", "filter", "filter", "solve", "project"])
    if kind == "project":
        n = int(loguniform(2000, 1.15e6))
        m = min(int(loguniform(8, 576)), n // 4)
        return {"kind": kind, "n": n, "m": m, "b": min(rng.choice([4, 8, 16, 31, 32]), m)}
    body = rng.choice(["planet", "planet", "planet", "ball"])
    h = round(loguniform(0.055, 0.3) if body == "planet" else loguniform(0.15, 0.45), 4)
    b = rng.choice([rng.randint(1, 64), 8, 16, 24, 32, 48, 64])
    prec = rng.choice(["mixed", "mixed", "mixed", "f32", "f64"])
    if prec == "f64" and h < 0.1:
        h = round(h + 0.05, 4)
    c = {"kind": kind, "body": body, "h": h, "b": b, "prec": prec, "k": rng.randint(18, 40)}
    if kind == "filter":
        # columns x inner steps x degree x nodes: at most 3/4 of the benchmark filter's
        most = 0.75 * 32 * 18 * 8 * (h / 0.05) ** 3
        c["b"] = min(b, max(1, int(most / (2 * c["k"]))))
        c["degree"] = max(2, min(rng.randint(4, 16), int(most / (c["b"] * c["k"]))))
    return c


# ----------------------------------------------------------------- what a program keeps
@functools.lru_cache(maxsize=None)
def _ctx():
    return nm.Context(torch.cuda.current_device())


def _mesh(body, h, seed):
    return homogeneous_ball(h=h, seed=seed) if body == "ball" else layered_planet(h=h, seed=seed)


@functools.lru_cache(maxsize=4)
def _problem(body, h):
    mesh, model = _mesh(body, h, 2)
    return nm.Problem(_ctx(), mesh, model, self_gravity=body == "planet_sg")


@functools.lru_cache(maxsize=16)
def _bounds(body, h):
    return _problem(body, h).spectrum_bounds(steps=40, k_M=40, seed=1)


def _normal(shape, seed, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


# ----------------------------------------------------------------- state and pass
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "project":
        # an orthonormal-like basis and a block to project, as the Lanczos step holds them
        n, m, b = case["n"], case["m"], case["b"]
        s["ctx"] = _ctx()
        s["V"] = _normal((n, m), seed).mul_(1.0 / math.sqrt(n))
        s["W"] = _normal((n, b), seed + 1)
        s["C"] = torch.zeros((b, m), device="cuda", dtype=torch.float64)   # column-major m x b
        s["D"] = torch.zeros((n, b), device="cuda", dtype=torch.float64)
        return s
    if kind == "assemble":
        # the arriving mesh's coordinates and coefficients are the seed's; its size is the kept problem's
        s["ctx"] = _ctx()
        s["mesh"], s["model"] = _mesh(case["body"], case["h"], 100 + seed % 100000)
        n = _problem(case["body"], case["h"]).n
        s["X"] = _normal((n, case["b"]), seed)
        s["KX"], s["MX"] = torch.zeros_like(s["X"]), torch.zeros_like(s["X"])
        return s
    P = s["P"] = _problem(case["body"], case["h"])
    if kind == "ritz":
        s["V"] = _normal((P.n, case["m"]), seed)
        s["hi"] = 1.1 * _bounds(case["body"], case["h"])[1]
        s["side"] = _normal((P.n,), 5)
        return s
    if kind == "slice":
        s["seed"] = int(seed) % (1 << 30)
        s["side"] = _normal((P.n,), 5)
        return s
    dtype = torch.float32 if case["prec"] == "f32" else torch.float64
    s["X"] = _normal((P.n, case["b"]), seed, dtype)
    s["Y"] = torch.zeros_like(s["X"])
    if kind == "filter":
        lo, hi = _bounds(case["body"], case["h"])
        s["gamma"], s["c"], s["e"] = nm.filter_design(lo, hi, 16.0, 42.25, case["degree"])
    return s


def _oriented(X, side):
    """Eigenvectors with their signs fixed against one direction, as a program that compares modes does."""
    return X * torch.sign(side @ X)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "filter":
        s["P"].filter_apply(s["gamma"], s["c"], s["e"], case["k"], s["X"], s["Y"], prec=PREC[case["prec"]])
        return s["Y"]
    if kind == "solve":
        s["P"].solve_M(s["X"], s["Y"], case["k"], prec=PREC[case["prec"]])
        return s["Y"]
    if kind == "apply":
        s["P"].apply_K(s["X"], s["Y"], k_P=case["k"], prec=PREC[case["prec"]])
        return s["Y"]
    if kind == "project":
        s["ctx"].gemm_tn(s["V"], s["W"], s["C"])
        s["ctx"].gemm_nn(s["V"], s["C"], s["D"])
        return {"C": s["C"], "D": s["D"]}
    if kind == "ritz":
        s["P"].set_interval(-1.0, s["hi"], nm.NM_UNIT_OMEGA2)
        r = s["P"].ritz(s["V"])
        out = {"lam": r.lam, "resid": r.resid, "X": _oriented(r.vectors(), s["side"])}
        r.free()
        return out
    if kind == "slice":
        s["P"].set_interval(case["lo"], case["hi"])
        r = s["P"].lanczos_slice(block=case["b"], degree=case["degree"], k_M=case["k"], k_P=case["k"], max_blocks=16,
                                 seed=s["seed"])
        out = {"lam": r.lam, "X": _oriented(r.vectors(), s["side"])}
        r.free()
        return out
    if kind == "assemble":
        P = nm.Problem(s["ctx"], s["mesh"], s["model"])
        P.apply_K(s["X"], s["KX"], k_P=40)
        P.apply_M(s["X"], s["MX"])
        g = P.gravity()
        P.free()
        return {"g": g, "KX": s["KX"], "MX": s["MX"]}
    raise ValueError(kind)


# ----------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "project":
        n, m, b = case["n"], case["m"], case["b"]
        return {"bytes": 8.0 * (2 * n * m + 2 * n * b + 2 * m * b), "flops": 4.0 * n * m * b}
    i = _problem(case["body"], case["h"]).info
    n, Nu, Np, zu, zp, ze = i["n"], i["Nu"], i["Np"], i["nnz_u"], i["nnz_p"], i["nnz_e"]
    b = case.get("b", case.get("m"))
    k = case.get("k", 80)
    vs = 4 if case.get("prec") == "f32" else 8        # bytes of a value of the blocks and of K_eff
    ms = 8 if case.get("prec", "f64") == "f64" else 4  # ... of the semi-iterations
    mixed = case.get("prec") == "mixed"

    def solve(nodes, z, comps):
        """One mass or pressure solve: (bytes of its steps, flops)."""
        steps = 2 * (k - 1) + 1 if mixed else k - 1
        step = z * (ms + 4) + 4 * (nodes + 1) + ms * nodes + 4 * ms * nodes * comps * b
        return steps * step, steps * (2.0 * z * comps * b + 6.0 * nodes * comps * b)

    K_bytes = zu * (9 * vs + 4) + 4 * (Nu + 1) + 2 * ze * (3 * vs + 4) + 2 * vs * n * b + 2 * vs * Np * b
    K_flops = 18.0 * zu * b + 12.0 * ze * b
    pb, pf = solve(Np, zp, 1) if Np else (0, 0.0)
    mb, mf = solve(Nu, zu, 3)
    once = zu * (9 * vs + ms + 8) + 2 * ze * (3 * vs + 4) + zp * (ms + 4) + 2 * vs * n * b
    # the steps of a recurrence stream whole blocks; only what outgrows the L2 cache has to cross HBM each time
    big = zu * (ms + 4) + 4 * ms * n * b > L2_BYTES
    if kind == "solve":
        return {"bytes": mb if big else zu * (ms + 4) + 2 * vs * n * b, "flops": mf}
    if kind == "filter":
        d = case["degree"]
        return {"bytes": d * (K_bytes + pb + mb + 4 * vs * n * b) if big else once, "flops": d * (K_flops + pf + mf)}
    if kind == "apply":
        pts = i["n_charges"]
        return {"bytes": once, "flops": K_flops + pf + float(pts) ** 2 * (9 + 2 * b)}
    if kind == "ritz":
        m = case["m"]
        return {"bytes": 3 * 8.0 * n * m + zu * 84, "flops": 8.0 * n * m * m + K_flops + pf + 6.0 * zu * m}
    if kind == "slice":
        passes = 13   # blocks the slice takes
        return {"bytes": once, "flops": passes * case["degree"] * (K_flops + pf + mf)}
    if kind == "assemble":
        return {"bytes": zu * 84.0 + i["nt"] * 60, "flops": 20.0 * Nu * i["nt"] + i["nt"] * 1e4}
    raise ValueError(kind)


# ----------------------------------------------------------------- the same in 64 bits
class _Exact:
    """The operators in plain torch FP64, on the matrices that the handle holds."""

    def __init__(self, P):
        self.P = P
        self.Nu, self.Np, self.n = P.Nu, P.Np, P.n
        self.A = self._csr(0, 3, 3, self.Nu, self.Nu)
        self.M = self._csr(1, 1, 1, self.Nu, self.Nu)
        self.dM = self._diag(1)
        if self.Np:
            self.Q = self._csr(2, 1, 1, self.Np, self.Np)
            self.dQ = self._diag(2)
            self.E = self._csr(3, 3, 1, self.Nu, self.Np)
            self.Et = self._csr(4, 1, 3, self.Np, self.Nu)

    def _csr(self, which, rb, cb, nr, nc):
        rp, col, val = self.P.export(which)
        rp, col, val = (torch.from_numpy(a).cuda() for a in (rp, col.astype(np.int64), val))
        cnt = rp[1:] - rp[:-1]
        crow = torch.zeros(nr * rb + 1, dtype=torch.int64, device="cuda")
        crow[1:] = torch.cumsum(torch.repeat_interleave(cnt * cb, rb), 0)
        row = torch.repeat_interleave(torch.arange(nr, device="cuda"), cnt)
        e = torch.arange(len(col), device="cuda")
        cols = torch.empty(len(col) * rb * cb, dtype=torch.int64, device="cuda")
        vals = torch.empty(len(col) * rb * cb, dtype=torch.float64, device="cuda")
        val = val.reshape(-1, rb, cb)
        for a in range(rb):
            at = crow[row * rb + a] + (e - rp[row]) * cb
            for c in range(cb):
                cols[at + c] = col * cb + c
                vals[at + c] = val[:, a, c]
        return torch.sparse_csr_tensor(crow, cols, vals, (nr * rb, nc * cb))

    def _diag(self, which):
        rp, col, val = self.P.export(which)
        row = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
        d = np.zeros(len(rp) - 1)
        on = row == col
        d[row[on]] = val[on]
        return torch.from_numpy(d).cuda()

    def m(self, X):
        return (self.M @ X.reshape(self.Nu, -1)).reshape(self.n, -1)

    def _cheb(self, apply, d, w, k):
        """k steps of the Jacobi-Chebyshev semi-iteration from zero (w: one row per node)."""
        th, de = 0.5 * (MASS_HI + MASS_LO), 0.5 * (MASS_HI - MASS_LO)
        f = 4.0 * (th / de) ** 2
        prev, x = torch.zeros_like(w), w / (d[:, None] * th)
        om = 2.0
        for _ in range(2, k + 1):
            om = 1.0 / (1.0 - om / f)
            prev, x = x, prev + om * (x - prev + (w - apply(x)) / (d[:, None] * th))
        return x

    def _solve(self, A, d, w, k, refine):
        apply = lambda x: A @ x  # noqa: E731
        x = self._cheb(apply, d, w, k)
        return x + self._cheb(apply, d, w - apply(x), k) if refine else x

    def solve_m(self, W, k, refine):
        return self._solve(self.M, self.dM, W.reshape(self.Nu, -1).contiguous(), k, refine).reshape(self.n, -1)

    def k_eff(self, X, k, refine):
        Y = self.A @ X
        if self.Np:
            Y += self.E @ self._solve(self.Q, self.dQ, self.Et @ X, k, refine)
        return Y


def _mass_product(P, mesh, model, X):
    """M X from the mesh: affine P2 tets, element mass matrix in closed form, in the problem's node order."""
    tet = torch.from_numpy(mesh.tet.astype(np.int64)).cuda()
    v = torch.from_numpy(mesh.xyz).cuda()[tet]
    vol = torch.linalg.det(v[:, 1:] - v[:, :1]).abs() / 6.0
    edges = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))
    ref = torch.empty((10, 10), dtype=torch.float64, device="cuda")
    for i in range(10):
        for j in range(10):
            if i < 4 and j < 4:
                r = 6.0 if i == j else 1.0
            elif i >= 4 and j >= 4:
                r = (8.0, 16.0, 32.0)[len(set(edges[i - 4]) & set(edges[j - 4]))]
            else:
                a, e = (i, edges[j - 4]) if i < 4 else (j, edges[i - 4])
                r = -4.0 if a in e else -6.0
            ref[i, j] = r / 420.0
    nv = len(mesh.xyz)
    pair = torch.stack([tet[:, list(e)] for e in edges], 1).sort(-1).values
    key = pair[..., 0] * nv + pair[..., 1]
    uniq, inv = torch.unique(key, return_inverse=True)
    p2 = torch.cat([tet, nv + inv.reshape(-1, 6)], 1)
    fluid = torch.from_numpy(mesh.region.astype(np.int64)).cuda() == 1
    touch = [torch.zeros(nv + len(uniq), dtype=torch.bool, device="cuda") for _ in range(2)]
    for f in (0, 1):
        touch[f][p2[fluid == bool(f)].reshape(-1)] = True
    ids = [torch.cumsum(touch[0].long(), 0) - 1, touch[0].sum() + torch.cumsum(touch[1].long(), 0) - 1]
    canon = torch.where(fluid[:, None], ids[1][p2], ids[0][p2])
    order = torch.from_numpy(P.unodes()[0]).cuda()          # canonical id of each internal node
    internal = torch.empty_like(order)
    internal[order] = torch.arange(len(order), device="cuda")
    at = internal[canon]
    x = X.reshape(P.Nu, -1)
    y = torch.zeros_like(x)
    w = (vol * torch.from_numpy(model.rho).cuda())[:, None, None]
    y.index_add_(0, at.reshape(-1), (w * (ref @ x[at])).reshape(-1, x.shape[1]))
    # node positions in internal order, and the point masses of the reference field
    mid = torch.from_numpy(mesh.xyz).cuda()
    ends = torch.stack([uniq // nv, uniq % nv], 1)
    pos = torch.cat([mid, mid[ends].mean(1)])[torch.from_numpy(P.unodes()[1]).cuda()]
    src = v.mean(1)
    g = torch.zeros_like(pos)
    mass = vol * torch.from_numpy(model.rho).cuda() * model.G
    for i in range(0, len(pos), 2048):
        r = pos[i:i + 2048, None, :] - src[None]
        g[i:i + 2048] = -(r * (mass / r.square().sum(-1) ** 1.5)[..., None]).sum(1)
    return y.reshape(X.shape), g


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        return None   # the charges of the self-gravitation term are not part of the handle
    s = prepare(case, seed)
    if kind == "project":
        C = s["V"].T @ s["W"]
        return {"C": C.T.contiguous(), "D": s["V"] @ C}
    if kind == "assemble":
        P = nm.Problem(s["ctx"], s["mesh"], s["model"])
        mx, g = _mass_product(P, s["mesh"], s["model"], s["X"])
        P.free()
        return {"g": g, "KX": None, "MX": mx}
    op = _Exact(s["P"])
    if kind == "slice":
        eye = torch.eye(op.n, dtype=torch.float64, device="cuda")
        lam, X = _dense_pencil(op.k_eff(eye, 80, False), op.m(eye))
        on = (lam >= case["lo"] ** 2) & (lam <= case["hi"] ** 2)
        return {"lam": lam[on], "X": _oriented(X[:, on], s["side"])}
    if kind == "ritz":
        V = s["V"]
        KV, MV = torch.cat([op.k_eff(c, 80, False) for c in V.split(64, 1)], 1), op.m(V)
        lam, S = _dense_pencil(V.T @ KV, V.T @ MV)
        KX, MX = KV @ S, MV @ S
        res = (KX - lam * MX).norm(dim=0) / (MX.norm(dim=0) * lam.abs().clamp(min=1e-3 * s["hi"]))
        return {"lam": lam, "resid": res, "X": _oriented(V @ S, s["side"])}
    X = s["X"].double()
    mixed = case["prec"] == "mixed"
    if kind == "solve":
        return op.solve_m(X, case["k"], mixed)
    g, c, e, k = s["gamma"], s["c"], s["e"], case["k"]
    prev, cur = None, X
    Z = g[0] * X
    for j in range(case["degree"]):
        t = op.solve_m(op.k_eff(cur, k, mixed), k, mixed) - c * cur
        nxt = t / e if prev is None else 2.0 / e * t - prev
        Z += g[j + 1] * nxt
        prev, cur = cur, nxt
    return Z


def _dense_pencil(H, G):
    """Eigenvalues and G-orthonormal eigenvectors of H x = lam G x."""
    L = torch.linalg.cholesky(0.5 * (G + G.T))
    B = torch.linalg.solve_triangular(L, 0.5 * (H + H.T), upper=False)
    B = torch.linalg.solve_triangular(L, B.T.contiguous(), upper=False)
    lam, Y = torch.linalg.eigh(0.5 * (B + B.T))
    return lam, torch.linalg.solve_triangular(L.T.contiguous(), Y, upper=True)
