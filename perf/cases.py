"""The work that users of this library have it do: M = L + S decompositions of matrices on the GPU (and in
host memory) through the Python binding's entry points, over the range of sizes, ranks, storage
types and options the library takes in earnest.

A case is a dict of plain values; `kind` selects the call:
  adm      one FR-ADM solve (solve_torch), float64 or mixed precision
  noalloc  the same through sfr_solve_noalloc, into buffers the caller holds
  host     the same on pinned host buffers (M in, S and the factors out)
  nys      FR-Nys with l sampled columns and rows (solve_torch, nys_l)
  stream   many uneven requests queued on one context with the grouped engine (submit / poll)
  tsvd     a rank-r truncated SVD by FixedRankOptFull (opt_full_torch)

Float64 solves return their factors U, B, V and S.  Mixed-precision solves and FR-Nys return L and S in
float32: the problem determines L = U B V^T, but not the rotation that U, B and V share
((U Q)(Q^T B Q)(V Q)^T is the same L), which bfloat16 storage moves by 1e-4.
"""
import math
import random

import torch

from paper_1503_03004_gb300 import binding as B

RHO, TOL, MU_MAX, MAX_ITER = 1.5, 1e-9, 1e9, 300
STORE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
CODE = {"f64": B.F64, "f32": B.F32, "bf16": B.BF16}


def listed():
    return [
        # the smallest calls: a fixed pool owns the device memory, the solve is all latency
        {"name": "noalloc 200x160 r5 f64", "kind": "noalloc", "m": 200, "n": 160, "r": 5, "store": "f64", "prec": "fp64",
         "p": 0.08, "amp": 50.0},
        # the plain single problem in float64
        {"name": "square 500 r25 f64", "kind": "adm", "m": 500, "n": 500, "r": 25, "store": "f64", "prec": "fp64",
         "p": 0.1, "amp": 50.0},
        # a row of the paper's scale experiment (Sec. 5.1): unit outliers, mu_0 from ||M||_2
        {"name": "table 2000 r10 f64", "kind": "adm", "m": 2000, "n": 2000, "r": 10, "store": "f64", "prec": "fp64",
         "p": 0.1, "amp": 1.0},
        # a large float64 solve of float32 data at the highest rank
        {"name": "square 4096 r64 f32 fp64", "kind": "adm", "m": 4096, "n": 4096, "r": 64, "store": "f32", "prec": "fp64",
         "p": 0.05, "amp": 50.0},
        # the large square problem in mixed precision
        {"name": "square 16384 r64 bf16", "kind": "adm", "m": 16384, "n": 16384, "r": 64, "store": "bf16", "prec": "mixed",
         "p": 0.05, "amp": 50.0},
        # an ordinary rectangular bfloat16 matrix, not a multiple of any tile
        {"name": "rect 3000x2040 r48 bf16", "kind": "adm", "m": 3000, "n": 2040, "r": 48, "store": "bf16", "prec": "mixed",
         "p": 0.06, "amp": 50.0},
        # float32 storage above rank 32 in mixed precision
        {"name": "square 2048 r40 f32", "kind": "adm", "m": 2048, "n": 2048, "r": 40, "store": "f32", "prec": "mixed",
         "p": 0.05, "amp": 50.0},
        # photometric stereo: a million pixels, 40 images, rank 3
        {"name": "photometric 1048576x40 r3", "kind": "adm", "m": 1048576, "n": 40, "r": 3, "store": "f32", "prec": "mixed",
         "scene": True},
        # spectral clustering: 20 clusters, Nystrom sampling
        {"name": "affinity 32768 r20 l2048", "kind": "nys", "n": 32768, "r": 20, "l": 2048, "store": "bf16"},
        # a serving load: uneven requests, most of them with rows off 16-byte boundaries
        {"name": "stream of 48 bf16", "kind": "stream", "count": 48, "sizes": 1004, "store": "bf16"},
        # truncated SVD of the large matrix, five steps
        {"name": "tsvd 16384 r64 bf16", "kind": "tsvd", "m": 16384, "n": 16384, "r": 64, "store": "bf16", "steps": 5,
         "p": 0.05, "amp": 50.0},
        # data that lives in host memory
        {"name": "host 4096x2048 r32 bf16", "kind": "host", "m": 4096, "n": 2048, "r": 32, "store": "bf16", "prec": "mixed",
         "p": 0.05, "amp": 50.0},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["f64", "f64", "f64", "tc", "tc", "simt", "simt", "simt", "f32", "tall", "nys", "stream", "tsvd", "host",
                       "noalloc"])
    p = round(rng.uniform(0.02, 0.1), 3)
    if kind in ("f64", "noalloc"):
        top = 260 if kind == "noalloc" else 2500
        m, n = log(100, top), log(100, top)
        r = min(log(2, 64), min(m, n) // 8)
        return {"kind": "noalloc" if kind == "noalloc" else "adm", "m": m, "n": n, "r": r, "prec": "fp64", "p": p,
                "amp": 50.0, "store": rng.choice(["f64", "f64", "f32", "bf16"])}
    if kind == "tc":
        return {"kind": "adm", "m": 8 * log(64, 1024), "n": 8 * log(64, 1024), "r": rng.randint(33, 64), "store": "bf16",
                "prec": "mixed", "p": p, "amp": 50.0}
    if kind in ("simt", "host"):
        m, n = log(400, 6000), log(400, 3000)
        return {"kind": "host" if kind == "host" else "adm", "m": m, "n": n, "r": log(3, 32),
                "store": rng.choice(["f32", "bf16"]), "prec": "mixed", "p": p, "amp": 50.0}
    if kind == "f32":
        return {"kind": "adm", "m": log(500, 3000), "n": log(500, 3000), "r": rng.randint(33, 60), "store": "f32",
                "prec": "mixed", "p": p, "amp": 50.0}
    if kind == "tall":
        side = log(64, 700)
        return {"kind": "adm", "m": side * side, "n": rng.randint(24, 64), "r": 3, "store": "f32", "prec": "mixed", "scene": True}
    if kind == "nys":
        n = log(2000, 16000)
        r = rng.randint(8, 24)
        return {"kind": "nys", "n": n, "r": r, "l": min(16 * r + rng.randint(0, 300), n // 4), "store": "bf16"}
    if kind == "stream":
        return {"kind": "stream", "count": log(4, 48), "sizes": rng.randint(1, 1 << 20), "store": rng.choice(["bf16", "f32"])}
    return {"kind": "tsvd", "m": 8 * log(64, 1500), "n": 8 * log(64, 1500), "r": rng.randint(33, 64), "store": "bf16",
            "steps": rng.randint(3, 8), "p": p, "amp": 50.0}


# ---------------------------------------------------------------- inputs
def _planted(g, m, n, r, p, amp, dtype):
    """L0 + S0: standard normal factors, uniform outliers in [-amp, amp] on a Bernoulli(p) support."""
    t = torch.float64 if dtype == torch.float64 else torch.float32
    u = torch.randn((m, r), generator=g, device="cuda", dtype=t)
    v = torch.randn((n, r), generator=g, device="cuda", dtype=t)
    s = torch.rand((m, n), generator=g, device="cuda", dtype=t).mul_(2 * amp).sub_(amp)
    s.mul_(torch.rand((m, n), generator=g, device="cuda") < p)
    return s.addmm_(u, v.T).to(dtype)


def _scene(g, m, n, dtype):
    """Lambertian images (pixels x images) of a smooth height field, with attached shadows and specular outliers."""
    side = math.isqrt(m)
    ax = torch.linspace(0, 1, side, device="cuda", dtype=torch.float64)
    rnd = torch.rand((16, 4), generator=g, device="cuda", dtype=torch.float64)
    nx = torch.zeros((side, side), device="cuda", dtype=torch.float64)
    ny = torch.zeros_like(nx)
    for a, b, c, d in rnd.tolist():
        cx, cy, w, h = 0.05 + 0.9 * a, 0.05 + 0.9 * b, 0.05 + 0.15 * c, 0.6 * d - 0.3
        dx, dy = ax[None, :] - cx, ax[:, None] - cy
        bump = h * torch.exp(-(dx * dx + dy * dy) / (2 * w * w)) / (w * w)
        nx += bump * dx
        ny += bump * dy
    N = torch.stack([nx, ny, torch.ones_like(nx)], dim=-1).reshape(-1, 3)
    N /= N.norm(dim=1, keepdim=True)
    N *= 0.2 + 0.8 * torch.rand((m, 1), generator=g, device="cuda", dtype=torch.float64)
    lo = math.sin(math.radians(15.0))
    z = lo + (1 - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    az = 2 * math.pi * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    xy = (1 - z * z).sqrt()
    lights = torch.stack([xy * az.cos(), xy * az.sin(), z], dim=1)
    M = (N @ lights.T).clamp_(min=0)
    spec = torch.rand((m, n), generator=g, device="cuda", dtype=torch.float64)
    M += torch.where(torch.rand((m, n), generator=g, device="cuda") < 0.1, spec, torch.zeros_like(spec))
    return M.to(dtype)


def _affinity(g, n, k, dtype):
    """Symmetric affinity of k clusters: 0.8 within, 0.05 across, noise, and 3 % symmetric outliers."""
    label = (torch.arange(n, device="cuda") % k)[torch.randperm(n, generator=g, device="cuda")]
    same = label[:, None] == label[None, :]
    up = torch.randn((n, n), generator=g, device="cuda", dtype=torch.float32).triu_()
    up *= torch.where(same, 0.05, 0.02)
    up += torch.where(same, 0.8, 0.05)
    hit = torch.rand((n, n), generator=g, device="cuda", dtype=torch.float32) < 0.03
    up += hit * torch.rand((n, n), generator=g, device="cuda", dtype=torch.float32)
    up.triu_()
    return (up + up.triu(1).T).to(dtype)


def _mu0(case, M):
    """0.05 for outliers of size 50, 1 for data in [0, 1], 1.25 / ||M||_2 for unit outliers (the paper's scale experiment)."""
    if "amp" not in case:
        return 1.0
    if case["amp"] > 1:
        return 0.05
    A, x = M.double(), torch.ones((M.shape[1], 1), device=M.device, dtype=torch.float64)
    for _ in range(30):
        x = A.T @ (A @ x)
        x = x / x.norm()
    return 1.25 / float((A @ x).norm())


def _matrix(case, seed):
    g = torch.Generator("cuda").manual_seed(int(seed))
    dt = STORE[case["store"]]
    if case.get("scene"):
        return _scene(g, case["m"], case["n"], dt)
    if case["kind"] == "nys":
        return _affinity(g, case["n"], case["r"], dt)
    return _planted(g, case["m"], case["n"], case["r"], case["p"], case["amp"], dt)


def _stream_shapes(case):
    """(m, n, r, p) of the requests of a stream: sizes belong to the case, values to the seed."""
    rnd = random.Random(case["sizes"])
    out = []
    for _ in range(case["count"]):
        m, n = rnd.randint(256, 8192), rnd.randint(16, 512)
        r = rnd.choice([r for r in (3, 5, 10, 25) if r <= max(3, n // 5)])
        out.append((m, n, r, rnd.uniform(0.02, 0.1)))
    return out


def _stream_matrices(case, seed):
    g = torch.Generator("cuda").manual_seed(int(seed))
    return [_planted(g, m, n, r, p, 50.0, STORE[case["store"]]) for m, n, r, p in _stream_shapes(case)]


# ---------------------------------------------------------------- prepare and run
_CONTEXTS = {}


def _context(grouped):
    """The library handles a program keeps: one for single solves, one that serves requests in groups."""
    if grouped not in _CONTEXTS:
        _CONTEXTS[grouped] = B.Context(0, max_batch=256) if grouped else B.Context(0)
    return _CONTEXTS[grouped]


def _prec(case):
    return B.PREC_FP64 if case["prec"] == "fp64" else B.PREC_MIXED


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "ctx": _context(kind == "stream")}
    if kind == "stream":
        Ms = _stream_matrices(case, seed)
        shapes = _stream_shapes(case)
        area = sum(m * n for m, n, _, _ in shapes)
        st["S"] = torch.empty(area, device="cuda", dtype=torch.float32)
        st["L"] = torch.empty(area, device="cuda", dtype=torch.float32)
        st["M"], st["calls"], at = Ms, [], 0
        for M, (m, n, r, _) in zip(Ms, shapes):
            prob = B.make_problem(m=m, n=n, r=r, M_ptr=M.data_ptr(), m_dtype=CODE[case["store"]], mu0=0.05, rho=RHO,
                                  tol=TOL, max_iter=MAX_ITER, precision=B.PREC_MIXED)
            res = B.make_result(S_ptr=st["S"][at:].data_ptr(), L_ptr=st["L"][at:].data_ptr(), s_dtype=B.F32, lds=n)
            st["calls"].append((prob, res))
            at += m * n
        torch.cuda.synchronize()
        return st
    M = _matrix(case, seed)
    st["M"] = M
    if kind == "tsvd":
        return st
    st["mu0"] = _mu0(case, M)
    m, n = M.shape
    r = case["r"]
    if kind == "nys":
        st["perm"] = torch.randperm(n, generator=torch.Generator("cuda").manual_seed(int(seed) + 1), device="cuda")
        return st
    if kind in ("noalloc", "host"):
        host = kind == "host"
        where = {"pin_memory": True} if host else {"device": "cuda"}
        if host:
            st["M"] = M = torch.empty((m, n), dtype=M.dtype, pin_memory=True).copy_(M)
        fp64 = case["prec"] == "fp64"
        f64, out = dict(where, dtype=torch.float64), dict(where, dtype=torch.float64 if fp64 else torch.float32)
        st["out"] = {"U": torch.empty((m, r), **f64), "B": torch.empty((r, r), **f64), "V": torch.empty((n, r), **f64),
                     "S": torch.empty((m, n), **out), "L": torch.empty((m, n), **out)}
        at = {k + "_ptr": t.data_ptr() for k, t in st["out"].items()}
        st["prob"] = B.make_problem(m=m, n=n, r=r, M_ptr=M.data_ptr(), m_dtype=CODE[case["store"]], mu0=st["mu0"], rho=RHO,
                                    tol=TOL, max_iter=MAX_ITER, precision=_prec(case),
                                    mem=B.MEM_HOST if host else B.MEM_DEVICE)
        st["res"] = B.make_result(s_dtype=B.F64 if fp64 else B.F32, lds=n, **at)
        torch.cuda.synchronize()
    return st


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "stream":
        tickets = [ctx.submit(prob, res) for prob, res in state["calls"]]
        for t in tickets:
            st = ctx.poll(t)
            if st != B.OK:
                raise B.SfrError(st, ctx.last_error())
        return {"L": state["L"], "S": state["S"]}
    if kind == "tsvd":
        sol = B.opt_full_torch(ctx, state["M"], case["r"], max_iter=case["steps"], precision=B.PREC_MIXED)
        return {"U": sol.U.float(), "B": sol.B.float(), "V": sol.V.float()}
    if kind in ("noalloc", "host"):
        st = (ctx.solve_noalloc if kind == "noalloc" else ctx.solve)(state["prob"], state["res"])
        if st != B.OK:
            raise B.SfrError(st, ctx.last_error())
        got = state["out"]
    else:
        fp64 = case.get("prec") == "fp64"
        kw = dict(nys_l=case["l"], nys_perm=state["perm"]) if kind == "nys" else {}
        sol = B.solve_torch(ctx, state["M"], case["r"], precision=B.PREC_FP64 if fp64 else B.PREC_MIXED,
                            s_dtype=B.F64 if fp64 else B.F32, want_L=not fp64, mu0=state["mu0"], rho=RHO, tol=TOL,
                            max_iter=MAX_ITER, **kw)
        got = {"U": sol.U, "B": sol.B, "V": sol.V, "S": sol.S, "L": sol.L}
    return {k: got[k] for k in ("UBVS" if case.get("prec") == "fp64" else "LS")}


# ---------------------------------------------------------------- work
def work(case):
    """M read once, the results written once; the three thin products of each of about 45 iterations."""
    es = {"f64": 8, "f32": 4, "bf16": 2}[case["store"]]
    kind = case["kind"]
    if kind == "stream":
        b = f = 0.0
        for m, n, r, _ in _stream_shapes(case):
            b += m * n * (es + 8.0)
            f += 45 * 6.0 * m * n * r
        return {"bytes": b, "flops": f}
    r = case["r"]
    if kind == "nys":
        n, l = case["n"], case["l"]
        return {"bytes": n * n * (es + 8.0), "flops": 2 * 40 * 6.0 * n * l * r + 2.0 * n * n * r}
    m, n = case["m"], case["n"]
    thin = 8.0 * (m + n + r) * r
    if kind == "tsvd":
        return {"bytes": es * m * n + thin, "flops": case["steps"] * 4.0 * m * n * r}
    return {"bytes": m * n * (es + 8.0) + thin, "flops": 45 * 6.0 * m * n * r}


# ---------------------------------------------------------------- the same in 64 bits
def _polar(A):
    w, E = torch.linalg.eigh(A.T @ A)
    return A @ ((E * w.rsqrt()) @ E.T)


def _step(X, Bm, V):
    U = _polar(X @ V @ Bm)
    W = X.T @ U
    V = _polar(W @ Bm)
    Bm = W.T @ V
    return U, (Bm + Bm.T) / 2, V


def _fr_adm(M, r, mu0):
    """Algorithm 1 with every matrix dense in float64: U, B, V, L, S."""
    n = M.shape[1]
    eye = {"dtype": torch.float64, "device": M.device}
    Bm, V = torch.eye(r, **eye), torch.eye(n, r, **eye)
    S, Y, mu, scale = torch.zeros_like(M), torch.zeros_like(M), mu0, float(M.norm())
    for _ in range(MAX_ITER):
        X = M - S
        X.add_(Y, alpha=1 / mu)
        U, Bm, V = _step(X, Bm, V)
        L = U @ Bm @ V.T
        Z = M - L
        S = torch.nn.functional.softshrink(Z.add(Y, alpha=1 / mu), 1 / mu)
        Z -= S
        Y.add_(Z, alpha=mu)
        mu = min(MU_MAX, RHO * mu)
        if float(Z.norm()) <= TOL * scale:
            break
    return U, Bm, V, L, S


def exact(case, seed):
    kind = case["kind"]
    if kind == "stream":
        got = [_fr_adm(M.double(), r, 0.05)[3:] for M, (_, _, r, _) in zip(_stream_matrices(case, seed), _stream_shapes(case))]
        return {"L": torch.cat([L.reshape(-1) for L, _ in got]), "S": torch.cat([S.reshape(-1) for _, S in got])}
    st = prepare(case, seed)
    M = st["M"].cuda().double()
    r = case["r"]
    if kind == "tsvd":
        Bm, V = torch.eye(r, dtype=M.dtype, device="cuda"), torch.eye(M.shape[1], r, dtype=M.dtype, device="cuda")
        for _ in range(case["steps"]):
            U, Bm, V = _step(M, Bm, V)
        return {"U": U, "B": Bm, "V": V}
    if kind == "nys":
        l, perm = case["l"], st["perm"]
        U, Bl, _, _, _ = _fr_adm(M[perm, :l], r, st["mu0"])
        T = _fr_adm(M[perm[:l], :], r, st["mu0"])
        # L_L (L_L[:l, :l])^+ L_T with L_L = U Bl Vl^T: U Bl A^+ L_T, A = U[:l] Bl of full column rank
        core = torch.linalg.lstsq(U[:l] @ Bl, T[0]).solution @ T[1]
        L = torch.empty_like(M)
        L[perm] = (U @ (Bl @ core)) @ T[2].T
        return {"L": L, "S": M - L}
    got = dict(zip("UBVLS", _fr_adm(M, r, st["mu0"])))
    return {k: got[k] for k in ("UBVS" if case["prec"] == "fp64" else "LS")}
