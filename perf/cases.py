"""Workloads of the coded QR through its public entry points, for timing and comparison.

Five kinds, over the sizes that the configurations, tests and benchmark use:
  square  coded_qr_run on an m = n problem: encode, panels, one erasure event recovered on the
          way, post-orthogonalisation, solve (FP64, FP32 on the CUDA cores, FP32 in 3xTF32)
  tall    the step verbs on a tall problem: encode, panels, erasure, recovery, panels,
          post-orthogonalisation into the caller's buffer, least squares for k right-hand sides
  code    the checksum code alone: encode, lose tiles, recover them
  batch   many uneven tall-skinny FP32 problems in one batch handle, one erasure each
  grad    differentiable least squares: forward with one erasure, and the gradients

The matrices of square, tall and grad have a set 2-norm condition number (U diag(sigma) V^T with
geometric sigma); it is small enough in FP32 that two roundings of the same factors can be told
from an error.  code and batch take i.i.d. N(0,1) entries.
"""
import math
import random

import torch

from paper_2311_11943_gb300 import binding as B
from paper_2311_11943_gb300.autograd import coded_lstsq


def listed():
    return [
        # the smallest problem of the configurations in the library's default precision: FP64,
        # one node lost at panel 3; latency and launches
        dict(name="square f64 256", kind="square", m=256, n=256, p_r=4, p_c=4, f=1, b=32,
             dtype="f64", mma="simt", reorth=False, lost=1, panel=3, k=1, kappa=100.0),
        # FP64 on the 4096 x 4096 workload: the paper's own arithmetic
        dict(name="square f64 4096", kind="square", m=4096, n=4096, p_r=8, p_c=8, f=2, b=128,
             dtype="f64", mma="simt", reorth=False, lost=2, panel=9, k=1, kappa=100.0),
        # FP32 on the CUDA cores, an odd size
        dict(name="square f32 1420", kind="square", m=1420, n=1420, p_r=5, p_c=4, f=2, b=96,
             dtype="f32", mma="simt", reorth=False, lost=2, panel=4, k=1, kappa=4.0),
        # the 4096 x 4096 workload in mixed precision (register panel, look-ahead)
        dict(name="square 3xtf32 4096", kind="square", m=4096, n=4096, p_r=8, p_c=8, f=2, b=128,
             dtype="f32", mma="3xtf32", reorth=True, lost=2, panel=9, k=1, kappa=4.0),
        # the largest square: the grid, checksum count and panel width of the 16384 x 16384
        # workload at 8192 (at 16384 the FP32 sums over 20480 rows leave R 4e-5 off the exact
        # factor, more than two FP32 results of the same quality may be apart)
        dict(name="square 3xtf32 8192", kind="square", m=8192, n=8192, p_r=16, p_c=16, f=4,
             b=256, dtype="f32", mma="3xtf32", reorth=True, lost=4, panel=18, k=1, kappa=4.0),
        # the tall panels of the 16384 x 16384 workload (256 columns over many thread-block
        # clusters), on its first 2048 columns
        dict(name="tall 3xtf32 16384x2048", kind="tall", m=16384, n=2048, p_r=16, p_c=16, f=2,
             b=256, dtype="f32", mma="3xtf32", reorth=True, lost=2, panel=3, k=1, kappa=4.0),
        # small least squares with ragged rows and three right-hand sides
        dict(name="tall 3xtf32 1003x96", kind="tall", m=1003, n=96, p_r=6, p_c=4, f=2, b=32,
             dtype="f32", mma="3xtf32", reorth=False, lost=2, panel=1, k=3, kappa=4.0),
        # a mid-size tall problem with ragged rows and a ragged last panel
        dict(name="tall 3xtf32 6151x1320", kind="tall", m=6151, n=1320, p_r=8, p_c=6, f=2, b=128,
             dtype="f32", mma="3xtf32", reorth=True, lost=2, panel=5, k=1, kappa=4.0),
        # encode and decode on a matrix larger than the L2 cache
        dict(name="code f32 8192", kind="code", m=8192, n=8192, p_r=16, p_c=16, f=4, b=256,
             dtype="f32", mma="3xtf32", reorth=False, lost=4, panel=0, k=1, kappa=0.0),
        # the 512 uneven problems of the batch recipe, and a batch that does not fill the GPU
        dict(name="batch 512", kind="batch", count=512, shapes=4, m_lo=256, m_hi=8192, n_lo=32,
             n_hi=256, p_r=8, p_c=4, f=2, lost=2, graph=True, post_orth=False),
        dict(name="batch 40", kind="batch", count=40, shapes=7, m_lo=256, m_hi=2048, n_lo=32,
             n_hi=128, p_r=8, p_c=4, f=2, lost=1, graph=False, post_orth=True),
        # differentiable least squares on a batch of 16: forward with one erasure, gradients
        dict(name="grad 3xtf32 16x8192x1024", kind="grad", count=16, m=8192, n=1024, p_r=8, p_c=8,
             f=1, b=128, dtype="f32", mma="3xtf32", lost=1, panel=4, k=1, kappa=4.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["square", "square", "square", "tall", "tall", "code", "batch", "grad"])
    if kind == "batch":
        m_hi = _log(rng, 512, 8192)
        return dict(kind=kind, count=_log(rng, 4, 512), shapes=rng.randrange(1 << 20), m_lo=256,
                    m_hi=m_hi, n_lo=32, n_hi=min(256, m_hi // 8 // 4 * 4), p_r=8, p_c=4, f=2,
                    lost=rng.randint(1, 2), graph=rng.random() < 0.5,
                    post_orth=rng.random() < 0.5)
    f = rng.choice([1, 1, 2, 2, 4])
    p_c = rng.randint(max(4, 2 * f), 16)
    mode = rng.choice(["3xtf32", "3xtf32", "simt", "f64"])
    if kind == "grad":
        f, p_c = min(f, 2), min(p_c, 8)
        f64 = mode == "f64"
        n = max(1, _log(rng, 32, 256 if f64 else 1024) // p_c) * p_c
        m = _log(rng, 3 * n, 8 * n)
        return dict(kind=kind, count=rng.randint(1, 6), m=m, n=n, p_r=p_c, p_c=p_c, f=f,
                    b=rng.choice([16, 32, 64, 128]), dtype="f64" if f64 else "f32",
                    mma="simt" if f64 else "3xtf32", lost=f, panel=0, k=rng.randint(1, 2),
                    kappa=4.0)
    top = {"3xtf32": 7000, "simt": 2400, "f64": 3000}[mode]
    n = max(2, _log(rng, 160, top) // p_c) * p_c
    b = rng.choice([32, 48, 64, 96, 128, 128, 192, 256])
    p_r = p_c
    m = n
    if kind != "square":
        f = f if kind == "code" else min(f, 2)
        n = max(2, n // rng.randint(1, 4) // p_c) * p_c
        p_r = rng.randint(max(4, 2 * f), 16)
        m = min(n + rng.randint(1, 3 * n), max(n + 1, 12000))
    c = dict(kind=kind, m=m, n=n, p_r=p_r, p_c=p_c, f=f, b=b, dtype="f64" if mode == "f64" else "f32",
             mma="simt" if mode == "f64" else mode, reorth=mode == "3xtf32" and (kind == "tall" or rng.random() < 0.7),
             lost=f, panel=rng.randint(0, (n + b - 1) // b - 1), k=rng.randint(1, 2), kappa=4.0)
    if kind == "code":
        c.update(panel=0, kappa=0.0, reorth=False)
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _signs(n, g, dt):
    return torch.randint(0, 2, (n,), generator=g, device="cuda").to(dt) * 2 - 1


def _hartley(x):
    """The orthonormal discrete Hartley transform along the last dimension."""
    y = torch.fft.fft(x)
    return (y.real - y.imag) / math.sqrt(x.shape[-1])


def _matrix(m, n, kappa, dt, g):
    """A (m x n, column-major) = U diag(sigma) V^T, sigma_i = kappa^(-i/(n-1)), with U and V
    from Hartley transforms, random signs and a random choice of U's columns; kappa = 0: i.i.d.
    N(0,1)."""
    if not kappa:
        return torch.randn((n, m), generator=g, device="cuda", dtype=dt).t()
    sig = kappa ** (-torch.arange(n, device="cuda", dtype=torch.float64) / max(n - 1, 1))
    Vt = _hartley(torch.eye(n, device="cuda", dtype=dt)) * _signs(n, g, dt)[None, :]
    At = torch.zeros((n, m), device="cuda", dtype=dt)
    pick = torch.randperm(m, generator=g, device="cuda")[:n]
    At[:, pick] = Vt.t() * (sig.to(dt) * _signs(n, g, dt))[None, :]
    return (_hartley(At) * _signs(m, g, dt)[None, :]).contiguous().t()


def _dt(c):
    return torch.float64 if c.get("dtype") == "f64" else torch.float32


def _rhs(rows, k, dt, g):
    return torch.randn((k, rows), generator=g, device="cuda", dtype=dt).t()


def _tiles(c, rows, cols, count, rng):
    """`count` nodes of the rows x cols grid, no two in one grid row or column, whose tiles the
    code gives back without losing digits (the weight that a decode divides by is not small)."""
    G, Gh = _generator(c["f"], c["p_r"], c["p_c"])
    good_i = [i for i in range(rows) if i >= c["p_r"] or abs(G[0, i]) >= 0.4]
    good_j = [j for j in range(cols) if j >= c["p_c"] or Gh[j, 0] >= 0.4]
    return list(zip(rng.sample(good_i, count), rng.sample(good_j, count)))


def _shapes(c):
    rng = random.Random(c["shapes"])
    out = []
    while len(out) < c["count"]:
        m = rng.randint(c["m_lo"], c["m_hi"])
        n = rng.randint(c["n_lo"] // c["p_c"], c["n_hi"] // c["p_c"]) * c["p_c"]
        if m >= 4 * n:
            out.append((m, n))
    return out


def _inputs(c, seed):
    """The arrays of a case, the same for prepare and exact."""
    g, dt = _gen(seed), _dt(c)
    if c["kind"] == "batch":
        return [torch.randn((n, m), generator=g, device="cuda").t() for m, n in _shapes(c)]
    if c["kind"] == "grad":
        A = torch.stack([_matrix(c["m"], c["n"], c["kappa"], dt, g) for _ in range(c["count"])])
        y = torch.randn((c["count"], c["m"], c["k"]), generator=g, device="cuda", dtype=dt)
        W = [torch.randn(s, generator=g, device="cuda", dtype=dt) for s in (
            (c["count"], c["m"], c["n"]), (c["count"], c["n"], c["n"]),
            (c["count"], c["n"], c["k"]))]
        return A.contiguous(), y, W
    return _matrix(c["m"], c["n"], c["kappa"], dt, g), _rhs(c["m"], c["k"], dt, g)


GENERATOR_SEED = 11


def prepare(case, seed):
    c = case
    rng = random.Random(c["n_hi"] if c["kind"] == "batch" else c["m"] * 31 + c["n"])
    if c["kind"] == "grad":
        A, y, W = _inputs(c, seed)
        tiles = _tiles(c, c["p_r"] + c["f"], c["p_c"] + c["f"], c["lost"], rng)
        return dict(c=c, A=A.requires_grad_(), y=y.requires_grad_(), W=W,
                    erasures={c["panel"]: tiles})
    if c["kind"] == "batch":
        As = _inputs(c, seed)
        bt = B.CodedQRBatch(_shapes(c), c["p_r"], c["p_c"], c["f"], b=0, seed=GENERATOR_SEED)
        flat, plan = [], []
        for i, g in enumerate(bt.geo):
            for v, ld, cols in zip(bt.factors(i), (g["ldq"], g["ldr"]), (g["n"], g["N"])):
                # the columns of the factor as they lie in memory, with zero padding rows
                flat.append(torch.as_strided(v, (cols * ld,), (1,)))
                flat[-1].zero_()
            for t in _tiles(c, g["grid_rows"], g["grid_cols"], rng.randint(1, c["lost"]), rng):
                plan.append((i, g["panels"] // 2) + t)
        return dict(c=c, As=As, bt=bt, flat=flat, plan=plan)
    A, y = _inputs(c, seed)
    q = B.CodedQR(c["m"], c["n"], c["p_r"], c["p_c"], c["f"], c["b"], dtype=c["dtype"],
                  mma=c["mma"], reorth_block=c["reorth"], nrhs_max=c["k"], seed=GENERATOR_SEED)
    g = q.geo
    tiles = _tiles(c, g["grid_rows"], g["grid_cols"], c["lost"], rng)
    s = dict(c=c, A=A, y=y, q=q, tiles=tiles, x=B.colmajor_empty(c["n"], c["k"], _dt(c)))
    Q, R = q.factors()
    if c["kind"] == "square":
        s.update(plan=[(c["panel"],) + t for t in tiles], out=(Q[:g["m_pad"], :c["n"]], R))
    elif c["kind"] == "tall":
        s.update(out=(Q[:, : c["n"]], R), Qo=B.colmajor_empty(g["m_pad"], c["n"], _dt(c)))
    else:
        s.update(out=(Q,))
    for v in s["out"]:
        v.handle = q  # the factors are the handle's memory: keep it as long as they are kept
    return s


def run(state):
    s = state
    c = s["c"]
    if c["kind"] == "grad":
        Q, R, x = coded_lstsq(s["A"], s["y"], c["p_r"], c["p_c"], c["f"], c["b"],
                              seed=GENERATOR_SEED, erasures=s["erasures"], mma=c["mma"])
        loss = (s["W"][0] * Q).sum() + (s["W"][1] * R).sum() + (s["W"][2] * x).sum()
        gA, gy = torch.autograd.grad(loss, (s["A"], s["y"]))
        return dict(Q=Q, R=R, x=x, gA=gA, gy=gy)
    if c["kind"] == "batch":
        s["bt"].run(s["As"], s["plan"], graph=c["graph"], post_orth=c["post_orth"])
        return dict(Q=torch.cat(s["flat"][0::2]), R=torch.cat(s["flat"][1::2]))
    q = s["q"]
    if c["kind"] == "square":
        q.run(s["A"], s["y"], s["x"], plan=s["plan"])
        return dict(Q=s["out"][0], R=s["out"][1], x=s["x"])
    q.encode(s["A"])
    if c["kind"] == "code":
        q.inject(s["tiles"])
        q.recover()
        return dict(Q=s["out"][0])
    if c["panel"]:
        q.factor(0, c["panel"])
    q.inject(s["tiles"])
    q.recover()
    q.factor(c["panel"], -1)
    q.post_orth(s["Qo"])
    q.solve_ls(s["y"], s["x"])
    return dict(Q=s["out"][0], R=s["out"][1], Qo=s["Qo"], x=s["x"])


# ------------------------------------------------------------------ what a pass cannot do without
def _one(m, n, p_r, p_c, f, e, k=0, qo=False):
    """(bytes, flops) of one coded QR: A and the right-hand sides in, the coded factors out."""
    mb = -(-m // p_r)
    M, N = (p_r + f) * mb, n + f * (n // p_c)
    out = M * N + N * N + (p_r * mb * n if qo else 0)
    return e * (m * n + out + k * (m + n)), 2.0 * M * n * (2 * N - n)


def work(case):
    c = case
    e = 8 if c.get("dtype") == "f64" else 4
    if c["kind"] == "batch":
        each = [_one(m, n, c["p_r"], c["p_c"], c["f"], 4) for m, n in _shapes(c)]
        return dict(bytes=float(sum(x[0] for x in each)), flops=float(sum(x[1] for x in each)))
    if c["kind"] == "code":
        b, _ = _one(c["m"], c["n"], c["p_r"], c["p_c"], c["f"], e)
        N = c["n"] + c["f"] * (c["n"] // c["p_c"])
        return dict(bytes=float(b - e * N * N), flops=4.0 * c["f"] * c["m"] * c["n"])
    b, fl = _one(c["m"], c["n"], c["p_r"], c["p_c"], c["f"], e, c["k"], c["kind"] != "square")
    if c["kind"] == "grad":
        # the reverse rule: two m n^2 products and a triangular solve beside the forward pass
        return dict(bytes=float(c["count"] * (b + 3 * e * c["m"] * c["n"])),
                    flops=float(c["count"]) * (fl + 5.0 * c["m"] * c["n"] ** 2))
    return dict(bytes=float(b), flops=float(fl))


# ------------------------------------------------------------------ the same in plain 64-bit torch
def _generator(f, p_r, p_c):
    """G~ (f x p_r) and G~_h (p_c x f) in Python: V~ and G~_h from SplitMix64 as Unif(0,1),
    G~ = [-1/2 V~ V~^T, V~]."""
    s, mask = GENERATOR_SEED, (1 << 64) - 1

    def unif():
        nonlocal s
        while True:
            s = (s + 0x9E3779B97F4A7C15) & mask
            z = s
            z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            z = (z ^ (z >> 31)) >> 11
            if z:
                return z * 2.0 ** -53
    V = torch.tensor([[unif() for _ in range(p_r - f)] for _ in range(f)], dtype=torch.float64)
    Gh = torch.tensor([[unif() for _ in range(f)] for _ in range(p_c)], dtype=torch.float64)
    return torch.cat([-0.5 * V @ V.T, V], 1), Gh


def _checksums(G, X, mb):
    """(G~ (x) I_mb) X for the block rows of X."""
    return torch.einsum("it,trc->irc", G.to(X), X.reshape(G.shape[1], mb, -1)).reshape(-1, X.shape[1])


def _g0(G, X, mb):
    """G_0 X, G_0 = [[I + G~_1, V~], [V~^T, -I]] on the block rows of X."""
    f, p = G.shape
    K = torch.zeros((p, p), dtype=torch.float64)
    K[:f], K[f:, :f] = G, G[:, f:].t()
    K[:f, :f] += torch.eye(f)
    K[f:, f:] = -torch.eye(p - f)
    return _checksums(K, X, mb)


def _qr(X, passes):
    """Thin QR with a positive diagonal, by Cholesky of X^T X (twice for full 64 bits)."""
    R = None
    for _ in range(passes):
        n = X.shape[1]
        S = torch.empty((n, n), dtype=X.dtype, device=X.device)
        for j in range(0, n, 2048):  # the upper half only
            S[: j + 2048, j : j + 2048] = X[:, : j + 2048].t() @ X[:, j : j + 2048]
        C = torch.linalg.cholesky(torch.triu(S) + torch.triu(S, 1).t()).t().contiguous()
        X = torch.linalg.solve_triangular(C, X, upper=True, left=False)
        R = C if R is None else C @ R
    return X, R


def _factor(A, p_r, p_c, f, passes=2):
    """The coded factors of A in 64 bits: Q~ (its n columns that are not zero), R~, G~ and mb."""
    G, Gh = _generator(f, p_r, p_c)
    m, n = A.shape
    mb = -(-m // p_r)
    X = torch.zeros((p_r * mb, n), dtype=torch.float64, device="cuda")
    X[:m] = A
    X = torch.cat([X, _checksums(G, X, mb)])
    Q, R1 = _qr(X, passes)
    nb = n // p_c
    R2 = torch.einsum("rtc,tl->rlc", R1.reshape(n, p_c, nb), Gh.to(R1)).reshape(n, f * nb)
    N = n + f * nb
    R = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    R[:n, :n], R[:n, n:] = R1, R2
    return Q, R, G, mb


def _exact_grad(c, seed):
    A0, y0, W = _inputs(c, seed)
    W = [w.double() for w in W]
    mb = -(-c["m"] // c["p_r"])
    G, _ = _generator(c["f"], c["p_r"], c["p_c"])
    out = {k: [] for k in ("Q", "R", "x", "gA", "gy")}
    for i in range(c["count"]):
        A = A0[i].double().requires_grad_()
        y = y0[i].double().requires_grad_()
        pad = torch.zeros((c["p_r"] * mb - c["m"], c["n"]), dtype=torch.float64, device="cuda")
        Q, R = torch.linalg.qr(_g0(G, torch.cat([A, pad]), mb))
        d = torch.sign(torch.diagonal(R)).detach()
        Q, R = (Q * d)[: c["m"]], torch.triu(d[:, None] * R)
        x = torch.linalg.solve(A.t() @ A, A.t() @ y)
        loss = (W[0][i] * Q).sum() + (W[1][i] * R).sum() + (W[2][i] * x).sum()
        gA, gy = torch.autograd.grad(loss, (A, y))
        for k, v in zip(out, (Q, R, x, gA, gy)):
            out[k].append(v.detach())
    return {k: torch.stack(v) for k, v in out.items()}


def exact(case, seed):
    c = case
    if c["kind"] == "grad":
        return _exact_grad(c, seed)
    if c["kind"] == "batch":
        Qs, Rs = [], []
        for A in _inputs(c, seed):
            Q, R, G, mb = _factor(A.double(), c["p_r"], c["p_c"], c["f"])
            if c["post_orth"]:
                Q[: c["p_r"] * mb] = _g0(G, Q[: c["p_r"] * mb], mb)
            for X, to in ((Q, Qs), (R, Rs)):
                ld = -(-X.shape[0] // 32) * 32
                Y = torch.zeros((X.shape[1], ld), dtype=torch.float64, device="cuda")
                Y[:, : X.shape[0]] = X.t()
                to.append(Y.reshape(-1))
        return dict(Q=torch.cat(Qs), R=torch.cat(Rs))
    A, y = _inputs(c, seed)
    if c["kind"] == "code":
        G, Gh = _generator(c["f"], c["p_r"], c["p_c"])
        mb = -(-c["m"] // c["p_r"])
        X = torch.zeros((c["p_r"] * mb, c["n"]), dtype=torch.float64, device="cuda")
        X[: c["m"]] = A
        X = torch.cat([X, _checksums(G, X, mb)])
        H = torch.einsum("rtc,tl->rlc", X.reshape(X.shape[0], c["p_c"], -1), Gh.to(X))
        return dict(Q=torch.cat([X, H.reshape(X.shape[0], -1)], 1))
    # one pass of Cholesky QR holds 64 bits less log2(kappa^2): enough beside FP32 factors
    Q, R, G, mb = _factor(A, c["p_r"], c["p_c"], c["f"], 2 if c["dtype"] == "f64" else 1)
    mp, n = c["p_r"] * mb, c["n"]
    Qo = _g0(G, Q[:mp], mb)
    if c["kind"] == "square":
        # G_0 A x = G_0 y and G_0 A = Qo R
        yo = _g0(G, y.double(), mb)
        x = torch.linalg.solve_triangular(R[:n, :n], Qo.t() @ yo, upper=True)
        return dict(Q=Qo, R=R, x=x)
    Qa, Ra = _qr(A.double(), 2)
    x = torch.linalg.solve_triangular(Ra, Qa.t() @ y.double(), upper=True)
    return dict(Q=Q, R=R, Qo=Qo, x=x)
