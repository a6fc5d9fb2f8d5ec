"""Performance cases of the EXCMG solver: the calls a user of the package makes.

Each case is one pass through the public entry points on inputs made on the
GPU from a seed.  The operations and what they stand for in real use:

  apply    stencil_apply: one application of A_h or its transpose to a node
           array (residuals, a user's own Krylov method)
  bicg     bicg_solve: a fixed number of Bi-CG iterations on one grid from a
           starting guess (smoothing, a level of the cascade, a capped solve)
  setup    what Alg. 1 does on entering a level: right-hand side assembly and
           the extrapolated, interpolated initial guess with its boundary
  true     midpoint_extrapolate: the final extrapolation on the finest grid
  solve    excmg_solve: the whole cascade to a relative residual tolerance
  mixed    excmg_solve in the FP32-correction / FP64-refinement precision
  batch    many independent solves through the batch engine
  bicg2d   bicg_solve2d: the 2D problem's Bi-CG

All grid functions are float64 (the ABI's only type); the mixed case runs its
inner solves in float32.  "kind" is the kind of Dirichlet data (1 or 2).
"""
import math

import numpy as np
import torch

from paper_1901_05118_gb300 import binding as B

F8 = torch.float64
DEV = "cuda"


def listed():
    return [
        # a tiny grid: one application is all launch and synchronisation cost
        dict(name="apply_17", op="apply", n=17, kind=2, transpose=False),
        # the operator at the benchmark's size, transposed (A^T of Alg. 2)
        dict(name="apply_512_t", op="apply", n=512, kind=1, transpose=True),
        # Bi-CG where a level's vectors live in cache: most iterations of a
        # cascade are spent on such grids
        dict(name="bicg_64", op="bicg", n=64, kind=1, iters=200),
        # a ragged grid of the middle range
        dict(name="bicg_133", op="bicg", n=133, kind=2, iters=60),
        # the finest level of the 512^3 benchmark (22 iterations there)
        dict(name="bicg_512", op="bicg", n=512, kind=1, iters=16),
        # entering the finest level of the benchmark
        dict(name="setup_512", op="setup", n=512, kind=1),
        # the final extrapolation of a 256^3 solve (the largest request size
        # of the serving stream)
        dict(name="true_256", op="true", n=256),
        # the small workload: 4^3 .. 32^3, tol 1e-10, first-kind data
        dict(name="solve_32", op="solve", n=32, coarsest=4, kind=1, tol=1e-10, problem="sines"),
        # the headline workload: 8^3 .. 512^3, tol 1e-10
        dict(name="solve_512", op="solve", n=512, coarsest=8, kind=1, tol=1e-10, problem="exp"),
        # FP32 correction solves inside FP64 refinement
        dict(name="mixed_48", op="mixed", n=48, coarsest=6, kind=2, tol=1e-12, problem="exp"),
        # a burst of small requests, kinds and sizes mixed
        dict(name="batch_8", op="batch", count=8, nmax=64, mix=1, tol=1e-10),
        # the 2D problem
        dict(name="bicg2d_512", op="bicg2d", n=512, kind=1, iters=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["apply", "apply", "bicg", "bicg", "bicg", "setup", "true", "solve", "solve", "mixed", "batch",
                     "bicg2d"])
    kind = rng.choice([1, 2])
    if op == "apply":
        return dict(op=op, n=_log_int(rng, 9, 512), kind=kind, transpose=rng.choice([False, True]))
    if op == "bicg":
        n = _log_int(rng, 16, 512)
        # short of convergence, and below the cost of the largest listed case
        most = min(3 * n, 200) if n <= 160 else 40 if n <= 320 else 16
        return dict(op=op, n=n, kind=kind, iters=_log_int(rng, 8, most))
    if op == "setup":
        return dict(op=op, n=4 * _log_int(rng, 4, 128), kind=kind)
    if op == "true":
        return dict(op=op, n=2 * _log_int(rng, 8, 256))
    if op in ("solve", "mixed"):
        # n = c 2^k as the cascade asks; first-kind data needs many more
        # iterations, so it is drawn up to 64^3 (mixed: both kinds up to 64^3)
        c = rng.choice([4, 5, 6, 7, 8])
        top = 256 if op == "solve" and kind == 2 else 64
        ks = [k for k in range(2, 7) if c * 2 ** k <= top]
        n = c * 2 ** rng.choice(ks)
        if op == "mixed":
            return dict(op=op, n=n, coarsest=c, kind=kind, tol=1e-12, problem="exp")
        return dict(op=op, n=n, coarsest=c, kind=kind, tol=1e-10,
                    problem=rng.choice(["exp", "sines"]) if n <= 64 else "exp")
    if op == "batch":
        return dict(op=op, count=rng.randint(4, 8), nmax=rng.choice([32, 48, 64]), mix=rng.randint(2, 1000), tol=1e-10)
    return dict(op="bicg2d", n=_log_int(rng, 32, 1024), kind=kind, iters=_log_int(rng, 16, 100))


# ------------------------------------------------------------------- inputs
def _rand(shape, seed, lo=-1.0, hi=1.0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return torch.empty(shape, dtype=F8, device=DEV).uniform_(lo, hi, generator=g)


def _terms(problem, seed):
    """[(A, (factor x, factor y, factor z))] of a manufactured solution: four
    seeded sines with integer wave numbers 1..4, or one exponential."""
    r = np.random.Generator(np.random.PCG64(int(seed)))
    if problem == "sines":
        return [(float(r.standard_normal()), tuple(("sin", math.pi * int(v)) for v in r.integers(1, 5, size=3)))
                for _ in range(4)]
    return [(1.0, tuple(("exp", float(v)) for v in r.uniform(0.8, 1.2, size=3)))]


def _fn(f, d, s):
    """d-th derivative of the factor f at s."""
    name, w = f
    if name == "exp":
        return w ** d * torch.exp(w * s)
    return w ** d * torch.sin(w * s + 0.5 * math.pi * d)


def _data(n, kind, problem, seed):
    """(f, g1, g2) on the grid with n intervals: f = Laplacian^2 u, g1 = u,
    g2 = outward du/dn (kind 1) or d2u/dn2 (kind 2) on the six faces."""
    s = torch.arange(n + 1, dtype=F8, device=DEV) / n
    end = [torch.zeros(1, dtype=F8, device=DEV), torch.ones(1, dtype=F8, device=DEV)]
    f = torch.zeros((n + 1,) * 3, dtype=F8, device=DEV)
    u = torch.zeros_like(f)
    g2 = torch.zeros((6, n + 1, n + 1), dtype=F8, device=DEV)
    for A, fac in _terms(problem, seed):
        v = [_fn(q, 0, s) for q in fac]
        prod = v[2][:, None, None] * v[1][None, :, None] * v[0][None, None, :]
        sq = sum(w * w if name == "exp" else -w * w for name, w in fac)
        u += A * prod
        f += (A * sq * sq) * prod
        for face in range(6):
            axis, side = divmod(face, 2)
            lo, hi = [v[a] for a in range(3) if a != axis]
            d = _fn(fac[axis], kind, end[side])
            g2[face] += (A * (d if kind == 2 or side else -d)) * (hi[:, None] * lo[None, :])
    return f, u, g2


def _batch_items(case, seed):
    """(n, coarsest, kind, seed) of the instances of a batch: the sizes of the
    batched workload up to nmax and the kinds, drawn by the case's mix."""
    r = np.random.Generator(np.random.PCG64(case["mix"]))
    sizes = [v for v in ((32, 8), (48, 6), (64, 8)) if v[0] <= case["nmax"]]
    return [sizes[int(r.integers(len(sizes)))] + (int(r.integers(1, 3)), int(seed) * 64 + i)
            for i in range(case["count"])]


def prepare(case, seed):
    op, n = case["op"], case.get("n")
    if op == "apply":
        return dict(case=case, level=B.Level(n, case["kind"]), u=_rand((n + 1,) * 3, seed))
    if op == "bicg":
        return dict(case=case, level=B.Level(n, case["kind"]), b=_rand((n + 1,) * 3, 2 * seed),
                    x0=_rand((n + 1,) * 3, 2 * seed + 1, -0.1, 0.1))
    if op == "bicg2d":
        return dict(case=case, b=_rand((n + 1,) * 2, 2 * seed), x0=_rand((n + 1,) * 2, 2 * seed + 1, -0.1, 0.1))
    if op == "setup":
        # the two coarser solutions carry an h^2 error, as solutions of the scheme do
        f, g1, g2 = _data(n, case["kind"], "sines", seed)
        err = _rand((n // 4 + 1,) * 3, seed)
        u4 = g1[::4, ::4, ::4] + (4.0 / n) ** 2 * err
        u2 = g1[::2, ::2, ::2] + (2.0 / n) ** 2 * _linear(err)
        return dict(case=case, level=B.Level(n, case["kind"]), f=f, g1=g1, g2=g2, u2=u2.contiguous(),
                    u4=u4.contiguous())
    if op == "true":
        err = _rand((n // 2 + 1,) * 3, seed)
        u = _data(n, 1, "sines", seed)[1]
        return dict(case=case, uh=(u + _linear(err) / n ** 2).contiguous(),
                    u2=(u[::2, ::2, ::2] + 4 * err / n ** 2).contiguous())
    if op in ("solve", "mixed"):
        return dict(case=case, data=_data(n, case["kind"], case["problem"], seed))
    items = _batch_items(case, seed)
    return dict(case=case, items=items, data=[_data(m, kind, "sines", sd) for m, _, kind, sd in items])


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "apply":
        return B.stencil_apply(state["level"], state["u"], transpose=case["transpose"])
    if op == "bicg":
        x = state["x0"].clone()
        it, rel, _ = B.bicg_solve(state["level"], state["b"], x, 0.0, case["iters"])
        return [x, rel, it]
    if op == "bicg2d":
        x = state["x0"].clone()
        it, rel, _ = B.bicg_solve2d(case["n"], case["kind"], state["b"], x, 0.0, case["iters"])
        return [x, rel, it]
    if op == "setup":
        n = case["n"]
        fh = B.excmg_assemble_rhs(state["level"], n, state["f"], state["g1"], state["g2"])
        return [fh, B.extrapolate_interpolate(n, state["u2"], state["u4"], g1_fine=state["g1"])]
    if op == "true":
        return B.midpoint_extrapolate(case["n"], state["uh"], state["u2"])
    if op in ("solve", "mixed"):
        uh = torch.empty_like(state["data"][0])
        ut = B.excmg_solve(case["n"], case["coarsest"], case["kind"], *state["data"], case["tol"], u_h_out=uh,
                           precision="fp64" if op == "solve" else "mixed")
        return [ut, uh]
    batch = B.Batch(max_instances=len(state["items"]))
    out = [batch.submit(m, c, kind, *d, case["tol"], precision="fp64")[1]
           for (m, c, kind, _), d in zip(state["items"], state["data"])]
    batch.run()
    batch.close()
    return out


# --------------------------------------------------------------------- work
def work(case):
    """Bytes: inputs read and outputs written once; for Bi-CG the five state
    vectors of Alg. 2 (x, r, r*, p, p*) read and written once per iteration.
    Operations: the 25-point (13-point) rows, about 50 (26) each, twice per
    Bi-CG iteration, and its vector updates and inner products."""
    op, n = case["op"], case.get("n")
    if op == "batch":
        pts = float(sum(m ** 3 for m, _, _, _ in _batch_items(case, 0)))
        return dict(bytes=(24 + 20 * 80) * pts, flops=20 * 114 * pts)
    if op == "bicg2d":
        return dict(bytes=80.0 * n ** 2 * case["iters"], flops=66.0 * n ** 2 * case["iters"])
    pts = float(n) ** 3
    if op == "apply":
        return dict(bytes=16 * pts, flops=50 * pts)
    if op == "bicg":
        return dict(bytes=80 * pts * case["iters"], flops=114 * pts * case["iters"])
    if op == "setup":
        return dict(bytes=(16 + 8 + 9 * 0.125) * pts, flops=12 * pts)
    if op == "true":
        return dict(bytes=17 * pts, flops=6 * pts)
    # whole solves: about 20 iterations on the finest grid
    return dict(bytes=(24 + 20 * 80) * pts, flops=20 * 114 * pts)


# -------------------------------------------------------------------- exact
# The method in plain torch, 64 bits: grid functions as [k, j, i] tensors.
def _along(d, axis, fn):
    return fn(d.movedim(axis, -1)).movedim(-1, axis)


def _linear(d):
    """Multilinear interpolation onto the grid twice as fine."""
    def one(v):
        o = torch.empty(v.shape[:-1] + (2 * v.shape[-1] - 1,), dtype=F8, device=v.device)
        o[..., ::2] = v
        o[..., 1::2] = 0.5 * (v[..., :-1] + v[..., 1:])
        return o
    for a in range(d.dim()):
        d = _along(d, a, one)
    return d


def _quadratic(W):
    """Lagrange interpolation of degree 2 per axis, cells of two intervals of
    W, onto the grid twice as fine."""
    def one(v):
        o = torch.empty(v.shape[:-1] + (2 * v.shape[-1] - 1,), dtype=F8, device=v.device)
        w0, w1, w2 = v[..., 0:-2:2], v[..., 1:-1:2], v[..., 2::2]
        o[..., ::2] = v
        o[..., 1::4] = 0.375 * w0 + 0.75 * w1 - 0.125 * w2
        o[..., 3::4] = -0.125 * w0 + 0.75 * w1 + 0.375 * w2
        return o
    for a in range(W.dim()):
        W = _along(W, a, one)
    return W


def _exp_finite(u1, u0):
    sub = u1[tuple(slice(None, None, 2) for _ in range(u1.dim()))]
    return _quadratic(u1 + 0.25 * _linear(sub - u0))


def _exp_true(uh, u2):
    return uh + _linear(uh[tuple(slice(None, None, 2) for _ in range(uh.dim()))] - u2) / 3.0


def _shift(P, off, m, lead):
    return P[(Ellipsis,) + tuple(slice(2 + o, 2 + o + m) for o in off)] if lead else \
        P[tuple(slice(2 + o, 2 + o + m) for o in off)]


def _taps(P, m, dim, lead=False):
    """The stencil's sum without its diagonal correction, at the m^dim nodes
    inside a padding of 2: weights (42, -12, 1, 2) in 3D, (20, -8, 1, 2) in 2D."""
    ctr, near = (42.0, -12.0) if dim == 3 else (20.0, -8.0)
    zero = (0,) * dim

    def off(*pairs):
        o = list(zero)
        for a, v in pairs:
            o[a] = v
        return _shift(P, o, m, lead)

    y = ctr * off()
    for a in range(dim):
        y += near * (off((a, 1)) + off((a, -1)))
        y += off((a, 2)) + off((a, -2))
        for b in range(a + 1, dim):
            y += 2.0 * (off((a, 1), (b, 1)) + off((a, 1), (b, -1)) + off((a, -1), (b, 1)) + off((a, -1), (b, -1)))
    return y


class _Op:
    """A_h on the interior of a grid with n intervals (dim 2 or 3)."""

    def __init__(self, n, kind, dim):
        self.n, self.m, self.dim, self.kind = n, n - 1, dim, kind
        e = torch.zeros(n - 1, dtype=F8, device=DEV)
        e[0] += 1
        e[-1] += 1
        c = sum(e.reshape([-1 if b == a else 1 for b in range(dim)]) for a in range(dim))
        self.diag = (1.0 if kind == 1 else -1.0) * c

    def __call__(self, v):
        lead = v.dim() > self.dim
        P = torch.nn.functional.pad(v, (2, 2) * self.dim)
        return _taps(P, self.m, self.dim, lead) + self.diag * v

    def inner(self, a):
        return a[(slice(1, -1),) * self.dim]


def _bicg(A, b, x, tol, bnorm, iters):
    """Alg. 2 with M = I and r*_0 = r_0: A_h is symmetric, so the shadow
    sequence is the primal one.  Interior arrays; returns (x, ||r||, steps)."""
    r = b - A(x)
    p = r.clone()
    rho = torch.dot(r.flatten(), r.flatten())
    k = 0
    while k < iters and float(rho) ** 0.5 > tol * bnorm:
        q = A(p)
        alpha = rho / torch.dot(p.flatten(), q.flatten())
        x = x + alpha * p
        r = r - alpha * q
        new = torch.dot(r.flatten(), r.flatten())
        p = r + (new / rho) * p
        rho = new
        k += 1
    return x, float(rho) ** 0.5, k


def _rhs(n, kind, f, g1, g2):
    """f_h: h^4 f minus every known boundary value and ghost datum a row touches."""
    h = 1.0 / n
    E = torch.zeros((n + 3,) * 3, dtype=F8, device=DEV)   # nodes -1 .. n+1
    E[1:-1, 1:-1, 1:-1] = g1
    E[2:-2, 2:-2, 2:-2] = 0.0
    s = slice(1, -1)
    for face in range(6):
        axis, side = divmod(face, 2)      # x is the last dimension
        at = [s, s, s]
        at[2 - axis] = -1 if side else 0
        g = g1.select(2 - axis, n if side else 0)
        E[tuple(at)] = 2.0 * h * g2[face] if kind == 1 else 2.0 * g + h * h * g2[face]
    fh = torch.zeros_like(f)
    i = slice(1, -1)
    fh[i, i, i] = h ** 4 * f[i, i, i] - _taps(E, n - 1, 3)
    return fh


def _solve(n, coarsest, kind, f, g1, g2, tol):
    """Alg. 1 with the uniform tolerance; returns (u~, u_h)."""
    lv = []
    N = coarsest
    while N <= n:
        t = n // N
        A = _Op(N, kind, 3)
        fl, gl = f[::t, ::t, ::t], g1[::t, ::t, ::t]
        fh = _rhs(N, kind, fl, gl, g2[:, ::t, ::t])
        b = A.inner(fh)
        u = gl.clone()
        norm = float(torch.linalg.vector_norm(b))
        if len(lv) < 2:
            m3 = (N - 1) ** 3
            M = A(torch.eye(m3, dtype=F8, device=DEV).reshape((m3,) + (N - 1,) * 3)).reshape(m3, m3)
            x = torch.linalg.solve(M, b.reshape(-1)).reshape(b.shape)
        else:
            x = A.inner(_exp_finite(lv[-1], lv[-2])).clone()
            bad, rel = 0, float(torch.linalg.vector_norm(b - A(x))) / norm
            while rel > tol:
                last = rel
                x, _, _ = _bicg(A, b, x, tol, norm, 100000)
                rel = float(torch.linalg.vector_norm(b - A(x))) / norm
                bad = bad + 1 if rel > 0.5 * last else 0
                if bad >= 2:
                    break
        A.inner(u).copy_(x)
        lv.append(u)
        N *= 2
    return _exp_true(lv[-1], lv[-2]), lv[-1]


def exact(case, seed):
    op, n = case["op"], case.get("n")
    if op in ("bicg", "bicg2d"):
        dim = 3 if op == "bicg" else 2
        b = _rand((n + 1,) * dim, 2 * seed)
        x = _rand((n + 1,) * dim, 2 * seed + 1, -0.1, 0.1)
        A = _Op(n, case["kind"], dim)
        b = A.inner(b).contiguous()
        xi, rn, k = _bicg(A, b, A.inner(x).clone(), 0.0, 1.0, case["iters"])
        A.inner(x).copy_(xi)
        return [x, rn / float(torch.linalg.vector_norm(b)), k]
    if op == "apply":
        A = _Op(n, case["kind"], 3)
        u = _rand((n + 1,) * 3, seed)
        y = torch.zeros_like(u)
        A.inner(y).copy_(A(A.inner(u)))
        return y
    if op == "setup":
        s = prepare(case, seed)
        w = _exp_finite(s["u2"], s["u4"])
        out = s["g1"].clone()
        i = slice(1, -1)
        out[i, i, i] = w[i, i, i]
        return [_rhs(n, case["kind"], s["f"], s["g1"], s["g2"]), out]
    if op == "true":
        s = prepare(case, seed)
        return _exp_true(s["uh"], s["u2"])
    if op in ("solve", "mixed"):
        return list(_solve(n, case["coarsest"], case["kind"], *_data(n, case["kind"], case["problem"], seed),
                           case["tol"]))
    return [_solve(m, c, kind, *_data(m, kind, "sines", sd), case["tol"])[0]
            for m, c, kind, sd in _batch_items(case, seed)]
