"""The work that users of the solver have it do, as cases that can be timed and checked.

A case names one public entry point ("call") and its sizes:

    solve    Plan.solve: diag(G) of a whole batch of frequencies by the rank-k
             low-rank correction (p > 1), or the exact slice recursion (p = 1)
    xmatvec  dyson_xmatvec: u = X q, factorization and preconditioner included,
             as a caller with its own Krylov loop uses it
    apply_H  dyson_apply_H_c64: the stencil product y = H x

Inputs are those of inputs.py (trap potential, Sigma = a - i b sign(w), start
vector U[-1, 1]), drawn on the GPU.  The states of one geometry share its plan,
as the iterations of a self-consistency loop do.

The rank caps stay where the truncated diagonal is reproducible: with k close to
the number of interface sites, or k >= 32 with many high frequencies, two
roundings of the same method differ by 1e-6 and more, and a comparison would say
nothing.
"""
from __future__ import annotations

import math
import weakref

import numpy as np
import torch

from paper_1102_3137_gb300 import dyson as D
from paper_1102_3137_gb300 import inputs as I


def _case(name, call, L, K, p=1, k=1, precision="mixed", beta=20.0, eta=0.0, block=1, host=False, trap=0.01,
          b_max=0.5):
    c = dict(call=call, Lx=L[0], Ly=L[1], Lz=L[2] if len(L) > 2 else 1, K=K, p=p, k=k, precision=precision,
             beta=beta, eta=eta, block=block, host=host, trap=trap, b_max=b_max)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest lattice of the workload table, host arrays in and out as in the
        # README's example: latency, launches and copies
        _case("solve_16x16_host", "solve", (16, 16), 8, p=2, k=8, beta=10.0, host=True),
        # a small request of the serving stream
        _case("solve_64x64", "solve", (64, 64), 16, p=4, k=12),
        # the paper's own run: 101 x 101 sites, 63 frequencies (odd extents, ragged strips)
        _case("solve_101x101", "solve", (101, 101), 63, p=4, k=16, beta=40.0),
        # the plain FP64 form, the reference a user checks the mixed form against
        _case("solve_128x128_fp64", "solve", (128, 128), 16, p=4, k=32, precision="fp64"),
        # the largest 2D request of the serving stream
        _case("solve_256x256", "solve", (256, 256), 32, p=8, k=16),
        # the benchmark's lattice and batch
        _case("solve_512x512", "solve", (512, 512), 32, p=16, k=16, beta=10.0),
        # block Lanczos on the middle lattice (degenerate spectra)
        _case("block_128x128", "solve", (128, 128), 16, p=4, k=16, block=2),
        # a 3D request of the serving stream: slabs, slices of 144 sites
        _case("solve_24x24x24", "solve", (24, 24, 24), 16, p=4, k=8),
        # one operator application on the 3D workload's lattice: slices of 128 sites
        _case("xmatvec_32x32x32", "xmatvec", (32, 32, 32), 16, p=8, beta=40.0, trap=0.005, b_max=1.0),
        # one operator application on the real-frequency axis
        _case("xmatvec_128x128_real", "xmatvec", (128, 128), 32, p=4, eta=0.1),
        # the exact diagonal (one subdomain): what the truncation error is measured against
        _case("exact_128x128", "solve", (128, 128), 32, p=1),
        # the stencil product of many frequencies, bound by memory bandwidth
        _case("apply_H_128x128", "apply_H", (128, 128), 1024, p=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mixed", "mixed", "mixed", "fp64", "block", "slab", "xmatvec", "xmatvec3", "exact", "apply"])
    if kind in ("mixed", "fp64", "block", "xmatvec"):
        Lx = _log(rng, 32, {"mixed": 512, "fp64": 160, "block": 192, "xmatvec": 384}[kind])
        Ly = max(32, min(512, int(Lx * rng.uniform(0.7, 1.4))))
        h = rng.randint(12, 32)                              # strip height aimed at
        p = max(2, min(16, -(-(Ly + 1) // (h + 1))))
        p = max(p, min(16, -(-(Ly + 1) // 33)))
        top = {"mixed": 32 * 512 * 512, "fp64": 12 * 128 * 128, "block": 24 * 128 * 128, "xmatvec": 64 * 128 * 128}[kind]
        K = max(2, min(_log(rng, 4, 64), top // (Lx * Ly)))
        k = 2 * rng.randint(3, 6)
        if kind == "xmatvec":
            eta = rng.choice([0.0, 0.1])
            return _case(None, "xmatvec", (Lx, Ly), K, p=p, eta=eta, precision=rng.choice(["mixed", "fp64"]) if Lx * Ly * K < 2e5 else "mixed")
        return _case(None, "solve", (Lx, Ly), K, p=p, k=k, precision="fp64" if kind == "fp64" else "mixed",
                     beta=rng.choice([20.0, 40.0]), block=2 if kind == "block" else 1)
    if kind in ("slab", "xmatvec3"):
        Lx, Ly = rng.randint(10, 24), rng.randint(12, 24)
        h = rng.randint(4, 6)                                # slab thickness aimed at: W = Ly h
        p = rng.randint(2, 4)
        Lz = p * h + p - 1
        K = rng.randint(2, 16)
        if kind == "slab":
            return _case(None, "solve", (Lx, Ly, Lz), K, p=p, k=8, beta=rng.choice([20.0, 40.0]))
        return _case(None, "xmatvec", (Lx, Ly, Lz), K, p=p, beta=40.0, trap=0.005, b_max=1.0)
    if kind == "exact":
        return _case(None, "solve", (rng.randint(40, 128), rng.randint(40, 128)), _log(rng, 4, 32), p=1)
    Lx, Ly = _log(rng, 31, 512), _log(rng, 31, 512)
    return _case(None, "apply_H", (Lx, Ly), max(1, _log(rng, 2 ** 18, 2 ** 24) // (Lx * Ly)), p=2)


# ------------------------------------------------------------------ preparation
_plans = weakref.WeakValueDictionary()


def _shape(c):
    return (c["Lx"], c["Ly"]) if c["Lz"] == 1 else (c["Lx"], c["Ly"], c["Lz"])


def _plan(c):
    cap = 1 if c["call"] == "apply_H" else c["K"]            # device calls of apply_H take any K
    key = tuple(c[n] for n in ("call", "Lx", "Ly", "Lz", "K", "p", "k", "precision", "eta", "block"))
    pl = _plans.get(key)
    if pl is None:
        prec = D.DYSON_FP64 if c["precision"] == "fp64" else D.DYSON_MIXED
        pl = D.Plan(_shape(c), t=-1.0, mu=0.0, p=c["p"], k_max=c["k"], precision=prec, max_freqs=cap, eta=c["eta"],
                    block_size=c["block"])
        _plans[key] = pl
    return pl


def _omega(c):
    return I.real_grid(-1.0, c["K"]) if c["eta"] > 0 else I.matsubara(c["beta"], c["K"])


def _inputs(c, seed):
    """omega [K], V [N], sigma [K][N], q1 [block][N] and a complex vector per frequency."""
    N, K = c["Lx"] * c["Ly"] * c["Lz"], c["K"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    u = torch.rand((2 + c["block"], N), dtype=torch.float64, device="cuda", generator=gen)
    omega = torch.from_numpy(_omega(c)).cuda()
    V = torch.from_numpy(I.trap_potential(_shape(c), c["trap"])).cuda()
    sign = torch.ones_like(omega) if c["eta"] > 0 else torch.sign(omega)
    sigma = torch.complex((2 * u[0] - 1).expand(K, N), -(c["b_max"] * u[1])[None, :] * sign[:, None]).contiguous()
    q1 = (2 * u[2:] - 1).reshape(-1).contiguous()
    x = None
    if c["call"] != "solve":
        f = torch.float32 if c["call"] == "apply_H" else torch.float64
        x = torch.view_as_complex(torch.randn((K, N, 2), dtype=f, device="cuda", generator=gen))
    return omega, V, sigma, q1, x


def prepare(case, seed):
    c = case
    omega, V, sigma, q1, x = _inputs(c, seed)
    N, K = V.numel(), c["K"]
    s = dict(call=c["call"], plan=_plan(c), K=K, omega=omega, V=V, sigma=sigma, q1=q1, x=x)
    if c["call"] == "solve":
        s["out"] = torch.zeros((K, N), dtype=torch.complex128, device="cuda")
        s["status"] = torch.zeros(K, dtype=torch.int32, device="cuda")
        if c["host"]:
            for n in ("omega", "V", "sigma", "q1", "out", "status"):
                s[n] = s[n].cpu().numpy()
    else:
        s["out"] = torch.zeros_like(x)
    return s


def run(state):
    s = state
    if s["call"] == "solve":
        s["plan"].solve(s["omega"], s["V"], s["sigma"], s["q1"], s["out"], s["status"])
        return {"diagG": s["out"], "status": s["status"]}
    if s["call"] == "xmatvec":
        D.dyson_xmatvec(s["plan"].handle, s["K"], s["omega"], s["V"], s["sigma"], s["x"], s["out"])
    else:
        D.dyson_apply_H_c64(s["plan"].handle, s["K"], s["omega"], s["V"], s["sigma"], s["x"], s["out"])
    return {"y": s["out"]}


def work(case):
    """Inputs read once and results written once; the slice recursion's block products
    (about 2 w^3 complex multiply-adds a slice), two subdomain solves per operator
    application (2 w^2 a slice each), the Lanczos projections (two passes over j vectors)."""
    c = case
    N, K, Lx = c["Lx"] * c["Ly"] * c["Lz"], c["K"], c["Lx"]
    if c["call"] == "apply_H":
        return {"bytes": K * N * 32.0 + 8.0 * (N + K), "flops": 16.0 * K * N}
    io = K * N * 32.0 + 8.0 * N * (1 + c["block"]) + (K * N * 16.0 if c["call"] == "xmatvec" else 0.0)
    T, slow = (1, c["Ly"]) if c["Lz"] == 1 else (c["Ly"], c["Lz"])
    p = c["p"]
    h = [(slow - p + 1) // p + (1 if i < (slow - p + 1) % p else 0) for i in range(p)]
    macs = sum(2.0 * (T * v) ** 3 for v in h) * Lx
    if p > 1:
        steps = c["k"] if c["call"] == "solve" else 1
        macs += steps * 2.0 * sum(2.0 * (T * v) ** 2 for v in h) * Lx
        if c["call"] == "solve":
            macs += N * steps * (steps + 1.0)
    return {"bytes": io, "flops": 8.0 * K * macs}


# ------------------------------------------------------------------ 64-bit values
def _tridiag(z, T, slow, Lx, t):
    """Block-tridiagonal structure along x of a box: z [K][slow][T][Lx] -> g_s and diag(G_ss)."""
    K, n = z.shape[0], T * slow
    zz = z.reshape(K, n, Lx)
    A = torch.zeros((n, n), dtype=torch.complex128, device=z.device)
    i = torch.arange(n, device=z.device)
    if T > 1:
        a = i[i % T < T - 1]
        A[a, a + 1] = A[a + 1, a] = t
    a = i[i + T < n]
    A[a, a + T] = A[a + T, a] = t
    g = []
    for s in range(Lx):
        M = A.expand(K, n, n).clone()
        M.diagonal(dim1=1, dim2=2).add_(zz[:, :, s])
        if s:
            M -= t * t * g[-1]
        g.append(torch.linalg.inv(M))
    return g


def _diag_of(g, t):
    out, G = [None] * len(g), g[-1]
    out[-1] = G.diagonal(dim1=1, dim2=2)
    for s in range(len(g) - 2, -1, -1):
        G = g[s] + t * t * (g[s] @ G @ g[s])
        out[s] = G.diagonal(dim1=1, dim2=2)
    return torch.stack(out, -1)                               # [K][n][Lx]


def _tri_solve(g, t, b):
    """b [K][n][Lx]."""
    Lx, y = len(g), [None] * len(g)
    for s in range(Lx):
        r = b[:, :, s] if s == 0 else b[:, :, s] - t * y[s - 1]
        y[s] = (g[s] @ r[:, :, None])[:, :, 0]
    for s in range(Lx - 2, -1, -1):
        y[s] = y[s] - t * (g[s] @ y[s + 1][:, :, None])[:, :, 0]
    return torch.stack(y, -1)


def exact(case, seed):
    c, t = case, -1.0
    K, Lx, p = c["K"], c["Lx"], c["p"]
    T, slow = (1, c["Ly"]) if c["Lz"] == 1 else (c["Ly"], c["Lz"])
    if c["block"] > 1 or (c["call"] != "apply_H" and Lx * float(T * slow) ** 3 * K * 22 > 5e12):
        return None                                           # too long, or no scalar recurrence
    omega, V, sigma, q1, x = _inputs(c, seed)
    om = omega[:, None].to(torch.complex128)
    z = (om + 1j * c["eta"] if c["eta"] > 0 else 1j * om) - V[None, :] - sigma
    if c["call"] == "apply_H":
        v = x.to(torch.complex128).reshape(K, slow, T, Lx)
        y = z.reshape(v.shape) * v
        for d in (1, 2, 3):
            n = v.shape[d]
            y.narrow(d, 0, n - 1).add_(t * v.narrow(d, 1, n - 1))
            y.narrow(d, 1, n - 1).add_(t * v.narrow(d, 0, n - 1))
        return {"y": y.reshape(K, -1)}
    z4 = z.reshape(K, slow, T, Lx)
    full = _tridiag(z4, T, slow, Lx, t)
    if p == 1:
        return {"diagG": _diag_of(full, t).reshape(K, -1), "status": None}
    base, extra, cuts, s0 = (slow - p + 1) // p, (slow - p + 1) % p, [], 0
    for i in range(p):
        h = base + (1 if i < extra else 0)
        cuts.append((s0, s0 + h))
        s0 += h + 1
    strips = [_tridiag(z4[:, a:b].contiguous(), T, b - a, Lx, t) for a, b in cuts]

    def H(v):
        y = z4 * v
        for d in (1, 2, 3):
            n = v.shape[d]
            y.narrow(d, 0, n - 1).add_(t * v.narrow(d, 1, n - 1))
            y.narrow(d, 1, n - 1).add_(t * v.narrow(d, 0, n - 1))
        return y

    def X(q):                                                 # H^-1 (q - H w), w = blkdiag(B^-1, 0) q
        v = q.reshape(K, slow, T, Lx)
        w = torch.zeros_like(v)
        for g, (a, b) in zip(strips, cuts):
            w[:, a:b] = _tri_solve(g, t, v[:, a:b].reshape(K, T * (b - a), Lx)).reshape(K, b - a, T, Lx)
        r = v - H(w)
        for a, b in cuts:
            r[:, a:b] = 0
        u = _tri_solve(full, t, r.reshape(K, T * slow, Lx)).reshape(v.shape)
        r = r - H(u)                                          # one correction: residual at rounding
        u = u + _tri_solve(full, t, r.reshape(K, T * slow, Lx)).reshape(v.shape)
        return u.reshape(K, -1)

    if c["call"] == "xmatvec":
        return {"y": X(x)}
    diag = torch.zeros_like(z4)
    for g, (a, b) in zip(strips, cuts):
        diag[:, a:b] = _diag_of(g, t).reshape(K, b - a, T, Lx)
    diag = diag.reshape(K, -1)
    q = (q1 / torch.sqrt(q1 @ q1)).to(torch.complex128).expand(K, -1)
    Q, beta = [], None
    top = torch.zeros(K, dtype=torch.float64, device=z.device)
    live = torch.ones(K, dtype=torch.bool, device=z.device)
    for j in range(c["k"]):                                   # complex-symmetric Lanczos, bilinear form
        r = X(q)
        alpha = (q * r).sum(1)
        add = alpha[:, None] * q * q
        if j:
            add = add + 2 * beta[:, None] * Q[-1] * q
        diag = diag + torch.where(live[:, None], add, torch.zeros_like(add))
        Q.append(q)
        B = torch.stack(Q, 1)                                 # [K][j+1][N]
        for _ in range(2):
            r = r - (B.transpose(1, 2) @ (B @ r[:, :, None]))[:, :, 0]
        top = torch.maximum(top, alpha.abs())
        live = live & (r.norm(dim=1) > 1e-12 * top)           # an invariant subspace ends a frequency's sum
        beta = torch.sqrt((r * r).sum(1))
        top = torch.maximum(top, beta.abs())
        q = torch.where(live[:, None], r / beta[:, None], torch.zeros_like(r))
    return {"diagG": diag, "status": None}
