"""Performance cases of the sketched-Krylov f(A)b library.

One case is one piece of work a user's program asks for through the package's
public entry points: a solve with one of the basis types, sketches and methods,
both approximants from one basis, a batch of uneven problems, a solve with the
stopping criterion, a sketch applied to a block of vectors.  Operators are built
on the device from the case's sizes; right-hand sides, velocities, graph edges
and sketches come from the seed.

``exact`` restates each computation in plain torch FP64 (an unfused truncated
Arnoldi process, the dense QR whitening, quadrature of high order), with no code
of this repository.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2208_11447_gb300 as skf

DEV = "cuda"
SGMRES, SFOM = "sgmres", "sfom"


def listed():
    return [
        # a small problem solved many times (parameter studies, inner solves):
        # 2D, N = 1e4; launches, barriers and the dense tail's latency decide
        {"name": "solve2d_n100_m40", "kind": "solve", "basis": "f64", "dims": 2, "n": 100, "m": 40, "k": 2, "s": 160,
         "func": "invsqrt", "method": SGMRES, "sketch": "sparse"},
        # a somewhat larger grid carried to a converged f(A)b: the dense FP64 tail
        # (QR, node solves, level sums) takes as long as the recurrence
        {"name": "solve2d_n160_m240", "kind": "solve", "basis": "f64", "dims": 2, "n": 160, "m": 240, "k": 2, "s": 960,
         "func": "invsqrt", "method": SFOM, "sketch": "sparse"},
        # the stopping criterion of Sec. 4.3: the dimension is not known ahead,
        # every 20 steps a checkpoint's tail decides on the device
        {"name": "stop2d_n64", "kind": "stop", "basis": "f64", "dims": 2, "n": 64, "m": 160, "k": 2, "s": 640,
         "func": "invsqrt", "method": SFOM, "sketch": "sparse", "every": 20, "stop_tol": 1e-2},
        # the main FP64 workload: 100^3 grid, both approximants from one basis
        {"name": "pair3d_n100_m200", "kind": "pair", "basis": "f64", "dims": 3, "n": 100, "m": 200, "k": 2, "s": 800,
         "func": "log1p_over_z", "method": "both", "sketch": "sparse"},
        # the largest FP64 operators of a batch (about 4e6 rows, an odd grid)
        {"name": "solve3d_n159_m100", "kind": "solve", "basis": "f64", "dims": 3, "n": 159, "m": 100, "k": 2, "s": 400,
         "func": "invsqrt", "method": SGMRES, "sketch": "sparse"},
        # the paper's own sketch (subsampled randomised DCT) on a 2D grid
        {"name": "srdct2d_n600_m60", "kind": "solve", "basis": "f64", "dims": 2, "n": 600, "m": 60, "k": 2, "s": 240,
         "func": "invsqrt", "method": SFOM, "sketch": "srdct"},
        # a reduced-precision basis at the batch's ordinary size
        {"name": "fp32_3d_n100_m80", "kind": "solve", "basis": "f32", "dims": 3, "n": 100, "m": 80, "k": 2, "s": 320,
         "func": "invsqrt", "method": SGMRES, "sketch": "sparse"},
        # the large reduced-precision problem: 256^3 grid, m = 120
        {"name": "fp32_3d_n256_m120", "kind": "solve", "basis": "f32", "dims": 3, "n": 256, "m": 120, "k": 2, "s": 480,
         "func": "invsqrt", "method": SGMRES, "sketch": "sparse"},
        # a BF16 basis: half the memory again
        {"name": "bf16_3d_n150_m40", "kind": "solve", "basis": "bf16", "dims": 3, "n": 150, "m": 40, "k": 2, "s": 160,
         "func": "invsqrt", "method": SFOM, "sketch": "sparse"},
        # a directed power-law graph, k = 3: irregular rows, random gathers
        {"name": "graph_n1m_m12", "kind": "graph", "basis": "f32", "n": 1000000, "m": 12, "k": 3, "s": 48,
         "func": "invsqrt", "method": SGMRES, "sketch": "sparse"},
        # many right-hand sides over uneven operators, one call
        {"name": "batch_4ops_8rhs", "kind": "batch", "nrhs": 8, "n2": 400, "n3": 100, "m_lo": 50, "m_hi": 120, "k": 2,
         "lanes": 4, "func": "invsqrt", "method": SGMRES, "sketch": "sparse"},
        # the embedding on its own, on a block of vectors
        {"name": "sketch_n1m_c16", "kind": "sketch", "n": 1000000, "cols": 16, "s": 800, "sketch": "sparse"},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng: random.Random):
    kind = rng.choice(["solve", "solve", "pair", "stop", "f32", "f32", "bf16", "graph", "batch", "sketch", "dense"])
    func = rng.choice(["invsqrt", "invsqrt", "log1p_over_z"])
    method = rng.choice([SGMRES, SFOM])
    k = rng.choice([2, 2, 2, 3, 4])
    if kind == "sketch":
        return {"kind": "sketch", "n": int(_log(rng, 5e3, 4e6)), "cols": rng.randint(1, 24),
                "s": rng.randint(100, 1600), "sketch": rng.choice(["sparse", "sparse", "srht"])}
    if kind == "batch":
        return {"kind": "batch", "nrhs": rng.randint(4, 10), "n2": rng.randint(200, 700), "n3": rng.randint(70, 110),
                "m_lo": 40, "m_hi": rng.randint(60, 110), "k": 2, "lanes": rng.choice([2, 4, 8]), "func": "invsqrt",
                "method": method, "sketch": "sparse"}
    if kind == "graph":
        m = rng.randint(6, 12)
        return {"kind": "graph", "basis": rng.choice(["f32", "f64"]), "n": int(_log(rng, 2e5, 3e6)), "m": m, "k": 3,
                "s": 4 * m, "func": "invsqrt", "method": SGMRES, "sketch": "sparse"}
    if kind in ("f32", "bf16"):
        n = int(_log(rng, 30, 220))
        m = rng.randint(20, min(2 * n, 100 if kind == "f32" else 40))
        return {"kind": "solve", "basis": kind, "dims": 3, "n": n, "m": m, "k": 2, "s": 4 * m,
                "func": "invsqrt", "method": method, "sketch": "sparse"}
    if kind == "dense":
        m = rng.randint(20, 60)
        return {"kind": "solve", "basis": "f64", "dims": 2, "n": rng.choice([200, 243, 250, 441, 500, 625, 700]),
                "m": m, "k": 2, "s": 4 * m, "func": func, "method": method, "sketch": rng.choice(["srdct", "srht"])}
    dims = rng.choice([2, 3])
    if kind == "stop":
        return {"kind": "stop", "basis": "f64", "dims": 2, "n": rng.randint(48, 76), "m": 160, "k": 2, "s": 640,
                "func": "invsqrt", "method": method, "sketch": "sparse", "every": rng.choice([16, 20, 32]),
                "stop_tol": rng.choice([1e-2, 3e-2])}
    n = int(round(_log(rng, 2e3, 4e6) ** (1.0 / dims)))
    m = rng.randint(20, max(20, min(120, int(1.6 * n))))   # no further than the basis stays independent
    return {"kind": kind, "basis": "f64", "dims": dims, "n": n, "m": m, "k": k,
            "s": 4 * m, "func": func, "method": "both" if kind == "pair" else method, "sketch": "sparse"}


# ------------------------------------------------------------------ operators
def _stencil(n, dims, nu, dtype):
    """Centred convection-diffusion on an n^dims grid (CSR, x fastest)."""
    N, ih2, h = n ** dims, float((n + 1) ** 2), 1.0 / (n + 1)
    idx = torch.arange(N, device=DEV)
    slots = []
    for d in reversed(range(dims)):
        slots.append((-(n ** d), (idx // n ** d) % n > 0, -ih2 - nu[d] / (2 * h)))
    slots.append((0, torch.ones(N, dtype=torch.bool, device=DEV), 2.0 * dims * ih2))
    for d in range(dims):
        slots.append((n ** d, (idx // n ** d) % n < n - 1, -ih2 + nu[d] / (2 * h)))
    valid = torch.stack([v for _, v, _ in slots], 1)
    rowptr = torch.zeros(N + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(valid.sum(1), 0, out=rowptr[1:])
    cols = torch.stack([(idx + o).to(torch.int32) for o, _, _ in slots], 1)[valid]
    vals = torch.tensor([v for _, _, v in slots], dtype=dtype, device=DEV).expand(N, -1)[valid]
    return rowptr, cols, vals


def _graph(n, gen, dtype):
    """A = D + 0.1 I - W^T of a directed graph, Zipf(2.1) out-degrees of mean 10, unit weights."""
    u = torch.rand(n, generator=gen, device=DEV, dtype=torch.float64).clamp_min(1e-6)
    z = torch.floor(u ** (-1.0 / 1.1)).clamp_max(1e5)
    deg = torch.round(z * (10.0 / z.mean())).clamp(1, n - 1).long()
    src = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    dst = torch.randint(0, n - 1, (src.numel(),), generator=gen, device=DEV)
    dst = dst + (dst >= src)
    key = torch.unique(src * n + dst)
    src, dst = key // n, key % n
    diag = 0.5 * (torch.bincount(src, minlength=n) + torch.bincount(dst, minlength=n)).double() + 0.1
    i = torch.arange(n, device=DEV)
    key = torch.sort(torch.cat([dst * n + src, i * n + i]))[0]
    r, c = key // n, key % n
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(r, minlength=n), 0, out=rowptr[1:])
    vals = torch.where(r == c, diag[r], torch.full_like(diag[r], -1.0)).to(dtype)
    return rowptr, c.to(torch.int32), vals


def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * seed + salt)
    return g


def _rhs(n, seed, salt=1):
    b = torch.randn(n, generator=_gen(seed, salt), device=DEV, dtype=torch.float64)
    return b / b.norm()


def _scale(func, lam_lo, lam_hi):
    """Scale of the rule's Moebius map, from a cheap enclosure of the spectrum."""
    return math.sqrt(lam_lo * lam_hi) if func == "invsqrt" else math.sqrt(1.0 + lam_hi)


def _lam_lo(n, dims):
    return dims * (2.0 - 2.0 * math.cos(math.pi / (n + 1))) * (n + 1) ** 2


def _problem(case, seed, salt=0):
    """(csr tensors, lam_lo) of a grid or graph case."""
    dt = torch.float64 if case["basis"] == "f64" else torch.float32
    if case["kind"] == "graph":
        return _graph(case["n"], _gen(seed, 7), dt), 0.1
    rng = random.Random(seed * 31 + salt)
    # convection-dominated: a weak component lets the truncated basis lose independence
    nu = [rng.uniform(40.0, 100.0) for _ in range(case["dims"])]
    return _stencil(case["n"], case["dims"], nu, dt), _lam_lo(case["n"], case["dims"])


_BASIS = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
_SKETCH = {"sparse": skf.SPARSE_SIGN, "srht": skf.SRHT, "srdct": skf.SRDCT}


def _batch_layout(case):
    """Four operators (2D FP64, 3D FP32, and a smaller one of each) and the
    right-hand sides spread unevenly over them, each with its own m."""
    ops = [{"kind": "solve", "basis": "f64", "dims": 2, "n": case["n2"]},
           {"kind": "solve", "basis": "f32", "dims": 3, "n": case["n3"]},
           {"kind": "solve", "basis": "f64", "dims": 2, "n": max(8, case["n2"] // 2 + 1)},
           {"kind": "solve", "basis": "f32", "dims": 3, "n": max(6, (2 * case["n3"]) // 3)}]
    rng = random.Random(case["n2"] * 1009 + case["n3"] * 17 + case["nrhs"])
    return ops, [(r if r < 4 else rng.choice([0, 0, 1, 2, 3]), rng.randint(case["m_lo"], case["m_hi"]))
                 for r in range(case["nrhs"])]


# --------------------------------------------------------------------- passes
def prepare(case, seed):
    kind = case["kind"]
    if kind == "sketch":
        S = skf.Sketch(_SKETCH[case["sketch"]], case["n"], case["s"], 8, seed=100 + seed)
        X = torch.randn((case["cols"], case["n"]), generator=_gen(seed, 1), device=DEV, dtype=torch.float64).t()
        return {"case": case, "S": S, "X": X,
                "SX": torch.empty((case["cols"], case["s"]), device=DEV, dtype=torch.float64)}
    if kind == "batch":
        mats, rhs = _batch_layout(case)
        ops = []
        for i, o in enumerate(mats):
            (rp, ci, va), lo = _problem(o, seed, i)
            op = skf.upload_csr(rp, ci, va)
            ops.append((op, skf.make_func(case["func"], _scale(case["func"], lo, op.csr.norm_inf()))))
        probs = []
        for r, (i, m) in enumerate(rhs):
            op, f = ops[i]
            S = skf.Sketch(skf.SPARSE_SIGN, op.csr.n, 4 * m, 8, seed=100 + seed + r)
            b = _rhs(op.csr.n, seed, 10 + r)
            p = skf.make_params(m, case["k"], basis_dtype=_BASIS[mats[i]["basis"]])
            probs.append((skf.SGMRES if case["method"] == SGMRES else skf.SFOM, op.csr, S, b, f, p,
                          torch.empty_like(b), skf.new_info()))
        return {"case": case, "ops": ops, "probs": probs, "f32": [mats[i]["basis"] != "f64" for i, _ in rhs]}
    (rp, ci, va), lo = _problem(case, seed)
    op = skf.upload_csr(rp, ci, va)
    n = op.csr.n
    S = skf.Sketch(_SKETCH[case["sketch"]], n, case["s"], 8, seed=100 + seed)
    f = skf.make_func(case["func"], _scale(case["func"], lo, op.csr.norm_inf()))
    p = skf.make_params(case["m"], case["k"], basis_dtype=_BASIS[case["basis"]],
                        check_every=case.get("every", 0), stop_tol=case.get("stop_tol", 0.0))
    b = _rhs(n, seed)
    return {"case": case, "op": op, "S": S, "f": f, "p": p, "b": b, "x": torch.empty_like(b),
            "x2": torch.empty_like(b) if kind == "pair" else None, "info": skf.new_info(), "info2": skf.new_info()}


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "sketch":
        return skf.sketch_apply(st["S"], st["X"], st["SX"])
    if kind == "batch":
        xs = skf.solve_batched(st["probs"], lanes=case["lanes"])
        # the consumer of a reduced-precision solve takes x in single precision
        return [x.float() if single else x for x, single in zip(xs, st["f32"])]
    if kind == "pair":
        xf, xg = skf.sfom_sgmres(st["op"].csr, st["S"], st["b"], st["f"], st["p"], st["x"], st["x2"], st["info"],
                                 st["info2"])
        return {"fom": xf, "gmres": xg, "status": [_status(st["info"]), _status(st["info2"])]}
    solve = skf.sgmres if case["method"] == SGMRES else skf.sfom
    x = solve(st["op"].csr, st["S"], st["b"], st["f"], st["p"], st["x"], st["info"])
    return {"x": x if case["basis"] == "f64" else x.float(), "status": _status(st["info"])}


def _status(info):
    """(status, m_eff), the words a caller reads to know what it got."""
    return info[:8].view(torch.int32)


# ----------------------------------------------------------------------- work
def _solve_work(N, nnz, m, k, s, basis, methods=1):
    """m products with A, the window read and the new column written per step,
    the basis read once for x; the dense tail's QR."""
    bv = {"f64": 8, "f32": 4, "bf16": 2}[basis]
    av = 8 if basis == "f64" else 4
    step = nnz * (av + 4) + 4 * (N + 1) + (k + 1) * N * bv
    return {"bytes": m * step + m * N * bv + 8 * N * (1 + methods),
            "flops": m * (2 * nnz + (4 * k + 3) * N + 16 * N) + 2 * m * N * methods + 4 * s * m * m}


def work(case):
    if case["kind"] == "sketch":
        n, c = case["n"], case["cols"]
        return {"bytes": 8 * n * c + 8 * n + 8 * case["s"] * c,
                "flops": c * n * (16 if case["sketch"] == "sparse" else math.log2(n))}
    if case["kind"] == "batch":
        mats, rhs = _batch_layout(case)
        total = {"bytes": 0, "flops": 0}
        for i, m in rhs:
            o = mats[i]
            N = o["n"] ** o["dims"]
            w = _solve_work(N, (2 * o["dims"] + 1) * N, m, case["k"], 4 * m, o["basis"])
            total = {q: total[q] + w[q] for q in total}
        return total
    if case["kind"] == "graph":
        N, nnz = case["n"], 11 * case["n"]
    else:
        N = case["n"] ** case["dims"]
        nnz = (2 * case["dims"] + 1) * N
    return _solve_work(N, nnz, case["m"], case["k"], case["s"], case["basis"], 2 if case["kind"] == "pair" else 1)


# ---------------------------------------------------------------------- exact
_M64 = (1 << 64) - 1


def _signed(v):
    v &= _M64
    return v - (1 << 64) if v >> 63 else v


def _mix(z):
    """SplitMix64 finaliser on int64 tensors (two's complement)."""
    for sh, mul in ((30, 0xBF58476D1CE4E5B9), (27, 0x94D049BB133111EB), (31, None)):
        z = z ^ ((z >> sh) & ((1 << (64 - sh)) - 1))
        if mul is not None:
            z = z * _signed(mul)
    return z


def _mix_int(z):
    z &= _M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _words(seed, i):
    return _mix((i + 1) * _signed(0x9E3779B97F4A7C15) + _signed(seed))


def _sampled(seed, s, np_):
    """The first s entries of the seeded partial Fisher-Yates shuffle of [0, np_)."""
    key, swap, out = _mix_int(seed), {}, []
    for i in range(s):
        w = _mix_int(key + (i + 1) * 0x9E3779B97F4A7C15)
        j = i + w % (np_ - i)
        out.append(swap.get(j, j))
        swap[j] = swap.get(i, i)
    return torch.tensor(out, device=DEV)


class _S64:
    """The embedding applied to one vector in FP64."""

    def __init__(self, kind, n, s, seed, zeta=8):
        self.kind, self.n, self.s = kind, n, s
        if kind == "sparse":
            c = torch.arange(n, device=DEV)
            self.rows, self.signs = [], []
            for q in range(zeta):
                a, e = q * s // zeta, (q + 1) * s // zeta
                u = (_words(seed, c * 2 + q // 4) >> (16 * (q % 4))) & 0xFFFF
                self.rows.append((a + (((u >> 1) * (e - a)) >> 15)).to(torch.int32))
                self.signs.append((1 - 2 * (u & 1)).to(torch.int8))
            self.scale = 1.0 / math.sqrt(zeta)
        else:
            self.np = 1 << (n - 1).bit_length() if kind == "srht" else n
            self.signs = (1 - 2 * (_words(seed, torch.arange(n, device=DEV)) & 1)).double()
            self.P = _sampled(seed, s, self.np)

    def __call__(self, x):
        if self.kind == "sparse":
            out = torch.zeros(self.s, device=DEV, dtype=torch.float64)
            for r, g in zip(self.rows, self.signs):
                out += torch.bincount(r, weights=x * g, minlength=self.s)
            return out * self.scale
        y = x * self.signs
        if self.kind == "srht":
            y = torch.cat([y, y.new_zeros(self.np - self.n)])
            h = 1
            while h < self.np:
                y = y.view(-1, 2, h)
                y = torch.stack([y[:, 0] + y[:, 1], y[:, 0] - y[:, 1]], 1).reshape(-1)
                h *= 2
            return y[self.P] / math.sqrt(self.s)
        n = self.n   # orthonormal DCT-II through an FFT of the even-odd reordering
        v = torch.cat([y[::2], y[1::2].flip(0)])
        k = torch.arange(n, device=DEV, dtype=torch.float64)
        d = (torch.fft.fft(v) * torch.exp(-0.5j * math.pi * k / n)).real * math.sqrt(2.0 / n)
        d[0] /= math.sqrt(2.0)
        return d[self.P] * math.sqrt(n / self.s)


def _rule(func, c, ell=512):
    if func == "invsqrt":   # Gauss-Chebyshev
        x = np.cos((2 * np.arange(1, ell + 1) - 1) * math.pi / (2 * ell))
        th = (2 * np.arange(1, ell + 1) - 1) * math.pi / (2 * ell)
        t = c * np.tan(th / 2) ** 2
        return t, math.sqrt(c) / (ell * np.cos(th / 2) ** 2)
    x, w = np.polynomial.legendre.leggauss(ell)
    t = 1 + c * (1 - x) / (1 + x)
    return t, w * 2 * c / (1 + x) ** 2 / t


def _tail(method, SV, SAV, beta, t, w):
    """Coefficients y (x = V y) of one approximant from S V and S A V (s x m)."""
    m = SV.shape[1]
    Q, R = torch.linalg.qr(SV)
    Z = torch.linalg.solve_triangular(R, SAV, upper=True, left=False)
    Mm = Q.T @ Z
    c = torch.zeros(m, 1, device=DEV, dtype=torch.float64)
    c[0] = beta * R[0, 0]
    t, w = (torch.as_tensor(v, device=DEV, dtype=torch.float64)[:, None, None] for v in (t, w))
    eye = torch.eye(m, device=DEV, dtype=torch.float64)
    if method == SFOM:
        q = (w * torch.linalg.solve(t * eye + Mm, c.expand(len(t), m, 1))).sum(0)
    else:
        R2 = torch.linalg.qr(Z - Q @ Mm)[1]
        q = torch.zeros_like(c)
        for a in range(0, len(t), 64):
            K = torch.cat([t[a:a + 64] * eye + Mm, R2.expand(len(t[a:a + 64]), -1, -1)], 1).cpu()
            q2, r2 = torch.linalg.qr(K)
            rhs = (q2[:, :m].transpose(1, 2) @ c.cpu())
            q += (w[a:a + 64] * torch.linalg.solve_triangular(r2, rhs, upper=True).to(DEV)).sum(0)
    return torch.linalg.solve_triangular(R, q, upper=True)[:, 0]


def _solve64(csr, b, m, k, S, func, c, methods, every=0, stop_tol=0.0):
    rp, ci, va = csr
    n = b.numel()
    A = torch.sparse_csr_tensor(rp, ci.long(), va.double(), size=(n, n))
    V = torch.empty((m, n), device=DEV, dtype=torch.float64)
    SV, SAV = (torch.empty((S.s, m), device=DEV, dtype=torch.float64) for _ in range(2))
    beta = float(b.norm())
    t, w = _rule(func, c)
    V[0] = b / beta
    prev = None
    for j in range(m):
        SV[:, j] = S(V[j])
        y = A @ V[j]
        SAV[:, j] = S(y)
        p = j + 1
        if every and p % every == 0 and p < m:   # the stopping criterion's checkpoint
            z = _tail(methods[0], SV[:, :p], SAV[:, :p], beta, t, w)
            if prev is not None:
                eps = float(((SV[:, :p] ** 2).sum(0) - 1).abs().max())
                d = float((SV[:, :p] @ (z - torch.nn.functional.pad(prev, (0, p - len(prev))))).norm())
                if eps < 1 and d / math.sqrt(1 - eps) <= stop_tol * float((SV[:, :p] @ z).norm()) / math.sqrt(1 + eps):
                    return [z @ V[:p]]
            prev = z
        if j + 1 < m:
            for i in range(max(0, j - k + 1), j + 1):
                y -= torch.dot(V[i], y) * V[i]
            V[j + 1] = y / y.norm()
    return [_tail(q, SV, SAV, beta, t, w) @ V for q in methods]


def exact(case, seed):
    kind = case["kind"]
    if kind == "sketch":
        S = _S64(case["sketch"], case["n"], case["s"], 100 + seed)
        X = torch.randn((case["cols"], case["n"]), generator=_gen(seed, 1), device=DEV, dtype=torch.float64)
        return torch.stack([S(x) for x in X]).t()
    norm = lambda q: float(torch.zeros(q[0].numel() - 1, device=DEV, dtype=torch.float64).index_add_(   # noqa: E731
        0, torch.repeat_interleave(torch.arange(q[0].numel() - 1, device=DEV), q[0].diff()), q[2].double().abs()).max())
    if kind == "batch":
        mats, rhs = _batch_layout(case)
        probs = [_problem(o, seed, i) for i, o in enumerate(mats)]
        scale = [_scale(case["func"], lo, norm(q)) for q, lo in probs]
        out = []
        for r, (i, m) in enumerate(rhs):
            n = probs[i][0][0].numel() - 1
            out += _solve64(probs[i][0], _rhs(n, seed, 10 + r), m, case["k"],
                            _S64("sparse", n, 4 * m, 100 + seed + r), case["func"], scale[i], [case["method"]])
        return out
    csr, lo = _problem(case, seed)
    n = csr[0].numel() - 1
    S = _S64(case["sketch"], n, case["s"], 100 + seed)
    methods = [SFOM, SGMRES] if kind == "pair" else [case["method"]]
    x = _solve64(csr, _rhs(n, seed), case["m"], case["k"], S, case["func"], _scale(case["func"], lo, norm(csr)),
                 methods, case.get("every", 0), case.get("stop_tol", 0.0))
    if kind == "pair":
        return {"fom": x[0], "gmres": x[1], "status": [None, None]}
    return {"x": x[0], "status": None}
