"""The work a user of this library has it do, as cases that can be timed and compared.

Each case is one call (or the few calls of one task) through the public binding:
fixed-rank and adaptive column IDs in every precision triple, batches of small
kernel blocks, and the CUR / two-sided ID / stable-X task that follows an ID.
The matrices are the families of the benchmark and the tests: prescribed
spectra (polynomial, geometric), a Gaussian-factor product plus noise, and
Gaussian-kernel blocks between the leaves of a k-d tree.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2310_09417_gb300 import binding as B
from paper_2310_09417_gb300 import workloads as W

DEV = "cuda:0"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: one ID inside a larger program, where latency and launches count
        {"name": "fixed_f64_small", "kind": "fixed", "prec": "f64", "m": 600, "n": 400, "k": 48, "l": 56,
         "block": 64, "spectrum": "geometric", "decay": 20.0},
        # the fixed-rank benchmark: 2000 x 2000, k = 100 from 120 sketch rows
        {"name": "fixed_f64emu", "kind": "fixed", "prec": "f64emu", "m": 2000, "n": 2000, "k": 100, "l": 120,
         "block": 64, "spectrum": "geometric", "decay": 20.0},
        # the README's first call, plain FP64 throughout
        {"name": "adaptive_f64", "kind": "adaptive", "prec": "f64", "m": 4000, "n": 1000, "block": 64,
         "k_max": 640, "tol": 1e-8, "spectrum": "geometric", "decay": 40.0},
        # the reduced benchmark matrix, run to full rank (its late rounds: few columns left, long products)
        {"name": "adaptive_f64emu_full", "kind": "adaptive", "prec": "f64emu", "m": 16384, "n": 4096, "block": 64,
         "k_max": 4096, "tol": 1e-10, "spectrum": "poly", "decay": 2.0},
        # the benchmark's size at a tolerance with a low rank, the use an ID is made for
        {"name": "adaptive_f64emu", "kind": "adaptive", "prec": "f64emu", "m": 40000, "n": 10000, "block": 64,
         "k_max": 3072, "tol": 1e-4, "spectrum": "poly", "decay": 2.0},
        # FP32 on the SIMT units, odd sizes in both dimensions
        {"name": "adaptive_f32_odd", "kind": "adaptive", "prec": "f32", "m": 12007, "n": 3001, "block": 64,
         "k_max": 1024, "tol": 1e-3, "spectrum": "poly", "decay": 2.0},
        # FP32 data with the FP32-accurate tensor-core sketch
        {"name": "adaptive_f32emu", "kind": "adaptive", "prec": "f32emu", "m": 40000, "n": 10000, "block": 64,
         "k_max": 1536, "tol": 5e-4, "spectrum": "poly", "decay": 2.0},
        # mixed precision at the benchmark's size: BF16 storage and sketch, FP32 LU; stops just after the signal
        {"name": "adaptive_bf16", "kind": "adaptive", "prec": "bf16", "m": 100000, "n": 20000, "block": 64,
         "k_max": 3072, "tol": 3e-2, "spectrum": "lowrank", "decay": 1500.0},
        # FP8 storage with block scales: a fixed number of columns of a large matrix, ragged sizes
        {"name": "fixed_fp8", "kind": "fixed", "prec": "fp8", "m": 50001, "n": 12003, "k": 512, "l": 576,
         "block": 64, "spectrum": "lowrank", "decay": 400.0},
        # hierarchical-matrix compression: blocks of a Gaussian kernel, uneven sizes, one batched call
        {"name": "batched_f64", "kind": "batched", "prec": "f64", "points": 65536, "count": 512, "leaf": 512,
         "block": 32, "tol": 1e-8},
        # the same in FP32 with larger blocks, at a tolerance FP32 can certify
        {"name": "batched_f32", "kind": "batched", "prec": "f32", "points": 262144, "count": 512, "leaf": 1024,
         "block": 32, "tol": 1e-5},
        # what follows an ID: row skeletons, the CUR middle factor and the stable interpolation matrix
        {"name": "cur_f64", "kind": "cur", "prec": "f64", "m": 4000, "n": 2000, "k": 96, "spectrum": "geometric",
         "decay": 40.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fixed", "fixed", "adaptive", "adaptive", "adaptive", "adaptive", "batched", "cur"])
    if kind == "fixed":
        prec = rng.choice(["f64", "f64emu", "fp8"])
        hi = (60000, 14000) if prec == "fp8" else (5000, 4000)
        m, n = _log_int(rng, 300, hi[0]), _log_int(rng, 300, hi[1])
        k = _log_int(rng, 16, min(600 if prec == "fp8" else 200, min(m, n) // 2))
        c = {"kind": kind, "prec": prec, "m": m, "n": n, "k": k, "l": k + rng.randint(4, 64),
             "block": rng.choice([32, 64, 64, 100])}
        if prec == "fp8":
            return {**c, "spectrum": "lowrank", "decay": float(max(8, int(k * rng.uniform(0.5, 1.0))))}
        return {**c, "spectrum": "geometric", "decay": max(rng.uniform(15.0, 40.0), k / 5.0)}
    if kind == "adaptive":
        prec = rng.choice(["f64", "f64emu", "f32", "f32emu", "bf16"])
        hi = {"f64": 6000, "f64emu": 30000, "f32": 12000, "f32emu": 30000, "bf16": 60000}[prec]
        m = _log_int(rng, 1000, hi)
        n = max(300, min(m, int(m / rng.uniform(1.0, 6.0))))
        c = {"kind": kind, "prec": prec, "m": m, "n": n, "block": rng.choice([32, 64, 64, 64, 96])}
        if prec == "bf16":
            c = {**c, "tol": 3e-2, "spectrum": "lowrank", "decay": float(_log_int(rng, 32, n // 5))}
        elif prec in ("f64", "f64emu"):
            c = {**c, "tol": 10.0 ** rng.uniform(-8.0, -4.0), "spectrum": "geometric",
                 "decay": rng.uniform(0.02, 0.06) * n}
        else:
            c = {**c, "tol": 10.0 ** rng.uniform(-3.0, -2.0), "spectrum": "poly", "decay": 2.0}
        return {**c, "k_max": min(m, n, int(1.6 * _rank(c)) + 128)}
    if kind == "batched":
        prec = rng.choice(["f64", "f32"])
        leaf = _log_int(rng, 128, 1024)
        count = _log_int(rng, 24, 512)
        return {"kind": kind, "prec": prec, "points": _log_int(rng, 32768, 262144), "count": count, "leaf": leaf,
                "block": rng.choice([16, 32, 32]), "tol": 10.0 ** (rng.uniform(-9.0, -6.0) if prec == "f64"
                                                                   else rng.uniform(-5.0, -3.5))}
    m, n = _log_int(rng, 500, 6000), _log_int(rng, 400, 3000)
    return {"kind": kind, "prec": "f64", "m": m, "n": n, "k": _log_int(rng, 24, 160), "spectrum": "geometric",
            "decay": rng.uniform(30.0, 60.0)}


# ------------------------------------------------------------------ inputs
def _singular_values(case, r):
    if case["spectrum"] == "poly":
        return W.spectrum("poly", r, power=case["decay"])
    return W.spectrum("geometric", r, per_decade=case["decay"])


def _matrix(case, seed):
    """The input of one ID, column-major on the GPU, in the type the program stores it in."""
    m, n, prec = case["m"], case["n"], case["prec"]
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + 17)
    tf32 = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False
    try:
        if case["spectrum"] == "lowrank":
            # Gaussian factors of the stated rank plus 1e-4 noise, rounded to BF16 (rows padded for TMA)
            r = int(case["decay"])
            G1t = torch.randn(r, m, generator=g, device=DEV)
            G2t = torch.randn(n, r, generator=g, device=DEV)
            ld = -(-m // 8) * 8
            At = torch.zeros((n, ld), dtype=torch.bfloat16, device=DEV)
            for j0 in range(0, n, 4096):
                blk = G2t[j0:j0 + 4096] @ G1t
                blk += 1e-4 * torch.randn(blk.shape, generator=g, device=DEV)
                At[j0:j0 + 4096, :m] = blk
            A = At[:, :m].t()
            return B.quantize_fp8(A) if prec == "fp8" else A
        r = min(m, n)
        if case["spectrum"] == "geometric":  # values below 1e-18 of the largest vanish in the sum
            r = min(r, int(18 * case["decay"]) + 1)
        s = torch.as_tensor(_singular_values(case, r), device=DEV)
        big = m * n > 8_000_000  # large matrices: the product in FP32 (a full-rank floor of about 1e-7)
        dt = torch.float32 if big or prec in ("f32", "f32emu") else torch.float64
        U = torch.randn(m, r, generator=g, device=DEV, dtype=dt) / math.sqrt(m)
        V = torch.randn(n, r, generator=g, device=DEV, dtype=dt) / math.sqrt(n)
        if not big:
            U, V = torch.linalg.qr(U)[0], torch.linalg.qr(V)[0]
        At = (V * s.to(dt)) @ U.t()
        return At.to(torch.float64 if prec in ("f64", "f64emu") else torch.float32).t()
    finally:
        torch.backends.cuda.matmul.allow_tf32 = tf32


@functools.lru_cache(maxsize=4)
def _tree(points, count, leaf):
    return W.kernel_block_pairs(points, count, 7, leaf_max=leaf, size_min=min(64, leaf // 3))


def _kernel_blocks(case, seed):
    # one partition of the points; the points themselves move a little with the seed
    pts, leaves, pairs = _tree(case["points"], case["count"], case["leaf"])
    P = torch.as_tensor(pts + 0.003 * np.random.default_rng(int(seed)).standard_normal(pts.shape), device=DEV)
    idx = {i: torch.as_tensor(leaves[i], device=DEV) for p in pairs for i in p}
    dt = torch.float64 if case["prec"] == "f64" else torch.float32
    out = []
    for a, c in pairs:
        X, Y = P[idx[a]], P[idx[c]]
        d2 = (Y * Y).sum(1)[:, None] + (X * X).sum(1)[None, :] - 2.0 * (Y @ X.t())
        out.append(torch.exp(-d2.clamp_min(0.0) / 0.09).to(dt).contiguous().t())  # h = 0.3
    return out


def _sketch_prec(case):
    return {"f64emu": B.F64_EMU, "f32emu": B.F32_EMU}.get(case["prec"])


def prepare(case, seed):
    st = {"case": case, "seed": int(seed)}
    if case["kind"] == "batched":
        st["As"] = _kernel_blocks(case, seed)
        # one buffer for all factors, as a program that stores a compressed matrix lays them out
        dt = st["As"][0].dtype
        caps = [min(a.shape) for a in st["As"]]
        sizes = [a.shape[1] * c for a, c in zip(st["As"], caps)]
        st["X"] = torch.zeros(sum(sizes), dtype=dt, device=DEV)
        st["J"] = torch.zeros(sum(caps), dtype=torch.int64, device=DEV)
        st["outs"] = [(j, x.view(-1, c)) for j, x, c in zip(st["J"].split(caps), st["X"].split(sizes), caps)]
        # which entry of a problem's rank range each stored value belongs to
        st["X_row"] = torch.cat([torch.arange(c, device=DEV, dtype=torch.int16).repeat(a.shape[1])
                                 for a, c in zip(st["As"], caps)])
        st["J_row"] = torch.cat([torch.arange(c, device=DEV, dtype=torch.int16) for c in caps])
        st["X_of"] = torch.repeat_interleave(torch.tensor(sizes, device=DEV))
        st["J_of"] = torch.repeat_interleave(torch.tensor(caps, device=DEV))
        return st
    st["A"] = _matrix(case, seed)
    if case["kind"] == "cur":
        st["J"] = _column_skeleton(st["A"], case["k"], seed)
    return st


def _column_skeleton(A, k, seed):
    """k columns that an ID picks: partial pivoting on a Gaussian sketch, in plain torch."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 5)
    Y = torch.randn(k + 8, A.shape[0], generator=g, device=DEV, dtype=A.dtype) @ A
    return _pivot_rows(Y.t().contiguous(), k)[0][:k].contiguous()


# ------------------------------------------------------------------ one pass
def run(state):
    c = state["case"]
    if c["kind"] == "fixed":
        r = B.id_fixed_rank(state["A"], c["k"], c["l"], block=c["block"], seed=state["seed"],
                            sketch_prec=_sketch_prec(c))
        return {"J": r.J, "X": r.X, "est": r.est_err, "norm": r.norm_A}
    if c["kind"] == "adaptive":
        r = B.id_adaptive(state["A"], c["tol"], block=c["block"], k_max=c["k_max"], seed=state["seed"],
                          sketch_prec=_sketch_prec(c))
        # stored in a slot of the largest rank the program admits, whatever rank the run stopped at
        free = c["k_max"] - r.k
        return {"J": F.pad(r.J, (0, free), value=-1), "Xt": F.pad(r.X.t(), (0, free)), "k": r.k, "est": r.est_err,
                "norm": r.norm_A}
    if c["kind"] == "batched":
        rs = B.id_batched(state["As"], c["tol"], block=c["block"], seed=state["seed"], outs=state["outs"])
        k = torch.tensor([r.k for r in rs], dtype=torch.int16).to(DEV)
        # rows beyond a problem's rank are unspecified: a stored factor has zeros there
        X = torch.where(state["X_row"] < k[state["X_of"]], state["X"], 0.0)
        J = torch.where(state["J_row"] < k[state["J_of"]], state["J"], -1)
        return {"J": J, "X": X, "k": k, "est": np.array([r.est_err for r in rs])}
    A, J = state["A"], state["J"]
    I, Wm = B.cur_from_id(A, J)
    U = B.cur_middle(A, I, J, B.CUR_PSEUDOINVERSE)
    return {"I": I, "W": Wm, "U": U, "X": B.stable_x(A, J)}


# ------------------------------------------------------------------ necessary work
_BYTES = {"f64": 8, "f64emu": 8, "f32": 4, "f32emu": 4, "bf16": 2, "fp8": 1}


def _rank(case):
    """About the rank an adaptive run stops at (the spectrum's tail at the tolerance, an ID's loss included)."""
    cap = case.get("k_max", min(case["m"], case["n"]))
    if case["spectrum"] == "lowrank":
        k = 1.5 * case["decay"]
    elif case["spectrum"] == "poly":
        k = 1.4 * (6.0 / case["tol"]) ** (2.0 / 3.0)
    else:
        k = case["decay"] * (math.log10(1.0 / case["tol"]) + 1.3)
    return min(cap, case["block"] * math.ceil(k / case["block"]))


def _id_work(m, n, k, l, b, esz, xsz):
    # sketch, the triangular factorisation of its transpose, and the interpolation matrix
    return {"bytes": m * n * esz + k * n * xsz + 8 * k, "flops": 2.0 * m * n * l + n * float(k) * k
            + float(k) * k * (n - k)}


def work(case):
    if case["kind"] == "batched":
        s = 0.55 * case["leaf"]  # mean size of a leaf
        k = 48 if case["prec"] == "f64" else 40
        w = _id_work(s, s, k, k + case["block"], case["block"], _BYTES[case["prec"]], _BYTES[case["prec"]])
        return {key: v * case["count"] for key, v in w.items()}
    m, n, e = case["m"], case["n"], _BYTES[case["prec"]]
    x = 8 if case["prec"] in ("f64", "f64emu") else 4
    if case["kind"] == "fixed":
        return _id_work(m, n, case["k"], case["l"], case["block"], e, x)
    if case["kind"] == "adaptive":
        k = _rank(case)
        return _id_work(m, n, k, min(k + case["block"], m), case["block"], e, x)
    k = case["k"]
    # LUPP of C; QRs of C (twice) and R^T; Q^T A (twice), one more k x k product and the solves
    return {"bytes": e * (2.0 * m * n + 2 * m * k + k * k + k * n),
            "flops": m * k * k + 2.0 * (2 * m + n) * k * k + 2 * 2.0 * m * n * k + 2.0 * n * k * k}


# ------------------------------------------------------------------ the same in 64 bits, plain torch
_LOW = 0xFFFFFFFF


def _shift(x, s):
    """Logical right shift of int64 bit patterns."""
    return (x >> s) & ((1 << (64 - s)) - 1)


def _mulhi(c, x):
    """High 64 bits of c times x, x int64 bit patterns."""
    c0, c1, x0, x1 = c & _LOW, c >> 32, x & _LOW, _shift(x, 32)
    p01, p10 = x1 * c0, x0 * c1
    mid = _shift(x0 * c0, 32) + (p01 & _LOW) + (p10 & _LOW)
    return x1 * c1 + _shift(p01, 32) + _shift(p10, 32) + _shift(mid, 32)


def _signed(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _gaussian_rows(seed, row0, rows, m):
    """Philox4x64-10 keyed (seed, 0) at counters (column / 4, row, 0, 0), Box-Muller on 53-bit uniforms."""
    q = torch.arange(-(-m // 4), device=DEV)
    x0 = q[None, :].expand(rows, -1).contiguous()
    x1 = (row0 + torch.arange(rows, device=DEV))[:, None].expand_as(x0).contiguous()
    x2, x3 = torch.zeros_like(x0), torch.zeros_like(x0)
    k0, k1 = int(seed) & ((1 << 64) - 1), 0
    m0, m1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157
    for _ in range(10):
        y0, y2 = _mulhi(m1, x2) ^ x1 ^ _signed(k0), _mulhi(m0, x0) ^ x3 ^ _signed(k1)
        x1, x3 = x2 * _signed(m1), x0 * _signed(m0)
        x0, x2 = y0, y2
        k0, k1 = k0 + 0x9E3779B97F4A7C15, k1 + 0xBB67AE8584CAA73B
    z = []
    for a, b in ((x0, x1), (x2, x3)):
        u1 = (_shift(a, 11) + 1).double() * 2.0 ** -53
        u2 = (_shift(b, 11) + 1).double() * 2.0 ** -53
        r = torch.sqrt(-2.0 * torch.log(u1))
        z += [r * torch.cos(2.0 * math.pi * u2), r * torch.sin(2.0 * math.pi * u2)]
    return torch.stack(z, 2).reshape(rows, -1)[:, :m]


def _omega(case, seed, row0, rows, m):
    z = _gaussian_rows(seed, row0, rows, m)
    if case["prec"] == "f64emu":  # that path's Omega lies on the grid 2^-11
        z = torch.clamp(torch.round(z * 2048.0), -16383, 16383) / 2048.0
    return z


def _pivot_rows(Yt, k):
    """Partial pivoting of the rows of Yt (n x >= k): (row order, unit lower n x k, U)."""
    lu, piv = torch.linalg.lu_factor(Yt[:, :k].contiguous() if Yt.shape[0] >= k else Yt)
    order = list(range(Yt.shape[0]))
    for i, p in enumerate(piv.tolist()):
        order[i], order[p - 1] = order[p - 1], order[i]
    return torch.tensor(order, device=Yt.device), lu


def _interpolation(order, lu, k):
    """X (k x n) with X(:, order[:k]) = I from the packed factors of the first k pivots."""
    n = lu.shape[0]
    L = lu[:, :k].tril(-1)
    L1 = L[:k] + torch.eye(k, dtype=lu.dtype, device=lu.device)
    T = torch.linalg.solve_triangular(L1, L[k:], upper=False, left=False, unitriangular=True)
    X = torch.zeros(k, n, dtype=lu.dtype, device=lu.device)
    X[:, order[:k]] = torch.eye(k, dtype=lu.dtype, device=lu.device)
    if n > k:
        X[:, order[k:]] = T.t()
    return X


def _exact_adaptive(case, seed, A, Om, tol, cap):
    """(rank, order, packed factors, estimate) of the adaptive loop; Om(row0, rows) gives sketch rows."""
    n, b = A.shape[1], case["block"]
    thr = tol * float(torch.linalg.norm(A))
    rows, Y = 0, None
    while True:
        want = min(max(8 * b, 2 * rows), -(-cap // b) * b + b)
        new = Om(rows, want - rows) @ A
        Y, rows = (new if Y is None else torch.cat([Y, new])), want
        width = min(rows, n)
        order, lu = _pivot_rows(Y.t().contiguous(), width)
        for t in range(1, rows // b + 1):
            tb = min(t * b, cap)
            if tb == n:
                return n, order, lu, 0.0
            hi = min(tb + b, rows)
            if hi - tb < b:
                break
            # the Schur complement of the next b rows at rank tb, from the factors
            w = min(hi, width) - tb
            L = lu[tb:, tb:tb + w].tril(-1)
            L[:w] += torch.eye(w, dtype=lu.dtype, device=lu.device)
            S = L @ lu[tb:tb + w, tb:tb + w].triu()
            if w < b:  # fewer columns than rows are left: the estimate needs all b rows
                T = _interpolation(order, lu, tb)[:, order[tb:]].t()
                S = Y[tb:hi, order[tb:]].t() - T @ Y[tb:hi, order[:tb]].t()
            E = float(torch.linalg.norm(S)) / math.sqrt(b)
            if E <= thr or tb == cap:
                return tb, order, lu, E
        if rows >= cap + b:
            raise RuntimeError("the loop did not stop")


def exact(case, seed):
    if case["prec"] in ("bf16", "fp8"):
        return None  # Omega rounded to 16 or 8 bits decides the pivots: no 64-bit value of the same call
    if case["prec"] in ("f32", "f32emu") and case["kind"] != "cur":
        # hundreds of pivots among thousands of candidates in single precision: in 64 bits other columns win
        # near-ties, and X and the estimate are another skeleton's
        if case["kind"] == "batched":
            return None
        return {"J": None, "Xt": None, "k": None, "est": None,
                "norm": float(torch.linalg.norm(_matrix(case, seed).double()))}
    if case["kind"] == "batched":
        As = _kernel_blocks(case, seed)
        cols = max(a.shape[0] for a in As)
        cache = _omega(case, seed, 0, 256, cols)
        Xs, Js, ks, es = [], [], [], []
        for a in As:
            A, cap = a.double(), min(a.shape)

            def rows_of(r0, r):
                Z = cache[r0:r0 + r, :A.shape[0]] if r0 + r <= 256 else _omega(case, seed, r0, r, A.shape[0])
                return Z
            k, order, lu, E = _exact_adaptive(case, seed, A, rows_of, case["tol"], cap)
            X = torch.zeros(A.shape[1], cap, dtype=torch.float64, device=DEV)
            X[:, :k] = _interpolation(order, lu, k).t()
            J = torch.full((cap,), -1, dtype=torch.int64, device=DEV)
            J[:k] = order[:k]
            Xs.append(X.reshape(-1))
            Js.append(J)
            ks.append(k)
            es.append(E)
        return {"J": torch.cat(Js), "X": torch.cat(Xs), "k": torch.tensor(ks, dtype=torch.int16),
                "est": np.array(es)}
    A = _matrix(case, seed).double()
    norm = float(torch.linalg.norm(A))
    if case["kind"] == "fixed":
        k, l = case["k"], case["l"]
        Y = _omega(case, seed, 0, l, case["m"]) @ A
        order, lu = _pivot_rows(Y.t().contiguous(), k)
        X = _interpolation(order, lu, k)
        est = float(torch.linalg.norm(Y[k:] - Y[k:, order[:k]] @ X)) / math.sqrt(l - k)
        return {"J": order[:k], "X": X, "est": est, "norm": norm}
    if case["kind"] == "adaptive":
        k, order, lu, E = _exact_adaptive(case, seed, A, lambda r0, r: _omega(case, seed, r0, r, case["m"]),
                                          case["tol"], case["k_max"])
        free = case["k_max"] - k
        return {"J": F.pad(order[:k], (0, free), value=-1), "Xt": F.pad(_interpolation(order, lu, k).t(), (0, free)),
                "k": k, "est": E, "norm": norm}
    k = case["k"]
    J = _column_skeleton(A, k, seed)
    C = A[:, J].contiguous()
    order, lu = _pivot_rows(C, k)
    I = order[:k]
    Wm = _interpolation(order, lu, k).t()
    Qc, Rc = torch.linalg.qr(C)
    Qr, Rr = torch.linalg.qr(A[I].t().contiguous())
    U = torch.linalg.solve_triangular(Rc, Qc.t() @ A @ Qr, upper=True)
    U = torch.linalg.solve_triangular(Rr, U.t().contiguous(), upper=True).t()
    return {"I": I, "W": Wm, "U": U, "X": torch.linalg.solve_triangular(Rc, Qc.t() @ A, upper=True)}
