"""The work this library is used for, as cases that can be timed and checked.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (plans are
built once per setting and kept, as a program keeps them; signals come from the seed), ``run`` is one
pass through the public entry points, ``work`` the bytes and operations that pass cannot do without,
``exact`` the same outputs from a 64-bit restatement of the method in plain numpy / torch.

Kinds: project (S_K S_K^* y, and the truncated pseudoinverse and Tikhonov operators on the same path),
prolate (B y alone), coeffs / expand (T2^* y and T1 c), ragged (one plan per signal), host (signals in
pinned host memory), plan (a new setting: plan, then its first projection).
"""
from __future__ import annotations

import math
from collections import OrderedDict

import numpy as np
import torch

from paper_1611_04950_gb300 import fst, workloads

DEV = "cuda"
_REAL = {"f32": torch.float32, "f64": torch.float64, "c64": torch.float32, "c128": torch.float64}
_CPLX = ("c64", "c128")
EXACT_STEPS = 70000      # samples of serial recurrence that exact() walks per case


def listed():
    return [
        # one interactive request in double precision: a pair of signals of the smallest configuration
        dict(name="short-f64-pair", kind="project", op="project", N=4096, W=1 / 16, eps=1e-6, dtype="f64", batch=2),
        # one interactive request at the headline length: latency, launches and an almost idle chip
        dict(name="single-65536", kind="project", op="project", N=65536, W=1 / 8, eps=1e-4, dtype="f32", batch=1),
        # many short records of an odd length (sensor frames)
        dict(name="frames-3001", kind="project", op="project", N=3001, W=1 / 4, eps=1e-6, dtype="f32", batch=999),
        # the headline batch
        dict(name="batch-65536", kind="project", op="project", N=65536, W=1 / 8, eps=1e-4, dtype="f32", batch=1024),
        # long complex baseband records
        dict(name="complex-1m", kind="project", op="project", N=1 << 20, W=0.05, eps=1e-6, dtype="c64", batch=64),
        # the longest records, tight tolerance: projection, then the compressed coefficient vector
        dict(name="long-4m", kind="project", op="project", N=1 << 22, W=1 / 4, eps=1e-8, dtype="f32", batch=16),
        dict(name="coeffs-4m", kind="coeffs", op="project", N=1 << 22, W=1 / 4, eps=1e-8, dtype="f32", batch=16),
        # decompression: coefficient vectors back to samples
        dict(name="expand-65536", kind="expand", op="project", N=65536, W=1 / 8, eps=1e-4, dtype="c64", batch=256),
        # signals of mixed lengths, bandwidths and tolerances, one plan each
        dict(name="ragged-256", kind="ragged", op="project", plan_seed=3, n_lo=1000, n_hi=262144, dtype="f32", batch=256),
        # double-precision least squares (truncated pseudoinverse), a length that is no power of two
        dict(name="pinv-40000-f64", kind="project", op="pinv", N=40000, W=1 / 4, eps=1e-6, dtype="f64", batch=64),
        # signals that live in host memory: copies both ways are part of the call
        dict(name="host-65536", kind="host", op="project", N=65536, W=1 / 8, eps=1e-4, dtype="f32", batch=1024),
        # a new setting: build its plan, project one signal with it
        dict(name="plan-65536", kind="plan", op="project", N=65536, W=1 / 8, eps=1e-4, dtype="f32", batch=1),
    ]


def draw(rng):
    """One more case: lengths and batches over the logarithm of their ranges, odd lengths among them."""
    kind = rng.choice(["project", "project", "project", "prolate", "coeffs", "expand", "ragged", "host", "plan"])
    log = lambda lo, hi: int(math.exp(rng.uniform(math.log(lo), math.log(hi))))  # noqa: E731
    W, eps = rng.uniform(1 / 64, 1 / 4), rng.choice([1e-3, 1e-4, 1e-6, 1e-8])
    if kind == "ragged":
        return dict(kind=kind, op="project", plan_seed=rng.randrange(1 << 20), n_lo=1000, n_hi=rng.choice([8192, 65536, 262144]),
                    dtype=rng.choice(["f32", "f32", "c64", "f64"]), batch=log(8, 128))
    c = dict(kind=kind, op="project", N=0, W=W, eps=eps, dtype=rng.choice(["f32", "f32", "f32", "c64", "c64", "f64", "c128"]), batch=1)
    wide = c["dtype"] in ("f64", "c128")
    if kind in ("coeffs", "expand"):
        c["N"] = 1 << rng.randint(12, 16 if wide else 19)
        if kind == "expand":
            c["dtype"] = "c128" if wide else "c64"
    else:
        c["N"] = log(1000, 1 << 17 if wide or kind == "plan" else 1 << 20)
        if kind == "project" and rng.random() < 0.25:
            c["op"] = rng.choice(["pinv", "tikhonov"])
    if kind != "plan":
        c["batch"] = log(1, min(2048, (1 << (22 if wide else 24)) // c["N"] + 2))
    return c


# ---- what a program holds before the call ----------------------------------------------------

_plans: OrderedDict = OrderedDict()   # settings -> plan, as a program keeps them


def _alpha(case):
    return 1e-3 if case["op"] == "tikhonov" else 0.0


def _ragged_params(case):
    return workloads.ragged_params(case["batch"], case["plan_seed"], case["n_lo"], case["n_hi"])


def _plan(case):
    ragged = case["kind"] == "ragged"
    key = (case["batch"], case["plan_seed"], case["n_lo"], case["n_hi"]) if ragged else (case["op"], case["N"], case["W"], case["eps"])
    if key not in _plans:
        _plans[key] = fst.PlanSet(_ragged_params(case)) if ragged else fst.Plan(
            case["N"], case["W"], eps=case["eps"], op=case["op"], alpha=_alpha(case))
        while len(_plans) > 16:
            _plans.popitem(last=False)[1].close()
    _plans.move_to_end(key)
    return _plans[key]


def _signals(batch, N, W, dtype, gen):
    """The first half white noise, the second half limited to |f| <= W at unit power."""
    real, cplx = _REAL[dtype], dtype in _CPLX
    shape = (batch, N, 2) if cplx else (batch, N)
    y = torch.randn(shape, generator=gen, device=DEV, dtype=real)
    if cplx:
        y = torch.view_as_complex(y) * math.sqrt(0.5)
    h = batch - batch // 2
    for b in range(h, batch, 64):
        e = min(batch, b + 64)
        if cplx:
            keep = torch.fft.fftfreq(N, device=DEV).abs() <= W
            v = torch.fft.ifft(torch.fft.fft(y[b:e]) * keep)
        else:
            keep = torch.fft.rfftfreq(N, device=DEV) <= W
            v = torch.fft.irfft(torch.fft.rfft(y[b:e]) * keep, n=N)
        y[b:e] = v / (v.abs().square().mean(dim=1, keepdim=True).sqrt() + 1e-30)
    return y


def _sizes(case):
    """(h, r_H, r_A, r_B) of the coefficient vector: F bins -h..h and the ranks of the low-rank part."""
    N, eps = case["N"], case["eps"]
    rH = max(1, math.ceil(math.log(8.0 * N - 4.0) * math.log(4.0 * math.pi / (4.0 * math.pi * eps / 15.0)) / math.pi ** 2))
    rA = max(1, math.ceil(math.log(2.0 / (3.0 * math.pi * 7.0 * eps / 30.0)) / (2.0 * math.log(2.0))))
    rB = max(1, math.ceil(math.log(3.0 / (2.0 * 7.0 * eps / 30.0)) / (2.0 * math.log(6.0 / math.pi))))
    return math.floor(N * case["W"]), rH, rA, rB


def _inputs(case, seed, r=0):
    """The signals (or coefficient vectors, r of whose entries belong to the transition band)."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    kind, dtype = case["kind"], case["dtype"]
    if kind == "ragged":
        ns = [n for n, _, _ in _ragged_params(case)]
        return [v.clone() for v in _signals(1, sum(ns), 0.5, dtype, gen)[0].split(ns)]
    if kind == "expand":
        h, rH, rA, rB = _sizes(case)
        kp = 2 * h + 1 + 4 * rH + 4 * rA + 2 * (2 * rB - 1) + r
        # coefficient vectors of white noise: entries of order one
        c = torch.randn((case["batch"], kp, 2), generator=gen, device=DEV, dtype=_REAL[dtype])
        return torch.view_as_complex(c) * math.sqrt(0.5)
    return _signals(case["batch"], case["N"], case["W"], dtype, gen)


def _padded(case):
    """Lengths of the ragged outputs side by side in one buffer, each on a 16-byte boundary."""
    return [(n + 3) // 4 * 4 for n, _, _ in _ragged_params(case)]


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, kind=kind)
    if kind != "plan":
        s["plan"] = _plan(case)
    s["y"] = y = _inputs(case, seed, s["plan"].r if kind == "expand" else 0)
    if kind == "host":
        s["y"] = y.cpu().pin_memory()
        s["out"] = torch.empty_like(s["y"], pin_memory=True)
    if kind == "ragged":
        pad = _padded(case)
        s["out"] = torch.zeros(sum(pad), dtype=y[0].dtype, device=DEV)
        s["outs"] = [v[:u.numel()] for v, u in zip(s["out"].split(pad), y)]
        s["cut"] = sum(pad[:_walked(case)])
    return s


def run(s):
    kind = s["kind"]
    if kind == "project":
        return s["plan"].project(s["y"])
    if kind == "prolate":
        return s["plan"].apply_prolate(s["y"])
    if kind == "coeffs":
        c, r = s["plan"].coeffs(s["y"]), s["plan"].r
        return [c[:, : c.shape[1] - r], c[:, c.shape[1] - r:]]       # F and L parts, U part
    if kind == "expand":
        return s["plan"].expand(s["y"])
    if kind == "ragged":
        s["plan"].project(s["y"], s["outs"])
        return [s["out"][: s["cut"]], s["out"][s["cut"]:]]
    if kind == "host":
        return s["plan"].project_host(s["y"], s["out"])
    case = s["case"]
    p = fst.Plan(case["N"], case["W"], eps=case["eps"], op=case["op"], alpha=_alpha(case))
    e = p.export(with_vectors=False)
    out = p.project(s["y"])
    p.close()
    return [out, e["idx"], e["lam"], e["D"]]


# ---- what a pass cannot do without -----------------------------------------------------------

def _rank(N, eps):
    """Width of the transition band, 2/pi^2 ln N ln(1/eps - 1)."""
    return 2.0 / math.pi ** 2 * math.log(max(N, 2)) * math.log(1.0 / eps - 1.0)


def work(case):
    kind, dtype, batch = case["kind"], case["dtype"], case["batch"]
    size = (8 if dtype in ("f64", "c128") else 4) * (2 if dtype in _CPLX else 1)
    reals = 2 if dtype in _CPLX else 1      # real signals per signal
    rsz = size // reals

    def project(N, eps, count):
        M, r = 2.0 ** math.ceil(math.log2(2 * N)), _rank(N, eps) if kind != "prolate" else 0.0
        return (2.0 * count * N * size + rsz * (N * r + M),
                count * reals * (2 * 2.5 * M * math.log2(M) + M + 4.0 * N * r))

    if kind == "ragged":
        both = [project(n, e, 1) for n, _, e in _ragged_params(case)]
        return dict(bytes=sum(b for b, _ in both), flops=sum(f for _, f in both))
    N, eps = case["N"], case["eps"]
    if kind in ("coeffs", "expand"):
        h, rH, rA, rB = _sizes(case)
        low, r = 2 * rH + 2 * rA + 2 * (2 * rB - 1), _rank(N, eps)
        kp = 2 * h + 1 + 4 * rH + 4 * rA + 2 * (2 * rB - 1) + r
        n_in, n_out = (N * reals, 2 * kp) if kind == "coeffs" else (2 * kp, 2 * N)
        # one FFT, and per sample the columns of the low-rank part (generated once, applied to each signal)
        return dict(bytes=batch * (n_in + n_out) * rsz + N * r * rsz,
                    flops=batch * reals * (2.5 * N * math.log2(N) + N * (4.0 * low + 2.0 * r)) + N * 4.0 * low)
    b, f = project(N, eps, batch)
    if kind == "plan":
        # the vectors written in both precisions, an eigenvalue check (one convolution) per vector
        M, r = 2.0 ** math.ceil(math.log2(2 * N)), _rank(N, eps)
        b += N * r * 12.0
        f += r * (5.0 * M * math.log2(M) + 40.0 * N)
    return dict(bytes=b, flops=f)


# ---- the same in 64 bits ---------------------------------------------------------------------

def _walked(case):
    """How many of the ragged signals exact() computes (from the front)."""
    left, m = 2 * EXACT_STEPS, 0
    for n, _, _ in _ragged_params(case):
        if n > left:
            break
        left, m = left - n, m + 1
    return m


def _cos2piw(W):
    return math.cos(2.0 * math.pi * W) if W != 0.25 else 0.0


def _signed(s, lo):
    """Each vector's own symmetry, made exact, and its sign: positive sum (even l), positive first moment (odd l)."""
    n = np.arange(s.shape[1])
    for i in range(s.shape[0]):
        odd = (lo + i) % 2
        s[i] = 0.5 * (s[i] + (-1) ** odd * s[i][::-1])
        s[i] /= np.linalg.norm(s[i])
        if (s[i] * (s.shape[1] - 1 - 2 * n) if odd else s[i]).sum() < 0:
            s[i] = -s[i]
    return s


def _dpss(N, W, lo, hi):
    """Slepian vectors s^(l), lo <= l <= hi, as rows: eigenvectors of Slepian's tridiagonal matrix by
    Sturm multisection and Rayleigh-quotient steps on the twisted factorisation."""
    if N <= 600:
        n = np.arange(N, dtype=np.float64)
        T = np.diag(((N - 1) / 2 - n) ** 2 * _cos2piw(W))
        off = n[1:] * (N - n[1:]) / 2
        T += np.diag(off, 1) + np.diag(off, -1)
        return _signed(np.linalg.eigh(T)[1].T[::-1][lo:hi + 1].copy(), lo)
    n = np.arange(N, dtype=np.float64)
    d = ((N - 1) / 2 - n) ** 2 * _cos2piw(W)
    e = n[1:] * (N - n[1:]) / 2                       # e[i] couples i and i + 1
    scale = float(np.max(np.abs(d)) + 2 * np.max(e))
    d, e = d / scale, e / scale
    e2 = e * e
    asc = N - 1 - np.arange(lo, hi + 1)               # ascending index of each target
    a, b = np.full(asc.size, -1.01), np.full(asc.size, 1.01)
    pts = 16
    dl, el = d.tolist(), e2.tolist()
    for _ in range(7):                                # 17^7: neighbours are apart well before that
        x = (a[:, None] + (b - a)[:, None] * (np.arange(1, pts + 1) / (pts + 1))[None, :]).ravel()
        q, t, neg = dl[0] - x, np.empty_like(x), np.empty(x.size, bool)
        cnt = (q < 0).astype(np.int64)
        with np.errstate(divide="ignore"):
            for i in range(1, N):
                np.divide(el[i - 1], q, out=t)
                np.subtract(dl[i], x, out=q)
                np.subtract(q, t, out=q)
                np.less(q, 0.0, out=neg)
                cnt += neg
        k = (cnt.reshape(asc.size, pts) <= asc[:, None]).sum(1)
        step = (b - a) / (pts + 1)
        a, b = a + k * step, a + (k + 1) * step
    th = 0.5 * (a + b)
    D, Um = np.empty((N, asc.size)), np.empty((N, asc.size))
    for _ in range(3):
        D[0], Um[N - 1] = dl[0] - th, dl[N - 1] - th
        t = np.empty_like(th)
        for i in range(1, N):
            np.divide(el[i - 1], D[i - 1], out=t)
            np.subtract(dl[i] - th, t, out=D[i])
            j = N - 1 - i
            np.divide(el[j], Um[j + 1], out=t)
            np.subtract(dl[j] - th, t, out=Um[j])
        g = np.abs(D + Um - (d[:, None] - th[None, :]))
        z = np.zeros((N, asc.size))
        for c in range(asc.size):
            k = int(np.argmin(g[:, c]))
            z[k, c] = 1.0
            if k + 1 < N:
                z[k + 1:, c] = np.cumprod(-e[k:] / Um[k + 1:, c])
            if k:
                z[:k, c] = np.cumprod((-e[:k] / D[:k, c])[::-1])[::-1]
        z /= np.linalg.norm(z, axis=0)
        th = np.clip((d[:, None] * z * z).sum(0) + 2.0 * (e[:, None] * z[1:] * z[:-1]).sum(0), a, b)
    # one step of inverse iteration with partial pivoting at the Rayleigh quotients
    U, V, X, Y = np.empty((N, asc.size)), np.zeros((N, asc.size)), np.zeros((N, asc.size)), np.empty((N, asc.size))
    ell, cd, cu, cur = e.tolist() + [0.0, 0.0], dl[0] - th, np.full(asc.size, e[0]), z[0].copy()
    for i in range(N - 1):
        li, nd, nu, b = ell[i], dl[i + 1] - th, ell[i + 1], z[i + 1]
        swap = np.abs(cd) < li
        U[i], V[i], X[i] = np.where(swap, li, cd), np.where(swap, nd, cu), swap * nu
        Y[i] = np.where(swap, b, cur)
        f = np.where(swap, cd, li) / U[i]
        cd, cu = np.where(swap, cu, nd) - f * V[i], np.where(swap, -f * nu, nu)
        cur = np.where(swap, cur, b) - f * Y[i]
    U[N - 1], Y[N - 1] = np.where(np.abs(cd) < 1e-17, 1e-17, cd), cur
    x1 = z[N - 1] = Y[N - 1] / U[N - 1]
    x2 = np.zeros_like(x1)
    for i in range(N - 2, -1, -1):
        z[i] = (Y[i] - V[i] * x1 - X[i] * x2) / np.where(np.abs(U[i]) < 1e-17, 1e-17, U[i])
        x1, x2 = z[i], x1
    return _signed((z / np.abs(z).max(0)).T.copy(), lo)


def _sinc_row(N, W):
    """2W sinc(2W k), the phase reduced exactly (2W k split into two exact products)."""
    k = torch.arange(N, dtype=torch.float64, device=DEV)
    w2 = 2.0 * W
    hi = float(np.float32(w2))
    ph = torch.remainder(hi * k, 2.0) + (w2 - hi) * k
    r = torch.sin(math.pi * ph) / (math.pi * k)
    r[0] = w2
    return r


def _prolate(N, W, y):
    """B_{N,W} y along the last axis (64-bit rows)."""
    r = _sinc_row(N, W)
    L = 1 << (2 * N - 1).bit_length()
    c = torch.zeros(L, dtype=torch.float64, device=DEV)
    c[:N] = r
    c[L - N + 1:] = r[1:].flip(0)
    f = torch.fft.fft(c).real
    out = torch.empty_like(y)
    for b in range(0, y.shape[0], 32):
        z = torch.fft.ifft(torch.fft.fft(y[b:b + 32], n=L) * f)[:, :N]
        out[b:b + 32] = z if y.is_complex() else z.real
    return out


def _transition(case):
    """(idx, lam, D, S rows) of the transition band, all in 64 bits."""
    N, W, eps, op, alpha = case["N"], case["W"], case["eps"], case["op"], _alpha(case)
    K = math.floor(2.0 * N * W + 0.5)
    R = math.ceil(0.6 * _rank(N, eps)) + 8
    while True:
        lo, hi = max(0, K - R), min(N - 1, K + R)
        S = torch.as_tensor(_dpss(N, W, lo, hi), device=DEV)
        lam = (S * _prolate(N, W, S)).sum(1).cpu().numpy()
        l = np.arange(lo, hi + 1)
        one = (l < K).astype(np.float64)
        if op == "tikhonov":
            keep = (lam > alpha * (1 + alpha) * eps) & (lam < 1 - eps / 3)
            D = lam / (lam * lam + alpha) - lam / (1 + alpha)
        else:
            keep = np.abs(one - lam) > eps
            D = np.where(l < K, 1.0 / lam, 0.0) - lam if op == "pinv" else one - lam
        if (lo == 0 or not keep[0]) and (hi == N - 1 or not keep[-1]):
            return l[keep], lam[keep], D[keep], S[torch.as_tensor(keep, device=DEV)]
        R *= 2


def _wide(y):
    return y.to(DEV).to(torch.complex128 if y.is_complex() else torch.float64)


def _project(case, y, T):
    y = _wide(y)
    S = T[3].to(y.dtype)
    D = torch.as_tensor(T[2], device=DEV)
    beta = 1.0 / (1.0 + _alpha(case))
    return beta * _prolate(case["N"], case["W"], y) + ((y @ S.T) * D) @ S


def _shifts(N, r):
    """Optimal CF-ADI shifts b dn((2k-1) K / 2r, m), b = N - 1/2, 1 - m = (1/(2N-1))^2."""
    m1 = (0.5 / (N - 0.5)) ** 2
    a, b, c = [1.0], math.sqrt(m1), [math.sqrt(1.0 - m1)]
    while abs(c[-1]) > 1e-17 and len(a) < 60:
        an, c1, b = 0.5 * (a[-1] + b), 0.5 * (a[-1] - b), math.sqrt(a[-1] * b)
        a.append(an)
        c.append(c1)
    K = math.pi / (2.0 * a[-1])
    p = []
    for k in range(1, r + 1):
        phi = nxt = 2.0 ** (len(a) - 1) * a[-1] * (2 * k - 1) / (2.0 * r) * K
        for i in range(len(a) - 1, 0, -1):
            nxt, phi = phi, 0.5 * (phi + math.asin(c[i] / a[i] * math.sin(phi)))
        p.append((N - 0.5) * math.cos(phi) / math.cos(nxt - phi))
    return p


def _lowrank(case):
    """What the low-rank part needs: shifts, mixing matrices C_A and C_B, sizes."""
    N, W = case["N"], case["W"]
    h, rH, rA, rB = _sizes(case)
    t = math.pi * (W - (2 * h + 1) / (2.0 * N)) * N
    alpha = [0.0] + [1.0 - (1.0 - 2.0 ** (1 - 2 * k)) * _zeta(2 * k) for k in range(1, rA + 1)]
    beta = [(-1) ** k * t ** (2 * k + 1) / math.factorial(2 * k + 1) for k in range(rB)]

    def mix(D, terms):
        C = np.zeros((D, D))
        for d, w in terms:
            for i in range(d + 1):
                C[i, d - i] += 2.0 / (N * math.pi) * w * math.comb(d, i) * (-1) ** (d - i)
        return torch.as_tensor(C, device=DEV)

    CA = mix(2 * rA, [(2 * k - 1, alpha[k]) for k in range(1, rA + 1)])
    CB = mix(2 * rB - 1, [(2 * k, beta[k]) for k in range(rB)])
    return h, rH, 2 * rA, 2 * rB - 1, _shifts(N, rH), CA, CB


def _zeta(s):
    n = np.arange(1, 40001, dtype=np.float64)
    return float(np.sum(n[::-1] ** -float(s))) + 40000.5 ** (1.0 - s) / (s - 1.0)


def _columns(case, low, n):
    """Z(n), Z(N-1-n) [r_H], centred monomials, and the phase ramps exp(-j 2 pi W' n), exp(-j pi (W + W') n)."""
    N, W = case["N"], case["W"]
    h, rH, DA, DB, p, _, _ = low
    x = n.to(torch.float64) + 0.5

    def z(x):
        cols = [math.sqrt(2.0 * p[0]) / (x + p[0])]
        for k in range(1, rH):
            cols.append(cols[-1] * math.sqrt(p[k] / p[k - 1]) * (x - p[k - 1]) / (x + p[k]))
        return torch.stack(cols)

    u = (n.to(torch.float64) - 0.5 * (N - 1)) / N
    mono = torch.stack([u ** i for i in range(max(DA, DB))])
    odd = 2 * h + 1
    a = torch.remainder(odd * n, 2 * N).to(torch.float64) / (2 * N)          # W' n in cycles
    hi = float(np.float32(W))
    nd = n.to(torch.float64)
    b = 0.5 * (torch.remainder(hi * nd, 2.0) + (W - hi) * nd) + 0.5 * torch.remainder(odd * n, 4 * N).to(torch.float64) / (2 * N)
    return z(x), z(N - x), mono, torch.polar(torch.ones_like(a), -2 * math.pi * a), torch.polar(torch.ones_like(b), -2 * math.pi * b)


def _coeffs(case, y):
    N, low = case["N"], _lowrank(case)
    h, rH, DA, DB, _, CA, CB = low
    y = _wide(y)
    F = torch.cat([torch.cat([v[:, N - h:], v[:, : h + 1]], 1) for v in (torch.fft.fft(y[b:b + 4]) for b in range(0, y.shape[0], 4))]) / math.sqrt(N)
    acc = None
    for n0 in range(0, N, 1 << 18):
        n = torch.arange(n0, min(N, n0 + (1 << 18)), device=DEV)
        zf, zr, mono, pa, pb = _columns(case, low, n)
        col = torch.cat([zr, zf, mono[:DA]]).T.to(torch.complex128)
        mon = mono[:DB].T.to(torch.complex128)
        yc = y[:, n0:n0 + n.numel()].to(torch.complex128)
        part = [(yc * pa) @ col, (yc * pa.conj()) @ col, (yc * pb) @ mon, (yc * pb.conj()) @ mon]
        acc = part if acc is None else [q + w for q, w in zip(acc, part)]
    am, ap, bm, bp = acc
    CA, CB = CA.to(torch.complex128), CB.to(torch.complex128)
    return torch.cat([F, am[:, : 2 * rH], ap[:, : 2 * rH], am[:, 2 * rH:] @ CA.T, ap[:, 2 * rH:] @ CA.T, bm @ CB.T, bp @ CB.T], 1)


def _expand(case, c, T):
    N, low = case["N"], _lowrank(case)
    h, rH, DA, DB, _, _, _ = low
    c = _wide(c)
    n = torch.arange(N, device=DEV)
    zf, zr, mono, pa, pb = _columns(case, low, n)
    X = torch.zeros((c.shape[0], N), dtype=torch.complex128, device=DEV)
    X[:, : h + 1] = c[:, h:2 * h + 1]
    if h:
        X[:, N - h:] = c[:, :h]
    out = torch.fft.ifft(X) * math.sqrt(N)
    b = torch.split(c[:, 2 * h + 1:], [rH] * 4 + [DA] * 2 + [DB] * 2 + [len(T[2])], dim=1)
    mm = lambda v, col: v @ col.to(torch.complex128)  # noqa: E731
    q = 1.0 / (2j * math.pi)
    out += pa.conj() * (q * (mm(b[0], zf) - mm(b[1], zr)) + mm(b[4], mono[:DA]) / 2j)
    out += pa * (q * (mm(b[3], zr) - mm(b[2], zf)) - mm(b[5], mono[:DA]) / 2j)
    out += pb.conj() * (0.5 * mm(b[6], mono[:DB])) + pb * (0.5 * mm(b[7], mono[:DB]))
    w = torch.as_tensor(np.sign(T[2]) * np.sqrt(np.abs(T[2])), device=DEV)
    return out + mm(b[8] * w, T[3])


def exact(case, seed):
    kind = case["kind"]
    if kind == "ragged":
        y, pad, m = _inputs(case, seed), _padded(case), _walked(case)
        got = torch.zeros(sum(pad[:m]), dtype=_wide(y[0][:1]).dtype, device=DEV)
        for v, u, (N, W, eps) in zip(got.split(pad[:m]), y, _ragged_params(case)):
            one = dict(case, N=N, W=W, eps=eps)
            v[:N] = _project(one, u[None], _transition(one))[0]
        return [got, None]
    big = case["N"] > EXACT_STEPS
    if big and kind not in ("prolate", "coeffs"):
        return None
    T = None if big or kind == "prolate" else _transition(case)
    y = _inputs(case, seed, len(T[0]) if kind == "expand" else 0)
    if kind == "prolate":
        return _prolate(case["N"], case["W"], _wide(y))
    if kind == "coeffs":
        first = _coeffs(case, y)
        if big:
            return [first, None]
        u = _wide(y) @ T[3].to(_wide(y[:, :1]).dtype).T * torch.as_tensor(np.sqrt(np.abs(T[2])), device=DEV)
        return [first, u.to(torch.complex128)]
    if kind == "expand":
        return _expand(case, y, T)
    out = _project(case, y, T)
    return [out, T[0], T[1], T[2]] if kind == "plan" else out
