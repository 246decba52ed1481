"""Performance cases of the PSD-cone projection: the calls that a first-order SDP solver makes.

Every case goes through the public binding (``paper_2507_09165_gb300.binding``) on
device-resident FP32 matrices, the way a solver calls it: one dense cone per call
(``psd_project_ex``), a block-diagonal cone per call (``psd_project_batched``), a cone
with dominant eigenpairs (``psd_project_deflate``), the norm bound alone
(``psd_norm_bound``) and a burst of requests to one server (``psd_server_*``).

``listed()`` gives the named cases, ``draw(rng)`` further ones from the same ranges,
``prepare(case, seed)`` a call's inputs, ``run(state)`` one call, ``work(case)`` the
bytes and operations that the result cannot do without, and ``exact(case, seed)`` the
result in 64 bits from plain torch and numpy.
"""
import math

import numpy as np
import torch

from paper_2507_09165_gb300 import binding as b
from paper_2507_09165_gb300 import synth

DEV = torch.device("cuda")


def listed():
    return [
        # the smallest single cone: latency of one call, nothing to hide it behind
        {"name": "fp32_256", "kind": "project", "n": 256, "ld": 256, "prec": "fp32", "matrix": "gaussian"},
        # a small cone of odd order inside a padded array of the solver's
        {"name": "bf16_701", "kind": "project", "n": 701, "ld": 704, "prec": "bf16", "matrix": "gaussian"},
        # one iteration's cone of a mid-size max-cut SDP, warm-start precision
        {"name": "fp16_2000", "kind": "project", "n": 2000, "ld": 2000, "prec": "fp16", "matrix": "wigner"},
        # an odd order with an unaligned leading dimension, in the precision a solver finishes with
        {"name": "fp32_3001", "kind": "project", "n": 3001, "ld": 3001, "prec": "fp32", "matrix": "wigner"},
        # a dense cone with a spread spectrum, the accurate half-precision mode
        {"name": "mixed_4096", "kind": "project", "n": 4096, "ld": 4096, "prec": "mixed", "matrix": "uniform"},
        # the same order where a coarse projection is enough (early iterations)
        {"name": "fp8_late_4096", "kind": "project", "n": 4096, "ld": 4096, "prec": "fp8_late", "matrix": "uniform"},
        # the large dense cone, in the accurate half-precision mode and in FP32
        {"name": "mixed_10000", "kind": "project", "n": 10000, "ld": 10000, "prec": "mixed", "matrix": "wigner"},
        {"name": "fp32_10000", "kind": "project", "n": 10000, "ld": 10000, "prec": "fp32", "matrix": "wigner"},
        # a block-diagonal cone: hundreds of blocks of very different orders in one call
        {"name": "batched_fp16_512", "kind": "batched", "count": 512, "sizes_seed": 7, "prec": "fp16"},
        # a cone whose few dominant eigenvalues are taken out before the filter
        {"name": "deflate_mixed_4096", "kind": "deflate", "n": 4096, "ld": 4096, "prec": "mixed",
         "matrix": "powerlaw", "kmax": 16},
        # the norm bound alone, as a solver's step-size rule uses it
        {"name": "norm_bound_6007", "kind": "norm_bound", "n": 6007, "ld": 6007, "matrix": "lowrank"},
        # several solves' projections arriving at one server at the same time
        {"name": "server_mix", "kind": "server", "small": 8, "mid": 3, "large": 1, "prec": "fp16"},
    ]


def _order(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project"] * 5 + ["batched", "deflate", "norm_bound", "server"])
    if kind == "project":
        n = _order(rng, 256, 10000)
        return {"kind": kind, "n": n, "ld": rng.choice([n, n, (n + 7) // 8 * 8]),
                "prec": rng.choice(["fp16", "fp16", "mixed", "mixed", "fp32", "fp32", "bf16", "fp8_late"]),
                "matrix": rng.choice(["gaussian", "wigner", "lowrank"])}
    if kind == "batched":
        return {"kind": kind, "count": _order(rng, 16, 512), "sizes_seed": rng.randrange(1, 10 ** 6),
                "prec": rng.choice(["fp16", "fp16", "bf16", "mixed", "fp32"])}
    if kind == "deflate":
        n = _order(rng, 700, 5000)
        return {"kind": kind, "n": n, "ld": n, "prec": rng.choice(["fp16", "mixed", "fp32"]), "matrix": "powerlaw",
                "kmax": rng.choice([8, 16])}
    if kind == "norm_bound":
        n = _order(rng, 256, 10000)
        return {"kind": kind, "n": n, "ld": rng.choice([n, (n + 3) // 4 * 4]),
                "matrix": rng.choice(["gaussian", "wigner", "lowrank"])}
    return {"kind": kind, "small": rng.randrange(2, 13), "mid": rng.randrange(0, 5), "large": rng.randrange(0, 2),
            "prec": rng.choice(["fp16", "bf16"])}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _symmetric(n, g, scale):
    G = torch.randn(n, n, generator=g, device=DEV)
    return (G + G.T) * (0.5 * scale)


def _matrix(kind, n, ld, seed):
    """An exactly symmetric FP32 matrix of order n in rows of ld elements."""
    g = _gen(seed)
    if kind == "gaussian":
        X = _symmetric(n, g, 1.0)
    elif kind == "wigner":
        X = _symmetric(n, g, 1.0 / math.sqrt(n))
    elif kind == "lowrank":  # positive and negative parts of rank 50 over noise
        k = min(50, max(1, n // 8))
        U = torch.linalg.qr(torch.randn(n, 2 * k, generator=g, device=DEV)).Q
        s = 1.0 + 9.0 * torch.rand(2 * k, generator=g, device=DEV)
        s[k:] *= -1.0
        X = (U * s) @ U.T + _symmetric(n, g, 1e-2)
        X = (X + X.T) * 0.5
    else:  # orthogonal similarity of a given spectrum
        Q = torch.linalg.qr(torch.randn(n, n, generator=g, device=DEV)).Q
        lam = torch.from_numpy(synth.spectrum(kind, n, seed + 1).astype(np.float32)).to(DEV)
        X = (Q * lam) @ Q.T
        X = (X + X.T) * 0.5
    if ld == n:
        return X.contiguous()
    out = torch.zeros(n, ld, device=DEV)
    out[:, :n] = X
    return out


def _blocks(case, seed):
    """Wigner blocks one after another in one buffer, and where each begins."""
    sizes = synth.block_sizes(case["count"], case["sizes_seed"])
    offs = np.concatenate([[0], np.cumsum([n * n for n in sizes])]).tolist()
    g = _gen(seed)
    X = torch.randn(offs[-1], generator=g, device=DEV)
    for n, o in zip(sizes, offs):
        V = X[o:o + n * n].view(n, n)
        V.copy_((V + V.T) * (0.5 / math.sqrt(n)))
    return sizes, offs, X


_SERVER_ORDERS = (("small", 500), ("mid", 2000), ("large", 8000))
_server = None


def _get_server():
    """The one server that a serving program keeps for all its requests."""
    global _server
    if _server is None:
        _server = b.psd_server_create(12 << 30, 0, 8192, 64)
    return _server


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batched":
        sizes, offs, X = _blocks(case, seed)
        out = torch.zeros_like(X)
        info = torch.zeros(len(sizes), b.INFO_BYTES, dtype=torch.uint8, device=DEV)
        descs = b.block_descs([(n, X.data_ptr() + 4 * o, n, out.data_ptr() + 4 * o, n, info[i])
                               for i, (n, o) in enumerate(zip(sizes, offs))], DEV)
        return {"case": case, "X": X, "out": out, "info": info, "descs": descs}
    if kind == "server":
        reqs = []
        for i, n in enumerate(n for key, n in _SERVER_ORDERS for _ in range(case[key])):
            X = _matrix("wigner", n, n, 1000 * seed + i)
            reqs.append((n, X, torch.empty_like(X)))
        return {"case": case, "server": _get_server(), "reqs": reqs}
    n, ld = case["n"], case["ld"]
    X = _matrix(case["matrix"], n, ld, seed)
    info = torch.zeros(b.INFO_BYTES // 8, dtype=torch.float64, device=DEV)
    st = {"case": case, "X": X, "info": info}
    if kind != "norm_bound":
        st["out"] = torch.zeros_like(X)
    if kind == "deflate":
        st["kused"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    return st


# -------------------------------------------------------------------- calls
def run(state):
    case = state["case"]
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "project":
        n, ld = case["n"], case["ld"]
        b.psd_project_ex(n, state["X"], ld, state["out"], ld, case["prec"], state["info"], stream=stream)
        return state["out"][:, :n]
    if kind == "deflate":
        n, ld = case["n"], case["ld"]
        b.psd_project_deflate(n, state["X"], ld, state["out"], ld, case["prec"], case["kmax"], state["info"],
                              state["kused"], stream=stream)
        return [state["out"], state["kused"]]
    if kind == "norm_bound":
        b.psd_norm_bound(case["n"], state["X"], case["ld"], state["info"], stream=stream)
        return state["info"][1:6]  # lambda_bound, lanczos_sigma, lanczos_resid, fro_X, max_diag
    if kind == "batched":
        b.psd_project_batched(case["count"], state["descs"], case["prec"], stream)
        return state["out"]
    ready = torch.cuda.Event()
    ready.record(stream)
    tickets = [b.psd_server_submit(state["server"], n, X, n, out, n, case["prec"], ready)
               for n, X, out in state["reqs"]]
    for t in tickets:
        b.psd_server_wait(state["server"], t)
    return [out for _, _, out in state["reqs"]]


# --------------------------------------------------------------------- work
_STEPS = 20  # Lanczos steps of the norm bound


def _products(prec):
    return 31 if prec == "fp32" else 22


def _bound_flops(n):
    return (2.0 * _STEPS + 2.0) * 2.0 * n * n


def work(case):
    """The triangle read once, the whole result written once; a product of two commuting symmetric
    matrices is n^3 operations (half of it is formed), a product with a vector 2 n^2."""
    kind = case["kind"]
    if kind == "norm_bound":
        n = case["n"]
        return {"bytes": 2.0 * n * n, "flops": _bound_flops(n)}
    if kind == "batched":
        orders = synth.block_sizes(case["count"], case["sizes_seed"])
    elif kind == "server":
        orders = [n for key, n in _SERVER_ORDERS for _ in range(case[key])]
    else:
        orders = [case["n"]]
    bounds = 2 if kind == "deflate" else 1
    return {"bytes": sum(6.0 * n * n for n in orders),
            "flops": sum(_products(case["prec"]) * float(n) ** 3 + bounds * _bound_flops(n) for n in orders)}


# -------------------------------------------------------------------- exact
# The paper's optimised coefficients: Table 2 (half, 7 stages), Table 1 (single, 10 stages).
_HALF = [(8.2885332412, -22.5927099246, 15.8201383114), (4.1666196466, -2.9679004036, 0.5307623217),
         (4.0611848147, -2.9698947955, 0.5492133813), (3.6678301399, -2.7561018955, 0.5421513305),
         (2.7632556383, -2.0607754898, 0.4695405857), (2.0527445797, -1.4345145882, 0.4070669182),
         (1.8804816691, -1.2583997294, 0.3779501813)]
_SINGLE = [(8.3119043343, -23.0739115930, 16.4664144722), (4.1439360087, -2.9176674704, 0.5246212487),
           (4.0257813209, -2.9025002398, 0.5334261214), (3.5118574347, -2.5740236523, 0.5050097282),
           (2.4398158400, -1.7586675341, 0.4191290613), (1.9779835097, -1.3337358510, 0.3772169049),
           (1.9559726949, -1.3091355170, 0.3746734515), (1.9282822454, -1.2823649693, 0.3704626545),
           (1.9220135179, -1.2812524618, 0.3707011753), (1.8942192942, -1.2613293407, 0.3676616051)]
_EXACT_ORDER = 5000  # a 64-bit eigendecomposition of a larger matrix takes too long


def _start_vector(n):
    """2 u - 1 with u from SplitMix64 (Steele, Lea & Flood 2014), of unit length."""
    with np.errstate(over="ignore"):
        z = np.uint64(0x243F6A8885A308D3) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    v = 2.0 * ((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1.0
    return v / np.linalg.norm(v)


def _bound(X):
    """(bound, sigma, residual, Frobenius norm, largest diagonal) of a 64-bit matrix: 20 Lanczos steps on
    X^2 with full re-orthogonalisation, then sqrt(sigma + ||X^2 q - sigma q||)."""
    n = X.shape[0]
    fro, diag = float(torch.linalg.norm(X)), float(X.diagonal().abs().max())
    Q = torch.zeros(n, _STEPS + 1, dtype=torch.float64, device=X.device)
    Q[:, 0] = torch.from_numpy(_start_vector(n)).to(X.device)
    alpha, beta = [], []
    for j in range(_STEPS):
        w = X @ (X @ Q[:, j])
        a = 0.0
        for _ in range(2):
            h = Q[:, :j + 1].T @ w
            w = w - Q[:, :j + 1] @ h
            a += float(h[j])
        alpha.append(a)
        beta.append(float(torch.linalg.norm(w)))
        if beta[-1] <= 1e-12 * fro * fro:
            break
        Q[:, j + 1] = w / beta[-1]
    m = len(alpha)
    T = np.diag(alpha) + np.diag(beta[:m - 1], 1) + np.diag(beta[:m - 1], -1)
    lam, Y = np.linalg.eigh(T)
    q = Q[:, :m] @ torch.from_numpy(Y[:, -1].copy()).to(X.device)
    q = q / torch.linalg.norm(q)
    sigma = float(lam[-1])
    resid = float(torch.linalg.norm(X @ (X @ q) - sigma * q))
    lt = max(math.sqrt(sigma + resid), fro / math.sqrt(n), diag)
    return lt, sigma, resid, fro, diag


def _filtered(X, prec):
    """The composite filter's result for a 64-bit matrix, through its eigenvalues."""
    lt = _bound(X)[0]
    coef, last, rescale = (_SINGLE, 8, 1.001) if prec == "fp32" else (_HALF, 6, 1.01)
    lam, Q = torch.linalg.eigh(X)
    x = lam / lt
    for t, (a1, a3, a5) in enumerate(coef):
        x = x * (a1 + x * x * (a3 + x * x * a5))
        if t < last:
            x = x / rescale
    return (Q * (lam * (1.0 + x) * 0.5)) @ Q.T


def exact(case, seed):
    kind = case["kind"]
    if kind == "batched":
        sizes, offs, X = _blocks(case, seed)
        out = torch.empty(offs[-1], dtype=torch.float64, device=DEV)
        for n, o in zip(sizes, offs):
            out[o:o + n * n] = _filtered(X[o:o + n * n].view(n, n).double(), case["prec"]).reshape(-1)
        return out
    if kind == "server":
        outs = []
        for i, n in enumerate(n for key, n in _SERVER_ORDERS for _ in range(case[key])):
            outs.append(_filtered(_matrix("wigner", n, n, 1000 * seed + i).double(), case["prec"])
                        if n <= _EXACT_ORDER else None)
        return outs
    n = case["n"]
    if kind == "norm_bound":
        X = _matrix(case["matrix"], n, n, seed).double()
        return torch.tensor(_bound(X), dtype=torch.float64)
    if n > _EXACT_ORDER:
        return None
    X = _matrix(case["matrix"], n, n, seed).double()
    if kind == "deflate":  # deflation is there to come nearer to the projection itself
        lam, Q = torch.linalg.eigh(X)
        return [(Q * lam.clamp(min=0.0)) @ Q.T, None]
    return _filtered(X, case["prec"])
