"""Cases that the library's speed is measured on, each one call (or one burst of calls) through
the public entry points of ``paper_2607_22484_gb300``.

The listed cases span what callers use it for: the smallest single solves, where launches and
waits count; the shapes the paper measures; large square, tall and wide solves in both tensor-core
tiers; Corollary 1's rank-r mode; the FP64 tier; the uneven batch; matrix completion on the
device; and a burst of mixed serving requests. ``draw`` gives further ones of the same ranges.
"""
from __future__ import annotations

import math
import random
import time

import torch

import paper_2607_22484_gb300 as svt

NOISE = 0.01  # entries of the noise part of low-rank inputs


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # A 64 x 64 block with a gap around tau, FP32 tier, cubic Newton-Schulz: the smallest
        # solve in use (per-patch thresholding); nothing but launches and dependent steps.
        {"name": "gap_64_fp32_ns3", "kind": "polar", "m": 64, "n": 64, "prec": "fp32", "iters": 30,
         "schedule": "ns3", "input": "gap", "mode": "svt", "pad": 0},
        # A small odd tall matrix in the default tier, a view of a wider buffer.
        {"name": "gap_97x61_bf16", "kind": "polar", "m": 97, "n": 61, "prec": "bf16", "iters": 20,
         "schedule": "pe5", "input": "gap", "mode": "svt", "pad": 3},
        # The FP64 correctness tier with an FP64 result, as used to check other tiers.
        {"name": "gap_256x192_fp64", "kind": "f64", "m": 256, "n": 192, "iters": 20, "input": "gap"},
        # The paper's accuracy test: a 300 x 301 Gaussian matrix (wide, odd sizes).
        {"name": "gauss_300x301_bf16", "kind": "polar", "m": 300, "n": 301, "prec": "bf16",
         "iters": 20, "schedule": "pe5", "input": "gauss", "mode": "svt", "pad": 0},
        # The paper's timing test at its small end: m x (m + 1) Gaussian, 25 steps.
        {"name": "gauss_1000x1001_bf16", "kind": "polar", "m": 1000, "n": 1001, "prec": "bf16",
         "iters": 25, "schedule": "pe5", "input": "gauss", "mode": "svt", "pad": 0},
        # A mid-size denoising solve in the FP32 tier (the stricter of serving's two tiers).
        {"name": "lowrank_2048x1024_fp32", "kind": "polar", "m": 2048, "n": 1024, "prec": "fp32",
         "iters": 20, "schedule": "pe5", "input": "lowrank", "mode": "svt", "pad": 0},
        # The benchmark's workload: 4096 x 4096 Marchenko-Pastur, BF16 tier, 20 steps.
        {"name": "gauss_4096_bf16", "kind": "polar", "m": 4096, "n": 4096, "prec": "bf16",
         "iters": 20, "schedule": "pe5", "input": "gauss", "mode": "svt", "pad": 0},
        # Tall low-rank-plus-noise denoising (the A^T A branch).
        {"name": "lowrank_8192x2048_bf16", "kind": "polar", "m": 8192, "n": 2048, "prec": "bf16",
         "iters": 20, "schedule": "pe5", "input": "lowrank", "mode": "svt", "pad": 0},
        # Corollary 1: best rank-r approximation of a wide matrix (the A A^T branch).
        {"name": "rank_2048x8192_bf16", "kind": "polar", "m": 2048, "n": 8192, "prec": "bf16",
         "iters": 20, "schedule": "pe5", "input": "lowrank", "mode": "rank_r", "pad": 0},
        # Six proximal-gradient steps of matrix completion as one device-resident loop.
        {"name": "complete_2048_bf16", "kind": "complete", "m": 2048, "n": 2048, "prec": "bf16",
         "iters": 20, "rank": 20, "steps": 6},
        # The uneven batch: 256 low-rank-plus-noise matrices of 128 to 1024, one grouped call.
        {"name": "batch_256_bf16", "kind": "batch", "count": 256, "lo": 128, "hi": 1024,
         "prec": "bf16", "iters": 20, "shapes": 1004},
        # A burst of serving requests, 256 to 2048, three in ten of them in the FP32 tier.
        {"name": "serve_24_mixed", "kind": "serve", "count": 24, "lo": 256, "hi": 2048, "iters": 20,
         "shapes": 1005},
    ]


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        case = _draw(rng)
        if _cost(case) <= most:
            return case


def _draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def shape(lo, hi, aspects):
        s, a = size(lo, hi), rng.choice(aspects)
        return (s, s + 1) if a == 0 else (max(8, int(s * min(1.0, a))), max(8, int(s / max(1.0, a))))

    kind = rng.choices(["small", "polar", "f64", "batch", "complete", "serve"],
                       [0.22, 0.44, 0.08, 0.10, 0.08, 0.08])[0]
    if kind == "small":
        m, n = shape(16, 192, [0, 1.0, 1.5, 0.5, 2.0])
        prec = rng.choice(["bf16", "fp32"])
        sched = "ns3" if prec == "fp32" and rng.random() < 0.5 else "pe5"
        return {"kind": "polar", "m": m, "n": n, "prec": prec, "schedule": sched, "input": "gap",
                "iters": 30 if sched == "ns3" else rng.choice([8, 11, 20, 25]),
                "mode": "svt", "pad": rng.choice([0, 0, 1, 4])}
    if kind == "polar":
        m, n = shape(192, 8192, [0, 1.0, 1.0, 0.5, 2.0, 0.25, 4.0])
        inp = rng.choice(["gauss", "lowrank"])
        return {"kind": "polar", "m": m, "n": n, "prec": rng.choice(["bf16", "bf16", "fp32"]),
                "schedule": "pe5", "input": inp, "iters": rng.choice([8, 11, 20, 20, 25]),
                "mode": "rank_r" if inp == "lowrank" and rng.random() < 0.25 else "svt",
                "pad": rng.choice([0, 0, 1, 4])}
    if kind == "f64":
        m, n = shape(32, 448, [0, 1.0, 0.5, 2.0])
        return {"kind": "f64", "m": m, "n": n, "iters": rng.choice([11, 20]), "input": "gap"}
    if kind == "batch":
        lo = size(48, 384)
        return {"kind": "batch", "count": rng.choice([7, 16, 33, 64, 128]), "lo": lo,
                "hi": min(1024, lo * rng.choice([2, 4])), "prec": rng.choice(["bf16", "bf16", "fp32"]),
                "iters": rng.choice([11, 20]), "shapes": rng.randrange(1 << 20)}
    if kind == "complete":
        m, n = shape(256, 2048, [1.0, 0.75, 1.5])
        return {"kind": "complete", "m": m, "n": n, "prec": rng.choice(["bf16", "fp32"]),
                "iters": 20, "rank": rng.randrange(5, 21), "steps": rng.randrange(3, 7)}
    return {"kind": "serve", "count": rng.choice([8, 16, 24]), "lo": 256,
            "hi": rng.choice([512, 1024, 2048]), "iters": 20, "shapes": rng.randrange(1 << 20)}


# ------------------------------------------------------------------ sizes and work

def _shapes(case):
    """(m, n, rank, tier) of each matrix of a batch or a burst of requests: sizes log-uniform,
    aspect 1, 2 or 1/2, rank 5 to 50."""
    r = random.Random(case["shapes"])
    out = []
    for _ in range(case["count"]):
        s = int(round(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"])))))
        m, n = r.choice([(s, s), (s, max(1, s // 2)), (max(1, s // 2), s)])
        rank = min(r.randint(5, 50), m, n)
        tier = "fp32" if r.random() < 0.3 else "bf16"
        out.append((m, n, rank, case.get("prec", tier)))
    return out


def _flops(m, n, iters, mode="svt", quintic=True):
    """Flops of one solve's products, symmetric ones at half."""
    M, N = max(m, n), min(m, n)
    s_step = (3 if quintic else 2) * N ** 3
    p_step = 3 * M * N * N + (N ** 3 if quintic else 0)
    if mode == "rank_r":
        return iters * s_step + 3 * M * N * N + 2 * N ** 3
    return iters * (s_step + p_step) + 6 * M * N * N + 2 * N ** 3


def work(case):
    kind = case["kind"]
    if kind in ("polar", "f64"):
        m, n = case["m"], case["n"]
        return {"bytes": m * n * (12 if kind == "f64" else 8),
                "flops": _flops(m, n, case["iters"], case.get("mode", "svt"),
                                case.get("schedule") != "ns3")}
    if kind == "complete":
        m, n = case["m"], case["n"]
        return {"bytes": case["steps"] * m * n * 13, "flops": case["steps"] * _flops(m, n, case["iters"])}
    shapes = _shapes(case)
    return {"bytes": sum(8 * m * n for m, n, _, _ in shapes),
            "flops": sum(_flops(m, n, case["iters"]) for m, n, _, _ in shapes)}


def _cost(case):
    """A case's work for the draw's limit: the FP32 tier takes three BF16 products for one, the
    FP64 tier runs without tensor cores, and short products leave much of the GPU idle."""
    kind = case["kind"]
    if kind in ("polar", "complete"):
        f = 2.6 if case["prec"] == "fp32" else 1.0
    else:
        f = 2000.0 if kind == "f64" else 4.0 * (2.6 if case.get("prec") == "fp32" else 1.0)
    return f * work(case)["flops"]


# ------------------------------------------------------------------ inputs

def _edge(m, n):
    return NOISE * (math.sqrt(m) + math.sqrt(n))


def _basis(g, m, r):
    return torch.linalg.qr(torch.randn(m, r, generator=g, device="cuda"))[0]


def _matrix(g, kind, m, n, rank=32):
    """An m x n FP32 matrix and its threshold.

    gauss: iid N(0, 1/max(m, n)) entries (no gap), tau 0.5. gap: three quarters of the singular
    values log-spaced in [0.01, 0.24], the rest in [0.36, 1], tau 0.3. lowrank: a signal with
    singular values in [2, 10] plus N(0, 0.01^2) noise, tau just above the noise."""
    if kind == "gauss":
        return torch.randn(m, n, generator=g, device="cuda").div_(math.sqrt(max(m, n))), 0.5
    if kind == "gap":
        k = min(m, n)
        lo = max(1, (3 * k) // 4)
        s = torch.cat([torch.logspace(math.log10(0.24), -2, lo, device="cuda"),
                       torch.logspace(0, math.log10(0.36), k - lo, device="cuda")])
        return (_basis(g, m, k) * s) @ _basis(g, n, k).T, 0.3
    r = min(rank, m, n)
    s = torch.rand(r, generator=g, device="cuda") * 8 + 2
    a = (_basis(g, m, r) * s) @ _basis(g, n, r).T
    return a.add_(torch.randn(m, n, generator=g, device="cuda"), alpha=NOISE), _edge(m, n) + 0.5


def _inputs(case, seed):
    """The case's matrices and thresholds (for completion: M, mask and lambda)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    kind = case["kind"]
    if kind in ("polar", "f64"):
        return [_matrix(g, case["input"], case["m"], case["n"])]
    if kind == "complete":
        m, n, r = case["m"], case["n"], min(case["rank"], case["m"], case["n"])
        a = _basis(g, m, r) * (torch.rand(r, generator=g, device="cuda") * 8 + 2)
        M = a @ _basis(g, n, r).T
        mask = (torch.rand(m, n, generator=g, device="cuda") < 0.2).to(torch.uint8)
        return M, mask, 0.2  # 0.1 of the observed part's norm (a fifth of the signal's 10)
    return [_matrix(g, "lowrank", m, n, r) for m, n, r, _ in _shapes(case)]


def _strided(a, pad):
    """The matrix as the left part of a buffer with `pad` more columns."""
    if not pad:
        return a.contiguous()
    buf = torch.zeros(a.shape[0], a.shape[1] + pad, device=a.device)
    buf[:, : a.shape[1]] = a
    return buf[:, : a.shape[1]]


def _pool(shapes):
    """One buffer that holds all results, and the matrices' views of it."""
    flat = torch.zeros(sum(m * n for m, n, _, _ in shapes), device="cuda")
    views, at = [], 0
    for m, n, _, _ in shapes:
        views.append(flat[at: at + m * n].view(m, n))
        at += m * n
    return flat, views


def prepare(case, seed):
    kind, inp = case["kind"], _inputs(case, seed)
    st = {"case": case}
    if kind in ("polar", "f64"):
        (a, tau), = inp
        m, n = case["m"], case["n"]
        opts = {"iters": case["iters"]}
        if kind == "polar":
            opts.update(prec=case["prec"], schedule=case["schedule"], mode=case["mode"])
        need = svt.workspace_bytes(m, n, **dict({"prec": "fp64"}, **opts))
        st.update(a=_strided(a, case.get("pad", 0)), tau=tau, opts=opts,
                  out=torch.zeros(m, n, device="cuda",
                                  dtype=torch.float64 if kind == "f64" else torch.float32),
                  status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    elif kind == "complete":
        M, mask, lam = inp
        m, n = M.shape
        st.update(M=M, mask=mask, lam=lam, opts={"iters": case["iters"], "prec": case["prec"]},
                  X=torch.zeros_like(M), Z=torch.zeros_like(M), Xprev=torch.zeros_like(M),
                  stats=torch.zeros(svt.binding.COMPLETION_STATS_BYTES, dtype=torch.uint8, device="cuda"))
        need = svt.workspace_bytes(m, n, **st["opts"])
    else:
        shapes = _shapes(case)
        flat, views = _pool(shapes)
        st.update(a=[x for x, _ in inp], tau=[t for _, t in inp], out=views, flat=flat,
                  opts=[{"iters": case["iters"], "prec": p} for _, _, _, p in shapes],
                  status=torch.zeros(case["count"], dtype=torch.int32, device="cuda"))
        sizes = [svt.workspace_bytes(m, n, **o) for (m, n, _, _), o in zip(shapes, st["opts"])]
        # A serving loop's memory budget holds the largest 16 requests at once; a batch's holds
        # all its matrices and launch tables.
        need = sum(sorted(sizes)[-16:]) + (16 << 20) if kind == "serve" else \
            sum(sizes) + case["count"] * (2 * 70 << 10) * 2
    st["ctx"] = svt.Context(0, workspace_bytes=need)
    torch.cuda.synchronize()
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "polar":
        ctx.polar(st["a"], st["tau"], out=st["out"], status=st["status"], **st["opts"])
        return {"y": st["out"], "status": st["status"]}
    if kind == "f64":
        ctx.polar_f64(st["a"], st["tau"], out=st["out"], status=st["status"], **st["opts"])
        return {"y": st["out"], "status": st["status"]}
    if kind == "complete":
        st["X"].zero_()
        ctx.complete_on_device(st["M"], st["mask"], st["lam"], case["steps"], X=st["X"], Z=st["Z"],
                               Xprev=st["Xprev"], stats=st["stats"], **st["opts"])
        return {"x": st["X"], "z": st["Z"]}
    if kind == "batch":
        ctx.batch(st["a"], st["tau"], outs=st["out"],
                  statuses=[st["status"][i: i + 1] for i in range(case["count"])],
                  opts=st["opts"][0])
        return {"y": st["flat"], "status": st["status"]}
    tickets = [ctx.submit(a, t, y, **o)
               for a, t, y, o in zip(st["a"], st["tau"], st["out"], st["opts"])]
    status = []
    for t in tickets:
        s, _ = ctx.poll(t)
        while s == svt.binding.ERR_NOT_READY:
            time.sleep(5e-5)
            s, _ = ctx.poll(t)
        status.append(s)
        ctx.release(t)
    return {"y": st["flat"], "status": status}


# ------------------------------------------------------------------ 64 bits

def _threshold(a, tau, rank_r=False):
    """A_tau = U max(Sigma - tau, 0) V^T (or the part with sigma > tau) in FP64, from the
    eigenvectors of the smaller Gram matrix."""
    tau = float(torch.tensor(tau, dtype=torch.float32))  # the entry points take an FP32 tau
    tall = a.shape[0] >= a.shape[1]
    w, v = torch.linalg.eigh(a.T @ a if tall else a @ a.T)
    s = w.clamp_min(0).sqrt()
    f = (s > tau).double() if rank_r else (1 - tau / s.clamp_min(1e-300)).clamp_min(0)
    p = (v * f) @ v.T
    return a @ p if tall else p @ a


def exact(case, seed):
    kind, inp = case["kind"], _inputs(case, seed)
    if kind in ("polar", "f64"):
        (a, tau), = inp
        return {"y": _threshold(a.double(), tau, case.get("mode") == "rank_r"), "status": None}
    if kind == "complete":
        M, mask, lam = inp
        M, x = M.double(), torch.zeros(M.shape, dtype=torch.float64, device="cuda")
        for _ in range(case["steps"]):
            z = torch.where(mask.bool(), M, x)
            x = _threshold(z, lam)
        return {"x": x, "z": z}
    flat = torch.cat([_threshold(a.double(), t).reshape(-1) for a, t in inp])
    return {"y": flat, "status": None}
