"""Serving windows change their tile width while requests run: a lone small request, then bursts of
growing size in all tiers, against single solves.

Tolerances: 1e-5, the bound between execution paths of one solve (FP64 tier: 1e-10)."""
import time

import numpy as np
import pytest
import torch

import paper_2607_22484_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,hi", [(1, 300), (2, 1100), (3, 1700)])
def test_serving_window_widths(seed, hi):
    rng = np.random.default_rng(seed)
    ctx = pkg.Context(0, workspace_bytes=2 << 30)
    single = pkg.Context(0, workspace_bytes=1 << 20)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    reqs = []
    for size, count in ((140, 1), (hi, 6), (hi // 2, 14)):
        for k in range(count):
            m, n = (int(x) for x in rng.integers(max(1, size // 3), size + 1, 2))
            prec = "fp64" if k == 4 and size < 600 else ("bf16", "fp32")[k % 2]
            a = torch.randn(m, n, generator=g, device="cuda") / max(m, n) ** 0.5
            reqs.append((a, float(rng.uniform(0.3, 0.7)), torch.empty_like(a), prec))
    refs = [single.polar(a, t, iters=8, prec=p).clone() for a, t, _, p in reqs]
    torch.cuda.synchronize()
    for _ in range(2):
        tickets = []
        for i, (a, t, y, p) in enumerate(reqs):
            tickets.append(ctx.submit(a, t, y, iters=8, prec=p))
            if i in (0, 6):
                time.sleep(2e-4)
        for k in tickets:
            end = time.time() + 60
            st, _ = ctx.poll(k)
            while st == pkg.binding.ERR_NOT_READY and time.time() < end:
                time.sleep(1e-4)
                st, _ = ctx.poll(k)
            assert st == 0
            ctx.release(k)
        for (a, t, y, p), r in zip(reqs, refs):
            tol = 1e-10 if p == "fp64" else 1e-5
            assert float((y - r).double().norm()) <= tol * float(r.double().norm()), (a.shape, p)
            y.fill_(float("nan"))
