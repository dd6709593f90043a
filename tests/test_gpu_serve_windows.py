"""Serving windows that carry several stages of every active request in one fused launch."""
import numpy as np
import pytest
import torch

import paper_2607_22484_gb300 as pkg
import svt_workloads as wl

pytestmark = pytest.mark.gpu


def test_serving_windows_of_many_stages():
    """More requests than slots, of both tile widths and with ops the grouped kernels do not cover
    (rank-r mode, the FP64 tier) among them: every result equals the same solve alone."""
    rng = np.random.default_rng(8)
    shapes = [(int(rng.integers(40, 700)), int(rng.integers(40, 700))) for _ in range(24)]
    opts = [dict(prec="bf16", iters=20) if i % 3 else dict(prec="fp32", iters=12) for i in range(24)]
    opts[5] = dict(prec="bf16", iters=20, mode="rank_r")
    opts[11] = dict(prec="fp64", iters=11)
    mats = [torch.from_numpy(wl.low_rank_plus_noise(m, n, min(m, n, 20), 60 + i)).cuda()
            for i, (m, n) in enumerate(shapes)]
    outs = [torch.full_like(a, float("nan")) for a in mats]
    taus = [wl.noise_edge(m, n) + 0.5 for m, n in shapes]
    ctx = pkg.Context(0, workspace_bytes=256 << 20)
    torch.cuda.synchronize()
    tickets = [ctx.submit(a, t, y, **o) for a, t, y, o in zip(mats, taus, outs, opts)]
    for t in tickets:
        s, _ = ctx.poll(t)
        while s == pkg.binding.ERR_NOT_READY:
            s, _ = ctx.poll(t)
        assert s == 0
        ctx.release(t)
    alone = pkg.Context(0, workspace_bytes=1 << 20)
    for a, t, y, o in zip(mats, taus, outs, opts):
        ref = alone.polar(a, t, **o)
        torch.cuda.synchronize()
        assert float((y - ref).double().norm()) <= 1e-5 * float(ref.double().norm()), (a.shape, o)
