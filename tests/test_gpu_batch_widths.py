"""Grouped batches at the sizes where each tile configuration is the automatic choice (128 x 64,
128 x 128, 128 x 256, pairs on 256 x 256), captured graph included, against single solves.

Tolerance: 1e-5, the bound between execution paths of one solve."""
import numpy as np
import pytest
import torch

import paper_2607_22484_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,lo,hi,prec", [(5, 60, 250, "bf16"), (40, 100, 400, "bf16"),
                                              (24, 256, 512, "bf16"), (60, 256, 512, "bf16"),
                                              (12, 800, 1023, "bf16"), (16, 600, 900, "fp32"),
                                              (3, 2100, 2200, "bf16"), (130, 1, 40, "bf16")])
def test_batch_widths(count, lo, hi, prec):
    rng = np.random.default_rng(count + lo)
    g = torch.Generator(device="cuda")
    g.manual_seed(lo)
    shapes = [tuple(int(x) for x in rng.integers(lo, hi + 1, 2)) for _ in range(count)]
    As = [torch.randn(m, n, generator=g, device="cuda") / max(m, n) ** 0.5 for m, n in shapes]
    taus = [float(t) for t in rng.uniform(0.3, 0.7, count)]
    opts = {"iters": 8, "prec": prec}
    ctx, single = (pkg.Context(0, workspace_bytes=1 << 20) for _ in range(2))
    refs = [single.polar(a, t, **opts).clone() for a, t in zip(As, taus)]
    for _ in range(2):  # the first call, then the recorded one
        outs = ctx.batch(As, taus, opts=opts)
        torch.cuda.synchronize()
        for y, r in zip(outs, refs):
            assert float((y - r).double().norm()) <= 1e-5 * float(r.double().norm())
