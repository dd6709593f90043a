"""Solves on 128 x 64 tiles: the automatic choice while a step's tiles are few per SM. Shapes at both
sides of that line (of each tier and of rank-r mode) and of multiples of 64 and 128, tall and wide, with
each option that changes the products; against 128 x 128 tiles and the oracle.

Tolerances: the tiers' (2e-2, 1e-4) against Eq. 1; 1e-5 between execution paths of one solve."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_22484_gb300 as pkg
import svt_workloads as wl

pytestmark = pytest.mark.gpu

BOUND = {"bf16": 2e-2, "fp32": 1e-4}


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
@pytest.mark.parametrize("m,n", [(129, 1), (129, 65), (190, 64), (1000, 63), (257, 256), (384, 705),
                                 (960, 1216), (961, 1216), (2432, 512), (2433, 512),
                                 (1152, 1088), (1300, 1290), (520, 8100), (9000, 500)])
def test_tiles_128x64(m, n, prec):
    k = min(m, n)
    hi = max(1, k // 4)
    s = np.concatenate([np.linspace(1.0, 0.36, hi), np.linspace(0.24, 0.01, k - hi)])
    a = wl.spectrum_matrix(s, m, n, m + 3 * n)
    exact = oracle.svt_definition(a.astype(np.float64), 0.3)
    dev = torch.from_numpy(a).cuda()
    ctx = pkg.Context(0, workspace_bytes=pkg.workspace_bytes(m, n, prec=prec))
    for o in (dict(), dict(polish=False), dict(mode="rank_r"), dict(schedule="ns3")):
        sts = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(2)]
        y = ctx.polar(dev, 0.3, status=sts[0], prec=prec, **o)
        ref = ctx.polar(dev, 0.3, status=sts[1], prec=prec, **dict(o, tile=128))
        assert int(sts[0]) == int(sts[1]) == 0
        assert float((y - ref).double().norm()) <= 1e-5 * float(ref.double().norm()), o
        if not o:
            assert oracle.relerr(y.cpu().numpy(), exact) < BOUND[prec]


def test_tuned_128_keeps_the_finer_tiles():
    """A tuned or imported 128 stands for the automatic choice where that is 128 x 64."""
    m, n = 300, 300
    a = torch.randn(m, n, device="cuda") / n**0.5
    ctx = pkg.Context(0, workspace_bytes=pkg.workspace_bytes(m, n))
    before = ctx.polar(a, 0.5)
    ctx.autotune(a, 0.5, reps=2)
    text = ctx.tuning_export()
    other = pkg.Context(0, workspace_bytes=pkg.workspace_bytes(m, n))
    other.tuning_import(text)
    for c in (ctx, other):
        y = c.polar(a, 0.5)
        assert float((y - before).double().norm()) <= 1e-5 * float(before.double().norm())
