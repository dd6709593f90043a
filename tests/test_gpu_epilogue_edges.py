"""Product-kernel epilogues where their 32-column blocks, 64-column units and diagonal blocks end:
solves whose smaller side lies around multiples of 32 and 64 above one tile, in every tile mode,
fused and launch by launch, against the oracle and against each other.

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
@pytest.mark.parametrize("m,n", [(129, 129), (130, 159), (160, 160), (161, 193), (300, 191),
                                 (192, 256), (255, 257), (289, 288), (321, 140), (516, 383)])
def test_epilogue_edges(m, n, prec):
    k = min(m, n)
    hi = k // 4
    s = np.concatenate([np.linspace(1.0, 0.36, hi), np.linspace(0.24, 0.01, k - hi)])
    a = wl.spectrum_matrix(s, m, n, 3 * m + n)
    exact = oracle.svt_definition(a.astype(np.float64), 0.3)
    ctx = pkg.Context(0, workspace_bytes=pkg.workspace_bytes(m, n, prec=prec))
    dev = torch.from_numpy(a).cuda()
    first = None
    for o in (dict(tile=128), dict(tile=256), dict(tile=512), dict(fuse=False), dict()):
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        y = ctx.polar(dev, 0.3, status=st, prec=prec, **o)
        assert int(st) == 0
        assert oracle.relerr(y.cpu().numpy(), exact) < BOUND[prec], o
        if first is None:
            first = y
        assert float((y - first).double().norm()) <= 1e-5 * float(first.double().norm()), o


@pytest.mark.parametrize("m,n,prec", [(700, 523, "fp32"), (531, 900, "fp32"), (1100, 257, "fp32"),
                                      (4100, 300, "bf16"), (260, 4300, "bf16"), (1500, 1601, "bf16"),
                                      (2600, 130, "fp32")])
def test_pairs_of_256x128(m, n, prec):
    """Shapes that the automatic choice runs on CTA pairs of 256 x 128 tiles (long K), ragged in
    both directions, against 128 x 128 tiles: 1e-5, the bound between execution paths."""
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n)
    a = torch.randn(m, n, generator=g, device="cuda") / max(m, n) ** 0.5
    ctx = pkg.Context(0, workspace_bytes=pkg.workspace_bytes(m, n, prec=prec))
    for o in (dict(), dict(mode="rank_r"), dict(polish=False), dict(schedule="ns3")):
        sts = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(2)]
        y = ctx.polar(a, 0.5, status=sts[0], prec=prec, iters=8, **o)
        ref = ctx.polar(a, 0.5, status=sts[1], prec=prec, iters=8, tile=128, **o)
        assert int(sts[0]) == int(sts[1]) == 0
        assert float((y - ref).double().norm()) <= 1e-5 * float(ref.double().norm()), o
