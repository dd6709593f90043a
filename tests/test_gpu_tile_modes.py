"""Which tiles a call runs on, and solves and batches on tiles that only the automatic choice has. Each case
first checks the choice itself, so that a moved line of the rule fails the test instead of emptying it.

Tolerances: 1e-5, the bound between execution paths of one solve; 2e-2 and 1e-4, the tiers', against Eq. 1."""
import json

import numpy as np
import pytest
import torch

import oracle
import paper_2607_22484_gb300 as pkg
import svt_workloads as wl

pytestmark = pytest.mark.gpu

PAIR128, PAIR = 384, 512


def _rel(y, r):
    return float((y - r).double().norm()) / float(r.double().norm())


@pytest.mark.parametrize("m,n,prec", [(1601, 1701, "bf16"), (2300, 1501, "bf16"), (1301, 2500, "bf16"),
                                      (4096, 1024, "bf16"), (650, 8000, "bf16"), (1300, 1290, "fp32"),
                                      (2100, 1030, "fp32"), (9000, 500, "fp32"), (531, 8100, "fp32")])
def test_pairs_of_256x128_by_choice(m, n, prec):
    ctx = pkg.Context(0, workspace_bytes=pkg.workspace_bytes(m, n, prec=prec))
    g = torch.Generator(device="cuda")
    g.manual_seed(m + 2 * n)
    a = torch.randn(m, n, generator=g, device="cuda") / max(m, n) ** 0.5
    for o in (dict(), dict(mode="rank_r"), dict(polish=False), dict(schedule="ns3")):
        assert ctx.tile_mode([(m, n)], prec=prec, iters=8, **o) == PAIR128, o
        sts = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(2)]
        y = ctx.polar(a, 0.5, status=sts[0], prec=prec, iters=8, **o)
        ref = ctx.polar(a, 0.5, status=sts[1], prec=prec, iters=8, tile=128, **o)
        assert int(sts[0]) == int(sts[1]) == 0
        assert _rel(y, ref) <= 1e-5, o


@pytest.mark.parametrize("prec,bound", [("bf16", 2e-2), ("fp32", 1e-4)])
def test_pairs_of_256x128_against_the_oracle(prec, bound):
    m, n = 1701, 1601
    s = np.concatenate([np.linspace(1.0, 0.36, n // 4), np.linspace(0.24, 0.01, n - n // 4)])
    a = wl.spectrum_matrix(s, m, n, 17)
    ctx = pkg.Context(0, workspace_bytes=pkg.workspace_bytes(m, n, prec=prec))
    assert ctx.tile_mode([(m, n)], prec=prec) == PAIR128
    y = ctx.polar(torch.from_numpy(a).cuda(), 0.3, prec=prec)
    torch.cuda.synchronize()
    assert oracle.relerr(y.cpu().numpy(), oracle.svt_definition(a.astype(np.float64), 0.3)) < bound


def test_modes_of_single_solves():
    """The automatic choice, an explicit tile, and an imported choice, of which 128 stands for the automatic
    one where that is finer."""
    ctx = pkg.Context(0, workspace_bytes=1 << 20)
    for (m, n), auto in (((128, 90), 1), ((300, 300), 64), ((1000, 1001), 64), ((4096, 4096), PAIR)):
        assert ctx.tile_mode([(m, n)]) == auto
        for tile in (128, 256, 512):
            assert ctx.tile_mode([(m, n)], tile=tile) == tile
    assert ctx.tile_mode([(300, 300)], prec="fp64") == ctx.tile_mode([(300, 300)], fuse=False) == 0
    a = torch.randn(300, 300, device="cuda") / 300 ** 0.5
    ctx.autotune(a, 0.5)
    doc = json.loads(ctx.tuning_export())
    for width, mode in ((128, 64), (256, 256), (512, 512)):
        doc["entries"][0]["widths"] = [width] * len(doc["entries"][0]["widths"])
        other = pkg.Context(0, workspace_bytes=1 << 20)
        other.tuning_import(json.dumps(doc))
        assert other.tile_mode([(300, 300)]) == mode
        assert _rel(other.polar(a, 0.5), ctx.polar(a, 0.5, tile=128)) <= 1e-5


@pytest.mark.parametrize("count,lo,hi,prec,mode", [(5, (60, 60), (250, 250), "bf16", 64),
                                                   (40, (100, 100), (400, 400), "bf16", 128),
                                                   (150, (243, 590), (256, 601), "bf16", 256),
                                                   (12, (800, 800), (1023, 1023), "bf16", PAIR),
                                                   (16, (600, 600), (900, 900), "fp32", PAIR)])
def test_batch_modes(count, lo, hi, prec, mode):
    rng = np.random.default_rng(count)
    shapes = [tuple(int(x) for x in rng.integers(lo, np.array(hi) + 1)) for _ in range(count)]
    ctx, single = (pkg.Context(0, workspace_bytes=1 << 20) for _ in range(2))
    opts = dict(iters=8, prec=prec)
    assert ctx.tile_mode(shapes, **opts) == mode
    for tile in (128, 256):
        assert ctx.tile_mode(shapes, tile=tile, **opts) == tile
    g = torch.Generator(device="cuda")
    g.manual_seed(count)
    As = [torch.randn(m, n, generator=g, device="cuda") / max(m, n) ** 0.5 for m, n in shapes]
    for y, a in zip(ctx.batch(As, [0.5] * count, opts=opts), As):
        assert _rel(y, single.polar(a, 0.5, **opts)) <= 1e-5
