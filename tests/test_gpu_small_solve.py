"""One-launch solves of matrices that fit one tile (both sides at most 128) against the general
path (an explicit tile mode) on the same inputs.

Both run the same products with the same segment and K order, scalings and roundings; they may
differ by the order of FP64 sums (1e-16 relative in a norm), which at worst moves an FP32 scale
by one unit in the last place. Bound: 1e-5 relative, the suite's bound between execution paths.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_22484_gb300 as pkg
import svt_workloads as wl
from paper_2607_22484_gb300 import binding as B

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (5, 3), (16, 17), (33, 128), (61, 97), (64, 64), (65, 127), (97, 61), (100, 100),
          (127, 65), (128, 1), (1, 128), (128, 128)]
OPTIONS = [dict(prec="bf16"), dict(prec="fp32"), dict(prec="fp32", schedule="ns3", iters=30),
           dict(prec="bf16", mode="rank_r"), dict(prec="fp32", norm="fro", iters=11),
           dict(prec="bf16", schedule="ns3", norm="gram", iters=25), dict(prec="bf16", iters=0),
           dict(prec="bf16", iters=1), dict(prec="bf16", iters=6, hp_steps=0),
           dict(prec="bf16", iters=128)]


def _gap(m, n, seed):
    k = min(m, n)
    hi = max(1, k // 4)
    s = np.concatenate([np.linspace(1.0, 0.36, hi), np.linspace(0.24, 0.01, k - hi)])
    return wl.spectrum_matrix(s, m, n, seed)


@pytest.fixture(scope="module")
def ctx():
    return pkg.Context(0, workspace_bytes=64 << 20)


def _both(ctx, a, tau, **o):
    sts = [torch.full((1,), -1, dtype=torch.int32, device="cuda") for _ in range(2)]
    before = ctx.launch_count()
    y = ctx.polar(a, tau, status=sts[0], **o)
    assert ctx.launch_count() == before + 1  # one launch: the small path took it
    ref = ctx.polar(a, tau, status=sts[1], tile=128, **o)
    torch.cuda.synchronize()
    return y, ref, int(sts[0]), int(sts[1])


@pytest.mark.parametrize("opts", OPTIONS, ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()))
def test_small_equals_general(ctx, opts):
    for m, n in SHAPES:
        a = torch.from_numpy(_gap(m, n, 7 * m + n)).cuda()
        y, ref, s, t = _both(ctx, a, 0.3, **opts)
        assert s == t == B.OK, (m, n)
        d = float((y - ref).double().norm())
        assert d <= 1e-5 * max(float(ref.double().norm()), 1e-3), (m, n, d)


@pytest.mark.parametrize("prec,bound", [("bf16", 2e-2), ("fp32", 1e-4)])
def test_small_against_the_oracle(ctx, prec, bound):
    for m, n in [(64, 64), (128, 100), (61, 97)]:
        a = _gap(m, n, m + n)
        y = ctx.polar(torch.from_numpy(a).cuda(), 0.3, prec=prec)
        assert oracle.relerr(y.cpu().numpy(), oracle.svt_definition(a.astype(np.float64), 0.3)) < bound


@pytest.mark.parametrize("m,n", [(97, 61), (61, 97), (64, 64), (128, 128)])
@pytest.mark.parametrize("pad_a,pad_y", [(0, 1), (1, 0), (3, 5), (4, 4)])
def test_small_strided(ctx, m, n, pad_a, pad_y):
    """Rows that are not 16-byte aligned on either side; nothing outside Y is written."""
    a = torch.from_numpy(_gap(m, n, 3)).cuda()
    buf = torch.full((m, n + pad_a), float("nan"), device="cuda")
    buf[:, :n] = a
    ybuf = torch.full((m + 1, n + pad_y), 7.5, device="cuda")
    ctx.polar(buf[:, :n], 0.3, out=ybuf[:m, :n], prec="bf16")
    ref = ctx.polar(a, 0.3, prec="bf16")
    torch.cuda.synchronize()
    assert torch.equal(ybuf[:m, :n], ref)
    ybuf[:m, :n] = 7.5
    assert bool((ybuf == 7.5).all())


def test_small_status_and_zero(ctx):
    a = torch.from_numpy(_gap(80, 50, 4)).cuda()
    for bad in (float("nan"), float("inf")):
        b = a.clone()
        b[79, 49] = bad
        _, _, s, t = _both(ctx, b, 0.3, prec="bf16")
        assert s == t == B.ERR_NONFINITE
    y, ref, s, t = _both(ctx, torch.zeros(30, 40, device="cuda"), 0.3, prec="fp32")
    assert s == t == B.OK and float(y.abs().max()) == float(ref.abs().max()) == 0.0
    # theta (the chain's norm) overflows FP32 sums in both paths: divergence is reported alike
    _, _, s, t = _both(ctx, a * 1e30, 0.3, prec="bf16")
    assert s == t


def test_small_scales(ctx):
    """||A||_F far from 1 (and exactly a power of two): the exact scaling by alpha."""
    a = torch.from_numpy(_gap(96, 64, 5)).cuda()
    for sc in (2.0 ** -40, 1e-6, 1.0, 3e5, 2.0 ** 40):
        y, ref, s, t = _both(ctx, a * sc, 0.3 * sc, prec="fp32")
        assert s == t == B.OK
        assert float((y - ref).double().norm()) <= 1e-5 * float(ref.double().norm())
    y, ref, s, t = _both(ctx, torch.eye(32, device="cuda"), 0.25, prec="fp32")
    assert s == t and float((y - ref).abs().max()) <= 1e-5


def test_small_in_the_completion_graph(ctx):
    """The launch inside a captured loop body: the device loop equals the host loop."""
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    M = torch.randn(96, 4, generator=g, device="cuda") @ torch.randn(4, 72, generator=g, device="cuda")
    mask = (torch.rand(96, 72, generator=g, device="cuda") < 0.5).to(torch.uint8)
    x, st = ctx.complete_on_device(M, mask, 0.5, 4, prec="fp32", iters=20)
    h = ctx.complete(M, mask, 0.5, 4, prec="fp32", iters=20)
    torch.cuda.synchronize()
    assert pkg.read_completion_stats(st)["status"] == B.OK
    assert float((x - h).double().norm()) <= 1e-5 * float(h.double().norm())
