"""Long, narrow solves in one launch: the shifted Gram reads X0^T for longer than the P chain needs to
reach the product that overwrites it. Alone, in a batch and served together, tall and wide, against
the same solves launch by launch.

Tolerance: 1e-5, the bound between execution paths of one solve."""
import time

import pytest
import torch

import paper_2607_22484_gb300 as pkg

pytestmark = pytest.mark.gpu

SHAPES = [(16384, 256), (50000, 64), (300, 16000), (131, 40000)]


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
def test_long_narrow_solves(prec):
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    As = []
    for m, n in SHAPES:
        k = min(m, n)
        a = torch.randn(max(m, n), k, generator=g, device="cuda") / max(m, n) ** 0.5
        a *= torch.linspace(0.05, 1.0, k, device="cuda")
        As.append((a if m > n else a.T).contiguous())
    opts = dict(iters=12, prec=prec)
    one = pkg.Context(0, workspace_bytes=1 << 20)
    refs = [one.polar(a, 0.3, fuse=False, **opts).clone() for a in As]

    def same(y, r):
        assert float((y - r).double().norm()) <= 1e-5 * float(r.double().norm()), tuple(r.shape)

    for a, r in zip(As, refs):
        same(one.polar(a, 0.3, **opts), r)
        same(one.polar(a, 0.3, tile=128, **opts), r)
    for _ in range(2):
        for y, r in zip(one.batch(As, [0.3] * len(As), opts=opts), refs):
            same(y, r)
    ctx = pkg.Context(0, workspace_bytes=1 << 30)
    for order in ([0, 1, 2, 3], [3, 1, 0, 2], [1]):
        outs = [torch.full_like(As[i], float("nan")) for i in order]
        torch.cuda.synchronize()
        tickets = [ctx.submit(As[i], 0.3, y, **opts) for i, y in zip(order, outs)]
        for t in tickets:
            end = time.time() + 60
            st, _ = ctx.poll(t)
            while st == pkg.binding.ERR_NOT_READY and time.time() < end:
                time.sleep(1e-4)
                st, _ = ctx.poll(t)
            assert st == 0
            ctx.release(t)
        for i, y in zip(order, outs):
            same(y, refs[i])
