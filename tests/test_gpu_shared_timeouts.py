"""Launches that several solves share (batches, serving windows) when a dependency wait gives up: with a
limit of 1 ns, waits of more than a few dozen polls (about 0.1 ms) do. In one of the solves they last
longer (50000 x 64: a tile of the Gram sums over 2346 k-blocks, some 0.3 ms). Every solve then is right or
reports SVT_ERR_TIMEOUT, that one reports it, and with the default limit the context solves all again.

Tolerance: 1e-5, the bound between execution paths of one solve."""
import time

import pytest
import torch

import paper_2607_22484_gb300 as pkg

pytestmark = pytest.mark.gpu
B = pkg.binding

SHAPES = [(200, 180), (50000, 64), (140, 300)]
LONG = 1
ORDERS = [[0, 1, 2], [1, 0, 2], [2, 0, 1]]
OPTS = dict(iters=10, prec="bf16")


def _problems():
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    As = [torch.randn(m, n, generator=g, device="cuda") / max(m, n) ** 0.5 for m, n in SHAPES]
    one = pkg.Context(0, workspace_bytes=1 << 20)
    return As, [one.polar(a, 0.3, **OPTS).clone() for a in As]


def _check(order, As, refs, outs, sts, limited):
    for i, y, st in zip(order, outs, sts):
        assert st in ((B.OK, B.ERR_TIMEOUT) if limited else (B.OK,)), (i, st)
        if st == B.OK:
            assert float((y - refs[i]).double().norm()) <= 1e-5 * float(refs[i].double().norm()), i
    if limited:
        assert sts[order.index(LONG)] == B.ERR_TIMEOUT


@pytest.mark.parametrize("order", ORDERS)
def test_batch(order):
    As, refs = _problems()
    ctx = pkg.Context(0, workspace_bytes=256 << 20)
    for limit in (1, 0, 1, 0):
        ctx.debug("wait_limit_ns", limit)
        outs = [torch.full_like(As[i], float("nan")) for i in order]
        sts = [torch.full((1,), -1, dtype=torch.int32, device="cuda") for _ in order]
        ctx.batch([As[i] for i in order], [0.3] * 3, outs=outs, statuses=sts, opts=OPTS)
        torch.cuda.synchronize()
        _check(order, As, refs, outs, [int(s) for s in sts], limit == 1)


@pytest.mark.parametrize("order", ORDERS)
def test_serving(order):
    As, refs = _problems()
    ctx = pkg.Context(0, workspace_bytes=256 << 20)
    ctx.debug("admit_delay_us", 20000)  # the three are admitted together
    for limit in (1, 0):
        ctx.debug("wait_limit_ns", limit)
        outs = [torch.full_like(As[i], float("nan")) for i in order]
        torch.cuda.synchronize()
        tickets = [ctx.submit(As[i], 0.3, y, **OPTS) for i, y in zip(order, outs)]
        sts = []
        for t in tickets:
            end = time.time() + 60
            st, _ = ctx.poll(t)
            while st == B.ERR_NOT_READY and time.time() < end:
                time.sleep(1e-4)
                st, _ = ctx.poll(t)
            sts.append(st)
            ctx.release(t)
        _check(order, As, refs, outs, sts, limit == 1)
