"""Products over very long K through the diagnostic entry points: around 2^22 (BF16) and 2^23 (e4m3), where
a segment has 2^16 k-blocks, and past them; every segment count and tile mode, with and without a remainder.

Exact: the operands hold 0, 1 and -1, and R so few of them that every sum is a small whole number."""
import pytest
import torch

import paper_2607_22484_gb300 as pkg

pytestmark = pytest.mark.gpu

M, N = 40, 24


def _operand(rows, k, keep, seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randint(0, 2, (rows, k), generator=g, device="cuda", dtype=torch.int8) * 2 - 1
    if keep > 1:
        x[:, torch.randint(0, keep, (k,), generator=g, device="cuda") != 0] = 0
    x[:, -1] = 1
    return x.to(dtype)


def _exact(L, R):
    out = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    for k in range(0, L.shape[1], 1 << 20):
        out += L[:, k:k + (1 << 20)].double() @ R[:, k:k + (1 << 20)].double().T
    return out


@pytest.fixture(scope="module")
def ctx():
    return pkg.Context(0, workspace_bytes=1 << 20)


@pytest.mark.parametrize("k", [(1 << 22) - 8, 1 << 22, (1 << 22) + 72, 5000000])
def test_bf16_long_k(ctx, k):
    Lh, Ll = (_operand(M, k, 1, s, torch.bfloat16) for s in (1, 2))
    Rh, Rl = (_operand(N, k, 4096, s, torch.bfloat16) for s in (3, 4))
    d = torch.empty(M, N, device="cuda")
    want = _exact(Lh, Rh)
    for nseg, tile in ((1, 128), (1, 256), (1, 512), (2, 0), (3, 0)):
        if nseg == 2:
            want = want + _exact(Lh, Rl)
        elif nseg == 3:
            want = want + _exact(Ll, Rh)
        d.fill_(float("nan"))
        ctx.debug_gemm_bf16(nseg, Lh, Ll if nseg == 3 else None, Rh, Rl if nseg > 1 else None, d, tile=tile)
        torch.cuda.synchronize()
        assert torch.equal(d.double(), want), (nseg, tile)


@pytest.mark.parametrize("k", [1 << 23, (1 << 23) + 144])
def test_e4m3_long_k(ctx, k):
    L = _operand(M, k, 1, 5, torch.float8_e4m3fn)
    R = _operand(N, k, 4096, 6, torch.float8_e4m3fn)
    d = torch.full((M, N), float("nan"), device="cuda")
    ctx.debug_gemm_e4m3(L.view(torch.uint8), R.view(torch.uint8), d)
    torch.cuda.synchronize()
    assert torch.equal(d.double(), _exact(L, R))
