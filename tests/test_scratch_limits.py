"""Workspace sizes at the fixed 32 MiB of the no-allocation call: the largest of these shapes that fit.

A longer product table would shut them out (256 bytes more a product did: 65 shapes of width 64 alone)."""
import pytest
import torch

import paper_2607_22484_gb300 as pkg

LIMIT = pkg.binding.NOALLOC_SCRATCH_BYTES
CASES = [((36904, 64), {}), ((25856, 64), dict(prec="fp32")), ((35478, 64), dict(iters=100)),
         ((25664, 128), dict(mode="rank_r")), ((832, 832), {})]


@pytest.mark.parametrize("shape,opts", CASES)
def test_shapes_that_fit_the_fixed_scratch(shape, opts):
    assert pkg.workspace_bytes(*shape, **opts) <= LIMIT


def test_workspace_of_a_solve():
    assert pkg.workspace_bytes(1000, 1000) <= 47319040
    assert pkg.workspace_bytes(1000, 1000, prec="fp32") <= 57559040


@pytest.mark.gpu
@pytest.mark.parametrize("shape,opts", CASES[:2])
def test_no_allocation_call_at_the_limit(shape, opts):
    a = torch.randn(*shape, device="cuda") / shape[0] ** 0.5
    st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    y = torch.empty_like(a)
    pkg.polar_noalloc(a, 0.5, out=y, status=st, **opts)
    ref = pkg.Context(0, workspace_bytes=1 << 20).polar(a, 0.5, **opts)
    torch.cuda.synchronize()
    assert int(st) == 0
    assert float((y - ref).double().norm()) <= 1e-5 * float(ref.double().norm())
