"""Autotuning shapes that run as one launch in shared memory: there is no mode to choose, so nothing is
stored, and a choice imported for one (a cache written before) leaves its solves as they are.

Tolerance: 0, the same launch on the same input."""
import json

import pytest
import torch

import paper_2607_22484_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [dict(prec="bf16"), dict(prec="fp32", mode="rank_r"), dict(prec="bf16", tile=256)])
@pytest.mark.parametrize("m,n", [(128, 128), (96, 80), (1, 5)])
def test_nothing_is_stored_for_one_launch_solves(m, n, opts):
    a = torch.randn(m, n, device="cuda") / max(m, n) ** 0.5
    ctx = pkg.Context(0, workspace_bytes=1 << 20)
    plain = {k: v for k, v in opts.items() if k != "tile"}
    want = ctx.polar(a, 0.3, **plain).clone()
    y = ctx.autotune(a, 0.3, **opts)  # synchronises
    assert torch.equal(y, want)
    assert json.loads(ctx.tuning_export())["entries"] == []


def test_imported_choice_has_no_effect():
    a = torch.randn(100, 90, device="cuda") / 10
    ctx = pkg.Context(0, workspace_bytes=1 << 20)
    ctx.autotune(torch.randn(300, 280, device="cuda"), 0.3)
    doc = json.loads(ctx.tuning_export())
    doc["entries"][0].update(m=100, n=90)
    want = ctx.polar(a, 0.3).clone()
    ctx.tuning_import(json.dumps(doc))
    before = ctx.launch_count()
    y = ctx.polar(a, 0.3)
    torch.cuda.synchronize()
    assert ctx.launch_count() - before == 1
    assert torch.equal(y, want)
