"""FP64 tier at the edges of its 8 x 8 product tiles and 32-deep K stages, against the oracle.

Tolerance: the tier's 1e-9 relative, on its FP64 result, for the FP32 value of tau."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_22484_gb300 as pkg
import svt_workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule,norm", [("pe5", "auto"), ("ns3", "fro"), ("ns3", "gram")])
@pytest.mark.parametrize("m,n", [(1, 1), (7, 8), (8, 8), (9, 7), (31, 33), (32, 32), (40, 64),
                                 (65, 63), (129, 257), (300, 96)])
def test_f64_tile_edges(m, n, schedule, norm):
    k = min(m, n)
    hi = max(1, k // 4)
    s = np.concatenate([np.linspace(1.0, 0.36, hi), np.linspace(0.24, 0.05, k - hi)])
    a = wl.spectrum_matrix(s, m, n, 11 * m + n)
    ctx = pkg.Context(0, workspace_bytes=pkg.workspace_bytes(m, n, prec="fp64", iters=40))
    buf = torch.full((m, n + 3), float("nan"), device="cuda")
    buf[:, :n] = torch.from_numpy(a)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    y = ctx.polar_f64(buf[:, :n], 0.3, status=st, iters=40, schedule=schedule, norm=norm)
    exact = oracle.svt_definition(a.astype(np.float64), float(np.float32(0.3)))
    assert int(st) == 0
    assert oracle.relerr(y.cpu().numpy(), exact) < 1e-9
