"""Serving beside a large request: no window waits for the load of a kernel.

In a process of its own (kernels are loaded once a process): a lone small request first, which loads what
any window needs, then bursts that move the windows through their tile widths, each beside a large one that
keeps the GPU busy for some 30 ms. The scheduler's trace has the host time of each window; one that loads a
kernel holds it until the large lane's launches in flight are done (4.4 to 6.4 ms), others take under 0.5 ms."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import time
import torch
import paper_2607_22484_gb300 as pkg

def serve(ctx, items):
    ts = [ctx.submit(a, 0.3, y, **o) for a, y, o in items]
    return ts

def wait(ctx, ts):
    for t in ts:
        while ctx.poll(t)[0] == pkg.binding.ERR_NOT_READY:
            time.sleep(1e-4)
        assert ctx.poll(t)[0] == 0

def item(m, n, **o):
    a = torch.randn(m, n, device="cuda") / max(m, n) ** 0.5
    return a, torch.empty_like(a), dict(dict(iters=20, prec="bf16"), **o)

ctx = pkg.Context(0, workspace_bytes=pkg.workspace_bytes(8192, 4096, prec="fp32") + (1 << 30))
big = item(8192, 4096, prec="fp32")
lone = item(200, 180)
bursts = [[item(300, 280)], [item(512, 500) for _ in range(8)], [item(900, 700) for _ in range(8)],
          [item(1000, 900) for _ in range(10)], [item(2000, 1500) for _ in range(4)]]
torch.cuda.synchronize()
wait(ctx, serve(ctx, [lone]))
for b in bursts:
    t = serve(ctx, [big])
    time.sleep(0.004)
    wait(ctx, serve(ctx, b))
    wait(ctx, t)
"""


def test_no_window_waits_for_a_kernel_to_load(tmp_path):
    trace = tmp_path / "trace.txt"
    env = dict(os.environ, SVT_SERVE_TRACE=str(trace), PYTHONPATH=ROOT)
    env.pop("CUDA_MODULE_LOADING", None)
    subprocess.run([sys.executable, "-c", PROGRAM], check=True, env=env, cwd=ROOT, timeout=300)
    events = [line.split() for line in trace.read_text().splitlines()]
    start = next(i for i, e in enumerate(events) if e[1] == "large_launch")
    us = [int(e[3]) for e in events[start:] if e[1] == "window"]
    print("host time of a window, us:", sorted(us)[-5:])
    assert len(us) > 10
    assert max(us) < 2500
