"""Chain-mode dependencies of fused launches (csrc/fused_deps.h), checked exactly on the host.

tests/chain_order_check.cpp derives the conditions of a solve's products, whole and cut into
windows, and requires a chain of waits between any two that touch the same memory: a product
that lags behind everything not waiting for it must still find its operands unchanged.
Without the wait of the P chain's second X Z for the shifted Gram (both use X0^T) it fails."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2607_22484_gb300", "csrc")


def test_chain_waits_order_all_shared_memory(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-I", CSRC,
                    os.path.join(HERE, "chain_order_check.cpp"), "-o", exe],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert " 0 failures" in r.stdout, r.stdout
