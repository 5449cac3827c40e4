"""The stage traffic that bench.py reports is that of the kernels it timed: the
committed summary of the sum-factorised kernels does not stand for runs on the
fused kernel (x3 on mma.sync, the diffusion operator)."""
import argparse
import os
import sys

import pytest

pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("head,backend,diffusion,fused", [
    ("x3", "tcgen05", 0.0, False), ("learned-x3", "tcgen05", 0.0, False), ("x3", "mma", 0.0, True),
    ("learned-x3", "mma", 0.0, True), ("f32", "mma", 0.0, False), ("f32", "tcgen05", 1e-3, True),
    ("x3", "tcgen05", 1e-3, True)])
def test_traffic_of_the_kernels_that_ran(monkeypatch, head, backend, diffusion, fused):
    monkeypatch.setattr(bench, "profiled_traffic", lambda variant, N: (variant, N))
    name, traffic = bench.stage_kernels(head, argparse.Namespace(x3_backend=backend, diffusion=diffusion, N=64))
    assert traffic == (None if fused else (head, 64))
    assert name.startswith("k_tile" if fused else "k_sf")
