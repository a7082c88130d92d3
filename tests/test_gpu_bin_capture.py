"""Binning in groups of views under stream capture: the captured launches are
the eager ones, whatever was called before them, so the lists are equal bit
for bit."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2403_01444_gb300 import gs3
from paper_2403_01444_gb300.engine import Rasterizer

pytestmark = pytest.mark.gpu
DEV = "cuda"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# 920 bins a view, so groups of two views, the last of one
V, N, W, H, BIN, CAP = 5, 200_003, 1920, 1080, 3, 16_000_000


def _sorter():
    g = torch.Generator(device=DEV).manual_seed(11)
    p = gs3.Projected.empty(V, N)
    p.mean2d.uniform_(-0.1, 1.1, generator=g).mul_(torch.tensor([W, H], device=DEV, dtype=torch.float32))
    p.depth.uniform_(0.5, 8.0, generator=g)
    p.radius.random_(0, 40, generator=g)
    r = Rasterizer(0, V, W, H, CAP, DEV, bin=BIN)
    ws = torch.empty(gs3.gs_bin_sort_workspace_size(N, V, W, H, CAP), dtype=torch.uint8, device=DEV)
    return r, lambda: gs3.gs_bin_sort(p, N, V, W, H, BIN, CAP, r.vals, r.ranges, None, r.d_count, r.d_err, ws)


def _captured(r, sort):
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        sort()
    r.vals.zero_()
    r.ranges.zero_()
    graph.replay()
    torch.cuda.synchronize()
    return r.count(), r.vals.clone(), r.ranges.clone()


def _assert_equal(got, r, sort):
    r.vals.zero_()
    r.ranges.zero_()
    sort()
    n = r.count()
    assert got[0] == n > 0 and int(r.d_err) == 0
    assert torch.equal(got[1], r.vals) and torch.equal(got[2], r.ranges)


@pytest.mark.parametrize("before", ["the same call", "a call of one small view"])
def test_captured_after_eager_calls(before):
    bins = gs3.bins_of(W, H, BIN)
    assert 2 * bins <= 2048 < 3 * bins and V % 2 == 1
    r, sort = _sorter()
    sort()
    if before != "the same call":
        q = Rasterizer(100, 1, 64, 48, 1000, DEV, bin=1)
        p = gs3.Projected.empty(1, 100)
        p.radius.zero_()
        ws = torch.empty(gs3.gs_bin_sort_workspace_size(100, 1, 64, 48, 1000), dtype=torch.uint8, device=DEV)
        gs3.gs_bin_sort(p, 100, 1, 64, 48, 1, 1000, q.vals, q.ranges, None, q.d_count, q.d_err, ws)
    _assert_equal(_captured(r, sort), r, sort)


def test_captured_as_a_process_s_first_call():
    code = ("import sys; sys.path[:0] = [%r, %r]\n"
            "import test_gpu_bin_capture as t\n"
            "r, sort = t._sorter()\n"
            "t._assert_equal(t._captured(r, sort), r, sort)\n" % (ROOT, os.path.join(ROOT, "tests")))
    p = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
