"""Binning whose keys are taken in groups of views: the same lists as binning
each view by itself, bit for bit, and nothing usable over capacity."""
import pytest
import torch

from paper_2403_01444_gb300 import gs3
from paper_2403_01444_gb300.engine import Rasterizer

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2403_01444_gb300 import build
    build.build()
    gs3.lib()


def _records(V, N, W, H):
    g = torch.Generator(device=DEV)
    g.manual_seed(V * N)
    p = gs3.Projected.empty(V, N)
    p.mean2d.uniform_(-0.1, 1.1, generator=g).mul_(torch.tensor([W, H], device=DEV, dtype=torch.float32))
    p.depth.uniform_(0.5, 8.0, generator=g)
    p.depth[:, ::7] = p.depth[:, :1]     # equal depths: ties by index
    p.radius.random_(0, 40, generator=g)
    for t in (p.conic_opacity, p.rgb, p.tiles_touched):
        t.zero_()
    return p


def _sort(p, N, V, W, H, bin, capacity):
    r = Rasterizer(0, V, W, H, capacity, DEV, bin=bin)
    ws = torch.empty(gs3.gs_bin_sort_workspace_size(N, V, W, H, capacity), dtype=torch.uint8, device=DEV)
    keys = torch.zeros(max(capacity, 1), dtype=torch.int64, device=DEV)
    gs3.gs_bin_sort(p, N, V, W, H, bin, capacity, r.vals, r.ranges, keys, r.d_count, r.d_err, ws)
    return r, keys


# groups of one view each (2 040 bins a view), and of two views, the last of one
@pytest.mark.parametrize("V,N,W,H,bin", [(2, 400_001, 1920, 1080, 2), (5, 200_003, 1920, 1080, 3)])
def test_groups_of_views_equal_single_views(V, N, W, H, bin):
    bins = gs3.bins_of(W, H, bin)
    assert V * bins > 2048 >= bins
    p = _records(V, N, W, H)
    cap = 16_000_000
    r, keys = _sort(p, N, V, W, H, bin, cap)
    total = r.count()
    assert int(r.d_err) == 0 and 0 < total <= cap
    at = 0
    for v in range(V):
        one = gs3.Projected(*(getattr(p, f)[v:v + 1] for f in ("mean2d", "conic_opacity", "rgb", "depth", "radius",
                                                              "tiles_touched")))
        q, k = _sort(one, N, 1, W, H, bin, cap)
        c = q.count()
        assert torch.equal(r.vals[at:at + c], q.vals[:c])
        assert torch.equal(keys[at:at + c], k[:c] + ((v * bins) << 32))
        mine, want = r.ranges.view(V, bins, 2)[v], q.ranges.view(bins, 2)
        full = want[:, 1] > want[:, 0]
        assert torch.equal(mine[full], want[full] + at) and not mine[~full].any()
        at += c
    assert at == total
    for capacity in (total - 1, total // (2 * V)):
        q, _ = _sort(p, N, V, W, H, bin, capacity)
        assert q.count() == total and int(q.d_err) == gs3.GS_ERR_CAPACITY and not q.ranges.any()
