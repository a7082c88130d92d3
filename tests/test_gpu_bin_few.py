"""The binning's depth sort at and around the number of entries one cluster of
blocks sorts (49 152): every view's list, with one bin a view, is its visible
entries in a stable sort of the depth bits, bit for bit."""
import pytest
import torch

from paper_2403_01444_gb300 import gs3
from paper_2403_01444_gb300.engine import Rasterizer

pytestmark = pytest.mark.gpu
DEV = "cuda"
W, H, BIN = 512, 480, 64


@pytest.mark.parametrize("culled", [False, True])
@pytest.mark.parametrize("depths", ["random", "one", "low byte", "high bytes"])
@pytest.mark.parametrize("V,N", [(1, 1), (1, 33), (3, 700), (1, 8191), (2, 4097), (1, 40961), (5, 6553), (4, 12288),
                                 (1, 49153)])
def test_lists_are_stable_sorts_of_the_depth_bits(V, N, depths, culled):
    gen = torch.Generator(device=DEV).manual_seed(V * N)
    r = Rasterizer(N, V, W, H, V * N + 1, DEV, bin=BIN)
    p = r.proj
    p.mean2d.copy_(torch.rand(V, N, 2, device=DEV, generator=gen) * torch.tensor([W, H], device=DEV))
    bits = torch.randint(0, 1 << 23, (V, N), device=DEV, generator=gen, dtype=torch.int32)
    base = 0x40000000   # 2.0
    if depths == "random":
        bits[:, ::5] = bits[:, :1].clone()
    elif depths == "one":
        bits[:] = 77
    elif depths == "low byte":
        bits &= 0xff
    else:
        bits &= 0x7f0000
    p.depth.copy_((bits + base).view(torch.float32))
    p.radius.fill_(5)
    if culled:
        p.radius.copy_(torch.randint(0, 3, (V, N), device=DEV, generator=gen, dtype=torch.int32))
    for t in (p.conic_opacity, p.rgb, p.tiles_touched):
        t.zero_()
    for _ in range(2):   # a second call meets the first one's scratch
        gs3.gs_bin_sort(p, N, V, W, H, BIN, r.capacity, r.vals, r.ranges, None, r.d_count, r.d_err, r.ws)
    assert gs3.bins_of(W, H, BIN) == 1 and int(r.d_err) == 0
    at = 0
    for v in range(V):
        seen = (p.radius[v] > 0).nonzero()[:, 0]
        want = seen[torch.sort(bits[v][seen], stable=True).indices]
        c = len(seen)
        assert r.ranges[v].tolist() == ([at, at + c] if c else [0, 0])
        assert torch.equal(r.vals[at:at + c].long(), want)
        at += c
    assert r.count() == at
