"""The compositing reverse on both sides of the line at which a warp takes 8x8
or 8x16 pixels (40 tiles per SM): sixteen views in one launch, above the line,
against the same views one at a time, below it, with images that end inside
either warp's pixels, with and without the forward's lists.

The same pixels take part in the same records either way and only the order of
the FP32 additions differs: at most 2^10 terms of either sign, each rounding
below 2^-24 of a partial sum, bounded by 1e-5 of the tensor."""
import pytest
import torch

from paper_2403_01444_gb300 import gs3
from paper_2403_01444_gb300.engine import Rasterizer

pytestmark = pytest.mark.gpu
DEV = "cuda"
BG = (0.1, 0.2, 0.3)
FEW_TILES = 40


def _scene(V, N, W, H):
    gen = torch.Generator(device=DEV).manual_seed(N + W)
    u = lambda *s: torch.rand(*s, device=DEV, generator=gen)
    r = Rasterizer(N, V, W, H, 64 * N * V, DEV, bin=4)
    p = r.proj
    p.mean2d.copy_(u(V, N, 2) * torch.tensor([W, H], device=DEV))
    a, c = 0.02 + 0.2 * u(V, N), 0.02 + 0.2 * u(V, N)
    b = (u(V, N) - 0.5) * (a * c).sqrt()
    p.conic_opacity.copy_(torch.stack([a, b, c, 0.05 + 0.95 * u(V, N)], -1))
    p.rgb.copy_(u(V, N, 3))
    p.depth.copy_(1.0 + u(V, N))
    p.radius.fill_(24)
    d_img = u(V, 3, H, W) - 0.5
    return r, d_img


def _gradients(r, d_img, lists):
    V, N, W, H = r.V, r.n, r.W, r.H
    g = torch.zeros(V, N, 8, device=DEV)
    o = torch.zeros(V, N, device=DEV)
    gs3.gs_bin_sort(r.proj, N, V, W, H, r.bin, r.capacity, r.vals, r.ranges, None, r.d_count, r.d_err, r.ws)
    gs3.gs_raster_fwd(r.proj, N, V, W, H, r.bin, BG, r.vals, r.ranges, r.img, r.T_final, r.last, lists=r.lists)
    gs3.gs_raster_bwd(r.proj, N, V, W, H, r.bin, BG, r.vals, r.ranges, r.T_final, r.last, d_img, g, o,
                      lists=r.lists if lists else None)
    torch.cuda.synchronize()
    assert int(r.d_err.item()) == 0
    return g, o


@pytest.mark.parametrize("lists", [True, False])
@pytest.mark.parametrize("N,W,H", [(2000, 313, 305), (700, 316, 312)])
def test_reverse_is_the_same_on_both_sides_of_the_line(N, W, H, lists):
    V = 16
    tiles = ((W + 15) // 16) * ((H + 15) // 16)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert tiles <= FEW_TILES * sms < V * tiles
    r, d_img = _scene(V, N, W, H)
    g, o = _gradients(r, d_img, lists)
    one = Rasterizer(N, 1, W, H, 64 * N, DEV, bin=4)
    for v in range(V):
        for f in ("mean2d", "conic_opacity", "rgb", "depth", "radius"):
            getattr(one.proj, f).copy_(getattr(r.proj, f)[v:v + 1])
        g1, o1 = _gradients(one, d_img[v:v + 1].contiguous(), lists)
        for k in range(8):
            a, b = g[v, :, k].double(), g1[0, :, k].double()
            assert float((a - b).norm()) <= 1e-5 * float(b.norm())
        a, b = o[v].double(), o1[0].double()
        assert float((a - b).norm()) <= 1e-5 * float(b.norm())
