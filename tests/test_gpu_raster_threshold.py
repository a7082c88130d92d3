"""Compositing of records whose opacity is 1/255 or the next floats to it: the
threshold power log2(255 o) is 0 or its rounding, of either sign.  Only the
pixel on the mean can reach alpha >= 1/255 there, so every other pixel keeps
the background, T = 1 and no contributor, bit for bit; on the mean a record
that takes part has alpha = o, and the reverse gives a colour gradient exactly
where the forward added."""
import numpy as np
import pytest
import torch

from paper_2403_01444_gb300 import gs3
from paper_2403_01444_gb300.engine import Rasterizer

pytestmark = pytest.mark.gpu
DEV = "cuda"
BG = (0.25, 0.5, 0.75)


@pytest.mark.parametrize("lists", [True, False])
@pytest.mark.parametrize("bin", [1, 4])
def test_opacities_at_the_threshold(bin, lists):
    N = 64
    W, H = 16 * N, 16
    o = np.full(N, np.float32(1.0) / np.float32(255.0), np.float32)
    for k in range(N):   # 8 floats below, the others above
        for _ in range(abs(k - 8)):
            o[k] = np.nextafter(o[k], np.float32(0.0 if k < 8 else 1.0))
    assert (np.float32(255.0) * o < 1).any() and (np.float32(255.0) * o == 1).any()
    r = Rasterizer(N, 1, W, H, 64 * N, DEV, bin=bin)
    p = r.proj
    x = torch.arange(N, device=DEV) * 16
    p.mean2d.copy_(torch.stack([x + 5.5, torch.full_like(x, 9.5, dtype=torch.float32)], -1)[None])
    conic = torch.tensor([0.5, 0.125, 0.25, 0.0], device=DEV).repeat(1, N, 1)
    conic[..., 3] = torch.from_numpy(o).to(DEV)
    p.conic_opacity.copy_(conic)
    p.rgb.fill_(1.0)
    p.depth.fill_(1.0)
    p.radius.fill_(5)
    gs3.gs_bin_sort(p, N, 1, W, H, bin, r.capacity, r.vals, r.ranges, None, r.d_count, r.d_err, r.ws)
    gs3.gs_raster_fwd(p, N, 1, W, H, bin, BG, r.vals, r.ranges, r.img, r.T_final, r.last,
                      lists=r.lists if lists else None)
    d_img = torch.full((1, 3, H, W), 2.0, device=DEV)
    g, d_op = torch.zeros(1, N, 8, device=DEV), torch.zeros(1, N, device=DEV)
    gs3.gs_raster_bwd(p, N, 1, W, H, bin, BG, r.vals, r.ranges, r.T_final, r.last, d_img, g, d_op,
                      lists=r.lists if lists else None)
    torch.cuda.synchronize()
    T, last = r.T_final[0], r.last[0]
    on = torch.zeros(H, W, dtype=torch.bool, device=DEV)
    on[9, x + 5] = True
    bg = torch.tensor(BG, device=DEV)[:, None]
    assert bool((T[~on] == 1).all()) and not last[~on].any()
    assert bool((r.img[0][:, ~on] == bg).all())
    added = (last[on] > 0)
    od = torch.from_numpy(o).to(DEV)
    assert bool(added[od * 255 > 1 + 1e-6].all()) and not added[od * 255 < 1].any()
    assert bool((T[on][~added] == 1).all()) and bool((r.img[0][:, on][:, ~added] == bg).all())
    assert float((T[on] - torch.where(added, 1 - od, 1.0)).abs().max()) <= 2.0 ** -23
    assert torch.equal(g[0, :, 5] != 0, added) and torch.equal(d_op[0] != 0, added)
    assert bool(torch.isfinite(g).all()) and bool(torch.isfinite(d_op).all())
