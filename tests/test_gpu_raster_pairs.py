"""The reverse's pair counts: a pixel walks the records of its tile's list that
lie before its last contributor, however the launch cuts the tile between warps
and whether the records come from the forward's lists or from the bins', and
the pairs that contribute are those that the forward added."""
import pytest
import torch

from paper_2403_01444_gb300 import gs3
from paper_2403_01444_gb300.engine import Rasterizer
from test_gpu_raster_few_tiles import BG, DEV, FEW_TILES, _scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opacity_gradient", [False, True])
@pytest.mark.parametrize("V,N,W,H", [(1, 700, 61, 45), (2, 1500, 316, 305), (16, 2000, 313, 305)])
def test_walked_and_contributing_pairs(V, N, W, H, opacity_gradient):
    r, d_img = _scene(V, N, W, H)
    tx, ty = (W + 15) // 16, (H + 15) // 16
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (V * tx * ty > FEW_TILES * sms) == (V == 16)
    gs3.gs_bin_sort(r.proj, N, V, W, H, r.bin, r.capacity, r.vals, r.ranges, None, r.d_count, r.d_err, r.ws)
    fwd = torch.zeros(2, dtype=torch.int64, device=DEV)
    gs3.gs_raster_fwd(r.proj, N, V, W, H, r.bin, BG, r.vals, r.ranges, r.img, r.T_final, r.last, fwd, lists=r.lists)
    got = []
    for lists in (r.lists, None):
        bwd = torch.zeros(2, dtype=torch.int64, device=DEV)
        g = torch.zeros(V, N, 8, device=DEV)
        o = torch.zeros(V, N, device=DEV) if opacity_gradient else None
        gs3.gs_raster_bwd(r.proj, N, V, W, H, r.bin, BG, r.vals, r.ranges, r.T_final, r.last, d_img, g, o, bwd,
                          lists=lists)
        got.append(bwd.tolist())
    torch.cuda.synchronize()
    assert int(r.d_err.item()) == 0
    count = r.lists.count.view(V, ty, tx).long()
    assert int(count.min()) >= 0   # every tile has its list
    cap = r.lists.rec.view(V, ty, tx, -1, 2).shape[3]
    pos = r.lists.rec.view(V, ty, tx, cap, 2)[..., 1].long()
    pos = torch.where(torch.arange(cap, device=DEV) < count[..., None], pos, 1 << 40)
    last = torch.zeros(V, 16 * ty, 16 * tx, dtype=torch.int64, device=DEV)
    last[:, :H, :W] = r.last
    last = last.view(V, ty, 16, tx, 16).permute(0, 1, 3, 2, 4).reshape(V, ty, tx, 256)
    walked = int(torch.searchsorted(pos.contiguous(), last.contiguous()).sum())   # records before each pixel's last
    assert got[0] == got[1] == [walked, int(fwd[1])] and walked > int(fwd[1]) > 0
