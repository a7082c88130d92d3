"""The compositing reverse where its division of the work can go wrong: lists
shorter and longer than a chunk, a batch and the length that sends a tile
first; images that end inside a warp's 8x16 pixels; an odd number of tiles;
capped opacities; a pixel gradient that is not finite.

Tolerances: the oracle's as in test_gpu_kernels.py (1e-3 relative per tensor).
With and without the forward's lists the same records are walked by the same
arithmetic and only the order of the FP32 additions differs: at most 2^10 terms
of either sign, each rounding below 2^-24 of a partial sum, bounded by 1e-5."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_01444_gb300 import gs3, scenes
from paper_2403_01444_gb300.engine import Rasterizer

pytestmark = pytest.mark.gpu
DEV = "cuda"
BG = (0.1, 0.2, 0.3)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2403_01444_gb300 import build
    build.build()
    gs3.lib()
    oracle.build()


def _t(a, dtype=torch.float32):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, dtype)


def _rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30))


def _setup(rec, W, H, bin, cap):
    V, N = rec["depth"].shape
    r = Rasterizer(N, V, W, H, 4 * N * V * 64 + 16, DEV, bin=bin)
    p = r.proj
    p.mean2d.copy_(_t(rec["mean2d"]))
    p.conic_opacity.copy_(_t(np.concatenate([rec["conic"], rec["opacity"][..., None]], -1)))
    p.rgb.copy_(_t(rec["rgb"]))
    p.depth.copy_(_t(rec["depth"]))
    p.radius.copy_(_t(rec["radius"], torch.int32))
    p.tiles_touched.zero_()
    r.lists = gs3.TileLists(V, W, H, cap, DEV)
    gs3.gs_bin_sort(p, N, V, W, H, bin, r.capacity, r.vals, r.ranges, None, r.d_count, r.d_err, r.ws)
    gs3.gs_raster_fwd(p, N, V, W, H, bin, BG, r.vals, r.ranges, r.img, r.T_final, r.last, lists=r.lists)
    return r


def _reverse(r, d_img, lists, opacity=True):
    V, N, W, H = r.V, r.n, r.W, r.H
    g = torch.full((V, N, 8), 7.0, device=DEV)
    o = torch.full((V, N), 7.0, device=DEV) if opacity else None
    gs3.gs_raster_bwd(r.proj, N, V, W, H, r.bin, BG, r.vals, r.ranges, r.T_final, r.last, d_img, g, o,
                      lists=r.lists if lists else None)
    torch.cuda.synchronize()
    return g.cpu().numpy(), None if o is None else o.cpu().numpy()


@pytest.mark.parametrize("V,N,W,H,bin,cap,opacity", [
    (1, 5, 16, 16, 1, 64, None),          # fewer records than a chunk
    (1, 40, 8, 16, 1, 64, None),          # half a tile, a batch and a bit
    (3, 300, 17, 33, 1, 1024, None),      # 2 x 3 tiles, ragged both ways
    (1, 1400, 40, 24, 4, 1024, 0.01),     # lists above 256 records
    (2, 1400, 40, 24, 4, 400, 0.01),      # some tiles without a list, long bin lists
    (1, 400, 47, 20, 2, 200, 1.0),        # opacities at and above the cap
])
def test_reverse_against_oracle_and_without_lists(V, N, W, H, bin, cap, opacity):
    rec = scenes.random_projected(V, N, W, H, np.random.default_rng(N + W), radius_range=(4, 30), margin=8)
    if opacity is not None:
        rec["opacity"][:] = np.float32(opacity)
        rec["opacity"][:, ::3] *= np.float32(0.9)
    r = _setup(rec, W, H, bin, cap)
    cnt = r.lists.count.cpu().numpy()
    if opacity == 0.01:
        assert cnt.max() >= 256 or cap < 1024
        assert (cnt == -1).any() == (cap < 1024)
    _, Tf, last, amb = oracle.raster_fwd(rec, W, H, BG)
    d_img = np.random.default_rng(N).normal(size=(V, 3, H, W)) * (amb == 0)[:, None]
    want, want_o = oracle.raster_bwd(rec, W, H, Tf, last, d_img, BG, want_opacity=True)
    g1, o1 = _reverse(r, _t(d_img), True)
    g2, o2 = _reverse(r, _t(d_img), False)
    g3, _ = _reverse(r, _t(d_img), True, opacity=False)
    for sl in (slice(0, 2), slice(2, 5), slice(5, 8)):
        assert _rel(g1[..., sl], want[..., sl]) <= 1e-3
        assert _rel(g2[..., sl], g1[..., sl]) <= 1e-5
        assert _rel(g3[..., sl], g1[..., sl]) <= 1e-5
    assert _rel(o1, want_o) <= 1e-3
    assert _rel(o2, o1) <= 1e-5


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_pixel_gradient_stays_with_the_records_at_the_pixel(value):
    """Records that no pixel with a non-finite gradient takes part in keep
    the gradients they have when that pixel's gradient is zero."""
    N, W, H = 60, 32, 32
    rec = scenes.random_projected(1, N, W, H, np.random.default_rng(5), cull_frac=0.0, radius_range=(2, 4), margin=0)
    rec["opacity"][:] = np.float32(0.3)
    r = _setup(rec, W, H, 1, 256)
    d_img = _t(np.random.default_rng(6).normal(size=(1, 3, H, W)))
    d_img[0, :, 9, 21] = 0.0
    want, want_o = _reverse(r, d_img, True)
    d_img[0, 1, 9, 21] = value
    got, got_o = _reverse(r, d_img, True)
    m = rec["mean2d"][0].astype(np.float64)
    dx, dy = 21.5 - m[:, 0], 9.5 - m[:, 1]
    A, B, C = rec["conic"][0].astype(np.float64).T
    alpha = 0.3 * np.exp(-0.5 * (A * dx * dx + C * dy * dy) - B * dx * dy)
    at, away = alpha > 1.01 / 255, alpha < 0.99 / 255
    assert at.any() and away.sum() > N // 2
    assert not np.isfinite(got[0, at]).all(axis=1).any()
    np.testing.assert_allclose(got[0, away], want[0, away], rtol=1e-4, atol=1e-5 * np.abs(want).max())
    np.testing.assert_allclose(got_o[0, away], want_o[0, away], rtol=1e-4, atol=1e-5 * np.abs(want_o).max())
