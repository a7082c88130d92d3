"""The loss at the edges of its 54 x 32 output tiles and of the tests-free path
of windows that lie inside the image, against the FP64 oracle.

Tolerances: those of test_gpu_kernels.py's loss parity (1e-5 on the loss and
the SSIM, 1e-3 relative on the gradient); a gradient of images that are equal
everywhere is zero to the rounding of its coefficients: they cancel terms of up
to 2 / C2 with 2^-24 each, times a dozen roundings, 1e-3 of lambda / (3 V H W)
at most 1e-2 with the window's sum."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_01444_gb300 import gs3

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2403_01444_gb300 import build
    build.build()
    gs3.lib()
    oracle.build()


def _loss(x, y, lam=0.2):
    V, _, H, W = x.shape
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(DEV)
    ws = torch.empty(gs3.gs_loss_workspace_size(3 * V, H, W), dtype=torch.uint8, device=DEV)
    gd, gl, gs = torch.full(x.shape, 7.0, device=DEV), torch.zeros(1, device=DEV), torch.zeros(1, device=DEV)
    gs3.gs_loss_l1_dssim(t(x), t(y), 3 * V, H, W, lam, gd, gl, gs, ws)
    torch.cuda.synchronize()
    return gl.item(), gs.item(), gd.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("V,H,W", [(1, 1, 1), (1, 31, 53), (1, 32, 54), (2, 33, 55), (1, 43, 65), (1, 74, 118),
                                   (1, 75, 119), (1, 106, 172)])
def test_loss_at_tile_edges(V, H, W):
    rng = np.random.default_rng(H * 1000 + W)
    x = rng.uniform(size=(V, 3, H, W)).astype(np.float32)
    y = np.clip(x + rng.normal(0, 0.15, size=x.shape), 0, 1).astype(np.float32)
    L, d, ss = oracle.loss_l1_dssim(x, y, 0.2)
    gl, gs, gd = _loss(x, y)
    assert abs(gl - L) <= 1e-5 * abs(L)
    assert abs(gs - ss) <= 1e-5
    assert np.linalg.norm(gd - d) <= 1e-3 * np.linalg.norm(d)
    assert np.abs(gd - d).max() <= 1e-2 * np.abs(d).max()


def test_equal_images_and_a_non_finite_pixel():
    rng = np.random.default_rng(1)
    x = rng.uniform(size=(1, 3, 80, 130)).astype(np.float32)
    x[0, 1] = 0.0                      # a black channel: an exact zero gradient
    gl, gs, gd = _loss(x, x)
    assert abs(gl) <= 1e-6 and abs(gs - 1) <= 1e-6
    assert np.abs(gd).max() <= 1e-2 * 0.2 / x.size
    assert not gd[0, 1].any()
    # a NaN spoils the gradient where a window of a window reaches it, no further
    y = x.copy()
    y[0, 0, 40, 60] = np.nan
    gl, gs, gd = _loss(x, y)
    assert np.isnan(gl) and np.isnan(gs)
    bad = ~np.isfinite(gd[0, 0])
    r, c = np.nonzero(bad)
    assert bad[40, 60] and r.min() >= 30 and r.max() <= 50 and c.min() >= 50 and c.max() <= 70
    assert np.isfinite(gd[0, 1:]).all()
