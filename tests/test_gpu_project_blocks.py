"""The projection reverse on both sides of the lines at which a block takes more
Gaussians.  It does a Gaussian's arithmetic the same way in every block size, so
a call over all rows equals calls over a few of them bit for bit."""
import numpy as np
import pytest
import torch

from paper_2403_01444_gb300 import gs3, scenes

pytestmark = pytest.mark.gpu
DEV = "cuda"
W, H = 200, 150


def _inputs(V, N, deg, frac):
    rng = np.random.default_rng(V + N)
    g = gs3.Gaussians.from_numpy(scenes.make_gaussians(N, deg, rng))
    cams = gs3.cameras_to_device(scenes.ring_cameras(np.linspace(0, 300, V), [5.0] * V, W, H))
    gen = torch.Generator(device=DEV).manual_seed(N)
    grads = torch.randn(V, N, 8, device=DEV, generator=gen)
    grads[..., 2:5] *= 0.1
    grads *= torch.rand(1, N, 1, device=DEV, generator=gen) < frac
    return g, cams, grads


def _rows(g, a, b):
    return gs3.Gaussians(*(getattr(g, f)[a:b].clone() for f in ("mean", "quat", "scale", "opacity_logit", "sh")),
                         g.sh_deg)


# blocks of 128, 64, 32 and fewer Gaussians on a chip of 152 SMs
@pytest.mark.parametrize("V,N,frac", [(1, 80_001, 0.5), (2, 77_700, 0.1), (2, 90_001, 0.1), (4, 50_003, 1.0),
                                      (8, 20_001, 1.0), (8, 80_003, 0.1), (16, 50_001, 0.3), (16, 160_003, 0.1),
                                      (32, 2_001, 1.0), (32, 9_999, 0.3), (32, 50_001, 0.1), (32, 157_001, 0.05)])
def test_mean_and_rotation_do_not_depend_on_the_block(V, N, frac):
    g, cams, grads = _inputs(V, N, 1, frac)
    f = lambda *s: torch.full(s, 7.0, device=DEV)
    dm, dq = f(N, 3), f(N, 4)
    gs3.gs_project_bwd(g, cams, V, W, H, grads, dm, dq)
    assert bool(torch.isfinite(dm).all()) and bool(dm.any()) and bool(dq.any())
    assert not bool(dm[~(grads != 0).any(-1).any(0)].any())
    for a, b in ((0, 1), (0, 777), (N // 2, N // 2 + 130), (N - 513, N)):
        pm, pq = f(b - a, 3), f(b - a, 4)
        gs3.gs_project_bwd(_rows(g, a, b), cams, V, W, H, grads[:, a:b].contiguous(), pm, pq)
        assert torch.equal(pm, dm[a:b]) and torch.equal(pq, dq[a:b])

