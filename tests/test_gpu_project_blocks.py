"""The projection reverses on both sides of the lines at which a block takes more
Gaussians and at which a thread walks a Gaussian's views by itself.

The reverse for mean and rotation does a Gaussian's arithmetic the same way in
every block size, so a call over all rows equals calls over a few of them bit
for bit.  The reverse of every parameter sums at most 32 views in another
order: 1e-5 of a tensor's norm (33 roundings of 2^-24 of terms of either
sign)."""
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


@pytest.mark.parametrize("deg,V,N", [(0, 2, 210_000), (0, 4, 101_000), (0, 16, 32_768), (0, 16, 32_767), (1, 4, 200_001),
                                     (1, 32, 33_000), (2, 16, 60_000)])
def test_every_parameter_whichever_kernel(deg, V, N):
    g, cams, grads = _inputs(V, N, deg, 0.7)
    op = torch.randn(V, N, device=DEV, generator=torch.Generator(device=DEV).manual_seed(1))
    K = (deg + 1) ** 2

    def run(first, count):
        o = [torch.full(s, 7.0, device=DEV) for s in ((count, 3), (count, 4), (count, 3), (count,), (count, K, 3))]
        gs3.gs_project_bwd_full(g, cams, V, W, H, grads, op, first, count, *o)
        return o

    whole = run(0, N)
    for a, b in ((0, 1000), (N - 3001, N)):
        for x, y in zip(whole, run(a, b - a)):
            x, y = x[a:b].double(), y.double()
            assert bool(torch.isfinite(x).all()) and float((x - y).norm()) <= 1e-5 * float(y.norm())
