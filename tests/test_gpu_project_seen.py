"""The projection reverse over the Gaussians that have a gradient: every number
of views on its lanes (and one more than there are lanes), blocks that are
empty, full and ragged, a rotation or scale that has no finite gradient.

A Gaussian none of whose records has a gradient gets zeros; the others get what
the reverse of every parameter gives them from the same records, by the same
arithmetic up to the compiler's contractions: 1e-5 of the tensor (some hundred
roundings of 2^-24 a term)."""
import numpy as np
import pytest
import torch

from paper_2403_01444_gb300 import gs3, scenes

pytestmark = pytest.mark.gpu
DEV = "cuda"
W, H = 200, 150


@pytest.mark.parametrize("V,N,frac,deg", [(1, 1, 1.0, 0), (1, 129, 0.1, 3), (2, 128, 0.0, 1), (3, 1000, 0.1, 3),
                                          (5, 700, 1.0, 2), (16, 300, 0.05, 3), (32, 127, 0.3, 1), (33, 200, 0.3, 3)])
def test_seen_gaussians_get_the_full_reverse_and_the_others_zero(V, N, frac, deg):
    rng = np.random.default_rng(V + N)
    g = gs3.Gaussians.from_numpy(scenes.make_gaussians(N, deg, rng))
    cams = gs3.cameras_to_device(scenes.ring_cameras(np.linspace(0, 300, V), [5.0] * V, W, H))
    seen = rng.uniform(size=N) < frac
    grads = rng.normal(size=(V, N, 8)).astype(np.float32)
    grads[..., 2:5] *= 0.1
    grads *= (rng.uniform(size=(V, N, 1)) < 0.5) & seen[None, :, None]
    grads = torch.from_numpy(grads).to(DEV)
    seen = (grads != 0).any(-1).any(0)
    odd = [] if N < 100 else [3, N - 1]
    if odd:   # no finite gradient, seen or not
        g.quat[odd[0]] = 0.0
        g.scale[odd[1], 1] = float("inf")
    f = lambda *s: torch.full(s, 7.0, device=DEV)
    dm, dq, fm, fq = f(N, 3), f(N, 4), f(N, 3), f(N, 4)
    gs3.gs_project_bwd(g, cams, V, W, H, grads, dm, dq)
    gs3.gs_project_bwd_full(g, cams, V, W, H, grads, None, 0, N, fm, fq, f(N, 3), f(N), f(N, 3 * (deg + 1) ** 2))
    torch.cuda.synchronize()
    for i in odd:
        assert not bool(torch.isfinite(fq[i]).all())
        assert bool((torch.isfinite(dq[i]) == torch.isfinite(fq[i])).all())
    keep = torch.ones(N, dtype=torch.bool, device=DEV)
    keep[odd] = False
    for a, b in ((dm, fm), (dq, fq)):
        assert not bool(a[keep & ~seen].any())
        a, b = a[keep].double(), b[keep].double()
        assert float((a - b).norm()) <= 1e-5 * float(b.norm())
