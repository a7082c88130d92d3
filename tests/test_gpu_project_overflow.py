"""The projection reverse of Gaussians that no record gradient reaches and whose
covariance is not finite although their scales and records are: an axis seen end
on, whose square overflows.  The reverse for mean and rotation says so in the
gradient exactly where the reverse of every parameter, which leaves no Gaussian
out, does, and gives zeros elsewhere."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2403_01444_gb300 import gs3

pytestmark = pytest.mark.gpu
DEV = "cuda"
W, H = 64, 48
AXIS = [1.0, 1e4, 1e18, 2e19, 1e25, 3e38]


@pytest.mark.parametrize("deg", [0, 3])
@pytest.mark.parametrize("V", [1, 3, 32, 33])
def test_unseen_gaussians_of_an_overflowing_covariance(V, deg):
    N = 40 * len(AXIS)
    cam = SimpleNamespace(viewmat=np.eye(3, 4) + np.array([0, 0, 0, 4.0]) * np.array([[0], [0], [1]]), fx=50.0, fy=50.0,
                          cx=W / 2, cy=H / 2, W=W, H=H, campos=np.array([0, 0, -4.0]))
    z = lambda *s: torch.zeros(*s, device=DEV)
    g = gs3.Gaussians(z(N, 3), z(N, 4), torch.full((N, 3), 0.1, device=DEV), z(N), z(N, (deg + 1) ** 2, 3), deg)
    g.quat[:, 0] = 1.0
    g.scale[:, 2] = torch.tensor(AXIS, device=DEV).repeat(40)
    cams = gs3.cameras_to_device([cam] * V)
    p = gs3.Projected.empty(V, N)
    err = torch.zeros(1, dtype=torch.int32, device=DEV)
    gs3.gs_project(g, cams, V, W, H, p, d_err=err)
    f = lambda *s: torch.full(s, 7.0, device=DEV)
    dm, dq, fm, fq = f(N, 3), f(N, 4), f(N, 3), f(N, 4)
    grads = z(V, N, 8)
    gs3.gs_project_bwd(g, cams, V, W, H, grads, dm, dq)
    gs3.gs_project_bwd_full(g, cams, V, W, H, grads, None, 0, N, fm, fq, f(N, 3), f(N), f(N, (deg + 1) ** 2, 3))
    torch.cuda.synchronize()
    assert int(err) == 0 and bool((p.radius > 0).all())   # every record is there
    assert bool(torch.isfinite(fm).any()) and not bool(torch.isfinite(fm).all())
    for a, b in ((dm, fm), (dq, fq)):
        assert torch.equal(torch.isfinite(a), torch.isfinite(b))
        assert not bool(a[torch.isfinite(a)].any())
