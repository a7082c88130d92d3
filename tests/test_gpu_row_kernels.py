"""Kernels whose work is divided over rows, segments or views, at the edges of
those divisions: the SH rotation, the selection above a threshold, the added
rows' Adam step and the reverse projection of every parameter.

Tolerances: the rotation, the selection and the Adam step compute each value
independently of its neighbours, so a call on the first rows equals the first
rows of a longer call bit for bit.  The reverse projection sums over the views
in another order than the sum of single-view calls: each of its sums has at
most 33 terms, so the two differ by less than 33 roundings of 2^-24 of the
terms' absolute sum; with the terms of either sign, 1e-5 of a tensor's norm."""
import numpy as np
import pytest
import torch

from paper_2403_01444_gb300 import gs3, scenes

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2403_01444_gb300 import build
    build.build()
    gs3.lib()


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 129])
def test_sh_rotate_rows_are_independent(deg, n):
    g, N = _gen(deg), 300
    sh = torch.randn(N, (deg + 1) ** 2, 3, generator=g, device=DEV)
    qa, qb = torch.randn(N, 4, generator=g, device=DEV), torch.randn(N, 4, generator=g, device=DEV)
    full, part = torch.empty_like(sh), torch.full_like(sh, 7.0)
    gs3.gs_sh_rotate(qa, qb, sh, N, deg, full)
    gs3.gs_sh_rotate(qa, qb, sh, n, deg, part)
    inplace = sh.clone()
    gs3.gs_sh_rotate(qa, qb, inplace, n, deg, inplace)
    assert torch.equal(part[:n], full[:n]) and bool((part[n:] == 7.0).all())
    assert torch.equal(inplace[:n], full[:n]) and torch.equal(inplace[n:], sh[n:])


@pytest.mark.parametrize("count", [0, 1, 31, 33, 255, 8191, 8193, 65536, 100003])
@pytest.mark.parametrize("tau", [0.25, 0.0, -0.5])
def test_select_above_in_index_order(count, tau):
    g = _gen(count)
    # quotients at, just above and far from the threshold; unseen ones (denom 0) never
    denom = torch.randint(0, 4, (max(count, 1),), generator=g, device=DEV, dtype=torch.int32)
    accum = torch.randn(max(count, 1), generator=g, device=DEV)
    accum[::3] = tau * denom[::3].float()
    accum[::7] = torch.nextafter(accum[::7], torch.full_like(accum[::7], 9.0))
    idx = torch.full((max(count, 1) + 1,), -1, dtype=torch.int32, device=DEV)
    nsel = torch.full((1,), -1, dtype=torch.int64, device=DEV)
    gs3.gs_select_above(accum, denom, count, tau, idx, nsel)
    want = torch.nonzero((denom > 0) & (accum / denom.float() > tau)).flatten().to(torch.int32)
    want = want[want < count]
    assert int(nsel) == want.numel()
    assert torch.equal(idx[:want.numel()], want) and bool((idx[want.numel():] == -1).all())


@pytest.mark.parametrize("deg", [0, 3])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 17])
def test_added_adam_rows_are_independent(deg, n):
    g, N, K = _gen(n), 40, (deg + 1) ** 2
    P = gs3.added_cols(deg)
    rows = torch.randn(N, P, generator=g, device=DEV) * 0.1
    m, v = torch.randn(N, P, generator=g, device=DEV) * 1e-3, torch.rand(N, P, generator=g, device=DEV) * 1e-5
    grads = [torch.randn(N, c, generator=g, device=DEV).reshape(s) for c, s in
             ((3, (N, 3)), (4, (N, 4)), (3, (N, 3)), (1, (N,)), (3 * K, (N, K, 3)))]
    res = []
    for k in (N, n):
        r = [rows.clone(), m.clone(), v.clone()]
        out = gs3.Gaussians(*(torch.full(s, 7.0, device=DEV) for s in ((N + 2, 3), (N + 2, 4), (N + 2, 3), (N + 2,),
                                                                       (N + 2, K, 3))), deg)
        gs3.gs_added_adam(gs3.added_struct(*r, deg), k, *grads, (1e-3, 2e-3, 3e-3, 4e-3, 5e-3, 6e-3), 0.9, 0.999,
                          1e-15, gs3.new_train_state(1.0), out, 2)
        res.append((r, out))
    for a, b, start in zip(res[0][0], res[1][0], (rows, m, v)):
        assert torch.equal(a[:n], b[:n]) and torch.equal(b[n:], start[n:])
    for f in ("mean", "quat", "scale", "opacity_logit", "sh"):
        a, b = getattr(res[0][1], f), getattr(res[1][1], f)
        assert torch.equal(a[:2 + n], b[:2 + n]) and bool((b[2 + n:] == 7.0).all()) and bool((b[:2] == 7.0).all())


@pytest.mark.parametrize("V,deg", [(1, 0), (3, 1), (5, 2), (4, 3), (17, 3), (33, 1)])
def test_project_bwd_full_sums_its_views(V, deg):
    W, H, N, first, count = 96, 80, 150, 20, 101
    g = gs3.Gaussians.from_numpy(scenes.make_gaussians(N, deg, np.random.default_rng(V)))
    cams = gs3.cameras_to_device(scenes.ring_cameras(np.linspace(0, 300, V), [5] * V, W, H))
    gen, K = _gen(V), (deg + 1) ** 2
    grads = torch.randn(V, N, 8, generator=gen, device=DEV)
    d_op = torch.randn(V, N, generator=gen, device=DEV)

    def call(vs, cd, gr, op):
        o = [torch.full((count,) + s, 7.0, device=DEV) for s in ((3,), (4,), (3,), (), (K, 3))]
        gs3.gs_project_bwd_full(g, cd, vs, W, H, gr, op, first, count, *o)
        return o

    got = call(V, cams, grads, d_op)
    want = [0.0] * 5
    for v in range(V):
        one = call(1, gs3.camera_slice(cams, v, 1).clone(), grads[v:v + 1].contiguous(), d_op[v:v + 1].contiguous())
        want = [w + o.double() for w, o in zip(want, one)]
    for a, b in zip(got, want):
        assert float((a.double() - b).norm()) <= 1e-5 * float(b.norm())
