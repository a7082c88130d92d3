"""Spawn, Adam and render of the added rows at every SH degree, whose rows take 16,
32 or 64 threads, or one where 65 536 of degree 0 or 1 are rendered: a call on
the first rows equals the first rows of a longer call bit for bit, spawned and
rendered columns that are copies are their sources', and nothing is written
outside the rows."""
import pytest
import torch

from paper_2403_01444_gb300 import gs3

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _added(rows, m, v, deg):
    a = gs3.GsAdded(gs3._ptr(rows), gs3._ptr(m), gs3._ptr(v), rows.shape[0], deg)
    a._keep = (rows, m, v)
    return a


def _set(n, deg, fill=7.0):
    K = (deg + 1) ** 2
    return gs3.Gaussians(*(torch.full(s, fill, device=DEV) for s in ((n, 3), (n, 4), (n, 3), (n,), (n, K, 3))), deg)


def _fields(g):
    return [getattr(g, f) for f in ("mean", "quat", "scale", "opacity_logit", "sh")]


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 15, 16, 17, 33, 65_499, 65_536])
def test_first_rows_of_a_longer_call(deg, n):
    N, K, P = n + 37, (deg + 1) ** 2, gs3.added_cols(deg)
    gen = torch.Generator(device=DEV).manual_seed(97 * deg + n)
    r = lambda *s: torch.randn(*s, device=DEV, generator=gen)
    # spawn: n of N selected rows, in an order of their own
    src = gs3.Gaussians(r(N, 3), r(N, 4), r(N, 3).exp(), r(N), r(N, K, 3), deg)
    order, z = torch.randperm(N, device=DEV, generator=gen).to(torch.int32), r(N, 3)
    got = []
    for count in (N, n):
        rows, m, v = (torch.full((N + 3, P), 7.0, device=DEV) for _ in range(3))
        nsel = torch.tensor([count], dtype=torch.int64, device=DEV)
        nadd, err = torch.tensor([2], dtype=torch.int64, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
        gs3.gs_added_spawn(src, order, nsel, z, 0.1, _added(rows, m, v, deg), nadd, err)
        assert int(nadd) == 2 + count and int(err) == 0
        for t in (rows, m, v):
            assert bool((t[:2] == 7.0).all()) and bool((t[2 + count:] == 7.0).all())
        assert not m[2:2 + count].any() and not v[2:2 + count].any()
        got.append(rows[2:2 + count])
    assert torch.equal(got[0][:n], got[1])
    at = order[:n].long()
    assert torch.equal(got[1][:, P - 3 * K:], src.sh[at].reshape(n, 3 * K))
    assert torch.equal(got[1][:, 3:7], torch.tensor([1.0, 0, 0, 0], device=DEV).expand(n, 4))
    # Adam (with the render) and render
    start = [r(N, P) * 0.1, r(N, P) * 1e-3, r(N, P).abs() * 1e-5]
    grads = [r(N, 3), r(N, 4), r(N, 3), r(N), r(N, K, 3)]
    state = torch.tensor([1065353216, 0, 3, 0], dtype=torch.int32, device=DEV)
    res = []
    for count in (N, n):
        t, out, again = [x.clone() for x in start], _set(N + 2, deg), _set(N + 2, deg)
        a = _added(*t, deg)
        gs3.gs_added_adam(a, count, *grads, [1e-3] * 6, 0.9, 0.999, 1e-15, state, out, 1)
        gs3.gs_added_to_render(a, count, again, 1)
        for x, y in zip(_fields(out), _fields(again)):
            assert torch.equal(x, y) and bool((x[0] == 7.0).all()) and bool((x[1 + count:] == 7.0).all())
        for x, y in zip(t, start):
            assert torch.equal(x[count:], y[count:]) and not torch.equal(x[:count], y[:count])
        assert torch.equal(out.sh[1:1 + count].reshape(count, 3 * K), t[0][:count, P - 3 * K:])
        res.append((t, out))
    for x, y in zip(res[0][0], res[1][0]):
        assert torch.equal(x[:n], y[:n])
    for x, y in zip(_fields(res[0][1]), _fields(res[1][1])):
        assert torch.equal(x[:1 + n], y[:1 + n])
