"""The FP32 MLP's reverse over a list of rows and a count on the device: counts
of none, one, the edges of a chunk of 64 rows and more chunks than resident
blocks, below the list's length, in no order.

Bounds are accumulated roundings as in test_gpu_mlp_f32.py.  Rows that are not
listed, or are past the count, take no part and keep their d_enc."""
import pytest
import torch

from paper_2403_01444_gb300 import gs3
from test_gpu_mlp_f32 import DEV, U, _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("n,count", [(300, 0), (300, 1), (300, 63), (300, 65), (39000, 20011)])
def test_fp32_mlp_reverse_over_listed_rows(n, count, bf16):
    W, x, go = _inputs(n, bf16)
    gen = torch.Generator(device=DEV).manual_seed(n + count)
    order = torch.randperm(n, device=DEV, generator=gen)
    rows = order.to(torch.int32)   # the count is below the list's length
    mlp = gs3.mlp_struct(gs3.GS_MLP_FP32, torch.cat([w.reshape(-1) for w in W]))
    enc = x.bfloat16() if bf16 else x
    dW = torch.zeros(gs3.MLP_PARAMS, device=DEV)
    d_enc = torch.full((n, 32), 7.0, device=DEV)
    d_rows = torch.tensor([count], dtype=torch.int64, device=DEV)
    gs3.ntc_mlp_bwd(enc, n, mlp, go, None, dW, d_enc, rows=rows, d_rows=d_rows)
    torch.cuda.synchronize()
    at = order[:count]
    rest = torch.ones(n, dtype=torch.bool, device=DEV)
    rest[at] = False
    assert bool((d_enc[rest] == 7.0).all())

    W1, W2, W3 = (w.double() for w in W)
    xd, g = x[at].double(), go[at].double()
    h1 = (xd @ W1.T).relu()
    E1 = 32 * U * xd.abs() @ W1.abs().T
    h2 = (h1 @ W2.T).relu()
    E2 = E1 @ W2.abs().T + 64 * U * h1 @ W2.abs().T
    m1, m2 = (h1 > 0).double(), (h2 > 0).double()
    g2 = (g @ W3) * m2
    F2 = 7 * U * (g.abs() @ W3.abs()) * m2
    g1 = (g2 @ W2) * m1
    F1 = (F2 @ W2.abs() + 64 * U * g2.abs() @ W2.abs()) * m1
    Ee = F1 @ W1.abs() + 64 * U * g1.abs() @ W1.abs()
    assert bool(((d_enc[at].double() - g1 @ W1).abs() <= Ee).all())
    want = [g1.T @ xd, g2.T @ h1, g.T @ h2]
    err = [F1.T @ xd.abs() + count * U * g1.abs().T @ xd.abs(),
           F2.T @ h1 + g2.abs().T @ E1 + count * U * g2.abs().T @ h1,
           g.abs().T @ E2 + count * U * g.abs().T @ h2]
    want, err = (torch.cat([a.reshape(-1) for a in v]) for v in (want, err))
    assert bool(((dW.double() - want).abs() <= err).all())
