"""The FP32 MLP where its tiling can go wrong: the edges of a chunk of 64 rows,
more chunks than resident blocks, encodings that do not start on a 16-byte
boundary, BF16 encodings, and no gradient of the encoding asked for.

The bound of every value is its accumulated rounding: a chain of k FP32
multiply-adds is off by at most k u sum |a b| with u = 2^-24 (any order), on
top of its inputs' own errors, carried through the layers below; the factor
1.01 covers the products of errors.  Rows with an activation whose sign is
within its bound are left out, so both sides see the same gates."""
import pytest
import torch

from paper_2403_01444_gb300 import gs3

pytestmark = pytest.mark.gpu
DEV = "cuda"
U = 1.01 * 2.0 ** -24


def _inputs(n, bf16):
    gen = torch.Generator(device=DEV).manual_seed(n + 7 * bf16)
    W = [torch.randn(o, i, device=DEV, generator=gen) * (2.0 / i) ** 0.5 for o, i in ((64, 32), (64, 64), (7, 64))]
    x = torch.randn(2 * n + 64, 32, device=DEV, generator=gen)
    if bf16:
        x = x.bfloat16().float()
    W1, W2, W3 = (w.double() for w in W)
    xd = x.double()
    z1 = xd @ W1.T
    E1 = 32 * U * xd.abs() @ W1.abs().T
    z2 = z1.relu() @ W2.T
    E2 = E1 @ W2.abs().T + 64 * U * z1.relu() @ W2.abs().T
    sure = ((z1.abs() > E1).all(1) & (z2.abs() > E2).all(1)).nonzero()[:n, 0]
    assert len(sure) == n
    go = torch.randn(n, 7, device=DEV, generator=gen)
    return W, x[sure].contiguous(), go


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("n,offset,want_enc", [(1, 0, True), (63, 0, True), (64, 1, True), (65, 2, False),
                                               (20011, 0, True), (39000, 3, True)])
def test_fp32_mlp_within_its_rounding(n, offset, want_enc, bf16):
    W, x, go = _inputs(n, bf16)
    wflat = torch.cat([w.reshape(-1) for w in W])
    mlp = gs3.mlp_struct(gs3.GS_MLP_FP32, wflat)
    enc = torch.empty(32 * n + offset, device=DEV, dtype=torch.bfloat16 if bf16 else torch.float32)[offset:]
    enc = enc.view(n, 32).copy_(x)
    raw = torch.full((n, 7), float("nan"), device=DEV)
    gs3.ntc_mlp_fwd(enc, n, mlp, raw)
    dW = torch.zeros(gs3.MLP_PARAMS, device=DEV)
    d_enc = torch.full((32 * n + offset,), float("nan"), device=DEV)[offset:].view(n, 32) if want_enc else None
    scale = torch.tensor([4.0], device=DEV)
    gs3.ntc_mlp_bwd(enc, n, mlp, go, scale, dW, d_enc)
    torch.cuda.synchronize()

    W1, W2, W3 = (w.double() for w in W)
    xd, g = x.double(), 4.0 * go.double()
    h1 = (xd @ W1.T).relu()
    E1 = 32 * U * xd.abs() @ W1.abs().T
    h2 = (h1 @ W2.T).relu()
    E2 = E1 @ W2.abs().T + 64 * U * h1 @ W2.abs().T
    Eo = E2 @ W3.abs().T + 64 * U * h2 @ W3.abs().T
    assert ((raw.double() - h2 @ W3.T).abs() <= Eo).all()
    m1, m2 = (h1 > 0).double(), (h2 > 0).double()
    g2 = (g @ W3) * m2
    F2 = 7 * U * (g.abs() @ W3.abs()) * m2
    g1 = (g2 @ W2) * m1
    F1 = (F2 @ W2.abs() + 64 * U * g2.abs() @ W2.abs()) * m1
    if want_enc:
        Ee = F1 @ W1.abs() + 64 * U * g1.abs() @ W1.abs()
        assert ((d_enc.double() - g1 @ W1).abs() <= Ee).all()
    want = [g1.T @ xd, g2.T @ h1, g.T @ h2]
    err = [F1.T @ xd.abs() + n * U * g1.abs().T @ xd.abs(),
           F2.T @ h1 + g2.abs().T @ E1 + n * U * g2.abs().T @ h1,
           g.abs().T @ E2 + n * U * g.abs().T @ h2]
    want, err = (torch.cat([a.reshape(-1) for a in v]) for v in (want, err))
    assert ((dW.double() - want).abs() <= err).all()
