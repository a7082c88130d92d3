"""Weight gradients of the FP32 MLP over many rows.

Every row is the same and the weights are zeros and ones, so that activations
and row gradients are the inputs themselves and each weight's gradient is n
times one product: with equal terms the roundings of a running sum all have
one sign over most of it, and a chain of k additions is off by a good part of
its worst case, k u |sum| with u = 2^-24.  Allowed is what the three levels of
the sum add up to: 32 rows (and the even rows' sum to the odd ones', or eight
warps), the chunks of a block, the blocks."""
import pytest
import torch

from paper_2403_01444_gb300 import gs3

pytestmark = pytest.mark.gpu
DEV = "cuda"
ROWS = 64   # of a chunk


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("n", [19456, 4_000_000])
def test_no_chain_over_all_rows(n, bf16):
    gen = torch.Generator(device=DEV).manual_seed(n)
    i, j, q = torch.arange(32, device=DEV), torch.arange(64, device=DEV), torch.arange(7, device=DEV)
    W = [(j[:, None] % 32 == i).float(), (j[:, None] == j).float(), (j % 7 == q[:, None]).float()]
    x = torch.rand(32, device=DEV, generator=gen) + 0.5
    dtype = torch.bfloat16 if bf16 else torch.float32
    x = x.to(dtype)
    go = torch.randn(7, device=DEV, generator=gen)
    mlp = gs3.mlp_struct(gs3.GS_MLP_FP32, torch.cat([w.reshape(-1) for w in W]))
    enc = x.repeat(n, 1)
    d_raw = go.repeat(n, 1)
    dW = torch.zeros(gs3.MLP_PARAMS, device=DEV)
    gs3.ntc_mlp_bwd(enc, n, mlp, d_raw, None, dW, None)
    torch.cuda.synchronize()
    h = x.double()[j % 32]
    g2 = go.double()[j % 7]
    one = torch.cat([(g2[:, None] * x.double()).reshape(-1), (g2[:, None] * h).reshape(-1),
                     (go.double()[:, None] * h).reshape(-1)])
    chunks = -(-n // ROWS)
    blocks = min(chunks, 2 * torch.cuda.get_device_properties(0).multi_processor_count)
    k = 32 + 1 + -(-chunks // blocks) + 8 + blocks
    err = (dW.double() - n * one).abs()
    assert float((err / (n * one.abs())).max()) <= 1.01 * k * 2.0 ** -24
