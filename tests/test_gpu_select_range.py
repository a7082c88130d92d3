"""gs_select_above at the ends of FP32's range, where the product of threshold and
count overflows, underflows or is not a number: the selection is that of the
quotient alone."""
import pytest
import torch

from paper_2403_01444_gb300 import gs3

pytestmark = pytest.mark.gpu
DEV = "cuda"
INF, NAN = float("inf"), float("nan")


@pytest.mark.parametrize("tau", [3.4e38, 1e38, 1e-38, 1e-45, 0.0, -0.0, -1e-45, -1e38, -3.4e38, INF, -INF, NAN])
def test_selection_is_the_quotient_s(tau):
    a = torch.tensor([INF, 3.4028235e38, 3e38, 1e38, 1.0, 1e-38, 7e-45, 4.2e-45, 1e-45, 0.0], device=DEV)
    a = torch.cat([a, -a, torch.tensor([NAN], device=DEV)])
    d = torch.tensor([-1, 0, 1, 2, 3, 5, 1000, 2 ** 31 - 1], dtype=torch.int32, device=DEV)
    accum, denom = a.repeat_interleave(len(d)), d.repeat(len(a))
    idx = torch.full((len(accum),), -1, dtype=torch.int32, device=DEV)
    nsel = torch.full((1,), -1, dtype=torch.int64, device=DEV)
    gs3.gs_select_above(accum, denom, len(accum), tau, idx, nsel)
    t = torch.tensor(tau, dtype=torch.float32, device=DEV)
    want = torch.nonzero((denom > 0) & (accum / denom.float() > t)).flatten().to(torch.int32)
    assert int(nsel) == want.numel() and torch.equal(idx[:want.numel()], want)
