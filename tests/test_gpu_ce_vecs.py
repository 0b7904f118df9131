"""Cross-entropy forward at the row lengths where its vectors per thread and
step (1 to 6) and its number of steps change, with masked and invalid logits."""

import pytest
import torch

from paper_2412_04787_gb300 import dqt

pytestmark = pytest.mark.gpu

EDGES = [8] + [2048 * k + d for k in range(1, 10) for d in (0, 8)] + [24576, 24584, 32000, 50304]


@pytest.mark.parametrize("V", EDGES)
def test_cross_entropy_forward_row_lengths(V):
    g = torch.Generator(device="cuda").manual_seed(V)
    x = (torch.randn(6, V, generator=g, device="cuda") * 3).bfloat16()
    x[1, : V - 3] = float("-inf")  # masked but for the last three
    x[2] = torch.finfo(torch.bfloat16).min
    x[3] = float("-inf")
    x[4, V - 1] = float("nan")
    x[5, 0] = float("inf")
    t = torch.full((6,), V - 1, device="cuda", dtype=torch.int64)
    lse, loss = dqt.dqt_cross_entropy_fwd_bf16(x, t)
    ref = torch.logsumexp(x.double(), 1)
    # the terms' 2^-22 each, at most 64 roundings of 2^-24 on a term's way
    # through the sums (rows of a few thousand to 50000), then the logarithm and
    # the last addition
    tol = 68 * 2.0 ** -24 + 2.0 ** -22 * ref.abs()
    assert ((lse.double() - ref).abs() <= tol)[:3].all()
    assert lse[3] == float("-inf") and lse[4].isnan() and lse[5].isnan()
    assert ((loss.double() - (ref - x[:, V - 1].double())).abs() <= 2 * tol)[:2].all()
