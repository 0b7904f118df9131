"""The dequantised activation image X_tilde = bf16(RN(q / s_x)), written by a
multiplication with 1 / s_x where that provably rounds alike and by a division
otherwise, against the division on the CPU, bit for bit: rows of scales over
twelve decades (about 1.8 % of them divide), zero rows, infinite and NaN
inputs, on both activation types and from stored int8 codes.  Row counts about
one CTA per row (152), row lengths of one vector, ragged and long ones (the
ring's chunks hold several rows, one row, and at most a few)."""
import pytest
import torch

from paper_2412_04787_gb300 import dqt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_04787_gb300 import build
    build.build()
    dqt.lib()
    yield
    torch.cuda.synchronize()


def _same(a, b):
    # bf16 results bit for bit; a NaN is a NaN
    an, bn = torch.isnan(a), torch.isnan(b)
    return torch.equal(an, bn) and torch.equal(a.view(torch.int16)[~an], b.view(torch.int16)[~bn])


@pytest.mark.parametrize("T,K", [(1, 16), (151, 768), (153, 16), (3001, 1040), (20000, 48), (307, 5632),
                                 (160, 24576), (5, 49152)])
def test_xdq_is_the_correctly_rounded_quotient(T, K):
    g = torch.Generator().manual_seed(T + K)
    X = torch.randn(T, K, generator=g)
    X *= torch.exp(torch.empty(T, 1).uniform_(-14.0, 14.0, generator=g))
    X[T // 2] = 0.0
    if T > 100:
        X[T // 3, 3] = float("inf")
        X[T // 4, 5] = float("nan")
    X = X.to(torch.bfloat16)
    q, s, img, xdq = (t.cpu() for t in dqt.dqt_act_quant_images(X.cuda()))
    q8, s8, xdq8 = (t.cpu() for t in dqt.dqt_act_quant_fp8(X.cuda()))
    again = dqt.dqt_codes_to_xdq(q.cuda(), s.cuda()).cpu()
    dqt.dqt_check_device_status()
    want = torch.div(q.float(), s[:, None]).to(torch.bfloat16)
    assert _same(xdq, want) and _same(again, want)
    assert torch.equal(img.float(), q.float())
    v8 = q8.view(torch.float8_e4m3fn).float()
    assert _same(xdq8, torch.div(v8, s8[:, None]).to(torch.bfloat16))


@pytest.mark.parametrize("s", [1e-39, 1e-31, 1e-29, 0.3, 1e29, 1e31, 2e38])
def test_codes_to_xdq_at_extreme_scales(s):
    """Scales a caller may pass: where 1 / s or a quotient leaves the normal
    range the rows divide."""
    q = torch.arange(-128, 128, dtype=torch.int8).repeat(7, 1).contiguous()
    sx = torch.full((7,), s)
    got = dqt.dqt_codes_to_xdq(q.cuda(), sx.cuda()).cpu()
    assert _same(got, torch.div(q.float(), sx[:, None]).to(torch.bfloat16))
