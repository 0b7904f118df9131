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
                                 (457, 2048), (457, 2064), (700, 4096),
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


@pytest.mark.parametrize("T,K", [(8192, 5632), (16384, 768), (8192, 2048), (8192, 1040), (4096, 4112), (8192, 4096),
                                 (8192, 3584)])
def test_row_ring_many_rounds(T, K):
    """Several rounds of the shared-memory row ring (each place of it used up to
    five times), launched again and again: a warp that took a slot's old rows, or
    released a slot early, would change bytes or run into a wait's limit."""
    x = torch.randn(T, K, generator=torch.Generator().manual_seed(K)).to(torch.bfloat16).cuda()
    first = None
    for _ in range(60):
        out = list(dqt.dqt_act_quant_images(x)) + list(dqt.dqt_act_quant_fp8(x))
        out.append(dqt.dqt_codes_to_xdq(out[0], out[1]))
        if first is None:
            first = out
        else:
            for a, b in zip(out, first):
                assert torch.equal(a, b)
    dqt.dqt_check_device_status()
    s = 127.0 / x.float().abs().amax(1).double().clamp_min(1e-5)
    assert torch.equal(first[1], s.float())
    want = (x.float() * first[1][:, None]).round().clamp_(-128, 127)
    assert torch.equal(first[0].float(), want)


@pytest.mark.parametrize("T,K", [(8192, 2048), (8192, 4096), (16384, 768), (16384, 3584), (8192, 5632),
                                 (16384, 272), (4096, 8192), (3000, 1040)])
def test_each_output_alone(T, K):
    """Codes, code image and X_tilde written alone, and E4M3 codes alone: rings
    of other sizes than the call that writes all outputs has, the same bytes."""
    x = torch.randn(T, K, generator=torch.Generator().manual_seed(T + K)).to(torch.bfloat16).cuda()
    q, s, img, xdq = dqt.dqt_act_quant_images(x)
    q8, s8, _ = dqt.dqt_act_quant_fp8(x)
    for _ in range(20):
        a, sa = dqt.dqt_act_quant(x)
        assert torch.equal(a, q) and torch.equal(sa, s)
        assert torch.equal(dqt.dqt_act_quant_images(x, want=("Xq_img",))[2], img)
        assert torch.equal(dqt.dqt_act_quant_images(x, want=("Xdq",))[3], xdq)
        b, sb, none = dqt.dqt_act_quant_fp8(x, want_xdq=False)
        assert none is None and torch.equal(b, q8) and torch.equal(sb, s8)
    dqt.dqt_check_device_status()
