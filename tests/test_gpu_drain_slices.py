"""The exact forward of codes wider than 4 bits (its fp32 accumulator drained
into int32 every 1024 elements) with its last wave cut into reduction slices:
int32 partials, so Y and the int32 accumulators equal the uncut kernel's bit
for bit.  Shapes: the 5632-long down projection (256 tiles), a ragged one
whose slices are no multiple of the drained chunk and whose tail holds the
partial last row and column tiles, two stacked weights, and all-equal codes of
the largest magnitude (a slice's sums pass 2^24)."""
import pytest
import torch

from paper_2412_04787_gb300 import dqt, inputs

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


@pytest.mark.parametrize("T,K,N,kind", [(8192, 5632, 2048, "random"), (4896, 4104, 1032, "random"),
                                        (4896, 4104, 1032, "largest"), (4096, 4160, 1536, "pair")])
def test_cut_drained_forward_equals_uncut(T, K, N, kind):
    assert dqt.dqt_fwd_img_workspace_size(T, K, N) > 0
    if kind == "largest":
        x, c = torch.full((T, K), -128, dtype=torch.int8), torch.full((N, K), -128, dtype=torch.int8)
    else:
        g = torch.Generator().manual_seed(K)
        x = torch.randint(-128, 128, (T, K), generator=g, dtype=torch.int8)
        c = torch.randint(-128, 128, (N, K), generator=g, dtype=torch.int8)
    xi, ci = dqt.dqt_codes_to_bf16(x.cuda()), dqt.dqt_codes_to_bf16(c.cuda())
    s_x = inputs.normal((T,), 1.0, seed=1).abs().add_(0.5).cuda()
    ws = torch.full((dqt.dqt_fwd_img_workspace_size(T, K, N),), 0x3F, dtype=torch.uint8, device="cuda")
    got = []
    for w in (False, ws, ws, None):  # (a workspace used again, and new ones)
        acc = torch.empty((T, N), dtype=torch.int32, device="cuda")
        if kind == "pair":
            Y = dqt.dqt_bitlinear_fwd_img_pair(xi, s_x, ci, 512, 31.0, 77.0, 8, acc_out=acc, ws=w)
        else:
            Y = dqt.dqt_bitlinear_fwd_img(xi, s_x, ci, 31.0, 8, acc_out=acc, ws=w)
        got.append((Y, acc))
    dqt.dqt_check_device_status()
    ref = x[::257].double() @ c.double().t()
    assert torch.equal(got[0][1][::257].cpu().double(), ref)
    for Y, acc in got[1:]:
        assert torch.equal(acc, got[0][1]) and torch.equal(Y.view(torch.int16), got[0][0].view(torch.int16))
