"""The weight gradient of few output tiles: one token slice whose fp32 gradient
goes to the workspace and a streaming update after it (at most 3/4 as many
256 x 256 tiles as SM pairs, reductions too short to cut further).

The gradient is the one the fused kernel forms, so codes, moments, images,
counts and dW_out equal the fused call's (ws=False) bit for bit.  Sizes: one
ragged tile and the smallest reduction, ragged rows and columns, a whole tile,
and either side of the line (57 tiles of 76 pairs: slab; 58: fused both ways).
"""
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


@pytest.mark.parametrize("T,K,N", [(8, 16, 8), (129, 264, 520), (256, 512, 512), (200, 776, 4856),
                                   (200, 256, 14848)])
@pytest.mark.parametrize("form", ["int8", "8bit", "dev", "packed"])
def test_one_slab_equals_fused(T, K, N, form):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-N // 256) * -(-K // 256)
    assert (dqt.dqt_bwd_dw_img_workspace_size(T, N, K) == 4 * N * K) == (4 * tiles <= 3 * (sms // 2))
    g = dqt.grid(8 if form == "8bit" else 1.58)
    W0, s_w = dqt.dqt_absmean_init(inputs.normal((N, K), 0.02, seed=N).cuda(), g)
    dY = inputs.normal((T, N), 1e-2, seed=T, dtype=torch.bfloat16).cuda()
    Xdq = inputs.normal((T, K), 1.0, seed=K, dtype=torch.bfloat16).cuda()
    m0 = inputs.normal((N, K), 1e-4, seed=5).cuda()
    v0 = inputs.normal((N, K), 1e-4, seed=6).square().cuda()
    hp, sr = dqt.adamw(lr=1e-2, step=7), dqt.sr_stream(seed=9, tensor_id=2)
    got = []
    for ws in (None, False):
        W = dqt.dqt_pack_ternary(W0) if form == "packed" else W0.clone()
        m, v = m0.clone(), v0.clone()
        dW = torch.full((N, K), float("nan"), device="cuda")
        ch = torch.zeros(1, dtype=torch.int64, device="cuda")
        out = [W, m, v, dW, ch]
        if form == "packed":
            dqt.dqt_bitlinear_bwd_dw_update_packed(dY, Xdq, W, s_w, m, v, hp, sr, dW_out=dW,
                                                   changed_out=ch, ws=ws)
        else:
            img = torch.zeros((N, K), dtype=torch.bfloat16, device="cuda")
            if form == "dev":
                consts = dqt.dqt_update_consts(hp, sr, g, s_w).cuda()
                dqt.dqt_bitlinear_bwd_dw_update_dev(dY, Xdq, W, m, v, consts, dW_out=dW,
                                                    changed_out=ch, ws=ws, W_img_next=img)
            else:
                dqt.dqt_bitlinear_bwd_dw_update_img(dY, Xdq, W, s_w, m, v, hp, sr, g, dW_out=dW,
                                                    changed_out=ch, ws=ws, W_img_next=img)
            out.append(img)
        got.append(out)
    only = torch.full((N, K), float("nan"), device="cuda")  # gradient only, no update
    dqt.dqt_bitlinear_bwd_dw_update_img(dY, Xdq, None, s_w, None, None, None, None, g, dW_out=only)
    dqt.dqt_check_device_status()
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert torch.equal(only, got[0][3])
    assert int(got[0][4]) > 0


@pytest.mark.parametrize("T,K,N", [(2048, 2048, 2816), (4104, 5632, 1800)])
def test_whole_tiles_beside_token_slices(T, K, N):
    """One wave or more of whole tiles (updated in the GEMM's epilogue) and a
    last wave of token slices (stored and updated after it) in one launch: the
    two kinds of epilogue run side by side in a CTA's warps.  Every element's
    gradient against 64 bits (fp32 sums of T products: T 2^-24 of the sum of
    magnitudes, an O(1) error where blocks were mixed up), and the update is
    the standalone one on that gradient, bit for bit."""
    g = dqt.grid(1.58)
    W0, s_w = dqt.dqt_absmean_init(inputs.normal((N, K), 0.02, seed=N).cuda(), g)
    dY = inputs.normal((T, N), 1e-2, seed=T, dtype=torch.bfloat16).cuda()
    Xdq = inputs.normal((T, K), 1.0, seed=K, dtype=torch.bfloat16).cuda()
    need = dqt.dqt_bwd_dw_img_workspace_size(T, N, K)
    assert 0 < need < 4 * N * K  # last-wave slices
    hp, sr = dqt.adamw(lr=1e-2, step=7), dqt.sr_stream(seed=9, tensor_id=2)
    ref = dY.double().t() @ Xdq.double()
    bound = T * 2.0 ** -24 * (dY.double().abs().t() @ Xdq.double().abs())
    for _ in range(3):
        W, m, v = W0.clone(), torch.zeros((N, K), device="cuda"), torch.zeros((N, K), device="cuda")
        dW = torch.empty((N, K), device="cuda")
        dqt.dqt_bitlinear_bwd_dw_update_img(dY, Xdq, W, s_w, m, v, hp, sr, g, dW_out=dW)
        only = torch.empty((N, K), device="cuda")
        dqt.dqt_bitlinear_bwd_dw_update_img(dY, Xdq, None, s_w, None, None, None, None, g, dW_out=only)
        W2, m2, v2 = W0.clone(), torch.zeros_like(m), torch.zeros_like(v)
        dqt.dqt_sr_update(dW, W2, s_w, m2, v2, hp, sr, g)
        dqt.dqt_check_device_status()
        assert bool(((dW.double() - ref).abs() <= bound).all())
        assert torch.equal(only, dW)
        assert torch.equal(W, W2) and torch.equal(m, m2) and torch.equal(v, v2)
