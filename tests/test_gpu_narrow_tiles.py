"""The 2-SM kernels' 256 x 128 tiles, taken where they give each SM pair at most
one unit of work, against the 1-SM kernel (128 x 256 tiles): Y, the int32
accumulators and dX bit for bit; the E4M3 forward against the same rows run in
a launch of wide tiles.  Sizes: one vector, either side of a 128- and a
256-wide tile, ragged reductions, and either side of the rule's line (19 row
tiles x 4 = 76 units of 76 pairs; 20 x 4 = 80)."""
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


@pytest.mark.parametrize("T,K,N", [(1, 8, 8), (257, 64, 128), (255, 520, 136), (300, 136, 264),
                                   (256, 512, 512), (4864, 512, 512), (5120, 512, 512)])
def test_narrow_tiles_equal_one_sm_tiles(T, K, N):
    x = inputs.normal((T, K), 1.0, seed=T, dtype=torch.bfloat16).cuda()
    dy = inputs.normal((T, N), 1e-2, seed=N, dtype=torch.bfloat16).cuda()
    W, s_w = dqt.dqt_absmean_init(inputs.normal((N, K), 0.02, seed=K).cuda(), 1.58)
    _, s_x, xi, _ = dqt.dqt_act_quant_images(x)
    img = dqt.dqt_codes_to_bf16(W)
    got = []
    try:
        for mode in (0, 1):
            dqt.dqt_set_gemm_tiles(mode)
            acc = torch.empty((T, N), dtype=torch.int32, device="cuda")
            Y = dqt.dqt_bitlinear_fwd_img(xi, s_x, img, s_w, 1.58, acc_out=acc)
            got.append((Y, acc, dqt.dqt_bitlinear_bwd_dx_img(dy, img, s_w)))
    finally:
        dqt.dqt_set_gemm_tiles(0)
    dqt.dqt_check_device_status()
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("T,K,N", [(1, 16, 8), (257, 64, 128), (255, 528, 136), (300, 144, 264)])
def test_narrow_fp8_tiles_equal_wide_ones(T, K, N):
    """Rows repeated until the launch takes wide tiles: the same row, the same Y."""
    x = inputs.normal((T, K), 1.0, seed=T, dtype=torch.bfloat16).cuda()
    W, s_w = dqt.dqt_absmean_init(inputs.normal((N, K), 0.02, seed=K).cuda(), 4)
    w8 = dqt.dqt_codes_to_fp8(W, 4)
    q8, s8, _ = dqt.dqt_act_quant_fp8(x)
    acc = torch.empty((T, N), device="cuda")
    Y = dqt.dqt_bitlinear_fwd_fp8(q8, s8, w8, s_w, 4, acc_out=acc)
    reps = -(-256 * 80 // T)
    wide = dqt.dqt_bitlinear_fwd_fp8(q8.repeat(reps, 1), s8.repeat(reps), w8, s_w, 4)
    dqt.dqt_check_device_status()
    # E4M3 products summed in fp32 (the order is the instruction's): K 2^-24 of
    # the sum of magnitudes, and one bf16 rounding
    v = q8.view(torch.float8_e4m3fn).double()
    ref, mag = v @ W.double().t(), v.abs() @ W.double().abs().t()
    assert bool(((acc.double() - ref).abs() <= K * 2.0 ** -24 * mag + 1e-30).all())
    tol = 2.0 ** -8 * Y.double().abs() + 2 * K * 2.0 ** -24 * mag / (s8.double()[:, None] * s_w)
    assert bool(((wide[:T].double() - Y.double()).abs() <= tol).all())
