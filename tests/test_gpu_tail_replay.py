"""A forward or dX whose last wave is cut into reduction slices, captured alone
in a CUDA graph with a workspace of its own and replayed: every replay finds the
slice counters as the one before it left them, and has to write the whole
output.  Each replay gets new inputs and an output filled with NaN; the result
equals the eager call bit for bit (the forward: the uncut kernel; dX, whose
fp32 sums depend on the slices: the cut call on a workspace of its own).
Shapes: the 5632-long down projection and dX, and ragged ones whose tail holds
the partial last row and column tiles."""
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


def _capture(fn):
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        fn()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fn()
    return graph


# (rows, reduction, columns): tiles beyond the last full wave, reduction >= 4096
@pytest.mark.parametrize("M,R,C", [(8192, 5632, 2048), (4896, 4104, 1032)])
@pytest.mark.parametrize("kind", ["ternary", "8-bit", "pair", "8-bit pair", "int8 call", "dx"])
def test_replayed_cut_launch_writes_its_output(kind, M, R, C):
    g = torch.Generator().manual_seed(R)
    top = 128 if "8-bit" in kind else 2
    lo = -128 if "8-bit" in kind else -1
    bits = 8 if "8-bit" in kind else 1.58
    codes = torch.randint(lo, top, (R, C) if kind == "dx" else (C, R), generator=g,
                          dtype=torch.int8).cuda()
    img = dqt.dqt_codes_to_bf16(codes)
    out = torch.empty((M, C), dtype=torch.bfloat16, device="cuda")
    if kind == "dx":
        dy = torch.empty((M, R), dtype=torch.bfloat16, device="cuda")
        nws = dqt.dqt_bwd_dx_img_workspace_size(M, R, C)

        def load(seed):
            dy.copy_(inputs.normal((M, R), 1e-2, seed=seed, dtype=torch.bfloat16))

        def call(y, ws):
            return dqt.dqt_bitlinear_bwd_dx_img(dy, img, 31.0, dX=y, ws=ws)
    else:
        xq = torch.empty((M, R), dtype=torch.int8, device="cuda")
        xi = torch.empty((M, R), dtype=torch.bfloat16, device="cuda")
        s_x = inputs.normal((M,), 1.0, seed=1).abs().add_(0.5).cuda()
        nws = (dqt.dqt_fwd_workspace_size(M, R, C) if kind == "int8 call"
               else dqt.dqt_fwd_img_workspace_size(M, R, C))

        def load(seed):
            gs = torch.Generator().manual_seed(seed)
            xq.copy_(torch.randint(-128, 128, (M, R), generator=gs, dtype=torch.int8))
            dqt.dqt_codes_to_bf16(xq, xi)

        def call(y, ws):
            if kind == "int8 call" and ws is not False:
                return dqt.dqt_bitlinear_fwd(xq, s_x, codes, 31.0, bits, Y=y, ws=ws)
            if "pair" in kind:
                return dqt.dqt_bitlinear_fwd_img_pair(xi, s_x, img, 512, 31.0, 77.0, bits, Y=y, ws=ws)
            return dqt.dqt_bitlinear_fwd_img(xi, s_x, img, 31.0, bits, Y=y, ws=ws)
    assert nws > 0
    ws = torch.full((nws,), 0x3F, dtype=torch.uint8, device="cuda")
    load(1)
    graph = _capture(lambda: call(out, ws))
    for replay in range(4):
        load(10 + replay)
        out.fill_(float("nan"))
        graph.replay()
        if kind == "dx":
            ref = call(None, torch.zeros(nws, dtype=torch.uint8, device="cuda"))
        else:
            ref = call(None, False)
        dqt.dqt_check_device_status()
        assert torch.equal(out.view(torch.int16), ref.view(torch.int16)), replay
