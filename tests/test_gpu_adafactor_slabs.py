"""Adafactor statistics at the sizes where the rows per block change (32, 16,
8: the grid of 1024-column blocks against two blocks per SM), with ragged last
slabs and columns."""

import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2412_04787_gb300 import dqt, inputs

pytestmark = pytest.mark.gpu


# 8 rows: fewer than 304 blocks of 16; 16 rows: fewer than 304 of 32
@pytest.mark.parametrize("N,K", [(1, 8), (9, 4), (4848, 1024), (4841, 1000), (4849, 1024),
                                 (9696, 1024), (9697, 1020), (2431, 2056)])
def test_adafactor_stats_slabs(N, K):
    c, s_w, _ = oracle.absmean_init(inputs.normal((N, K), 0.02, seed=N).numpy(), -1, 1)
    hp = dict(lr=1e-2, relative_step=True, scale_parameter=True, weight_decay=0.1)
    R, C = np.zeros(N, np.float32), np.zeros(K, np.float32)
    Rg, Cg = torch.zeros(N, device="cuda"), torch.zeros(K, device="cuda")
    for t in (1, 2):
        g = inputs.normal((N, K), 1e-3, seed=10 * t + K).numpy()
        R, C, st = oracle.adafactor_stats(g, c, float(s_w), R, C, t, oracle.AdafactorHP(**hp))
        a, b, sc = dqt.dqt_adafactor_stats(torch.from_numpy(g).cuda(), torch.from_numpy(c).cuda(),
                                           float(s_w), Rg, Cg, dqt.adafactor(step=t, **hp))
        # fp32 sums of positive terms, each term through at most 32 + N / 128 + 8
        # (columns) or K / 128 + 7 (rows) additions, 2^-24 each: below 128 * 2^-24
        for got, ref in ((Rg, R), (Cg, C), (a, st["a"]), (b, st["b"])):
            assert np.allclose(got.cpu().numpy(), ref, rtol=1e-5, atol=0)
        s = sc.cpu().numpy().astype(np.float64)
        for i, key in enumerate(["rbar", "step", "decay", "rms_u", "rms_x", "alpha"]):
            assert s[i] == pytest.approx(float(st[key]), rel=1e-5), (t, key)
