"""The fused FP32 arm at the edges of its tiles (32 stationary rows, 64 streamed rows, eight warps sharing the streamed ones).

Tolerance as in test_gpu_fp32_baseline.py: the BF16 cast of the results leaves 0.17 %; 0.3 % bounds it on small tensors.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_34272_b200 as g
from paper_2609_34272_b200.workloads import Workload, bits, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("N", [2, 31, 33, 64, 65, 97, 130, 321])
def test_fp32_arm_at_tile_edges(N, d, causal):
    w = Workload("fp32_edge", 2, 2, N, d, causal, k_offset=4.0, seed=31 * N + d)
    inp = make_inputs(w)
    dev = {k: v.cuda() for k, v in inp.items()}
    O, saved = g.gproj_fp32_attn_fwd(dev["Q"], dev["K"], dev["V"], w.softmax_scale, causal)
    dQ, dK, dV = g.gproj_fp32_attn_bwd(dev["Q"], dev["K"], dev["V"], dev["dO"], saved, w.softmax_scale, causal)
    ex = oracle.attn_fwd_bwd_f64(*(bits(inp[k]) for k in ("Q", "K", "V", "dO")), w.softmax_scale, causal)
    for n, t in (("O", O), ("dQ", dQ), ("dK", dK), ("dV", dV)):
        t = t.float().cpu().numpy()
        assert np.all(np.isfinite(t)), n
        assert oracle.rel_l2_percent(t, ex[n]) <= 0.3, n
        assert np.abs(t - ex[n]).max() <= 0.01 * np.abs(ex[n]).max(), n


@pytest.mark.parametrize("d", [64, 128])
def test_fp32_arm_keeps_a_nan_in_the_normaliser(d):
    # Keys 0..3 go to one share of the streamed rows and are all that it sees of rows 0..5: its maximum stays -inf while its
    # normaliser is NaN.  Every row sees such a key, so all probabilities and with them all gradients are NaN.
    gen = torch.Generator().manual_seed(d)
    Q, K, V, dO = (torch.randn(1, 1, 6, d, generator=gen).to(torch.bfloat16).cuda() for _ in range(4))
    K[0, 0, :4] = float("nan")
    O, saved = g.gproj_fp32_attn_fwd(Q, K, V, d ** -0.5, True)
    for t in (O,) + tuple(g.gproj_fp32_attn_bwd(Q, K, V, dO, saved, d ** -0.5, True)):
        assert t.isnan().all()
