"""Forward kernels at the edges of their dispatch rules and of their tiles (through the C ABI, against the oracle).

Tolerances as in test_gpu_clusters.py: BF16 operands and results leave up to 0.26 % relative L2 against FP64, one BF16 step of the
largest value is 0.4 % of it; a wrong tile, part or rescale moves a result by several per cent.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_34272_b200 as g

pytestmark = pytest.mark.gpu


def tobits(t):
    return t.contiguous().view(torch.int16).numpy().view(np.uint16)


def kernel():
    return g.FWD_KERNELS[g.gproj_last_form(g.FORM_FWD_KERNEL)]


def check_forward(B, H, Hkv, Nq, Nk, causal, d, fma):
    """Run the call; compare whole batches or, of more than 24 heads, the first and the last KV heads with the oracle."""
    gen = torch.Generator().manual_seed(Nq * 7 + Nk + d)
    Q = torch.randn(B, H, Nq, d, generator=gen).to(torch.bfloat16)
    K = torch.randn(B, Hkv, Nk, d, generator=gen) + 0.5
    K[:, :, Nk // 2:] *= 3.0                      # the running maximum moves on the way
    K = K.to(torch.bfloat16)
    V = torch.randn(B, Hkv, Nk, d, generator=gen).to(torch.bfloat16)
    q, k, v = Q.cuda(), K.cuda(), V.cuda()
    O, LSE = torch.full_like(q, float("nan")), torch.full(q.shape[:3], float("nan"), device="cuda")
    g.gproj_attn_fwd_rect(q, k, v, d ** -0.5, causal, O=O, LSE=LSE, fwd_flags=fma * g.FWD_FLAG_FMA_SOFTMAX)
    rc, detail = g.gproj_last_device_status()
    assert rc == 0, hex(detail)
    assert bool(torch.isfinite(O).all()) and not bool(torch.isnan(LSE).any())
    if H > 24:
        few, G = max(1, 8 // B), H // Hkv
        kv = sorted({*range(min(few, Hkv)), *range(max(0, Hkv - few), Hkv)})
        heads = [h for i in kv for h in range(i * G, (i + 1) * G)]
        Q, K, V, O, LSE = Q[:, heads], K[:, kv], V[:, kv], O[:, heads], LSE[:, heads]
    ex = oracle.attn_rect_f64(tobits(Q), tobits(K), tobits(V), tobits(torch.zeros_like(Q)), d ** -0.5, causal)
    O, LSE = O.float().cpu().numpy().astype(np.float64), LSE.cpu().numpy().astype(np.float64)
    empty = np.isinf(ex["LSE"])
    assert np.array_equal(np.isposinf(LSE), empty) and np.all(O[empty] == 0.0)
    assert np.all(np.abs(LSE[~empty] - ex["LSE"][~empty]) <= 1e-4 + 1e-5 * np.abs(ex["LSE"][~empty]))
    assert oracle.rel_l2_percent(O, ex["O"]) <= 0.3
    assert np.abs(O - ex["O"]).max() <= 0.01 * np.abs(ex["O"]).max()


# On 148 SMs.  d = 64: single tiles on three warpgroups whatever the call.  d = 128: pairs of query tiles need 222 pairs; an odd tile
# at the end, one or two rows in the last tile, ends of key tiles.  Single tiles: with one item per CTA two and three key tiles, then
# more items than CTAs on both sides of three key tiles per item.
SHAPES = [  # B, H, Hkv, Nq, Nk, causal, kernel at d = 128
    (1, 112, 112, 257, 257, True, "pairs"), (1, 112, 56, 258, 385, True, "pairs"), (2, 75, 25, 300, 130, True, "pairs"), (1, 222, 222, 256, 1, False, "pairs"),
    (1, 112, 112, 384, 640, False, "pairs"), (1, 111, 111, 384, 130, False, "pairs"), (1, 110, 110, 384, 130, False, "split"), (1, 60, 60, 513, 513, True, "split, rings"),
    (1, 223, 223, 129, 128, True, "pairs"), (3, 100, 100, 128, 200, True, "one tile"), (2, 150, 75, 77, 77, True, "one tile"), (1, 222, 222, 100, 500, False, "one tile"),
    (1, 221, 221, 100, 500, False, "split, rings"), (1, 3, 3, 256, 256, True, "split"), (1, 3, 3, 257, 257, True, "split, rings"), (1, 16, 4, 300, 300, True, "split, rings"),
    (1, 60, 60, 384, 384, True, "split"), (1, 40, 40, 640, 640, True, "split, rings"), (1, 2, 2, 1, 385, False, "split, rings"), (1, 5, 5, 200, 64, True, "split"),
    (1, 3, 1, 130, 1030, True, "split, rings"), (1, 128, 128, 512, 512, False, "pairs"), (1, 296, 296, 256, 256, False, "pairs"), (1, 96, 96, 1000, 1000, False, "pairs"),
]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("fma", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_forward_forms(shape, d, fma):
    check_forward(*shape[:6], d, fma)
    assert kernel() == ("three" if d == 64 else shape[6])
    assert g.gproj_last_form(g.FORM_FWD_CTAS) == 1


# Folded query heads, one CTA to a tile, on both sides of four key tiles at d = 128; clusters of two, four and eight, which have at
# least four key tiles to a CTA.  The last two: the same sizes with the fused exponent, which has no cluster form, and whole heads.
MERGED = [  # B, H, Hkv, Nq, Nk, causal, fma, kernel at d = 64, at d = 128
    (40, 8, 2, 1, 384, True, 0, "cluster", "cluster"), (40, 8, 2, 1, 385, True, 0, "cluster", "cluster, rings"), (13, 3, 3, 1, 2047, True, 0, "cluster", "cluster, rings"),
    (1, 2, 2, 130, 2048, False, 0, "cluster", "cluster, rings"), (1, 1, 1, 64, 4097, False, 0, "cluster", "cluster, rings"),
    (40, 8, 2, 1, 385, True, 1, "three", "one tile"), (13, 3, 3, 1, 1900, True, 0, "three", "split, rings"),
]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("shape", MERGED)
def test_forward_forms_merged_by_a_cluster(shape, d):
    check_forward(*shape[:6], d, shape[6])
    assert kernel() == shape[7 + (d == 128)]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("lens", [[1 + (7 * i) % 64 for i in range(300)], [64] * 40 + [65, 129, 1, 0, 193, 400, 63] * 12], ids=["one_step", "mixed"])
def test_packed_forward_of_many_short_sequences(lens, d):
    """Items of one, two and three 64-key steps behind one another on every CTA."""
    H = 8
    cu = np.concatenate([[0], np.cumsum(lens)])
    T = int(cu[-1])
    gen = torch.Generator().manual_seed(T + d)
    Q, K, V = (torch.randn(H, T, d, generator=gen).to(torch.bfloat16) for _ in range(3))
    plan = g.VarlenPlan([int(c) for c in cu], causal=True)
    O, LSE = g.gproj_attn_fwd_varlen(Q.cuda(), K.cuda(), V.cuda(), plan, d ** -0.5)
    assert kernel() == ("three" if d == 64 else "split")
    rc, detail = g.gproj_last_device_status()
    assert rc == 0, hex(detail)
    O, LSE = O.double().cpu(), LSE.double().cpu()
    for a, b in zip(cu[:-1], cu[1:]):
        if a == b:
            continue
        s = (Q[:, a:b].double() @ K[:, a:b].double().transpose(1, 2)) * d ** -0.5
        s = s.masked_fill(torch.ones(b - a, b - a, dtype=torch.bool).triu(1), -float("inf"))
        ex = torch.softmax(s, -1) @ V[:, a:b].double()
        assert float((O[:, a:b] - ex).norm() / ex.norm()) <= 3e-3
        assert float((O[:, a:b] - ex).abs().max()) <= 0.01 * float(ex.abs().max())
        assert float((LSE[:, a:b] - torch.logsumexp(s, -1)).abs().max()) <= 2e-4
