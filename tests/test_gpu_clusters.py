"""Kernels that run as thread-block clusters, at the edges of their dispatch rules (through the C ABI, against the oracle).

Tolerances: BF16 operands and results leave 0.11 to 0.26 % relative L2 against FP64 at these sizes, and one BF16 step of the largest
value is 0.4 % of it; 0.3 % and 1 % of the largest value bound them, while one wrong weight among the sixteen parts of a merge
moves a result by several per cent.  LSE to 1e-4 + 1e-5 |LSE|.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_34272_b200 as g

pytestmark = pytest.mark.gpu


def tobits(t):
    return t.contiguous().view(torch.int16).numpy().view(np.uint16)


# The forward splits a query tile's key range over 2, 4 or 8 CTAs from 16, 16 and 32 key tiles on, when the tiles are few;
# grouped queries without a mask are folded into one head first, with one those of the second half of the list.
FWD = [  # B, H, Hkv, Nq, Nk, causal, CTAs per tile, query heads taken as one (at d = 64, at d = 128)
    (1, 2, 2, 128, 1921, True, 4, 1, 1), (1, 2, 2, 130, 2048, False, 4, 1, 1), (13, 3, 3, 1, 2047, True, 2, 1, 1), (1, 2, 2, 257, 4100, True, 8, 1, 1),
    (1, 1, 1, 64, 5000, False, 8, 1, 1), (1, 8, 2, 16, 4096, True, 8, 1, 1), (9, 6, 2, 127, 2500, True, 2, 1, 1), (1, 4, 1, 33, 300, True, 1, 1, 1),
    (1, 4, 2, 100, 40, True, 1, 1, 1), (1, 6, 2, 200, 2100, False, 4, 3, 3), (1, 8, 1, 1, 1, True, 1, 1, 1), (3, 4, 1, 96, 2049, True, 4, 1, 1),
    (40, 8, 2, 1, 300, True, 1, 4, 4), (50, 8, 2, 20, 130, True, 1, 4, 4), (70, 8, 1, 33, 300, True, 1, 1, 8), (3, 64, 8, 5, 2300, True, 4, 8, 8),
    (20, 12, 3, 60, 2100, True, 1, 4, 4), (8, 16, 4, 16, 8192, True, 4, 4, 4), (60, 8, 1, 3, 2, True, 1, 8, 8),
]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("shape", FWD)
def test_forward_with_the_key_range_split_over_a_cluster(shape, d):
    B, H, Hkv, Nq, Nk, causal, ctas, heads64, heads128 = shape
    gen = torch.Generator().manual_seed(Nq * 7 + Nk + d)
    Q = torch.randn(B, H, Nq, d, generator=gen).to(torch.bfloat16)
    K = (torch.randn(B, Hkv, Nk, d, generator=gen) + 0.5).to(torch.bfloat16)
    V = torch.randn(B, Hkv, Nk, d, generator=gen).to(torch.bfloat16)
    ex = oracle.attn_rect_f64(tobits(Q), tobits(K), tobits(V), tobits(torch.zeros_like(Q)), d ** -0.5, causal)
    q, k, v = Q.cuda(), K.cuda(), V.cuda()
    O, LSE = torch.full_like(q, float("nan")), torch.full(q.shape[:3], float("nan"), device="cuda")
    g.gproj_attn_fwd_rect(q, k, v, d ** -0.5, causal, O=O, LSE=LSE)
    assert g.gproj_last_form(g.FORM_FWD_CTAS) == ctas and g.gproj_last_form(g.FORM_FWD_HEADS) == (heads64 if d == 64 else heads128)
    rc, detail = g.gproj_last_device_status()
    assert rc == 0, hex(detail)
    O, LSE = O.float().cpu().numpy().astype(np.float64), LSE.cpu().numpy().astype(np.float64)
    empty = np.isinf(ex["LSE"])
    assert np.array_equal(np.isposinf(LSE), empty) and np.all(O[empty] == 0.0) and np.all(np.isfinite(O))
    assert np.all(np.abs(LSE[~empty] - ex["LSE"][~empty]) <= 1e-4 + 1e-5 * np.abs(ex["LSE"][~empty]))
    assert oracle.rel_l2_percent(O, ex["O"]) <= 0.3
    assert np.abs(O - ex["O"]).max() <= 0.01 * np.abs(ex["O"]).max()


# query heads folded on one CTA per tile; clusters with and without folding; the last without either, for comparison
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("shape", [(50, 8, 2, 20, 130, True), (8, 16, 4, 16, 8192, True), (1, 2, 2, 128, 4100, False), (1, 2, 2, 600, 600, True)])
def test_a_nan_reaches_every_output_row_that_sees_it(shape, d):
    B, H, Hkv, Nq, Nk, causal = shape
    gen = torch.Generator().manual_seed(Nq + Nk + d)
    rand = lambda h, n: torch.randn(B, h, n, d, generator=gen).to(torch.bfloat16).cuda()
    for name in ("Q", "K", "V"):
        x = {"Q": rand(H, Nq), "K": rand(Hkv, Nk), "V": rand(Hkv, Nk)}
        at = 1 if name == "Q" else Nk // 3
        x[name][0, 0, at, 3] = float("nan")
        O, _ = g.gproj_attn_fwd_rect(x["Q"], x["K"], x["V"], d ** -0.5, causal)
        want = torch.zeros(B, H, Nq, dtype=torch.bool)
        if name == "Q":
            want[0, 0, at] = True
        else:                                     # the queries of the KV head's group that see key `at`
            want[0, :H // Hkv] = (torch.arange(Nq) + Nk - Nq >= at) if causal else True
        nan = O.isnan().cpu()
        if name == "V":                           # one column of those rows; elsewhere 0 x NaN of a masked key may appear
            assert nan[..., 3][want].all()
        else:
            assert nan[want].all()
            if name == "Q":
                assert not nan[~want].any()
    rc, detail = g.gproj_last_device_status()
    assert rc == 0, hex(detail)


@pytest.mark.parametrize("causal", [True, False])
def test_packed_forward_with_split_keys_repeats_bitwise(causal):
    # one long and some short sequences: parts of a tile without any key tile, tiles of different length in one launch
    lens, H, Hkv, d = [2500, 3, 200, 0, 129], 2, 1, 64
    gen = torch.Generator().manual_seed(5)
    T = sum(lens)
    Q = torch.randn(H, T, d, generator=gen).to(torch.bfloat16)
    K, V = (torch.randn(Hkv, T, d, generator=gen).to(torch.bfloat16) for _ in range(2))
    cu = np.concatenate([[0], np.cumsum(lens)])
    plan = g.VarlenPlan(cu, causal)
    q, k, v = Q.cuda(), K.cuda(), V.cuda()
    O, LSE = g.gproj_attn_fwd_varlen(q, k, v, plan, 0.125)
    assert g.gproj_last_form(g.FORM_FWD_CTAS) == 2
    for _ in range(5):
        O2, LSE2 = g.gproj_attn_fwd_varlen(q, k, v, plan, 0.125)
        assert torch.equal(O, O2) and torch.equal(LSE, LSE2)
    rc, detail = g.gproj_last_device_status()
    assert rc == 0, hex(detail)
    for a, b in zip(cu, cu[1:]):
        if b > a:
            part = lambda t: tobits(t[None, :, a:b])
            ex = oracle.attn_rect_f64(part(Q), part(K), part(V), part(torch.zeros_like(Q)), 0.125, causal)
            assert oracle.rel_l2_percent(O[:, a:b].float().cpu().numpy()[None], ex["O"]) <= 0.3


@pytest.mark.parametrize("rows,d", [(1, 64), (7, 128), (8, 64), (255, 64), (257, 64), (129, 128), (513, 64), (2047, 64), (4097, 64), (2049, 128), (9000, 64)])
def test_key_smoothing_at_the_edges_of_its_row_split(rows, d):
    # one row, fewer rows than a pass, the edges of a batch of eight passes, one to eight CTAs.  FP32 sums of n values in
    # any order lie within n 2^-24 of each other relative to the sum of magnitudes; one BF16 step of the output covers it.
    gen = torch.Generator().manual_seed(rows + d)
    X = (torch.randn(3, rows, d, generator=gen) + 4.0 * torch.randn(3, 1, d, generator=gen)).to(torch.bfloat16)
    want = (X.float() - X.double().mean(dim=1, keepdim=True).float())
    buf = X.cuda()
    g.gproj_key_smooth(buf, Y=buf, cu_seqlens=[0, 0, rows, rows])
    got = buf.float().cpu()
    assert torch.all((got - want).abs() <= 2.0 ** -8 * want.abs() + 2.0 ** -20 * X.float().abs().max())


# Both backward kernels share tiles between two CTAs where whole tiles cannot be dealt evenly: one-step tiles (a CTA without a
# step of its own), odd and even step counts, query heads split between the CTAs, ragged ends, keys no query sees, rows that
# see no key; the last four have more tiles than the 74 clusters that run at once, i.e. two tiles for some of them (three on
# the dK/dV side of the last one and, at d = 64, on its dQ side).
BWD = [  # B, H, Hkv, Nq, Nk, causal, CTAs per tile: dQ and dK/dV side at d = 64, the same at d = 128
    (1, 1, 1, 700, 700, True, 2, 2, 1, 2), (1, 3, 1, 333, 333, True, 1, 2, 1, 2), (2, 4, 2, 1000, 1000, False, 2, 2, 1, 2), (1, 2, 1, 900, 130, True, 1, 2, 1, 1),
    (1, 2, 1, 641, 257, False, 1, 2, 1, 2), (1, 2, 2, 600, 1100, True, 2, 2, 2, 2), (1, 8, 2, 1025, 1025, True, 2, 2, 1, 2), (1, 1, 1, 5, 1700, True, 2, 1, 2, 1),
    (2, 5, 5, 1290, 1290, True, 2, 2, 1, 2), (1, 4, 4, 2500, 2500, True, 2, 2, 2, 2), (1, 6, 3, 2500, 2500, True, 2, 2, 2, 2), (1, 6, 6, 3100, 3100, True, 2, 2, 1, 2),
]


@pytest.mark.parametrize("flags", [0, g.FLAG_NO_K_CORRECTION])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("shape", BWD)
def test_backward_with_tiles_shared_by_two_ctas(shape, d, flags):
    B, H, Hkv, Nq, Nk, causal, *ctas = shape
    gen = torch.Generator().manual_seed(Nq + 3 * Nk + d)
    Q, dO = (torch.randn(B, H, Nq, d, generator=gen).to(torch.bfloat16) for _ in range(2))
    K = (torch.randn(B, Hkv, Nk, d, generator=gen) + 0.5).to(torch.bfloat16)
    V = torch.randn(B, Hkv, Nk, d, generator=gen).to(torch.bfloat16)
    ex = oracle.attn_rect_f64(tobits(Q), tobits(K), tobits(V), tobits(dO), d ** -0.5, causal)
    q, k, v, u = (t.cuda() for t in (Q, K, V, dO))
    O, LSE = g.gproj_attn_fwd_rect(q, k, v, d ** -0.5, causal)
    runs = []
    for _ in range(3):
        out = [torch.full_like(t, float("nan")) for t in (q, k, v)]
        runs.append(g.gproj_attn_bwd_rect(q, k, v, O, LSE, u, d ** -0.5, causal, flags=flags, dQ=out[0], dK=out[1], dV=out[2]))
    assert [g.gproj_last_form(g.FORM_DQ_CTAS), g.gproj_last_form(g.FORM_DKV_CTAS)] == (ctas[:2] if d == 64 else ctas[2:])
    rc, detail = g.gproj_last_device_status()
    assert rc == 0, hex(detail)
    assert all(torch.equal(a, b) for r in runs[1:] for a, b in zip(runs[0], r))
    for n, t in zip(("dQ", "dK", "dV"), runs[0]):
        t = t.float().cpu().numpy().astype(np.float64)
        assert np.all(np.isfinite(t)), n
        assert oracle.rel_l2_percent(t, ex[n]) <= 0.3, n
        assert np.abs(t - ex[n]).max() <= 0.01 * np.abs(ex[n]).max(), n
