"""Workloads the attention path is timed on: what users of this package have it do, through its public calls.

Most cases are one training step of one attention layer (forward, then backward with the GProj correction); the others are
the forward of a block of new queries behind a key history, the host-buffer call, and the two comparison arms (key
smoothing, fused FP32).  Inputs follow ``workloads.py``: unit normals in BF16 with one common offset per KV head added to
the keys, the regime the correction exists for.
"""
import math
import random

import torch

import paper_2609_34272_b200 as g

OFFSET_NORM = 16.0      # norm of the common key offset, as in the 4096-token workloads


# ---------------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------------
def _dense(B, H, Hkv, N, d, causal):
    return {"kind": "dense", "B": B, "H": H, "Hkv": Hkv, "N": N, "d": d, "causal": causal}


def _packed(H, Hkv, total, docs, lens_seed, d, causal):
    return {"kind": "packed", "H": H, "Hkv": Hkv, "total": total, "docs": docs, "lens_seed": lens_seed, "d": d, "causal": causal}


def _rect(B, H, Hkv, Nq, Nk, d):
    return {"kind": "rect", "B": B, "H": H, "Hkv": Hkv, "Nq": Nq, "Nk": Nk, "d": d, "causal": True}


def listed():
    return [
        # Workload 1: the smallest step, four tiles in all.  Unit tests, toy models; what counts is launches and host time.
        {"name": "step_tiny_d64", **_dense(1, 2, 2, 256, 64, True)},
        # Workload 2: one layer of a small language model at 4096 tokens, batch one; the benchmark's default.
        {"name": "step_h16_n4096_d64", **_dense(1, 16, 16, 4096, 64, True)},
        # Workload 3: the same sequence length with the other head dimension.
        {"name": "step_h8_n4096_d128", **_dense(1, 8, 8, 4096, 128, True)},
        # Workload 6: the paper's own layer, 16 query heads on 4 KV heads.
        {"name": "step_h16_kv4_n4096_d64", **_dense(1, 16, 4, 4096, 64, True)},
        # Workload 4: throughput-scale batch, bidirectional (encoder training).
        {"name": "step_b4_h32_n8192_d128_full", **_dense(4, 32, 32, 8192, 128, False)},
        # Workload 5: long-context training, one sequence.
        {"name": "step_h8_n32768_d128", **_dense(1, 8, 8, 32768, 128, True)},
        # Documents of very different lengths packed into one row axis: pre-training and fine-tuning batches.
        {"name": "step_packed_16k_h16_kv4_d64", **_packed(16, 4, 16384, 24, 1, 64, True)},
        # Packed pairs with their own query and key lengths: cross-attention over a ragged batch.
        {"name": "step_packed_qk_h12_d128", "kind": "packed_qk", "H": 12, "Hkv": 12, "total": 4000, "total_k": 9000, "docs": 12,
         "lens_seed": 2, "d": 128, "causal": False},
        # Sixteen new tokens for each of eight sequences behind an 8192-key history: scoring continuations with the trained layer
        # (one new token at a time is the lower end of this range).
        {"name": "fwd_b8_q16_k8192_h16_kv4_d64", **_rect(8, 16, 4, 16, 8192, 64)},
        # Host buffers in, gradients back to host buffers: callers whose tensors live in page-locked host memory.
        {"name": "host_h16_n4096_d64", "kind": "host", "B": 1, "H": 16, "Hkv": 16, "N": 4096, "d": 64, "causal": True},
        # Key-smoothing comparison arm on packed documents: mean key removed per document, uncorrected backward, dK fixed up.
        {"name": "smooth_packed_8k_h16_kv4_d64", "kind": "smooth", **{k: v for k, v in _packed(16, 4, 8192, 16, 3, 64, True).items()
                                                                      if k != "kind"}},
        # Fused FP32 comparison arm (no tensor cores), at the length its accuracy is compared at.
        {"name": "fp32_h4_n2048_d64", "kind": "fp32", "B": 1, "H": 4, "N": 2048, "d": 64, "causal": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _heads(rng, most):
    """(query heads, KV heads): head counts up to `most`, grouped in half of the cases."""
    Hkv = rng.choice([h for h in (2, 4, 8, 12, 16) if h <= most])
    G = rng.choice([1, 1, 2, 4])
    return (Hkv * G, Hkv) if Hkv * G <= most else (Hkv, Hkv)


def draw(rng: random.Random):
    kind = rng.choice(["dense"] * 4 + ["packed"] * 2 + ["packed_qk", "rect", "rect", "host", "smooth", "fp32"])
    d = rng.choice([64, 128])
    H, Hkv = _heads(rng, 16 if kind.startswith("packed") or kind == "smooth" else 32)
    if kind == "dense":
        causal = rng.random() < 0.7
        N = _log_int(rng, 200, 16000 if causal else 10000)
        B = max(1, min(_log_int(rng, 1, 16), int((1 << 31) / (H * N * N)), (1 << 18) // (H * N)))     # an eighth of the largest listed step
        return _dense(B, H, Hkv, N, d, causal)
    if kind in ("packed", "smooth"):
        c = _packed(H, Hkv, _log_int(rng, 2000, 20000), rng.randint(4, 40), rng.randrange(1 << 30), d, kind == "smooth" or rng.random() < 0.8)
        c["kind"] = kind
        return c
    if kind == "packed_qk":
        return {"kind": kind, "H": H, "Hkv": Hkv, "total": _log_int(rng, 500, 10000), "total_k": _log_int(rng, 1000, 20000),
                "docs": rng.randint(2, 24), "lens_seed": rng.randrange(1 << 30), "d": d, "causal": rng.random() < 0.3}
    if kind == "rect":
        Nk = _log_int(rng, 1000, 40000)
        return _rect(max(1, min(_log_int(rng, 1, 16), (1 << 28) // (Hkv * Nk * d))), H, Hkv, rng.choice([1, 1, _log_int(rng, 2, 700)]), Nk, d)
    if kind == "host":
        N = _log_int(rng, 300, 8000)
        return {"kind": kind, "B": rng.choice([1, 1, 2]), "H": H, "Hkv": Hkv, "N": N, "d": d, "causal": rng.random() < 0.8}
    return {"kind": kind, "B": rng.choice([1, 2]), "H": rng.randint(1, 6), "N": _log_int(rng, 200, 3000), "d": d, "causal": rng.random() < 0.8}


# ---------------------------------------------------------------------------------------------------------------------
# sizes
# ---------------------------------------------------------------------------------------------------------------------
def _offsets(total, docs, seed):
    """`docs` sequence lengths that add up to `total`, spread over two orders of magnitude, as cumulative offsets."""
    rng = random.Random(seed)
    weights = [math.exp(rng.uniform(0.0, math.log(60.0))) for _ in range(docs)]
    s = sum(weights)
    cu, acc = [0], 0.0
    for w in weights:
        acc += w
        cu.append(min(total, max(cu[-1] + 1, int(round(total * acc / s)))))
    cu[-1] = total
    return cu


def _pairs(nq, nk, causal):
    """Score elements of one head: all of them, or those at or before the diagonal that ends at the last query and key."""
    if not causal:
        return nq * nk
    first = max(0, nq - nk)                      # leading queries without a key
    n = nq - first
    lo = max(0, nk - nq) + 1
    return n * (2 * lo + n - 1) // 2


def _problem(case):
    """Query rows and key rows per head over all batches or sequences, and score elements per query head."""
    kind = case["kind"]
    if kind in ("packed", "smooth"):
        cu = _offsets(case["total"], case["docs"], case["lens_seed"])
        return cu[-1], cu[-1], sum(_pairs(b - a, b - a, case["causal"]) for a, b in zip(cu, cu[1:]))
    if kind == "packed_qk":
        cq = _offsets(case["total"], case["docs"], case["lens_seed"])
        ck = _offsets(case["total_k"], case["docs"], case["lens_seed"] + 1)
        return cq[-1], ck[-1], sum(_pairs(q1 - q0, k1 - k0, case["causal"]) for q0, q1, k0, k1 in zip(cq, cq[1:], ck, ck[1:]))
    nq, nk = (case["Nq"], case["Nk"]) if kind == "rect" else (case["N"], case["N"])
    return case["B"] * nq, case["B"] * nk, case["B"] * _pairs(nq, nk, case["causal"])


def work(case):
    rows_q, rows_k, pairs = _problem(case)
    H, Hkv, d = case["H"], case.get("Hkv", case["H"]), case["d"]
    q, kv, row = 2 * H * rows_q * d, 2 * Hkv * rows_k * d, 4 * H * rows_q
    unit = 2.0 * H * pairs * d                   # one contraction over the score elements
    if case["kind"] == "rect":
        return {"bytes": 2 * q + 2 * kv + row, "flops": 2 * unit}
    # in: Q, K, V, dO; out: O, LSE, dQ, dK, dV.  Forward 2 contractions; backward 5, and 2 more for the correction.
    if case["kind"] == "fp32":
        return {"bytes": 4 * q + 4 * kv, "flops": 7 * unit}
    if case["kind"] == "host":
        return {"bytes": 3 * q + 4 * kv, "flops": 9 * unit}
    return {"bytes": 4 * q + 4 * kv + row, "flops": (7 if case["kind"] == "smooth" else 9) * unit}


def tolerance(case):
    # BF16 operands and outputs: every tensor is 0.17-0.25 % (relative 2-norm) from the same problem in 64 bits, and two
    # implementations with different summation orders lie within 0.3 % of each other.
    return {"rel": 7e-3 if case["kind"] == "fp32" else 1e-2}


# ---------------------------------------------------------------------------------------------------------------------
# inputs and one pass
# ---------------------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind, H, Hkv, d = case["kind"], case["H"], case.get("Hkv", case["H"]), case["d"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if kind in ("packed", "smooth", "packed_qk"):
        nq = case["total"]
        nk = case.get("total_k", nq)
        lead = ()
    else:
        nq, nk = (case["Nq"], case["Nk"]) if kind == "rect" else (case["N"], case["N"])
        lead = (case["B"],)

    def normal(heads, rows):
        return torch.randn(lead + (heads, rows, d), generator=gen, device="cuda")

    def bf16(t):
        return t.to(torch.bfloat16).contiguous()

    s = {"case": case, "scale": 1.0 / math.sqrt(d)}
    offset = normal(Hkv, 1)
    s["Q"] = bf16(normal(H, nq))
    s["K"] = bf16(normal(Hkv, nk) + offset * (OFFSET_NORM / offset.norm(dim=-1, keepdim=True)))
    s["V"] = bf16(normal(Hkv, nk))
    if kind != "rect":
        s["dO"] = bf16(normal(H, nq))
    if kind in ("packed", "smooth"):
        s["cu"] = _offsets(nq, case["docs"], case["lens_seed"])
        s["plan"] = g.VarlenPlan(s["cu"], case["causal"])
    elif kind == "packed_qk":
        s["plan"] = g.VarlenPlan(_offsets(nq, case["docs"], case["lens_seed"]), case["causal"],
                                 cu_seqlens_k=_offsets(nk, case["docs"], case["lens_seed"] + 1))
    elif kind == "host":
        for n in ("Q", "K", "V", "dO"):
            s[n] = s[n].cpu().pin_memory()
        for n, like in (("dQ", "Q"), ("dK", "K"), ("dV", "V")):
            s[n] = torch.empty_like(s[like]).pin_memory()
        s["staging"] = torch.empty(g.gproj_attn_host_staging_bytes(case["B"], H, Hkv, nq, d), dtype=torch.uint8, device="cuda")
    return s


def run(state):
    s, case = state, state["case"]
    kind, scale, causal = case["kind"], s["scale"], case["causal"]
    Q, K, V = s["Q"], s["K"], s["V"]
    if kind == "rect":
        O, LSE = g.gproj_attn_fwd_rect(Q, K, V, scale, causal)
        return {"O": O, "LSE": LSE}
    dO = s["dO"]
    if kind == "dense":
        O, LSE = g.gproj_attn_fwd(Q, K, V, scale, causal)
        dQ, dK, dV = g.gproj_attn_bwd(Q, K, V, O, LSE, dO, scale, causal)
    elif kind == "packed":
        O, LSE = g.gproj_attn_fwd_varlen(Q, K, V, s["plan"], scale)
        dQ, dK, dV = g.gproj_attn_bwd_varlen(Q, K, V, O, LSE, dO, s["plan"], scale)
    elif kind == "packed_qk":
        O, LSE = g.gproj_attn_fwd_varlen_qk(Q, K, V, s["plan"], scale)
        dQ, dK, dV = g.gproj_attn_bwd_varlen_qk(Q, K, V, O, LSE, dO, s["plan"], scale)
    elif kind == "smooth":
        Ks = g.gproj_key_smooth(K, cu_seqlens=s["cu"])
        O, LSE = g.gproj_attn_fwd_varlen(Q, Ks, V, s["plan"], scale, fwd_flags=g.FWD_FLAG_FMA_SOFTMAX)
        dQ, dKs, dV = g.gproj_attn_bwd_varlen(Q, Ks, V, O, LSE, dO, s["plan"], scale,
                                              flags=g.FLAG_NO_Q_CORRECTION | g.FLAG_NO_K_CORRECTION)
        dK = g.gproj_key_smooth(dKs, cu_seqlens=s["cu"])
    elif kind == "fp32":
        O, saved = g.gproj_fp32_attn_fwd(Q, K, V, scale, causal)
        dQ, dK, dV = g.gproj_fp32_attn_bwd(Q, K, V, dO, saved, scale, causal)
        return {"O": O, "dQ": dQ, "dK": dK, "dV": dV}
    else:
        dQ, dK, dV = s["dQ"], s["dK"], s["dV"]
        g.gproj_attn_fwd_bwd_host(Q, K, V, dO, dQ, dK, dV, scale, causal, s["staging"])
        return {"dQ": dQ, "dK": dK, "dV": dV}
    return {"O": O, "LSE": LSE, "dQ": dQ, "dK": dK, "dV": dV}
