"""Tensors that would make a kernel read or write out of bounds are refused before the library is called (no GPU needed: CPU
tensors that claim to be CUDA ones, and a library that only counts its calls)."""
import pytest
import torch

from paper_2609_34272_b200 import binding

D = 64


class Cuda(torch.Tensor):
    is_cuda = True
    index = 0

    def get_device(self):
        return self.index


def bf16(*shape):
    return torch.zeros(*shape, dtype=torch.bfloat16).as_subclass(Cuda)


def f32(*shape):
    return torch.zeros(*shape, dtype=torch.float32).as_subclass(Cuda)


def host(*shape, dtype=torch.bfloat16):
    return torch.zeros(*shape, dtype=dtype)


@pytest.fixture
def calls(monkeypatch):
    made = []

    class Library:
        def __getattr__(self, name):
            return (lambda *a: 4096) if name.endswith("_bytes") else (lambda *a: made.append(name) or 0)

    lib = Library()
    monkeypatch.setattr(binding, "_lib", lib)
    monkeypatch.setattr(binding, "load", lambda: lib)
    monkeypatch.setattr(binding, "_on_device", lambda index: binding._HERE)
    monkeypatch.setattr(binding, "_raw_stream", lambda index: 0)
    return made


class Plan:
    def __init__(self, total, total_k=None):
        self.cu = self.cu_k = (binding.ctypes.c_int * 2)(0, total)
        self.num_seqs, self.total, self.total_k, self.causal, self.device = 1, total, total if total_k is None else total_k, True, bf16(16)


X, KV, L = (1, 4, 32, D), (1, 2, 32, D), (1, 4, 32)
P, PKV = (4, 32, D), (2, 32, D)
U8 = dict(dtype=torch.uint8)


def other_device(t):
    t.index = 1
    return t


BAD_LSE = [lambda: host(*L, dtype=torch.float32), lambda: f32(1, 4, 31), lambda: bf16(*L), lambda: f32(1, 4, 64)[..., ::2], lambda: other_device(f32(*L))]
BAD_BUFFER = [lambda: host(1 << 16, **U8), lambda: host(1 << 17, **U8).as_subclass(Cuda)[::2], lambda: other_device(host(1 << 16, **U8).as_subclass(Cuda))]


@pytest.mark.parametrize("lse", BAD_LSE)
def test_a_supplied_lse_is_checked(calls, lse):
    q, k = bf16(*X), bf16(*KV)
    with pytest.raises((TypeError, ValueError)):
        binding.gproj_attn_fwd(q, k, k, 0.1, True, LSE=lse())
    with pytest.raises((TypeError, ValueError)):
        binding.gproj_attn_fwd_rect(q, k, k, 0.1, True, LSE=lse())
    assert calls == []
    binding.gproj_attn_fwd(q, k, k, 0.1, True, LSE=f32(*L))
    binding.gproj_attn_fwd_rect(q, k, k, 0.1, True, LSE=f32(4 * 32 + 5))        # a larger buffer of another shape, as before
    assert len(calls) == 2


@pytest.mark.parametrize("buffer", BAD_BUFFER)
def test_a_supplied_workspace_is_checked(calls, buffer):
    q, k, lse = bf16(*X), bf16(*KV), f32(*L)
    p, pk, plse = bf16(*P), bf16(*PKV), f32(4, 32)
    for call in (lambda w: binding.gproj_attn_bwd(q, k, k, q, lse, q, 0.1, True, workspace=w),
                 lambda w: binding.gproj_attn_bwd_rect(q, k, k, q, lse, q, 0.1, True, workspace=w),
                 lambda w: binding.gproj_attn_bwd_varlen(p, pk, pk, p, plse, p, Plan(32), 0.1, workspace=w),
                 lambda w: binding.gproj_attn_bwd_varlen_qk(p, pk, pk, p, plse, p, Plan(32), 0.1, workspace=w),
                 lambda w: binding.gproj_fp32_attn_fwd(q, q, q, 0.1, True, saved=w),
                 lambda w: binding.gproj_fp32_attn_bwd(q, q, q, q, w, 0.1, True)):
        n = len(calls)
        with pytest.raises(TypeError):
            call(buffer())
        assert len(calls) == n
        call(host(1 << 16, **U8).as_subclass(Cuda))
        assert len(calls) == n + 1


@pytest.mark.parametrize("plan,kv", [(Plan(40), PKV), (Plan(32, 48), PKV), (Plan(32), (2, 31, D)), (Plan(32), (2, 32, 128)), (Plan(32), (3, 32, D))])
def test_packed_shapes_are_checked_against_the_plan(calls, plan, kv):
    q, k, lse = bf16(*P), bf16(*kv), f32(4, 32)
    with pytest.raises(ValueError):
        binding.gproj_attn_fwd_varlen(q, k, k, plan, 0.1)
    with pytest.raises(ValueError):
        binding.gproj_attn_bwd_varlen(q, k, k, q, lse, q, plan, 0.1)
    assert calls == []


def test_offsets_of_key_smoothing_are_checked(calls):
    for heads, cu in ((1, [0, 33]), (2, [0, 10, 40]), (2, [0, 31])):
        with pytest.raises(ValueError):
            binding.gproj_key_smooth(bf16(heads, 32, D), cu_seqlens=cu)
    assert calls == []
    binding.gproj_key_smooth(bf16(1, 32, D), cu_seqlens=[0, 31])                 # one head: the leading rows, as before
    binding.gproj_key_smooth(bf16(2, 32, D), cu_seqlens=[0, 5, 32])
    assert len(calls) == 2


@pytest.mark.parametrize("name", ["K", "V", "dO", "dQ", "dK", "dV", "O", "LSE"])
def test_host_tensors_of_the_host_call_are_checked(calls, name):
    t = {n: host(*(X if n in ("Q", "dO", "dQ", "O") else KV)) for n in ("Q", "K", "V", "dO", "dQ", "dK", "dV", "O")}
    t["LSE"] = host(*L, dtype=torch.float32)
    staging = host(1 << 16, **U8).as_subclass(Cuda)
    run = lambda: binding.gproj_attn_fwd_bwd_host(t["Q"], t["K"], t["V"], t["dO"], t["dQ"], t["dK"], t["dV"], 0.1, True, staging, O=t["O"], LSE=t["LSE"])
    run()
    t[name] = t[name][:, :, :31].contiguous()
    with pytest.raises(ValueError):
        run()
    assert len(calls) == 1


def test_a_missing_tensor_is_a_type_error(calls):
    q, k, lse = bf16(*X), bf16(*KV), f32(*L)
    for at in range(4):
        args = [q, k, k, q]
        args[at] = None
        with pytest.raises(TypeError):
            binding.gproj_attn_bwd(*args, lse, q, 0.1, True)
    assert calls == []
