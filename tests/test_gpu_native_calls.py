"""The dense calls as one native step: same results and the same refusals as by way of ctypes."""
import ctypes
import subprocess

import pytest
import torch

import paper_2609_34272_b200 as g
from paper_2609_34272_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture
def x():
    torch.manual_seed(0)
    return [torch.randn(*s, device="cuda").to(torch.bfloat16) for s in ((2, 4, 130, 64), (2, 2, 130, 64), (2, 2, 130, 64), (2, 4, 130, 64))]


def step(x, fwd, bwd, **kw):
    Q, K, V, dO = x
    O, LSE = fwd(Q, K, V, 0.125, True, **kw)
    return (O, LSE) + tuple(bwd(Q, K, V, O, LSE, dO, 0.125, True))


@pytest.mark.parametrize("names", [("gproj_attn_fwd", "gproj_attn_bwd"), ("gproj_attn_fwd_rect", "gproj_attn_bwd_rect")])
def test_same_results_with_and_without(x, names, monkeypatch):
    g.gproj_last_device_status()
    assert binding._calls is not None
    native = step(x, *(getattr(g, n) for n in names), fwd_flags=g.FWD_FLAG_FMA_SOFTMAX)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        other = step(x, *(getattr(g, n) for n in names), fwd_flags=g.FWD_FLAG_FMA_SOFTMAX)
    torch.cuda.current_stream().wait_stream(side)
    monkeypatch.setattr(binding, "_calls", None)
    plain = step(x, *(getattr(g, n) for n in names), fwd_flags=g.FWD_FLAG_FMA_SOFTMAX)
    for a, b, c in zip(native, plain, other):
        assert a.shape == b.shape and a.dtype == b.dtype and a.device == b.device and torch.equal(a, b) and torch.equal(a, c)


def test_refusals_are_those_of_the_checks(x):
    Q, K, V, dO = x
    O, LSE = g.gproj_attn_fwd(Q, K, V, 0.125, True)
    with pytest.raises(TypeError):
        g.gproj_attn_fwd(Q.transpose(1, 2), K, V, 0.125, True)
    with pytest.raises(TypeError):
        g.gproj_attn_fwd(Q.float(), K, V, 0.125, True)
    with pytest.raises(TypeError):
        g.gproj_attn_fwd(Q, K.cpu(), V, 0.125, True)
    with pytest.raises(ValueError):
        g.gproj_attn_fwd(Q, K[:, :, :100].contiguous(), V[:, :, :100].contiguous(), 0.125, True)
    with pytest.raises(ValueError):
        g.gproj_attn_bwd(Q, K, V, O, LSE, dO[:, :2].contiguous(), 0.125, True)
    with pytest.raises(TypeError):
        g.gproj_attn_bwd(Q, K, V, O, LSE[:, :2].contiguous(), dO, 0.125, True)
    for scale in (0.0, float("nan")):
        with pytest.raises(g.GprojError):
            g.gproj_attn_fwd(Q, K, V, scale, True)
    with pytest.raises(g.GprojError):
        g.gproj_attn_bwd(Q, K, V, O, LSE, dO, 0.125, True, flags=1 << 10)
    assert all(torch.equal(a, b) for a, b in zip(g.gproj_attn_fwd(Q, K, V, torch.tensor(0.125), 1), (O, LSE)))     # numbers of other types


def test_an_exception_out_of_the_library_leaves_the_call_to_the_checks(x, tmp_path):
    source = tmp_path / "throws.cpp"
    source.write_text('#include <new>\nextern "C" int f() { throw std::bad_alloc(); }\nextern "C" unsigned long bytes() { return 4096; }\n')
    subprocess.run(["g++", "-shared", "-fPIC", "-o", str(tmp_path / "throws.so"), str(source)], check=True)
    fake, lib = ctypes.CDLL(str(tmp_path / "throws.so")), binding.load()
    address = lambda f: ctypes.cast(f, ctypes.c_void_p).value
    Q, K, V, dO = x
    O, LSE = g.gproj_attn_fwd(Q, K, V, 0.125, True)
    expected = g.gproj_attn_bwd(Q, K, V, O, LSE, dO, 0.125, True)
    try:
        binding._calls.bind(address(fake.f), address(fake.f), address(fake.bytes))
        assert binding._calls.fwd(Q, K, V, 0.125, True, 0, True) is None
        assert all(torch.equal(a, b) for a, b in zip(g.gproj_attn_fwd(Q, K, V, 0.125, True), (O, LSE)))
        assert all(torch.equal(a, b) for a, b in zip(g.gproj_attn_bwd(Q, K, V, O, LSE, dO, 0.125, True), expected))
    finally:
        binding._calls.bind(*(address(getattr(lib, n)) for n in ("gproj_attn_fwd_rect", "gproj_attn_bwd_rect", "gproj_attn_bwd_workspace_bytes")))


def test_function_and_dispatch_modes_see_the_call(x):
    from torch.overrides import TorchFunctionMode
    from torch.utils._python_dispatch import TorchDispatchMode

    seen = []

    class Function(TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            seen.append(func)
            return func(*args, **(kwargs or {}))

    class Dispatch(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            seen.append(func)
            return func(*args, **(kwargs or {}))

    Q, K, V, _ = x
    for mode in (Function, Dispatch):
        seen.clear()
        with mode():
            g.gproj_attn_fwd(Q, K, V, 0.125, True)
        assert seen
