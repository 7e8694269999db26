"""The native call layer is optional: what the binding and the build do where it is unusable (no GPU needed)."""
import os
import subprocess
import sys
import warnings

import pytest

import __graft_entry__ as entry
from paper_2609_34272_b200 import binding, build


@pytest.fixture
def unloaded(monkeypatch):
    """The binding as in a new process."""
    entry.build()
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_calls", None)


def test_a_file_that_does_not_load_leaves_the_calls_to_ctypes(unloaded, tmp_path, monkeypatch):
    bad = tmp_path / "_torch_calls.so"
    bad.write_bytes(b"not a shared object")
    monkeypatch.setattr(binding, "CALLS_PATH", str(bad))
    with pytest.warns(RuntimeWarning, match="ctypes"):
        lib = binding.load()                       # the first call is as good as any later one ...
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        assert binding.load() is lib               # ... and says so once
    assert binding._calls is None and lib.gproj_attn_bwd_workspace_bytes(1, 2, 256, 64) > 0


def test_a_call_that_fails_half_way_through_loading_is_repeated(unloaded, monkeypatch):
    def fail(lib):
        raise MemoryError
    monkeypatch.setattr(binding, "_bind_native_calls", fail)
    for _ in range(2):
        with pytest.raises(MemoryError):
            binding.load()


def test_another_torch_or_python_gets_a_layer_of_its_own(monkeypatch):
    entry.build()
    made = []
    monkeypatch.setattr(build, "_run", lambda cmd, verbose=False: made.append(cmd[0]))
    build.build()
    assert made == [] and build.calls_path() == binding.CALLS_PATH
    for owner, name in ((sys.modules["torch"], "__version__"), (sys.implementation, "cache_tag")):
        with monkeypatch.context() as m:
            m.setattr(owner, name, "0.0")
            assert build.calls_path() != binding.CALLS_PATH
            build.build()
            assert made == ["g++"]
        made.clear()


def test_a_host_compiler_that_fails_does_not_fail_the_build(monkeypatch, tmp_path):
    entry.build()
    stale = tmp_path / "_torch_calls.so"
    monkeypatch.setattr(build, "calls_path", lambda: str(stale))
    for command in (["false"], ["/nonexistent/g++"]):
        stale.write_bytes(b"")
        os.utime(stale, (0, 0))
        monkeypatch.setattr(build, "calls_command", lambda: command)
        with pytest.warns(RuntimeWarning, match="native call layer"):
            assert build.build() == build.LIB
        assert not stale.exists()                  # an old one might call the library by another signature


def test_the_layer_calls_by_the_headers_signatures(tmp_path, monkeypatch):
    entry.build()
    # a call that does not fit a changed signature no longer compiles ...
    changed = tmp_path / "gproj_attn.h"
    changed.write_text(open(build.ABI_HEADER).read().replace("int gproj_attn_bwd_rect(", "int gproj_attn_bwd_rect(long long added, ", 1))
    command = [c for c in build.calls_command() if c != "-shared"]
    out = command.index("-o")
    done = subprocess.run([command[0], "-fsyntax-only", f"-I{tmp_path}"] + command[1:out] + [command[out + 2]], capture_output=True, text=True)
    assert done.returncode != 0 and "bwd_fn" in done.stderr
    # ... and a changed header makes the layer out of date
    made = []
    monkeypatch.setattr(build, "_run", lambda cmd, verbose=False: made.append(cmd[0]))
    monkeypatch.setattr(build, "ABI_HEADER", str(changed))
    build.build()
    assert made == ["g++"]


def test_the_forward_encodes_each_tensor_map_once():
    # an encoded map is 0.15 us of host time; the smallest calls are bound by that
    source = open(build.SOURCES[0]).read()
    body = source[source.index("int launch_fwd(", source.index("int launch_fwd(") + 1):]
    assert body[:body.index("\n}\n")].count("make_map(&") == 4
