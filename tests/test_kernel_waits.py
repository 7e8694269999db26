"""Limits of the kernels' waits, checked without a GPU: by arithmetic, and by which wait has which limit."""
import ctypes
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_34272_b200", "csrc")
CLOCKS_PER_STEP = 2000          # upper end of what a step of any kernel takes


@pytest.fixture(scope="module")
def budget(tmp_path_factory):
    d = tmp_path_factory.mktemp("wait_budget")
    (d / "b.cpp").write_text('#include "wait_budget.h"\nextern "C" long long budget(long long s) { return gproj::tile_wait_budget(s); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "b.so"), str(d / "b.cpp")], check=True)
    f = ctypes.CDLL(str(d / "b.so")).budget
    f.restype, f.argtypes = ctypes.c_longlong, [ctypes.c_longlong]
    return f


# (query heads per KV head, queries): a single key tile's steps of 64 queries; the last is the largest that the entry points take
@pytest.mark.parametrize("G,Nq", [(1, 128), (64, 1 << 18), (16, 1 << 20), (64, 1 << 20), (127, 1 << 24)])
def test_a_wait_for_a_whole_tile_outlasts_the_tile(budget, G, Nq):
    steps = G * (Nq // 64 + 1)
    assert budget(steps) >= 4 * steps * CLOCKS_PER_STEP and budget(steps) >= budget(0) > 0


def test_a_stage_wait_outlasts_a_tile_of_the_kernel_in_front(budget):
    # the dK/dV side starts beside the dQ side's last tiles; a tile of that has at most 2^24 / 64 steps
    assert budget(0) >= (2 ** 24 // 64 + 1) * CLOCKS_PER_STEP


def test_every_wait_that_may_span_a_tile_has_the_tile_limit():
    # loaders of a stationary tile, epilogues, parts of another CTA (what waits for an epilogue waits for its last microseconds)
    bars = "res_free|acc_done|mass_ready|peer_mass|peer_ready|peer_full|peer_free|q_free"
    found = 0
    for name in ("attn_fwd.cuh", "attn_fwd_w64.cuh", "attn_bwd.cuh", "attn_bwd_w128.cuh"):
        here = found
        for line in open(os.path.join(CSRC, name)):
            for call in re.findall(r"mbar_wait(?:_cluster)?\(&bar_(?:%s)\b[^;]*;" % bars, line):
                found += 1
                assert any(b in call for b in ("tile_budget()", "kTileBudget", "tile_wait_budget(")), (name, call)
        assert found > here, name
    assert found >= 17


def test_a_cta_that_skips_its_work_still_waits_for_the_previous_kernel():
    # after a wait has given up, the CTAs of later launches return at once; one that was launched early (programmatic
    # dependent launch) must not let its grid end before the one in front of it, which may still be writing
    found = 0
    for name, kernels in (("attn_fwd.cuh", 1), ("attn_fwd_w64.cuh", 1), ("attn_bwd.cuh", 2), ("attn_bwd_w128.cuh", 1)):
        bodies = open(os.path.join(CSRC, name)).read().split("__global__")[1:]
        assert len(bodies) == kernels, name
        for body in bodies:
            for skip in re.finditer(r"if \([^()]*cta_skip != 0\)", body):
                found += 1
                # the wait stands in the branch, in front of the return, or on everybody's way before the branch
                branch = body[skip.start():body.index("return;", skip.start())]
                assert "griddep_wait();" in branch or "griddep_wait();" in body[:skip.start()], name
    assert found == 6


def test_softmax_warps_that_disagree_about_an_item_neither_hang_nor_leave_the_tensors():
    # the forward's Q loader leaves an item's rank and head in shared memory for the softmax warps.  After a wait has given up they
    # may read a slot too early or too late, each warp something else: it has to be an item of the launch all the same, so the
    # slots are written before the kernel's first barrier, and no barrier without a limit may depend on what the item is
    for name in ("attn_fwd.cuh", "attn_fwd_w64.cuh"):
        body = open(os.path.join(CSRC, name)).read().split("__global__")[1]
        setup = body[:body.index("fence_mbar_init();")]
        assert re.search(r"for \(auto &slot : s_item\) slot\[0\] = slot\[1\] = 0;", setup), name
        role = body[body.index("setmaxnreg_inc"):]
        barriers = re.findall(r"named_bar_sync\([^;]*;|__syncthreads\(\);", role)
        # behind the item loop, and in the cluster form, whose single item every warp reaches the barrier of (warp_bar_sync is one warp's own)
        assert barriers == (["named_bar_sync(3, 256);", "__syncthreads();", "__syncthreads();"] if name == "attn_fwd.cuh" else ["__syncthreads();"]), (name, barriers)
