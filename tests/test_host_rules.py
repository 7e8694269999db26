"""The host's choices between kernels and launch shapes, checked without a GPU (host_rules.h compiled with g++)."""
import ctypes
import os
import random
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_34272_b200", "csrc")
HARNESS = r"""
#include "host_rules.h"
#include "tile_schedule.h"
using namespace gproj;
extern "C" {
int count(int ok, int n) { return count_or_none([&](int *out) { *out = n; return ok != 0; }); }
int folds(int kv_heads, int G, int N, int Nk, int d) { const int fit[4] = {0, 74, 36, 16}; return fwd_folds_heads(kv_heads, G, N, Nk, d, 148, fit); }
int smooth(long long pairs, long long rows, int longest, int d) { return smooth_cluster(pairs, rows, longest, d, 148); }
long long key_tiles(int lq, int lk, int causal) { return fwd_key_tiles(lq, lk, causal != 0); }
int short_tiles(long long key_tiles, long long tiles, int causal) { return dq_short_tiles(key_tiles, tiles, causal != 0); }
int packed_rings(const int *key_tiles, int n, int heads, int solo) { return fwd_separate_rings(std::vector<int>(key_tiles, key_tiles + n), heads, 148, solo); }
double item_cost(int d, int pairs) { return fwd_item_cost(d, pairs != 0); }
int cluster_rings(int key_tiles, int lg) { return fwd_cluster_separate_rings(key_tiles, lg); }
int rings(long long key_tiles, long long tiles) { return fwd_separate_rings(key_tiles, tiles); }
double deal(const int *steps, int n, int heads, int ctas, int solo, double per_item) {
  return deal_tiles(std::vector<int>(steps, steps + n), heads, ctas, [&](int s) { return s + per_item; }, solo);
}
double walk(const int *steps, int n, int heads, int ctas, int solo, double per_item, int *taken) {
  const int items = n * heads, G = std::min(items, ctas);
  double most = 0.0;
  for (int c = 0; c < G; ++c) {
    TileSched sched(items, solo, G, c);
    double sum = 0.0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next()) { sum += steps[lin / heads] + per_item; ++taken[lin]; }
    most = std::max(most, sum);
  }
  return most;
}
int form(const int *cu_q, const int *cu_k, int num, int causal, int packed, int key_side, int G, int heads, int tiles) {
  const DealForm f = deal_form(PackedSeqs{cu_q, cu_k, num, causal != 0}, packed != 0, key_side != 0, G, heads, tiles, 148, 74, DealCosts{64, 3.0, 8.0});
  return f.pairs ? -1 : f.solo;
}
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_rules")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "h.so"), str(d / "h.cpp")], check=True)
    return ctypes.CDLL(str(d / "h.so"))


def test_a_failed_cluster_query_means_no_clusters(rules):
    assert rules.count(1, 74) == 74 and rules.count(1, 0) == 0
    assert rules.count(0, 74) == 0                       # whatever a failing query left behind
    # ... and does not fail the set-up of a device, which calls without clusters need as well
    text = open(os.path.join(CSRC, "gproj_attn.cu")).read()
    assert "count_or_none" in text and not re.search(r"ok[^;]*=[^;]*max_clusters\(", text)


# batch x KV heads, group, queries, keys, and which form measured faster at d = 64 and at d = 128 (folded, else whole)
FOLD = [(256, 4, 100, 100, 0, 0), (64, 4, 100, 100, 0, 0), (32, 4, 100, 100, 0, 0), (256, 4, 64, 64, 0, 0), (256, 4, 32, 32, 0, 1), (2048, 4, 1, 1000, 1, 1),
        (512, 4, 16, 2048, 1, 1), (512, 4, 64, 2048, 1, 1), (128, 16, 120, 600, 0, 0), (128, 16, 64, 600, 0, 1), (128, 2, 64, 600, 1, 1), (512, 2, 100, 256, 0, 0),
        (512, 2, 16, 256, 0, 1), (8, 8, 100, 1000, 0, 0), (16, 8, 100, 1000, 0, 0), (1024, 8, 1, 64, 1, 1), (128, 4, 1, 1000, 1, 1), (64, 4, 1, 1900, 1, 1),
        (64, 2, 64, 300, 0, 0), (64, 2, 100, 1900, 0, 0), (400, 2, 64, 300, 0, 1), (60, 2, 90, 2000, 0, 0), (32, 8, 127, 1000, 0, 0), (1, 8, 1, 1, 0, 0),
        (4, 4, 10, 10, 0, 0), (184, 4, 13, 13, 0, 1), (288, 2, 47, 63, 0, 0), (368, 16, 56, 97, 0, 0), (456, 4, 108, 1567, 0, 1), (70, 8, 33, 300, 0, 1),
        (80, 4, 1, 300, 1, 1), (100, 4, 20, 130, 1, 1), (60, 8, 3, 2, 1, 1), (32, 4, 16, 8192, 1, 1), (18, 3, 127, 2500, 0, 0), (112, 2, 102, 17113, 0, 1)]


@pytest.mark.parametrize("kv_heads,G,N,Nk,folded64,folded128", FOLD)
def test_query_heads_are_folded_where_that_is_faster(rules, kv_heads, G, N, Nk, folded64, folded128):
    assert [rules.folds(kv_heads, G, N, Nk, d) for d in (64, 128)] == [folded64, folded128]
    assert rules.folds(kv_heads, G, 128, Nk, 64) == 0


# pairs, rows of each (dense), head dimension, CTAs per pair that measured fastest or within 10 % of it
SMOOTH = [(2048, 200, 64, 1), (2048, 20, 64, 1), (2048, 1000, 64, 2), (2048, 2048, 64, 4), (512, 512, 64, 1), (256, 200, 64, 1), (256, 4000, 64, 4),
          (100, 300, 64, 1), (100, 3000, 64, 4), (128, 4096, 64, 4), (16, 4096, 64, 4), (4, 8000, 64, 8), (1, 32768, 64, 8), (16, 32768, 64, 8),
          (2048, 200, 128, 1), (2048, 512, 128, 2), (2048, 1000, 128, 4), (2048, 2048, 128, 4), (512, 512, 128, 1), (128, 1000, 128, 2),
          (128, 4096, 128, 4), (64, 3000, 128, 4), (4, 8000, 128, 8), (1000, 100, 128, 1)]


@pytest.mark.parametrize("pairs,N,d,ctas", SMOOTH)
def test_key_smoothing_splits_a_sequence_where_that_is_faster(rules, pairs, N, d, ctas):
    f = rules.smooth
    f.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    assert f(pairs, pairs * N, N, d) == ctas


def walked(lq, lk, causal):
    """Key tiles of every query tile, as the forward's decode_rank counts them."""
    off = lk - lq
    return sum(max(1, -(-max(min(lk, r + 128 + off) if causal else lk, 0) // 128)) for r in range(0, lq, 128))


def test_key_tiles_of_a_sequence(rules):
    f = rules.key_tiles
    f.restype = ctypes.c_longlong
    for causal in (0, 1):
        for lq in (0, 1, 127, 128, 129, 256, 300, 1000, 1024):
            for lk in (0, 1, 100, 128, 129, 255, 256, 257, 640, 1000, 1024, 3000):
                # the closed form takes the tile in which the diagonal passes key 0 and the last, ragged one as whole tiles
                assert abs(f(lq, lk, causal) - walked(lq, lk, causal)) <= (1 if causal and lq > 0 else 0), (lq, lk, causal)


@pytest.mark.parametrize("rows,causal,two", [(128, 1, 0), (200, 0, 0), (256, 1, 0), (256, 0, 0), (512, 1, 0), (384, 0, 1), (640, 1, 1), (1500, 1, 1), (4096, 1, 1)])
def test_separate_rings_from_three_key_tiles_on(rules, rows, causal, two):
    key_tiles, tiles = ctypes.c_longlong(walked(rows, rows, causal)), ctypes.c_longlong(-(-rows // 128))
    assert rules.rings(key_tiles, tiles) == two


@pytest.mark.parametrize("rows,causal,short", [(1, 1, 1), (128, 1, 1), (500, 1, 1), (700, 1, 1), (1000, 1, 0), (4096, 1, 0), (128, 0, 1), (256, 0, 1), (384, 0, 0), (700, 0, 0)])
def test_row_constants_of_short_tiles_by_the_compute_warps(rules, rows, causal, short):
    assert rules.short_tiles(ctypes.c_longlong(walked(rows, rows, causal)), ctypes.c_longlong(-(-rows // 128)), causal) == short


def test_the_weighed_deal_is_the_kernels_deal(rules):
    rng = random.Random(1)
    args = [ctypes.POINTER(ctypes.c_int), ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_double]
    rules.deal.restype = rules.walk.restype = ctypes.c_double
    rules.deal.argtypes, rules.walk.argtypes = args, args + [ctypes.POINTER(ctypes.c_int)]
    for _ in range(300):
        n, heads, ctas = rng.randint(1, 40), rng.randint(1, 30), rng.choice([1, 2, 7, 74, 148])
        steps = sorted((rng.randint(1, 100) for _ in range(n)), reverse=True)
        solo = rng.randint(0, ctas // 2) if n * heads > ctas else 0
        arr, taken = (ctypes.c_int * n)(*steps), (ctypes.c_int * (n * heads))()
        assert abs(rules.deal(arr, n, heads, ctas, solo, 2.5) - rules.walk(arr, n, heads, ctas, solo, 2.5, taken)) < 1e-6
        assert set(taken) == {1}


def test_tiles_are_not_listed_where_the_deal_does_not_matter(rules):
    # null offsets: listing the tiles would read them
    assert rules.form(None, None, 8000, 1, 1, 0, 1, 2, 8000) == 0 and rules.form(None, None, 8000, 1, 1, 1, 1, 2, 8000) == 0
    assert rules.form(None, None, 1, 1, 0, 0, 1, 100, 12) == 0
    one = lambda n: (ctypes.c_int * 2)(0, n)
    assert rules.form(one(4096), one(4096), 1, 1, 0, 0, 1, 4, 32) == -1             # 128 tiles of very different length: pairs
    short = [128 * i for i in range(101)]
    cu_q, cu_k = ((ctypes.c_int * 102)(0, *[first + x for x in short]) for first in (300, 9000))
    assert rules.form(cu_q, cu_k, 101, 0, 1, 0, 1, 12, 103) == 36                   # three long tiles of 12 heads, 1200 short ones


def test_one_cost_of_an_item_in_every_weighing_of_the_forward(rules):
    rules.item_cost.restype = ctypes.c_double
    assert [rules.item_cost(64, 0), rules.item_cost(128, 0), rules.item_cost(128, 1)] == [1.8, 2.1, 1.45]
    text = open(os.path.join(CSRC, "gproj_attn.cu")).read()
    body = text[text.rindex("int launch_fwd("):text.index("gproj_attn_bwd_workspace_bytes(")]
    assert re.findall(r"(?:solo_ctas|tile_group_of)\(.*?fwd_item_cost\(d, [^)]*\)", body, re.S).__len__() == 2


def test_separate_rings_in_clusters_from_four_key_tiles_of_a_cta_on(rules):
    assert [rules.cluster_rings(n, 0) for n in (1, 3, 4, 5)] == [0, 0, 1, 1]
    assert [rules.cluster_rings(n, 2) for n in (15, 16)] == [0, 1] and rules.cluster_rings(16, 1) == 1


def test_separate_rings_of_a_packed_call_follow_its_longest_cta(rules):
    def rings(lens, heads, solo=0):
        tiles = sorted((-(-min(r + 128, n) // 128) for n in lens for r in range(0, n, 128)), reverse=True)
        return rules.packed_rings((ctypes.c_int * len(tiles))(*tiles), len(tiles), heads, solo)
    # sequences of one length: as their mean says
    assert [rings([n] * 60, 16) for n in (128, 256, 512, 1024)] == [0, 0, 0, 1]
    # a few long ones among many short ones: one CTA with the longest tile, the others with up to three of one key tile
    assert rings([2000] + [100] * 60, 4) == 1 and rings([100] * 80, 4) == 0
