"""The host's choices between kernels and launch shapes, checked without a GPU (host_rules.h compiled with g++)."""
import ctypes
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_34272_b200", "csrc")
HARNESS = r"""
#include "host_rules.h"
using namespace gproj;
extern "C" {
int count(int ok, int n) { return count_or_none([&](int *out) { *out = n; return ok != 0; }); }
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
