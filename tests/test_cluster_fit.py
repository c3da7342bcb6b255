"""The sizes of the clusters, and a device that has no room for one: the kernels
that need no cluster are taken (asked through a fake, no device needed)."""
import os
import shutil
import subprocess

import pytest

from paper_1808_00270_gb300 import build as B

SRC = r"""
#include <cstdio>
#include "cluster_fit.h"
#define CHECK(x) do { if (!(x)) { std::printf("line %d\n", __LINE__); return 1; } } while (0)
using namespace gld;
int main() {
    CHECK(cluster_ctas(1, 8) == 1 && cluster_ctas(64, 8) == 1 && cluster_ctas(65, 8) == 2);
    CHECK(cluster_ctas(1024, 8) == 16 && cluster_ctas(4096, 8) == 16 && cluster_ctas(8192, 4) == 16);
    CHECK(cluster_lanes(1024, 16) == 8 && cluster_lanes(1025, 16) == 4 && cluster_lanes(2049, 16) == 2);
    CHECK(scan_totals(1) == 16 && scan_totals(8192) == 16 && scan_totals(8193) == 17);  // a word per CTA at least
    int a = 0, b = 0, asked = 0;
    size_t seen = 0;
    ClusterFit fit;
    auto none = [&](size_t s) { ++asked; seen = s; return 0; };  // nothing resident, or the question failed
    auto some = [&](size_t s) { ++asked; seen = s; return 3; };
    CHECK(!fit(0, &a, 16, 70000, none) && asked == 1 && seen >= 70000);
    CHECK(!fit(0, &a, 16, 70001, some) && asked == 1);      // the answer is kept
    CHECK(fit(0, &a, 8, 70000, some) && asked == 2);        // another shape,
    CHECK(fit(0, &b, 16, 70000, some) && asked == 3);       // kernel,
    CHECK(fit(1, &a, 16, 70000, some) && asked == 4);       // device,
    CHECK(fit(0, &a, 16, 50000, some) && asked == 5);       // or size
    CHECK(fit(0, &a, 16, 50000, none) && asked == 5);
    std::puts("ok");
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no C++ compiler")
def test_cluster_fit(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", B.CSRC, str(src), "-o", str(exe), "-lpthread"],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout


def test_the_cluster_kernels_ask_first():
    """Both rules that send work to a cluster end in the question."""
    s = open(os.path.join(B.CSRC, "k_cluster.cu")).read()
    for rule in ("bool cluster_ok(", "bool rebuild_in_cluster("):
        body = s[s.index(rule):]
        assert "cluster_fits(" in body[: body.index("\n}\n")]


def test_cluster_barriers_take_lanes_one_by_one():
    """The barriers stand behind loops that lanes leave by break and continue: the
    form that presumes a converged warp is not used."""
    asm = [x for x in open(os.path.join(B.CSRC, "k_cluster.cu")) if "barrier.cluster" in x]
    assert asm and not any(".aligned" in x for x in asm)
