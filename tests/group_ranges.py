"""csrc/group_ranges.h through the host C++ compiler: the ranges that calls get."""
import os
import shutil
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_22586_gb300", "csrc")

HARNESS = r"""
#include "group_ranges.h"
#include <cstdio>
int main() {
  int G, RG, ar, nsm;
  long long keyu;
  while (std::scanf("%d %d %d %lld %d", &G, &RG, &ar, &keyu, &nsm) == 5) {
    const mmshift::GroupRanges r = mmshift::choose_ranges(G, RG, ar, 64, keyu, nsm);
    std::printf("%d %d %d", r.gper, r.ngr, (int)r.own);
    for (int i = 0; i < r.ngr; ++i) {
      int g0, g1;
      mmshift::range_groups(r, G, i, g0, g1);
      std::printf(" %d %d", g0, g1);
    }
    std::printf("\n");
  }
}
"""


def ranges(calls):
    """calls: (groups, rows a group, anchor rows, key tiles x KV heads x layers, SMs).
    For each: groups per range, whether the anchor has its own, [g0, g1) of each."""
    cxx = shutil.which("g++") or shutil.which("c++")
    assert cxx, "needs a host C++ compiler"
    with tempfile.TemporaryDirectory() as tmp:
        src, exe = os.path.join(tmp, "r.cpp"), os.path.join(tmp, "r")
        with open(src, "w") as f:
            f.write(HARNESS)
        subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, src, "-o", exe], check=True)
        out = subprocess.run([exe], input="\n".join(" ".join(map(str, c)) for c in calls), text=True,
                             capture_output=True, check=True).stdout
    got = []
    for line in out.splitlines():
        gper, ngr, own, *g = map(int, line.split())
        assert len(g) == 2 * ngr
        got.append((gper, bool(own), list(zip(g[::2], g[1::2]))))
    assert len(got) == len(calls)
    return got
