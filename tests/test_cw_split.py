"""How gemv_cw shares the resident clusters between the layers of a group (csrc/cw_split.h, host arithmetic):
the passes are the fewest that fit, every layer has a cluster, and the search ends also where there are more
layers than resident clusters (three clusters of eight with two token tiles on 64 SMs)."""
import itertools
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include <cstdio>
#include "cw_split.h"
int main() {
    int n, cap, r[4];
    while (std::scanf("%d %d %d %d %d %d", &n, &cap, r, r + 1, r + 2, r + 3) == 6)
        std::printf("%d\n", aq::cw_group_passes(r, n, cap));
}
"""


def test_group_passes(tmp_path):
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2606_12876_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    heights = (1, 2, 3, 31, 32, 449, 67108864)
    cases = [(n, cap, r) for n in (1, 2, 3, 4) for cap in (1, 2, 3, 8, 16, 76, 152)
             for r in itertools.combinations_with_replacement(heights, n) if n < 4 or sum(r) < 2000 or r[0] > 32]
    text = "".join("%d %d %s\n" % (n, cap, " ".join(map(str, (r + (0, 0, 0, 0))[:4]))) for n, cap, r in cases)
    out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True, timeout=60).stdout
    got = list(map(int, out.split()))
    assert len(got) == len(cases)
    for (n, cap, r), p in zip(cases, got):
        need = lambda q: sum(-(-b // q) for b in r)
        assert p >= 1 and need(p) <= max(cap, n), (n, cap, r, p)
        if p > 1:
            assert need(p - 1) > max(cap, n), (n, cap, r, p)
