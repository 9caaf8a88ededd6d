"""split_parts: the patches of a level share a scratch of bounded size, in order, each
in exactly one part and none overlapping another of its part."""
import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include "parts.hpp"
#include <cstdio>
int main() {
    long long cap, n;
    while (std::scanf("%lld %lld", &cap, &n) == 2) {
        std::vector<long long> size(n), off;
        std::vector<int> first;
        for (auto& x : size) if (std::scanf("%lld", &x) != 1) return 1;
        std::printf("%lld", split_parts(size, cap, off, first));
        for (long long x : off) std::printf(" %lld", x);
        std::printf(" |");
        for (int x : first) std::printf(" %d", x);
        std::printf("\n");
    }
}
"""


def test_parts_are_bounded_and_disjoint(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "parts")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2407_07253_gb300", "csrc"), "-o", exe,
                    str(tmp_path / "main.cpp")], check=True)
    rng = np.random.default_rng(0)
    cases = [(10, []), (10, [10]), (10, [11, 3, 12]), (1 << 29, [100_000] * 12_000)]
    cases += [(int(rng.integers(1, 200)), rng.integers(1, 60, int(rng.integers(1, 80))).tolist()) for _ in range(60)]
    text = "\n".join(f"{cap} {len(size)} " + " ".join(map(str, size)) for cap, size in cases)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
    for (cap, size), line in zip(cases, out):
        left, first = line.split("|")
        most, *off = map(int, left.split())
        first = list(map(int, first.split()))
        assert first == sorted(set(first)) and first[0] == 0 and first[-1] == len(size)
        tops = [0]
        for a, b in zip(first, first[1:]):
            assert off[a] == 0 and off[a:b] == np.cumsum([0] + size[a:b - 1]).tolist()
            tops.append(off[b - 1] + size[b - 1])
            assert tops[-1] <= cap or b == a + 1
            assert b == len(size) or tops[-1] + size[b] > cap        # no part ends early
        assert most == max(tops)
