"""Which host frames gmm_apply_host ticks in place: page-locked to the last
byte (not at the two ends alone), aligned, the mask apart from the frame, and
never for the staged kernel. The rule is plain C++ and is run here with made-up
registrations."""
import os
import subprocess

import pytest

import paper_2110_14934_gb300._build as B

MAIN = r"""
#include <stdio.h>
#include <stdlib.h>
#include <vector>
#include "gmm_host_frames.h"
using gmmlib::HostSpan;
// staged r d m pixels mask_bytes, then pairs lo hi of registrations
int main(int argc, char **argv) {
    std::vector<unsigned long long> v;
    for (int i = 1; i < argc; ++i)
        v.push_back(strtoull(argv[i], nullptr, 0));
    auto span_of = [&](uintptr_t q) {
        for (size_t i = 6; i + 1 < v.size(); i += 2)
            if (v[i] <= q && q < v[i + 1])
                return HostSpan{(uintptr_t)v[i], (uintptr_t)v[i + 1]};
        return HostSpan{q, q};
    };
    printf("%d\n", (int)gmmlib::frame_in_place(v[0] != 0, v[1], v[2], v[3], v[4], v[5], span_of));
    return 0;
}
"""

# 1000 pixels: rgb 3000 bytes at 0x10000, depth 2000 at 0x20000, mask 128 at 0x30000
R, D, K, N, MB = 0x10000, 0x20000, 0x30000, 1000, 128
ALL = [(R, R + 3000), (D, D + 2000), (K, K + 128)]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I", B.CSRC, "-o", str(d / "rule"), str(d / "main.cpp")], check=True)

    def run(spans, staged=0, r=R, dep=D, m=K):
        args = [staged, r, dep, m, N, MB] + [x for s in spans for x in s]
        return subprocess.run([str(d / "rule")] + [str(a) for a in args], check=True, capture_output=True, text=True).stdout.strip() == "1"

    return run


def test_whole_buffers(rule):
    assert rule(ALL)
    assert rule([(0, 1 << 20)])  # one allocation around everything
    assert rule([(R, R + 1000), (R + 1000, R + 3000)] + ALL[1:])  # registrations side by side


@pytest.mark.parametrize("which", [0, 1, 2])
def test_a_gap_anywhere_rules_it_out(rule, which):
    lo, hi = ALL[which]
    rest = ALL[:which] + ALL[which + 1:]
    assert not rule(rest)
    assert not rule(rest + [(lo, hi - 1)])                      # the last byte
    assert not rule(rest + [(lo + 1, hi)])                      # the first one
    assert not rule(rest + [(lo, lo + 50), (lo + 51, hi)])      # both ends, not the middle


def test_alignment_overlap_and_the_staged_kernel(rule):
    space = [(0, 1 << 20)]
    assert not rule(space, dep=D + 1)
    assert not rule(space, m=K + 2)
    assert not rule(space, m=R + 2996)       # over the colour frame's end
    assert rule(space, m=R + 3000)
    assert not rule(space, m=D - 124)        # over the depth frame's start
    assert not rule(space, staged=1)
