"""How a pool's tick is cut into launches and tiles, and the shapes its tuner
tries (plain C++, compiled here): a launch's tiles follow the pixels of that
launch, and the tuner's shapes are those that run, each once."""
import subprocess

import pytest

import paper_2110_14934_gb300._build as B

MAIN = r"""
#include <stdio.h>
#include <stdlib.h>
#include "gmm_pool_plan.h"
using namespace gmmlib;
// plan threads ctas tile blocks, or tune sms; then per camera: M n_pad
int main(int argc, char **argv) {
    const bool tune = argv[1][0] == 't';
    std::vector<TickCam> cams;
    for (int i = tune ? 3 : 6, k = 0; i + 1 < argc; i += 2, ++k)
        cams.push_back({k, atoi(argv[i]), atoll(argv[i + 1])});
    if (!tune) {
        std::vector<LaunchPlan> plan;
        plan_launches(cams, Shape{atoi(argv[2]), atoi(argv[3]), atoi(argv[4])}, atoi(argv[5]), plan);
        for (const LaunchPlan &l : plan)
            printf("%d %d %d %d\n", l.first, l.count, l.m, l.unit);
        return 0;
    }
    const int sms = atoi(argv[2]);
    std::vector<Shape> shapes;
    for (int t : {64, 128, 256})
        for (int c : {1024 / t, 512 / t})
            for (int tp : {256, 512, 1024, 2048, 8192})
                shapes.push_back({t, c, tp});
    for (const Shape &s : distinct_shapes(shapes, cams, [&](const Shape &x) { return sms * x.ctas; }))
        printf("%d %d %d\n", s.threads, s.ctas, s.tile);
    return 0;
}
"""


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I", B.CSRC, "-o", str(d / "plan"), str(d / "main.cpp")], check=True)

    def run(*args):
        out = subprocess.run([str(d / "plan")] + [str(a) for a in args], check=True, capture_output=True, text=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]

    return run


def _cams(*groups):
    return [x for M, n_pad, count in groups for _ in range(count) for x in (M, n_pad)]


def test_tiles_follow_the_launch_not_the_tick(planner):
    one = planner("plan", 128, 8, 2048, 1216, *_cams((5, 76800, 128)))
    two = planner("plan", 128, 8, 2048, 1216, *_cams((5, 76800, 256)))
    assert len(one) == 1 and [(f, c) for f, c, _, _ in two] == [(0, 128), (128, 128)]
    assert [u for _, _, _, u in two] == [one[0][3]] * 2
    # a last launch of a few cameras has small tiles, whatever ran before it
    three = planner("plan", 128, 8, 2048, 1216, *_cams((5, 2073600, 128), (3, 76800, 2)))
    few = planner("plan", 128, 8, 2048, 1216, *_cams((3, 76800, 2)))
    assert three[0][3] == 2048 and three[1][3] == few[0][3] == 128


@pytest.mark.parametrize("threads,tile", [(64, 64), (96, 960), (128, 2048), (256, 8192)])
def test_every_launch_is_whole(planner, threads, tile):
    for n in (1, 127, 128, 129, 300):
        for n_pad in (32, 306560, 2073600):
            for ctas in (2, -1):
                cams = _cams((5, n_pad, n), (4, 32, 1), (3, n_pad, 2))
                plan = planner("plan", threads, ctas, 32 if ctas < 0 else tile, 304, *cams)
                assert [f for f, _, _, _ in plan] == [sum(c for _, c, _, _ in plan[:i]) for i in range(len(plan))]
                assert sum(c for _, c, _, _ in plan) == n + 3
                assert all(0 < c <= 128 for _, c, _, _ in plan)
                for first, count, m, unit in plan:
                    if ctas < 0:
                        assert unit == 32 and {cams[2 * (first + i)] for i in range(count)} == {m}
                    else:
                        assert m == 0 and threads <= unit <= tile and unit % threads == 0


def test_the_tuner_tries_each_shape_that_runs_once(planner):
    large = planner("tune", 152, *_cams((5, 2073600, 64)))
    assert len(large) == 30 and {t for _, _, t in large} >= {256, 512, 1024, 2048}
    small = planner("tune", 152, *_cams((5, 76800, 4)))
    assert len(set(small)) == len(small) < 30
    for threads, ctas, tile in small:  # the tile is the one that runs, and stays so
        assert planner("plan", threads, ctas, tile, 152 * ctas, *_cams((5, 76800, 4)))[0][3] == tile
