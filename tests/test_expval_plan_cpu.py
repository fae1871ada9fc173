"""Which Pauli strings share a tile pass, on the CPU: a small program around the planner's header checks
that every run is placed once, that a pass keeps the tile's limits, that the choice is the first fit by
plain scans, and that many masks (fitting tiles and not) are planned in a bounded time."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "sv_evplan.h"
using namespace svg;

static void scans(std::vector<EvRun> runs, const std::vector<uint64_t> &xs, const EvTileLimits &lim, std::vector<std::vector<EvRun>> *tiles,
                  std::vector<EvRun> *left)
{
    auto x = [&](const EvRun &r) { return xs[(size_t)r.pos]; };
    while (!runs.empty()) {
        uint64_t lam = 31;
        int strings = 0, passes = 0;
        std::vector<EvRun> took, rest;
        for (const EvRun &r : runs)
            if (__builtin_popcountll(lam | x(r)) <= lim.qubits && strings + r.m <= lim.strings && 2 * (int)(took.size() + 1) <= lim.groups) {
                lam |= x(r);
                strings += r.m;
                passes += (r.m + lim.per_pass - 1) / lim.per_pass;
                took.push_back(r);
            } else {
                rest.push_back(r);
            }
        if (took.empty()) {
            left->insert(left->end(), rest.begin(), rest.end());
            return;
        }
        if (passes < lim.passes) left->insert(left->end(), took.begin(), took.end());
        else tiles->push_back(took);
        runs.swap(rest);
    }
}

int main(int argc, char **argv)
{
    const int n = 28, count = atoi(argv[1]), weight = atoi(argv[2]), check = atoi(argv[3]);
    const EvTileLimits lim{12, 64, 32, 2, 8};
    std::mt19937_64 rng(7);
    std::vector<EvRun> runs, left, want_left;
    std::vector<uint64_t> x;
    for (int i = 0; i < count; ++i) {   // here a run's position is its number
        uint64_t m = 0;
        for (int w = (int)(rng() % (weight + 1)); w > 0; --w) m |= uint64_t(1) << rng() % n;
        x.push_back(m);
        runs.push_back(EvRun{i, rng() % 8 ? 1 : 1 + (int)(rng() % 32)});
    }
    std::vector<EvTilePass> tiles;
    const auto began = std::chrono::steady_clock::now();
    plan_tiles(runs, x, n, lim, &tiles, &left);
    printf("%.3f\n", std::chrono::duration<double>(std::chrono::steady_clock::now() - began).count());
    std::vector<int> seen((size_t)count, 0);
    for (const EvRun &r : left) ++seen[(size_t)r.pos];
    for (const EvTilePass &t : tiles) {
        int strings = 0;
        if (__builtin_popcountll(t.lam) != 12 || (t.lam & 31) != 31 || t.lam >> n) return 2;
        for (const EvRun &r : t.runs) {
            ++seen[(size_t)r.pos];
            strings += r.m;
            if (x[(size_t)r.pos] & ~t.lam) return 3;
        }
        if (strings > 64 || t.runs.size() > 16) return 4;
    }
    for (int s : seen)
        if (s != 1) return 5;
    if (check) {
        std::vector<std::vector<EvRun>> want;
        scans(runs, x, lim, &want, &want_left);
        if (want.size() != tiles.size() || want_left.size() != left.size()) return 6;
        for (size_t t = 0; t < want.size(); ++t) {
            if (want[t].size() != tiles[t].runs.size()) return 7;
            for (size_t i = 0; i < want[t].size(); ++i)
                if (want[t][i].pos != tiles[t].runs[i].pos) return 8;
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("evplan")
    (d / "plan.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2602_09604_gb300", "csrc"), str(d / "plan.cpp"), "-o", str(d / "plan")], check=True)
    return str(d / "plan")


@pytest.mark.parametrize("count", [0, 1, 2, 15, 16, 17, 64, 300, 2000])
@pytest.mark.parametrize("weight", [0, 2, 4, 14])
def test_first_fit(program, count, weight):
    assert subprocess.run([program, str(count), str(weight), "1"]).returncode == 0


@pytest.mark.parametrize("count,weight", [(50000, 4), (50000, 26), (200000, 26)])
def test_many_masks(program, count, weight):
    r = subprocess.run([program, str(count), str(weight), "0"], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and float(r.stdout) < 5.0
    print(r.stdout)
