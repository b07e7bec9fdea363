"""The tile lists of the backward GEMMs (csrc/backward_plan.h, plain host code): every output tile is computed exactly once."""
import subprocess

from paper_2603_05168_b200 import build as sbn_build

PROGRAM = r"""
#include <cstdio>
#include <random>
#include <vector>
#include "backward_plan.h"

int main() {
    std::mt19937 gen(7);
    auto upto = [&](int n) { return 1 + static_cast<int>(gen() % n); };
    for (int it = 0; it < 20000; ++it) {
        const int form = static_cast<int>(gen() % 3), hint = gen() % 4 == 0 ? static_cast<int>(gen() % 2) : -1;
        const int most = it % 2 ? 40 : 6000;
        const int tiles[2] = {form == 1 ? 0 : upto(most), form == 2 ? 0 : upto(most)}, stages[2] = {upto(200), upto(200)};
        const sbn::BackwardPlan plan = sbn::plan_backward(tiles, stages, hint);
        std::vector<int> halves[2] = {std::vector<int>(tiles[0]), std::vector<int>(tiles[1])};        // bit 0, 1: the halves done
        bool ok = plan.segments >= 1 && plan.segments <= 3;
        for (int g = 0; ok && g < plan.segments; ++g) {
            const sbn::BackwardSegment& s = plan.seg[g];
            for (int pair = 0; ok && pair < sbn::kBackwardPairs; ++pair)
                for (int i = 0; ok && i < s.count(pair); ++i) {
                    const int u = s.index(pair, i), tile = s.half ? s.first_tile + (u >> 1) : u;
                    const int bits = s.half ? 1 << (u & 1) : 3;
                    ok = u >= 0 && tile < tiles[s.part] && (halves[s.part][tile] & bits) == 0;
                    if (ok) halves[s.part][tile] |= bits;
                }
        }
        for (int part = 0; part < 2; ++part)
            for (int b : halves[part]) ok = ok && b == 3;
        if (!ok) {
            std::printf("tiles %d %d stages %d %d hint %d\n", tiles[0], tiles[1], stages[0], stages[1], hint);
            return 1;
        }
    }
    return 0;
}
"""


def test_tile_lists_cover_every_tile_once(tmp_path):
    # either gradient alone, both, each split hint; fewer tiles than CTA pairs and many rounds of them
    source, program = tmp_path / "plan.cpp", tmp_path / "plan"
    source.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-I", sbn_build.CSRC, "-o", str(program), str(source)], check=True)
    run = subprocess.run([str(program)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
