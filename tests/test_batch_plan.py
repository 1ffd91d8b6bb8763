"""The equal shares of a batch's 3D columns (csrc/batch_plan.h): a host program
walks them as the persistent step does, for random batches of both precisions."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1510_05061_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include <cstdio>
#include <random>
#include <cuda_runtime.h>
#include "batch_plan.h"
using namespace hydro;
#define CHECK(c) do { if (!(c)) { std::printf("case %d: %s\n", n, #c); return 1; } } while (0)
int main()
{
    std::mt19937 rng(7);
    for (int n = 0; n < 400; ++n) {
        const bool fp32 = n % 2 == 0;
        const int count = 1 + rng() % (n < 300 ? 12 : 60), hi = n < 100 ? 12 : 130;
        std::vector<hydro_problem> probs(count);
        std::vector<const hydro_problem *> pp;
        double cells = 0.0;
        for (hydro_problem &p : probs) {
            for (int d = 0; d < 3; ++d) p.n[d] = 2 + rng() % hi;
            pp.push_back(&p);
            cells += (double)p.n[0] * p.n[1] * p.n[2];
        }
        BatchPlan plan = batch_plan(pp.data(), count, fp32, -1);
        if (fp32 && cells * 20 > 160e6) { CHECK(plan.shares == 0); continue; }   // chunks there
        if (n % 5 == 4) {
            const int v = rng() % 8;   // the kernel chosen before a change of membership, or none modelled
            plan = batch_plan(pp.data(), count, fp32, v);
            if (plan.shares == 0) { CHECK(fp32 ? v % 4 == 0 : v % 4 == 3); continue; }
            CHECK(plan.variant == v);
        }
        const TileShape s = TILE3D_SHAPES[plan.variant];
        std::vector<BatchItem> cut;
        CutState c{};
        std::vector<int> tiles(count), pieces(count);
        long long planes = 0, capacity = 0;
        for (int i = 0; i < count; ++i) {
            tiles[i] = ((probs[i].n[0] + s.tx - 1) / s.tx) * ((probs[i].n[1] + s.ty - 1) / s.ty);
            planes += (long long)tiles[i] * probs[i].n[2];
            cut_columns(plan, i, tiles[i], probs[i].n[2], c, cut, &pieces[i]);
            CHECK(pieces[i] <= tiles[i] * probs[i].n[2]);
        }
        CHECK(c.shares >= 1 && c.shares <= plan.shares);
        const std::vector<BatchItem> items = claim_order(cut);
        CHECK(items.size() == cut.size());
        // every plane of every column once, by the shares' links from the claimed items
        std::vector<std::vector<char>> seen(count), slot(count);
        for (int i = 0; i < count; ++i) {
            seen[i].assign((size_t)tiles[i] * probs[i].n[2], 0);
            slot[i].assign(pieces[i], 0);
        }
        size_t visited = 0;
        double longest = 0.0;
        for (int k = 0; k < c.shares; ++k) {
            double cost = 0.0;
            for (int it = k; it >= 0; it = items[it].next) {
                const BatchItem w = items[it];
                CHECK(it == k || it >= c.shares);
                CHECK(w.z0 >= 0 && w.z0 < w.z1 && w.z1 <= probs[w.inst].n[2] && w.tile >= 0 && w.tile < tiles[w.inst]);
                for (int z = w.z0; z < w.z1; ++z) CHECK(seen[w.inst][(size_t)w.tile * probs[w.inst].n[2] + z]++ == 0);
                CHECK(w.local >= 0 && w.local < pieces[w.inst] && slot[w.inst][w.local]++ == 0);
                cost += w.z1 - w.z0 + plan.fixed;
                CHECK(++visited <= items.size());
            }
            longest = std::max(longest, cost);
        }
        CHECK(visited == items.size());
        for (int i = 0; i < count; ++i)
            for (char x : seen[i]) CHECK(x == 1);
        // a share passes its budget by less than a plane and one piece's cost
        CHECK(longest <= plan.budget + plan.fixed + 1.0);
    }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.isdir(os.path.join(CUDA, "include")),
                    reason="needs g++ and the CUDA headers")
def test_shares_cover_the_columns(tmp_path):
    src, exe = str(tmp_path / "t.cpp"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(CUDA, "include"), src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
