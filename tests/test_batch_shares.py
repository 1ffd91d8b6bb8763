"""Which FP32 batches take equal shares of their columns and which claim
chunks (csrc/batch_plan.h, host only): shares cost more pieces, so they must not
be taken where three batches at once were measured slower with them."""

import os
import subprocess

from test_plan2d import CSRC, CUDA, needs_gxx

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <cuda_runtime.h>
#include "batch_plan.h"
int main()
{
    int count;
    while (std::scanf("%d", &count) == 1) {
        std::vector<hydro_problem> probs(count);
        std::vector<const hydro_problem *> pp;
        for (hydro_problem &p : probs) {
            std::memset(&p, 0, sizeof p);
            std::scanf("%d", &p.n[0]);
            p.n[1] = p.n[2] = p.n[0];
            pp.push_back(&p);
        }
        const hydro::BatchPlan plan = hydro::batch_plan(pp.data(), count, true, -1);
        std::printf("%d\n", plan.shares > 0 && hydro::shares_pay(plan, pp.data(), count, 7));
    }
}
"""

# (smallest, largest, boxes): time of three batches in turn, chunks over shares
MEASURED = {(17, 113, 4): 2.68, (31, 67, 7): 1.31, (18, 66, 16): 1.26, (23, 99, 6): 1.09, (39, 91, 9): 1.05,
            (19, 98, 11): 1.03, (25, 96, 16): 1.02, (32, 128, 14): 1.00, (35, 115, 6): 0.952, (24, 123, 9): 0.937,
            (36, 128, 6): 0.969, (20, 127, 10): 0.980, (39, 142, 8): 0.984, (18, 116, 14): 0.986, (27, 110, 16): 0.991, (22, 112, 10): 0.977, (38, 134, 6): 0.992,
            (18, 125, 5): 0.936, (18, 96, 9): 1.01, (24, 90, 5): 1.03}


def cubes(lo, hi, n):
    """The 3D boxes of a batch: sizes spread over their logarithm, every fourth box 2D."""
    sizes = [int(round(lo * (hi / lo) ** (i / (n - 1)))) for i in range(n)]
    return [s for i, s in enumerate(sizes) if i % 4 != 3]


@needs_gxx
def test_shares_only_where_they_cost_no_work(tmp_path):
    src, exe = str(tmp_path / "t.cpp"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(CUDA, "include"), src, "-o", exe], check=True)
    lists = [cubes(*m) for m in MEASURED]
    r = subprocess.run([exe], input="".join(f"{len(b)} {' '.join(map(str, b))}\n" for b in lists), capture_output=True,
                       text=True, check=True)
    for (m, ratio), taken in zip(MEASURED.items(), r.stdout.split()):
        assert (taken == "1") == (ratio >= 1.0), (m, ratio)
