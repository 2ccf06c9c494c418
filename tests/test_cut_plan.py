"""The plan of the steps on the cut rows (k_cut.cu, cut_plan), on the host: every problem that
the cluster form takes has a grid form as well, for a device that cannot schedule its cluster,
and each form fits the shared memory it is launched with."""
import os
import subprocess

import pytest

SOURCE = r"""
#include <cstdio>
#include "kernels.h"
using namespace hh;
// as the solver fills it; prints: cluster allowed, taken, shared memory
template <typename T> static void one(int Sx, int L, int r, int b_max) {
    for (int allowed = 1; allowed >= 0; --allowed) {
        CutProb p{};
        p.Sx = Sx; p.L = L; p.r = r; p.ncut = (1 << L) - 1; p.D = 2 * r * p.ncut;
        const size_t sm = cut_plan<T>(p, b_max, allowed != 0);
        const bool items = p.MG >= 1 && p.ngrp * p.MG >= b_max && p.nch * p.XC >= Sx && p.nA == (p.ncut + 1) * p.ngrp &&
                           p.nB == p.ncut * p.nch;
        std::printf("%d %d %d %d %d %d %d %zu %d\n", (int)sizeof(T), Sx, L, r, b_max, allowed, p.cl, sm, (int)items);
    }
}
int main() {
    for (int L = 1; L <= 4; ++L)
        for (int Sx : {8, 16, 33, 64, 65, 100, 129, 200, 257, 300})
            for (int r : {1, 4, 8, 16, 32}) {
                if ((Sx >> L) < 4 || r > Sx) continue;
                one<float>(Sx, L, r, (Sx >> L) + 3);
                one<double>(Sx, L, r, (Sx >> L) + 3);
            }
}
"""


def test_every_cluster_problem_has_a_grid_form(tmp_path):
    from paper_2512_12538_gb300 import build
    lib = build.build()
    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text(SOURCE)
    cmd = [build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", build.INCLUDE,
           str(src), "-o", str(exe), lib, "-Xlinker", f"-rpath={os.path.dirname(lib)}"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    rows = [list(map(int, line.split())) for line in
            subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    taken = {tuple(r[:5]) for r in rows if r[5] == 1 and r[6] == 1}
    assert len(taken) > 10 and all(size == 4 for size, *_ in taken)
    for size, Sx, L, r, b, allowed, cl, smem, items in rows:
        case = (size, Sx, L, r, b)
        assert items or smem == 0, case
        assert smem <= 210 * 1024, case
        if not allowed:
            assert cl == 0, case
            if case in taken:
                assert smem > 0, case
