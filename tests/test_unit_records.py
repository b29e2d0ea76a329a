"""Which problems cut units into parts, and what a unit's record holds at its limits (csrc/common.cuh, host side)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2403_01254_gb300", "csrc")

PROGRAM = r"""
#include "common.cuh"
using namespace rk;
int main() {
    FrameDev f[3] = {};
    f[0].n_pts = f[1].n_pts = CUT_EDGE + 1;
    f[2].n_pts = CUT_EDGE;
    EdgeDev e[2] = {};
    e[0].a = 0, e[0].b = 1, e[1].a = 0, e[1].b = 2;
    GridParams gp{};
    if (cut_edge_for(gp, e, 1, f, 1 << 20) != 0) return 1;         // its only edge is too large
    if (cut_edge_for(gp, e, 2, f, 1 << 20) != CUT_EDGE) return 2;
    if (cut_edge_for(gp, e, 2, f, (1LL << 30) - 1) != CUT_EDGE) return 3;
    if (cut_edge_for(gp, e, 2, f, 1LL << 30) != 0) return 4;       // 2 Q records would pass 31 bits
    gp.top_k = 8;
    if (cut_edge_for(gp, e, 2, f, 1 << 20) != 0) return 5;
    for (int edge : {0, 1, 8386559, (1 << 23) - 1})                // 4096 frames have 8 386 560 pairs
        for (int n : {1, 2, 31, 32})
            for (int s = 0; s <= 3; ++s)
                for (int part = 0; part < 1 << s; ++part) {
                    const int2 u = unit_record(0x7fffffbf, edge, n, s, part);
                    const unsigned y = (unsigned)u.y;
                    int top = 0;
                    while ((y & 15) >> (top + 1)) ++top;
                    if (u.x != 0x7fffffbf || y >> 9 != (unsigned)edge || (int)((y >> 4) & 31) + 1 != n || top != s ||
                        (int)(y & 15) - (1 << s) != part)
                        return 6;
                }
    return 0;
}
"""


def test_cut_rule_and_records(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no CUDA compiler")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I" + CSRC,
                    "-I" + os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
