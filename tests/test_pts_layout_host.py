"""Host arithmetic of the point-owner projection's shared memory
(csrc/pts_layout.cuh), compiled with the system C++ compiler: the blocks are
aligned and disjoint, and whatever a launch that returns multipliers reserves for the
fixed columns' rows is what the kernel's own layout asks for, at every n_p and
group size, unless it would cost an SM its second CTA.  No GPU needed."""
import shutil
import subprocess

import pytest

from test_grid_layout_host import CSRC, INC, cuda_include

DRIVER = r"""
#include <cstdio>
#include "pts_layout.cuh"

using namespace priest;
using namespace priest::pts;

int main() {
    for (int G = 16; G <= 32; G += 16)
        for (int form = 0; form < 3; ++form) {
            const int dims = form == 1 ? 3 : 2, nf = form == 2 ? 7 : 5;
            if (G == 16 && form) continue;
            const int sf = sample_floats(G, dims, nf);
            if (sf % 8 || moved_at(G, dims, nf) % 4 || moved_at(G, dims, nf) + 2 * nf * dims > sf) {
                std::printf("sample block %d %d %d\n", G, dims, nf);
                return 1;
            }
            for (int n_p = 2; n_p <= G * kMaxStrides; ++n_p)
                for (int n_obs = 0; n_obs <= 400; n_obs += 100)
                    for (int warps = 1; warps <= kMaxWarps; ++warps) {
                        const PtsLayout L = pts_layout(G, dims, nf, 11, n_p, n_obs, n_obs - n_obs / 10, warps, warps % 2 ? 0 : warps / 2);
                        if (L.np < n_p || L.np % (2 * G) || L.np > n_p + 2 * G) { std::printf("np %d\n", n_p); return 1; }
                        if (L.rows < size_t(kRows) || L.rows % 8 || L.vrows % 8 || L.node % 8 || L.tv % 8 || L.obs % 8 ||
                            L.obq % 8 || L.mov % 8 || L.grid % 8 || L.warp0 % 8 || L.wsz % 8 || L.xch % 8 || L.fix % 8) {
                            std::printf("alignment %d %d\n", G, n_p);
                            return 1;
                        }
                        const size_t smem = 4 * L.total, fix = 4 * L.total_fix;
                        if (fix - smem != size_t(3) * ((11 - nf + 3) / 4) * L.np * 16) { std::printf("rows %d\n", n_p); return 1; }
                        for (int two = 0; two < 2; ++two) {
                            const size_t got = pts_smem_with_fix(smem, fix, two);
                            if (smem > kSmemCap) continue;  // another tiling or kernel
                            const bool costs = two && smem <= kSmemHalf && fix > kSmemHalf;
                            if (got > kSmemCap || got < (costs || fix > kSmemCap ? smem : fix) ||
                                (two && smem <= kSmemHalf && got > kSmemHalf)) {
                                std::printf("reserved %d %d %d %d\n", G, n_p, n_obs, two);
                                return 1;
                            }
                        }
                    }
        }
    // one sample per warp, 371 obstacles: the rows fit beside the tables
    for (int n_p : {65, 77, 150}) {
        const PtsLayout L = pts_layout(32, 2, 5, 11, n_p, 371, 333, 6, 0);
        if (pts_smem_with_fix(4 * L.total, 4 * L.total_fix, false) != 4 * L.total_fix) { std::printf("not staged %d\n", n_p); return 1; }
    }
    std::puts("ok");
    return 0;
}
"""


def test_fixed_columns_reserved(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = cuda_include()
    if not cxx or not inc:
        pytest.skip("no C++ compiler or CUDA headers")
    src = tmp_path / "pts_layout_check.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "pts_layout_check"
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", INC, "-I", inc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("ok")
