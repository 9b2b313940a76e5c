"""Launch shapes are host arithmetic: a small C++ program asks the library for them, without a GPU."""

import os
import subprocess

from paper_2607_16892_gb300 import build as kbuild

PROGRAM = r"""
#include <cstdio>
#include "kvdro_internal.cuh"
int main() {
    using kvdro::Prec;
    const int R = 1 << 20, K = 4096;  // the largest grid of one regime that the entry points take
    for (Prec p : {Prec::EXACT, Prec::ENVELOPE})
        for (int NL = 1; NL <= 256; NL++)
            for (int E : {1, 64}) {
                const kvdro::GridShape s = kvdro::grid_shape(p, R, NL, E, K, 1, 152);
                if ((long long)K * s.r_blocks > 0x7fffffffLL || (long long)s.rows * s.r_blocks < R || s.smem > 227 * 1024) {
                    std::printf("mode %d, %d lam, %d eps: %d rows, %d blocks, %zu bytes\n", (int)p, NL, E, s.rows, s.r_blocks, s.smem);
                    return 1;
                }
            }
    return 0;
}
"""


def run_program(tmp_path, source):
    lib = os.path.dirname(kbuild.build())
    src, exe = tmp_path / "shapes.cpp", str(tmp_path / "shapes")
    src.write_text(source)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(kbuild.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-I", kbuild.CSRC, "-I", cuda, str(src), "-L", lib, "-lkvdro", f"-Wl,-rpath,{lib}",
                    "-o", exe], check=True)
    return subprocess.run([exe], capture_output=True, text=True)


def test_the_largest_grid_of_one_regime_fits_a_launch(tmp_path):
    """A launch holds at most 2^31 - 1 CTAs: grids of 129 lam values and more, one row to a CTA where that
    fills its warps best, take more rows where 4096 classes x 2^20 reservations need it."""
    out = run_program(tmp_path, PROGRAM)
    assert out.returncode == 0, out.stdout


DUAL = r"""
#include <cstdio>
#include "kvdro_internal.cuh"
int main() {
    const long long most = 0x7fffffffLL * 256;  // cells that the entry point takes
    for (long long cells : {1LL, 127LL, 128LL, 129LL, most / 2 - 127, most / 2, most / 2 + 1, most - 128, most}) {
        const dim3 g = kvdro::dual_grid(cells);
        if (g.x > 0x7fffffffu || g.y > 65535 || g.z != 1 || (long long)g.x * g.y * 128 < cells) {
            std::printf("%lld cells: %u x %u blocks\n", cells, g.x, g.y);
            return 1;
        }
    }
    return 0;
}
"""


def test_the_dual_launch_covers_every_cell_that_the_entry_point_takes(tmp_path):
    """Up to 2^31 - 1 times 256 cells, in blocks of 128."""
    out = run_program(tmp_path, DUAL)
    assert out.returncode == 0, out.stdout
