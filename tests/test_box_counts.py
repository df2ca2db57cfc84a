"""The counts by which the boxes of the resident step wait for one another are 32
bits wide and run on over a context's life: their arithmetic, compiled for the
host with the checks for undefined behaviour, holds across both wraps of 32 bits
(a signed count overflows at 2^31, after 2.7e8 steps of 8 warps).  On the GPU
every context passes 2^31 in its first steps: its counts start just below."""
import os
import subprocess

from paper_1812_00118_gb300 import build as B

SOURCE = r"""
#include <cstdio>
#include "lbm_box.cuh"
using namespace lbm;

int main() {
    const unsigned starts[] = {0u, kBoxFirstCount, 0x7fffffffu, 0x80000000u, 0xfffffff0u, 0xffffffffu};
    for (unsigned first : starts)
        for (int warps : {1, 4, 8})
            for (int step = 1; step < 5000; ++step) {
                const unsigned want = box_count(first, step, warps);
                if (want != (unsigned)(first + (unsigned long long)step * warps)) return 1;
                // a neighbour is at most one step ahead or behind, counted by warps
                for (int d = -2 * warps; d <= 2 * warps; ++d)
                    if (box_reached(want + (unsigned)d, want) != (d >= 0)) return 2;
            }
    const unsigned far = box_count(kBoxFirstCount, 2147483647, 8);   // the longest call
    if (!box_reached(far, far) || box_reached(far - 1, far)) return 3;
    if (kBoxFirstCount >= 0x80000000u || box_count(kBoxFirstCount, 20, 1) < 0x80000000u) return 4;
    std::puts("ok");
    return 0;
}
"""


def test_counts_wrap(tmp_path):
    src, exe = tmp_path / "counts.cu", str(tmp_path / "counts")
    src.write_text(SOURCE)
    subprocess.run([B.nvcc(), *B.ARCH, "-std=c++17", "-w", "-Xcompiler", "-fsanitize=undefined,-fno-sanitize-recover",
                    "-I" + B.INCLUDE, "-I" + B.CSRC, "-o", exe, str(src)], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0 and "ok" in r.stdout, (r.returncode, r.stderr)
