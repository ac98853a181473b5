"""The grid barrier's arrival count over its wrap at 2^32 (host code, no GPU): max_iter
and fixed_iters go up to 2^24 iterations a step, with up to three barriers of several
hundred blocks each."""
import os
import subprocess

from paper_1904_00861_gb300 import build

SRC = r"""
#include <cstdio>
#include "grid_barrier.cuh"
int main()
{
    using dtsph::barrier_reached;
    const unsigned int grid = 456;
    const unsigned long long half = (1ull << 31) / grid, wrap = (1ull << 32) / grid;
    for (unsigned long long epoch : {1ull, 2ull, half, half + 1, wrap - 1, wrap, wrap + 1, wrap + 2, 3ull << 24}) {
        const unsigned int target = (unsigned int)(epoch * grid);
        // from all blocks of the barrier before to all of the one after
        for (long long a = (long long)((epoch - 1) * grid); a <= (long long)((epoch + 1) * grid); ++a)
            if (barrier_reached((unsigned int)a, target) != (a >= (long long)(epoch * grid))) {
                printf("epoch %llu arrivals %lld\n", epoch, a);
                return 1;
            }
    }
    return 0;
}
"""


def test_arrival_count_wraps(tmp_path):
    src, exe = tmp_path / "count.cu", tmp_path / "count"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I" + build.CSRC, "-I" + os.path.join(build.ROOT, "include"),
                    str(src), "-o", str(exe)], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
