"""Agent indices of the kernels that give an agent several lanes (no GPU needed).

The index arithmetic is compiled for the host and evaluated around the sizes
where a 32-bit thread number wraps: every agent belongs to exactly the lanes
that the launch gives it.  No kernel forms such an index another way.
"""
import glob
import os
import re
import subprocess

from paper_2008_11578_gb300 import _lib

CSRC = os.path.join(os.path.dirname(_lib.__file__), "csrc")

PROGRAM = r"""
#include <cstdio>
#include "orca_kernels.cuh"
int main() {
    const long long sizes[] = {1, 33, (1ll << 27) - 1, 1ll << 27, (1ll << 27) + 5,
                               (1ll << 30) + 3, (1ll << 31) - 1};
    int bad = 0;
    for (unsigned lanes : {4u, 32u})
        for (unsigned threads : {32u, 64u, 96u, 128u})
            for (long long n : sizes) {
                const long long blocks = (n * lanes + threads - 1) / threads;
                for (long long b : {0ll, blocks / 2, blocks - 1})
                    for (unsigned t = 0; t < threads; ++t) {
                        const long long want = (b * threads + t) / lanes;
                        if (want >= n) continue;   // (past the last agent)
                        bad += orca::lane_group((unsigned)b, threads, t, lanes) != want;
                    }
            }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_lane_group_at_the_wrap(tmp_path):
    src, exe = tmp_path / "lane_groups.cu", tmp_path / "lane_groups"
    src.write_text(PROGRAM)
    subprocess.check_call([_lib._nvcc(), *_lib.ARCH_FLAGS, "-std=c++17", f"-I{CSRC}", str(src),
                           "-o", str(exe)])
    assert subprocess.run([str(exe)], stdout=subprocess.PIPE).stdout.decode().strip() == "0"


def test_no_kernel_divides_a_thread_number():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        assert not re.search(r"blockDim\.x \+ threadIdx\.x\)\s*(>>|/)", text), path
