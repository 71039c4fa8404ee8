"""The loss kernels' scratch holds what they write on any GPU: two partials a
block, or one a block and the image loss's last sums after them.  A GPU with
few SMs (a partition of one) runs few blocks."""
import os
import subprocess

from paper_2510_26358_gb300 import build as B

PROGRAM = r"""
#include "gs_internal.cuh"
#include <cstdio>
int main() {
    for (int sms = 1; sms <= 512; ++sms)
        std::printf("%d %lld\n", sms, (long long)gs::red_part_count(2 * sms));
    std::printf("%d\n", gs::kImageLossSlices);
}
"""


def test_scratch_holds_every_block_and_slice(tmp_path):
    src, exe = tmp_path / "count.cu", tmp_path / "count"
    src.write_text(PROGRAM)
    subprocess.run([B.nvcc(), "-std=c++17", "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"), "-o", str(exe), str(src)],
                   check=True, capture_output=True, text=True)
    *rows, slices = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()
    for row in rows:
        sms, count = map(int, row.split())
        blocks = 2 * sms
        assert count >= 2 * blocks and count >= blocks + 2 * int(slices), row
