"""Default block sizes on the host: a launch of any length a 256-thread block can take fits a grid of
2^31 - 1 blocks, in FP64 too, whose blocks are a warp otherwise."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_15632_gb300", "csrc")
COUNTS = [1, 31, 4096, 1 << 26, (1 << 36) - 32, (1 << 36) - 31, 1 << 36, 1 << 37, (1 << 38) + 1, (1 << 39) - 256]


def test_every_launch_fits_a_grid(tmp_path):
    src, exe = tmp_path / "block.cpp", tmp_path / "block"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "qmcrt_block.h"\n'
                   'int main(int c, char **v) { for (int i = 1; i < c; ++i) for (int d = 0; d < 2; ++d) '
                   'std::printf("%d\\n", qmcrt::default_block(std::strtoull(v[i], nullptr, 10), d)); }\n')
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)])
    out = subprocess.check_output([str(exe)] + [str(n) for n in COUNTS], text=True).split()
    for n, f32, f64 in zip(COUNTS, map(int, out[::2]), map(int, out[1::2])):
        for b in (f32, f64):
            assert b in (32, 64, 128, 256)
            assert (n + b - 1) // b <= 0x7fffffff
    assert out[7] == "32"  # 2^26 FP64 packets: still a warp a block
