"""Index arithmetic of the prefill kernels, compiled for the host: every chunk whose bias or landmark a lane may read for its
position lies inside tensors that hold no more rows than the call's last token needs."""
import subprocess

from paper_2607_02980_b200 import build

PROGRAM = r"""
#include <cstdio>
#include "common.cuh"
using namespace hils;
int main() {
    long wrong = 0, beyond = 0;
    for (int W : {1, 64, 65, 130, 512, 897})
        for (int pos0 = 0; pos0 < 400; ++pos0)
            for (int R : {1, 2, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 1000}) {
                Shape s = {};
                s.pos0 = pos0; s.R = R; s.W = W; s.S = 64;
                const int C = local_lo(pos0 + R - 1, W, 64) / 64;        // the fewest rows that the entry points accept
                for (int tok = R / 64 * 64; tok < (R + 63) / 64 * 64; ++tok) {
                    wrong += local_lo(lane_position(s, tok, R), W, 64) / 64 > C;
                    if (tok < R) wrong += lane_position(s, tok, R) != pos0 + tok;
                    beyond += local_lo(pos0 + tok, W, 64) / 64 > C;
                }
            }
    printf("%ld %ld\n", wrong, beyond);
}
"""


def test_lanes_past_the_last_token_stay_inside_the_tensors(tmp_path):
    src, exe = tmp_path / "lanes.cu", tmp_path / "lanes"
    src.write_text(PROGRAM)
    subprocess.run([build._nvcc(), "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, str(src), "-o", str(exe)], check=True)
    wrong, beyond = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert wrong == 0
    assert beyond > 0, "no case whose tile reaches past the last token's candidates: the test shows nothing"
