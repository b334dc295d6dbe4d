"""The word by which a running solve reports ||r||^2 to the host: whatever the
bits of ||r||^2, it is told from an empty slot, and its sign bit is the stop
flag alone.  Compiled for the host; no GPU needed."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "internal.h"
using namespace xdcg;
int main() {
    // 0, the least and a common value, infinity; NaNs: quiet, with the sign, with
    // a payload, the empty slot's own bits with and without the sign, signalling
    const unsigned long long bits[] = {0ull, 1ull, 0x3ff0000000000000ull, 0x7ff0000000000000ull,
        0x7ff8000000000000ull, 0xfff8000000000000ull, 0x7fffffffffffffffull,
        0xffffffffffffffffull, kNoReport, kNoReport | kStopBit, 0x7ff0000000000001ull};
    for (unsigned long long b : bits)
        for (int stopped = 0; stopped < 2; ++stopped) {
            const unsigned long long w = report_word(b, stopped != 0);
            const unsigned long long v = w & ~kStopBit;
            const bool nan = (b & ~kStopBit) > 0x7ff0000000000000ull;
            if (w == kNoReport || ((w & kStopBit) != 0) != (stopped != 0) ||
                (nan ? v <= 0x7ff0000000000000ull : v != b)) {
                std::printf("%llx %d -> %llx\n", b, stopped, w);
                return 1;
            }
        }
    return 0;
}
"""


def test_report_word(tmp_path):
    from paper_2111_09294_gb300 import build as b
    src, exe = tmp_path / "word.cu", tmp_path / "word"
    src.write_text(PROGRAM)
    r = subprocess.run([b.nvcc(), "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", b.CSRC,
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
