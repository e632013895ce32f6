"""The chunk of samples that fits into device memory (csrc/chunk.h), with an allocator that runs out."""

import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_14450_gb300", "csrc")
SOURCE = r"""
#include <cstdio>
#include <vector>
#include "chunk.h"
// memory of `room` samples, taken in two parts so that a failure leaves the first one held
static int fit(int want, long room) {
    long held = 0;
    const int c = wd::largest_chunk(
        want,
        [&](int n) {
            for (int part = 0; part < 2; ++part) {
                if (held + n > 2 * room) return false;
                held += n;
            }
            return true;
        },
        [&]() { held = 0; });
    if (held != 2L * c) return -1;
    return c;
}
int main() {
    const int cases[][2] = {{1, 1}, {1, 0}, {4, 9}, {5, 4}, {5, 3}, {65535, 700}, {7, 1}, {7, 0}};
    for (auto& c : cases) std::printf("%d ", fit(c[0], c[1]));
}
"""


def test_chunk_is_halved_until_it_fits(tmp_path):
    (tmp_path / "t.cpp").write_text(SOURCE)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", exe, str(tmp_path / "t.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1", "0", "4", "3", "3", "512", "1", "0"]
