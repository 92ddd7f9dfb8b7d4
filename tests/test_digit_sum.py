"""Integer recombination of the sliced update's eight accumulators
(csrc/digit_sum.h), compiled for the host with signed overflow and invalid
shifts as traps: exact against Python integers over the accumulators' range
(|S_d| <= 40960 K, K <= 64)."""
import os
import subprocess

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2508_04370_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "digit_sum.h"
using namespace ipm::sliced;
static uint32_t biased(int a) {
    const float f = (float)a + 12582912.0f;
    uint32_t u;
    std::memcpy(&u, &f, 4);
    return u;
}
int main() {
    int s[8];
    for (;;) {
        for (int d = 0; d < 8; d++)
            if (std::scanf("%d", &s[d]) != 1) return 0;
        int32_t p[4];
        for (int d = 0; d < 4; d++) p[d] = digit_pair(biased(s[2 * d]), biased(s[2 * d + 1]));
        std::printf("%d %lld\n", p[0], (long long)digit_sum(digit_low(p[2], p[3]), p[0], p[1]));
    }
}
"""


def test_recombination_without_overflow(tmp_path):
    src, exe = tmp_path / "digits.cpp", tmp_path / "digits"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-fsanitize=signed-integer-overflow,shift",
                    "-fsanitize-undefined-trap-on-error", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    top = 40960 * 64
    rng = np.random.default_rng(1)
    rows = [[top] * 8, [-top] * 8, [0] * 8, [top, -top] * 4, [-top, top] * 4, [0, 0, 0, 0, 0, 0, 0, -1]]
    rows += rng.integers(-top, top + 1, size=(2000, 8)).tolist()
    rows += (rng.integers(-2, 3, size=(200, 8))).tolist()
    text = "\n".join(" ".join(map(str, r)) for r in rows)
    run = subprocess.run([str(exe)], input=text, capture_output=True, text=True)
    assert run.returncode == 0, f"the host program stopped with {run.returncode}"
    got = [tuple(map(int, line.split())) for line in run.stdout.splitlines()]
    assert len(got) == len(rows)
    for s, (pair, t) in zip(rows, got):
        assert pair == 128 * s[0] + s[1]
        # T 2^-8 rounded down: digits 0..5 are whole multiples of 2^-8 T's unit
        assert t == sum(v << (7 * (7 - d)) for d, v in enumerate(s)) >> 8
