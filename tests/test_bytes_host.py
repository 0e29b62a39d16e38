"""The integer arithmetic on byte rows (csrc/itc_bytes.cuh), compiled for the host with the undefined-
behaviour checks of the compiler on."""
import os
import subprocess

import pytest

from paper_1310_7114_gb300 import build as itc_build

HEAD = """
#define __host__
#define __device__
#define __forceinline__ inline
#include "itc_bytes.cuh"
#include <stdio.h>
#include <string.h>
"""


def run_host(tmp_path, source):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(HEAD + source)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-Wno-unknown-pragmas",
                    "-I", itc_build.CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True)


@pytest.mark.parametrize("R", range(3, 14))
def test_window_bits(tmp_path, R):
    """Every run of ones and of zeros in a row pass window of 4 + 2 R inputs, the bytes around the window
    of either value: bit i is input i."""
    r = run_host(tmp_path, """
int main() {
    constexpr int R = %d, OFF = (16 - R) & 3, N = 4 + 2 * R, NQ = (OFF + N + 3) / 4;
    for (int a = 0; a <= N; ++a)
        for (int b = a; b <= N; ++b)
            for (int flip = 0; flip < 4; ++flip) {
                unsigned char row[4 * NQ];
                uint32_t want = 0, w[NQ];
                for (int i = 0; i < 4 * NQ; ++i) {
                    const int k = i - OFF;
                    const int x = k < 0 || k >= N ? flip >> 1 : ((k >= a && k < b) ? 1 : 0) ^ (flip & 1);
                    row[i] = (unsigned char)x;
                    if (k >= 0 && k < N && x) want |= 1u << k;
                }
                memcpy(w, row, sizeof(w));
                const uint32_t got = itc::window_bits<OFF, N>(w);
                if (got != want) { printf("R %%d run [%%d, %%d) flip %%d: %%08x, not %%08x\\n", R, a, b, flip, got, want); return 1; }
            }
    return 0;
}
""" % R)
    assert r.returncode == 0, r.stdout + r.stderr
