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


@pytest.mark.parametrize("W,pitch", [(1, 1), (1, 2), (2, 2), (1, 3), (3, 3), (4, 4), (5, 5), (5, 7), (9, 9), (37, 37), (61, 64), (131, 133)])
def test_row_words(tmp_path, W, pitch):
    """The words of every row of a byte image on each of the four boundaries, as the kernels take them: whole
    words inside the image, the bytes that those leave out by themselves; every byte once, and no read
    outside the image."""
    r = run_host(tmp_path, """
int main() {
    const int W = %d, pitch = %d;
    alignas(16) unsigned char mem[4096];
    for (int i = 0; i < 4096; ++i) mem[i] = (unsigned char)(i * 37 + 11) | 1;
    for (int H = 1; H <= 9; ++H)
        for (int shift = 0; shift < 4; ++shift) {
            const unsigned char *data = mem + 64 + shift, *end = data + (H - 1) * pitch + W;
            for (int u = -9; u < H + 9; ++u) {   // rows above and below the image: nothing
                const unsigned char* row = data + u * pitch;
                if (u >= 0 && u < H) continue;
                for (int c = -((int)((uintptr_t)row & 3)) - 4; c < W; c += 4)
                    if (c + 3 >= 0 && itc::ByteSpan((H - 1) * pitch + W).whole_word((long long)u * pitch + c)) { printf("row %%d\\n", u); return 1; }
            }
            for (int u = 0; u < H; ++u) {
                const itc::RowRoom room(u, H, pitch);
                const unsigned char* row = data + u * pitch;
                const int off = (int)((uintptr_t)row & 3);
                for (int c = -off - 8; c < W + 12; c += 4) {   // words
                    const bool whole = room.whole(c, W);
                    if (whole != (c + 3 >= 0 && c < W && itc::ByteSpan((H - 1) * pitch + W).whole_word((long long)u * pitch + c))) { printf("by offset\\n"); return 1; }
                    if (whole && (row + c < data || row + c + 4 > end)) { printf("H %%d boundary %%d row %%d word %%d: outside\\n", H, shift, u, c); return 1; }
                    if (whole && (c + 3 < 0 || c >= W)) { printf("word without a byte of the row\\n"); return 1; }
                }
                for (int c = -8; c < W + 12; ++c) {
                    const uint32_t b = itc::row_bytes(row, c, W, room);
                    for (int j = 0; j < 4; ++j) {
                        const int k = c + j;
                        const bool in = k >= 0 && k < W, whole = room.whole(k - (int)((uintptr_t)(row + k) & 3), W);
                        const int want = in && !whole ? row[k] : 0;
                        if ((int)((b >> (8 * j)) & 255) != want) { printf("H %%d boundary %%d row %%d column %%d\\n", H, shift, u, k); return 1; }
                    }
                }
            }
        }
    return 0;
}
""" % (W, pitch))
    assert r.returncode == 0, r.stdout + r.stderr
