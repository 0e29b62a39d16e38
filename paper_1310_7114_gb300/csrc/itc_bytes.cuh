// itc_bytes.cuh -- integer arithmetic on the byte rows of an image, free of CUDA types so that it also
// compiles for the host.
#pragma once

#include <stdint.h>

namespace itc {

// The low bits of the N bytes from byte OFF on of the words w: bit i is byte OFF + i.  One 32-bit word
// takes them (N <= 31, so that 1 << N is a value too): each word's 4 bits go to their final place, the
// first OFF of them shifted out, so that no bit passes through a place above 31.
template <int OFF, int N, int NQ>
__host__ __device__ __forceinline__ uint32_t window_bits(const uint32_t (&w)[NQ]) {
    static_assert(OFF >= 0 && OFF < 4 && N <= 31 && 4 * NQ >= OFF + N, "the window lies in the words and fits a word of bits");
    uint32_t m = 0u;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        // the low bits of the 4 bytes in 4 bits (no carries: the 16 partial products land on distinct bits)
        const uint32_t b = ((w[q] & 0x01010101u) * 0x01020408u) >> 24;
        m |= 4 * q >= OFF ? b << (4 * q - OFF) : b >> (OFF - 4 * q);
    }
    return m & ((1u << N) - 1u);
}

// Rows on any boundary are read as the aligned 4-byte words that hold their bytes.  A word may hold bytes of
// the rows around (or the padding between them), but must not reach beyond the image: in row u of H rows of
// W bytes, `pitch` apart, RowRoom has the bytes of the image before and after the row that a word can reach
// (up to 3).  A word that begins at column c (a multiple of 4 bytes from a boundary) is taken whole or not at
// all; row_bytes puts together what is left, the image's first and last bytes.
struct RowRoom {
    int before, after;
    __host__ __device__ __forceinline__ RowRoom(int u, int H, int pitch) {
        const int p = pitch < 3 ? pitch : 3, a = u < 3 ? u : 3, z = H - 1 - u < 3 ? H - 1 - u : 3;
        before = a * p < 3 ? a * p : 3;
        after = z * p < 3 ? z * p : 3;
    }
    __host__ __device__ __forceinline__ bool whole(int c, int W) const { return c >= -before && c < W + after - 3; }
};
// The same test by the word's offset from the image's first byte, for an image of `bytes` bytes in all.
struct ByteSpan {
    unsigned long long last, shift;   // images of less than a word: no offset passes
    __host__ __device__ __forceinline__ explicit ByteSpan(long long bytes)
        : last(bytes < 4 ? 0ull : (unsigned long long)bytes - 4), shift(bytes < 4 ? 1ull << 62 : 0ull) {}
    __host__ __device__ __forceinline__ bool whole_word(long long at) const { return (unsigned long long)at + shift <= last; }
};
// the bytes of columns c to c + 3 of a row that lie in words not taken whole (the others: zeros)
__host__ __device__ __forceinline__ uint32_t row_bytes(const unsigned char* row, int c, int W, const RowRoom& room) {
    uint32_t w = 0u;
#pragma unroll 1
    for (int j = 0; j < 4; ++j)
        if (c + j >= 0 && c + j < W && !room.whole(c + j - (int)(reinterpret_cast<uintptr_t>(row + c + j) & 3), W))
            w |= (uint32_t)row[c + j] << (8 * j);
    return w;
}

}  // namespace itc
