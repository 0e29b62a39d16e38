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

}  // namespace itc
