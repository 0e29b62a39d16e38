// itc_pairs.cuh -- the codebook pair sums of Eq. (origupdate), shared by the iterations (itc_run.cu) and the
// backward's codebook kernel (itc_backward.cu):
//   s_k = sum_j g_rho(w_j - w_k),  E_k = sum_j g_rho(w_j - w_k)(w_j - w_k)
#pragma once

#include <type_traits>

#include "itc_internal.cuh"

namespace itc {
namespace {

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// 2^x by the PTX instruction ex2.approx.ftz.f32 (relative error about 2^-22; results below the
// smallest normal float flush to zero, which for the pair kernel means a weight under 1e-38)
__device__ __forceinline__ float ex2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Position of the padding entries past an image's last vector: its weight 2^(-1e38 c) is 0
constexpr float kFar = 1e19f;
// Pair-loop steps whose arithmetic is kept in flight together: kPairU, and half of them for the rest;
// positions are padded to the latter.  (4096 ragged shapes, 50 iterations: 0.426 ms with 8, 0.438
// with 4, 0.470 with 2; one image of M = 128, 100 iterations: 171, 186 and 225 us.)
constexpr int kPairU = 8;
constexpr int kPairPad = kPairU;   // two positions per step

// pair kernel g_rho(d) = exp(-sum_i d_i^2 / (2 rho_i^2)) = 2^(sum_i d_i^2 nc_i), nc_i = -log2(e) /
// (2 rho_i^2); rho = sigma unless the codebook width is set apart.  iso: equal widths in 2-D, where
// the exponent is nc (d0^2 + d1^2): one product fewer per pair, and on the lattice d0^2 + d1^2 is an
// exact integer, rounded once by the product.
template <int ND>
struct PairWidths {
    float nc[3];
    bool iso;
    __device__ __forceinline__ explicit PairWidths(const ImageDesc& Dg) {
#pragma unroll
        for (int i = 0; i < 3; ++i) nc[i] = i < ND ? -(float)(1.4426950408889634 * (double)Dg.pinv2s2[i]) : 0.f;
        iso = ND == 2 && nc[0] == nc[1];
    }
};

// offsets and weights of two positions at once, as packed FP32 operations
template <int ND, bool ISO>
__device__ __forceinline__ float2 pair_weights(const float4 q, const float2 z, const float2 (&nw)[ND], const float (&nc)[3],
                                               float2 (&d)[ND]) {
    d[0] = __fadd2_rn(f2(q.x, q.y), nw[0]);
    d[1] = __fadd2_rn(f2(q.z, q.w), nw[1]);
    float2 x;
    if constexpr (ISO) {
        x = __fmul2_rn(__ffma2_rn(d[1], d[1], __fmul2_rn(d[0], d[0])), f2(nc[0], nc[0]));
    } else {
        x = __fmul2_rn(__fmul2_rn(d[0], d[0]), f2(nc[0], nc[0]));
        x = __ffma2_rn(__fmul2_rn(d[1], d[1]), f2(nc[1], nc[1]), x);
    }
    if constexpr (ND == 3) {
        d[2] = __fadd2_rn(z, nw[2]);
        x = __ffma2_rn(__fmul2_rn(d[2], d[2]), f2(nc[2], nc[2]), x);
    }
    return f2(ex2_ftz(x.x), ex2_ftz(x.y));
}

// Pair sums of one vector over mp positions (a multiple of kPairPad): (x_j, x_j+1, y_j, y_j+1) per
// even j with one 16-byte broadcast load, z by itself; the even j accumulate in the .x halves and
// the odd j in the .y halves.  kPairU steps run side by side: a lone image has one warp per SM
// sub-partition, and one step at a time it waited for its chain of load, exponent and ex2 (74
// clocks a step; the ex2 pipe needs 16).
template <int ND, bool ISO>
__device__ __forceinline__ void pair_sums(const float* sxy, const float* sz, int mp, const float (&w)[ND],
                                          const float (&nc)[3], float& s, float (&E)[ND]) {
    float2 nw[ND], sp = f2(0.f, 0.f), ep[ND];
#pragma unroll
    for (int i = 0; i < ND; ++i) { nw[i] = f2(-w[i], -w[i]); ep[i] = f2(0.f, 0.f); }
    int j = 0;
    auto block = [&](auto steps) {
        constexpr int U = decltype(steps)::value;
        float2 g[U], d[U][ND];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float4 q = *reinterpret_cast<const float4*>(sxy + 2 * (j + 2 * u));
            const float2 z = ND == 3 ? *reinterpret_cast<const float2*>(sz + j + 2 * u) : f2(0.f, 0.f);
            g[u] = pair_weights<ND, ISO>(q, z, nw, nc, d[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            sp = __fadd2_rn(sp, g[u]);
#pragma unroll
            for (int i = 0; i < ND; ++i) ep[i] = __ffma2_rn(g[u], d[u][i], ep[i]);
        }
        j += 2 * U;
    };
#pragma unroll 1
    while (j + 2 * kPairU <= mp) block(std::integral_constant<int, kPairU>());
    if (j < mp) block(std::integral_constant<int, kPairU / 2>());
    s = sp.x + sp.y;
#pragma unroll
    for (int i = 0; i < ND; ++i) E[i] = ep[i].x + ep[i].y;
}

}  // namespace
}  // namespace itc
