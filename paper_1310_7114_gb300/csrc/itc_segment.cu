// itc_segment.cu -- segmentation of the data pixels by the codebook (the segments of Figs. 3 and 6).
//
// Every pixel with data (h != 0; in 3-D the voxel (u, v, gray(u, v))) gets the index of the
// codebook vector whose lattice site r_k = round(w_k) gives the largest kernel value
// g_tau(x - r_k), i.e. the smallest
//     D_k(x) = sum_i d_i^2 q_i,   d_i = x_i - r_{k,i},  q_i = 1 / tau_i^2 (rounded once to float),
// evaluated in single precision term by term (each product rounded, the terms added in axis
// order with one rounding each, no fused multiply-add), lowest k on ties; pixels without data
// get -1.
//
// A warp takes 64 x 64 pixel blocks (16 x 64 where there are few) in turn, each on its own (no block-wide barrier after the sites are
// staged): the block's data as bit masks first, one column of each half per lane, so that blocks
// and 16 x 16 tiles without data only write -1.  For the others the codebooks that can win somewhere
// are listed, first for the block and from that list for each tile: with dmin_k / dmax_k the metric
// of the nearest / farthest point of the box, every k with dmin_k <= min_j dmax_j (the same rounded
// arithmetic, which is monotone in each |d_i|, so the bounds hold for every pixel; a list is never empty).  Lists keep k
// order, so the first strict minimum over one is the lowest index on ties.  A lane then takes 8 rows
// of one column: the column's term once per codebook, the rows' terms and sums as packed operations.
// Bound by instruction issue (the bytes take 38 us).  1024 ragged shapes (64 to 512 px a side, M 16 to
// 128, 84 Mpx): 0.67 -> 0.18 ms; before, every 16 x 16 tile listed from the whole codebook, with or
// without data, and each pixel ran through its list in integers.
#include <algorithm>
#include <type_traits>

#include "itc_internal.cuh"

namespace itc {
namespace {

constexpr int kSegBlock = 64;            // block side
constexpr int kSegTile = 16;             // tile side (8 x 32 tiles list 1.4 times the codebooks)
constexpr int kSegRows = kSegTile / 2;   // rows per lane
constexpr int kSegWarps = 4;             // most warps of a CTA
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float site_round(float x, int n) {
    const float r = floorf(x + 0.5f);
    return fminf(fmaxf(r, 0.f), (float)(n - 1));
}

// d^2 q, both products rounded (d is a whole number below 2^24, so d^2 is rounded once)
__device__ __forceinline__ float term(float d, float q) { return __fmul_rn(__fmul_rn(d, d), q); }
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
// Sites and the per-warp lists in shared memory.
struct SegSmem {
    float2* site;             // (r_u, r_v) of every codebook vector
    float* site_g;            // r_g (3-D)
    unsigned short* block;    // this warp's list for its current block, ascending k
    unsigned short* tile;     // and for its current tile
};

// The codebooks of `from` (n of them; null: 0 .. n - 1) that can win in rows u0..u1 and columns v0..v1, in
// order, into `to`; returns their number.  Whole warp.
template <int ND>
__device__ __forceinline__ int list_box(const SegSmem& S, const unsigned short* from, int n, unsigned short* to, int u0,
                                        int u1, int v0, int v1, int G, const float (&q)[3]) {
    const int lane = threadIdx.x & 31;
    const float fu0 = (float)u0, fu1 = (float)u1, fv0 = (float)v0, fv1 = (float)v1, fg1 = (float)(G - 1);
    // the least farthest-point metric bounds the winner at every pixel
    float bound = __int_as_float(0x7f800000);
    for (int i = lane; i < n; i += 32) {
        const int k = from ? from[i] : i;
        const float2 r = S.site[k];
        float m = __fadd_rn(term(fmaxf(fabsf(fu0 - r.x), fabsf(fu1 - r.x)), q[0]),
                            term(fmaxf(fabsf(fv0 - r.y), fabsf(fv1 - r.y)), q[1]));
        if constexpr (ND == 3) m = __fadd_rn(m, term(fmaxf(S.site_g[k], fg1 - S.site_g[k]), q[2]));
        bound = fminf(bound, m);
    }
    for (int o = 16; o > 0; o >>= 1) bound = fminf(bound, __shfl_xor_sync(kFull, bound, o));
    int nl = 0;
    for (int base = 0; base < n; base += 32) {
        const int i = base + lane;
        int k = 0;
        bool hit = false;
        if (i < n) {
            k = from ? from[i] : i;
            const float2 r = S.site[k];
            // (not greater, so that a NaN, an infinite q times 0, stays: at such widths all metrics are
            // infinite or NaN, no comparison holds and the first vector keeps every pixel)
            hit = !(__fadd_rn(term(fmaxf(fmaxf(fu0 - r.x, r.x - fu1), 0.f), q[0]),
                              term(fmaxf(fmaxf(fv0 - r.y, r.y - fv1), 0.f), q[1])) > bound);
        }
        const unsigned bal = __ballot_sync(kFull, hit);
        if (hit) to[nl + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)k;
        nl += __popc(bal);
    }
    __syncwarp();
    return nl;
}

// The blocks (bh rows, 64 or 16) t0, t0 + step, .. of one image.  T: type of the data that says where the image has some.
template <int ND, typename T>
__device__ __forceinline__ void segment_blocks(const ImageDesc& D, const T* data, const SegSmem& S, short* out, int t0,
                                               int step, int bh, const float (&q)[3]) {
    const int lane = threadIdx.x & 31, c = lane & 15, r0 = (lane >> 4) * kSegRows;   // column, first row in a tile
    const int H = D.H, Wd = D.W, G = D.G, pitch = D.pitch, M = D.M;
    const unsigned char* gray = reinterpret_cast<const unsigned char*>(D.data);   // 3-D
    const int blocks_v = (Wd + kSegBlock - 1) / kSegBlock, nblocks = blocks_v * ((H + bh - 1) / bh);
    // up to 32 vectors are a step of the tile's own list, and an image of one tile needs no other
    const bool tile_only = M <= 32 || (H <= kSegTile && Wd <= kSegTile);
    for (int t = t0; t < nblocks; t += step) {
        const int ub = (t / blocks_v) * bh, vb = (t % blocks_v) * kSegBlock;
        // the block's list is made when a tile needs it
        int nb = tile_only ? M : -1;
        const unsigned short* from = tile_only ? nullptr : S.block;
        for (int half = 0; half < 2; ++half) {
            const int vh = vb + 32 * half;
            if (vh >= Wd) break;
            // bit r: data at row ub + r of column vh + lane (16 unconditional loads in flight)
            unsigned mask[2] = {0u, 0u};
            if (data) {
                const T* col = data + min(vh + lane, Wd - 1);
#pragma unroll
                for (int w = 0; w < 2; ++w) {
#pragma unroll
                    for (int p = 0; p < 32; p += 16) {
                        if (32 * w + p >= bh) break;
                        T x[16];
#pragma unroll
                        for (int r = 0; r < 16; ++r) x[r] = __ldg(col + (size_t)min(ub + 32 * w + p + r, H - 1) * pitch);
#pragma unroll
                        for (int r = 0; r < 16; ++r) mask[w] |= x[r] != (T)0 ? 1u << (p + r) : 0u;
                    }
                }
            } else {
                mask[0] = mask[1] = kFull;   // a gray image without weights
            }
            if (vh + lane >= Wd) mask[0] = mask[1] = 0u;
#pragma unroll 1
            for (int s = 0; s < bh / kSegTile * 2; ++s) {
                const int rb = s >> 1, co = (s & 1) * kSegTile;
                const int ut = ub + rb * kSegTile, v0 = vh + co, v = v0 + c, u0 = ut + r0;
                if (ut >= H || v0 >= Wd) continue;
                // this lane's 8 rows of its column, from the lane that holds the column
                const unsigned word = __shfl_sync(kFull, rb < 2 ? mask[0] : mask[1], co + c);
                const int nr = v < Wd ? min(kSegRows, max(0, H - u0)) : 0;
                const unsigned on = (word >> (kSegTile * (rb & 1) + r0)) & ((1u << nr) - 1u);
                short* o = out + (size_t)u0 * Wd + v;
                if (!__any_sync(kFull, on != 0u)) {
#pragma unroll
                    for (int i = 0; i < kSegRows; ++i)
                        if (i < nr) o[(size_t)i * Wd] = -1;
                    continue;
                }
                if (nb < 0)
                    nb = list_box<ND>(S, nullptr, M, S.block, ub, min(ub + bh, H) - 1, vb, min(vb + kSegBlock, Wd) - 1,
                                      G, q);
                // the box of the tile's data: rows and columns with any
                const unsigned rows = __reduce_or_sync(kFull, on << r0), cols2 = __ballot_sync(kFull, on != 0u);
                const unsigned cols = (cols2 | (cols2 >> 16)) & 0xffffu;
                const int nl = list_box<ND>(S, from, nb, S.tile, ut + __ffs(rows) - 1, ut + 31 - __clz(rows),
                                            v0 + __ffs(cols) - 1, v0 + 31 - __clz(cols), G, q);
                float fg[ND == 3 ? kSegRows : 1];
                if constexpr (ND == 3) {
#pragma unroll
                    for (int i = 0; i < kSegRows; ++i)
                        fg[i] = (float)__ldg(gray + (size_t)min(u0 + i, H - 1) * pitch + min(v, Wd - 1));
                }
                float bd[kSegRows];
                int best[kSegRows];
                const int first = S.tile[0];
#pragma unroll
                for (int i = 0; i < kSegRows; ++i) {
                    bd[i] = __int_as_float(0x7f800000);
                    best[i] = first;
                }
                const float fu = (float)u0, fv = (float)v;
#pragma unroll 2
                for (int l = 0; l < nl; ++l) {
                    const int k = S.tile[l];
                    const float2 r = S.site[k];
                    const float tv = term(fv - r.y, q[1]);
                    const float d0 = fu - r.x;
                    float rg = 0.f;
                    if constexpr (ND == 3) rg = S.site_g[k];
#pragma unroll
                    for (int i = 0; i < kSegRows; i += 2) {
                        const float2 d = __fadd2_rn(both(d0), make_float2((float)i, (float)(i + 1)));
                        // the sums one by one: a packed product and a packed sum become a fused
                        // multiply-add, which decides ties between equally near sites the other way
                        float2 m = __fmul2_rn(__fmul2_rn(d, d), both(q[0]));
                        m.x = __fadd_rn(m.x, tv);
                        m.y = __fadd_rn(m.y, tv);
                        if constexpr (ND == 3) {
                            m.x = __fadd_rn(m.x, term(fg[i] - rg, q[2]));
                            m.y = __fadd_rn(m.y, term(fg[i + 1] - rg, q[2]));
                        }
                        best[i] = m.x < bd[i] ? k : best[i];
                        bd[i] = fminf(bd[i], m.x);
                        best[i + 1] = m.y < bd[i + 1] ? k : best[i + 1];
                        bd[i + 1] = fminf(bd[i + 1], m.y);
                    }
                }
#pragma unroll
                for (int i = 0; i < kSegRows; ++i)
                    if (i < nr) o[(size_t)i * Wd] = (on >> i) & 1u ? (short)best[i] : (short)-1;
                __syncwarp();   // the tile list is rewritten
            }
        }
        __syncwarp();   // and the block list
    }
}

// split CTAs per image: their warps share out its blocks.  KIND: the images of the launch, bytes, weights or
// gray (others return).
template <int KIND, int NW>
__global__ void __launch_bounds__(32 * NW, (KIND == kSegGray ? 4 : 5) * kSegWarps / NW) segment_kernel(const __grid_constant__ SegmentLaunch L) {
    const int img = __ldg(L.order + blockIdx.x / L.split), part = blockIdx.x % L.split;
    const ImageDesc& D = L.descs[img];
    constexpr int nd = KIND == kSegGray ? 3 : 2;
    if ((D.ndim == 3 ? kSegGray : (D.dtype == ITC_U8 ? kSegBytes : kSegWeights)) != KIND) return;
    const int M = D.M, tid = threadIdx.x, wid = tid >> 5, nw = NW;
    const int blocks = D.bwd_tiles_u * D.bwd_tiles_v;
    static_assert(kSegBlock == kBwdTileH && kSegBlock == kBwdTileW, "blocks are the backward's tiles");
    // strips of 16 rows where there are few blocks for the image's warps: 770 images of up to 67 px with 8
    // vectors, whose one block would keep one warp, take 16 us instead of 25
    const int step = L.split * nw, bh = blocks < 2 * step ? kSegTile : kSegBlock;
    if (part * nw >= (bh == kSegTile ? D.bwd_tiles_v * ((D.H + kSegTile - 1) / kSegTile) : blocks)) return;
    // q_i = 1 / tau_i^2: the square of the float width in double (exact), one division, one
    // rounding to float
    float q[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) q[i] = i < nd ? (float)(1.0 / ((double)D.sigma[i] * (double)D.sigma[i])) : 0.f;
    extern __shared__ __align__(16) unsigned char ssm[];
    SegSmem S;
    S.site = reinterpret_cast<float2*>(ssm);
    S.site_g = reinterpret_cast<float*>(S.site + M);
    S.block = reinterpret_cast<unsigned short*>(S.site_g + M) + 2 * wid * M;
    S.tile = S.block + M;
    const float* Wk = L.W + D.w_off;
    for (int k = tid; k < M; k += 32 * NW) {
        S.site[k] = make_float2(site_round(Wk[k * nd], D.H), site_round(Wk[k * nd + 1], D.W));
        S.site_g[k] = nd == 3 ? site_round(Wk[k * nd + nd - 1], D.G) : 0.f;
    }
    __syncthreads();
    short* out = L.labels + D.gh_off;
    const int t0 = part * nw + wid;
    if constexpr (KIND == kSegGray) segment_blocks<3, float>(D, D.weight, S, out, t0, step, bh, q);
    else if constexpr (KIND == kSegBytes) segment_blocks<2>(D, reinterpret_cast<const unsigned char*>(D.data), S, out, t0, step, bh, q);
    else segment_blocks<2>(D, reinterpret_cast<const float*>(D.data), S, out, t0, step, bh, q);
}

template <int KIND, int NW>
cudaError_t launch_kind(const SegmentLaunch& L, int B, int max_M, int max_blocks, cudaStream_t s) {
    constexpr size_t per_vector = 3 * sizeof(float) + 2 * NW * sizeof(unsigned short);
    const size_t smem = (size_t)max_M * per_vector;
    cudaError_t e = allow_smem(segment_kernel<KIND, NW>, ITC_MAX_M * per_vector);
    if (e != cudaSuccess) return e;
    // a large image is shared out over several CTAs, eight blocks a warp (four: 5 % slower, more CTAs stage
    // the sites).  A batch that does not fill the GPU (152 SMs, five CTAs each) takes a block a warp, two if
    // that makes many CTAs, and as few as a strip while it leaves SMs without work (300 ragged images 86 ->
    // 64 us, 42 of 500 px with 327 vectors 75 -> 49, one of 300 px 19 -> 7).
    constexpr int nw = NW, slots = 152 * 5;
    auto ctas = [&](int blocks_per_warp) { return (max_blocks + blocks_per_warp * nw - 1) / (blocks_per_warp * nw); };
    SegmentLaunch L2 = L;
    if (B >= slots) L2.split = ctas(8);
    else if ((long long)B * ctas(1) >= 4 * slots) L2.split = ctas(2);
    else L2.split = std::max(ctas(1), std::min((kSegBlock / kSegTile * max_blocks + nw - 1) / nw, slots / B));
    segment_kernel<KIND, NW><<<(unsigned)(B * L2.split), 32 * NW, smem, s>>>(L2);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_segment(const SegmentLaunch& L, int B, int max_M, int max_blocks, int max_H, int max_W, int kinds, cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    static_assert(ITC_MAX_M <= 65535, "16-bit lists");
    // images of one strip: a warp each, three idle ones would keep others off the SM (10000 gray images of 4 to 16
    // px, 64 vectors: 189 us with four warps, 83 with one)
    const bool one = max_H <= kSegTile && max_W <= kSegBlock;
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto kind) {
        constexpr int K = decltype(kind)::value;
        if (e == cudaSuccess && (kinds & (1 << K)))
            e = one ? launch_kind<K, 1>(L, B, max_M, max_blocks, s) : launch_kind<K, kSegWarps>(L, B, max_M, max_blocks, s);
    };
    launch(std::integral_constant<int, kSegBytes>());
    launch(std::integral_constant<int, kSegWeights>());
    launch(std::integral_constant<int, kSegGray>());
    return e;
}

}  // namespace itc
