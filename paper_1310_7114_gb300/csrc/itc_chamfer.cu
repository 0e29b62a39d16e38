// itc_chamfer.cu -- the chamfer distance transform that weights the pixels of a binary shape for
// weighted ITC (Sec. 5): T(x) = 3-4 chamfer distance of a foreground pixel to the nearest
// background pixel, the outside of the image counted as background; 0 on the background.
//
// The chamfer distance is a norm, so T is the lesser of the distances to the background in the rows
// at or above a pixel and in the rows at or below it, and a path to a row above can take its row steps first:
//   c(u,j) = min(T(u-1,j-1) + 4, T(u-1,j) + 3, T(u-1,j+1) + 4), 0 on the background
//   T(u,j) = min_k c(u,k) + 3 |j - k|
// from the top row down, and the mirror image from the bottom row up, with frame columns and rows of
// zeros.  Two warps walk an image towards each other, keeping the distances of the rows they pass as
// 16-bit pairs in the first half of the output row; past the middle row each finds the other's
// distances, takes the minimum (any value carried on is the length of some path, so the minimum
// can be carried on too) and overwrites the row with the final floats.
// What bounds it is the chain of H rows of the tallest images (a batch of 1024 gives 13 warps per
// SM), so a row is kept short: lane l holds the C = 4, 8, 16 or 32 columns from l C on in registers, as
// 16-bit pairs of the columns i and i + C/2 (values stay below 3 * 1024 + 4).  Both halves run the
// prefix minimum T(j) = min(c(j), T(j-1) + 3) and the suffix minimum side by side in C/2 packed steps
// each, two warp scans carry the lanes' last values on (+ 3 per column between), and C/2 packed steps
// each add the carries in: integer minima, so the result is that of the sequential raster passes.
// Image and distance rows are copied to shared memory kAhead rows ahead.
// 1024 ragged shapes (64 to 512 px a side, 84 Mpx): 1.50 -> 0.28 ms.  Before, one warp per image walked it
// down and up again, 4 columns of each 128-column chunk per lane in 32 bits, a scan per chunk and the
// previous row in shared memory: about 3000 clocks a row of 512 columns; the same two walks with this row
// layout took 0.34 ms.
#include "itc_bytes.cuh"
#include "itc_internal.cuh"

namespace itc {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kAhead = 8;   // rows copied ahead (a power of two)

__device__ __forceinline__ unsigned pair16(int a) { return (unsigned)a * 0x00010001u; }
// asynchronous copies to shared memory of the first `bytes` of N bytes and zeros, grouped by row
template <int N>
__device__ __forceinline__ void copy_async(unsigned* dst, const void* src, int bytes = N) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(N), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copy_wait_oldest() { asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory"); }
// min(a + b, c) in both 16-bit halves
__device__ __forceinline__ unsigned addmin2(unsigned a, unsigned b, unsigned c) { return __viaddmin_s16x2(a, b, c); }
// bytes i of lo and j of hi, sign bits replicated, as the masks of a 16-bit pair
__device__ __forceinline__ unsigned mask_pair(unsigned lo, unsigned hi, int i, int j) {
    unsigned m;
    const int a = 8 | i, b = 8 | 4 | j;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(m) : "r"(lo), "r"(hi), "r"(a | (a << 4) | (b << 8) | (b << 12)));
    return m;
}
// a value below 2^16 as a float, exactly: the bits of 2^23 + v, minus 2^23
__device__ __forceinline__ float low_float(unsigned p) { return __uint_as_float(__byte_perm(p, 0x4B000000u, 0x7610)) - 8388608.f; }
__device__ __forceinline__ float high_float(unsigned p) { return __uint_as_float(__byte_perm(p, 0x4B000000u, 0x7632)) - 8388608.f; }

// The words of a lane's input bytes (columns from j0 on) that reach beyond the image: in its first and last
// rows, which the two walks start with
__device__ __noinline__ void first_words(unsigned* dst, int nw, const unsigned char* row, int j0, int W, RowRoom room) {
    const int c = j0 - (int)(reinterpret_cast<size_t>(row + j0) & 3);
    for (int q = 0; q <= nw; ++q)
        if (!room.whole(c + 4 * q, W)) dst[q] = row_bytes(row, c + 4 * q, W, room);
}

// The warp's rows of one image with up to 32 C columns.  VEC: rows on vector boundaries.  Rows come
// through a ring in shared memory that each lane fills and reads for itself; copies are unconditional,
// from clamped places, and rows past the image are run through without a store: the loop body has no
// branch.
template <int C, bool VEC>
struct Rows {
    static constexpr int R = C / 2;        // 16-bit pairs per lane: columns i and i + R
    static constexpr int NW = C / 4;       // 4-byte words of the lane's input bytes
    int lane, H, W, pitch, fp, j0;
    const unsigned char* X;
    float* T;
    unsigned* ring;                        // kAhead slots of 32 R words
    bool in;                               // the lane has columns

    __device__ __forceinline__ Rows(const ImageDesc& D, float* out, unsigned* ring_) : ring(ring_) {
        lane = threadIdx.x & 31;
        H = D.H; W = D.W; pitch = D.pitch; fp = D.fpitch;
        j0 = lane * C;
        X = reinterpret_cast<const unsigned char*>(D.data);
        T = out + D.pad_off;
        in = j0 < W;
    }
    __device__ __forceinline__ int inside(int u) const { return min(max(u, 0), H - 1); }
    // the lane's pairs of row u (lanes without columns: the first lane's)
    __device__ __forceinline__ unsigned* pairs_row(int u) const {
        return reinterpret_cast<unsigned*>(T + (size_t)u * fp) + (in ? lane * R : 0);
    }
    // the lane's input bytes of row u to the ring, zeros past W.  Rows without vector alignment: the 4-byte
    // words that hold the bytes, one more than NW, shifted into place when they are read; words that reach
    // beyond the image are left out (first_words)
    __device__ __forceinline__ void copy_in(int u, int t) const {
        const unsigned char* row = X + (size_t)inside(u) * pitch;
        const unsigned char* src = row + (in ? j0 : 0);
        if constexpr (VEC) {
            unsigned* dst = ring + (t & (kAhead - 1)) * 32 * R + lane * NW;
            constexpr int VB = C < 16 ? C : 16;
#pragma unroll
            for (int q = 0; q < NW; q += VB / 4)
                copy_async<VB>(dst + q, src + (j0 + 4 * q < W ? 4 * q : 0), min(max(W - j0 - 4 * q, 0), VB));
        } else {
            unsigned* dst = ring + (t & (kAhead - 1)) * 32 * R + lane * (NW + 1);
            const int off = (int)(reinterpret_cast<size_t>(src) & 3), c = (in ? j0 : 0) - off;
            const unsigned char* word = src - off;
            const RowRoom room(inside(u), H, pitch);
#pragma unroll
            for (int q = 0; q <= NW; ++q) {
                const bool ok = room.whole(c + 4 * q, W);
                copy_async<4>(dst + q, word + (ok ? 4 * q : 0), ok ? 4 : 0);
            }
        }
        copy_commit();
    }
    __device__ __forceinline__ void read_in(int u, int t, unsigned (&w)[NW]) const {
        copy_wait_oldest();
        if constexpr (VEC) {
            const unsigned* src = ring + (t & (kAhead - 1)) * 32 * R + lane * NW;
#pragma unroll
            for (int q = 0; q < NW; ++q) w[q] = src[q];
        } else {
            const unsigned* src = ring + (t & (kAhead - 1)) * 32 * R + lane * (NW + 1);
            const size_t at = reinterpret_cast<size_t>(X) + (size_t)inside(u) * pitch + (in ? j0 : 0);
            const int sh = 8 * (int)(at & 3);
#pragma unroll
            for (int q = 0; q < NW; ++q) w[q] = __funnelshift_r(src[q], src[q + 1], sh);
        }
    }
    // the same for the lane's pairs of row u
    __device__ __forceinline__ void copy_pairs(int u, int t) const {
        unsigned* dst = ring + (t & (kAhead - 1)) * 32 * R + lane * R;
        const unsigned* src = pairs_row(inside(u));
        if constexpr (R >= 4) {
#pragma unroll
            for (int i = 0; i < R; i += 4) copy_async<16>(dst + i, src + i);
        } else {
            copy_async<8>(dst, src);
        }
        copy_commit();
    }
    __device__ __forceinline__ void read_pairs(int t, unsigned (&f)[R]) const {
        copy_wait_oldest();
        const unsigned* src = ring + (t & (kAhead - 1)) * 32 * R + lane * R;
#pragma unroll
        for (int i = 0; i < R; ++i) f[i] = in ? src[i] : 0u;
    }
    // c of a row from the neighbouring row p (the one above or below): left and right columns + 4,
    // the same column + 3; the lanes' edge columns from the next lanes, 0 outside
    __device__ __forceinline__ void neighbours(const unsigned (&p)[R], unsigned (&c)[R]) const {
        unsigned a = __shfl_up_sync(kFull, p[R - 1], 1), b = __shfl_down_sync(kFull, p[0], 1);
        a = lane == 0 ? 0u : a;
        b = lane == 31 ? 0u : b;
        const unsigned first = __byte_perm(a, p[R - 1], 0x5432);   // columns j0 - 1 and j0 + R - 1
        const unsigned last = __byte_perm(p[0], b, 0x5432);        // columns j0 + R and j0 + C
        const unsigned three = pair16(3), four = pair16(4);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const unsigned l = i > 0 ? p[i - 1] : first, r = i < R - 1 ? p[i + 1] : last;
            c[i] = addmin2(p[i], three, addmin2(l, four, __vadd2(r, four)));
        }
    }

    // T of a row from its c: prefix and suffix minima over the whole row
    __device__ __forceinline__ void along_row(const unsigned (&c)[R], unsigned (&p)[R]) const {
        const unsigned three = pair16(3);
        unsigned l[R], r[R];
        l[0] = c[0];
        r[R - 1] = c[R - 1];
#pragma unroll
        for (int i = 1; i < R; ++i) {
            l[i] = addmin2(l[i - 1], three, c[i]);
            r[R - 1 - i] = addmin2(r[R - i], three, c[R - 1 - i]);
        }
        // the lane's last (first) column, carried over the lanes, 3 per column, from the frame's zeros
        const int ll = (int)(l[R - 1] & 0xffffu), lh = (int)(l[R - 1] >> 16);
        const int rl = (int)(r[0] & 0xffffu), rh = (int)(r[0] >> 16);
        int tl = min(lh, ll + 3 * R), tr = min(rl, rh + 3 * R);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {   // a lane without a source gets its own value back: no effect
            tl = min(tl, __shfl_up_sync(kFull, tl, o) + 3 * C * o);
            tr = min(tr, __shfl_down_sync(kFull, tr, o) + 3 * C * o);
        }
        const int bl = __shfl_up_sync(kFull, tl, 1), br = __shfl_down_sync(kFull, tr, 1);
        const int cl = lane == 0 ? 0 : min(bl, 3 * C * lane), cr = lane == 31 ? 0 : min(br, 3 * C * (31 - lane));
        const unsigned kl = (unsigned)cl | ((unsigned)min(ll, cl + 3 * R) << 16);
        const unsigned kr = (unsigned)min(rh, cr + 3 * R) | ((unsigned)cr << 16);
#pragma unroll
        for (int i = 0; i < R; ++i)
            p[i] = __vmins2(addmin2(kl, pair16(3 * (i + 1)), l[i]), addmin2(kr, pair16(3 * (R - i)), r[i]));
    }

    // The walk of one warp: down (rows 0, 1, ..) or up (rows H - 1, H - 2, ..), to the image's middle row
    // and then through the other warp's half.
    __device__ __forceinline__ void walk(bool down) const {
        const int mid = H / 2, own = down ? mid : H - mid;   // rows this warp reaches first
        auto row = [&](int t) { return down ? t : H - 1 - t; };
        unsigned valid[NW];   // 0x80 in the bytes of the lane's columns inside the image
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            valid[q] = 0u;
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (j0 + 4 * q + t < W) valid[q] |= 0x80u << (8 * t);
        }
        unsigned p[R];
#pragma unroll
        for (int i = 0; i < R; ++i) p[i] = 0u;   // the frame row
        for (int t = 0; t < kAhead; ++t) copy_in(row(t), t);
        if constexpr (!VEC) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            for (int t = 0; t < min(own, pitch < 3 ? 3 : 1) && in; ++t)
                first_words(ring + t * 32 * R + lane * (NW + 1), NW, X + (size_t)row(t) * pitch, j0, W, RowRoom(row(t), H, pitch));
        }
#pragma unroll 2
        for (int t = 0; t < own; ++t) {
            unsigned on[NW], c[R];
            read_in(row(t), t, on);
#pragma unroll
            for (int q = 0; q < NW; ++q)   // 0x80 in the bytes of foreground columns
                on[q] = (((on[q] & 0x7f7f7f7fu) + 0x7f7f7f7fu) | on[q]) & valid[q];
            copy_in(row(t + kAhead), t);   // into the slot just read
            neighbours(p, c);
#pragma unroll
            for (int i = 0; i < R; ++i) c[i] &= mask_pair(on[i / 4], on[(i + R) / 4], i & 3, (i + R) & 3);
            along_row(c, p);
            if (in) store_pairs(pairs_row(row(t)), p);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");   // the ring is filled anew
        __syncthreads();                                   // the other warp's half is there
        for (int t = own; t < own + kAhead; ++t) copy_pairs(row(t), t);
#pragma unroll 2
        for (int t = own; t < H; ++t) {
            unsigned f[R], c[R];
            read_pairs(t, f);
            copy_pairs(row(t + kAhead), t);
            neighbours(p, c);
#pragma unroll
            for (int i = 0; i < R; ++i) c[i] = __vmins2(c[i], f[i]);   // 0 on the background
            along_row(c, p);
            // every lane has used its pairs of this row (the shuffles came after), so the row can be
            // overwritten
            store_floats(T + (size_t)row(t) * fp + j0, p);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }

    __device__ __forceinline__ void store_pairs(unsigned* o, const unsigned (&p)[R]) const {
        if constexpr (R >= 4) {
#pragma unroll
            for (int i = 0; i < R; i += 4) *reinterpret_cast<uint4*>(o + i) = make_uint4(p[i], p[i + 1], p[i + 2], p[i + 3]);
        } else {
            *reinterpret_cast<uint2*>(o) = make_uint2(p[0], p[1]);
        }
    }
    __device__ __forceinline__ void store_floats(float* o, const unsigned (&p)[R]) const {
        float v[C];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            v[i] = low_float(p[i]);
            v[i + R] = high_float(p[i]);
        }
        if (j0 + C <= W) {
#pragma unroll
            for (int i = 0; i < C; i += 4) *reinterpret_cast<float4*>(o + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        } else {
#pragma unroll
            for (int i = 0; i < C; ++i)
                if (j0 + i < W) o[i] = v[i];
        }
    }
};

// An image of one column: the frame lies beside every pixel (the walks' pairs would take two columns of the row)
__device__ __noinline__ void one_column(const ImageDesc& D, float* out) {
    const unsigned char* X = reinterpret_cast<const unsigned char*>(D.data);
    for (int u = threadIdx.x; u < D.H; u += blockDim.x) out[D.pad_off + (size_t)u * D.fpitch] = X[(size_t)u * D.pitch] ? 3.f : 0.f;
}

template <int C>
__device__ __forceinline__ void run_rows(const ImageDesc& D, float* out, unsigned* ring) {
    constexpr int VB = C < 16 ? C : 16;   // bytes per vector load
    if (((reinterpret_cast<size_t>(D.data) | (size_t)D.pitch) & (VB - 1)) == 0) Rows<C, true>(D, out, ring).walk(threadIdx.x < 32);
    else Rows<C, false>(D, out, ring).walk(threadIdx.x < 32);
}

// A CTA of two warps per image, so that the images spread evenly over the SMs.
template <int CMAX>
__global__ void __launch_bounds__(64) chamfer_kernel(const __grid_constant__ ChamferLaunch L) {
    const ImageDesc& D = L.descs[__ldg(L.order + blockIdx.x)];
    const int W = D.W;
    __shared__ __align__(16) unsigned rings[2][kAhead * 32 * (CMAX / 2)];
    unsigned* ring = rings[threadIdx.x >> 5];
    if (W == 1) one_column(D, L.out);
    else if (W <= 128) run_rows<4>(D, L.out, ring);
    else if (W <= 256) { if constexpr (CMAX >= 8) run_rows<8>(D, L.out, ring); }
    else if (W <= 512) { if constexpr (CMAX >= 16) run_rows<16>(D, L.out, ring); }
    else { if constexpr (CMAX >= 32) run_rows<32>(D, L.out, ring); }
}

}  // namespace

cudaError_t launch_chamfer(const ChamferLaunch& L, int max_W, cudaStream_t s) {
    if (L.B <= 0) return cudaSuccess;
    static_assert(kChamferMaxW == 32 * 32, "the widest rows: 32 columns per lane");
    if (max_W <= 128) chamfer_kernel<4><<<(unsigned)L.B, 64, 0, s>>>(L);
    else if (max_W <= 256) chamfer_kernel<8><<<(unsigned)L.B, 64, 0, s>>>(L);
    else if (max_W <= 512) chamfer_kernel<16><<<(unsigned)L.B, 64, 0, s>>>(L);
    else chamfer_kernel<32><<<(unsigned)L.B, 64, 0, s>>>(L);
    return cudaGetLastError();
}

}  // namespace itc
