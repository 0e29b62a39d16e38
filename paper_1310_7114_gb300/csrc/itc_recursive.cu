// itc_recursive.cu -- 2-D fields for large widths by recursive filtering (Sec. 3.1 points to
// recursive filters, citing Deriche 1992): the cost per pixel does not grow with sigma.
//
// Deriche's recursive Gaussian fits the kernel by two damped sinusoids,
//     exp(-x^2/2) ~ sum_t Re(c_t exp((-b_t + i omega_t) x)),  x >= 0,
// so with z_t = exp((-b_t + i omega_t) / sigma) the sampled kernel is g(j) ~ Re sum_t c_t z_t^j and
// a convolution along one axis is four first-order complex recursions per signal:
//   causal       s0[n] = x[n] + z s0[n-1],          s1[n] = z (s1[n-1] + s0[n-1])
//   anticausal   r0[n] = z (r0[n+1] + x[n+1]),      r1[n] = z (r1[n+1] + r0[n+1] + x[n+1])
//   g * x  = Re sum_t c_t (s0 + r0),     (d g) * x = Re sum_t c_t (r1 - s1)     (d = offset)
// with zero states at the ends (no data outside the image), so the kernel is untruncated.
//
// Lines of up to kRecMaxLine samples (rec_rows_scan, rec_cols_scan): a warp filters a line that lies in
// shared memory, each lane a contiguous segment of it.  The recursions are linear, so a segment's
// state is its own (from zero) plus the incoming state times a power of z:
//   s0' = z^n s0 + b0,   s1' = z^n s1 + n z^n s0 + b1
// Every lane runs its segment from zero for (b0, b1) of both directions, two warp scans carry the
// states across the lanes (powers z^(L 2^k) from the plan), and a second run writes the outputs.
// A line thus takes 4 L steps of a chain instead of 2 n, for 1.7 times the arithmetic.  A warp takes two
// neighbouring lines at once as the halves of packed FP32 operations.  Pass along v: lines are image
// rows, T = g_v * h, T_v = (d g)_v * h into two scratch planes.  Pass along u: a CTA takes 8 columns
// (32-byte row pieces of the planes), A = g_u * T and F_u = (d g)_u * T, in a launch of its own
// F_v = g_u * T_v; its h A sum is one S_XX partial (FP32 over 8 products, then FP64 in a fixed order).
// What bounds it now is the memory round trips between a CTA's phases (8 to 12 warps per SM at 101 KB
// of shared memory for 1024 samples): all loads of a phase are in flight together.
// 48 images of 128 to 1024 px a side (15 Mpx), microseconds, before and now: along v 431 and 102, along u
// 694 and 245, the self-overlap pass 361 and 60, 567 and 105.
//
// Longer lines, and small images where a batch has lines enough to fill the GPU (rec_seq_side in itc_api.cu),
// take one sequential recursion per row and column (rec_rows_kernel, rec_cols_kernel):
// along v one lane per row, rows staged through shared memory in 32 x 32 tiles, the causal part
// stored and the anticausal part added; along u one thread per column, 128 columns per CTA, rows in
// prefetched chunks, one S_XX partial per 32 columns.
// The self-overlap pass (mode 1) computes A alone into the A_s plane with one scratch plane.
#include "itc_internal.cuh"

namespace itc {
namespace {

struct Cplx {
    float r, i;
};
__device__ __forceinline__ Cplx cmul(Cplx a, Cplx b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }
__device__ __forceinline__ Cplx cadd(Cplx a, Cplx b) { return {a.r + b.r, a.i + b.i}; }
__device__ __forceinline__ float re_mul(Cplx c, Cplx s) { return c.r * s.r - c.i * s.i; }

// the image of the CTA: list entry blockIdx.x (blockIdx.y picks the CTA's block of rows or columns within it)
__device__ __forceinline__ const ImageDesc& rec_image(const RecursiveLaunch& L) {
    return L.descs[__ldg(L.img_list + blockIdx.x)];
}

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// A complex number for each of two neighbouring lines, in packed halves.
struct Cplx2 {
    float2 r, i;
};
__device__ __forceinline__ float2 both(float a) { return f2(a, a); }
// z s and z s + t, one z for both lines
__device__ __forceinline__ Cplx2 cmul2(const Cplx& z, const Cplx2& s) {
    return {__ffma2_rn(both(z.r), s.r, __fmul2_rn(both(-z.i), s.i)), __ffma2_rn(both(z.r), s.i, __fmul2_rn(both(z.i), s.r))};
}
__device__ __forceinline__ Cplx2 cfma2(const Cplx& z, const Cplx2& s, const Cplx2& t) {
    return {__ffma2_rn(both(z.r), s.r, __ffma2_rn(both(-z.i), s.i, t.r)),
            __ffma2_rn(both(z.r), s.i, __ffma2_rn(both(z.i), s.r, t.i))};
}
template <bool UP>
__device__ __forceinline__ float shfl_by(float v, int o) {
    return UP ? __shfl_up_sync(0xffffffffu, v, o) : __shfl_down_sync(0xffffffffu, v, o);
}
template <bool UP>
__device__ __forceinline__ Cplx2 shfl_by(const Cplx2& s, int o) {
    return {f2(shfl_by<UP>(s.r.x, o), shfl_by<UP>(s.r.y, o)), f2(shfl_by<UP>(s.i.x, o), shfl_by<UP>(s.i.y, o))};
}

// One axis of the recursion: z, the weights and z^(seg 2^k) of both terms.
struct RecAxis {
    Cplx z[2], c[2], zp[2][5];
    __device__ __forceinline__ RecAxis(const RecCoef& rc, int a) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            z[t] = {rc.zr[a][t], rc.zi[a][t]};
            c[t] = {rc.cr[t], rc.ci[t]};
#pragma unroll
            for (int k = 0; k < 5; ++k) zp[t][k] = {rc.pr[a][t][k], rc.pi[a][t][k]};
        }
    }
};

// States of the two terms: s0 (and, MOM, s1) of one direction.
template <bool MOM>
struct RecState {
    Cplx2 s0[2], s1[MOM ? 2 : 1];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            s0[t] = {f2(0.f, 0.f), f2(0.f, 0.f)};
            s1[MOM ? t : 0] = s0[t];
        }
    }
    // s1' = z s1 + z s0, s0' = z s0 + x: the state after sample x
    __device__ __forceinline__ void causal(const RecAxis& A, float2 x) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const Cplx2 p = cmul2(A.z[t], s0[t]);
            if constexpr (MOM) s1[t] = cfma2(A.z[t], s1[t], p);
            s0[t] = {__fadd2_rn(p.r, x), p.i};
        }
    }
    // r0' = z (r0 + x), r1' = z r1 + r0': the state one place to the left of sample x
    __device__ __forceinline__ void anticausal(const RecAxis& A, float2 x) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            s0[t] = cmul2(A.z[t], Cplx2{__fadd2_rn(s0[t].r, x), s0[t].i});
            if constexpr (MOM) s1[t] = cfma2(A.z[t], s1[t], s0[t]);
        }
    }
    // acc + sign Re sum_t c_t s_t
    static __device__ __forceinline__ float2 weigh(const RecAxis& A, const Cplx2* s, float sign, float2 acc) {
#pragma unroll
        for (int t = 0; t < 2; ++t)
            acc = __ffma2_rn(both(sign * A.c[t].r), s[t].r, __ffma2_rn(both(-sign * A.c[t].i), s[t].i, acc));
        return acc;
    }
    // the lanes' own states (from zero) become the states that enter their segments: inclusive scan,
    // then one lane on.  UP: from the lower lanes (causal)
    template <bool UP>
    __device__ __forceinline__ void scan(const RecAxis& A, int seg) {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const int o = 1 << k;
            const float2 n = both((float)(seg * o));
            const bool from = UP ? lane >= o : lane + o < 32;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const Cplx zp = {from ? A.zp[t][k].r : 0.f, from ? A.zp[t][k].i : 0.f};   // 0: no lane there
                const Cplx2 p = cmul2(zp, shfl_by<UP>(s0[t], o));
                if constexpr (MOM) {
                    s1[t] = cfma2(zp, shfl_by<UP>(s1[t], o), s1[t]);
                    s1[t] = {__ffma2_rn(n, p.r, s1[t].r), __ffma2_rn(n, p.i, s1[t].i)};
                }
                s0[t] = {__fadd2_rn(s0[t].r, p.r), __fadd2_rn(s0[t].i, p.i)};
            }
        }
        const bool none = UP ? lane == 0 : lane == 31;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            s0[t] = shfl_by<UP>(s0[t], 1);
            if constexpr (MOM) s1[t] = shfl_by<UP>(s1[t], 1);
        }
        if (none) clear();
    }
};

// The whole warp filters the two lines in x: seg samples per lane (zeros past the lines' end), lane
// l's at x + l * str, str odd.  o0 = g * x and (MOM) o1 = (d g) * x in the same layout.
template <bool MOM>
__device__ __forceinline__ void filter_lines(const RecAxis& A, const float2* x, float2* o0, float2* o1, int seg, int str) {
    const int lane = threadIdx.x & 31;
    x += lane * str;
    o0 += lane * str;
    o1 += lane * str;
    RecState<MOM> s, r;
    s.clear();
    r.clear();
    // (1) each segment from zero, both directions side by side
#pragma unroll 2
    for (int j = 0; j < seg; ++j) {
        s.causal(A, x[j]);
        r.anticausal(A, x[seg - 1 - j]);
    }
    // (2) states across the lanes
    s.template scan<true>(A, seg);
    r.template scan<false>(A, seg);
    // (3) the outputs: the causal part, then the anticausal part added
    const float2 zero = f2(0.f, 0.f);
#pragma unroll 4
    for (int j = 0; j < seg; ++j) {
        s.causal(A, x[j]);
        o0[j] = s.weigh(A, s.s0, 1.f, zero);
        if constexpr (MOM) o1[j] = s.weigh(A, s.s1, -1.f, zero);
    }
#pragma unroll 4
    for (int j = seg - 1; j >= 0; --j) {
        o0[j] = r.weigh(A, r.s0, 1.f, o0[j]);
        if constexpr (MOM) o1[j] = r.weigh(A, r.s1, 1.f, o1[j]);
        r.anticausal(A, x[j]);
    }
}

// Place of sample i of a line pair in its shared-memory layout, for i advancing by 32.
struct LineAt {
    int seg, str, q, r, dq, dr;
    __device__ __forceinline__ LineAt(int i, int seg_)
        : seg(seg_), str(seg_ | 1), q(i / seg_), r(i % seg_), dq(32 / seg_), dr(32 % seg_) {}
    __device__ __forceinline__ int at() const { return q * str + r; }
    __device__ __forceinline__ void next() {
        q += dq;
        r += dr;
        if (r >= seg) { r -= seg; ++q; }
    }
};

template <bool MOM>
__global__ void __launch_bounds__(32 * kRecPairs) rec_rows_scan(const __grid_constant__ RecursiveLaunch L, int nblk) {
    const ImageDesc& D = L.descs[__ldg(L.img_list + blockIdx.x / nblk)];
    const int H = D.H, W = D.W, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int u = (blockIdx.x % nblk) * kRecLines + 2 * wid;
    if (u >= H) return;   // no block-wide barrier below
    const int seg = (W + 31) / 32, str = seg | 1;
    const bool two = u + 1 < H;
    const RecAxis ax(MOM ? D.rc : D.rc_self, 1);
    extern __shared__ __align__(16) float2 rsm2[];
    float2* x = rsm2 + wid * rec_pair_floats2(W, MOM ? 3 : 2);
    float2 *o0 = x + 32 * str, *o1 = MOM ? o0 + 32 * str : o0;
    {
        LineAt p(lane, seg);
        const size_t second = two ? (size_t)D.pitch : 0;   // one row: filtered twice, written once
        // one loop per type, its 32 loads unconditional and in flight together (a type test or a
        // bounds branch between them would put one memory round trip after another)
        auto stage = [&](auto* row) {
            for (int t = 0; t < seg; t += 16) {
                float2 h[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const int v = min(32 * (t + q) + lane, W - 1);
                    h[q] = f2((float)__ldg(row + v), (float)__ldg(row + second + v));
                }
#pragma unroll
                for (int q = 0; q < 16; ++q)
                    if (t + q < seg) {
                        x[p.at()] = 32 * (t + q) + lane < W ? h[q] : f2(0.f, 0.f);
                        p.next();
                    }
            }
        };
        if (D.dtype == ITC_U8) stage(reinterpret_cast<const unsigned char*>(D.data) + (size_t)u * D.pitch);
        else stage(reinterpret_cast<const float*>(D.data) + (size_t)u * D.pitch);
    }
    __syncwarp();
    filter_lines<MOM>(ax, x, o0, o1, seg, str);
    __syncwarp();
    float* P0 = L.fields + (MOM ? D.field_off + 3 * D.plane_floats : D.self_off + D.plane_floats) + (size_t)u * D.fpitch;
    float* P1 = P0 + D.plane_floats;   // T_v (moments only)
    const int fp = D.fpitch;
    LineAt p(lane, seg);
#pragma unroll 4
    for (int t = 0; t < seg; ++t, p.next()) {
        const int v = 32 * t + lane;
        if (v < W) {
            const float2 a = o0[p.at()];
            P0[v] = a.x;
            if (two) P0[fp + v] = a.y;
            if constexpr (MOM) {
                const float2 m = o1[p.at()];
                P1[v] = m.x;
                if (two) P1[fp + v] = m.y;
            }
        }
    }
}

// PART 0: A and F_u from T; 1: F_v from T_v; 2: A_s (self-overlap pass).  0 and 2 with the S_XX share.
template <int PART>
__global__ void __launch_bounds__(32 * kRecPairs) rec_cols_scan(const __grid_constant__ RecursiveLaunch L, int nblk) {
    constexpr bool MOM = PART == 0;
    const ImageDesc& D = L.descs[__ldg(L.img_list + blockIdx.x / nblk)];
    const int H = D.H, W = D.W, fp = D.fpitch, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int blk = blockIdx.x % nblk, v0 = blk * kRecLines;
    if (v0 >= W) return;
    const int seg = (H + 31) / 32, str = seg | 1, ls = rec_pair_floats2(H, MOM ? 3 : 2);
    extern __shared__ __align__(16) float2 rsm2[];
    __shared__ double red[kRecPairs];
    const long long pl = D.plane_floats;
    const float* T = L.fields + (PART == 2 ? D.self_off + pl : D.field_off + (3 + PART) * pl);
    float* A = L.fields + (PART == 2 ? D.self_off : D.field_off + 2 * PART * pl);
    // when the CTA moves columns between global and shared memory: this thread's column pair and
    // first row (a warp moves 8 row pieces of 32 bytes)
    const int c = tid & (kRecPairs - 1), r0 = tid / kRecPairs, v = v0 + 2 * c;
    static_assert(32 * kRecPairs / kRecPairs == 32, "LineAt advances by 32 rows");
    const bool in = v < W, in2 = v + 1 < W;
    float2* const xc = rsm2 + c * ls;                // the arrays of this thread's column pair
    float2* const xw = rsm2 + wid * ls;              // and of this warp's
    {
        LineAt p(r0, seg);
        for (int t = 0; t < seg; ++t, p.next()) {   // copies of 8 bytes, zeros outside the image
            const int u = 32 * t + r0;
            const bool ok = in && u < H;
            const float* src = ok ? T + (size_t)u * fp + v : T;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(xc + p.at());
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(ok ? 8 : 0) : "memory");
        }
    }
    // h of 16 rows at a time for the S_XX share, the first of them loaded while the columns arrive
    float2 hv[PART != 1 ? 16 : 1];
    auto load_h = [&](int tb) {   // unconditional loads, as in rec_rows_scan
        const size_t pitch = (size_t)D.pitch;
        const int va = min(v, W - 1), vb = min(v + 1, W - 1);
        auto take = [&](auto* h) {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const size_t o = (size_t)min(32 * (tb + q) + r0, H - 1) * pitch;
                hv[q] = f2((float)__ldg(h + o + va), (float)__ldg(h + o + vb));
            }
        };
        // byte pairs on 2-byte boundaries with one load each (not in the CTA that holds the last column of an
        // odd W): a warp's load touches 8 image rows whatever it takes from each
        const unsigned char* hb = reinterpret_cast<const unsigned char*>(D.data);
        if (D.dtype == ITC_U8 && ((pitch | reinterpret_cast<size_t>(hb)) & 1) == 0 && ((W & 1) == 0 || v0 + kRecLines <= W)) {
            const int at = min(v, W - 2);
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const size_t o = (size_t)min(32 * (tb + q) + r0, H - 1) * pitch;
                const uchar2 b = __ldg(reinterpret_cast<const uchar2*>(hb + o + at));
                hv[q] = f2((float)b.x, (float)b.y);
            }
        } else if (D.dtype == ITC_U8) {
            take(hb);
        } else {
            take(reinterpret_cast<const float*>(D.data));
        }
    };
    if constexpr (PART != 1) load_h(0);
    const RecAxis ax(PART == 2 ? D.rc_self : D.rc, 0);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (v0 + 2 * wid < W) filter_lines<MOM>(ax, xw, xw + 32 * str, xw + (MOM ? 64 : 32) * str, seg, str);
    __syncthreads();
    double hs = 0.0;
    LineAt p(r0, seg);
    for (int tb = 0; tb < seg; tb += 16) {
        if constexpr (PART != 1)
            if (tb > 0) load_h(tb);
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int u = 32 * (tb + q) + r0;
            if (tb + q < seg) {
                if (in && u < H) {
                    // a pair's second column past the image lies in the row padding
                    const size_t o = (size_t)u * fp + v;
                    float2 a = xc[32 * str + p.at()];
                    if (!in2) a.y = 0.f;
                    *reinterpret_cast<float2*>(A + o) = a;
                    if constexpr (MOM) {
                        float2 m = xc[64 * str + p.at()];
                        if (!in2) m.y = 0.f;
                        *reinterpret_cast<float2*>(A + pl + o) = m;
                    }
                    if constexpr (PART != 1) sum = fmaf(hv[q].x, a.x, fmaf(hv[q].y, a.y, sum));
                }
                p.next();
            }
            if constexpr (PART != 1)
                if (q % 4 == 3) {
                    hs += (double)sum;
                    sum = 0.f;
                }
        }
    }
    if constexpr (PART != 1) {
        for (int o = 16; o > 0; o >>= 1) hs += __shfl_xor_sync(0xffffffffu, hs, o);
        if (lane == 0) red[wid] = hs;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int q = 0; q < kRecPairs; ++q) t += red[q];
            L.partials[(PART == 0 ? D.partial_off : D.sxx_off) + blk] = t;
        }
    }
}

// Along v: a warp takes 32 rows, one lane per row, and walks them in 32 x 32 tiles staged in
// shared memory (rows of 33 floats), so every global load and store is a coalesced row segment
// while each lane runs its row's recursion on the staged tile.
constexpr int kRecRowWarps = 4;                        // row blocks per CTA
constexpr int kRecTileFloats = 3 * 32 * 33;            // a warp's three 32 x 33 tiles
constexpr int kRecCh = 8;                              // rows per prefetched chunk in the column pass
constexpr int kRecColThreads = 128;                    // columns per CTA in the column pass

template <bool MOM>   // MOM: the moment fields too (else the self-overlap pass: A alone)
__global__ void __launch_bounds__(32 * kRecRowWarps) rec_rows_kernel(const __grid_constant__ RecursiveLaunch L) {
    const ImageDesc& D = rec_image(L);
    const int H = D.H, W = D.W, fp = D.fpitch, pitch = D.pitch;
    float* P0 = L.fields + (MOM ? D.field_off + 3 * D.plane_floats : D.self_off + D.plane_floats);
    float* P1 = P0 + D.plane_floats;   // T_v (moments only)
    const RecCoef& rc = MOM ? D.rc : D.rc_self;
    const Cplx z0 = {rc.zr[1][0], rc.zi[1][0]}, z1 = {rc.zr[1][1], rc.zi[1][1]};
    const Cplx c0 = {rc.cr[0], rc.ci[0]}, c1 = {rc.cr[1], rc.ci[1]};
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    extern __shared__ float rsm[];
    float (*X)[33] = reinterpret_cast<float (*)[33]>(rsm + wid * kRecTileFloats);
    float (*O0)[33] = X + 32;
    float (*O1)[33] = X + 64;
    const int ntc = (W + 31) / 32;
    // this warp's block of 32 rows (warps past the image's last row have nothing to do; the
    // kernel takes no block-wide barrier)
    const int r0 = (blockIdx.y * kRecRowWarps + wid) * 32;
    if (r0 >= H) return;
    const int nr = min(32, H - r0);
    float* const q0 = P0 + (size_t)r0 * fp;   // row r0 of the scratch planes
    float* const q1 = P1 + (size_t)r0 * fp;
    const bool u8 = D.dtype == ITC_U8;
    const unsigned char* const xb = reinterpret_cast<const unsigned char*>(D.data) + (size_t)r0 * pitch;
    const float* const xf = reinterpret_cast<const float*>(D.data) + (size_t)r0 * pitch;
    auto load_x = [&](int cb) {   // input tile: rows r0.., columns cb.. (8 loads in flight at a time)
        const int v = cb + lane;
        if (v < W && u8) {
#pragma unroll 8
            for (int rr = 0; rr < 32; ++rr)
                if (rr < nr) X[rr][lane] = (float)__ldg(xb + rr * pitch + v);
        } else if (v < W) {
#pragma unroll 8
            for (int rr = 0; rr < 32; ++rr)
                if (rr < nr) X[rr][lane] = __ldg(xf + rr * pitch + v);
        } else {
            for (int rr = 0; rr < nr; ++rr) X[rr][lane] = 0.f;
        }
        __syncwarp();
    };
    auto store_tile = [&](int cb, int nc) {   // the staged outputs back, one coalesced row segment per row
        if (lane < nc) {
            for (int rr = 0; rr < nr; ++rr) {
                q0[rr * fp + cb + lane] = O0[rr][lane];
                if (MOM) q1[rr * fp + cb + lane] = O1[rr][lane];
            }
        }
        __syncwarp();
    };
    // causal: tiles left to right
    Cplx a0 = {0.f, 0.f}, a1 = {0.f, 0.f}, m0 = {0.f, 0.f}, m1 = {0.f, 0.f};   // s0, s1 per term
    auto causal = [&](int cc) {
        const float x = X[lane][cc];
        m0 = cmul(z0, cadd(m0, a0));
        m1 = cmul(z1, cadd(m1, a1));
        a0 = cmul(z0, a0); a0.r += x;
        a1 = cmul(z1, a1); a1.r += x;
        O0[lane][cc] = re_mul(c0, a0) + re_mul(c1, a1);
        if (MOM) O1[lane][cc] = -(re_mul(c0, m0) + re_mul(c1, m1));
    };
    for (int tc = 0; tc < ntc; ++tc) {
        const int cb = tc * 32, nc = min(32, W - cb);
        load_x(cb);
        if (lane < nr) {
            if (nc == 32) {
#pragma unroll 8
                for (int cc = 0; cc < 32; ++cc) causal(cc);
            } else {
                for (int cc = 0; cc < nc; ++cc) causal(cc);
            }
        }
        __syncwarp();
        store_tile(cb, nc);
    }
    // anticausal: tiles right to left; x[v + 1] of a tile's last column is the first column
    // of the tile to its right
    a0 = a1 = m0 = m1 = Cplx{0.f, 0.f};   // r0, r1 per term
    float xnext = 0.f;
    auto anticausal = [&](int cc, float xn) {
        m0 = cmul(z0, cadd(cadd(m0, a0), Cplx{xn, 0.f}));
        m1 = cmul(z1, cadd(cadd(m1, a1), Cplx{xn, 0.f}));
        a0 = cmul(z0, cadd(a0, Cplx{xn, 0.f}));
        a1 = cmul(z1, cadd(a1, Cplx{xn, 0.f}));
        O0[lane][cc] += re_mul(c0, a0) + re_mul(c1, a1);
        if (MOM) O1[lane][cc] += re_mul(c0, m0) + re_mul(c1, m1);
    };
    for (int tc = ntc - 1; tc >= 0; --tc) {
        const int cb = tc * 32, nc = min(32, W - cb);
        load_x(cb);
        if (lane < nc) {
#pragma unroll 4
            for (int rr = 0; rr < 32; ++rr) {
                if (rr < nr) {
                    O0[rr][lane] = q0[rr * fp + cb + lane];
                    if (MOM) O1[rr][lane] = q1[rr * fp + cb + lane];
                }
            }
        }
        __syncwarp();
        if (lane < nr) {
            if (nc == 32) {
                anticausal(31, xnext);
#pragma unroll 8
                for (int cc = 30; cc >= 0; --cc) anticausal(cc, X[lane][cc + 1]);
            } else {
                for (int cc = nc - 1; cc >= 0; --cc) anticausal(cc, cc + 1 < nc ? X[lane][cc + 1] : xnext);
            }
            xnext = X[lane][0];
        }
        __syncwarp();
        store_tile(cb, nc);
    }
}

template <bool MOM>
__global__ void __launch_bounds__(kRecColThreads) rec_cols_kernel(const __grid_constant__ RecursiveLaunch L) {
    const ImageDesc& D = rec_image(L);
    const int H = D.H, W = D.W, fp = D.fpitch;
    const long long pl = D.plane_floats;
    const float* T = L.fields + (MOM ? D.field_off + 3 * pl : D.self_off + pl);
    const float* Tv = T + pl;
    float* A = L.fields + (MOM ? D.field_off : D.self_off);
    float* Fu = A + pl;
    float* Fv = A + 2 * pl;
    const RecCoef& rc = MOM ? D.rc : D.rc_self;
    const Cplx z0 = {rc.zr[0][0], rc.zi[0][0]}, z1 = {rc.zr[0][1], rc.zi[0][1]};
    const Cplx c0 = {rc.cr[0], rc.ci[0]}, c1 = {rc.cr[1], rc.ci[1]};
    const int lane = threadIdx.x & 31;
    const long long poff = MOM ? D.partial_off : D.sxx_off;
    // whole warps walk the columns so that each warp's partial covers 32 consecutive columns;
    // this CTA takes columns blockIdx.y * kRecColThreads ..
    const int wcols = (W + 31) & ~31;
    const int vb = blockIdx.y * kRecColThreads;
    if (vb + (threadIdx.x & ~31) >= wcols) return;   // whole warps past the image
    // rows go in chunks of kRecCh: a chunk's loads are all issued before its recursion steps,
    // so the sequential walk waits on one memory round trip per chunk, not per row.  S_XX of the
    // column: FP32 within a chunk (at most kRecCh non-negative products), FP64 across chunks.
    constexpr int CH = kRecCh;
    const int v = vb + threadIdx.x;
    double hs = 0.0;
    if (v < W) {
        const bool u8 = D.dtype == ITC_U8;
        const unsigned char* const hb = reinterpret_cast<const unsigned char*>(D.data) + v;
        const float* const hf = reinterpret_cast<const float*>(D.data) + v;
        const int pitch = D.pitch;
        Cplx a0 = {0.f, 0.f}, a1 = {0.f, 0.f}, m0 = {0.f, 0.f}, m1 = {0.f, 0.f}, b0 = {0.f, 0.f}, b1 = {0.f, 0.f};
        for (int ub = 0; ub < H; ub += CH) {
            float xs[CH], ys[CH];
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int u = ub + c;
                xs[c] = u < H ? T[(size_t)u * fp + v] : 0.f;
                ys[c] = (MOM && u < H) ? Tv[(size_t)u * fp + v] : 0.f;
            }
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int u = ub + c;
                if (u >= H) break;
                const size_t o = (size_t)u * fp + v;
                const float x = xs[c];
                m0 = cmul(z0, cadd(m0, a0));
                m1 = cmul(z1, cadd(m1, a1));
                a0 = cmul(z0, a0); a0.r += x;
                a1 = cmul(z1, a1); a1.r += x;
                A[o] = re_mul(c0, a0) + re_mul(c1, a1);
                if (MOM) {
                    const float y = ys[c];
                    b0 = cmul(z0, b0); b0.r += y;
                    b1 = cmul(z1, b1); b1.r += y;
                    Fu[o] = -(re_mul(c0, m0) + re_mul(c1, m1));
                    Fv[o] = re_mul(c0, b0) + re_mul(c1, b1);
                }
            }
        }
        a0 = a1 = m0 = m1 = b0 = b1 = Cplx{0.f, 0.f};
        for (int ue = H - 1; ue >= 0; ue -= CH) {
            // this chunk's inputs (the row below each row) and the causal parts it adds to
            float xn[CH], yn[CH], ao[CH], fu[CH], fv[CH], hv[CH];
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int u = ue - c;
                xn[c] = yn[c] = ao[c] = fu[c] = fv[c] = hv[c] = 0.f;
                if (u >= 0) {
                    const size_t o = (size_t)u * fp + v;
                    xn[c] = u + 1 < H ? T[o + fp] : 0.f;
                    ao[c] = A[o];
                    hv[c] = u8 ? (float)__ldg(hb + (size_t)u * pitch) : __ldg(hf + (size_t)u * pitch);
                    if (MOM) {
                        yn[c] = u + 1 < H ? Tv[o + fp] : 0.f;
                        fu[c] = Fu[o];
                        fv[c] = Fv[o];
                    }
                }
            }
            float hc = 0.f;
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int u = ue - c;
                if (u < 0) break;
                const size_t o = (size_t)u * fp + v;
                m0 = cmul(z0, cadd(cadd(m0, a0), Cplx{xn[c], 0.f}));
                m1 = cmul(z1, cadd(cadd(m1, a1), Cplx{xn[c], 0.f}));
                a0 = cmul(z0, cadd(a0, Cplx{xn[c], 0.f}));
                a1 = cmul(z1, cadd(a1, Cplx{xn[c], 0.f}));
                const float a = ao[c] + re_mul(c0, a0) + re_mul(c1, a1);
                A[o] = a;
                if (MOM) {
                    b0 = cmul(z0, cadd(b0, Cplx{yn[c], 0.f}));
                    b1 = cmul(z1, cadd(b1, Cplx{yn[c], 0.f}));
                    Fu[o] = fu[c] + (re_mul(c0, m0) + re_mul(c1, m1));
                    Fv[o] = fv[c] + (re_mul(c0, b0) + re_mul(c1, b1));
                }
                hc = fmaf(hv[c], a, hc);
            }
            hs += (double)hc;
        }
    }
    // S_XX share of these 32 columns: a fixed-order shuffle tree
    for (int o = 16; o > 0; o >>= 1) hs += __shfl_xor_sync(0xffffffffu, hs, o);
    if (lane == 0) L.partials[poff + (v >> 5)] = hs;
}

}  // namespace

cudaError_t launch_recursive_scan(const RecursiveLaunch& L, int axis, int nimg, int lines, int len, cudaStream_t s) {
    if (nimg <= 0) return cudaSuccess;
    auto go = [&](auto k, int arrays) -> cudaError_t {
        cudaError_t e = allow_smem(k, rec_smem_bytes(kRecMaxLine, arrays));
        if (e != cudaSuccess) return e;
        const int nblk = (lines + kRecLines - 1) / kRecLines;
        k<<<(unsigned)(nimg * nblk), 32 * kRecPairs, rec_smem_bytes(len, arrays), s>>>(L, nblk);
        return cudaGetLastError();
    };
    if (axis == 1) return L.mode == 0 ? go(rec_rows_scan<true>, 3) : go(rec_rows_scan<false>, 2);
    if (L.mode != 0) return go(rec_cols_scan<2>, 2);
    const cudaError_t e = go(rec_cols_scan<0>, 3);
    return e != cudaSuccess ? e : go(rec_cols_scan<1>, 2);
}

cudaError_t launch_recursive_seq(const RecursiveLaunch& L, int nimg, int max_H, int max_W, cudaStream_t s) {
    if (nimg <= 0) return cudaSuccess;
    cudaError_t e;
    const size_t smem = (size_t)kRecRowWarps * kRecTileFloats * sizeof(float);
    if ((e = allow_smem(rec_rows_kernel<true>, smem)) != cudaSuccess) return e;
    if ((e = allow_smem(rec_rows_kernel<false>, smem)) != cudaSuccess) return e;
    const dim3 grow((unsigned)nimg, (unsigned)((max_H + 32 * kRecRowWarps - 1) / (32 * kRecRowWarps)));
    const dim3 gcol((unsigned)nimg, (unsigned)((max_W + kRecColThreads - 1) / kRecColThreads));
    if (L.mode == 0) {
        rec_rows_kernel<true><<<grow, 32 * kRecRowWarps, smem, s>>>(L);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        rec_cols_kernel<true><<<gcol, kRecColThreads, 0, s>>>(L);
    } else {
        rec_rows_kernel<false><<<grow, 32 * kRecRowWarps, smem, s>>>(L);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        rec_cols_kernel<false><<<gcol, kRecColThreads, 0, s>>>(L);
    }
    return cudaGetLastError();
}

}  // namespace itc
