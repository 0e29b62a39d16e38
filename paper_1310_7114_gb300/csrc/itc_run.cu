// itc_run.cu -- the fixed-point iterations of Algorithm 1 (steps 3-11) on precomputed fields.
//
// run_kernel: a CTA owns its images for all of their iterations: one image of 65 to 128 codebook
// vectors, else 2, 4 or 8 images of up to 64, 32 or 16 vectors, a thread per vector.  Images do not
// wait for one another: those of up to 32 vectors live in one warp, those of 33 to 64 in two warps
// with a named barrier of their own.  run_large_kernel: a cluster of CTAs owns one image of more
// than 128 vectors.  W, the gathered field values and the codebook sums stay on chip, the fields are
// read from L2/HBM by gathers.  Per iteration:
//   gather   a_k = A(r_k), D_k = F(r_k) (- r_k a_k if absolute) + (r_k - w_k) a_k,
//            r_k = round(w_k) clamped to the lattice                  (Eq. (accupdate) data terms)
//   pairs    s_k = sum_j g_rho(w_j - w_k),  E_k = sum_j g_rho(w_j - w_k)(w_j - w_k)   (Eq. (origupdate))
//            as two chains, the even j in order and the odd j in order, added at the end;
//            g = 2^(-sum_i d_i^2 c_i) (ex2.approx.ftz) with log2(e) folded into c_i.
//   sums     S_XW = sum_k a_k, S_WW = sum_k s_k (FP32 shuffle trees, then the image's warps in order),
//            c = S_XW / S_WW, D_cs of Eq. (1) in double at the reported W
//   update   w_k' = w_k + step_scale (D_k - kappa c E_k) / a_k, kappa_i = tau_i^2 / rho_i^2 (the
//            factor differentiating Eq. (1) gives the pair term; 1 when tau = rho), rounded to the
//            lattice unless ITC_CONTINUOUS (floor(w) + round(w - floor(w) + delta), exact in FP32
//            up to the one sum of the fraction and delta; a real-valued W lands on the lattice
//            after its first update); a_k = 0 keeps w_k.  Jacobi: every k reads the old W.
// Every sum has one order, whichever kernel, span or cluster size runs it, so the results do not
// depend on how a batch is cut.
#include <cooperative_groups.h>
#include <math.h>

#include "itc_internal.cuh"
#include "itc_pairs.cuh"

namespace itc {
namespace {

namespace cg = cooperative_groups;

__device__ __forceinline__ double warp_sum_d(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float lattice_round(float x, int n) {
    float r = floorf(x + 0.5f);
    return fminf(fmaxf(r, 0.f), (float)(n - 1));
}

struct Sums {
    float sxw, sww;
    int empty;
};

// The stats record of an image, by the whole calling warp for the image whose first lane is
// `leader` (that lane writes): the three logarithms of D_cs on three lanes at once.
// dev_status: the image's status word from the fields pass (ITC_ERR_TIMEOUT when a bounded wait
// there gave up; its S_XX is then NaN)
__device__ __forceinline__ void write_stats(itc_stats* st, bool leader, int first, const Sums& s, double sxx, int moved,
                                            int iters_done, double dcs_const, int dev_status) {
    const int q = (threadIdx.x & 31) - first;
    const double l = log(q == 0 ? (double)s.sww : (q == 1 ? sxx : (double)s.sxw));
    const double lw = __shfl_sync(0xffffffffu, l, first), lx = __shfl_sync(0xffffffffu, l, first + 1),
                 lc = __shfl_sync(0xffffffffu, l, first + 2);
    if (!leader) return;
    itc_stats r;
    r.sxw = s.sxw;
    r.sww = s.sww;
    r.sxx = sxx;
    r.c = (double)s.sxw / (double)s.sww;
    r.dcs = s.sxw > 0 ? lw + lx - 2.0 * lc + dcs_const : INFINITY;
    r.empty = s.empty;
    r.moved = moved;
    r.iters_done = iters_done;
    r.status = dev_status == ITC_ERR_TIMEOUT ? ITC_ERR_TIMEOUT
               : (!(s.sxw > 0) || !isfinite(r.dcs) ? ITC_ERR_NONFINITE
                  : (s.empty > 0 ? ITC_WARN_EMPTY_SUPPORT : ITC_OK));
    *st = r;
}

// The image fields the iteration needs, copied to registers once.
struct Img {
    const float* A;
    long long plane;
    int n[3];   // H, W, G
    int fpitch, M, iters, flags;
    float step;
};

__device__ __forceinline__ Img load_img(const RunLaunch& L, const ImageDesc& Dg) {
    Img D;
    D.A = L.fields + Dg.field_off;
    D.plane = Dg.plane_floats;
    D.n[0] = Dg.H; D.n[1] = Dg.W; D.n[2] = Dg.G;
    D.fpitch = Dg.fpitch; D.M = Dg.M; D.iters = Dg.iters; D.flags = Dg.flags; D.step = Dg.step_scale;
    return D;
}

// Positions split by the parity of j, for threads that sum the even or the odd j alone: four j are
// stored as (x_j, x_j+2, y_j, y_j+2) and (x_j+1, x_j+3, y_j+1, y_j+3).
constexpr int kHalfPad = 2 * kPairU;   // positions are padded to whole (half) blocks of one parity
__device__ __forceinline__ int half_at(int k) { return (k >> 2) * 8 + (k & 1) * 4 + ((k >> 1) & 1); }
__device__ __forceinline__ int half_atz(int k) { return (k >> 2) * 4 + (k & 1) * 2 + ((k >> 1) & 1); }

// The pair sums of one vector over the even (or odd) j alone, in order; the offsets, exponents and
// weights of two of them go through packed operations as in pair_sums.
template <int ND, bool ISO>
__device__ __forceinline__ void half_sums(const float* pos, const float* posz, int mp, int half, const float (&w)[ND],
                                          const float (&nc)[3], float& s, float (&E)[ND]) {
    float2 nw[ND];
#pragma unroll
    for (int i = 0; i < ND; ++i) { nw[i] = f2(-w[i], -w[i]); E[i] = 0.f; }
    s = 0.f;
    pos += 4 * half;
    posz += 2 * half;
    int j = 0;
    auto block = [&](auto steps) {
        constexpr int U = decltype(steps)::value;
        float2 g[U], d[U][ND];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float4 q = *reinterpret_cast<const float4*>(pos + 2 * j + 8 * u);
            const float2 z = ND == 3 ? *reinterpret_cast<const float2*>(posz + j + 4 * u) : f2(0.f, 0.f);
            g[u] = pair_weights<ND, ISO>(q, z, nw, nc, d[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            s += g[u].x;
            s += g[u].y;
#pragma unroll
            for (int i = 0; i < ND; ++i) {
                E[i] = fmaf(g[u].x, d[u][i].x, E[i]);
                E[i] = fmaf(g[u].y, d[u][i].y, E[i]);
            }
        }
        j += 4 * U;
    };
#pragma unroll 1
    while (j + 4 * kPairU <= mp) block(std::integral_constant<int, kPairU>());
    if (j < mp) block(std::integral_constant<int, kPairU / 2>());
}

// n / a, correctly rounded, with the correctly rounded reciprocal ra of a at hand (Markstein, IBM
// J. Res. Dev. 34, 1990: one residual correction of n ra); the range test keeps the residual exact,
// and anything outside it divides.
__device__ __forceinline__ float quotient(float n, float a, float ra, bool a_mid) {
    const float m = fabsf(n);
    if (a_mid && (m >= 1e-18f || m == 0.f) && m <= 1e18f) {
        const float q = n * ra;
        return fmaf(fmaf(-a, q, n), ra, q);
    }
    return n / a;
}

// The field values at a vector's site: a = A(r) and the moments; site r.
template <int ND>
__device__ __forceinline__ void gather(const Img& D, const float (&w)[ND], float (&r)[ND], float& a, float (&f)[ND]) {
#pragma unroll
    for (int i = 0; i < ND; ++i) r[i] = lattice_round(w[i], D.n[i]);
    const long long o = ((long long)(ND == 3 ? (int)r[ND - 1] : 0) * D.n[0] + (int)r[0]) * D.fpitch + (int)r[1];
    a = __ldg(D.A + o);
#pragma unroll
    for (int i = 0; i < ND; ++i) f[i] = __ldg(D.A + (i + 1) * D.plane + o);
}

// One coordinate of the update: w + delta, snapped to the lattice or kept real, clamped to it.
// snapped: round(w + delta) = fl + round(fr + delta) with w = fl + fr, fl = floor(w): fl and fr are
// exact in FP32, and on the lattice (fr = 0, the state after the first update) this is
// w + round(delta) with the one rounding of delta + 0.5.  A real-valued initial W (from a continuous
// run, or optimised by gradients) is rounded onto the lattice by its first update.
__device__ __forceinline__ float moved_to(float w, float delta, int n, bool snap) {
    const float fl = floorf(w);
    const float v = snap ? fl + floorf((w - fl) + delta + 0.5f) : w + delta;
    return fminf(fmaxf(v, 0.f), (float)(n - 1));
}

// S_XX of the images of a CTA's group (or of its one image Dg) from their tile partials into s_sxx.
// A gray image (a partial per slice tile) is always added as four strided shares, a 2-D image as one, in
// one order whichever warps take them: a warp a share, or where there are as many images as warps an image
// with its shares side by side (400 images of 64 x 64 x 64: 27 us an evaluation, 29 share by share).  Called
// by the first kRunThreads threads; s_sxx is valid after the caller's next block barrier.
template <int ND>
constexpr int kSxxShares = ND == 3 ? 4 : 1;
constexpr int kSxxMost = kGroupMax * kSxxShares<3>;
template <int ND>
__device__ __forceinline__ void load_sxx(const RunLaunch& L, const int* grp, int n, const ImageDesc& Dg, double* s_sxx) {
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    constexpr int NS = kSxxShares<ND>, NW = kRunThreads / 32;
    constexpr long long step = 32 * NS;
    if (L.sxx_single) {
        if (tid < NS) s_sxx[tid] = tid == 0 ? *L.sxx_single : 0.0;
        return;
    }
    auto lane_sum = [&](const double* p, long long nt, int share) {   // eight loads in flight
        double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        long long i = (long long)share * 32 + lane;
        for (; i + 7 * step < nt; i += 8 * step)
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] += p[i + q * step];
        if (i < nt) {   // the rest, fewer than eight
            double x[7];
#pragma unroll
            for (int q = 0; q < 7; ++q) x[q] = i + q * step < nt ? p[i + q * step] : 0.0;
#pragma unroll
            for (int q = 0; q < 7; ++q)
                if (i + q * step < nt) v[0] += x[q];
        }
        return ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    };
    const bool images = ND == 3 && n >= NW;
    for (int g = wid; g < (images ? n : n * NS); g += NW) {
        const int im = images ? g : g / NS;
        const ImageDesc& ds = grp ? L.descs[__ldg(grp + 2 + im)] : Dg;
        const long long nt = ds.sxx_tiles;
        const double* p = L.partials + ds.sxx_off;
        if constexpr (ND == 3) {
            if (images) {
                double t[NS];
#pragma unroll
                for (int q = 0; q < NS; ++q) t[q] = 0;
                if (nt <= 7 * step) {   // the sums of lane_sum, all shares at once
#pragma unroll 2
                    for (long long i = lane; i < nt; i += step)
#pragma unroll
                        for (int q = 0; q < NS; ++q) t[q] += i + 32 * q < nt ? p[i + 32 * q] : 0.0;
                } else {
#pragma unroll
                    for (int q = 0; q < NS; ++q) t[q] = lane_sum(p, nt, q);
                }
#pragma unroll
                for (int q = 0; q < NS; ++q) t[q] = warp_sum_d(t[q]);
                if (lane == 0)
#pragma unroll
                    for (int q = 0; q < NS; ++q) s_sxx[g * NS + q] = t[q];
                continue;
            }
        }
        const double t = warp_sum_d(lane_sum(p, nt, g % NS));
        if (lane == 0) s_sxx[g] = t;
    }
}
// (after the barrier) S_XX of image `sub` of the group
template <int ND>
__device__ __forceinline__ double read_sxx(const double* s_sxx, int sub) {
    double t = 0;
#pragma unroll
    for (int q = 0; q < kSxxShares<ND>; ++q) t += s_sxx[sub * kSxxShares<ND> + q];
    return t;
}

// All iterations of the images of one group, SPAN threads each (a thread per codebook vector).
// The position array of an image is only read between its two synchronisations per iteration and
// only written after the first of them.
template <int ND, int SPAN>
__device__ __forceinline__ void iterate_group(const RunLaunch& L, const int* grp, int n, float* s_pos, float2* s_red,
                                              int* s_mv, const double* s_sxx) {
    constexpr int WPI = SPAN / 32;   // warps per image (0: two images per warp)
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int sub = tid / SPAN, kl = tid % SPAN;
    const int img = grp ? (sub < n ? __ldg(grp + 2 + sub) : -1) : (sub == 0 ? L.img_base + (int)blockIdx.x : -1);
    const bool has = img >= 0;
    if (!__any_sync(0xffffffffu, has)) return;   // a warp without images takes no further barrier
    const ImageDesc& Dg = L.descs ? L.descs[has ? img : (grp ? __ldg(grp + 2) : L.img_base + (int)blockIdx.x)] : L.one;
    Img D = load_img(L, Dg);
    if (!has) D.M = 0;
    const PairWidths<ND> pw(Dg);
    const bool mine = kl < D.M;
    const int mp = (D.M + kPairPad - 1) / kPairPad * kPairPad;
    float* sxy = s_pos + sub * SPAN * ND;
    float* sz = sxy + 2 * SPAN;
    auto sync_image = [&]() {
        if constexpr (SPAN <= 32) __syncwarp();
        else if constexpr (SPAN == 64) asm volatile("bar.sync %0, 64;" ::"r"(1 + sub) : "memory");
        else __syncthreads();
    };
    float w[ND];
    const float* Win = L.W_in + Dg.w_off;
#pragma unroll
    for (int i = 0; i < ND; ++i) w[i] = mine ? Win[kl * ND + i] : kFar;
    auto publish = [&]() {
        sxy[(kl >> 1) * 4 + (kl & 1)] = w[0];
        sxy[(kl >> 1) * 4 + 2 + (kl & 1)] = w[1];
        if constexpr (ND == 3) sz[kl] = w[ND - 1];
    };
    publish();
    sync_image();
    const bool snap = !(D.flags & ITC_CONTINUOUS);
    const bool stop_fixed = (D.flags & ITC_STOP_ON_FIXED) != 0;
    float kap[ND];
#pragma unroll
    for (int i = 0; i < ND; ++i) kap[i] = Dg.kappa[i];

    // every test below that steers synchronisation is uniform over an image (and, for images that
    // share a warp, taken by the whole warp)
    Sums s = {0.f, 0.f, 0};
    int moved = 0, done = 0;
    bool stop = false, live = has;
    for (int t = 0;; ++t) {
        if (!L.final_eval && t == D.iters) live = false;
        if (SPAN <= 16 ? !__any_sync(0xffffffffu, live) : !live) break;
        float a = 0.f, sk = 0.f, Dm[ND], Ek[ND];
#pragma unroll
        for (int i = 0; i < ND; ++i) Dm[i] = Ek[i] = 0.f;
        if (mine && live) {
            float r[ND], f[ND];
            gather<ND>(D, w, r, a, f);   // its latency overlaps the pair sums
            if (ND == 2 && pw.iso) pair_sums<ND, ND == 2>(sxy, sz, mp, w, pw.nc, sk, Ek);
            else pair_sums<ND, false>(sxy, sz, mp, w, pw.nc, sk, Ek);
#pragma unroll
            for (int i = 0; i < ND; ++i)   // centred moment about the real w_k
                Dm[i] = fmaf(r[i] - w[i], a, L.absolute ? f[i] - r[i] * a : f[i]);
        }
        const float av = a > 0.f ? a : 1.f;
        const float ra = __frcp_rn(av);   // while the sums are under way
        const bool a_mid = av >= 1e-18f && av <= 1e18f;
        // S_XW, S_WW: a shuffle tree over the image's lanes, then its warps in order.  Zeros from
        // threads past M leave a sum unchanged, so the result is the same for any span.
        float x = a, y = sk;
#pragma unroll
        for (int o = SPAN >= 32 ? 16 : SPAN / 2; o > 0; o >>= 1) {
            x += __shfl_xor_sync(0xffffffffu, x, o);
            y += __shfl_xor_sync(0xffffffffu, y, o);
        }
        const bool upd = live && t != D.iters && !stop;
        const bool last = !upd || (!L.final_eval && t == 0);   // the sums of this evaluation are reported
        if constexpr (SPAN > 32) {
            if (lane == 0) s_red[wid] = f2(x, y);
        }
        int e = 0;
        if (SPAN <= 16 ? __any_sync(0xffffffffu, last && live) : last && live) {
            const unsigned b = __ballot_sync(0xffffffffu, mine && live && !(a > 0.f));
            e = __popc(SPAN == 16 ? (b >> (lane & 16)) & 0xffffu : b);
            if (SPAN > 32 && lane == 0) s_mv[wid] = e;
        }
        sync_image();   // the warp sums are in, and every vector's pair reads are done
        if constexpr (SPAN > 32) {
            const float2* rd = s_red + sub * WPI;
            x = y = 0.f;
#pragma unroll
            for (int q = 0; q < WPI; ++q) { x += rd[q].x; y += rd[q].y; }
        }
        if (live) { s.sxw = x; s.sww = y; }
        if (last && live) {
            if constexpr (SPAN > 32) {
                e = 0;
#pragma unroll
                for (int q = 0; q < WPI; ++q) e += s_mv[sub * WPI + q];
            }
            s.empty = e;
        }
        if (!L.final_eval && t == 0 && L.stats && (SPAN <= 32 || kl < 32))
            write_stats(L.stats + (has ? img : 0), has && kl == 0, SPAN == 16 ? (lane & 16) : 0, s,
                        read_sxx<ND>(s_sxx, has ? sub : 0), 0, 0, Dg.dcs_const,
                        has && L.img_status ? L.img_status[img] : ITC_OK);
        if (!upd) live = false;
        // threads that do not update divide 1 by 1 (0 / 0 would take the slow division path and
        // hold the image's warps)
        const float c = (upd ? x : 1.f) / (upd ? y : 1.f);
        bool kmoved = false;
        if (upd && mine && a > 0.f) {
#pragma unroll
            for (int i = 0; i < ND; ++i) {
                // tau^2 / rho^2 on the pair term: 1 (exact) when tau = rho
                const float delta = quotient(D.step * (Dm[i] - (c * kap[i]) * Ek[i]), av, ra, a_mid);
                const float nv = moved_to(w[i], delta, D.n[i], snap);
                kmoved |= (nv != w[i]);
                w[i] = nv;
            }
            publish();
        }
        // vectors moved where the count is used: by the stopping test, and for the stats after an
        // image's last update
        const bool count = upd && (stop_fixed || t + 1 == D.iters);
        if (SPAN <= 16 ? __any_sync(0xffffffffu, count) : count) {
            const unsigned b = __ballot_sync(0xffffffffu, kmoved);
            int mv = __popc(SPAN == 16 ? (b >> (lane & 16)) & 0xffffu : b);
            if constexpr (SPAN > 32) {
                sync_image();   // the empty counts are read
                if (lane == 0) s_mv[wid] = mv;
                sync_image();
                mv = 0;
#pragma unroll
                for (int q = 0; q < WPI; ++q) mv += s_mv[sub * WPI + q];
            }
            if (count) {
                moved = mv;
                if (stop_fixed && moved == 0) stop = true;
            }
        }
        if (upd) ++done;
        sync_image();   // the new positions are in place
    }
    if (L.stats && L.final_eval && (SPAN <= 32 || kl < 32))
        write_stats(L.stats + (has ? img : 0), has && kl == 0, SPAN == 16 ? (lane & 16) : 0, s,
                    read_sxx<ND>(s_sxx, has ? sub : 0), moved, done, Dg.dcs_const,
                    has && L.img_status ? L.img_status[img] : ITC_OK);
    if (has && !L.final_eval && L.stats && kl == 0) {
        L.stats[img].moved = moved;
        L.stats[img].iters_done = done;
    }
    if (mine) {
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            L.W_out[Dg.w_off + kl * ND + i] = w[i];
            if (L.W_lattice) L.W_lattice[Dg.w_off + kl * ND + i] = (int)lattice_round(w[i], D.n[i]);
        }
    }
}

// All iterations of an image that has the CTA to itself, 33 to kRunThreads / 2 vectors: two threads
// per vector, the owner (first half of the CTA) and a helper that adds up the odd j.  A lone
// image's iteration is a chain of latencies, of which the pair loop is the longest: one image of
// M = 64 takes 1.22 us per iteration with one thread per vector and 1.05 us with two (101
// evaluations, 1024 x 1024: 124 and 113 us; 164 us when four idle or waiting warps shared every
// barrier and the pair loop ran one step at a time).
template <int ND>
__device__ __forceinline__ void iterate_wide(const RunLaunch& L, int img, const ImageDesc& Dg, float* pos, float4* s_half,
                                             float2* s_red, int* s_mv, const double* s_sxx) {
    constexpr int SPAN = kRunThreads / 2;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int kl = tid % SPAN;
    const bool owner = tid < SPAN;
    const Img D = load_img(L, Dg);
    const PairWidths<ND> pw(Dg);
    const bool mine = kl < D.M;
    const int mp = (D.M + kHalfPad - 1) / kHalfPad * kHalfPad;
    float* posz = pos + 2 * SPAN;
    float w[ND], kap[ND];
#pragma unroll
    for (int i = 0; i < ND; ++i) {
        w[i] = mine ? L.W_in[Dg.w_off + kl * ND + i] : kFar;
        kap[i] = Dg.kappa[i];
    }
    auto publish = [&]() {
        pos[half_at(kl)] = w[0];
        pos[half_at(kl) + 2] = w[1];
        if constexpr (ND == 3) posz[half_atz(kl)] = w[ND - 1];
    };
    auto sync_owners = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(SPAN) : "memory"); };
    if (owner) publish();
    if (tid == 0) s_mv[2] = 0;
    __syncthreads();
    const bool snap = !(D.flags & ITC_CONTINUOUS);
    const bool stop_fixed = (D.flags & ITC_STOP_ON_FIXED) != 0;
    Sums s = {0.f, 0.f, 0};
    int moved = 0, done = 0;
    for (int t = 0;; ++t) {
        if (!L.final_eval && t == D.iters) break;
        const bool upd = t != D.iters && !(stop_fixed && s_mv[2]);   // s_mv[2]: the image has stopped
        const bool last = !upd || (!L.final_eval && t == 0);
        float a = 0.f, sk = 0.f, r[ND], f[ND], Dm[ND], Ek[ND];
#pragma unroll
        for (int i = 0; i < ND; ++i) { r[i] = f[i] = Dm[i] = Ek[i] = 0.f; }
        if (!owner) {   // a helper reads its vector's position as the owner published it
            w[0] = pos[half_at(kl)];
            w[1] = pos[half_at(kl) + 2];
            if constexpr (ND == 3) w[ND - 1] = posz[half_atz(kl)];
        }
        if (mine) {
            if (owner) gather<ND>(D, w, r, a, f);   // its latency overlaps the pair sums
            if (ND == 2 && pw.iso) half_sums<ND, ND == 2>(pos, posz, mp, !owner, w, pw.nc, sk, Ek);
            else half_sums<ND, false>(pos, posz, mp, !owner, w, pw.nc, sk, Ek);
            if (!owner) s_half[kl] = make_float4(sk, Ek[0], Ek[1], ND == 3 ? Ek[ND - 1] : 0.f);
        }
        __syncthreads();   // the odd sums are in, and every pair read is done
        if (owner) {
            if (mine) {
                const float4 h = s_half[kl];
                sk += h.x;
                Ek[0] += h.y;
                Ek[1] += h.z;
                if constexpr (ND == 3) Ek[ND - 1] += h.w;
#pragma unroll
                for (int i = 0; i < ND; ++i)   // centred moment about the real w_k
                    Dm[i] = fmaf(r[i] - w[i], a, L.absolute ? f[i] - r[i] * a : f[i]);
            }
            const float av = a > 0.f ? a : 1.f;
            const float ra = __frcp_rn(av);
            const bool a_mid = av >= 1e-18f && av <= 1e18f;
            float x = a, y = sk;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                x += __shfl_xor_sync(0xffffffffu, x, o);
                y += __shfl_xor_sync(0xffffffffu, y, o);
            }
            if (lane == 0) s_red[wid] = f2(x, y);
            if (last) {
                const unsigned b = __ballot_sync(0xffffffffu, mine && !(a > 0.f));
                if (lane == 0) s_mv[wid] = __popc(b);
            }
            sync_owners();
            x = y = 0.f;
#pragma unroll
            for (int q = 0; q < SPAN / 32; ++q) { x += s_red[q].x; y += s_red[q].y; }
            s.sxw = x;
            s.sww = y;
            if (last) s.empty = s_mv[0] + s_mv[1];
            if (!L.final_eval && t == 0 && L.stats && kl < 32)
                write_stats(L.stats + img, kl == 0, 0, s, read_sxx<ND>(s_sxx, 0), 0, 0, Dg.dcs_const,
                            L.img_status ? L.img_status[img] : ITC_OK);
            if (upd) {
                const float c = x / y;
                bool kmoved = false;
                if (mine && a > 0.f) {
#pragma unroll
                    for (int i = 0; i < ND; ++i) {
                        const float delta = quotient(D.step * (Dm[i] - (c * kap[i]) * Ek[i]), av, ra, a_mid);
                        const float nv = moved_to(w[i], delta, D.n[i], snap);
                        kmoved |= (nv != w[i]);
                        w[i] = nv;
                    }
                    publish();
                }
                if (stop_fixed || t + 1 == D.iters) {
                    const unsigned b = __ballot_sync(0xffffffffu, kmoved);
                    sync_owners();   // the empty counts are read
                    if (lane == 0) s_mv[wid] = __popc(b);
                    sync_owners();
                    moved = s_mv[0] + s_mv[1];
                    if (tid == 0 && stop_fixed && moved == 0) s_mv[2] = 1;
                }
                ++done;
            }
        }
        __syncthreads();   // the new positions are in place
        if (!upd) break;
    }
    if (!owner) return;
    if (L.stats && L.final_eval && kl < 32)
        write_stats(L.stats + img, kl == 0, 0, s, read_sxx<ND>(s_sxx, 0), moved, done, Dg.dcs_const,
                    L.img_status ? L.img_status[img] : ITC_OK);
    if (!L.final_eval && L.stats && kl == 0) {
        L.stats[img].moved = moved;
        L.stats[img].iters_done = done;
    }
    if (mine) {
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            L.W_out[Dg.w_off + kl * ND + i] = w[i];
            if (L.W_lattice) L.W_lattice[Dg.w_off + kl * ND + i] = (int)lattice_round(w[i], D.n[i]);
        }
    }
}

// ------------------------------------------------------------- one image of more than kRunThreads vectors
constexpr int kLargeCluster = 8;        // most CTAs per image (the portable cluster size)
constexpr size_t kMergedSmem = 30 * 1024;   // 7 CTAs per SM
constexpr double kClusterWork = 1.5e5;      // pairs over all iterations of an image: about 20 us of one CTA
__host__ __device__ constexpr int large_threads(bool split) { return split ? 256 : 128; }
// Where a vector's position lies: split by the parity of k for half_sums, in pairs for pair_sums.
template <bool SPLIT>
__device__ __forceinline__ int large_at(int k) { return SPLIT ? half_at(k) : (k >> 1) * 4 + (k & 1); }
template <bool SPLIT>
__device__ __forceinline__ int large_atz(int k) { return SPLIT ? half_atz(k) : k; }

// Vectors owned by each CTA of a cluster of `csize`: whole warps of them.
__host__ __device__ inline int large_share(int M, int csize) { return ((M + csize - 1) / csize + 31) & ~31; }
__host__ __device__ inline size_t large_smem_floats(int M, int csize, int nd) {
    const int mp = (M + kHalfPad - 1) / kHalfPad * kHalfPad;
    return (size_t)mp * (nd + 2) + (size_t)large_share(M, csize) * (3 + 3 * nd);
}

// One image of more than kRunThreads vectors per cluster: each CTA owns a share of the vectors and
// keeps a copy of every position.  Per iteration: (1) each vector's pair sums and gathers, SPLIT:
// the even and the odd j by two threads in different warps; (2) a_k and s_k to every CTA, cluster
// barrier; (3) every CTA adds S_XW and S_WW in the one order (kRunThreads strided chains, shuffle
// trees, warps in order) and updates its share, the new positions to every CTA, cluster barrier.
// Bound by the pair weights, M^2 of them at 16 ex2 per clock and SM, so an image is spread over as
// many SMs as the launch leaves idle, and then (SPLIT) over more warps of each.  A launch with an
// image for every second SM or more takes one CTA per image and whole pair sums, whose packed
// accumulation issues fewer instructions.  M = 1024, 20 iterations of one image: 3.09 ms on one CTA of
// 128 threads, 0.18 ms on 8 CTAs.
template <int ND, bool SPLIT>
__device__ __forceinline__ void iterate_large(const RunLaunch& L) {
    constexpr int NT = large_threads(SPLIT);
    cg::cluster_group cluster = cg::this_cluster();
    const int csize = SPLIT ? (int)cluster.num_blocks() : 1, rank = SPLIT ? (int)cluster.block_rank() : 0;
    auto sync_all = [&]() {
        if constexpr (SPLIT) cluster.sync();
        else __syncthreads();
    };
    auto in_cta = [&](auto* p, int dst) {   // the same place in CTA dst of the cluster
        if constexpr (SPLIT) return cluster.map_shared_rank(p, dst);
        else return p;
    };
    const int cid = blockIdx.x / csize;
    const int* grp = L.groups ? L.groups + (size_t)cid * kGroupInts : nullptr;
    const int img = grp ? __ldg(grp + 2) : L.img_base + cid;
    const ImageDesc& Dg = L.descs ? L.descs[img] : L.one;
    if (!grp && (Dg.ndim != ND || Dg.M <= kRunThreads)) return;   // cluster-uniform
    const Img D = load_img(L, Dg);
    const PairWidths<ND> pw(Dg);
    const int M = D.M, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int PAD = SPLIT ? kHalfPad : kPairPad;
    const int mp = (M + PAD - 1) / PAD * PAD;
    const int share = large_share(M, csize), k0 = min(M, rank * share), own = min(M, k0 + share) - k0;
    extern __shared__ __align__(16) float lsm[];
    float* pos = lsm;                      // positions, 2 mp floats (layout: large_at)
    float* posz = pos + 2 * mp;            // third coordinate (3-D)
    float2* as = reinterpret_cast<float2*>(posz + (ND == 3 ? mp : 0));   // (a_k, s_k) of every vector
    float* st = reinterpret_cast<float*>(as + mp);   // this CTA's vectors: planes of `share` floats:
    // even s, even E[ND], odd s, odd E[ND], a, D[ND]
    __shared__ double s_sxx[kSxxMost];
    __shared__ float2 s_red[kRunThreads / 32];
    __shared__ int s_empty, s_mv, s_cnt[kLargeCluster];   // s_cnt: moved vectors of every CTA
    const float* Win = L.W_in + Dg.w_off;
    for (int k = tid; k < mp; k += NT) {
        pos[large_at<SPLIT>(k)] = k < M ? Win[k * ND] : kFar;
        pos[large_at<SPLIT>(k) + 2] = k < M ? Win[k * ND + 1] : kFar;
        if constexpr (ND == 3) posz[large_atz<SPLIT>(k)] = k < M ? Win[k * ND + 2] : kFar;
    }
    if (tid < kRunThreads) load_sxx<ND>(L, grp, 1, Dg, s_sxx);
    auto load_w = [&](int k, float (&w)[ND]) {
        w[0] = pos[large_at<SPLIT>(k)];
        w[1] = pos[large_at<SPLIT>(k) + 2];
        if constexpr (ND == 3) w[ND - 1] = posz[large_atz<SPLIT>(k)];
    };
    // warps of each half: as many as the share fills, so that a small share spreads over the SM's
    // sub-partitions
    const int hw = min(NT / 64, (own + 31) >> 5);
    const bool snap = !(D.flags & ITC_CONTINUOUS);
    const bool stop_fixed = (D.flags & ITC_STOP_ON_FIXED) != 0;
    sync_all();   // positions in place, and every CTA of the cluster is running

    Sums s = {0.f, 0.f, 0};
    int moved = 0, done = 0;
    bool stop = false;
    for (int t = 0;; ++t) {
        if (!L.final_eval && t == D.iters) break;
        // (1) pair sums and gathers
        const int half = SPLIT && wid >= hw;
        const int step = SPLIT ? 32 * hw : NT;
        for (int i = SPLIT ? (wid < 2 * hw ? tid - half * step : own) : tid; i < own; i += step) {
            float w[ND], r[ND], f[ND], a = 0.f, hs, he[ND];
            load_w(k0 + i, w);
            if (!half) gather<ND>(D, w, r, a, f);
            if constexpr (SPLIT) {
                if (ND == 2 && pw.iso) half_sums<ND, ND == 2>(pos, posz, mp, half, w, pw.nc, hs, he);
                else half_sums<ND, false>(pos, posz, mp, half, w, pw.nc, hs, he);
            } else {
                if (ND == 2 && pw.iso) pair_sums<ND, ND == 2>(pos, posz, mp, w, pw.nc, hs, he);
                else pair_sums<ND, false>(pos, posz, mp, w, pw.nc, hs, he);
            }
            float* o = st + (half ? 1 + ND : 0) * share + i;
            o[0] = hs;
#pragma unroll
            for (int q = 0; q < ND; ++q) o[(1 + q) * share] = he[q];
            if (!half) {
                st[(2 + 2 * ND) * share + i] = a;
#pragma unroll
                for (int q = 0; q < ND; ++q)   // centred moment about the real w_k
                    st[(3 + 2 * ND + q) * share + i] = fmaf(r[q] - w[q], a, L.absolute ? f[q] - r[q] * a : f[q]);
            }
        }
        __syncthreads();
        // (2) a_k and s_k to every CTA
        for (int e = tid; e < own * csize; e += NT) {
            const int i = e % own, dst = e / own;
            const float2 v = f2(st[(2 + 2 * ND) * share + i], SPLIT ? st[i] + st[(1 + ND) * share + i] : st[i]);
            in_cta(as, dst)[k0 + i] = v;
        }
        sync_all();
        // (3) sums, the same in every CTA
        if (tid == 0) s_empty = s_mv = 0;
        float x = 0.f, y = 0.f;
        int e = 0;
        if (tid < kRunThreads) {
            for (int k = tid; k < M; k += kRunThreads) {
                const float2 v = as[k];
                x += v.x;
                y += v.y;
                e += !(v.x > 0.f);
            }
            for (int o = 16; o > 0; o >>= 1) {
                x += __shfl_xor_sync(0xffffffffu, x, o);
                y += __shfl_xor_sync(0xffffffffu, y, o);
            }
            e = __reduce_add_sync(0xffffffffu, e);
            if (lane == 0) s_red[wid] = f2(x, y);
        }
        __syncthreads();
        if (tid < kRunThreads && lane == 0 && e) atomicAdd(&s_empty, e);
        x = y = 0.f;
#pragma unroll
        for (int q = 0; q < kRunThreads / 32; ++q) { x += s_red[q].x; y += s_red[q].y; }
        s.sxw = x;
        s.sww = y;
        if (!L.final_eval && t == 0 && L.stats) {   // uniform: the counts are complete after this barrier
            __syncthreads();
            s.empty = s_empty;
            if (rank == 0 && wid == 0)
                write_stats(L.stats + img, lane == 0, 0, s, read_sxx<ND>(s_sxx, 0), 0, 0, Dg.dcs_const,
                            L.img_status ? L.img_status[img] : ITC_OK);
        }
        if (t == D.iters || stop) break;   // uniform over the cluster
        const float c = x / y;
        int mv = 0;
        for (int i = tid; i < own; i += NT) {
            const float a = st[(2 + 2 * ND) * share + i];
            if (!(a > 0.f)) continue;
            const float ra = __frcp_rn(a);
            const bool a_mid = a >= 1e-18f && a <= 1e18f;
            float w[ND];
            load_w(k0 + i, w);
            bool km = false;
#pragma unroll
            for (int q = 0; q < ND; ++q) {
                const float Ek = SPLIT ? st[(1 + q) * share + i] + st[(2 + ND + q) * share + i] : st[(1 + q) * share + i];
                const float delta = quotient(D.step * (st[(3 + 2 * ND + q) * share + i] - (c * Dg.kappa[q]) * Ek), a, ra, a_mid);
                const float nv = moved_to(w[q], delta, D.n[q], snap);
                km |= (nv != w[q]);
                w[q] = nv;
            }
            mv += km;
            if (km) {
                for (int dst = 0; dst < csize; ++dst) {
                    float* p = in_cta(pos, dst) + large_at<SPLIT>(k0 + i);
                    p[0] = w[0];
                    p[2] = w[1];
                    if constexpr (ND == 3) in_cta(posz, dst)[large_atz<SPLIT>(k0 + i)] = w[ND - 1];
                }
            }
        }
        // vectors moved, where the count is used: by the stopping test and after the last update
        const bool count = stop_fixed || t + 1 == D.iters;   // uniform over the cluster
        if (count) {
            mv = __reduce_add_sync(0xffffffffu, mv);
            if (lane == 0 && mv) atomicAdd(&s_mv, mv);
            __syncthreads();
            if (tid < csize) in_cta(s_cnt, tid)[rank] = s_mv;
        }
        sync_all();   // the new positions (and counts) are in every CTA
        if (count) {
            moved = 0;
            for (int q = 0; q < csize; ++q) moved += s_cnt[q];
            if (stop_fixed && moved == 0) stop = true;
        }
        ++done;
    }
    __syncthreads();
    if (rank == 0 && L.stats && L.final_eval && wid == 0) {
        s.empty = s_empty;
        write_stats(L.stats + img, lane == 0, 0, s, read_sxx<ND>(s_sxx, 0), moved, done, Dg.dcs_const,
                    L.img_status ? L.img_status[img] : ITC_OK);
    }
    if (rank == 0 && L.stats && !L.final_eval && tid == 0) {
        L.stats[img].moved = moved;
        L.stats[img].iters_done = done;
    }
    for (int i = tid; i < own; i += NT) {
        float w[ND];
        load_w(k0 + i, w);
        const int k = k0 + i;
#pragma unroll
        for (int q = 0; q < ND; ++q) {
            L.W_out[Dg.w_off + k * ND + q] = w[q];
            if (L.W_lattice) L.W_lattice[Dg.w_off + k * ND + q] = (int)lattice_round(w[q], D.n[q]);
        }
    }
}

template <int ND, bool SPLIT>
__global__ void __launch_bounds__(large_threads(SPLIT), SPLIT ? 1 : (ND == 3 ? 6 : 7))
    run_large_kernel(const __grid_constant__ RunLaunch L) {
    iterate_large<ND, SPLIT>(L);
}

// ND: lattice dimension (2 or 3).
// Register budget: 7 CTAs per SM in 2-D and 6 in 3-D leave the per-iteration state in registers
// (8 CTAs per SM spilled it and lengthened every iteration).
template <int ND>
__global__ void __launch_bounds__(kRunThreads, ND == 3 ? 6 : 7) run_kernel(const __grid_constant__ RunLaunch L) {
    const int* grp = L.groups ? L.groups + (size_t)blockIdx.x * kGroupInts : nullptr;
    const int n = grp ? __ldg(grp) : 1;
    const ImageDesc& Dg = L.descs ? L.descs[grp ? __ldg(grp + 2) : L.img_base + (int)blockIdx.x] : L.one;
    // a range launch covers every image once per dimension and kernel (CTA-uniform)
    if (!grp && Dg.ndim != ND) return;
    const int M = Dg.M;
    if (M > kRunThreads) {   // with_large: the launch covers these too, else a launch of their own
        if (L.with_large) iterate_large<ND, false>(L);
        return;
    }
    const int span = grp ? __ldg(grp + 1) : (M <= 16 ? 16 : (M <= 32 ? 32 : (M <= 64 ? 64 : kRunThreads)));
    __shared__ __align__(16) float s_pos[ND * kRunThreads];
    __shared__ __align__(16) float2 s_red[kRunThreads / 32];
    __shared__ float4 s_half[kRunThreads / 2];
    __shared__ int s_mv[kRunThreads / 32];
    __shared__ double s_sxx[kSxxMost];
    load_sxx<ND>(L, grp, n, Dg, s_sxx);
    __syncthreads();
    if (span == 16) iterate_group<ND, 16>(L, grp, n, s_pos, s_red, s_mv, s_sxx);
    else if (span == 32) iterate_group<ND, 32>(L, grp, n, s_pos, s_red, s_mv, s_sxx);
    else if (span == 64 && n == 1)
        iterate_wide<ND>(L, grp ? __ldg(grp + 2) : L.img_base + (int)blockIdx.x, Dg, s_pos, s_half, s_red, s_mv, s_sxx);
    else if (span == 64) iterate_group<ND, 64>(L, grp, n, s_pos, s_red, s_mv, s_sxx);
    else iterate_group<ND, 128>(L, grp, n, s_pos, s_red, s_mv, s_sxx);
}

// CTAs per image of a launch with nlarge images of more than kRunThreads vectors: as many as give
// each of their CTAs an SM of its own, up to the portable cluster size, and a warp of vectors each
int cluster_size(int nlarge, int max_M, int sms) {
    int c = 1;
    while (c < kLargeCluster && 2 * c * nlarge <= sms && large_share(max_M, 2 * c) < large_share(max_M, c)) c *= 2;
    return c;
}

template <int ND>
cudaError_t launch_nd(RunLaunch L, int large_ctas, int nlarge, int ctas, int max_M, double work, cudaStream_t s) {
    cudaError_t e;
    size_t smem = 0;
    if (nlarge > 0) {
        int dev = 0, sms = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        const int csize = cluster_size(nlarge, max_M, sms);
        // One launch for all, a CTA per large image, where their shared memory still lets 7 CTAs share
        // an SM and clusters are not to be had (2000 images of M 64, 128 and 256, 50 iterations: 1.09
        // ms in two launches, 0.96 ms in one) or would not repay the second launch's 7 us: a CTA alone
        // takes about 0.13 ns per pair (101 images of M 34 to 136, no iterations: 17 and 12 us).
        const size_t one = large_smem_floats(max_M, 1, ND) * sizeof(float);
        const bool others = L.groups ? ctas > 0 : ctas > nlarge;
        if (one <= kMergedSmem && (csize == 1 || (others && work < kClusterWork))) {
            L.with_large = 1;
            smem = one;
            if (L.groups) ctas += large_ctas;   // their groups come first
        } else {
            smem = large_smem_floats(max_M, csize, ND) * sizeof(float);
            auto k = csize > 1 ? run_large_kernel<ND, true> : run_large_kernel<ND, false>;
            if ((e = allow_smem(k, large_smem_floats(ITC_MAX_M, 1, ND) * sizeof(float))) != cudaSuccess) return e;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(large_ctas * csize));
            cfg.blockDim = dim3((unsigned)large_threads(csize > 1));
            cfg.dynamicSmemBytes = smem;
            cfg.stream = s;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = (unsigned)csize;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            if ((e = cudaLaunchKernelEx(&cfg, k, L)) != cudaSuccess) return e;
            if (!others) return cudaSuccess;
            if (L.groups) L.groups += (size_t)large_ctas * kGroupInts;
            smem = 0;
        }
    }
    if (ctas <= 0) return cudaSuccess;
    run_kernel<ND><<<ctas, kRunThreads, smem, s>>>(L);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_run(const RunLaunch& L, int large_ctas, int nlarge, int ctas, int max_M, double work, cudaStream_t s,
                       int ndim) {
    return ndim == 3 ? launch_nd<3>(L, large_ctas, nlarge, ctas, max_M, work, s)
                     : launch_nd<2>(L, large_ctas, nlarge, ctas, max_M, work, s);
}

}  // namespace itc
