// itc_backward.cu -- gradient of the Cauchy-Schwarz divergence, Eq. (1), with respect to the
// codebook and to the per-pixel weights of weighted ITC (Sec. 5).
//
//   dD/dw_{k,i} = (2 / rho_i^2) E_{k,i} / S_WW - (2 / tau_i^2) D_{k,i} / S_XW
//   dD/dh(x)    = 2 A_s(x) / S_XX - (2 / S_XW) sum_k g_tau(x - w_k) [x in box(round(w_k))]
// (tau = sigma: the data kernel and its fields; rho: the codebook pair kernel; A_s: the field of h
// at the width s of V(X); rho = s = tau unless set apart, and then A_s = A.)
//
// Kernel 1 (one CTA per image): a_k, D_k from the stored fields or, for a real-valued codebook, as
// window sums around round(w_k) read directly from the image (kernel evaluated at the real w_k, one
// warp per k), the M x M sums s_k, E_k (one thread per k), S_XW, S_WW, grad_W and two per-image
// scalars for kernel 2.
// Kernel 2 (per dimension; 16 x 64 or 16 x 16 pixel tiles of a warp in 2-D, 32 x 32 or 16 x 16 of a CTA in 3-D): the codebooks
// whose box meets a tile are taken in k order (ballots), their Gaussians are stamped onto the tile in
// that order -- the transposed form of the gather in the forward update -- and every pixel
// combines the stored field A with the stamp.
#include <math.h>

#include <algorithm>

#include "itc_internal.cuh"
#include "itc_pairs.cuh"

namespace itc {
namespace {

__device__ __forceinline__ float warp_sum_f(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_sum_d(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ int lattice_round_i(float x, int n) {
    float r = floorf(x + 0.5f);
    return (int)fminf(fmaxf(r, 0.f), (float)(n - 1));
}
__device__ __forceinline__ int pixel_gray(const ImageDesc& D, int u, int v) {
    return (int)__ldg(reinterpret_cast<const unsigned char*>(D.data) + (size_t)u * D.pitch + v);
}

// Dynamic shared floats of the codebook kernel: positions, z, then a (1), D (3), s (1), E (3) per vector
__host__ __device__ constexpr size_t codebook_smem_floats(int M) { return (size_t)((M + kPairPad - 1) / kPairPad * kPairPad) * 11; }

// a_k and D_k summed over the box around round(w_k) with the kernel at the real w_k, by the calling warp: a
// lane adds every 32nd position of the box in turn, the loads of eight of them in flight together and the
// next position found by adding (8 weight images of 256 x 256, M = 32, R = 9: 41 us with a division and a
// dependent load per position and four warps per image; 12 us now, with sixteen).  A lane per column
// instead takes the same time, but leaves sums of one sign in each lane: the error of grad_W was 1.03e-7,
// and is 8.3e-8 in this order.
template <int ND>
__device__ __forceinline__ void window_sums(const ImageDesc& D, float w0, float w1, float w2, float* sa, float* sD) {
    const int lane = threadIdx.x & 31;
    const int H = D.H, Wd = D.W, Ru = D.R[0], Rv = D.R[1], Rg = D.R[2];
    const float c0 = D.inv2s2[0], c1 = D.inv2s2[1], c2 = D.inv2s2[2];
    const int r0 = lattice_round_i(w0, H), r1 = lattice_round_i(w1, Wd), r2 = ND == 3 ? lattice_round_i(w2, D.G) : 0;
    const int ua = max(0, r0 - Ru), ub = min(H - 1, r0 + Ru), va = max(0, r1 - Rv), vb = min(Wd - 1, r1 + Rv);
    const int nv = vb - va + 1, npos = (ub - ua + 1) * nv;
    const int su = 32 / nv, sv = 32 - su * nv;   // 32 positions on, as rows and columns
    int u = ua + lane / nv, v = va + lane % nv;
    float a = 0.f, d0 = 0.f, d1 = 0.f, d2 = 0.f;
    auto sums = [&](auto* h) {   // h: weights (null: ones); unconditional loads from clamped places
        int p = lane;
        auto block = [&](auto steps) {
            constexpr int U = decltype(steps)::value;
            float x[U], du[U], dv[U], gl[U];
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const size_t o = (size_t)min(u, ub) * D.pitch + v;
                x[q] = h ? (float)__ldg(h + o) : 1.f;
                gl[q] = ND == 3 ? (float)__ldg(reinterpret_cast<const unsigned char*>(D.data) + o) : 0.f;
                du[q] = (float)u - w0;
                dv[q] = (float)v - w1;
                u += su;
                v += sv;
                if (v > vb) {
                    v -= nv;
                    ++u;
                }
            }
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const float dg = ND == 3 ? gl[q] - w2 : 0.f;
                float e = du[q] * du[q] * c0 + dv[q] * dv[q] * c1;
                if (ND == 3) e += dg * dg * c2;
                const bool in = p + 32 * q < npos && x[q] != 0.f && (ND == 2 || fabsf(gl[q] - (float)r2) <= (float)Rg);
                const float g = in ? x[q] * expf(-e) : 0.f;
                a += g;
                d0 = fmaf(g, du[q], d0);
                d1 = fmaf(g, dv[q], d1);
                if (ND == 3) d2 = fmaf(g, dg, d2);
            }
            p += 32 * U;
        };
        // eight loads in flight, four where no more are left (10000 images of up to 16 px, whose boxes have
        // 36 to 256 positions, M = 64: 568 us with eight throughout)
        while (p - lane + 4 * 32 < npos) block(std::integral_constant<int, 8>());
        if (p - lane < npos) block(std::integral_constant<int, 4>());
    };
    if (ND == 3) sums(D.weight);
    else if (D.dtype == ITC_U8) sums(reinterpret_cast<const unsigned char*>(D.data));
    else sums(reinterpret_cast<const float*>(D.data));
    a = warp_sum_f(a);
    d0 = warp_sum_f(d0);
    d1 = warp_sum_f(d1);
    d2 = warp_sum_f(d2);
    if (lane == 0) {
        sa[0] = a;
        sD[0] = d0;
        sD[1] = d1;
        sD[2] = d2;
    }
}

template <int ND>
__device__ __forceinline__ void codebook_image(const BackwardLaunch& L, const ImageDesc& D, int img) {
    const int M = D.M, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nw = blockDim.x >> 5, mp = (M + kPairPad - 1) / kPairPad * kPairPad;
    extern __shared__ __align__(16) float sm[];
    float* sxy = sm;             // positions in pairs (pair_sums), padded
    float* sz = sxy + 2 * mp;
    float* sa = sz + mp;
    float* sD = sa + mp;         // 3 per vector
    float* ss = sD + 3 * mp;
    float* sE = ss + mp;
    __shared__ double red[4], coef[6];
    __shared__ double s_px[32];

    // S_XX from the image's tile partials: warp 0 alone, or for a gray image (a partial per
    // slice tile) the first four warps a strided share each with eight loads in flight per lane, the
    // warp sums added in warp order
    const int nws = ND == 3 ? kRunThreads / 32 : 1;
    if (wid < nws) {
        const long long nt = D.sxx_tiles, step = 32LL * nws;
        double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        long long i = tid;
        for (; i + 7 * step < nt; i += 8 * step)
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] += L.partials[D.sxx_off + i + q * step];
        for (; i < nt; i += step) v[0] += L.partials[D.sxx_off + i];
        const double t = warp_sum_d(((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])));
        if (lane == 0) s_px[wid] = t;
    }
    const float* Wk = L.W + D.w_off;
    const int n[3] = {D.H, D.W, D.G};
    int off_lattice = 0;
    for (int k = tid; k < mp; k += blockDim.x) {
        float w[3] = {kFar, kFar, kFar};
        if (k < M) {
#pragma unroll
            for (int i = 0; i < ND; ++i) {
                w[i] = Wk[k * ND + i];
                off_lattice |= (w[i] != rintf(w[i])) || !(w[i] >= 0.f) || !(w[i] <= (float)(n[i] - 1));
            }
        }
        sxy[(k >> 1) * 4 + (k & 1)] = w[0];
        sxy[(k >> 1) * 4 + 2 + (k & 1)] = w[1];
        sz[k] = w[2];
    }
    // a_k and D_k: on the lattice (every w_k integral and inside it) they are the stored field
    // values at w_k; otherwise window sums around round(w_k) with the kernel at the real w_k
    const bool gather = !__syncthreads_or(off_lattice);
    auto at = [&](int k, int i) { return i == 2 ? sz[k] : sxy[(k >> 1) * 4 + 2 * i + (k & 1)]; };
    if (!gather)
        for (int k = wid; k < M; k += nw) window_sums<ND>(D, at(k, 0), at(k, 1), at(k, 2), sa + k, sD + 3 * k);
    // codebook interaction sums: one thread per k, the gathers in flight beside them
    const PairWidths<ND> pw(D);
    const float* A = L.fields + D.field_off;
    for (int k = tid; k < M; k += blockDim.x) {
        float w[ND], E[ND], s, a = 0.f, f[ND];
#pragma unroll
        for (int i = 0; i < ND; ++i) w[i] = at(k, i);
        if (gather) {
            const long long o = ((long long)(ND == 3 ? (int)w[ND - 1] : 0) * D.H + (int)w[0]) * D.fpitch + (int)w[1];
            a = __ldg(A + o);
#pragma unroll
            for (int i = 0; i < ND; ++i) f[i] = __ldg(A + (i + 1) * D.plane_floats + o);
        }
        // equal widths share a product where the positions are on the lattice, which makes it exact
        if (ND == 2 && pw.iso && gather) pair_sums<ND, ND == 2>(sxy, sz, mp, w, pw.nc, s, E);
        else pair_sums<ND, false>(sxy, sz, mp, w, pw.nc, s, E);
        ss[k] = s;
        if (gather) sa[k] = a;
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            sE[k * 3 + i] = E[i];
            if (gather) sD[k * 3 + i] = f[i];
        }
    }
    __syncthreads();
    const double gD = L.grad_dcs ? (double)L.grad_dcs[img] : 1.0;
    if (wid == 0) {
        double x = 0, y = 0;
        int e = 0;
        for (int k = lane; k < M; k += 32) {
            x += (double)sa[k];
            y += (double)ss[k];
            e += !(sa[k] > 0.f);
        }
        x = warp_sum_d(x);
        y = warp_sum_d(y);
        e = __reduce_add_sync(0xffffffffu, e);
        // on a lane each: the coefficients of E and D in grad_W per axis, and of the two terms of grad_h
        double sxx = 0;
        for (int q = 0; q < nws; ++q) sxx += s_px[q];   // written before the barriers above
        const int i = lane < 6 ? lane % 3 : 0;
        const double width = lane < 3 ? (double)D.rho[i] : (double)D.sigma[i];
        const double den = lane < 3 ? width * width * y : (lane < 6 ? width * width * x : (lane == 6 ? sxx : x));
        const double c = 2.0 * gD / den;
        if (lane < 6) coef[lane] = c;
        if (lane == 6) L.scal[img * 4 + 0] = c;
        if (lane == 7) L.scal[img * 4 + 1] = c;
        if (lane == 0) {
            red[0] = x;
            red[1] = y;
            red[2] = (double)e;
            red[3] = sxx;
        }
    }
    __syncthreads();
    if (L.grad_W) {
        float* gW = L.grad_W + D.w_off;
        for (int k = tid; k < M; k += blockDim.x)
#pragma unroll
            for (int i = 0; i < ND; ++i)
                gW[k * ND + i] = (float)(coef[i] * (double)sE[k * 3 + i] - coef[3 + i] * (double)sD[k * 3 + i]);
    }
    if (tid == 0 && L.stats) {
        const double sxw = red[0], sww = red[1], sxx = red[3];
        itc_stats r;
        r.sxw = sxw;
        r.sww = sww;
        r.sxx = sxx;
        r.c = sxw / sww;
        r.dcs = sxw > 0 ? log(sww) + log(sxx) - 2.0 * log(sxw) + D.dcs_const : INFINITY;
        r.empty = (int)red[2];
        r.moved = 0;
        r.iters_done = 0;
        const int dev_status = L.img_status ? L.img_status[img] : ITC_OK;
        r.status = dev_status == ITC_ERR_TIMEOUT ? ITC_ERR_TIMEOUT
                   : (!(sxw > 0) || !isfinite(r.dcs) ? ITC_ERR_NONFINITE
                      : (r.empty > 0 ? ITC_WARN_EMPTY_SUPPORT : ITC_OK));
        L.stats[img] = r;
    }
}

constexpr int kCodebookThreads = 512;   // most threads of a codebook CTA

__global__ void __launch_bounds__(kCodebookThreads, 1) bwd_codebook_kernel(const __grid_constant__ BackwardLaunch L) {
    const int img = L.img_base + blockIdx.x;
    const ImageDesc& D = L.descs[img];
    if (D.ndim == 3) codebook_image<3>(L, D, img);
    else codebook_image<2>(L, D, img);
}

constexpr int kPixWarps = 4;    // warps of a 2-D pixel CTA
constexpr int kPixRows = kBwdStrip;   // rows of a warp's tile
constexpr int kPixSlots = 16;   // codebook vectors staged per turn

// 2-D pixel pass.  The stamp S(x) = sum_k g(x - w_k) [x in box(round(w_k))] is separable:
// g(x - w) = g_u(x_u - w_u) g_v(x_v - w_v) and the box is a product of two intervals, so for the vectors
// whose box meets a tile, taken in k order,
//   S(r, c) = sum_l a_l(r) b_l(c),  a_l(r) = g_u(u0 + r - w_lu) [|u0 + r - r_lu| <= R_u], ...
// Every warp walks 16 x 64 tiles of its image on its own: it loads the field (a lane has 8 rows x 4
// columns), finds the vectors by ballot, stages a and b of up to 16 of them in its own shared memory and adds
// them in l order with packed FMAs over pairs of rows (deterministic, no atomics).  HBM bounds it: 4 bytes
// read and 4 written per pixel.  Nothing waits for other warps, so that 20 of them per SM keep loads in flight
// (64 x 64 tiles of a CTA with a barrier per phase: 113 us for 256 images of 512 x 512, 6.3 TB/s in 85 us now;
// 589 and 464 us for 4096 ragged images).  Row pieces of 256 bytes: fields and gradients of ragged images start
// anywhere in a 128-byte line, and with 32 x 32 tiles the shared lines cost 514 us.
// COLS 16: where a batch has too few tiles for all warps, the chain of a warp over the vectors is the time of
// the pass, and 16 x 16 tiles (4 x 2 per lane) make a vector's step shorter.  Every pixel adds the same products in
// the same order (39 images of 16 x 16, 300 vectors, the whole backward: 62 us, 77 with 16 x 64 tiles).
template <int COLS>
__global__ void __launch_bounds__(32 * kPixWarps, 5) bwd_pixels2d_kernel(const __grid_constant__ BackwardLaunch L) {
    // split CTAs per image: the warps take its tiles in turn
    const int split = L.split;
    const int img = L.bwd_order ? __ldg(L.bwd_order + blockIdx.x / split) : L.img_base + (int)(blockIdx.x / split);
    const ImageDesc& D = L.descs[img];
    if (D.ndim != 2) return;
    const int M = D.M, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int RB = COLS == 64 ? 8 : 4, CB = COLS == 64 ? 4 : 2;   // a lane's rows and columns of a tile
    constexpr int STAGE = kPixRows + COLS;                             // floats of a staged vector: a, then b
    static_assert(kPixRows / RB * (COLS / CB) == 32, "a lane's block");
    const int H = D.H, Wd = D.W, fpitch = D.fpitch, Ru = D.R[0], Rv = D.R[1];
    const int tiles_v = (Wd + COLS - 1) / COLS, ntiles = tiles_v * ((H + kPixRows - 1) / kPixRows);
    const int first = (int)(blockIdx.x % split) * kPixWarps;
    if (first >= ntiles) return;
    // the separable factors exp(-d^2 c) = 2^(-d^2 c log2 e), log2 e folded into the widths
    const float l0 = (float)(1.4426950408889634 * (double)D.inv2s2[0]), l1 = (float)(1.4426950408889634 * (double)D.inv2s2[1]);
    // the S_XX term uses the field of h at the width of V(X): A itself unless set apart
    const float* A = L.fields + (D.self_off >= 0 ? D.self_off : D.field_off);
    float* gh = L.grad_h + D.gh_off;
    const float s1 = (float)L.scal[img * 4 + 0], s2 = (float)L.scal[img * 4 + 1];

    extern __shared__ __align__(16) unsigned char bsm[];
    float4* rec = reinterpret_cast<float4*>(bsm);   // per vector: position and site along u and v
    __shared__ __align__(16) float stage[kPixWarps][kPixSlots][STAGE];
    const float* Wk = L.W + D.w_off;
    for (int k = tid; k < M; k += blockDim.x) {
        const float w0 = Wk[k * 2], w1 = Wk[k * 2 + 1];
        rec[k] = make_float4(w0, w1, __int_as_float(lattice_round_i(w0, H)), __int_as_float(lattice_round_i(w1, Wd)));
    }
    __syncthreads();

    static_assert(kPixSlots * STAGE >= kPixRows * COLS, "a warp's stage holds a tile");
    float(*st)[STAGE] = stage[wid];
    const int br = lane / (COLS / CB) * RB, bc = lane % (COLS / CB) * CB;   // a lane's block of a tile
    const bool rows16 = (Wd & 3) == 0 && (reinterpret_cast<size_t>(gh) & 15) == 0;
    using Piece = std::conditional_t<CB == 4, float4, float2>;
    for (int t = first + wid; t < ntiles; t += split * kPixWarps) {
        const int u0 = t / tiles_v * kPixRows, v0 = (t - t / tiles_v * tiles_v) * COLS;
        const int u = u0 + lane, v = v0 + lane, nrow = min(kPixRows, H - u0);
        // this lane's block of the field, loaded first so that its latency overlaps the stamp
        union { Piece v; float e[CB]; } f[RB];
        {
            const float* p = A + min(v0 + bc, fpitch - CB);
#pragma unroll
            for (int i = 0; i < RB; ++i) f[i].v = __ldg(reinterpret_cast<const Piece*>(p + (size_t)min(u0 + br + i, H - 1) * fpitch));
        }
        float2 acc[RB / 2][CB];   // row pairs, columns
#pragma unroll
        for (int i = 0; i < RB / 2; ++i)
#pragma unroll
            for (int j = 0; j < CB; ++j) acc[i][j] = make_float2(0.f, 0.f);
        const float fu = (float)u, fv = (float)v;
        int ns = 0;
        auto add = [&] {
            __syncwarp();
#pragma unroll 1
            for (int l = 0; l < ns; ++l) {
                union { Piece v; float e[CB]; } b;
                b.v = *reinterpret_cast<const Piece*>(&st[l][kPixRows + bc]);
                float2 a[RB / 2];
#pragma unroll
                for (int i = 0; i < RB / 2; i += 2) {
                    const float4 a4 = *reinterpret_cast<const float4*>(&st[l][br + 2 * i]);
                    a[i] = make_float2(a4.x, a4.y);
                    a[i + 1] = make_float2(a4.z, a4.w);
                }
#pragma unroll
                for (int j = 0; j < CB; ++j)
#pragma unroll
                    for (int i = 0; i < RB / 2; ++i) acc[i][j] = __ffma2_rn(a[i], make_float2(b.e[j], b.e[j]), acc[i][j]);
            }
            __syncwarp();
            ns = 0;
        };
        for (int base = 0; base < M; base += 32) {
            bool hit = false;
            if (base + lane < M) {
                const float4 r = rec[base + lane];
                const int r0 = __float_as_int(r.z), r1 = __float_as_int(r.w);
                hit = r0 + Ru >= u0 && r0 - Ru < u0 + kPixRows && r1 + Rv >= v0 && r1 - Rv < v0 + COLS;
            }
            unsigned bal = __ballot_sync(0xffffffffu, hit);
            while (bal) {
                const float4 r = rec[base + __ffs(bal) - 1];
                bal &= bal - 1;
                if constexpr (COLS == 16) {   // the rows' factors on the first lanes, the columns' on the others
                    const bool row = lane < kPixRows;
                    const int x = row ? u : v - kPixRows;
                    const float d = (float)x - (row ? r.x : r.y);
                    const int site = __float_as_int(row ? r.z : r.w);
                    st[ns][lane] = abs(x - site) <= (row ? Ru : Rv) ? ex2_ftz(-(d * d) * (row ? l0 : l1)) : 0.f;
                } else {
                    const float du = fu - r.x, dv = fv - r.y;
                    const float dv2 = (float)(v + 32) - r.y;
                    if (lane < kPixRows) st[ns][lane] = abs(u - __float_as_int(r.z)) <= Ru ? ex2_ftz(-(du * du) * l0) : 0.f;
                    st[ns][kPixRows + lane] = abs(v - __float_as_int(r.w)) <= Rv ? ex2_ftz(-(dv * dv) * l1) : 0.f;
                    st[ns][kPixRows + 32 + lane] = abs(v + 32 - __float_as_int(r.w)) <= Rv ? ex2_ftz(-(dv2 * dv2) * l1) : 0.f;
                }
                if (++ns == kPixSlots) add();
            }
        }
        if (ns) add();
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const float* q = &acc[i >> 1][0].x + (i & 1);
#pragma unroll
            for (int j = 0; j < CB; ++j) f[i].e[j] = s1 * f[i].e[j] - s2 * q[2 * j];
        }
        if (rows16) {
            float* out = gh + (size_t)(u0 + br) * Wd + v0 + bc;
#pragma unroll
            for (int i = 0; i < RB; ++i)
                if (v0 + bc < Wd && br + i < nrow) *reinterpret_cast<Piece*>(out + (size_t)i * Wd) = f[i].v;
            continue;
        }
        // rows on any boundary: through the warp's shared memory, a row piece to each store
        float* tile = &st[0][0];
#pragma unroll
        for (int i = 0; i < RB; ++i) *reinterpret_cast<Piece*>(tile + (br + i) * COLS + bc) = f[i].v;
        __syncwarp();
        if constexpr (COLS == 16) {
#pragma unroll
            for (int i = 0; i < kPixRows; i += 2) {   // two rows at a time
                const int r = i + (lane >> 4), c = lane & 15;
                if (r < nrow && v0 + c < Wd) gh[(size_t)(u0 + r) * Wd + v0 + c] = tile[r * COLS + c];
            }
        } else {
            float* out = gh + (size_t)u0 * Wd + v;
            const bool in0 = v < Wd, in1 = v + 32 < Wd;
            if (nrow == kPixRows) {
#pragma unroll
                for (int i = 0; i < kPixRows; ++i, out += Wd) {
                    if (in0) out[0] = tile[i * COLS + lane];
                    if (in1) out[32] = tile[i * COLS + 32 + lane];
                }
            } else {
                for (int i = 0; i < nrow; ++i, out += Wd) {
                    if (in0) out[0] = tile[i * COLS + lane];
                    if (in1) out[32] = tile[i * COLS + 32 + lane];
                }
            }
        }
        __syncwarp();
    }
}

constexpr int kChunk = 64;   // codebooks staged per round in the 3-D pixel kernel

// 3-D pixel pass: a CTA walks T x T tiles of its image (images with the most tiles are launched first).  The
// codebooks whose box meets the tile are listed in k order; chunks of 64 of them are staged as a (64 x T) and
// b (64 x T) in shared memory and every thread accumulates a T / 16 square of pixels in l order.  The g factor
// depends on each pixel's gray level and is applied per pixel and codebook, so the pass is bound by its chain
// of exponentials where there are few pixels.  T = 32, or 16 where tiles of 32 would not fill the GPU: one
// 256 x 256 image with 64 vectors 21 us at T = 64, 6.4 at 32, 4.5 at 16; 16 of them 31, 20 and 29.
template <int T>
__global__ void __launch_bounds__(kThreads, 3) bwd_pixels3d_kernel(const __grid_constant__ BackwardLaunch L) {
    // split CTAs per image (few large images): CTA s of an image takes its tiles s, s + split, ...
    const int split = L.split;
    const int img = L.bwd_order ? __ldg(L.bwd_order + blockIdx.x / split) : L.img_base + (int)(blockIdx.x / split);
    const int part = blockIdx.x % split;
    const ImageDesc& D = L.descs[img];
    if (D.ndim != 3) return;
    const int M = D.M, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int H = D.H, Wd = D.W, G = D.G, fpitch = D.fpitch, tiles_v = (Wd + T - 1) / T;
    const int ntiles = tiles_v * ((H + T - 1) / T);
    const int Ru = D.R[0], Rv = D.R[1], Rg = D.R[2];
    const float c0 = D.inv2s2[0], c1 = D.inv2s2[1], c2 = D.inv2s2[2];
    // the separable factors exp(-d^2 c) = 2^(-d^2 c log2 e), log2 e folded into the widths
    const float l0 = (float)(1.4426950408889634 * (double)c0), l1 = (float)(1.4426950408889634 * (double)c1);
    // the S_XX term uses the field of h at the width of V(X): A itself unless set apart
    const float* A = L.fields + (D.self_off >= 0 ? D.self_off : D.field_off);
    float* gh = L.grad_h + D.gh_off;
    const float s1 = (float)L.scal[img * 4 + 0], s2 = (float)L.scal[img * 4 + 1];
    extern __shared__ __align__(16) unsigned char bsm[];
    // per listed codebook of the current tile one 16-byte record (position and site along u
    // and v), then the codebooks' positions, sites and the list itself
    float4* lc = reinterpret_cast<float4*>(bsm);
    float* cw = reinterpret_cast<float*>(lc + M);       // M x 3 codebook positions
    int* cr = reinterpret_cast<int*>(cw + 3 * M);       // M x 3 rounded lattice sites
    int* lk = cr + 3 * M;                               // listed codebooks of the current tile
    __shared__ __align__(16) float sa[kChunk][T];
    __shared__ __align__(16) float sb[kChunk][T];
    __shared__ __align__(16) int wcount[kThreads / 32];

    const float* Wk = L.W + D.w_off;
    for (int k = tid; k < M; k += blockDim.x) {
        const float w0 = Wk[k * 3], w1 = Wk[k * 3 + 1], w2 = Wk[k * 3 + 2];
        cw[k * 3] = w0;
        cw[k * 3 + 1] = w1;
        cw[k * 3 + 2] = w2;
        cr[k * 3] = lattice_round_i(w0, H);
        cr[k * 3 + 1] = lattice_round_i(w1, Wd);
        cr[k * 3 + 2] = lattice_round_i(w2, G);
    }
    __syncthreads();

    constexpr int P = T / 16;   // this thread's P x P block
    const int pr = (tid >> 4) * P, pc = (tid & 15) * P;
    if (part >= ntiles) return;
    for (int t = part; t < ntiles; t += split) {
        const int u0 = (t / tiles_v) * T, v0 = (t % tiles_v) * T;
        int gray[P][P];
        const bool cols_in = v0 + pc < Wd;
#pragma unroll
        for (int i = 0; i < P; ++i)
#pragma unroll
            for (int j = 0; j < P; ++j) {
                const int u = u0 + pr + i, v = v0 + pc + j;
                gray[i][j] = (u < H && v < Wd) ? pixel_gray(D, u, v) : 0;
            }

        // stable compaction of the codebooks whose box meets this tile
        int nl = 0;
        for (int base = 0; base < M; base += blockDim.x) {
            const int k = base + tid;
            bool hit = false;
            if (k < M) {
                const int r0 = cr[k * 3], r1 = cr[k * 3 + 1];
                hit = (r0 + Ru >= u0) && (r0 - Ru <= u0 + T - 1) &&
                      (r1 + Rv >= v0) && (r1 - Rv <= v0 + T - 1);
            }
            const unsigned bal = __ballot_sync(0xffffffffu, hit);
            if (lane == 0) wcount[wid] = __popc(bal);
            __syncthreads();
            static_assert(kThreads / 32 == 8, "eight warp counts");
            const int4 wc0 = *reinterpret_cast<const int4*>(wcount), wc1 = *reinterpret_cast<const int4*>(wcount + 4);
            const int cnt[8] = {wc0.x, wc0.y, wc0.z, wc0.w, wc1.x, wc1.y, wc1.z, wc1.w};
            int off = nl, tot = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                off += q < wid ? cnt[q] : 0;
                tot += cnt[q];
            }
            if (hit) {
                const int pos = off + __popc(bal & ((1u << lane) - 1u));
                lk[pos] = k;
                lc[pos] = make_float4(cw[k * 3], cw[k * 3 + 1], __int_as_float(cr[k * 3]), __int_as_float(cr[k * 3 + 1]));
            }
            nl += tot;
            __syncthreads();
        }

        float acc[P][P] = {};
        // factor staging: each thread fills one row / column r of the factors for every fourth l
        const int sr = tid & (T - 1), sl = tid / T;
        static_assert(kThreads % T == 0, "whole rows of threads");
        constexpr int kStageStep = kThreads / T;
        const int su = u0 + sr, sv = v0 + sr;
        const bool su_in = su < H, sv_in = sv < Wd;
        const float fu = (float)su, fv = (float)sv;
        for (int base = 0; base < nl; base += kChunk) {
            const int nc = min(kChunk, nl - base);
            for (int l = sl; l < nc; l += kStageStep) {
                const float4 rec = lc[base + l];
                float av = 0.f, bv = 0.f;
                if (su_in && abs(su - __float_as_int(rec.z)) <= Ru) { const float d = fu - rec.x; av = ex2_ftz(-(d * d) * l0); }
                if (sv_in && abs(sv - __float_as_int(rec.w)) <= Rv) { const float d = fv - rec.y; bv = ex2_ftz(-(d * d) * l1); }
                sa[l][sr] = av;
                sb[l][sr] = bv;
            }
            __syncthreads();
            for (int l = 0; l < nc; ++l) {
                float av[P], bv[P];
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    av[i] = sa[l][pr + i];
                    bv[i] = sb[l][pc + i];
                }
                const int k = lk[base + l];
                const float wg = cw[k * 3 + 2];
                const int rg = cr[k * 3 + 2];
#pragma unroll
                for (int i = 0; i < P; ++i)
#pragma unroll
                    for (int j = 0; j < P; ++j) {
                        const int gl = gray[i][j];
                        if (abs(gl - rg) <= Rg) {
                            const float d = (float)gl - wg;
                            acc[i][j] = fmaf(av[i] * bv[j], expf(-d * d * c2), acc[i][j]);
                        }
                    }
            }
            __syncthreads();   // sa / sb are rewritten by the next chunk or tile
        }
        if (!cols_in) continue;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const int u = u0 + pr + i;
            if (u >= H) break;
            float* out = gh + (long long)u * Wd + v0 + pc;
            {
#pragma unroll
                for (int j = 0; j < P; ++j) {
                    const int v = v0 + pc + j;
                    if (v >= Wd) break;
                    if (gray[i][j] >= G) {   // a voxel outside the lattice: no field value
                        out[j] = 0.f;
                        continue;
                    }
                    const long long o = ((long long)gray[i][j] * H + u) * fpitch + v;
                    out[j] = s1 * __ldg(A + o) - s2 * acc[i][j];
                }
            }
        }
    }
}

}  // namespace

cudaError_t launch_backward(const BackwardLaunch& L, int B, int max_M, long long pixel_tiles, int max_image_tiles,
                            int ndim_mask, cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    const size_t smem1 = codebook_smem_floats(max_M) * sizeof(float);
    cudaError_t e = allow_smem(bwd_codebook_kernel, codebook_smem_floats(ITC_MAX_M) * sizeof(float));
    if (e != cudaSuccess) return e;
    // few images: as many threads as keep a CTA's window sums and pair sums short
    bwd_codebook_kernel<<<B, B <= kSoloImages ? kCodebookThreads : kRunThreads, smem1, s>>>(L);
    e = cudaGetLastError();
    if (e != cudaSuccess || !L.grad_h || pixel_tiles <= 0) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    // each image's tiles are shared out over `split` CTAs: as many as fill the GPU, and up to `waves` times
    // that while an image's CTAs still have four times a tile for each warp (a batch's large images then
    // end together, and neighbouring tiles run at the same time: 4096 ragged images 541 us with a CTA each,
    // 514 with two; 256 of 512 x 512 127 us with three, 86 with sixteen)
    auto launch = [&](auto* kernel, int threads, size_t per_vector, long long waves, long long most) {
        int per_sm = 0;
        const size_t smem = (size_t)max_M * per_vector;
        e = allow_smem(kernel, ITC_MAX_M * per_vector);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
        if (e != cudaSuccess) return;
        const long long slots = (long long)sms * std::max(per_sm, 1);
        BackwardLaunch L2 = L;
        L2.split = (int)std::max({1LL, std::min((slots + B - 1) / B, most), waves > 1 ? std::min((slots * waves + B - 1) / B, most / 4) : 1LL});
        kernel<<<(unsigned)(B * (long long)L2.split), threads, smem, s>>>(L2);
        e = cudaGetLastError();
    };
    if (ndim_mask & 4) {
        // of 20 warps per SM; many vectors make the chain longer, few do not repay the shorter row pieces (244
        // images of 64 x 64, 976 strips: with 2, 16, 64 and 300 vectors 20.5, 22.3, 29.5 and 76.9 us in strips and
        // 21.6, 23.5, 29.9 and 67.7 in 16 x 16 tiles; 1952 strips, 300 vectors: 91 and 108)
        static_assert(kBwdStrip == kPixRows && kBwdTileW == 64, "a strip is a warp's tile");
        if (2 * L.strips <= (max_M > 64 ? 20LL : 10LL) * sms)
            launch(bwd_pixels2d_kernel<16>, 32 * kPixWarps, sizeof(float4), 1, 4LL * max_image_tiles);
        else
            launch(bwd_pixels2d_kernel<64>, 32 * kPixWarps, sizeof(float4), 6, max_image_tiles);
    }
    if (e == cudaSuccess && (ndim_mask & 8)) {   // list records, positions, sites, tile list
        constexpr size_t per_vector = 16 + 7 * sizeof(int);
        if (4 * pixel_tiles < 3LL * sms) launch(bwd_pixels3d_kernel<16>, kThreads, per_vector, 1, 16LL * max_image_tiles);
        else launch(bwd_pixels3d_kernel<32>, kThreads, per_vector, 1, 4LL * max_image_tiles);
    }
    return e;
}

}  // namespace itc
