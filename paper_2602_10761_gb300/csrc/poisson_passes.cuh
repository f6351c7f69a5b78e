// The split passes of the Poisson solve for compile-time transform lengths
// (x forward, z forward, y solve, z inverse, x inverse; Sec. 2.2 Poisson
// equation, second-order finite volumes of Sec. 3.1): kernels, their shared
// memory sizes and the list of compiled lengths.  The x and z transforms are
// instantiated and launched by poisson_x32/x64/z32/z64.cu (one translation
// unit per direction and precision, so that they compile side by side), the y
// solves by poisson_fast.cu and poisson_group.cu.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "fft.cuh"
#include "fft_reg.cuh"
#include "tribo_internal.cuh"

namespace tribo {
namespace {

constexpr int kThreads = 256;

// resident blocks per SM that leave a transform of length N room for the larger factor's values
// in registers (2 sizeof(R)/4 registers a value, and as many for the pass in flight): 64 registers
// a thread hold 16 FP32 or 8 FP64 values, 128 hold twice as many
template <class R, int N>
constexpr int fft_min_blocks() {
    return fft::FourStep<N, kThreads>::N2 * (int)sizeof(R) <= 64 ? 4
           : fft::FourStep<N, kThreads>::N2 * (int)sizeof(R) <= 128 ? 2 : 1;
}

// ---------------------------------------------------------------- double-single
struct ds {
    float hi, lo;
};
// Knuth's two-sum: s + e == a + b exactly
__device__ __forceinline__ ds two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    const float e = (a - (s - bb)) + (b - bb);
    return {s, e};
}
// Dekker's fast two-sum, |a| >= |b|
__device__ __forceinline__ ds fast_two_sum(float a, float b) {
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ ds ds_mul(ds a, ds b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return fast_two_sum(p, e);
}
__device__ __forceinline__ float ds_f(ds a) { return a.hi + a.lo; }

// ---------------------------------------------------------------- real transforms' split step
// Inverse: the half-length value Z_m of a real line from X_m = xa and X_M-m = xb,
//   Z = (xa + conj xb) + i conj(W^m) (xa - conj xb), w = W^m = exp(-2 pi i m / N),
// four additions and four fused multiply-adds (transforms in FP64 are bound by
// the FP64 pipe: operations are time).
template <class R>
__device__ __forceinline__ cplx<R> split_inv(cplx<R> xa, cplx<R> xb, cplx<R> w) {
    const R sr = xa.re + xb.re, si = xa.im - xb.im, dr = xa.re - xb.re, di = xa.im + xb.im;
    return {sr - w.re * di + w.im * dr, si + w.re * dr + w.im * di};
}
// the same of -i s X (s = sin(2 pi m / N) / dx, equal for m and M - m): E_x's spectrum from the potential's
template <class R>
__device__ __forceinline__ cplx<R> split_inv_dx(cplx<R> xa, cplx<R> xb, cplx<R> w, R s) {
    const R sr = xa.re + xb.re, si = xa.im - xb.im, dr = xa.re - xb.re, di = xa.im + xb.im;
    return {s * (di + w.re * sr + w.im * si), s * (w.re * si - w.im * sr - dr)};
}

// ---------------------------------------------------------------- x forward
// Thread group (line, r) per line (k, j) of the charge-sum array:
// z_n = x_2n + i x_2n+1 (scaled to -rho/eps), Z = FFT_M(z) by the register
// four-step, X_m = (Z_m + conj Z_M-m) - i W^m (Z_m - conj Z_M-m) for m = 0..M
// (the halves of the split step and the normalisation 1/(nx nz) of the inverse
// transforms are in the scale), X_m and X_M-m from one sum and product.  Each thread zeroes the charge sums it has read.  The source has
// type QT: the FP64 cell charge sums (or a caller's FP64 density), rounded to
// R as they are read, or the adjoint's R-typed charge adjoint.
// Bound by HBM.  Six resident blocks (40 registers) for FP32 factors up to 16 and M <= 192, one
// otherwise: 85 us against 115 at 384x256x256, 37 against 44 at 288x145x162, 58 against 68 at 256^3,
// although M = 192 and 144 spill 8 to 32 bytes so (the channel-table forms of 36 and 48 also 4 to 8).
// M = 256, with the same factor, runs with one.
template <class R, int M>
constexpr int xfwd_min_blocks() { return sizeof(R) == 4 && M <= 192 && fft::FourStep<M, kThreads>::N2 <= 16 ? 6 : 1; }

// whether v is not +-0: on the bits, as a comparison of doubles would go to the FP64 pipe
__device__ __forceinline__ bool is_nonzero(float v) { return v != 0.0f; }
__device__ __forceinline__ bool is_nonzero(double v) {
    return (((unsigned)__double2hiint(v) << 1) | (unsigned)__double2loint(v)) != 0u;
}

template <class R, int M, class QT, bool kTab = false>
__global__ void __launch_bounds__(kThreads, xfwd_min_blocks<R, M>()) k_xfwd4(QT* __restrict__ src, const double* __restrict__ scale_row,
                                                    int zero_src, cplx<R>* __restrict__ S, int ny, int nlines,
                                                    const cplx<R>* __restrict__ tw_g,
                                                    const FastTab<R>* __restrict__ tab) {
    pdl_wait();
    if constexpr (kTab) {
        const FastTab<R>& t = tab[blockIdx.y];
        src = reinterpret_cast<QT*>(t.src);
        scale_row = t.scale;
        S = t.S;
        tw_g = t.twx;
    }
    using F4 = fft::FourStep<M, kThreads>;
    constexpr int N1 = F4::N1, N2 = F4::N2, TPC = F4::TPC, LPB = F4::W, CS = F4::CS;
    constexpr int NX = 2 * M, NXH = M + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<R>* tw = reinterpret_cast<cplx<R>*>(smem_raw);   // exp(-2 pi i e / NX)
    cplx<R>* buf = tw + NX;
    const int r = threadIdx.x % TPC;
    const int l = threadIdx.x / TPC;
    const int line = blockIdx.x * LPB + l;
    const bool live = l < LPB && line < nlines;
    cplx<R>* lb = buf + l * CS;
    // the line's sums are loaded (and the nonzero ones rewritten with zero) before the block
    // fills its twiddle table, so that the table's round trip overlaps the loads
    cplx<R> y[N1];
    if (live && r < N2) {
        R s, s_lo = 0;               // the row's factor
        if constexpr (sizeof(R) == 4) {
            const float2 v = reinterpret_cast<const float2*>(scale_row)[line % ny];
            s = v.x;
            s_lo = v.y;
        } else {
            s = scale_row[line % ny];
        }
        using V2 = std::conditional_t<sizeof(QT) == 8, double2, float2>;   // (x_2n, x_2n+1)
        V2* row = reinterpret_cast<V2*>(src) + (size_t)line * M;
        unsigned nz_mask = 0;        // which element pairs hold a nonzero sum
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) {
            const V2 v = row[N2 * n1 + r];
            nz_mask |= is_nonzero(v.x) | is_nonzero(v.y) ? 1u << n1 : 0u;
            const R a = from_f64<R>(v.x), b = from_f64<R>(v.y);
            if constexpr (sizeof(R) == 4) y[n1] = cplx<R>{fmaf(a, s, a * s_lo), fmaf(b, s, b * s_lo)};
            else y[n1] = cplx<R>{a * s, b * s};
        }
        if (zero_src) {
            // most cells hold no particle: only pairs with a nonzero sum are rewritten, so the
            // sectors of empty cells stay clean in L2 and are never written back
            V2 zero;
            zero.x = (QT)0;
            zero.y = (QT)0;
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1)
                if (nz_mask & (1u << n1)) row[N2 * n1 + r] = zero;
        }
    }
    for (int i = threadIdx.x; i < NX; i += kThreads) tw[i] = tw_g[i];
    __syncthreads();
    if (live && r < N2) {
        fft::reg_dft<R, -1, N1, 2 * N2>(y, tw);
        // W_M^(r k1) from the thread-ordered copy after the table (consecutive in r)
#pragma unroll
        for (int k1 = 1; k1 < N1; ++k1) y[k1] = y[k1] * tw_g[NX + k1 * N2 + r];
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) lb[r * (N1 + 1) + k1] = y[k1];
    }
    __syncthreads();
    // the second step's threads are N1 a line: packed, so that whole warps are idle instead of
    // lanes where N1 < N2
    const int l2 = threadIdx.x / N1, r2 = threadIdx.x % N1;
    const bool live2 = l2 < LPB && blockIdx.x * LPB + l2 < nlines;
    cplx<R>* lb2 = buf + l2 * CS;
    cplx<R> z[N2];
    if (live2) {
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) z[n2] = lb2[n2 * (N1 + 1) + r2];
        fft::reg_dft<R, -1, N2, 2 * N1>(z, tw);
    }
    __syncthreads();
    if (live2) {
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) lb2[r2 + N1 * k2] = z[k2];
    }
    __syncthreads();
    if (live) {
        cplx<R>* out = S + (size_t)line * NXH;
        for (int m = r; 2 * m <= M; m += TPC) {
            const cplx<R> zm = lb[m], zc = lb[m == 0 ? 0 : M - m], w = tw[m];
            const R sr = zm.re + zc.re, si = zm.im - zc.im, dr = zm.re - zc.re, di = zm.im + zc.im;
            const R tr = w.re * dr - w.im * di, ti = w.re * di + w.im * dr;
            out[m] = cplx<R>{sr + ti, si - tr};
            if (2 * m < M) out[M - m] = cplx<R>{sr - ti, -si - tr};
        }
    }
}

// ---------------------------------------------------------------- y solve, double-single steps
// d - b c with one normalisation: the product's error terms (each exact to FP32
// rounding of an O(u) correction) are added to the low part of the two-sum of
// the high parts
__device__ __forceinline__ ds ds_sub_mul(ds d, ds b, ds c) {
    const float h = b.hi * c.hi;
    const float e = fmaf(b.lo, c.hi, fmaf(b.hi, c.lo, fmaf(b.hi, c.hi, -h)));
    ds s = two_sum(d.hi, -h);
    s.lo += d.lo - e;
    return fast_two_sum(s.hi, s.lo);
}
// the same for an FP32 r
__device__ __forceinline__ ds ds_sub_mul(float r, ds b, ds c) {
    const float h = b.hi * c.hi;
    const float e = fmaf(b.lo, c.hi, fmaf(b.hi, c.lo, fmaf(b.hi, c.hi, -h)));
    ds s = two_sum(r, -h);
    s.lo -= e;
    return fast_two_sum(s.hi, s.lo);
}
// a - b rounded to FP32: the high parts' difference is exact when they are
// within a factor two of each other (Sterbenz) and has no cancellation
// otherwise, so the result is within a few roundings of the difference
__device__ __forceinline__ float ds_diff_f(ds a, ds b) { return (a.hi - b.hi) + (a.lo - b.lo); }

// ---------------------------------------------------------------- y solve, twisted (two-ended) Thomas
// The elimination runs from both walls towards the middle row k = ny/2 at once
// (a twisted factorisation): the top half (rows 0..k-1) downwards, the bottom
// half (rows ny-1..k+1) upwards.  With the pivots' inverses i_j, FP64-computed
// at set-up per (|m_z|, m_x) and held as double-single pairs:
//   top     P_j = r_j - e_j P_j-1,  e_j = a_j i_j-1,  x_j = i_j (P_j - c_j x_j+1)
//   bottom  P_j = r_j - f_j P_j+1,  f_j = c_j i_j+1,  x_j = i_j (P_j - a_j x_j-1)
//   middle  x_k = g (r_k - e_k P_k-1 - f_k P_k+1).
// In local index t of a half (t = j in the top half, ny-1-j in the bottom half)
// both halves run the same recurrences.  E_y per cell j is A_j x_j + Bm_j (x_j -
// x_j-1) + Bp_j (x_j+1 - x_j) from the double-single values, one cell behind the
// substitution (the bottom half takes Bm and Bp with their roles and signs
// exchanged); the top half writes cell k; wall nodes E_y = ew0 phi_0 (bottom
// wall), ewN phi_ny-1 (top wall).
//
// The forward sweep keeps the value entering each chunk of C rows and the
// substitution recomputes each chunk's values from it (keeping all of them
// instead measured the same on small grids and 20 us more at 384x256x256).  A
// row's values are fetched C rows ahead, into the registers the row C before it
// has just left, and rows are addressed by 32-bit element indices: the kernel is
// bound by its instruction stream and its loads' latency together (51% issue,
// 34% of stalls on loads before this form).  NH = 1: a pencil's halves run in two
// lanes 16 apart and meet through shuffles; NH = 2: one thread runs both, two
// interleaved chains, in 168 registers, six blocks a SM (with E_y it spills 60 bytes, the
// channel-table form 72).
// Which one: NH = 1 needs 128 registers for C = 6 rows ahead, four blocks of 64
// pencils a SM; while the grid fits one such wave it is the faster (us, against
// 64-pencil blocks of NH = 2, C = 5 at 168 registers): 128^3 24 / 32, 192x128x128
// 26 / 32, 288x145x162 38 / 53, 256^3 85 / 105; past it (384x256x256, 1.27
// waves) 153 / 127.  Before: 33 at 128^3, 65 at 288x145x162, 150 at 384x256x256.
// te: e_j (j <= k) and f_j (j > k), f_k at row ny; ti: i_j, g at row k.
// cpl: ny couplings c_j (j < k), a_j (j > k).
// ck: (ceil(k / C) - 1) x 2 x (nz nxh) float4 of chunk checkpoints.
constexpr int kTwistC1 = 6, kTwistT1 = 128;  // NH = 1: rows per chunk, threads per block
constexpr int kTwistC2 = 5, kTwistT2 = 64;   // NH = 2
// shared memory: the E_y coefficients of both halves and the couplings
inline size_t ysolve_twist_smem(int ny) { return (2 * sizeof(float4) + sizeof(float2)) * (size_t)(ny + 1); }
// the pencils of one resident wave of the NH = 1 form
inline bool ysolve_two_lanes(int64_t pencils, int num_sms) { return pencils <= (int64_t)num_sms * 4 * (kTwistT1 / 2); }

template <int NH, bool EY = true, bool kTab = false>
__global__ void __launch_bounds__(NH == 1 ? kTwistT1 : kTwistT2, NH == 1 ? 4 : 6)
k_ysolve_twist(cplx<float>* __restrict__ S, cplx<float>* __restrict__ F, const float2* __restrict__ te,
               const float2* __restrict__ ti, const float2* __restrict__ cpl, const float4* __restrict__ ec,
               float4* __restrict__ ck, int ny, int nz, int nxh, const FastTab<float>* __restrict__ tab) {
    constexpr int C = NH == 1 ? kTwistC1 : kTwistC2;
    pdl_wait();
    if constexpr (kTab) {
        const FastTab<float>& t = tab[blockIdx.y];
        S = t.S;
        F = t.F;
        te = t.te;
        ti = t.ti;
        cpl = t.cpl;
        ec = t.yec;
        ck = t.yck;
    }
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4* se = reinterpret_cast<float4*>(smem_raw);                 // 2 x (ny + 1): top, bottom
    float2* sc = reinterpret_cast<float2*>(se + 2 * (ny + 1));        // ny
    for (int j = threadIdx.x; j <= ny; j += blockDim.x) {
        if (j < ny) sc[j] = cpl[j];
        const float4 c = ec[j];
        se[j] = c;
        se[ny + 1 + j] = make_float4(c.x, -c.z, -c.y, 0.f);
    }
    __syncthreads();
    constexpr int PW = NH == 1 ? 16 : 32;                             // pencils per warp
    const int lane = threadIdx.x & 31;
    const int h0 = NH == 1 ? (lane >> 4) : 0;                         // this thread's first half
    const uint32_t np = (uint32_t)nz * nxh, ni = (uint32_t)(nz / 2 + 1) * nxh;
    const uint32_t pencil = (blockIdx.x * blockDim.x + threadIdx.x) / 32 * PW + lane % PW;
    const bool live = pencil < np;
    if (NH == 2 && !live) return;
    const uint32_t mz = live ? pencil / nxh : 0, mx = live ? pencil - mz * nxh : 0;
    const uint32_t item = min(mz, (uint32_t)nz - mz) * nxh + mx;
    const int k = ny >> 1;
    // element indices of row 0 (a grid of at most 1024 cells a side has fewer than 2^32 elements)
    float2* const Sv = reinterpret_cast<float2*>(S);
    float2* const Yv = reinterpret_cast<float2*>(F + (size_t)nz * (ny + 2) * nxh);   // E_y spectrum
    const uint32_t rs = nxh;
    const uint32_t s0 = mz * ny * nxh + mx, f0 = mz * (ny + 2) * nxh + mx;
    auto pair = [](float2 v) { return ds{v.x, v.y}; };
    // per half of the thread: rows, row of local row 0 and its direction
    int H[NH], Hmin = 1 << 30, j0[NH];
    uint32_t d[NH];                                                   // +1, -1 (modulo 2^32)
#pragma unroll
    for (int hh = 0; hh < NH; ++hh) {
        const int h = h0 + hh;
        H[hh] = !live ? 0 : h == 0 ? k : ny - 1 - k;
        j0[hh] = h == 0 ? 0 : ny - 1;
        d[hh] = h == 0 ? 1u : ~0u;
        Hmin = min(Hmin, H[hh]);
    }
    // element index of local row t
    auto at = [&](uint32_t base, uint32_t stride, int hh, int t) {
        return base + ((uint32_t)j0[hh] + d[hh] * (uint32_t)t) * stride;
    };
    const int nch = live ? (k + C - 1) / C : 0;                       // the top half is the longer one
    // ---- forward elimination
    ds P[NH][2];
    float2 e[NH][C], r[NH][C];
#pragma unroll
    for (int hh = 0; hh < NH; ++hh) {
        P[hh][0] = P[hh][1] = ds{0.f, 0.f};
#pragma unroll
        for (int i = 0; i < C; ++i)
            if (i < H[hh]) {
                e[hh][i] = te[at(item, ni, hh, i)];
                r[hh][i] = Sv[at(s0, rs, hh, i)];
            }
    }
    for (int c = 0; c < nch; ++c) {
        const int t0 = c * C;
        auto rows = [&](auto full) {          // full: every row of the chunk lies in both halves
#pragma unroll
            for (int i = 0; i < C; ++i)
#pragma unroll
                for (int hh = 0; hh < NH; ++hh)
                    if (decltype(full)::value || t0 + i < H[hh]) {
                        P[hh][0] = ds_sub_mul(r[hh][i].x, pair(e[hh][i]), P[hh][0]);
                        P[hh][1] = ds_sub_mul(r[hh][i].y, pair(e[hh][i]), P[hh][1]);
                        if (t0 + i + C < H[hh]) {
                            e[hh][i] = te[at(item, ni, hh, t0 + i + C)];
                            r[hh][i] = Sv[at(s0, rs, hh, t0 + i + C)];
                        }
                    }
        };
        if (t0 + C <= Hmin) rows(std::true_type{});
        else rows(std::false_type{});
        if (c + 1 < nch)
#pragma unroll
            for (int hh = 0; hh < NH; ++hh)
                ck[((size_t)c * 2 + h0 + hh) * np + pencil] =
                    make_float4(P[hh][0].hi, P[hh][0].lo, P[hh][1].hi, P[hh][1].lo);
    }
    // ---- the middle row (the other half's last forward value through a shuffle when another
    // thread has it), and each half's row next to it
    auto other = [&](ds v) {
        return ds{__shfl_xor_sync(0xffffffffu, v.hi, 16), __shfl_xor_sync(0xffffffffu, v.lo, 16)};
    };
    ds xk[2], xn[NH][2], x1[NH][2];          // x1: x at local row t + 1
    float dn[NH][2];                         // x(t + 2) - x(t + 1), zero where the other half is empty
    {
        ds po[2];                            // the forward value of the first half's other half
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            if constexpr (NH == 2) po[m] = P[1][m];
            else po[m] = other(P[0][m]);
            xk[m] = xn[0][m] = ds{0.f, 0.f};
        }
        if (live) {
            const ds ek = pair(te[item + (uint32_t)k * ni]), fk = pair(te[item + (uint32_t)ny * ni]);
            const ds g = pair(ti[item + (uint32_t)k * ni]);
            const float2 rk = Sv[s0 + (uint32_t)k * rs];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const ds pt = h0 == 0 ? P[0][m] : po[m], pb = h0 == 0 ? po[m] : P[0][m];
                xk[m] = ds_mul(ds_sub_mul(ds_sub_mul(m ? rk.y : rk.x, ek, pt), fk, pb), g);
            }
        }
        // both lanes of a pencil have read row k before one of them stores it
        if constexpr (NH == 1) __syncwarp();
        if (live) {
            if (h0 == 0) Sv[s0 + (uint32_t)k * rs] = make_float2(ds_f(xk[0]), ds_f(xk[1]));
#pragma unroll
            for (int hh = 0; hh < NH; ++hh) {
                xn[hh][0] = xk[0];
                xn[hh][1] = xk[1];
                if (H[hh] > 0) {
                    const ds cj = pair(sc[j0[hh] + (int)d[hh] * (H[hh] - 1)]);
                    const ds iv = pair(ti[at(item, ni, hh, H[hh] - 1)]);
#pragma unroll
                    for (int m = 0; m < 2; ++m) xn[hh][m] = ds_mul(ds_sub_mul(P[hh][m], cj, xk[m]), iv);
                }
            }
        }
        const int Ho = h0 == 0 ? ny - 1 - k : k;      // rows of the first half's other half
#pragma unroll
        for (int hh = 0; hh < NH; ++hh)
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                ds xo;
                if constexpr (NH == 2) xo = xn[1 - hh][m];
                else xo = other(xn[hh][m]);
                x1[hh][m] = xk[m];
                dn[hh][m] = (hh == 0 ? Ho : k) > 0 ? ds_diff_f(xo, xk[m]) : 0.f;
            }
    }
    if (!live) return;
    // ---- substitution, chunks from the middle outwards
    float2 v[NH][C];
    float4 q[NH];                            // the value entering the chunk
    int Hs[NH];                              // E_y rows: the bottom half leaves row k to the top
    const float4* sh[NH];
#pragma unroll
    for (int hh = 0; hh < NH; ++hh) {
        Hs[hh] = h0 + hh == 0 ? k + 1 : ny - 1 - k;
        sh[hh] = se + (h0 + hh) * (ny + 1);
    }
    auto fetch = [&](int hh, int i, int t) {
        v[hh][i] = ti[at(item, ni, hh, t)];
        r[hh][i] = Sv[at(s0, rs, hh, t)];
        e[hh][i] = te[at(item, ni, hh, t)];
    };
    auto fetch_ck = [&](int c) {
#pragma unroll
        for (int hh = 0; hh < NH; ++hh)
            q[hh] = c > 0 ? ck[((size_t)(c - 1) * 2 + h0 + hh) * np + pencil] : make_float4(0.f, 0.f, 0.f, 0.f);
    };
#pragma unroll
    for (int hh = 0; hh < NH; ++hh)
#pragma unroll
        for (int i = 0; i < C; ++i)
            if ((nch - 1) * C + i < H[hh]) fetch(hh, i, (nch - 1) * C + i);
    fetch_ck(nch - 1);
    for (int c = nch - 1; c >= 0; --c) {
        const int t0 = c * C;
        auto rows = [&](auto full) {
            ds p[NH][C][2], w[NH][2];
#pragma unroll
            for (int hh = 0; hh < NH; ++hh) {
                w[hh][0] = ds{q[hh].x, q[hh].y};
                w[hh][1] = ds{q[hh].z, q[hh].w};
            }
#pragma unroll
            for (int i = 0; i < C; ++i)
#pragma unroll
                for (int hh = 0; hh < NH; ++hh)
                    if (decltype(full)::value || t0 + i < H[hh]) {
                        p[hh][i][0] = w[hh][0] = ds_sub_mul(r[hh][i].x, pair(e[hh][i]), w[hh][0]);
                        p[hh][i][1] = w[hh][1] = ds_sub_mul(r[hh][i].y, pair(e[hh][i]), w[hh][1]);
                    }
            fetch_ck(c - 1);
#pragma unroll
            for (int i = C - 1; i >= 0; --i)
#pragma unroll
                for (int hh = 0; hh < NH; ++hh)
                    if (decltype(full)::value || t0 + i < H[hh]) {
                        const int t = t0 + i, j = j0[hh] + (int)d[hh] * t;
                        const ds cj = pair(sc[j]), iv = pair(v[hh][i]);
                        const float4 cf = sh[hh][j + (int)d[hh]];      // coefficients of the row of x1
                        float xf[2], ey[2];
#pragma unroll
                        for (int m = 0; m < 2; ++m) {
                            const ds x = ds_mul(ds_sub_mul(p[hh][i][m], cj, x1[hh][m]), iv);
                            xf[m] = ds_f(x);
                            const float d0 = ds_diff_f(x1[hh][m], x);
                            ey[m] = cf.x * ds_f(x1[hh][m]) + cf.y * d0 + cf.z * dn[hh][m];
                            dn[hh][m] = d0;
                            x1[hh][m] = x;
                        }
                        Sv[at(s0, rs, hh, t)] = make_float2(xf[0], xf[1]);
                        if (EY && t + 1 < Hs[hh]) Yv[at(f0 + rs, rs, hh, t + 1)] = make_float2(ey[0], ey[1]);
                        if (c > 0) fetch(hh, i, t - C);
                    }
        };
        if (t0 + C <= Hmin) {
            rows(std::true_type{});
        } else {
            rows(std::false_type{});
            // rows past the end of a half hold nothing to replace: their registers take the next
            // chunk's values here
            if (c > 0)
#pragma unroll
                for (int hh = 0; hh < NH; ++hh)
#pragma unroll
                    for (int i = 0; i < C; ++i)
                        if (t0 + i >= H[hh]) fetch(hh, i, t0 + i - C);
        }
    }
    if (!EY) return;
    const float4 walls = se[ny];
#pragma unroll
    for (int hh = 0; hh < NH; ++hh) {
        const bool top = h0 + hh == 0;
        // top: cell 0 (node 1) and the wall node 0; bottom: cell ny-1 (node ny) unless it is cell k,
        // and the wall node ny+1
        const float4 cf = sh[hh][top ? 0 : ny - 1];
        const float x = ds_f(x1[hh][0]), y = ds_f(x1[hh][1]), w = top ? walls.x : walls.y;
        if (top || H[hh] > 0)
            Yv[f0 + (uint32_t)(top ? 1 : ny) * rs] = make_float2(cf.x * x + cf.z * dn[hh][0], cf.x * y + cf.z * dn[hh][1]);
        Yv[f0 + (uint32_t)(top ? 0 : ny + 1) * rs] = make_float2(w * x, w * y);
    }
}

// launch of the solve for np pencils (n channels): the form by the rule above
template <bool EY, bool kTab>
void ysolve_twist_launch(int64_t pencils, int n, int num_sms, int ny, cudaStream_t stream, cplx<float>* S,
                         cplx<float>* F, const float2* te, const float2* ti, const float2* cpl, const float4* ec,
                         float4* ck, int nz, int nxh, const FastTab<float>* tab) {
    const bool two = ysolve_two_lanes(pencils * n, num_sms);
    const int per = two ? kTwistT1 / 2 : kTwistT2;
    const dim3 grid((unsigned)((pencils + per - 1) / per), (unsigned)n);
    (void)launch_pdl(two ? k_ysolve_twist<1, EY, kTab> : k_ysolve_twist<2, EY, kTab>, grid,
                     dim3(two ? kTwistT1 : kTwistT2), ysolve_twist_smem(ny), stream, S, F, te, ti, cpl, ec, ck, ny, nz,
                     nxh, tab);
}

// ---------------------------------------------------------------- z passes (four-step)
// The columns of all planes are one run: element k of column c = plane * nxh + m_x
// sits at k * (planes nxh) + c, so a tile is any W neighbouring columns, planes
// straddled, and only the last tile of a pass has idle lanes.  (Tiles that ended
// with their plane left 31 of 64 lanes idle at nx = 64, where m_x runs to 32, and
// 15 of 80 at nx = 128: FP64 inverse z pass at 64^3
// 33.8 -> 22.7 us, at 128^3 182 -> 147.)
// one tile of the forward z transform of S in place; out of line so that each tile starts from a
// fresh register allocation
template <class R, int NZ>
__device__ __noinline__ void zfwd_tile(cplx<R>* __restrict__ S, int ncols, int t, const cplx<R>* __restrict__ tw,
                                       cplx<R>* buf) {
    using F4 = fft::FourStep<NZ, kThreads>;
    cplx<R>* base = S + (size_t)t * F4::W;
    fft::column_fft<R, -1, NZ, kThreads, false>(base, ncols, base, ncols, min(F4::W, ncols - t * F4::W), tw, nullptr,
                                                buf);
}

template <class R, int NZ, bool kTab = false>
__global__ void __launch_bounds__(kThreads, (fft_min_blocks<R, NZ>())) k_zfwd4(cplx<R>* __restrict__ S, int ny, int nxh,
                                                    const cplx<R>* __restrict__ tw_g,
                                                    const FastTab<R>* __restrict__ tab) {
    pdl_wait();
    if constexpr (kTab) {
        S = tab[blockIdx.y].S;
        tw_g = tab[blockIdx.y].twz;
    }
    using F4 = fft::FourStep<NZ, kThreads>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<R>* tw = reinterpret_cast<cplx<R>*>(smem_raw);
    cplx<R>* buf = tw + NZ;
    for (int i = threadIdx.x; i < NZ; i += kThreads) tw[i] = tw_g[i];
    __syncthreads();
    const int ncols = ny * nxh;
    for (int t = blockIdx.x; t * F4::W < ncols; t += gridDim.x) zfwd_tile<R, NZ>(S, ncols, t, tw, buf);
}

// Inverse z transforms: F1 = IFFT_z(E_y-hat) in place on all node planes; on the
// interior planes F0 = IFFT_z(phi-hat of cell jn-1) and F2 = IFFT_z(-i sin(2 pi
// m_z/nz)/dz phi-hat).  Out of line as above: one tile of F1, and one of F0 and F2
// (dz: F2 too).
template <class R, int NZ>
__device__ __noinline__ void zinv_tile_e(cplx<R>* __restrict__ Fy, int ncols, int t, const cplx<R>* __restrict__ tw,
                                         cplx<R>* buf) {
    using F4 = fft::FourStep<NZ, kThreads>;
    cplx<R>* base = Fy + (size_t)t * F4::W;
    fft::column_fft<R, 1, NZ, kThreads, false>(base, ncols, base, ncols, min(F4::W, ncols - t * F4::W), tw, nullptr,
                                               buf);
}
template <class R, int NZ, bool kDz>
__device__ __noinline__ void zinv_tile_phi(const cplx<R>* __restrict__ S, cplx<R>* __restrict__ F0, int ncols, int fcols,
                                           int t, size_t fstride, const cplx<R>* __restrict__ tw,
                                           const R* __restrict__ sz, cplx<R>* buf) {
    using F4 = fft::FourStep<NZ, kThreads>;
    const size_t c0 = (size_t)t * F4::W;
    const int ncol = min(F4::W, ncols - t * F4::W);
    fft::column_fft<R, 1, NZ, kThreads, false>(S + c0, ncols, F0 + c0, fcols, ncol, tw, nullptr, buf);
    if constexpr (kDz)
        fft::column_fft<R, 1, NZ, kThreads, true>(S + c0, ncols, F0 + 2 * fstride + c0, fcols, ncol, tw, sz, buf);
}

template <class R, int NZ, bool kTab = false>
__global__ void __launch_bounds__(kThreads, (fft_min_blocks<R, NZ>())) k_zinv4(const cplx<R>* __restrict__ S, cplx<R>* __restrict__ F,
                                                    int ny, int nxh, size_t fstride, const double* __restrict__ sinz,
                                                    const cplx<R>* __restrict__ tw_g, int phi_only,
                                                    const FastTab<R>* __restrict__ tab) {
    pdl_wait();
    if constexpr (kTab) {
        const FastTab<R>& t = tab[blockIdx.y];
        S = t.S;
        F = t.F;
        sinz = t.sinz;
        tw_g = t.twz;
    }
    using F4 = fft::FourStep<NZ, kThreads>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<R>* tw = reinterpret_cast<cplx<R>*>(smem_raw);
    cplx<R>* buf = tw + NZ;
    R* sz = reinterpret_cast<R*>(buf + F4::BUF);
    for (int i = threadIdx.x; i < NZ; i += kThreads) {
        tw[i] = tw_g[i];
        sz[i] = from_f64<R>(sinz[i]);
    }
    __syncthreads();
    const int ncols = ny * nxh, fcols = (ny + 2) * nxh;
    const int np = (ncols + F4::W - 1) / F4::W, ne = phi_only ? 0 : (fcols + F4::W - 1) / F4::W;
    // the longer tiles (two transforms) first
    for (int t = blockIdx.x; t < np + ne; t += gridDim.x) {
        if (t >= np) zinv_tile_e<R, NZ>(F + fstride, fcols, t - np, tw, buf);
        else if (phi_only) zinv_tile_phi<R, NZ, false>(S, F + nxh, ncols, fcols, t, fstride, tw, sz, buf);
        else zinv_tile_phi<R, NZ, true>(S, F + nxh, ncols, fcols, t, fstride, tw, sz, buf);
    }
}

// ---------------------------------------------------------------- x inverse
// Four-step variant.  Thread group (line, r) per node line (k, jn); for each
// field the thread with n2 = r forms Z_m for its m = N2 n1 + r straight from
// X_m and X_M-m in global memory (split step), then the register four-step
// inverse of length M = N1 N2, and the group stores x_2n, x_2n+1 as pairs.
// Wall lines (jn = 0, ny+1) carry E_x = E_z = 0.
template <class R>
__device__ __forceinline__ void store_pair(R* p, R a, R b) {
    if constexpr (sizeof(R) == 4) *reinterpret_cast<float2*>(p) = make_float2(a, b);
    else *reinterpret_cast<double2*>(p) = make_double2(a, b);
}

template <class R, int M, bool kTab = false>
__global__ void __launch_bounds__(kThreads, (fft_min_blocks<R, M>())) k_xinv4(const cplx<R>* __restrict__ F, R* __restrict__ E,
                                                    double* __restrict__ phi, int ny, int nz, size_t fstride,
                                                    const double* __restrict__ sinx,
                                                    const cplx<R>* __restrict__ tw_g, int want_phi, int want_e,
                                                    size_t nodes, const FastTab<R>* __restrict__ tab) {
    pdl_wait();
    if constexpr (kTab) {
        const FastTab<R>& t = tab[blockIdx.y];
        F = t.F;
        E = t.E;
        sinx = t.sinx;
        tw_g = t.twx;
    }
    using F4 = fft::FourStep<M, kThreads>;
    constexpr int N1 = F4::N1, N2 = F4::N2, TPC = F4::TPC, LPB = F4::W, CS = F4::CS;
    constexpr int NX = 2 * M, NXH = M + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<R>* tw = reinterpret_cast<cplx<R>*>(smem_raw);   // exp(-2 pi i e / NX)
    cplx<R>* buf = tw + NX;
    cplx<R>* t2 = buf + F4::BUF;    // t2[k1 N2 + r] = W_M^(r k1): consecutive in r, no bank conflicts
    R* sx = reinterpret_cast<R*>(t2 + N1 * N2);
    for (int i = threadIdx.x; i < NX; i += kThreads) tw[i] = tw_g[i];
    for (int i = threadIdx.x; i < N1 * N2; i += kThreads) t2[i] = tw_g[2 * (i % N2) * (i / N2)];
    for (int i = threadIdx.x; i < NXH; i += kThreads) sx[i] = from_f64<R>(sinx[i]);
    __syncthreads();
    const int nyn = ny + 2;
    // a caller's field without a context (tribo_poisson_noalloc) may be aligned to its elements only
    const bool pairs = (reinterpret_cast<uintptr_t>(E) & (2 * sizeof(R) - 1)) == 0;
    const int r = threadIdx.x % TPC;
    const int l = threadIdx.x / TPC;
    const int ntb = (nz * nyn + LPB - 1) / LPB;
    for (int tb = blockIdx.x; tb < ntb; tb += gridDim.x) {
    const int line = tb * LPB + l;
    const bool live = l < LPB && line < nz * nyn;
    const int jn = live ? line % nyn : 0;
    const bool interior = jn >= 1 && jn <= ny;
    // the second step's threads are N1 a line, packed as in the forward transform
    const int l2 = threadIdx.x / N1, r2 = threadIdx.x % N1;
    const int line2 = tb * LPB + l2;
    const bool live2 = l2 < LPB && line2 < nz * nyn;
    const int jn2 = live2 ? line2 % nyn : 0;
    const bool interior2 = jn2 >= 1 && jn2 <= ny;
    const int nf = want_phi ? 4 : 3;
    for (int f = want_e ? 0 : 3; f < nf; ++f) {
        const bool active = live && (f == 1 || interior);
        const int src = f == 3 ? 0 : f;
        if (active && r < N2) {
            const cplx<R>* X = F + (size_t)src * fstride + (size_t)line * NXH;
            cplx<R> y[N1];
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) {
                const int m = N2 * n1 + r;
                const cplx<R> xa = X[m], xb = X[M - m];
                y[n1] = f == 0 ? split_inv_dx(xa, xb, tw[m], sx[m]) : split_inv(xa, xb, tw[m]);
            }
            fft::reg_dft<R, 1, N1, 2 * N2>(y, tw);
#pragma unroll
            for (int k1 = 1; k1 < N1; ++k1) y[k1] = y[k1] * conj(t2[k1 * N2 + r]);
            cplx<R>* b = buf + l * CS + r * (N1 + 1);
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) b[k1] = y[k1];
        }
        __syncthreads();
        if (live2 && (f == 1 || interior2)) {
            cplx<R> z[N2];
            const cplx<R>* b = buf + l2 * CS + r2;
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2) z[n2] = b[n2 * (N1 + 1)];
            fft::reg_dft<R, 1, N2, 2 * N1>(z, tw);
            if (f < 3) {
                R* row = E + (size_t)f * nodes + (size_t)line2 * NX;
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) {
                    const int k = r2 + N1 * k2;
                    if (pairs) {
                        store_pair<R>(row + 2 * k, z[k2].re, z[k2].im);
                    } else {
                        row[2 * k] = z[k2].re;
                        row[2 * k + 1] = z[k2].im;
                    }
                }
            } else {
                double* prow = phi + ((size_t)(line2 / nyn) * ny + (jn2 - 1)) * NX;
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) {
                    const int k = r2 + N1 * k2;
                    prow[2 * k] = (double)z[k2].re;
                    prow[2 * k + 1] = (double)z[k2].im;
                }
            }
        }
        __syncthreads();
    }
    if (want_e && live && !interior) {
        R* ex = E + (size_t)line * NX;
        R* ez = E + 2 * nodes + (size_t)line * NX;
        for (int i = r; i < NX; i += TPC) {
            ex[i] = (R)0;
            ez[i] = (R)0;
        }
    }
    }
}

// ---------------------------------------------------------------- dispatch
template <class R, int M>
size_t xfwd_smem() { return sizeof(cplx<R>) * (2 * M + fft::FourStep<M, kThreads>::BUF); }
template <class R, int M>
size_t xinv_smem() {
    using F4 = fft::FourStep<M, kThreads>;
    return sizeof(cplx<R>) * (2 * M + F4::BUF + F4::N1 * F4::N2) + sizeof(R) * (M + 1);
}
template <class R, int NZ>
size_t zfwd_smem() { return sizeof(cplx<R>) * (NZ + fft::FourStep<NZ, kThreads>::BUF); }
template <class R, int NZ>
size_t zinv_smem() { return sizeof(cplx<R>) * (NZ + fft::FourStep<NZ, kThreads>::BUF) + sizeof(R) * NZ; }

// blocks of one resident wave of `kernel` (its occupancy is queried once per instantiation),
// at most `tiles`
template <class K>
int wave_blocks(K kernel, size_t smem, int num_sms, int64_t tiles, int* cache) {
    if (*cache == 0) {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kThreads, smem) != cudaSuccess || b < 1) b = 1;
        *cache = b;
    }
    return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)*cache * num_sms));
}

// every half length M = nx/2 and length nz of a supported grid: 2^a 3^b, nx and nz up to 1024
#define TRIBO_X_SIZES(X) \
    X(2) X(3) X(4) X(6) X(8) X(9) X(12) X(16) X(18) X(24) X(27) X(32) X(36) X(48) X(54) X(64) X(72) X(81) X(96) \
    X(108) X(128) X(144) X(162) X(192) X(216) X(243) X(256) X(288) X(324) X(384) X(432) X(486) X(512)
#define TRIBO_Z_SIZES(X) \
    X(4) X(6) X(8) X(9) X(12) X(16) X(18) X(24) X(27) X(32) X(36) X(48) X(54) X(64) X(72) X(81) X(96) \
    X(108) X(128) X(144) X(162) X(192) X(216) X(243) X(256) X(288) X(324) X(384) X(432) X(486) X(512) \
    X(576) X(648) X(729) X(768) X(864) X(972) X(1024)

}  // namespace
}  // namespace tribo
