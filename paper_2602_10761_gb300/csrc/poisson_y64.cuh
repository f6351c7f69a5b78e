// The FP64 y solve of the Poisson equation (Sec. 2.2, Sec. 3.1): the twisted
// elimination's kernel and factors, shared by a context's FP64 solve and the
// allocation-free solve.
#pragma once

#include "tribo_internal.cuh"

namespace tribo {
namespace {

// ---------------------------------------------------------------- y solve, FP64
// Twisted elimination from both walls to the middle row k = ny/2, as the mixed
// precision solve, in plain FP64.  With the pivots' inverses i_j (top half
// j < k from the lower wall, bottom half j > k from the upper wall) the
// recurrences need two table values a row and three operations a value:
//   top     P_j = r_j - e_j P_j-1,  e_j = a_j i_j-1,  x_j = i_j (P_j - c_j x_j+1)
//   bottom  P_j = r_j - f_j P_j+1,  f_j = c_j i_j+1,  x_j = i_j (P_j - a_j x_j-1)
//   middle  x_k = g (r_k - e_k P_k-1 - f_k P_k+1).
// A pencil's two halves and its real and imaginary parts are four threads (lanes
// 0-15 of a warp run the top halves of 8 pencils, lanes 16-31 the bottom halves;
// neighbouring lanes are one complex value, so a half warp reads 128 contiguous
// bytes), each with its own chain of FP64 operations and its rows' loads one
// chunk ahead.  P overwrites the spectrum row by row and is read back by the
// same thread, so the solve needs no scratch; with FP32 spectra (the allocation-
// free solve in mixed precision, everything between them FP64) P goes to the planes
// of the field spectra that the inverse z pass writes later, one double in the place
// of a complex value: real parts in the first plane, imaginary parts in the third.  The work is 6 FP64 operations a
// value (E_y included), 21 us of the FP64 pipe at 128^3; the kernel it replaces
// ran a |m_z| row's pencils in one thread (33 blocks at 128^3) with every row's
// load exposed: 291 -> 40 us at 128^3, a 64^3 step 269 -> 146 us.  Its error
// against an 80-bit solve is the one-sided sweep's but for scatter (phi 0.7 to
// 1.3 times it, 1.0 in the mean over six grids and three seeds; E 1.0).
// te: e_j (j <= k) and f_j (j > k), f_k at row ny; ti: i_j, g at row k.
constexpr int kY64Rows = 8;                  // rows per chunk
inline size_t ysolve64_smem(int ny) { return sizeof(double) * ((size_t)ny + 3 * (ny + 2)); }

template <class R>
__global__ void __launch_bounds__(128) k_ysolve64(cplx<R>* __restrict__ S, cplx<R>* F, const double* __restrict__ te, const double* __restrict__ ti,
                                                  const double* __restrict__ ycoef, const double* __restrict__ ey,
                                                  int ny, int nz, int nxh, int want_ey) {
    pdl_wait();
    extern __shared__ __align__(16) double sh64[];
    double* cpl = sh64;                       // coupling of the substitution: c_j (top), a_j (bottom)
    double* sey = sh64 + ny;                  // 3 per lattice node
    const int k = ny >> 1;
    for (int j = threadIdx.x; j < ny; j += blockDim.x) cpl[j] = j < k ? ycoef[2 * ny + j] : ycoef[j];
    for (int j = threadIdx.x; j < 3 * (ny + 2); j += blockDim.x) sey[j] = ey[j];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int h = lane >> 4, comp = lane & 1;
    const int np = nz * nxh, ni = (nz / 2 + 1) * nxh;
    const int pencil = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 8 + ((lane >> 1) & 7);
    const bool live = pencil < np;
    const int mz = live ? pencil / nxh : 0, mx = live ? pencil - mz * nxh : 0;
    const int item = min(mz, nz - mz) * nxh + mx;
    const int H = live ? (h == 0 ? k : ny - 1 - k) : 0;        // rows of this half
    const ptrdiff_t rs = 2 * (ptrdiff_t)nxh;
    const size_t fplane = (size_t)nz * (ny + 2) * nxh;
    R* srow = reinterpret_cast<R*>(S + (size_t)mz * ny * nxh + mx) + comp;
    R* frow = reinterpret_cast<R*>(F + fplane + (size_t)mz * (ny + 2) * nxh + mx) + comp;
    // local row t of a half: row t (top) or ny - 1 - t (bottom)
    const int j0 = h == 0 ? 0 : ny - 1, dj = h == 0 ? 1 : -1;
    R* sp = srow + j0 * rs;
    const ptrdiff_t ss = dj * rs, ts = (ptrdiff_t)dj * ni;
    double* pp;                              // P of local row t at pp[t * ps]
    ptrdiff_t ps;
    if constexpr (sizeof(R) == 8) {
        pp = sp;
        ps = ss;
    } else {
        pp = reinterpret_cast<double*>(F + 2 * comp * fplane + (size_t)mz * (ny + 2) * nxh + mx) + (ptrdiff_t)j0 * nxh;
        ps = (ptrdiff_t)dj * nxh;
    }
    const double* ep = te + (ptrdiff_t)j0 * ni + item;
    const double* ip = ti + (ptrdiff_t)j0 * ni + item;
    constexpr int C = kY64Rows;
    double P = 0.0;
    {
        double r[C], e[C], r2[C], e2[C];
#pragma unroll
        for (int i = 0; i < C; ++i)
            if (i < H) { r[i] = (double)sp[i * ss]; e[i] = ep[i * ts]; }
        for (int t0 = 0; t0 < H; t0 += C) {
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const int t = t0 + C + i;
                if (t < H) { r2[i] = (double)sp[t * ss]; e2[i] = ep[t * ts]; }
            }
#pragma unroll
            for (int i = 0; i < C; ++i)
                if (t0 + i < H) {
                    P = fma(-e[i], P, r[i]);
                    pp[(t0 + i) * ps] = P;
                }
#pragma unroll
            for (int i = 0; i < C; ++i) { r[i] = r2[i]; e[i] = e2[i]; }
        }
    }
    // the middle row, on both halves
    const double Po = __shfl_xor_sync(0xffffffffu, P, 16);
    double xk = 0.0, xn = 0.0;               // x_k, and the half's row next to it
    if (live) {
        const double Pt = h == 0 ? P : Po, Pb = h == 0 ? Po : P;
        xk = fma(-te[(size_t)ny * ni + item], Pb, fma(-te[(size_t)k * ni + item], Pt, (double)srow[k * rs])) *
             ti[(size_t)k * ni + item];
        if (H > 0) xn = fma(-cpl[j0 + (H - 1) * dj], xk, P) * ip[(H - 1) * ts];
    }
    const double xo = __shfl_xor_sync(0xffffffffu, xn, 16);   // the other half's row next to k
    __syncwarp();                            // both halves have read row k before one of them stores it
    if (!live) return;
    if (h == 0) srow[k * rs] = (R)xk;
    // substitution outwards; the E_y of a row one row behind it (the bottom half leaves row k to the top)
    double x1 = xk, x2 = xo;                 // x at local rows t + 1, t + 2
    const int om = h == 0 ? 0 : 2, op = h == 0 ? 2 : 0;       // coefficient of the row before, behind
    {
        double p[C], v[C], p2[C], v2[C];
        const int last = H > 0 ? (H - 1) / C * C : -C;
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int t = last + i;
            if (t >= 0 && t < H) { p[i] = pp[t * ps]; v[i] = ip[t * ts]; }
        }
        for (int t0 = last; t0 >= 0; t0 -= C) {
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const int t = t0 - C + i;
                if (t >= 0) { p2[i] = pp[t * ps]; v2[i] = ip[t * ts]; }
            }
#pragma unroll
            for (int i = C - 1; i >= 0; --i) {
                const int t = t0 + i;
                if (t < H) {
                    const double x = fma(-cpl[j0 + t * dj], x1, p[i]) * v[i];
                    sp[t * ss] = (R)x;
                    const int jc = j0 + (t + 1) * dj;         // row of x1
                    if (want_ey && (h == 0 || t + 1 < H)) {
                        const double* c = sey + 3 * (jc + 1);
                        frow[(jc + 1) * rs] = (R)fma(c[op], x2, fma(c[1], x1, c[om] * x));
                    }
                    x2 = x1;
                    x1 = x;
                }
            }
#pragma unroll
            for (int i = 0; i < C; ++i) { p[i] = p2[i]; v[i] = v2[i]; }
        }
    }
    if (!want_ey) return;
    // the row at the wall and the wall node
    if (h == 0) {
        frow[rs] = (R)fma(sey[5], x2, sey[4] * x1);
        frow[0] = (R)(sey[2] * x1);
    } else {
        if (H > 0) frow[ny * rs] = (R)fma(sey[3 * ny], x2, sey[3 * ny + 1] * x1);
        frow[(ny + 1) * rs] = (R)(sey[3 * (ny + 1)] * x1);
    }
}

__device__ __forceinline__ void put_factor(double* p, double v) { *p = v; }
__device__ __forceinline__ void put_factor(float2* p, double v) {
    const float hi = (float)v;
    *p = make_float2(hi, (float)(v - (double)hi));
}

// The factors of one wavenumber pair (lam, column item of the tables) in FP64: the top half (halves
// & 1), the bottom half (halves & 2); the middle row and f_k when both are this thread's, or
// meet through a shuffle of lanes 2i, 2i + 1 when they are two threads' (all 32 lanes call then).
template <class T>
__device__ __forceinline__ void y_factors(const double* __restrict__ ycoef, double lam, int ny, int ni, int item,
                                          int halves, T* __restrict__ te, T* __restrict__ ti) {
    const double *a = ycoef, *b = ycoef + ny, *c = ycoef + 2 * ny;
    const int k = ny >> 1;
    auto put = [&](int j, double e, double i) {
        put_factor(te + (size_t)j * ni + item, e);
        put_factor(ti + (size_t)j * ni + item, i);
    };
    double up = 0.0, dn = 0.0;
    if (halves & 1)
        for (int j = 0; j < k; ++j) {
            const double e = a[j] * up;
            up = 1.0 / ((b[j] - lam) - (j > 0 ? e * c[j - 1] : 0.0));
            put(j, e, up);
        }
    if (halves & 2)
        for (int j = ny - 1; j > k; --j) {
            const double f = c[j] * dn;
            dn = 1.0 / ((b[j] - lam) - (j < ny - 1 ? f * a[j + 1] : 0.0));
            put(j, f, dn);
        }
    if (halves != 3) {                        // two neighbouring lanes hold a half each
        const double o = __shfl_xor_sync(0xffffffffu, halves & 1 ? up : dn, 1);
        if (halves & 1) dn = o;
        else up = o;
        if (halves & 2) return;
    }
    const double e = a[k] * up, f = c[k] * dn;
    put(k, e, 1.0 / ((b[k] - lam) - (k > 0 ? e * c[k - 1] : 0.0) - (k < ny - 1 ? f * a[k + 1] : 0.0)));
    put_factor(te + (size_t)ny * ni + item, f);
}

}  // namespace
}  // namespace tribo
