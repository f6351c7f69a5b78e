// Poisson solve and E field of a context (Sec. 2.2 Poisson equation with
// grounded walls, second-order finite volumes of Sec. 3.1, E = -grad(phi) with
// Gauss-linear E_y and central E_x, E_z; the discretisation is described in
// poisson.cu).  Every supported length 2^a 3^b has compiled transforms and
// tabulated y factors (the field of a 288 x 145 x 162 grid in mixed precision:
// 160 us; 1167 us with shared-memory Stockham passes and an FP64 Thomas sweep
// with a division per row):
//  * the x transforms are real: a length-nx/2 complex FFT of the packed line
//    plus the split step (half the work and shared memory);
//  * the y factorisation depends only on lam = lam_x + lam_z, so the factors
//    are computed once in FP64 at set-up, one table row per (|m_z|, m_x): the
//    factors of a twisted elimination from both walls to the middle row;
//  * E_y is formed from phi in the y sweep, where phi still carries more than
//    FP32 precision (a difference of FP32 values would lose the near-wall
//    field); E_z takes its spectral multiplier before the inverse z transform
//    and E_x before the inverse x transform.
// In FP64 mode everything is FP64.  In mixed mode the sweeps run in
// double-single arithmetic (value = hi + lo, two FP32 numbers; Dekker's
// product and Knuth's sum), which keeps about 46 significant bits on the FP32
// pipes: on this GPU FP64 instructions, conversions included, issue at 1/64
// of the FP32 rate.
//  * the x and z transforms are register four-step FFTs (fft_reg.cuh): each
//    element passes through shared memory once, in one transpose.
// Passes: xfwd (zeroes the charge buffer), zfwd, ysolve, zinv, xinv.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "poisson_passes.cuh"
#include "poisson_y64.cuh"

namespace tribo {

namespace {

// The factors of the twisted elimination per (|m_z|, m_x), one thread each; T = double, or float2 for
// the double-single pairs of the mixed solve
template <class T>
__global__ void k_ytab(const double* __restrict__ ycoef, const double* __restrict__ lamx,
                       const double* __restrict__ lamz, int ny, int nz, int nxh, T* __restrict__ te,
                       T* __restrict__ ti) {
    const int ni = (nz / 2 + 1) * nxh;
    const int item = blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= ni) return;
    y_factors(ycoef, lamz[item / nxh] + lamx[item % nxh], ny, ni, item, 3, te, ti);
}

// ---------------------------------------------------------------- fused inverse pipeline
// The inverse z transforms of a node plane and its inverse x transforms with
// the field run as ONE persistent launch, the two transforms of a plane being
// tasks of one queue: producer tasks = tiles of m_x columns (inverse z
// transforms of phi-hat, of -i sin(2 pi m_z / nz)/dz phi-hat and of the E_y
// spectrum into three fields of a plane slot), consumer tasks = groups of x
// lines (inverse real x transforms of the slot's fields to E_x, E_y, E_z and
// phi).  The slots form a ring of P planes that stays in L2: the three
// intermediate fields never reach HBM, where the split passes wrote them
// (0.31 GB at 384x256x256) and read them back.  The spectra read and the
// field written pass with evict-first hints, so that they do not push the
// ring out of L2.
//
// Tasks are claimed in order from one counter.  Stage s holds the producer
// tasks of plane s and then the consumer tasks of plane s - L.  A consumer
// waits until all producer tasks of its plane are done; a producer of plane
// p >= P waits until all consumers of plane p - P (the slot's previous plane)
// are done, and P > L.  Every task therefore waits only on tasks claimed
// before it by blocks that are already running, so the queue drains whatever
// the residency; each wait is bounded, and a wait that runs out sets
// TRIBO_DEV_TIMEOUT in the device error word instead of hanging.  Data a
// task reads from the ring is loaded through L2 (ld.global.cg), never from a
// possibly stale L1 line; producers publish with a release increment after
// the barrier that ends the task, consumers acquire the counter before
// reading.  Both waits need slack: the resident blocks hold about 21 stages
// at once (608 blocks over 29 tasks per plane at 384x256x256), so a consumer
// should trail its producers by L = 32 stages and a producer its slot's
// previous consumers by P - L = 40 (FP32, 384x256x256: 302 us with L = 24,
// P = 32; 265 us with 40, 48; 248 us with 24, 64; 245 us with 32, 72, the
// ring then 86 MB of L2).  The split passes move the three fields through
// HBM only when they do not fit in L2: the pipeline is used where they take
// at least 64 MiB (at 128^3, 26 MB, the split passes measured 106 against
// 121 us for the whole solve).
constexpr int kMaxPlanes = 1026;            // node planes of the tallest grid (ny = 1024)
#ifndef TRIBO_PIPE_LOOK
#define TRIBO_PIPE_LOOK 32
#endif
#ifndef TRIBO_PIPE_SLOTS
#define TRIBO_PIPE_SLOTS 72
#endif
constexpr int kPipeLook = TRIBO_PIPE_LOOK;  // L: stages a plane's consumers trail its producers
constexpr int kPipeSlots = TRIBO_PIPE_SLOTS;  // P: ring slots (> L)
constexpr unsigned kSpinLimit = 1u << 22;   // polls of a wait (>= ~1 s with the back-off)

struct PipeSync {                           // one launch's counters: zero when it starts, and
                                            // zeroed again by its last block to finish
    unsigned next;                          // next task to claim
    unsigned exited;                        // blocks that have left the task loop
    unsigned pad[30];
    unsigned a_done[kMaxPlanes];            // finished producer tasks per plane
    unsigned b_done[kMaxPlanes];            // finished consumer tasks per plane
};

struct Pipe {
    int planes;      // planes of the stage
    int na, nb;      // producer and consumer tasks per plane
    int L, P;        // lookahead in stages, ring slots
    unsigned total;  // planes * (na + nb)
    int stall;       // testing: the plane whose consumers wait for a producer task that never
                     // comes (their bounded waits run out), or -1
};

Pipe make_pipe(int planes, int na, int nb) {
    Pipe p{};
    p.planes = planes;
    p.na = na;
    p.nb = nb;
    p.L = std::min(kPipeLook, planes);
    p.P = kPipeSlots;
    p.total = (unsigned)planes * (unsigned)(na + nb);
    p.stall = -1;
    return p;
}

// task t -> (consumer?, plane, index within the plane's tasks of that kind)
__device__ __forceinline__ void pipe_task(const Pipe& p, unsigned t, bool& cons, int& plane, int& idx) {
    const unsigned head = (unsigned)p.L * p.na;
    const unsigned per = (unsigned)(p.na + p.nb);
    const unsigned body = (unsigned)(p.planes - p.L) * per;
    if (t < head) {
        cons = false;
        plane = (int)(t / p.na);
        idx = (int)(t % p.na);
    } else if (t - head < body) {
        const unsigned u = t - head;
        const int st = p.L + (int)(u / per);
        const int r = (int)(u % per);
        cons = r >= p.na;
        plane = cons ? st - p.L : st;
        idx = cons ? r - p.na : r;
    } else {
        const unsigned u = t - head - body;
        cons = true;
        plane = p.planes - p.L + (int)(u / p.nb);
        idx = (int)(u % p.nb);
    }
}

// thread 0: wait until *ctr >= target (acquire), bounded
__device__ __forceinline__ void pipe_wait(const unsigned* ctr, unsigned target, unsigned* err) {
    unsigned it = 0;
    for (;;) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
        if (v >= target) return;
        if (++it >= kSpinLimit) {
            atomicOr(err, TRIBO_DEV_TIMEOUT);
            return;
        }
        __nanosleep(256);
    }
}

// Task loop of a fused launch.  A block claims its next task only when it
// can start it (claims in order are what keeps every wait pointed at tasks
// that are running), thread 0 issuing the claim as its own part of the
// current task ends, so that the round trip overlaps the rest of the block's
// work.  Thread 0 waits for a task's dependency before the block starts it,
// and publishes a finished task with a release increment after the barrier
// that ends it (the release covers every write the barrier ordered before it).
struct PipeLoop {
    unsigned* s_next;    // shared: the block's next task
    unsigned t;          // current task
};

__device__ __forceinline__ void pipe_start(PipeLoop& L, PipeSync* sy) {
    if (threadIdx.x == 0) *L.s_next = atomicAdd(&sy->next, 1u);
    __syncthreads();
    L.t = *L.s_next;
}

// thread 0 waits for the task's dependency; then the block may read
__device__ __forceinline__ void pipe_acquire(PipeLoop& L, const Pipe& p, PipeSync* sy, bool cons, int plane,
                                             unsigned* err) {
    if (threadIdx.x == 0) {
        if (cons) pipe_wait(&sy->a_done[plane], (unsigned)p.na + (plane == p.stall ? 1u : 0u), err);
        else if (plane >= p.P) pipe_wait(&sy->b_done[plane - p.P], (unsigned)p.nb, err);
    }
    __syncthreads();
}

// the block's writes of the task are done: claim the next task, publish this one
__device__ __forceinline__ void pipe_release(PipeLoop& L, PipeSync* sy, bool cons, int plane) {
    unsigned nt = 0;
    if (threadIdx.x == 0) nt = atomicAdd(&sy->next, 1u);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned* ctr = cons ? &sy->b_done[plane] : &sy->a_done[plane];
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
        *L.s_next = nt;
    }
    __syncthreads();
    L.t = *L.s_next;
}

template <class R, int M, int NZ>
constexpr int fused_min_blocks() { return sizeof(R) == 4 ? 4 : 2; }

// inverse producer: node plane jn, m_x columns of a tile: the three slot fields
// (0: IFFT_z phi-hat, 1: IFFT_z E_y spectrum, 2: IFFT_z -i sin_z phi-hat);
// without E only field 0
template <class R, int NZ>
__device__ __noinline__ void inv_ztask(const cplx<R>* __restrict__ S, const cplx<R>* __restrict__ Fy,
                                       cplx<R>* slot, int ny, int nxh, int jn, int tile, int want_e,
                                       const cplx<R>* __restrict__ tw, const R* __restrict__ sz, cplx<R>* buf) {
    using F4 = fft::FourStep<NZ, kThreads>;
    const int mx0 = tile * F4::W;
    const int ncol = min(F4::W, nxh - mx0);
    const size_t fs = (size_t)NZ * nxh;
    // the spectra are read once (phi-hat twice, the second time from L1): evict-first in L2
    if (want_e)
        fft::column_fft<R, 1, NZ, kThreads, false, fft::kStream>(Fy + (size_t)jn * nxh + mx0, (size_t)(ny + 2) * nxh,
                                                                 slot + fs + mx0, (size_t)nxh, ncol, tw, nullptr, buf);
    if (jn >= 1 && jn <= ny) {
        const cplx<R>* ph = S + (size_t)(jn - 1) * nxh + mx0;
        if (want_e) {
            fft::column_fft<R, 1, NZ, kThreads, false>(ph, (size_t)ny * nxh, slot + mx0, (size_t)nxh, ncol, tw,
                                                       nullptr, buf);
            fft::column_fft<R, 1, NZ, kThreads, true, fft::kStream>(ph, (size_t)ny * nxh, slot + 2 * fs + mx0,
                                                                    (size_t)nxh, ncol, tw, sz, buf);
        } else {
            fft::column_fft<R, 1, NZ, kThreads, false, fft::kStream>(ph, (size_t)ny * nxh, slot + mx0, (size_t)nxh,
                                                                     ncol, tw, nullptr, buf);
        }
    }
}

// inverse consumer: node lines (k, jn), k = grp * LPB + l: E_x (the slot's field 0
// with the x multiplier -i sin(2 pi m / nx) / dx), E_y (field 1), E_z (field 2),
// phi (field 0); wall lines carry E_x = E_z = 0
template <class R, int M>
__device__ __noinline__ void inv_xtask(const cplx<R>* slot, R* __restrict__ E, double* __restrict__ phi, int ny,
                                       int nz, int jn, int grp, int want_phi, int want_e, size_t nodes,
                                       const cplx<R>* __restrict__ tw, const cplx<R>* __restrict__ t2,
                                       const R* __restrict__ sx, cplx<R>* buf) {
    using F4 = fft::FourStep<M, kThreads>;
    constexpr int N1 = F4::N1, N2 = F4::N2, TPC = F4::TPC, LPB = F4::W, CS = F4::CS;
    constexpr int NX = 2 * M, NXH = M + 1;
    const int nyn = ny + 2;
    const int r = threadIdx.x % TPC;
    const int l = threadIdx.x / TPC;
    const int k = grp * LPB + l;
    const bool live = l < LPB && k < nz;
    const bool interior = jn >= 1 && jn <= ny;
    const size_t fs = (size_t)nz * NXH;
    const size_t line = (size_t)k * nyn + jn;
    // the second step's threads are N1 a line, packed (whole warps idle instead of lanes)
    const int l2 = threadIdx.x / N1, r2 = threadIdx.x % N1;
    const int kl2 = grp * LPB + l2;
    const bool live2 = l2 < LPB && kl2 < nz;
    const size_t line2 = (size_t)kl2 * nyn + jn;
    const int nf = want_phi ? 4 : 3;
    for (int f = want_e ? 0 : 3; f < nf; ++f) {
        const bool active = live && (f == 1 || interior);
        const int src = f == 3 ? 0 : f;
        if (active && r < N2) {
            const cplx<R>* X = slot + (size_t)src * fs + (size_t)k * NXH;
            cplx<R> y[N1];
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) {
                const int m = N2 * n1 + r;
                const cplx<R> xa = fft::ld_cplx<R, fft::kL2Only>(X + m), xb = fft::ld_cplx<R, fft::kL2Only>(X + M - m);
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
        // every thread of the block has its values of this field: the slot lines that lie
        // wholly in the task's rows are dropped from L2 unwritten (the slot is rewritten by a
        // later plane; a write-back would only add HBM traffic)
        if ((f != 0 || !want_phi) && (f == 1 || interior)) {
            const char* base = reinterpret_cast<const char*>(slot + (size_t)src * fs);
            const int k0 = grp * LPB, k1 = min(k0 + LPB, nz);
            const size_t b0 = ((size_t)k0 * NXH * sizeof(cplx<R>) + 127) & ~(size_t)127;
            const size_t b1 = ((size_t)k1 * NXH * sizeof(cplx<R>)) & ~(size_t)127;
            if ((reinterpret_cast<uintptr_t>(base) & 127) == 0)
                for (size_t b = b0 + (size_t)threadIdx.x * 128; b < b1; b += (size_t)blockDim.x * 128)
                    asm volatile("discard.global.L2 [%0], 128;" ::"l"(base + b) : "memory");
        }
        if (live2 && (f == 1 || interior)) {
            cplx<R> z[N2];
            const cplx<R>* b = buf + l2 * CS + r2;
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2) z[n2] = b[n2 * (N1 + 1)];
            fft::reg_dft<R, 1, N2, 2 * N1>(z, tw);
            if (f < 3) {       // written once: evict-first in L2
                cplx<R>* row = reinterpret_cast<cplx<R>*>(E + (size_t)f * nodes + line2 * NX);
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2)
                    fft::st_cplx<R, fft::kStream>(row + r2 + N1 * k2, z[k2]);
            } else {
                double2* prow = reinterpret_cast<double2*>(phi + ((size_t)kl2 * ny + (jn - 1)) * NX);
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2)
                    __stcs(prow + r2 + N1 * k2, make_double2((double)z[k2].re, (double)z[k2].im));
            }
        }
        __syncthreads();
    }
    if (want_e && live && !interior) {
        R* ex = E + line * NX;
        R* ez = E + 2 * nodes + line * NX;
        for (int i = r; i < NX; i += TPC) {
            ex[i] = (R)0;
            ez[i] = (R)0;
        }
    }
}

template <class R, int M, int NZ>
__global__ void __launch_bounds__(kThreads, (fused_min_blocks<R, M, NZ>())) k_inv_fused(
    const cplx<R>* __restrict__ S, const cplx<R>* __restrict__ Fy, cplx<R>* ring, R* __restrict__ E,
    double* __restrict__ phi, int ny, int want_phi, int want_e, size_t nodes,
    const double* __restrict__ sinx, const double* __restrict__ sinz, const cplx<R>* __restrict__ twx_g,
    const cplx<R>* __restrict__ twz_g, PipeSync* sy, Pipe pipe, unsigned* err) {
    pdl_wait();
    using FX = fft::FourStep<M, kThreads>;
    constexpr int NX = 2 * M, NXH = M + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<R>* twx = reinterpret_cast<cplx<R>*>(smem_raw);     // exp(-2 pi i e / NX)
    cplx<R>* t2 = twx + NX;                                    // t2[k1 N2 + r] = W_M^(r k1)
    cplx<R>* twz = t2 + FX::N1 * FX::N2;
    cplx<R>* buf = twz + NZ;
    constexpr int BZ = fft::FourStep<NZ, kThreads>::BUF;
    R* sx = reinterpret_cast<R*>(buf + (FX::BUF > BZ ? FX::BUF : BZ));
    R* sz = sx + NXH;
    __shared__ unsigned s_next;
    for (int i = threadIdx.x; i < NX; i += kThreads) twx[i] = twx_g[i];
    for (int i = threadIdx.x; i < FX::N1 * FX::N2; i += kThreads) t2[i] = twx_g[2 * (i % FX::N2) * (i / FX::N2)];
    for (int i = threadIdx.x; i < NXH; i += kThreads) sx[i] = from_f64<R>(sinx[i]);
    for (int i = threadIdx.x; i < NZ; i += kThreads) {
        twz[i] = twz_g[i];
        sz[i] = from_f64<R>(sinz[i]);
    }
    const size_t slot_elems = 3 * (size_t)NZ * NXH;
    PipeLoop L{&s_next, 0u};
    pipe_start(L, sy);
    while (L.t < pipe.total) {
        bool cons;
        int plane, idx;
        pipe_task(pipe, L.t, cons, plane, idx);
        pipe_acquire(L, pipe, sy, cons, plane, err);
        cplx<R>* slot = ring + (size_t)(plane % pipe.P) * slot_elems;
        if (cons) inv_xtask<R, M>(slot, E, phi, ny, NZ, plane, idx, want_phi, want_e, nodes, twx, t2, sx, buf);
        else inv_ztask<R, NZ>(S, Fy, slot, ny, NXH, plane, idx, want_e, twz, sz, buf);
        pipe_release(L, sy, cons, plane);
    }
    // the last block to leave zeroes the counters for the next launch (so no memset, which
    // would keep this launch from being scheduled while the y solve drains, sits between them)
    __shared__ unsigned s_last;
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&sy->exited, 1u) == gridDim.x - 1 ? 1u : 0u;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        for (int i = threadIdx.x; i < kMaxPlanes; i += kThreads) {
            sy->a_done[i] = 0u;
            sy->b_done[i] = 0u;
        }
        if (threadIdx.x == 0) {
            sy->next = 0u;
            sy->exited = 0u;
        }
    }
}

template <class R, int M, int NZ>
size_t inv_fused_smem() {
    using FX = fft::FourStep<M, kThreads>;
    return sizeof(cplx<R>) * (2 * M + FX::N1 * FX::N2 + NZ + std::max(FX::BUF, fft::FourStep<NZ, kThreads>::BUF)) +
           sizeof(R) * (M + 1 + NZ);
}

// resident blocks per SM of a fused kernel (queried once per instantiation)
template <class K>
int fused_grid(K kernel, size_t smem, int num_sms, unsigned tasks, int* cache) {
    if (*cache == 0) {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kThreads, smem) != cudaSuccess || b < 1) b = 1;
        *cache = b;
    }
    return (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)tasks, (int64_t)*cache * num_sms));
}

template <class R, int M, int NZ>
tribo_status launch_inv_fused(tribo_ctx* c, void* E, double* phi) {
    const Pipe pipe = make_pipe(c->ny + 2, (c->nxh + fft::FourStep<NZ, kThreads>::W - 1) / fft::FourStep<NZ, kThreads>::W,
                                (NZ + fft::FourStep<M, kThreads>::W - 1) / fft::FourStep<M, kThreads>::W);
    PipeSync* sy = (PipeSync*)c->d_pipe;     // zero (at set-up, then left so by every launch)
    Pipe pipe_t = pipe;
    pipe_t.stall = c->test_stall_plane;
    static int occ = 0;
    const size_t smem = inv_fused_smem<R, M, NZ>();
    const int grid = fused_grid(k_inv_fused<R, M, NZ>, smem, c->num_sms, pipe.total, &occ);
    const size_t fstride = (size_t)NZ * (c->ny + 2) * c->nxh;
    (void)launch_pdl(k_inv_fused<R, M, NZ>, dim3(grid), dim3(kThreads), smem, c->stream,
        (const cplx<R>*)c->S, (const cplx<R>*)c->F + fstride, (cplx<R>*)c->ring, (R*)E, phi, c->ny,
        phi != nullptr ? 1 : 0, E != nullptr ? 1 : 0, (size_t)NZ * (c->ny + 2) * c->nx, c->d_sinx, c->d_sinz, (const cplx<R>*)c->d_twx,
        (const cplx<R>*)c->d_twz, sy, pipe_t, &c->d_acc->err);
    return TRIBO_OK;
}

template <class R, int M, int NZ>
tribo_status attr_fused(int optin) {
    if (inv_fused_smem<R, M, NZ>() + 64 > (size_t)optin) return TRIBO_ERR_UNSUPPORTED;
    // the fused kernel also holds a few bytes of static shared memory: its dynamic limit is its
    // own (fixed) need, which leaves room for it
    TRIBO_CUDA(cudaFuncSetAttribute(k_inv_fused<R, M, NZ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)inv_fused_smem<R, M, NZ>()));
    return TRIBO_OK;
}

// (nx/2, nz) pairs with a fused inverse pipeline (the grids whose intermediate fields
// outgrow L2 at the usual heights); other lengths run the split passes
#define TRIBO_FUSED_PAIRS(X) X(128, 256) X(192, 256) X(256, 256)

bool fused_pair(int m, int nz) {
#define CASE(M, NZ) if (m == M && nz == NZ) return true;
    TRIBO_FUSED_PAIRS(CASE)
#undef CASE
    return false;
}

template <class R>
tribo_status dispatch_inv_fused(tribo_ctx* c, void* E, double* phi) {
#define CASE(M, NZ) if (c->nx / 2 == M && c->nz == NZ) return launch_inv_fused<R, M, NZ>(c, E, phi);
    TRIBO_FUSED_PAIRS(CASE)
#undef CASE
    return TRIBO_ERR_UNSUPPORTED;
}
template <class R>
tribo_status dispatch_attr_fused(int m, int nz, int optin) {
#define CASE(M, NZ) if (m == M && nz == NZ) return attr_fused<R, M, NZ>(optin);
    TRIBO_FUSED_PAIRS(CASE)
#undef CASE
    return TRIBO_ERR_UNSUPPORTED;
}

// tw[e] = exp(-2 pi i e / n), e < n; for the x length (with_inner) also the four-step's inner
// twiddles of M = n/2 = N1 N2 laid out by thread: tw[n + k1 N2 + r] = W_M^(r k1), so that the
// 16 threads of a column read 16 consecutive values (the lookup tw[2 r k1] hits one shared-memory
// bank several times over)
template <class R>
tribo_status twiddles(int n, void** dst, bool with_inner = false) {
    int n1 = 1, n2 = 0;
    if (with_inner) {
        const int m = n / 2;
        for (int d = 1; d * d <= m; ++d)
            if (m % d == 0) n1 = d;
        n2 = m / n1;
    }
    std::vector<cplx<R>> tw(n + (size_t)n1 * n2);
    for (int e = 0; e < n; ++e) {
        const double a = 2.0 * M_PI * (double)e / (double)n;
        tw[e] = cplx<R>{(R)std::cos(a), (R)(-std::sin(a))};
    }
    for (int k1 = 0; k1 < n1 && with_inner; ++k1)
        for (int r = 0; r < n2; ++r) tw[n + (size_t)k1 * n2 + r] = tw[(size_t)2 * r * k1];
    TRIBO_CUDA(cudaMalloc(dst, sizeof(cplx<R>) * tw.size()));
    TRIBO_CUDA(cudaMemcpy(*dst, tw.data(), sizeof(cplx<R>) * tw.size(), cudaMemcpyHostToDevice));
    return TRIBO_OK;
}

void split_ds(double v, float* hi, float* lo) {
    *hi = (float)v;
    *lo = (float)(v - (double)*hi);
}

template <class R>
tribo_status solve_fast(tribo_ctx* c, void* src, bool src_f64, const double* scale, bool zero_src, double* phi,
                        void* E) {
    const int ny = c->ny, nz = c->nz, nxh = c->nxh;
    // the inverse transforms as one pipelined launch where the grid has one, except in a batch,
    // whose channels solve side by side on their own streams (a launch that waits on its own
    // tasks would hold SMs the other channels' passes could use)
    // (the potential-only solves of the adjoint also keep the split passes)
    const bool fused = c->ring != nullptr && !c->in_batch && E != nullptr;
    const PassGrid<R> g{c->nx, ny, nz, nxh, c->num_sms, c->stream};
    const cplx<R>* twx = (const cplx<R>*)c->d_twx;
    const cplx<R>* twz = (const cplx<R>*)c->d_twz;
    phase_begin(c, PH_FWD_X);
    xfwd_launch<R>(g, src, src_f64, scale, zero_src, (cplx<R>*)c->S, twx);
    TRIBO_LAUNCHED(c);
    phase_begin(c, PH_FWD_Z);
    zfwd_launch<R>(g, (cplx<R>*)c->S, twz);
    TRIBO_LAUNCHED(c);
    const size_t fstride = (size_t)nz * (ny + 2) * nxh;
    const int ni = (nz / 2 + 1) * nxh;
    phase_begin(c, PH_SOLVE_Y);
    if constexpr (sizeof(R) == 8) {
        const double* te = (const double*)c->d_ytab;
        const unsigned nblk = (unsigned)(((int64_t)nz * nxh + 31) / 32);     // 32 pencils a block of 128
        (void)launch_pdl(k_ysolve64<double>, dim3(nblk), dim3(128), ysolve64_smem(ny), c->stream, (cplx<double>*)c->S,
                         (cplx<double>*)c->F, te, te + (size_t)(ny + 1) * ni, (const double*)c->d_ycoef,
                         (const double*)c->d_ey, ny, nz, nxh, E != nullptr ? 1 : 0);
    } else {
        // without E (the adjoint's potential-only solves) the E_y spectrum is not written
        const float2* te = (const float2*)c->d_ytab;
        auto solve = E ? ysolve_twist_launch<true, false> : ysolve_twist_launch<false, false>;
        solve((int64_t)nz * nxh, 1, c->num_sms, ny, c->stream, (cplx<float>*)c->S, (cplx<float>*)c->F, te,
              te + (size_t)(ny + 1) * ni, (const float2*)c->d_ycpl, (const float4*)c->d_yec, (float4*)c->d_yck, nz, nxh,
              nullptr);
    }
    TRIBO_LAUNCHED(c);
    if (fused) {
        phase_begin(c, PH_INV_Z);
        tribo_status st = dispatch_inv_fused<R>(c, E, phi);
        if (st) return st;
        TRIBO_LAUNCHED(c);
        return TRIBO_OK;
    }
    phase_begin(c, PH_INV_Z);
    zinv_launch<R>(g, (const cplx<R>*)c->S, (cplx<R>*)c->F, c->d_sinz, twz, E == nullptr);
    TRIBO_LAUNCHED(c);
    phase_begin(c, PH_INV_X);
    xinv_launch<R>(g, (const cplx<R>*)c->F, (R*)E, phi, c->d_sinx, twx);
    TRIBO_LAUNCHED(c);
    return TRIBO_OK;
}

}  // namespace

tribo_status poisson_fast_setup(tribo_ctx* c) {
    const int nx = c->nx, ny = c->ny, nz = c->nz, nxh = c->nxh;
    const int ni = (nz / 2 + 1) * nxh;
    const std::vector<double>& yf = c->yf;
    const std::vector<double>& yc = c->yc;
    const std::vector<double>& dy = c->dy;
    // the y operator, for the couplings and E_y coefficients of the mixed solve
    std::vector<double> a(ny, 0.0), b(ny), cc(ny, 0.0);
    for (int j = 0; j < ny; ++j) {
        if (j >= 1) a[j] = 1.0 / (dy[j] * (yc[j] - yc[j - 1]));
        if (j <= ny - 2) cc[j] = 1.0 / (dy[j] * (yc[j + 1] - yc[j]));
        b[j] = -(a[j] + cc[j]);
    }
    b[0] -= 1.0 / (dy[0] * (yc[0] - yf[0]));
    b[ny - 1] -= 1.0 / (dy[ny - 1] * (yf[ny] - yc[ny - 1]));
    const bool ds_mode = c->prec != TRIBO_FP64;
    const int kmid = ny / 2;         // the twisted solve's middle row
    const size_t rows = 2 * (size_t)ny + 1;
    TRIBO_CUDA(cudaMalloc(&c->d_ytab, 8 * rows * ni));
    if (ds_mode) {
        float2* te = (float2*)c->d_ytab;
        k_ytab<<<(ni + 127) / 128, 128>>>(c->d_ycoef, c->d_lamx, c->d_lamz, ny, nz, nxh, te,
                                          te + (size_t)(ny + 1) * ni);
    } else {
        double* te = (double*)c->d_ytab;
        k_ytab<<<(ni + 127) / 128, 128>>>(c->d_ycoef, c->d_lamx, c->d_lamz, ny, nz, nxh, te,
                                          te + (size_t)(ny + 1) * ni);
    }
    TRIBO_CUDA(cudaGetLastError());
    if (ds_mode) {
        // couplings of the substitution in double-single: c_j (rows 0..k-1), a_j (rows k..ny-1);
        // E_y coefficients per cell and walls
        std::vector<float2> cpl(ny);
        for (int j = 0; j < ny; ++j) split_ds(j < kmid ? cc[j] : a[j], &cpl[j].x, &cpl[j].y);
        auto w = [&](int f) { return (yf[f] - yc[f - 1]) / (yc[f] - yc[f - 1]); };
        std::vector<float4> ec(ny + 1, make_float4(0, 0, 0, 0));
        for (int j = 0; j < ny; ++j) {
            double A = 0, Bm = 0, Bp = 0;
            if (j == 0) A -= 1.0 / dy[j];           // -phi_f[1] / dy_0 = -(phi_0 + w_1 d1) / dy_0
            if (j == ny - 1) A += 1.0 / dy[j];      // +phi_f[ny-1] / dy = (phi_ny-1 - (1-w) d0) / dy
            if (j >= 1) Bm = -(1.0 - w(j)) / dy[j];
            if (j <= ny - 2) Bp = -w(j + 1) / dy[j];
            ec[j] = make_float4((float)A, (float)Bm, (float)Bp, 0.f);
        }
        ec[ny] = make_float4((float)(-1.0 / (yc[0] - yf[0])), (float)(1.0 / (yf[ny] - yc[ny - 1])), 0.f, 0.f);
        TRIBO_CUDA(cudaMalloc(&c->d_ycpl, sizeof(float2) * ny));
        TRIBO_CUDA(cudaMemcpy(c->d_ycpl, cpl.data(), sizeof(float2) * ny, cudaMemcpyHostToDevice));
        // chunk checkpoints of the twisted sweeps
        const int cmin = std::min(kTwistC1, kTwistC2);        // the launch with more chunks
        const size_t nck = (size_t)std::max(1, (kmid + cmin - 1) / cmin - 1) * 2 * (size_t)nz * nxh;
        TRIBO_CUDA(cudaMalloc(&c->d_yck, sizeof(float4) * nck));
        TRIBO_CUDA(cudaMalloc(&c->d_yec, sizeof(float4) * (ny + 1)));
        TRIBO_CUDA(cudaMemcpy(c->d_yec, ec.data(), sizeof(float4) * (ny + 1), cudaMemcpyHostToDevice));
    }
    int dev = 0, optin = 0;
    TRIBO_CUDA(cudaGetDevice(&dev));
    TRIBO_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    tribo_status st;
    // grids with a fused inverse pipeline: the ring of plane slots (three fields per slot) and
    // the launch's task counters
    const size_t csz0 = c->prec == TRIBO_FP64 ? sizeof(cplx<double>) : sizeof(cplx<float>);
    if (fused_pair(nx / 2, nz) && 3 * (size_t)nz * (ny + 2) * nxh * csz0 >= ((size_t)64 << 20)) {
        const size_t csz = c->prec == TRIBO_FP64 ? sizeof(cplx<double>) : sizeof(cplx<float>);
        st = c->prec == TRIBO_FP64 ? dispatch_attr_fused<double>(nx / 2, nz, optin)
                                   : dispatch_attr_fused<float>(nx / 2, nz, optin);
        if (st == TRIBO_OK) {
            TRIBO_CUDA(cudaMalloc(&c->ring, (size_t)kPipeSlots * 3 * nz * nxh * csz));
            TRIBO_CUDA(cudaMalloc(&c->d_pipe, sizeof(PipeSync)));
            TRIBO_CUDA(cudaMemset(c->d_pipe, 0, sizeof(PipeSync)));
        } else if (st != TRIBO_ERR_UNSUPPORTED) {
            return st;
        }
    }
    if (c->prec == TRIBO_FP64) {
        if ((st = twiddles<double>(nx, &c->d_twx, true)) || (st = twiddles<double>(nz, &c->d_twz))) return st;
        if ((st = zpass_attr<double>(nz, optin))) return st;
        return xpass_attr<double>(nx / 2, optin);
    }
    if ((st = twiddles<float>(nx, &c->d_twx, true)) || (st = twiddles<float>(nz, &c->d_twz))) return st;
    c->smem_optin = optin;
    if ((st = zpass_attr<float>(nz, optin))) return st;
    return xpass_attr<float>(nx / 2, optin);
}

void poisson_fast_free(tribo_ctx* c) {
    cudaFree(c->d_ytab);
    cudaFree(c->d_twx);
    cudaFree(c->d_twz);
    cudaFree(c->d_ycpl);
    cudaFree(c->d_yec);
    cudaFree(c->d_yck);
    c->d_yck = nullptr;
    cudaFree(c->ring);
    cudaFree(c->d_pipe);
    c->d_ytab = c->d_twx = c->d_twz = c->d_ycpl = c->d_yec = c->ring = c->d_pipe = nullptr;
}

tribo_status poisson_solve(tribo_ctx* c, void* src, bool src_f64, const double* scale, bool zero_src,
                           double* phi, void* E) {
    if (c->prec == TRIBO_FP64) return solve_fast<double>(c, src, true, scale, zero_src, phi, E);
    return solve_fast<float>(c, src, src_f64, scale, zero_src, phi, E);
}

}  // namespace tribo
