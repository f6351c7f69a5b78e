// 4-way coupling: hard-sphere particle-particle collisions (Sec. 2.2) with the
// condenser-model charge exchange of a particle-particle contact (Sec. 2.3.1),
// applied to the end-of-step state after the wall impacts.
//
// Candidates are the particles of the same cell (cell lists of the end-of-
// step positions).  A pair collides when the spheres overlap, approach each
// other ((v_i - v_j).(s_i - s_j) < 0) and each is the other's nearest such
// partner (ties to the lower index):
//   k_pp_partner  per particle, its nearest valid partner (or none);
//   k_pp_collide  the lower index of every mutual pair updates both particles:
//                 elastic impulse along the line of centres with the masses,
//                 v_i' = v_i - 2 m_j/(m_i+m_j) ((v_i - v_j).n) n (and the
//                 opposite for j), and the charge exchange
//                 dq_ij = C_i C_j/(C_i+C_j) (q_j/C_j - q_i/C_i) (1 - exp(-dt_12/T_12))
//                 with C = 4 pi eps d/2, T_12 = C_i C_j/(C_i+C_j) (d_i+d_j)/(2 A_12) phi_p,
//                 A_12 = pi d_i d_j/(2(d_i+d_j)) alpha_12, dt_12 = 2.94 alpha_12/|u_12|,
//                 alpha_12 = (d_i d_j/2)(5/8 pi rho_p (1+k_e) |u_12|^2 sqrt(d_i+d_j)/(d_i^3+d_j^3) el)^(2/5),
//                 el = 2 (1 - mu_p^2)/E_p (the two bodies' (1 - mu^2)/E of one material).
// Both particles of a pair share a cell, so the cell's deposited charge sum
// is unchanged.  Decisions and updates are formed in FP64 from the stored
// values (same-cell position differences of FP32 numbers are exact), so the
// choice of pairs does not depend on the precision of the state; pairs
// clearly apart are rejected first in the real type (with a 1e-4 relative
// margin on the squared contact distance, far above its rounding).
#include <algorithm>
#include <cmath>

#include "particle_math.cuh"

namespace tribo {
namespace {

constexpr uint32_t kNone = 0xffffffffu;

template <class R>
__global__ void __launch_bounds__(kThreads) k_pp_partner(PView p, const uint32_t* __restrict__ key,
                                                         const uint32_t* __restrict__ offsets,
                                                         const uint32_t* __restrict__ members, uint32_t ncell,
                                                         uint32_t* __restrict__ partner) {
    pdl_wait();
    const R* X = (const R*)p.x; const R* Y = (const R*)p.y; const R* Z = (const R*)p.z;
    const R* VX = (const R*)p.vx; const R* VY = (const R*)p.vy; const R* VZ = (const R*)p.vz;
    const R* D = (const R*)p.d;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < p.n; n += stride) {
        const uint32_t k = key[n];
        const uint32_t b = offsets[k];
        const uint32_t e = k + 1 < ncell ? offsets[k + 1] : (uint32_t)p.n;
        uint32_t best = kNone;
        if (e - b > 1) {
            double bd = 0.0;
            const R xr = X[n], yr = Y[n], zr = Z[n], dr = D[n];
            for (uint32_t m = b; m < e; ++m) {
                const uint32_t j = members[m];
                if (j == (uint32_t)n) continue;
                // cheap rejection in the real type, with a margin far above its rounding
                const R fx = xr - X[j], fy = yr - Y[j], fz = zr - Z[j];
                const R freach = (R)0.5 * (dr + D[j]);
                if (fx * fx + fy * fy + fz * fz > freach * freach * (R)1.0001) continue;
                // the few that remain are decided in FP64 (the conversions issue at its rate)
                const double rx = (double)xr - (double)X[j], ry = (double)yr - (double)Y[j], rz = (double)zr - (double)Z[j];
                const double d2 = rx * rx + ry * ry + rz * rz;
                const double reach = 0.5 * ((double)dr + (double)D[j]);
                if (!(d2 < reach * reach)) continue;
                const double dot = ((double)VX[n] - (double)VX[j]) * rx + ((double)VY[n] - (double)VY[j]) * ry +
                                   ((double)VZ[n] - (double)VZ[j]) * rz;
                if (!(dot < 0.0)) continue;
                if (best == kNone || d2 < bd || (d2 == bd && j < best)) {
                    best = j;
                    bd = d2;
                }
            }
        }
        partner[n] = best;
    }
}

// the collision of the mutual pair (n, j): both particles' velocities and charges
template <class R>
__device__ __forceinline__ void collide_pair(const PView& p, uint32_t n, uint32_t j, double rho_p, double k_e, double el,
                                             double eps, double phi_p) {
    const R* X = (const R*)p.x; const R* Y = (const R*)p.y; const R* Z = (const R*)p.z;
    R* VX = (R*)p.vx; R* VY = (R*)p.vy; R* VZ = (R*)p.vz;
    const R* D = (const R*)p.d;
    const double rx = (double)X[n] - (double)X[j], ry = (double)Y[n] - (double)Y[j],
                 rz = (double)Z[n] - (double)Z[j];
    const double inv = 1.0 / sqrt(rx * rx + ry * ry + rz * rz);
    const double nx = rx * inv, ny = ry * inv, nz = rz * inv;
    const double ui = VX[n], vi = VY[n], wi = VZ[n];
    const double uj = VX[j], vj = VY[j], wj = VZ[j];
    const double di = D[n], dj = D[j];
    const double vn = (ui - uj) * nx + (vi - vj) * ny + (wi - wj) * nz;
    const double mi = M_PI * rho_p * di * di * di / 6.0, mj = M_PI * rho_p * dj * dj * dj / 6.0;
    const double ci = 2.0 * mj / (mi + mj) * vn, cj = 2.0 * mi / (mi + mj) * vn;
    // charge exchange with the relative speed before the collision
    const double du = uj - ui, dv = vj - vi, dw = wj - wi;
    const double speed = sqrt(du * du + dv * dv + dw * dw);
    const double qi = p.q[n], qj = p.q[j];
    double dq = 0.0;
    if (speed > 0.0) {
        const double Ci = 2.0 * M_PI * eps * di, Cj = 2.0 * M_PI * eps * dj;
        const double alpha = 0.5 * di * dj *
                             pow04(0.625 * M_PI * rho_p * (1.0 + k_e) * speed * speed * sqrt(di + dj) /
                                   (di * di * di + dj * dj * dj) * el);
        const double A = M_PI * di * dj / (2.0 * (di + dj)) * alpha;
        const double dt = 2.94 * alpha / speed;
        const double Cs = Ci * Cj / (Ci + Cj);
        const double T = Cs * (di + dj) / (2.0 * A) * phi_p;
        dq = Cs * (qj / Cj - qi / Ci) * one_minus_exp(dt / T);
    }
    VX[n] = (R)(ui - ci * nx); VY[n] = (R)(vi - ci * ny); VZ[n] = (R)(wi - ci * nz);
    VX[j] = (R)(uj + cj * nx); VY[j] = (R)(vj + cj * ny); VZ[j] = (R)(wj + cj * nz);
    p.q[n] = qi + dq;
    p.q[j] = qj - dq;
}

// Few particles collide (about 1 in 1000 at 1M particles in 128^3 cells), and the exchange is some
// 400 FP64 operations: run where it is found, each pair held a warp of its own and an SM's FP64
// pipe, one lane in 32 in use (23.5 us a launch).  So the block lists the pairs of its particles
// in shared memory and works through the list with all its lanes: 14.0 us.
constexpr int kCollideThreads = 512;                  // at most; a block looks at 4 particles a thread per round
template <class R>
__global__ void __launch_bounds__(kCollideThreads) k_pp_collide(PView p, const uint32_t* __restrict__ partner,
                                                                double rho_p, double k_e, double el, double eps,
                                                                double phi_p) {
    pdl_wait();
    __shared__ uint32_t list[2 * 4 * kCollideThreads];
    __shared__ unsigned int count;
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    const unsigned per = 4 * blockDim.x;              // particles of a round
    const int64_t stride = (int64_t)gridDim.x * per;
    for (int64_t n0 = (int64_t)blockIdx.x * per; n0 < p.n; n0 += stride) {
        const int64_t n = n0 + 4 * threadIdx.x;
        uint32_t j[4] = {kNone, kNone, kNone, kNone};
        if (n + 4 <= p.n) {                           // one 16-byte load (n is a multiple of 4)
            const uint4 v = *reinterpret_cast<const uint4*>(partner + n);
            j[0] = v.x; j[1] = v.y; j[2] = v.z; j[3] = v.w;
        } else {
            for (int i = 0; i < 4; ++i)
                if (n + i < p.n) j[i] = partner[n + i];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t me = (uint32_t)(n + i);
            if (j[i] != kNone && j[i] > me && partner[j[i]] == me) list[atomicAdd(&count, 1u)] = me;
        }
        __syncthreads();
        const unsigned int m = count;
        __syncthreads();
        // a round adds at most `per`, so the list is emptied when it could not take another
        if (m > per || n0 + stride >= p.n) {
            for (unsigned int i = threadIdx.x; i < m; i += blockDim.x)
                collide_pair<R>(p, list[i], partner[list[i]], rho_p, k_e, el, eps, phi_p);
            if (threadIdx.x == 0) count = 0;
            __syncthreads();
        }
    }
}

template <class R>
tribo_status collide_impl(tribo_ctx* c, const PView& p, const uint32_t* members, uint32_t* partner) {
    const uint32_t ncell = (uint32_t)((size_t)c->nx * c->ny * c->nz);
    phase_begin(c, PH_AUX);
    (void)launch_pdl(k_pp_partner<R>, dim3(grid_for(p.n)), dim3(kThreads), 0, c->stream, p, (const uint32_t*)c->sort_key,
                     (const uint32_t*)c->sort_counts, members, ncell, partner);
    TRIBO_LAUNCHED(c);
    const tribo_params& P = c->P;
    phase_begin(c, PH_AUX);
    // Few particles in small blocks, up to two per SM, so that their pairs spread over the SMs; past
    // 2 x 1024 particles a SM blocks of 512, one a SM, whose lists fill the lanes.  A step of 2000
    // particles that all collide: 122 us in blocks of 512, 76 so; of 40,000: 136, 89; from 311,296
    // particles on the same launch as before.
    int threads = 64;
    while (threads < kCollideThreads && p.n > (int64_t)2 * c->num_sms * 4 * threads) threads *= 2;
    const int64_t blocks = std::min<int64_t>((p.n + 4 * threads - 1) / (4 * threads),
                                             (int64_t)c->num_sms * (threads == kCollideThreads ? 1 : 2));
    (void)launch_pdl(k_pp_collide<R>, dim3((unsigned)blocks), dim3(threads), 0, c->stream, p, (const uint32_t*)partner,
                     P.rho_p, P.k_e, 2.0 * (1.0 - P.mu_p * P.mu_p) / P.E_p, P.eps, P.phi_p);
    TRIBO_LAUNCHED(c);
    return TRIBO_OK;
}

}  // namespace

tribo_status particles_collide(tribo_ctx* c, const PView& p, const uint32_t* members, uint32_t* partner) {
    if (p.n == 0) return TRIBO_OK;
    if (c->prec == TRIBO_FP64) return collide_impl<double>(c, p, members, partner);
    return collide_impl<float>(c, p, members, partner);
}

}  // namespace tribo
