// Electrostatic Poisson solve and E = -grad(phi) on the channel grid.
//
// Sec. 2.2: laplacian(phi) = -rho_el / eps, the charge density of a grid cell
// being the sum of its particles' charges over the cell volume, and
// E = -grad(phi).  Sec. 3.1: second-order finite volumes; the walls are
// grounded conductors (phi = 0), which gives the image-charge attraction
// discussed in Sec. 4.2.
//
// Discretisation (the paper gives neither stencil nor gradient scheme): the
// 3-point operator in x and z and the flux form on the stretched y grid, with
// phi = 0 on the wall faces.  The DFT in x and z diagonalises the x and z
// parts with modified wavenumbers lam(m) = (4/h^2) sin^2(pi m / N), leaving a
// real tridiagonal system in y per (m_x, m_z) pencil.  E is formed in spectral space: the central difference in
// x (z) is the multiplier -i sin(2 pi m / N) / h, and the Gauss-linear E_y at
// each lattice node is a 3-point combination of phi in y; the spectra are then
// transformed back to the wall-extended lattice.
//
// The passes are in poisson_passes.cuh (transforms, mixed y solve) and
// poisson_y64.cuh (FP64 y solve); a context's solve is in poisson_fast.cu.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <algorithm>
#include <mutex>

#include "poisson_y64.cuh"
#include "tribo_internal.cuh"

namespace tribo {

tribo_status poisson_setup(tribo_ctx* c) {
    const int nx = c->nx, ny = c->ny, nz = c->nz, nxh = c->nxh;
    const std::vector<double>& yf = c->yf;
    const std::vector<double>& yc = c->yc;
    const std::vector<double>& dy = c->dy;
    // y operator coefficients (rows: a[j] phi[j-1] + b[j] phi[j] + c[j] phi[j+1])
    std::vector<double> coef(3 * ny, 0.0);
    double* a = coef.data();
    double* b = a + ny;
    double* cc = b + ny;
    for (int j = 0; j < ny; ++j) {
        if (j >= 1) a[j] = 1.0 / (dy[j] * (yc[j] - yc[j - 1]));
        if (j <= ny - 2) cc[j] = 1.0 / (dy[j] * (yc[j + 1] - yc[j]));
        b[j] = -(a[j] + cc[j]);
    }
    b[0] -= 1.0 / (dy[0] * (yc[0] - yf[0]));
    b[ny - 1] -= 1.0 / (dy[ny - 1] * (yf[ny] - yc[ny - 1]));
    std::vector<double> lamx(nx), lamz(nz), sinx(nxh), sinz(nz);
    for (int m = 0; m < nx; ++m) {
        const double s = std::sin(M_PI * m / nx);
        lamx[m] = 4.0 / (c->dx * c->dx) * s * s;
    }
    for (int m = 0; m < nz; ++m) {
        const double s = std::sin(M_PI * m / nz);
        lamz[m] = 4.0 / (c->dz * c->dz) * s * s;
        sinz[m] = std::sin(2.0 * M_PI * m / nz) / c->dz;
    }
    for (int m = 0; m < nxh; ++m) sinx[m] = std::sin(2.0 * M_PI * m / nx) / c->dx;
    // E_y at lattice node jn = cm phi[jn-2] + c0 phi[jn-1] + cp phi[jn]
    std::vector<double> ey(3 * (ny + 2), 0.0);
    auto w = [&](int f) { return (yf[f] - yc[f - 1]) / (yc[f] - yc[f - 1]); };  // interior face f
    for (int j = 0; j < ny; ++j) {
        const int jn = j + 1;
        double cm = 0, c0 = 0, cp = 0;
        // + phi_f[j] / dy_j
        if (j >= 1) { cm += (1.0 - w(j)) / dy[j]; c0 += w(j) / dy[j]; }
        // - phi_f[j+1] / dy_j
        if (j + 1 <= ny - 1) { c0 -= (1.0 - w(j + 1)) / dy[j]; cp -= w(j + 1) / dy[j]; }
        ey[3 * jn + 0] = cm;
        ey[3 * jn + 1] = c0;
        ey[3 * jn + 2] = cp;
    }
    ey[3 * 0 + 2] = -1.0 / (yc[0] - yf[0]);                    // bottom wall node
    ey[3 * (ny + 1) + 0] = 1.0 / (yf[ny] - yc[ny - 1]);        // top wall node

    TRIBO_CUDA(cudaMalloc(&c->d_ycoef, sizeof(double) * 3 * ny));
    TRIBO_CUDA(cudaMalloc(&c->d_lamx, sizeof(double) * nx));
    TRIBO_CUDA(cudaMalloc(&c->d_lamz, sizeof(double) * nz));
    TRIBO_CUDA(cudaMalloc(&c->d_sinx, sizeof(double) * nxh));
    TRIBO_CUDA(cudaMalloc(&c->d_sinz, sizeof(double) * nz));
    TRIBO_CUDA(cudaMalloc(&c->d_ey, sizeof(double) * 3 * (ny + 2)));
    TRIBO_CUDA(cudaMemcpy(c->d_ycoef, coef.data(), sizeof(double) * 3 * ny, cudaMemcpyHostToDevice));
    TRIBO_CUDA(cudaMemcpy(c->d_lamx, lamx.data(), sizeof(double) * nx, cudaMemcpyHostToDevice));
    TRIBO_CUDA(cudaMemcpy(c->d_lamz, lamz.data(), sizeof(double) * nz, cudaMemcpyHostToDevice));
    TRIBO_CUDA(cudaMemcpy(c->d_sinx, sinx.data(), sizeof(double) * nxh, cudaMemcpyHostToDevice));
    TRIBO_CUDA(cudaMemcpy(c->d_sinz, sinz.data(), sizeof(double) * nz, cudaMemcpyHostToDevice));
    TRIBO_CUDA(cudaMemcpy(c->d_ey, ey.data(), sizeof(double) * 3 * (ny + 2), cudaMemcpyHostToDevice));

    const size_t rsz = c->prec == TRIBO_FP64 ? sizeof(double) : sizeof(float);
    const size_t csz = 2 * rsz;
    TRIBO_CUDA(cudaMalloc(&c->S, csz * (size_t)nz * ny * nxh));
    TRIBO_CUDA(cudaMalloc(&c->F, csz * 4 * (size_t)nz * (ny + 2) * nxh));
    return poisson_fast_setup(c);
}

tribo_status poisson_free(tribo_ctx* c) {
    cudaFree(c->d_ycoef);
    cudaFree(c->d_lamx);
    cudaFree(c->d_lamz);
    cudaFree(c->d_sinx);
    cudaFree(c->d_sinz);
    cudaFree(c->d_ey);
    cudaFree(c->S);
    cudaFree(c->F);
    poisson_fast_free(c);
    return TRIBO_OK;
}

}  // namespace tribo

// ---------------------------------------------------------------------------
// tribo_poisson_noalloc: the standalone Poisson solve for callers that must
// not allocate device memory.  Some hosts cannot call cudaMalloc once they are
// running: a framework whose caching allocator has already reserved the
// device's memory, a real-time loop where an allocation's latency or failure
// mid-run is not acceptable, or a plug-in that is only ever handed
// pre-allocated buffers.  This variant keeps its scratch (coefficient tables,
// twiddles, y factors, spectra) in one fixed file-scope device
// array instead of a context's allocations.  It has no counterpart in the
// paper.  Its tables are written into the array by its first kernel, from the
// grid passed by value, so nothing is staged in or copied from host memory.
//
// The array is static device memory of this library: every GPU that loads
// the library holds it until the process exits.  Host code cannot use the
// array's name as a device address, so the first call on each device (with
// that device current) looks the address up once with cudaGetSymbolAddress
// and keeps it; it also loads the kernels of every transform length and both
// precisions (16 ms more than those of one grid), since code that CUDA loads at a
// kernel's first launch takes device memory then.  That first call should
// therefore come before any stream capture; later ones set nothing up, whatever
// their grid.  All calls share the array and it keeps the last call's contents:
// each call rewrites every byte it reads before reading it, and two calls
// whose work overlaps on the GPU (different streams or devices sharing
// nothing but this array on one device) race with each other.
namespace tribo {
namespace {

constexpr size_t kNoallocScratchBytes = size_t(32) << 20;   // 32 MiB
constexpr int kNoallocMaxN = 256;                            // nx, ny, nz limit
constexpr int kNoallocMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

struct NoallocDevice {
    unsigned char* base = nullptr;
    int num_sms = 1;
    bool ready = false;
};
NoallocDevice g_noalloc_dev[kNoallocMaxDevices];
std::mutex g_noalloc_mutex;

size_t round256(size_t b) { return (b + 255) / 256 * 256; }

// The rule by which the call takes a grid, part of its interface: the bytes that a spectrum, nf field
// spectra and 24 bytes per pencil and row beside the tables come to may not exceed the array.  It is
// an upper bound of the layout below (at most 26.7 MiB for every grid it lets through) and stays, so
// that what the call refuses does not depend on how the solve uses the array.
size_t noalloc_capacity(int nx, int ny, int nz, int nf, size_t rsz) {
    const size_t csz = 2 * rsz;
    const int nxh = nx / 2 + 1;
    const size_t tables = (size_t)3 * ny + nx + nz + nxh + nz + 3 * (ny + 2) + ny;
    return round256(tables * sizeof(double)) + round256((size_t)nx * csz) + round256((size_t)nz * csz) +
           round256((size_t)nz * ny * nxh * csz) + round256((size_t)nf * nz * (ny + 2) * nxh * csz) +
           round256((size_t)ny * nz * nxh * (sizeof(double2) + sizeof(double)));
}

// What the solve uses of the array: tables, twiddles (x: with their inner table), y factors (2 ny + 1
// rows of (nz/2+1) nxh doubles), the spectrum and three field spectra (the potential needs none).
struct NoallocLayout {
    size_t tables, twx, twz, te, S, F, total;
};
NoallocLayout noalloc_layout(int nx, int ny, int nz, size_t rsz) {
    const size_t csz = 2 * rsz;
    const int nxh = nx / 2 + 1;
    NoallocLayout L{};
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += round256(bytes); return o; };
    L.tables = take(((size_t)3 * ny + nxh + nz + 3 * (ny + 2) + ny) * sizeof(double));
    L.twx = take(((size_t)nx + nx / 2) * csz);
    L.twz = take((size_t)nz * csz);
    L.te = take((size_t)(2 * ny + 1) * (nz / 2 + 1) * nxh * sizeof(double));
    L.S = take((size_t)nz * ny * nxh * csz);
    L.F = take((size_t)3 * nz * (ny + 2) * nxh * csz);
    L.total = off;
    return L;
}

// Everything the solve needs besides the caller's arrays, passed by value to
// the table kernel (no host buffer is copied: the call neither blocks on nor
// reads host memory after it returns).
struct NoallocGeom {
    int nx, ny, nz, n1;
    double dx, dz, scale;        // scale: -1 / (2 eps nx nz)
    double yf[kNoallocMaxN + 1];
};

// The grid tables of the solve, written into the front of the scratch array: the y operator (a, b,
// c), the spectral derivative factors, the E_y node coefficients, the per-row RHS scale -1/(eps nx nz)
// and the x and z twiddles by block 0 (the same formulas as poisson_setup and the contexts' tables,
// Sec. 2.2, Sec. 3.1 FV operator), the y factors by the others, two neighbouring threads a wavenumber
// pair, from the y operator that each block forms for itself in shared memory.  Bound by the latency of
// a thread's chain of ny/2 FP64 divisions; the passes after it are those of a context (a mixed 64^3
// call: 202 us with one kernel a sweep over generic transforms, 62.5 us so).  Measured and not taken:
// one-warp blocks with a value a thread (64.4 us), factors by continuants without the divisions in the
// chain (72.8 us, more FP64 operations).
template <class R>
__global__ void __launch_bounds__(128) k_noalloc_tables(NoallocGeom g, double* __restrict__ T, cplx<R>* __restrict__ twx,
                                                        cplx<R>* __restrict__ twz, double* __restrict__ te) {
    pdl_wait();
    __shared__ double sy[3 * kNoallocMaxN];
    const int nx = g.nx, ny = g.ny, nz = g.nz, nxh = nx / 2 + 1;
    const double* yf = g.yf;
    auto yc = [&](int j) { return 0.5 * (yf[j] + yf[j + 1]); };
    auto dy = [&](int j) { return yf[j + 1] - yf[j]; };
    for (int j = threadIdx.x; j < ny; j += blockDim.x) {
        const double aj = (j >= 1) ? 1.0 / (dy(j) * (yc(j) - yc(j - 1))) : 0.0;
        const double cj = (j <= ny - 2) ? 1.0 / (dy(j) * (yc(j + 1) - yc(j))) : 0.0;
        double bj = -(aj + cj);
        if (j == 0) bj -= 1.0 / (dy(0) * (yc(0) - yf[0]));
        if (j == ny - 1) bj -= 1.0 / (dy(ny - 1) * (yf[ny] - yc(ny - 1)));
        sy[j] = aj;
        sy[ny + j] = bj;
        sy[2 * ny + j] = cj;
    }
    __syncthreads();
    if (blockIdx.x > 0) {
        const int ni = (nz / 2 + 1) * nxh;
        const int t = (blockIdx.x - 1) * blockDim.x + threadIdx.x;
        const int item = min(t >> 1, ni - 1);           // threads past the end repeat the last pair's work
        const double sx = sin(M_PI * (item % nxh) / nx), sz = sin(M_PI * (item / nxh) / nz);
        const double lam = 4.0 / (g.dz * g.dz) * sz * sz + 4.0 / (g.dx * g.dx) * sx * sx;
        y_factors(sy, lam, ny, ni, item, 1 + (t & 1), te, te + (size_t)(ny + 1) * ni);
        return;
    }
    double* sinx = T + 3 * ny;
    double* sinz = sinx + nxh;
    double* ey = sinz + nz;
    double* scale = ey + 3 * (ny + 2);
    for (int j = threadIdx.x; j < 3 * ny; j += blockDim.x) T[j] = sy[j];
    for (int j = threadIdx.x; j < ny; j += blockDim.x) {
        if constexpr (sizeof(R) == 8) scale[j] = g.scale;
        else reinterpret_cast<float2*>(scale)[j] = make_float2((float)g.scale, (float)(g.scale - (double)(float)g.scale));
        // E_y at lattice node jn = j + 1: cm phi[j-1] + c0 phi[j] + cp phi[j+1]
        double cm = 0, c0 = 0, cp = 0;
        if (j >= 1) {
            const double w = (yf[j] - yc(j - 1)) / (yc(j) - yc(j - 1));
            cm += (1.0 - w) / dy(j);
            c0 += w / dy(j);
        }
        if (j + 1 <= ny - 1) {
            const double w = (yf[j + 1] - yc(j)) / (yc(j + 1) - yc(j));
            c0 -= (1.0 - w) / dy(j);
            cp -= w / dy(j);
        }
        ey[3 * (j + 1) + 0] = cm;
        ey[3 * (j + 1) + 1] = c0;
        ey[3 * (j + 1) + 2] = cp;
    }
    if (threadIdx.x == 0) {
        ey[0] = 0.0;
        ey[1] = 0.0;
        ey[2] = -1.0 / (yc(0) - yf[0]);                       // bottom wall node
        ey[3 * (ny + 1) + 0] = 1.0 / (yf[ny] - yc(ny - 1));   // top wall node
        ey[3 * (ny + 1) + 1] = 0.0;
        ey[3 * (ny + 1) + 2] = 0.0;
    }
    for (int m = threadIdx.x; m < nx; m += blockDim.x) {
        double s, c;
        sincos(2.0 * M_PI * (double)m / (double)nx, &s, &c);
        twx[m] = cplx<R>{(R)c, (R)(-s)};
        if (m < nxh) sinx[m] = s / g.dx;
    }
    for (int m = threadIdx.x; m < nz; m += blockDim.x) {
        double s, c;
        sincos(2.0 * M_PI * (double)m / (double)nz, &s, &c);
        sinz[m] = s / g.dz;
        twz[m] = cplx<R>{(R)c, (R)(-s)};
    }
    __syncthreads();
    // the x transform's inner twiddles by thread: M = n1 n2, n1 the largest divisor not above sqrt(M)
    const int M = nx / 2, n2 = M / g.n1;
    for (int i = threadIdx.x; i < M; i += blockDim.x) twx[nx + i] = twx[2 * (i % n2) * (i / n2)];
}

template <class R>
tribo_status noalloc_solve(const tribo_grid* g, double eps, const double* rho, double* phi, void* E,
                           cudaStream_t stream, unsigned char* base, const NoallocLayout& L, int num_sms) {
    const int nx = g->nx, ny = g->ny, nz = g->nz, nxh = nx / 2 + 1;
    NoallocGeom geom{};
    geom.nx = nx; geom.ny = ny; geom.nz = nz;
    geom.dx = g->lx / nx; geom.dz = g->lz / nz;
    geom.scale = -0.5 / eps / ((double)nx * (double)nz);
    geom.n1 = 1;
    for (int d = 1; d * d <= nx / 2; ++d)
        if ((nx / 2) % d == 0) geom.n1 = d;
    for (int j = 0; j <= ny; ++j) geom.yf[j] = g->y_faces[j];
    double* T = reinterpret_cast<double*>(base + L.tables);
    cplx<R>* twx = reinterpret_cast<cplx<R>*>(base + L.twx);
    cplx<R>* twz = reinterpret_cast<cplx<R>*>(base + L.twz);
    double* te = reinterpret_cast<double*>(base + L.te);
    cplx<R>* S = reinterpret_cast<cplx<R>*>(base + L.S);
    cplx<R>* F = reinterpret_cast<cplx<R>*>(base + L.F);
    const double* sinx = T + 3 * ny;
    const double* sinz = sinx + nxh;
    const double* ey = sinz + nz;
    const double* scale = ey + 3 * (ny + 2);
    const int ni = (nz / 2 + 1) * nxh;
    (void)launch_pdl(k_noalloc_tables<R>, dim3(1 + (2 * ni + 127) / 128), dim3(128), 0, stream, geom, T, twx, twz, te);
    // the forward x transform reads pairs of densities: a density aligned to its elements only passes
    // through the field spectra's space, which is written later
    const double* src = rho;
    if (reinterpret_cast<uintptr_t>(rho) % sizeof(double2)) {
        const cudaError_t e = cudaMemcpyAsync(F, rho, sizeof(double) * (size_t)nx * ny * nz, cudaMemcpyDeviceToDevice, stream);
        if (e != cudaSuccess) return cuda_fail(e, "tribo_poisson_noalloc: copy of the density");
        src = reinterpret_cast<const double*>(F);
    }
    const PassGrid<R> pg{nx, ny, nz, nxh, num_sms, stream};
    xfwd_launch<R>(pg, const_cast<double*>(src), true, scale, false, S, twx);
    zfwd_launch<R>(pg, S, twz);
    (void)launch_pdl(k_ysolve64<R>, dim3((unsigned)(((int64_t)nz * nxh + 31) / 32)), dim3(128), ysolve64_smem(ny), stream,
                     S, F, (const double*)te, (const double*)(te + (size_t)(ny + 1) * ni), (const double*)T, ey, ny, nz,
                     nxh, 1);
    zinv_launch<R>(pg, S, F, sinz, twz, false);
    xinv_launch<R>(pg, F, (R*)E, phi, sinx, twx);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "tribo_poisson_noalloc: kernel launch");
    return TRIBO_OK;
}

bool noalloc_2a3b(int n) {
    if (n < 1) return false;
    while (n % 2 == 0) n /= 2;
    while (n % 3 == 0) n /= 3;
    return n == 1;
}

// the kernels of one precision on the current device: the shared-memory limits of the transforms of
// every length a grid may have (which loads their code: loaded when first launched, each would take
// device memory then), and the code of the other two
template <class R>
tribo_status noalloc_load(int optin) {
    tribo_status st;
    for (int n = 4; n <= kNoallocMaxN; ++n) {
        if (!noalloc_2a3b(n)) continue;
        if (n % 2 == 0 && (st = xpass_attr<R>(n / 2, optin))) return st;
        if ((st = zpass_attr<R>(n, optin))) return st;
    }
    cudaFuncAttributes at;
    cudaError_t e = cudaFuncGetAttributes(&at, k_noalloc_tables<R>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, k_ysolve64<R>);
    return e == cudaSuccess ? TRIBO_OK : cuda_fail(e, "tribo_poisson_noalloc: kernel attributes");
}

// set-up of the current device, by its first call: the array's device address and every kernel that a
// later call of either precision may launch
tribo_status noalloc_device(int dev, NoallocDevice* out) {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    NoallocDevice& d = g_noalloc_dev[dev];
    if (!d.ready) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "tribo_poisson_noalloc: cudaGetSymbolAddress");
        int optin = 0, sms = 0;
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return cuda_fail(e, "tribo_poisson_noalloc: device attribute");
        tribo_status st;
        if ((st = noalloc_load<float>(optin)) || (st = noalloc_load<double>(optin))) return st;
        d.base = static_cast<unsigned char*>(p);
        d.num_sms = std::max(1, sms);
        d.ready = true;
    }
    *out = d;
    return TRIBO_OK;
}

}  // namespace
}  // namespace tribo

extern "C" tribo_status tribo_poisson_noalloc(const tribo_grid* grid, double eps, int32_t precision,
                                              const double* rho, double* phi, void* E, void* stream) {
    using namespace tribo;
    if (!grid || !grid->y_faces || !rho || !E) {
        set_last_error("tribo_poisson_noalloc: grid, y_faces, rho and E must not be NULL");
        return TRIBO_ERR_ARG;
    }
    if (precision != TRIBO_FP64 && precision != TRIBO_MIXED) {
        set_last_error("tribo_poisson_noalloc: unknown precision");
        return TRIBO_ERR_ARG;
    }
    if (!(eps > 0) || !(grid->lx > 0) || !(grid->lz > 0)) {
        set_last_error("tribo_poisson_noalloc: eps, lx and lz must be positive");
        return TRIBO_ERR_ARG;
    }
    const int nx = grid->nx, ny = grid->ny, nz = grid->nz;
    if (nx < 4 || nz < 4 || nx % 2 || !noalloc_2a3b(nx) || !noalloc_2a3b(nz) || ny < 2) {
        set_last_error("tribo_poisson_noalloc: nx and nz must be 2^a 3^b >= 4 (nx even), ny >= 2");
        return TRIBO_ERR_UNSUPPORTED;
    }
    const size_t rsz = precision == TRIBO_FP64 ? sizeof(double) : sizeof(float);
    const size_t counted = noalloc_capacity(nx, ny, nz, phi ? 4 : 3, rsz);
    const NoallocLayout L = noalloc_layout(nx, ny, nz, rsz);
    if (nx > kNoallocMaxN || ny > kNoallocMaxN || nz > kNoallocMaxN || counted > kNoallocScratchBytes ||
        L.total > kNoallocScratchBytes) {
        char buf[256];
        snprintf(buf, sizeof buf,
                 "tribo_poisson_noalloc: a %dx%dx%d grid counts as %.1f MiB of static scratch; the limit is "
                 "%d MiB and %d cells per direction",
                 nx, ny, nz, counted / 1048576.0, (int)(kNoallocScratchBytes >> 20), kNoallocMaxN);
        set_last_error(buf);
        return TRIBO_ERR_CAPACITY;
    }
    if (grid->y_faces[0] != 0.0) {
        set_last_error("tribo_poisson_noalloc: y_faces[0] must be 0");
        return TRIBO_ERR_ARG;
    }
    for (int j = 0; j < ny; ++j)
        if (!(grid->y_faces[j + 1] > grid->y_faces[j])) {
            set_last_error("tribo_poisson_noalloc: y_faces must increase strictly");
            return TRIBO_ERR_ARG;
        }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "tribo_poisson_noalloc: cudaGetDevice");
    if (dev < 0 || dev >= kNoallocMaxDevices) {
        set_last_error("tribo_poisson_noalloc: device ordinal out of range");
        return TRIBO_ERR_UNSUPPORTED;
    }
    NoallocDevice d;
    const bool f64 = precision == TRIBO_FP64;
    tribo_status st = noalloc_device(dev, &d);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (f64) return noalloc_solve<double>(grid, eps, rho, phi, E, s, d.base, L, d.num_sms);
    return noalloc_solve<float>(grid, eps, rho, phi, E, s, d.base, L, d.num_sms);
}
