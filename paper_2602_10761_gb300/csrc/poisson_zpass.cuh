// Launch of the z transforms of the Poisson solve (Sec. 2.2, Sec. 3.1) for
// every length; instantiated once per precision (poisson_z32.cu,
// poisson_z64.cu).
#pragma once

#include "poisson_passes.cuh"

namespace tribo {
namespace {

template <class R, int NZ>
void zfwd_one(const PassGrid<R>& g, cplx<R>* S, const cplx<R>* twz) {
    constexpr int W = fft::FourStep<NZ, kThreads>::W;
    const int64_t tiles = ((int64_t)g.ny * g.nxh + W - 1) / W;
    if constexpr (sizeof(R) == 4) {
        if (g.tab) {
            static int occ_tab = 0;
            const int gx = std::max(1, wave_blocks(k_zfwd4<R, NZ, true>, zfwd_smem<R, NZ>(), g.num_sms, tiles, &occ_tab) / g.n);
            k_zfwd4<R, NZ, true><<<dim3(gx, g.n), kThreads, zfwd_smem<R, NZ>(), g.stream>>>(nullptr, g.ny, g.nxh,
                                                                                            nullptr, g.tab);
            return;
        }
    }
    static int occ = 0;
    const int nb = wave_blocks(k_zfwd4<R, NZ>, zfwd_smem<R, NZ>(), g.num_sms, tiles, &occ);
    (void)launch_pdl(k_zfwd4<R, NZ>, dim3(nb), dim3(kThreads), zfwd_smem<R, NZ>(), g.stream, S, g.ny, g.nxh, twz,
                     (const FastTab<R>*)nullptr);
}

template <class R, int NZ>
void zinv_one(const PassGrid<R>& g, const cplx<R>* S, cplx<R>* F, const double* sinz, const cplx<R>* twz,
              bool phi_only) {
    constexpr int W = fft::FourStep<NZ, kThreads>::W;
    const int64_t tiles = ((int64_t)g.ny * g.nxh + W - 1) / W + ((int64_t)(g.ny + 2) * g.nxh + W - 1) / W;
    const size_t fstride = (size_t)g.nz * (g.ny + 2) * g.nxh;
    if constexpr (sizeof(R) == 4) {
        if (g.tab) {
            static int occ_tab = 0;
            const int gx = std::max(1, wave_blocks(k_zinv4<R, NZ, true>, zinv_smem<R, NZ>(), g.num_sms, tiles, &occ_tab) / g.n);
            k_zinv4<R, NZ, true><<<dim3(gx, g.n), kThreads, zinv_smem<R, NZ>(), g.stream>>>(
                nullptr, nullptr, g.ny, g.nxh, fstride, nullptr, nullptr, 0, g.tab);
            return;
        }
    }
    static int occ = 0;
    const int nb = wave_blocks(k_zinv4<R, NZ>, zinv_smem<R, NZ>(), g.num_sms, tiles, &occ);
    (void)launch_pdl(k_zinv4<R, NZ>, dim3(nb), dim3(kThreads), zinv_smem<R, NZ>(), g.stream, S, F, g.ny, g.nxh, fstride,
                     sinz, twz, phi_only ? 1 : 0, (const FastTab<R>*)nullptr);
}

template <class R, int NZ>
tribo_status zattr_one(int optin) {
    if (zfwd_smem<R, NZ>() > (size_t)optin || zinv_smem<R, NZ>() > (size_t)optin) {
        set_last_error("grid needs more shared memory per block than the device offers");
        return TRIBO_ERR_UNSUPPORTED;
    }
    TRIBO_CUDA(cudaFuncSetAttribute(k_zfwd4<R, NZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    TRIBO_CUDA(cudaFuncSetAttribute(k_zinv4<R, NZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    if constexpr (sizeof(R) == 4) {
        TRIBO_CUDA(cudaFuncSetAttribute(k_zfwd4<R, NZ, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
        TRIBO_CUDA(cudaFuncSetAttribute(k_zinv4<R, NZ, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    }
    return TRIBO_OK;
}

}  // namespace

template <class R>
tribo_status zpass_attr(int nz, int optin) {
    switch (nz) {
#define CASE(N) case N: return zattr_one<R, N>(optin);
        TRIBO_Z_SIZES(CASE)
#undef CASE
        default: break;
    }
    set_last_error("no compiled transform of this z length");
    return TRIBO_ERR_UNSUPPORTED;
}

template <class R>
void zfwd_launch(const PassGrid<R>& g, cplx<R>* S, const cplx<R>* twz) {
    switch (g.nz) {
#define CASE(N) case N: zfwd_one<R, N>(g, S, twz); break;
        TRIBO_Z_SIZES(CASE)
#undef CASE
        default: break;
    }
}

template <class R>
void zinv_launch(const PassGrid<R>& g, const cplx<R>* S, cplx<R>* F, const double* sinz, const cplx<R>* twz,
                 bool phi_only) {
    switch (g.nz) {
#define CASE(N) case N: zinv_one<R, N>(g, S, F, sinz, twz, phi_only); break;
        TRIBO_Z_SIZES(CASE)
#undef CASE
        default: break;
    }
}

#define TRIBO_ZPASS_INSTANTIATE(R)                                                        \
    template tribo_status zpass_attr<R>(int, int);                                        \
    template void zfwd_launch<R>(const PassGrid<R>&, cplx<R>*, const cplx<R>*);           \
    template void zinv_launch<R>(const PassGrid<R>&, const cplx<R>*, cplx<R>*, const double*, const cplx<R>*, bool);

}  // namespace tribo
