// Launch of the x transforms of the Poisson solve (Sec. 2.2, Sec. 3.1) for
// every half length; instantiated once per precision (poisson_x32.cu,
// poisson_x64.cu).
#pragma once

#include "poisson_passes.cuh"

namespace tribo {
namespace {

template <class R, int M, class QT>
void xfwd_one(const PassGrid<R>& g, QT* src, const double* scale, bool zero, cplx<R>* S, const cplx<R>* twx) {
    constexpr int LPB = fft::FourStep<M, kThreads>::W;
    const int nlines = g.ny * g.nz;
    const unsigned nb = (unsigned)((nlines + LPB - 1) / LPB);
    if constexpr (sizeof(R) == 4 && sizeof(QT) == 8) {
        if (g.tab) {
            k_xfwd4<R, M, QT, true><<<dim3(nb, g.n), kThreads, xfwd_smem<R, M>(), g.stream>>>(
                nullptr, nullptr, 1, nullptr, g.ny, nlines, nullptr, g.tab);
            return;
        }
    }
    (void)launch_pdl(k_xfwd4<R, M, QT>, dim3(nb), dim3(kThreads), xfwd_smem<R, M>(), g.stream, src, scale,
                     zero ? 1 : 0, S, g.ny, nlines, twx, (const FastTab<R>*)nullptr);
}

template <class R, int M>
void xinv_one(const PassGrid<R>& g, const cplx<R>* F, R* E, double* phi, const double* sinx, const cplx<R>* twx) {
    constexpr int LPB = fft::FourStep<M, kThreads>::W;
    const int nlines = g.nz * (g.ny + 2);
    const size_t fstride = (size_t)g.nz * (g.ny + 2) * g.nxh, nodes = (size_t)nlines * g.nx;
    const int64_t tiles = (nlines + LPB - 1) / LPB;
    if constexpr (sizeof(R) == 4) {
        if (g.tab) {
            static int occ_tab = 0;
            const int gx = std::max(1, wave_blocks(k_xinv4<R, M, true>, xinv_smem<R, M>(), g.num_sms, tiles, &occ_tab) / g.n);
            k_xinv4<R, M, true><<<dim3(gx, g.n), kThreads, xinv_smem<R, M>(), g.stream>>>(
                nullptr, nullptr, nullptr, g.ny, g.nz, fstride, nullptr, nullptr, 0, 1, nodes, g.tab);
            return;
        }
    }
    static int occ = 0;
    const int nb = wave_blocks(k_xinv4<R, M>, xinv_smem<R, M>(), g.num_sms, tiles, &occ);
    (void)launch_pdl(k_xinv4<R, M>, dim3(nb), dim3(kThreads), xinv_smem<R, M>(), g.stream, F, E, phi, g.ny, g.nz, fstride,
                     sinx, twx, phi != nullptr ? 1 : 0, E != nullptr ? 1 : 0, nodes, (const FastTab<R>*)nullptr);
}

template <class R, int M>
tribo_status xattr_one(int optin) {
    if (xfwd_smem<R, M>() > (size_t)optin || xinv_smem<R, M>() > (size_t)optin) {
        set_last_error("grid needs more shared memory per block than the device offers");
        return TRIBO_ERR_UNSUPPORTED;
    }
    TRIBO_CUDA(cudaFuncSetAttribute(k_xfwd4<R, M, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    TRIBO_CUDA(cudaFuncSetAttribute(k_xfwd4<R, M, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    TRIBO_CUDA(cudaFuncSetAttribute(k_xinv4<R, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    if constexpr (sizeof(R) == 4) {
        TRIBO_CUDA(cudaFuncSetAttribute(k_xfwd4<R, M, double, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
        TRIBO_CUDA(cudaFuncSetAttribute(k_xinv4<R, M, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    }
    return TRIBO_OK;
}

}  // namespace

template <class R>
tribo_status xpass_attr(int m, int optin) {
    switch (m) {
#define CASE(M) case M: return xattr_one<R, M>(optin);
        TRIBO_X_SIZES(CASE)
#undef CASE
        default: break;
    }
    set_last_error("no compiled transform of this x length");
    return TRIBO_ERR_UNSUPPORTED;
}

template <class R>
void xfwd_launch(const PassGrid<R>& g, void* src, bool src_f64, const double* scale, bool zero, cplx<R>* S,
                 const cplx<R>* twx) {
    switch (g.nx / 2) {
#define CASE(M)                                                                        \
    case M:                                                                            \
        if (src_f64) xfwd_one<R, M, double>(g, (double*)src, scale, zero, S, twx);     \
        else xfwd_one<R, M, R>(g, (R*)src, scale, zero, S, twx);                       \
        break;
        TRIBO_X_SIZES(CASE)
#undef CASE
        default: break;
    }
}

template <class R>
void xinv_launch(const PassGrid<R>& g, const cplx<R>* F, R* E, double* phi, const double* sinx, const cplx<R>* twx) {
    switch (g.nx / 2) {
#define CASE(M) case M: xinv_one<R, M>(g, F, E, phi, sinx, twx); break;
        TRIBO_X_SIZES(CASE)
#undef CASE
        default: break;
    }
}

#define TRIBO_XPASS_INSTANTIATE(R)                                                                                 \
    template tribo_status xpass_attr<R>(int, int);                                                                 \
    template void xfwd_launch<R>(const PassGrid<R>&, void*, bool, const double*, bool, cplx<R>*, const cplx<R>*);  \
    template void xinv_launch<R>(const PassGrid<R>&, const cplx<R>*, R*, double*, const double*, const cplx<R>*);

}  // namespace tribo
