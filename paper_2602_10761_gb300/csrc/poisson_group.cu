// Channels with the same grid, solved together (a batch's channels): each
// split pass of the Poisson solve (Sec. 2.2; the passes of poisson_passes.cuh)
// is ONE launch over all of them, blockIdx.y selecting the channel, whose
// arrays the pass reads from a device table.  The result per channel is that
// of the channel's own split-pass solve.
#include <algorithm>
#include <new>
#include <vector>

#include "poisson_passes.cuh"

namespace tribo {
namespace {

struct Group {
    int n = 0;
    int nx = 0, ny = 0, nz = 0, nxh = 0;
    int num_sms = 152, smem_optin = 48 * 1024;
    FastTab<float>* d_tab = nullptr;
};

tribo_status group_attr(const Group& g) {
    tribo_status st;
    if ((st = xpass_attr<float>(g.nx / 2, g.smem_optin)) || (st = zpass_attr<float>(g.nz, g.smem_optin))) return st;
    return TRIBO_OK;
}

}  // namespace

bool poisson_group_ok(const tribo_ctx* c) { return c->prec == TRIBO_MIXED; }

tribo_status poisson_group_create(tribo_ctx* const* chans, int n, void** out) {
    *out = nullptr;
    if (n < 1) return TRIBO_ERR_ARG;
    const tribo_ctx* c0 = chans[0];
    std::vector<FastTab<float>> t(n);
    for (int i = 0; i < n; ++i) {
        tribo_ctx* c = chans[i];
        if (!poisson_group_ok(c) || c->nx != c0->nx || c->ny != c0->ny || c->nz != c0->nz) {
            set_last_error("a Poisson group needs mixed-precision channels of one grid");
            return TRIBO_ERR_ARG;
        }
        const int ni = (c->nz / 2 + 1) * c->nxh;
        FastTab<float>& f = t[i];
        f.src = c->Q;
        f.scale = c->d_scale_q;
        f.S = (cplx<float>*)c->S;
        f.F = (cplx<float>*)c->F;
        f.E = (float*)c->E_lat;
        f.twx = (const cplx<float>*)c->d_twx;
        f.twz = (const cplx<float>*)c->d_twz;
        f.sinx = c->d_sinx;
        f.sinz = c->d_sinz;
        f.te = (const float2*)c->d_ytab;
        f.ti = f.te + (size_t)(c->ny + 1) * ni;
        f.cpl = (const float2*)c->d_ycpl;
        f.yec = (const float4*)c->d_yec;
        f.yck = (float4*)c->d_yck;
    }
    Group* g = new (std::nothrow) Group();
    if (!g) { set_last_error("host allocation failed"); return TRIBO_ERR_OOM; }
    g->n = n;
    g->nx = c0->nx; g->ny = c0->ny; g->nz = c0->nz; g->nxh = c0->nxh;
    g->num_sms = c0->num_sms;
    g->smem_optin = c0->smem_optin;
    tribo_status st = group_attr(*g);
    if (st) {
        delete g;
        if (st == TRIBO_ERR_UNSUPPORTED) set_last_error("a Poisson group's transforms need more shared memory than the device has");
        return st;
    }
    cudaError_t e = cudaMalloc((void**)&g->d_tab, sizeof(FastTab<float>) * n);
    if (e == cudaSuccess) e = cudaMemcpy(g->d_tab, t.data(), sizeof(FastTab<float>) * n, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(g->d_tab);
        delete g;
        return cuda_fail(e, "Poisson group tables");
    }
    *out = g;
    return TRIBO_OK;
}

tribo_status poisson_group_solve(void* grp, cudaStream_t stream, int64_t* launches) {
    const Group* g = static_cast<const Group*>(grp);
    const PassGrid<float> pg{g->nx, g->ny, g->nz, g->nxh, g->num_sms, stream, g->d_tab, g->n};
    xfwd_launch<float>(pg, nullptr, true, nullptr, true, nullptr, nullptr);
    zfwd_launch<float>(pg, nullptr, nullptr);
    ysolve_twist_launch<true, true>((int64_t)g->nz * g->nxh, g->n, g->num_sms, g->ny, stream, nullptr, nullptr, nullptr,
                                    nullptr, nullptr, nullptr, nullptr, g->nz, g->nxh, g->d_tab);
    zinv_launch<float>(pg, nullptr, nullptr, nullptr, nullptr, false);
    xinv_launch<float>(pg, nullptr, nullptr, nullptr, nullptr, nullptr);
    TRIBO_CUDA(cudaGetLastError());
    if (launches) *launches += 5;
    return TRIBO_OK;
}

void poisson_group_free(void* grp) {
    Group* g = static_cast<Group*>(grp);
    if (!g) return;
    cudaFree(g->d_tab);
    delete g;
}

}  // namespace tribo
