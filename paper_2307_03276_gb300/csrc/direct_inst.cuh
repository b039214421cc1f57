// Instantiates the direct FP32 tile kernels (direct.cuh) for one gathered-mode
// count: DIRECT_NM1 (0 = runtime count), or DIRECT_PI with the materialised rows.  Included by the direct_*.cu units so that
// the instantiations compile in parallel.
#include "direct.cuh"

namespace cpapr {

namespace {
template <int NM1, int G, int OP, bool PI>
__global__ void __launch_bounds__(kDirectThreads, 8) direct_kernel(const __grid_constant__ PhiArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[kDirectThreads / 32];
    if (a.inner && a.inner->done) return;
    direct_tile<NM1, G, OP, PI>(a, blockIdx.x, smem_raw, red);
}

// win: persisting-L2 window for the launch, or null for a plain launch
template <int NM1, int RP, int OP, bool PI>
cudaError_t launch(const PhiArgs &a, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    auto k = direct_kernel<NM1, RP / 4, OP, PI>;
    constexpr size_t smem = direct_smem();
    static_assert(smem <= 48 * 1024, "within the default shared memory");
    if (a.ntiles <= 0) return cudaGetLastError();
    if (!win) {
        k<<<a.ntiles, kDirectThreads, smem, s>>>(a);
        return cudaGetLastError();
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
    attr[0].val.accessPolicyWindow = *win;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.ntiles);
    cfg.blockDim = dim3(kDirectThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, a);
}

#ifndef DIRECT_PI
// with two gathered modes MTTKRP is the staged kernel's (phi_inst.cuh)
template <int RP>
cudaError_t run_mttkrp(const PhiArgs &a, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    if constexpr (DIRECT_NM1 != 2) return launch<DIRECT_NM1, RP, OP_MTTKRP, false>(a, s, win);
    return cudaErrorInvalidValue;
}
#endif
}  // namespace

// Returns cudaErrorInvalidValue when the padded rank has no instantiation.
cudaError_t DIRECT_FN(const PhiArgs &a, int op, cudaStream_t s, const cudaAccessPolicyWindow *win) {
#ifdef DIRECT_PI
#define CPAPR_CASE(RP_) \
    case RP_: return op == OP_PHI ? launch<0, RP_, OP_PHI, true>(a, s, win) : cudaErrorInvalidValue;
#else
#define CPAPR_CASE(RP_)                                                                      \
    case RP_:                                                                                \
        return op == OP_PHI ? launch<DIRECT_NM1, RP_, OP_PHI, false>(a, s, win) : run_mttkrp<RP_>(a, s, win);
#endif
    switch (a.Rp) {
        CPAPR_CASE(4)
        CPAPR_CASE(8)
        CPAPR_CASE(16)
        CPAPR_CASE(32)
        CPAPR_CASE(64)
        CPAPR_CASE(128)
    }
#undef CPAPR_CASE
    return cudaErrorInvalidValue;
}

}  // namespace cpapr
