// Instantiates the FP64 tile kernels over float-pair Khatri-Rao rows
// (df_walk.cuh) for one gathered-mode count: DF_NM1 (0 = runtime count) with
// the rows formed in place, or DF_PI with the materialised rows.  Included by
// the phi_df_*.cu units so that the instantiations compile in parallel.
#include "df_walk.cuh"

namespace cpapr {

namespace {
// win: persisting-L2 window for the launch, or null for a plain launch
template <int RPL, int G, typename Kern>
cudaError_t launch_df(Kern k, const PhiArgs &a, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    constexpr int NG = kDfThreads / G;
    const size_t smem = (size_t)2 * NG * df_slot_stride(RPL * G) * sizeof(double) + (size_t)(2 * NG + 2) * 4;
    static_assert(2 * NG * (df_slot_stride(RPL * G) * 8 + 4) + 8 <= 48 * 1024, "within the default shared memory");
    if (a.ntiles <= 0) return cudaGetLastError();
    if (!win) {
        k<<<a.ntiles, kDfThreads, smem, s>>>(a);
        return cudaGetLastError();
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
    attr[0].val.accessPolicyWindow = *win;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.ntiles);
    cfg.blockDim = dim3(kDfThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, a);
}
}  // namespace

// Returns cudaErrorInvalidValue when the padded rank has no instantiation.  The
// kernel keeps 4 ranks per lane whatever lanes the other kernels of the mode use.
#ifdef DF_PI
cudaError_t DF_FN(const PhiArgs &a, int op, cudaStream_t s, const cudaAccessPolicyWindow *win) {
#define CPAPR_CASE(R_, G_, U_)                                                                              \
    case R_ * G_:                                                                                           \
        return op == OP_PHI ? launch_df<R_, G_>(phi_pair_kernel<0, R_, G_, OP_PHI, U_, true>, a, s, win)    \
                            : launch_df<R_, G_>(phi_pair_kernel<0, R_, G_, OP_LL, U_, true>, a, s, win);
#else
cudaError_t DF_FN(const PhiArgs &a, cudaStream_t s, const cudaAccessPolicyWindow *win) {
#define CPAPR_CASE(R_, G_, U_) \
    case R_ * G_: return launch_df<R_, G_>(phi_pair_kernel<DF_NM1, R_, G_, OP_PHI, U_, false>, a, s, win);
#endif
    switch (a.Rp) {
        CPAPR_CASE(2, 1, 2)
        CPAPR_CASE(4, 1, 2)
        CPAPR_CASE(4, 2, 2)
        CPAPR_CASE(4, 4, 4)
        CPAPR_CASE(4, 8, 4)
        CPAPR_CASE(4, 16, 4)
        CPAPR_CASE(4, 32, 4)
    }
#undef CPAPR_CASE
    return cudaErrorInvalidValue;
}

}  // namespace cpapr
