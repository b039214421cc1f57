// Instantiates the Phi tile kernels for one working type (PHI_T) and one
// gathered-mode count (PHI_NM1; 0 = runtime count) and exposes a launcher.
// Included by the small phi_<type>_<nm1>.cu units so that the template
// instantiations compile in parallel.
#include "phi_launch.cuh"

#ifndef PHI_T
#error "define PHI_T"
#endif
#ifndef PHI_NM1
#error "define PHI_NM1"
#endif
#ifndef PHI_FN
#error "define PHI_FN"
#endif

namespace cpapr {

namespace {
template <int RPL, int G, int OP, bool PI>
cudaError_t run(const PhiArgs &a, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    constexpr int U = unroll_for<RPL, G>();
    // the log-likelihood's underflow fallback needs more registers than four
    // blocks per SM allow (measured: 7% faster unconstrained)
    if constexpr (phi_occ4<PHI_T, RPL>() && OP != OP_LL) {
        return launch<RPL>(phi_tile_kernel_occ4<PHI_T, PHI_NM1, RPL, G, OP, kThreads, U, PI>, a, s, win);
    } else {
        return launch<RPL>(phi_tile_kernel<PHI_T, PHI_NM1, RPL, G, OP, kThreads, U, PI>, a, s, win);
    }
}
// Phi: FP32 runs the direct tiles (direct.cuh)
template <int RPL, int G>
cudaError_t run_phi(const PhiArgs &a, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    if constexpr (sizeof(PHI_T) == 8)
        return a.pi ? run<RPL, G, OP_PHI, true>(a, s, win) : run<RPL, G, OP_PHI, false>(a, s, win);
    return cudaErrorInvalidValue;
}
// MTTKRP: FP32 stays here for two gathered modes (0.187 ms on the 3-way tensor with
// 1e7 nonzeros, R = 32, against 0.192 as a direct tile; with three 0.99 against 0.89)
template <int RPL, int G>
cudaError_t run_mttkrp(const PhiArgs &a, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    if constexpr (sizeof(PHI_T) == 8 || PHI_NM1 == 2) return run<RPL, G, OP_MTTKRP, false>(a, s, win);
    return cudaErrorInvalidValue;
}
// log-likelihood: FP64 can stream the materialised rows, FP32 always gathers
template <int RPL, int G>
cudaError_t run_ll(const PhiArgs &a, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    if constexpr (sizeof(PHI_T) == 8) {
        if (a.pi) return run<RPL, G, OP_LL, true>(a, s, win);
    }
    return run<RPL, G, OP_LL, false>(a, s, win);
}
}  // namespace

// Returns cudaErrorInvalidValue when (rpl, lanes) has no instantiation.
// Phi reads the materialised Khatri-Rao rows when a.pi is set.
cudaError_t PHI_FN(const PhiArgs &a, int rpl, int lanes, int op, cudaStream_t s, const cudaAccessPolicyWindow *win) {
#define CPAPR_CASE(R_, G_)                                                                          \
    if (rpl == R_ && lanes == G_) {                                                                 \
        if (op == OP_PHI) return run_phi<R_, G_>(a, s, win);                                        \
        if (op == OP_MTTKRP) return run_mttkrp<R_, G_>(a, s, win);                                  \
        return run_ll<R_, G_>(a, s, win);                                                           \
    }
#if PHI_IS_DOUBLE
    CPAPR_CASE(2, 1)
    CPAPR_CASE(4, 1)
    CPAPR_CASE(8, 1)
    CPAPR_CASE(16, 1)
    CPAPR_CASE(8, 2)
    CPAPR_CASE(16, 2)
    CPAPR_CASE(8, 4)
    CPAPR_CASE(16, 4)
    CPAPR_CASE(8, 8)
    CPAPR_CASE(16, 8)
    CPAPR_CASE(8, 16)
#else
    CPAPR_CASE(4, 1)
    CPAPR_CASE(8, 1)
    CPAPR_CASE(16, 1)
    CPAPR_CASE(4, 2)
    CPAPR_CASE(8, 2)
    CPAPR_CASE(4, 4)
    CPAPR_CASE(8, 4)
    CPAPR_CASE(4, 8)
    CPAPR_CASE(8, 8)
    CPAPR_CASE(4, 16)
    CPAPR_CASE(8, 16)
#endif
#undef CPAPR_CASE
    return cudaErrorInvalidValue;
}

}  // namespace cpapr
