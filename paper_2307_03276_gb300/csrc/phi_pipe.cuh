// Instantiates the FP64 Phi kernel with FP64 rows and its divisor on the FP32 pipe
// (phi_tile_kernel_df) for one gathered-mode count: PIPE_NM1 (0 = runtime count).
// Units of its own: with these kernels beside MTTKRP's and the log-likelihood's the
// modules grew past the size from which nvcc compresses them, and the first MTTKRP of a
// process took 9 ms to load its kernel instead of 1.
#define PHI_T double
#include "phi_launch.cuh"

namespace cpapr {

// Returns cudaErrorInvalidValue when (rpl, lanes) has no instantiation.
cudaError_t PIPE_FN(const PhiArgs &a, int rpl, int lanes, cudaStream_t s, const cudaAccessPolicyWindow *win) {
#define CPAPR_CASE(R_, G_)                                                                                          \
    if (rpl == R_ && lanes == G_)                                                                                   \
        return a.pi ? launch<R_>(phi_tile_kernel_df<double, PIPE_NM1, R_, G_, OP_PHI, kThreads, unroll_for<R_, G_>(), true>, \
                                 a, s, win)                                                                         \
                    : launch<R_>(phi_tile_kernel_df<double, PIPE_NM1, R_, G_, OP_PHI, kThreads, unroll_for<R_, G_>(), false>, \
                                 a, s, win);
    CPAPR_CASE(2, 1)
    CPAPR_CASE(4, 1)
    CPAPR_CASE(8, 1)
    CPAPR_CASE(8, 2)
    CPAPR_CASE(8, 4)
    CPAPR_CASE(8, 8)
    CPAPR_CASE(8, 16)
#undef CPAPR_CASE
    return cudaErrorInvalidValue;
}

}  // namespace cpapr
