// Launch of a staged tile kernel, for the units that instantiate them
// (phi_inst.cuh, phi_pipe.cuh) for one working type (PHI_T).
#pragma once

#include "phi_kernels.cuh"

namespace cpapr {

namespace {
constexpr int kThreads = sizeof(PHI_T) == 8 ? 128 : 256;
// nonzeros per batch (U <= G when G > 1: after the reduce-scatter every lane
// finishes one of them, so a nonzero costs G / U divisions; one lane per
// nonzero takes two at a time for memory-level parallelism).  FP64 at 16
// ranks per lane has no registers to spare for a second batch entry; FP64 at
// 8 or fewer takes two: with four its kernel with the dot on the FP32 pipe
// needed 178 registers and ran 37% slower on the 3-way tensor (1.63 vs 1.19
// ms on GB300), and both kernels share the batch size.
template <int RPL, int G>
constexpr int unroll_for() {
    if (sizeof(PHI_T) == 8) return RPL >= 16 ? (G >= 2 ? 2 : 1) : 2;
    return G >= 4 ? 4 : 2;
}

// win: persisting-L2 window for the launch, or null for a plain launch
template <int RPL, typename K>
cudaError_t launch(K k, const PhiArgs &a, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    const size_t smem = phi_smem_bytes(a.T, a.pi ? 0 : a.nm1, (int)sizeof(PHI_T), kThreads, RPL);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    if (a.ntiles <= 0) return cudaGetLastError();
    if (!win) {
        k<<<a.ntiles, kThreads, smem, s>>>(a);
        return cudaGetLastError();
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
    attr[0].val.accessPolicyWindow = *win;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.ntiles);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, a);
}

}  // namespace

}  // namespace cpapr
