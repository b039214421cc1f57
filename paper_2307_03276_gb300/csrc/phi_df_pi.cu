// FP64 Phi and log-likelihood over materialised float-pair Khatri-Rao rows, the
// kernel that builds the rows, and the one that keeps the factors as pairs.
#define DF_PI 1
#define DF_FN launch_phi_df_pi
#include "phi_df.cuh"

#include <algorithm>

namespace cpapr {

namespace {

// largest entry of a factor as FP64 bits (entries are >= 0: bits order like values)
__global__ void __launch_bounds__(256) factor_max_kernel(const double *__restrict__ A, int64_t n,
                                                         unsigned long long *__restrict__ top) {
    double m = 0.0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        m = fmax(m, A[e]);
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0 && m > 0.0) atomicMax(top, ordered_bits(m));
}

// The pairs of one factor, scaled by 2^(kPairTop - k).  top: the largest entry's bits
// (k is its exponent, held to [-100, 100] so that products' scales stay far
// inside the FP64 range; entries outside the window escape), or null after a
// normalisation (entries <= 1: k = 0).  Bound by its 16 bytes per entry.
__global__ void __launch_bounds__(256) pair_factor_kernel(const double2 *__restrict__ A, float4 *__restrict__ P,
                                                          int64_t nv,
                                                          const unsigned long long *__restrict__ top,
                                                          int32_t *__restrict__ kexp) {
    int k = 0;
    if (top) {
        const unsigned long long b = *top;
        k = b ? max(-100, min(100, (int)(b >> 52) - 1022)) : 0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *kexp = k;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nv; e += (int64_t)gridDim.x * blockDim.x) {
        const double2 x = A[e];
        const float2 p = pair_factor(x.x, kPairTop - k), q = pair_factor(x.y, kPairTop - k);
        P[e] = make_float4(p.x, q.x, p.y, q.y);
    }
}

// Khatri-Rao rows of one mode as pairs, like pi_build_range: one thread per
// 16-byte vector (two elements).  The products are formed as the fused kernel
// forms them (form_rows in df_walk), so the two give the same bits.  No FP64: an
// element outside the pairs' window is marked, its value left to the few that need it.
template <int NM1>
__global__ void __launch_bounds__(256) pi_pair_kernel(const PhiArgs a, float4 *__restrict__ pi) {
    constexpr int MAXK = NM1 > 0 ? NM1 : kMaxNm1;
    const int nm1 = NM1 > 0 ? NM1 : a.nm1;
    const int vpr = a.Rp / 2;  // vectors per row, a power of two
    const int lg = 31 - __clz(vpr);
    const int64_t total = a.nnz << lg;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = e >> lg;
        const int v = (int)(e & (vpr - 1));
        int32_t ii[MAXK];
        PairProduct q0, q1;
#pragma unroll
        for (int k = 0; k < MAXK; ++k) {
            if (k < nm1) {
                ii[k] = __ldg(a.idx[k] + p);
                const float4 x = __ldg(reinterpret_cast<const float4 *>(a.P[k] + (int64_t)ii[k] * a.Rp) + v);
                if (k == 0) {
                    q0.start(make_float2(x.x, x.z));
                    q1.start(make_float2(x.y, x.w));
                } else {
                    q0.mul(make_float2(x.x, x.z));
                    q1.mul(make_float2(x.y, x.w));
                }
            }
        }
        float2 e0 = q0.p, e1 = q1.p;
        // pairs, then zeros (a padded rank's columns), then the rest; with four gathered
        // factors both at once (R = 33: 0.502 against 0.514 ms a mode at 3e6 nonzeros; three
        // factors, R = 16, 2e7: 0.696 against 0.684)
        const bool plain = NM1 == 4 ? q0.plain() && q1.plain()
                                    : (q0.pair_ok() && q1.pair_ok()) || (q0.plain_zero() && q1.plain_zero());
        if (!plain) {
            e0 = q0.value();
            e1 = q1.value();
        }
        __stcs(pi + e, make_float4(e0.x, e1.x, e0.y, e1.y));
    }
}

template <int NM1>
cudaError_t run_pi(const PhiArgs &a, float4 *pi, unsigned grid, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    if (!win) {
        pi_pair_kernel<NM1><<<grid, 256, 0, s>>>(a, pi);
        return cudaGetLastError();
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
    attr[0].val.accessPolicyWindow = *win;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, pi_pair_kernel<NM1>, a, pi);
}

}  // namespace

cudaError_t launch_pi_pairs(const PhiArgs &a, void *pi, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    const unsigned grid =
        (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(a.nnz * (a.Rp / 2), 256), 152 * 16));
    float4 *P = reinterpret_cast<float4 *>(pi);
    switch (a.nm1) {
        case 2: return run_pi<2>(a, P, grid, s, win);
        case 3: return run_pi<3>(a, P, grid, s, win);
        case 4: return run_pi<4>(a, P, grid, s, win);
        default: return run_pi<0>(a, P, grid, s, win);
    }
}

// Factor m's pairs from its FP64 entries; from_data: its exponent is measured
// first (else the factor comes from a normalisation: at most 1).
cpapr_status launch_factor_pairs(cpapr_ctx *ctx, int m, bool from_data) {
    const int64_t n = ctx->dims[m] * ctx->Rp;
    const double *A = reinterpret_cast<const double *>(ctx->A[m]);
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 512), 152 * 8));
    unsigned long long *top = nullptr;
    if (from_data) {
        top = ctx->pair_top + m;
        CPAPR_CUDA(ctx, cudaMemsetAsync(top, 0, 8, ctx->stream));
        factor_max_kernel<<<grid, 256, 0, ctx->stream>>>(A, n, top);
        CPAPR_CUDA(ctx, cudaGetLastError());
    }
    pair_factor_kernel<<<grid, 256, 0, ctx->stream>>>(reinterpret_cast<const double2 *>(A),
                                                      reinterpret_cast<float4 *>(ctx->P[m]), n / 2, top, ctx->kexp + m);
    CPAPR_CUDA(ctx, cudaGetLastError());
    count_launch(ctx, from_data ? 2 : 1);
    return CPAPR_OK;
}

}  // namespace cpapr
