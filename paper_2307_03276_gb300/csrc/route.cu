// When a large FP64 Phi leaves the float pairs.
//
// Along a solve, factor entries that a component does not need decay towards 0,
// and the Khatri-Rao elements with them.  Those below the pairs' window (df_pair.cuh)
// are left out of the FP32 sums, and a column of a row all of whose elements are
// small is summed again in FP64, nonzero by nonzero (pair_resum).  That is rare for
// some 20 outer iterations and then grows without end: an outer iteration of the
// 3-way tensor with 1e7 nonzeros (R = 32) takes 21.1 ms at first, 25.9 at the 16th, 33 at
// the 22nd and 75 at the 36th (rows formed in place: 25, 28, 34, 66), where the
// kernel that keeps the rows in FP64 and takes only the divisor on the FP32 pipe
// (phi_tile_kernel_df) takes 33.2 (44) throughout.  So the share of nonzeros that a
// launch would sum again is estimated from the current factors, on a sample of the
// runs that the kernel's groups take, once per outer iteration (and for a single
// Phi once per model), and a mode beyond kResumLimit takes that kernel.
//
// The share is a function of the tensor and the factors alone, counted in
// integers, and the limit is the same for both forms of the rows: a solve that is
// resumed from a checkpoint takes the same kernels, and gives the same bits, as one
// that did not stop, and the materialised form the bits of the fused one.
#include <algorithm>

#include "df_pair.cuh"
#include "internal.cuh"

namespace cpapr {

namespace {

constexpr int kProbeRuns = 1024;  // sampled runs per mode: 4% of a Phi launch at 3e6 nonzeros, 1% at 1e7
constexpr int kProbeWarps = 4;

struct ProbeMode {
    const int32_t *idx[kMaxModes - 1];
    const uint32_t *rstart;
    int32_t mode, vlen, nsamp;
    int64_t nruns;
};

struct RouteProbe {
    ProbeMode m[kMaxModes];  // the sampled modes, one per grid row
    const double *A[kMaxModes];
    const int32_t *kexp;
    uint32_t measured;  // factors whose exponent is in kexp (the others: 0)
    int64_t nnz;
    int32_t N, Rp;
    int32_t *count;  // [N][2] nonzeros in row parts that would be summed again; nonzeros
};

// One warp per sampled run: positions [p0, p0 + vlen) of the mode's order, lane c
// holding columns c, c + 32, ...; a part of a row counts if some column has elements
// below the window and none that makes up for what they leave out (pair kernel's
// flush: 2^55 times the window's edge, times the quotients, taken as alike).  An
// element's size is the sum of its factors' leading bits read as logarithms (within
// a tenth of a bit each).  Bound by the latency of its gathers, so those of 16
// positions are in flight.  With its synchronisation it adds 35 us to a first Phi of
// 1.3 ms (3-way 1e7, R = 32) and 65 to one of 1.1 (5-way 3e6, R = 33); with FP64 products
// and comparisons, which wait for the FP64 pipe, 160.
__global__ void __launch_bounds__(32 * kProbeWarps) route_probe_kernel(const __grid_constant__ RouteProbe a) {
    const ProbeMode &M = a.m[blockIdx.y];
    const int w = blockIdx.x * kProbeWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (w >= M.nsamp) return;
    constexpr unsigned full = 0xffffffffu;
    const int64_t p0 = M.nruns * w / M.nsamp * M.vlen;
    const int len = (int)min((int64_t)M.vlen, a.nnz - p0);
    const int nm1 = a.N - 1;
    int K = kPairTop;
    for (int m = 0; m < a.N; ++m)
        if (m != M.mode && ((a.measured >> m) & 1u)) K -= __ldg(a.kexp + m);
    constexpr int kFrac = 12;  // fraction bits of a logarithm
    const int low = (kPairLow - K) << kFrac, enough = low + (55 << kFrac);
    constexpr int U = 16;
    uint32_t some_low = 0, some_large = 0;  // a bit per column of the lane
    int part = 0, again = 0;
    for (int q = 0; q < len; q += U) {
        const int64_t mine = p0 + min(q + (lane & (U - 1)), len - 1);  // the position whose coordinates this lane loads
        uint32_t lo[U], hi[U];
#pragma unroll
        for (int u = 0; u < U; ++u) lo[u] = hi[u] = 0;
        for (int j = 0; j * 32 < a.Rp; ++j) {
            const int c = min(j * 32 + lane, a.Rp - 1);
            int d[U];            // log2 of the element
            uint32_t zero = 0u;  // a bit per position
#pragma unroll
            for (int u = 0; u < U; ++u) d[u] = 0;
#pragma unroll 2
            for (int k = 0; k < nm1; ++k) {
                const double *A = a.A[k + (k >= M.mode ? 1 : 0)] + c;
                const int i = __ldg(M.idx[k] + mine);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const double v = __ldg(A + (int64_t)__shfl_sync(full, i, u) * a.Rp);
                    const int h = __double2hiint(v);
                    d[u] += (h >> (20 - kFrac)) - (1023 << kFrac);
                    zero |= (h | __double2loint(v)) == 0 ? 1u << u : 0u;
                }
            }
            const uint32_t bit = j * 32 + lane < a.Rp ? 1u << j : 0u;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                lo[u] |= !((zero >> u) & 1u) && d[u] < low ? bit : 0u;
                hi[u] |= !((zero >> u) & 1u) && d[u] >= enough ? bit : 0u;
            }
        }
        const uint32_t starts =
            __ballot_sync(full, (__ldg(M.rstart + (mine >> 5)) >> (mine & 31)) & 1u);  // (of positions 0 .. U - 1)
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (q + u < len) {
                if (q + u > 0 && ((starts >> u) & 1u)) {
                    if (__any_sync(full, (some_low & ~some_large) != 0u)) again += part;
                    some_low = some_large = 0;
                    part = 0;
                }
                some_low |= lo[u];
                some_large |= hi[u];
                ++part;
            }
        }
    }
    if (__any_sync(full, (some_low & ~some_large) != 0u)) again += part;
    if (lane == 0) {
        if (again) atomicAdd(a.count + 2 * M.mode, again);
        atomicAdd(a.count + 2 * M.mode + 1, len);
    }
}

// Share of nonzeros summed again up to which the pairs are not slower, as measured
// over 36 outer iterations (ms an outer iteration with all modes on pairs against
// all on FP64 rows, and the share of the mode that has most).  3-way 1e7, R = 32,
// materialised: 31.4 against 33.2 at 0.0009, 33.1 at 0.0027, 41 at 0.012 (so it leaves them
// by the 23rd).  3-way 3e6, R = 64: 15.4 against 19.2 at 0.0022, 20.5 at 0.0061.  3-way 1.3e6,
// R = 16: 4.4 against 4.9 at 0.006.  4-way 1.5e6, R = 100: 56 against 25.4 at 0.07.  6-way 2e6,
// R = 40: 29.9 against 32.4 at 0.01.  In place they hold longer: 3-way 1e7 41 against 44 at
// 0.012.
constexpr double kResumLimit = 0.0015;

}  // namespace

cpapr_status queue_routes(cpapr_ctx *ctx, uint32_t modes) {
    RouteProbe a{};
    int rows = 0, most = 0;
    for (int n = 0; n < ctx->N; ++n) {
        if (!((modes >> n) & 1u) || !route_varies(ctx, n)) continue;
        const ModeLayout &L = ctx->mode[n];
        ProbeMode &M = a.m[rows++];
        for (int k = 0; k < ctx->N - 1; ++k) M.idx[k] = L.idx[k];
        M.rstart = L.rstart;
        M.mode = n;
        const int groups = 128 / std::max(1, ctx->Rp / 4);
        M.vlen = std::max(1, (L.tile_nnz << L.sh_df) / groups);
        M.nruns = ceil_div(ctx->nnz, M.vlen);
        M.nsamp = (int)std::min<int64_t>(M.nruns, kProbeRuns);
        most = std::max(most, M.nsamp);
    }
    if (rows == 0) return CPAPR_OK;
    for (int m = 0; m < ctx->N; ++m) {
        // a factor whose exponent is still to be measured; a normalised one has 0
        const bool read = rows > 1 || a.m[0].mode != m;
        if (read && ctx->pair_state[m] == kPairStale) {
            CPAPR_TRY(launch_factor_pairs(ctx, m, true));
            ctx->pair_state[m] = kPairCurrent;
        }
        if (ctx->pair_state[m] == kPairCurrent) a.measured |= 1u << m;
        a.A[m] = (const double *)ctx->A[m];
    }
    a.kexp = ctx->kexp;
    a.nnz = ctx->nnz;
    a.N = ctx->N;
    a.Rp = ctx->Rp;
    a.count = ctx->resum;
    CPAPR_CUDA(ctx, cudaMemsetAsync(ctx->resum, 0, sizeof(ctx->host->resum), ctx->stream));
    route_probe_kernel<<<dim3((unsigned)ceil_div(most, kProbeWarps), rows), 32 * kProbeWarps, 0, ctx->stream>>>(a);
    CPAPR_CUDA(ctx, cudaGetLastError());
    count_launch(ctx);
    CPAPR_CUDA(ctx, cudaMemcpyAsync(ctx->host->resum, ctx->resum, sizeof(ctx->host->resum), cudaMemcpyDeviceToHost,
                                    ctx->stream));
    return CPAPR_OK;
}

void take_routes(cpapr_ctx *ctx, uint32_t modes) {
    for (int n = 0; n < ctx->N; ++n) {
        if (!((modes >> n) & 1u)) continue;
        if (route_varies(ctx, n))
            ctx->mode[n].late = ctx->host->resum[n][0] > kResumLimit * ctx->host->resum[n][1];
        ctx->routes_known |= 1u << n;
    }
}

cpapr_status ensure_routes(cpapr_ctx *ctx, uint32_t modes) {
    uint32_t todo = 0;
    for (int n = 0; n < ctx->N; ++n)
        if (((modes >> n) & 1u) && !((ctx->routes_known >> n) & 1u) && route_varies(ctx, n)) todo |= 1u << n;
    if (!todo) return CPAPR_OK;
    CPAPR_TRY(queue_routes(ctx, todo));
    CPAPR_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    take_routes(ctx, todo);
    return CPAPR_OK;
}

}  // namespace cpapr
