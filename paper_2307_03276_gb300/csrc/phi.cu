// Launchers for the Phi family (Phi^(n), MTTKRP, log-likelihood sum).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "phi_kernels.cuh"

namespace cpapr {

cudaError_t launch_phi_f64_n0(const PhiArgs &, int, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_f64_n2(const PhiArgs &, int, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_f64_n3(const PhiArgs &, int, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_f64_n4(const PhiArgs &, int, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_f32_n0(const PhiArgs &, int, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_f32_n2(const PhiArgs &, int, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_f32_n3(const PhiArgs &, int, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_f32_n4(const PhiArgs &, int, int, int, cudaStream_t, const cudaAccessPolicyWindow *);

cudaError_t launch_phi_df_n0(const PhiArgs &, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_df_n2(const PhiArgs &, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_df_n3(const PhiArgs &, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_df_n4(const PhiArgs &, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_df_pi(const PhiArgs &, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_pipe_n0(const PhiArgs &, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_pipe_n2(const PhiArgs &, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_pipe_n3(const PhiArgs &, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_phi_pipe_n4(const PhiArgs &, int, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_direct_f32_n0(const PhiArgs &, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_direct_f32_n2(const PhiArgs &, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_direct_f32_n3(const PhiArgs &, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_direct_f32_n4(const PhiArgs &, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_direct_f32_pi(const PhiArgs &, int, cudaStream_t, const cudaAccessPolicyWindow *);
cudaError_t launch_pi_pairs(const PhiArgs &, void *, cudaStream_t, const cudaAccessPolicyWindow *);

bool phi_config_supported(int esize, int nm1, int rp, int lanes) {
    (void)nm1;
    if (lanes < 1 || rp % lanes) return false;
    const int rpl = rp / lanes;
    if (esize == 8) {
        static const int ok[][2] = {{2, 1}, {4, 1},  {8, 1}, {16, 1}, {8, 2},  {16, 2},
                                    {8, 4}, {16, 4}, {8, 8}, {16, 8}, {8, 16}};
        for (auto &p : ok)
            if (p[0] == rpl && p[1] == lanes) return true;
    } else {
        static const int ok[][2] = {{4, 1}, {8, 1}, {16, 1}, {4, 2}, {8, 2}, {4, 4},
                                    {8, 4}, {4, 8}, {8, 8}, {4, 16}, {8, 16}};
        for (auto &p : ok)
            if (p[0] == rpl && p[1] == lanes) return true;
    }
    return false;
}

// Shared memory of a tile kernel launch (staged streams + partial-row slots);
// a tile size is usable when it stays within kMaxPhiSmem.
size_t phi_smem_for(int esize, int nm1, int tile, int rp, int lanes) {
    return phi_smem_bytes(tile, nm1, esize, esize == 8 ? 128 : 256, rp / lanes);
}

static cudaError_t dispatch(const cpapr_ctx *ctx, const PhiArgs &a, int rpl, int lanes, int op) {
    const int nm1 = ctx->N - 1;
    // Phi over materialised rows gathers no factor rows: no window
    const cudaAccessPolicyWindow *win = (op == OP_PHI && a.pi) ? nullptr : l2_window(ctx);
    if (a.route == kRoutePairs && a.pi && op != OP_MTTKRP) return launch_phi_df_pi(a, op, ctx->stream, win);
    if (a.route == kRoutePairs && op == OP_PHI) {
        switch (nm1) {
            case 2: return launch_phi_df_n2(a, ctx->stream, win);
            case 3: return launch_phi_df_n3(a, ctx->stream, win);
            case 4: return launch_phi_df_n4(a, ctx->stream, win);
            default: return launch_phi_df_n0(a, ctx->stream, win);
        }
    }
    if (a.route == kRoutePipe && op == OP_PHI) {
        switch (nm1) {
            case 2: return launch_phi_pipe_n2(a, rpl, lanes, ctx->stream, win);
            case 3: return launch_phi_pipe_n3(a, rpl, lanes, ctx->stream, win);
            case 4: return launch_phi_pipe_n4(a, rpl, lanes, ctx->stream, win);
            default: return launch_phi_pipe_n0(a, rpl, lanes, ctx->stream, win);
        }
    }
    if (ctx->esize == 4 && op != OP_LL && !(op == OP_MTTKRP && nm1 == 2)) {
        if (a.pi) return launch_direct_f32_pi(a, op, ctx->stream, win);
        switch (nm1) {
            case 2: return launch_direct_f32_n2(a, op, ctx->stream, win);
            case 3: return launch_direct_f32_n3(a, op, ctx->stream, win);
            case 4: return launch_direct_f32_n4(a, op, ctx->stream, win);
            default: return launch_direct_f32_n0(a, op, ctx->stream, win);
        }
    }
    if (ctx->esize == 8) {
        switch (nm1) {
            case 2: return launch_phi_f64_n2(a, rpl, lanes, op, ctx->stream, win);
            case 3: return launch_phi_f64_n3(a, rpl, lanes, op, ctx->stream, win);
            case 4: return launch_phi_f64_n4(a, rpl, lanes, op, ctx->stream, win);
            default: return launch_phi_f64_n0(a, rpl, lanes, op, ctx->stream, win);
        }
    }
    switch (nm1) {
        case 2: return launch_phi_f32_n2(a, rpl, lanes, op, ctx->stream, win);
        case 3: return launch_phi_f32_n3(a, rpl, lanes, op, ctx->stream, win);
        case 4: return launch_phi_f32_n4(a, rpl, lanes, op, ctx->stream, win);
        default: return launch_phi_f32_n0(a, rpl, lanes, op, ctx->stream, win);
    }
}

// Host-side failure injection for the bounded staging wait: while the
// environment variable CPAPR_FAULT_STAGE_WAIT is "1", every tile's barrier
// expects 16 bytes more than its copies bring, so the wait runs out after
// its time limit, the tile is skipped and the call reports CPAPR_E_TIMEOUT.
// Nothing faults: the copies themselves are the normal ones.
uint32_t injected_stage_shortfall() {
    const char *s = std::getenv("CPAPR_FAULT_STAGE_WAIT");
    return (s && s[0] == '1' && s[1] == 0) ? 16u : 0u;
}

// Off the FP64 pipe an FP64 Phi is accurate relative to max(s, eps) for the eps its
// scales cover, and faster where the launch has at least a wave of tiles (4 per
// SM); a launch of a few tiles is bound by one tile's latency, which the longer
// FP32 instruction chains raise.
static bool off_fp64_pipe(const cpapr_ctx *ctx, int n) {
    const ModeLayout &L = ctx->mode[n];
    const int dot = ctx->opt.fp64_dot;
    if (L.tile_nnz == 0) return false;  // not configured yet
    return ctx->esize == 8 && ctx->nnz > 0 && ctx->Rp / L.lanes <= 8 && ctx->opt.eps >= 0x1p-43 &&
           ctx->opt.eps < 0x1p31 &&
           (dot == CPAPR_DOT_FP32_PIPE ||
            (dot == CPAPR_DOT_AUTO && ceil_div(ctx->nnz, (int64_t)L.tile_nnz << L.sh) >= kDfMinTiles));
}

static bool pairs_apply(const cpapr_ctx *ctx, int n) { return off_fp64_pipe(ctx, n) && ctx->opt.eps <= 0x1p20; }

bool route_varies(const cpapr_ctx *ctx, int n) {
    return ctx->P[0] && ctx->opt.fp64_dot == CPAPR_DOT_AUTO && pairs_apply(ctx, n);
}

PhiRoute phi_route(const cpapr_ctx *ctx, int n) {
    if (!off_fp64_pipe(ctx, n)) return kRouteFp64;
    if (!ctx->P[0] || !pairs_apply(ctx, n)) return kRoutePipe;
    return ctx->mode[n].late && ctx->opt.fp64_dot == CPAPR_DOT_AUTO ? kRoutePipe : kRoutePairs;
}

// The factors as pairs, where some mode's Phi would read them.  A context without
// the room for them (8 bytes per padded factor entry) keeps the kernels that need none.
cpapr_status ensure_pair_storage(cpapr_ctx *ctx) {
    bool any = false;
    for (int n = 0; n < ctx->N; ++n) any = any || pairs_apply(ctx, n);
    if (!any || ctx->P[0]) return CPAPR_OK;
    size_t ofs[CPAPR_MAX_MODES + 1] = {};
    for (int m = 0; m < ctx->N; ++m) ofs[m + 1] = ofs[m] + (((size_t)ctx->dims[m] * ctx->Rp * 8 + 255) & ~(size_t)255);
    void *p = nullptr;
    const cpapr_status st = dev_alloc(ctx, &p, ofs[ctx->N] + 256);
    if (st == CPAPR_E_NOMEM) {
        ctx->err.clear();
        return CPAPR_OK;
    }
    CPAPR_TRY(st);
    char *base = (char *)p;
    ctx->pair_top = (unsigned long long *)(base + ofs[ctx->N]);
    ctx->kexp = (int32_t *)(base + ofs[ctx->N] + 128);
    ctx->resum = (int32_t *)(base + ofs[ctx->N] + 192);
    for (int m = 0; m < ctx->N; ++m) {
        ctx->P[m] = (float2 *)(base + ofs[m]);
        ctx->pair_state[m] = kPairStale;
    }
    return CPAPR_OK;
}

// tiles of 2^sh table tiles
static void set_tiles(PhiArgs &a, const ModeLayout &L, int sh) {
    a.ksh = sh;
    a.T = L.tile_nnz << sh;
    a.ntiles = (int32_t)ceil_div(a.nnz, a.T);
}

static PhiArgs make_args(cpapr_ctx *ctx, int n, const void *B, void *out, InnerState *inner) {
    const ModeLayout &L = ctx->mode[n];
    PhiArgs a{};
    a.nnz = ctx->nnz;
    a.ntab = L.ntiles;
    set_tiles(a, L, L.sh);
    a.Rp = ctx->Rp;
    a.In = L.In;
    a.nm1 = ctx->N - 1;
    a.atomic = L.reduction == CPAPR_REDUCE_ATOMIC ? 1 : 0;
    a.rstart = L.rstart;
    a.nzrow = L.nzrow;
    a.krow = L.krow;
    int k = 0;
    for (int m = 0; m < ctx->N; ++m) {
        if (m == n) continue;
        a.idx[k] = L.idx[k];
        a.A[k] = ctx->A[m];
        a.Am[k] = ctx->A64[m];
        ++k;
    }
    a.Bm = ctx->B64;
    a.val = L.val;
    a.B = B;
    a.out = out;
    a.carry = ctx->carry;
    a.split = L.split;
    a.tsplit = L.tsplit;
    a.splitcnt = L.splitcnt;
    a.nsplit = L.nsplit;
    a.eps = ctx->opt.eps;
    a.inner = inner;
    a.llpart = ctx->llpart;
    a.err = ctx->errflag + 3;
    a.stage_extra = injected_stage_shortfall();
    a.route = phi_route(ctx, n);
    a.mode = n;
    a.kexp = ctx->kexp;
    for (int m = 0, j = 0; m < ctx->N; ++m)
        if (m != n) a.P[j++] = ctx->P[m];
    return a;
}

template <typename T>
static cudaError_t run_kkt_rows(const T *B, const T *P, int64_t n, InnerState *inner, cudaStream_t s) {
    int64_t g = std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), 152 * 8));
    kkt_rows_kernel<T><<<(unsigned)g, 256, 0, s>>>(B, P, n, inner);
    return cudaGetLastError();
}

static unsigned small_grid(int64_t n) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), 152 * 4));
}

// Zeros the rows of mode n that hold no nonzeros (the tile kernels never
// write them).
cpapr_status launch_zero_empty(cpapr_ctx *ctx, int n, void *out) {
    const ModeLayout &L = ctx->mode[n];
    if (L.nempty == 0) return CPAPR_OK;
    const int64_t m = (int64_t)L.nempty * ctx->Rp;
    if (ctx->esize == 8)
        zero_rows_kernel<double><<<small_grid(m), 256, 0, ctx->stream>>>(L.erows, L.nempty, ctx->Rp, (double *)out);
    else
        zero_rows_kernel<float><<<small_grid(m), 256, 0, ctx->stream>>>(L.erows, L.nempty, ctx->Rp, (float *)out);
    count_launch(ctx);
    CPAPR_CUDA(ctx, cudaGetLastError());
    return CPAPR_OK;
}

// KKT term of the empty rows for the first inner iteration (after S and B).
cpapr_status launch_empty_kkt(cpapr_ctx *ctx, int n, const void *B, InnerState *inner) {
    const ModeLayout &L = ctx->mode[n];
    if (L.nempty == 0 || ctx->nnz == 0 || L.reduction == CPAPR_REDUCE_ATOMIC) return CPAPR_OK;
    const int64_t m = (int64_t)L.nempty * ctx->Rp;
    if (ctx->esize == 8)
        empty_kkt_kernel<double><<<small_grid(m), 256, 0, ctx->stream>>>(L.erows, L.nempty, ctx->Rp,
                                                                         (const double *)B, inner);
    else
        empty_kkt_kernel<float><<<small_grid(m), 256, 0, ctx->stream>>>(L.erows, L.nempty, ctx->Rp,
                                                                        (const float *)B, inner);
    count_launch(ctx);
    CPAPR_CUDA(ctx, cudaGetLastError());
    return CPAPR_OK;
}

template <typename T, int NM1>
static cudaError_t launch_pi_kernel(const PhiArgs &a, T *pi, unsigned grid, cudaStream_t s,
                                    const cudaAccessPolicyWindow *win) {
    if (!win) {
        pi_build_kernel<T, NM1><<<grid, 256, 0, s>>>(a, pi);
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
    return cudaLaunchKernelEx(&cfg, pi_build_kernel<T, NM1>, a, pi);
}

template <typename T>
static cudaError_t run_pi_build(const PhiArgs &a, T *pi, cudaStream_t s, const cudaAccessPolicyWindow *win) {
    const int64_t total = a.nnz * (a.Rp / Vec16<T>::n);
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(total, 256), 152 * 16));
    switch (a.nm1) {
        case 2: return launch_pi_kernel<T, 2>(a, pi, grid, s, win);
        case 3: return launch_pi_kernel<T, 3>(a, pi, grid, s, win);
        case 4: return launch_pi_kernel<T, 4>(a, pi, grid, s, win);
        default: return launch_pi_kernel<T, 0>(a, pi, grid, s, win);
    }
}

cpapr_status prepare_phi(cpapr_ctx *ctx, int n) {
    if (uses_pairs(ctx, n))
        for (int m = 0; m < ctx->N; ++m)
            if (m != n && ctx->pair_state[m] != kPairCurrent) {
                CPAPR_TRY(launch_factor_pairs(ctx, m, ctx->pair_state[m] == kPairStale));
                ctx->pair_state[m] = kPairCurrent;
            }
    if (!ctx->mode[n].pi || ctx->nnz == 0) return CPAPR_OK;
    if (!ctx->pibuf) return fail(ctx, CPAPR_E_STATE, "materialised Pi selected without its buffer");
    PhiArgs a = make_args(ctx, n, nullptr, nullptr, nullptr);
    ProfScope ps(ctx, K_PI);
    count_launch(ctx);
    const cudaError_t e = a.route == kRoutePairs ? launch_pi_pairs(a, ctx->pibuf, ctx->stream, l2_window(ctx))
                          : ctx->esize == 8 ? run_pi_build<double>(a, (double *)ctx->pibuf, ctx->stream, l2_window(ctx))
                                            : run_pi_build<float>(a, (float *)ctx->pibuf, ctx->stream, l2_window(ctx));
    if (e != cudaSuccess) return cuda_fail(ctx, e, "Pi build kernel");
    ctx->pi_mode_built = n;
    ctx->pi_pairs = a.route == kRoutePairs;
    return CPAPR_OK;
}

cpapr_status launch_phi(cpapr_ctx *ctx, int n, PhiOp op, const void *B, void *out, InnerState *inner) {
    ModeLayout &L = ctx->mode[n];
    const int64_t nel = (int64_t)L.In * ctx->Rp;
    PhiArgs a = make_args(ctx, n, B, out, inner);
    if (op == OP_PHI && L.pi) a.pi = ctx->pibuf;
    if (op == OP_PHI) set_tiles(a, L, phi_shift(ctx, n));
    const bool atomic = a.atomic && op != OP_LL;
    if (ctx->nnz == 0 || atomic) {
        CPAPR_CUDA(ctx, cudaMemsetAsync(out, 0, (size_t)nel * ctx->esize, ctx->stream));
    } else if (op != OP_LL && out != ctx->Phi[n]) {
        // a shared output buffer: clear this mode's empty rows.  Phi[n] keeps
        // them zero from the moment the model is set.
        CPAPR_TRY(launch_zero_empty(ctx, n, out));
    }
    if (ctx->nnz > 0) {
        ProfScope ps(ctx, op == OP_MTTKRP ? K_MTTKRP : K_PHI);
        cudaError_t e = dispatch(ctx, a, ctx->Rp / L.lanes, L.lanes, op);
        count_launch(ctx);
        if (e == cudaErrorInvalidValue) return fail(ctx, CPAPR_E_ARG, "no kernel for this rank / lane choice");
        if (e != cudaSuccess) return cuda_fail(ctx, e, "phi tile kernel");
    }
    if (op == OP_PHI && inner && (atomic || ctx->nnz == 0)) {
        count_launch(ctx);
        cudaError_t e = ctx->esize == 8
                            ? run_kkt_rows<double>((const double *)B, (const double *)out, nel, inner, ctx->stream)
                            : run_kkt_rows<float>((const float *)B, (const float *)out, nel, inner, ctx->stream);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "kkt kernel");
    }
    return CPAPR_OK;
}

// Phi^(n) with the segmented reduction over tiles of 2^sh table tiles and a
// caller-supplied carry buffer (2 x tiles x Rp elements of the working type).
// Launches kernels only: no allocation, no event, no memset.
cpapr_status launch_phi_given_carry(cpapr_ctx *ctx, int n, const void *B, void *out, void *carry, int sh) {
    ModeLayout &L = ctx->mode[n];
    PhiArgs a = make_args(ctx, n, B, out, nullptr);
    a.atomic = 0;
    a.carry = carry;
    if (L.pi) a.pi = ctx->pibuf;
    set_tiles(a, L, sh);
    if (ctx->nnz == 0) return fail(ctx, CPAPR_E_ARG, "empty tensor");
    CPAPR_TRY(launch_zero_empty(ctx, n, out));
    cudaError_t e = dispatch(ctx, a, ctx->Rp / L.lanes, L.lanes, OP_PHI);
    count_launch(ctx);
    if (e == cudaErrorInvalidValue) return fail(ctx, CPAPR_E_ARG, "no kernel for this rank / lane choice");
    if (e != cudaSuccess) return cuda_fail(ctx, e, "phi tile kernel");
    return CPAPR_OK;
}

// Log-likelihood sum over the nonzeros, x log m with m = <lambda o A^(n)[i_n], Pi>.
// At the end of an outer iteration the materialised rows of the last mode
// were built from the final factors of all the other modes, so in FP64 the
// sum runs along that mode and streams them; otherwise it runs along mode 0
// with the rows formed in place.  (The FP32 form keeps the gathered rows: its
// underflow fallback recomputes products from the factors.)
cpapr_status launch_loglik(cpapr_ctx *ctx, double *dst) {
    const int N = ctx->N;
    if (ctx->nnz == 0) return launch_ll_total(ctx, ctx->llpart, 0, dst);  // the model total alone
    const bool use_pi = ctx->esize == 8 && ctx->pibuf && ctx->pi_mode_built == N - 1 && ctx->mode[N - 1].pi;
    const int n = use_pi ? N - 1 : 0;
    const ModeLayout &L = ctx->mode[n];
    CPAPR_TRY(launch_scale_b(ctx, n, ctx->B));
    PhiArgs a = make_args(ctx, n, ctx->B, nullptr, nullptr);
    a.atomic = 0;
    if (use_pi) {
        // (the mode's route may have changed since they were built)
        a.pi = ctx->pibuf;
        a.route = ctx->pi_pairs ? kRoutePairs : kRouteFp64;
        set_tiles(a, L, ctx->pi_pairs ? L.sh_df : L.sh);
    }
    {
        ProfScope ps(ctx, K_LL);
        cudaError_t e = dispatch(ctx, a, ctx->Rp / L.lanes, L.lanes, OP_LL);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "log-likelihood kernel");
        count_launch(ctx);
        CPAPR_TRY(launch_ll_total(ctx, ctx->llpart, a.ntiles, dst));
    }
    return CPAPR_OK;
}

}  // namespace cpapr
