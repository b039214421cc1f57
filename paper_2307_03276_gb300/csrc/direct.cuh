// FP32 Phi and MTTKRP tiles without a staged copy of the tile: every group of
// lanes streams its own run of nonzeros through registers.
//
// What it replaces: the staged tile kernel (phi_tile_body) copies a tile's
// streams into shared memory first, which its blocks wait for, and its fast and
// slow batches make long code (14.6 warp instructions per nonzero at 45% of the
// issue slots, 3-way R = 32).  Here a group works on aligned windows of four
// nonzeros: one vector load brings a window's coordinates per mode (single loads
// per nonzero took as many L1 wavefronts as the gathers themselves, 0.245 ms), one
// word its row starts; the next window's are loaded while a window is computed.
// A window with a row start inside takes one more pass over the rows it holds in
// registers; the warp stays converged.  A Phi launch went from 0.256 to 0.225 ms
// (3-way, 1e7 nonzeros, R = 32, rows formed in place; bound by the latency of the L2
// gathers and instruction issue at 57%) and from 0.650 to 0.561 ms (4-way, 5e7, R = 16,
// materialised rows; 0.89 of the HBM peak), with a smaller error: sums of 16 terms
// are compensated, and the quotient is within an ulp.  128 threads: with 256 the
// same launches took 0.231 and 0.582 ms at their best tiles, the batch 33 ms (27.5).
#pragma once

#include "phi_kernels.cuh"

namespace cpapr {

constexpr int kDirectThreads = 128;

// Index in nzrow of the row holding position qa of tile [p0, p1]: the tile's
// first row plus the row starts in (p0, qa], counted by the warp over the tile's
// words of row-start bits (every lane of the warp calls it).
__device__ __forceinline__ int run_first_row(const PhiArgs &a, int t, int p0, int p1, int qa, int wlane) {
    constexpr unsigned full = 0xffffffffu;
    int k = __ldg(a.krow + ((int64_t)t << a.ksh));
    const int w0 = p0 >> 5, w1 = p1 >> 5, wt = qa >> 5;
    int before = 0;
    for (int base = w0; base <= w1; base += 32) {
        const int w = base + wlane;
        uint32_t b = w <= w1 ? __ldg(a.rstart + w) : 0u;
        if (w == w0) b &= ~((2u << (p0 & 31)) - 1u);
        const int c = __popc(b);
        int x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(full, x, o);
            if (wlane >= o) x += y;
        }
        const int src = wt - base;
        const int ex = __shfl_sync(full, x - c, src & 31);
        const uint32_t bw = __shfl_sync(full, b, src & 31);
        if (src >= 0 && src < 32) k += before + ex + __popc(bw & (0xffffffffu >> (31 - (qa & 31))));
        before += __shfl_sync(full, x, 31);
    }
    return k;
}

// x / max(s, eps): the hardware reciprocal with one residual correction (within
// an ulp; a plain reciprocal product is within two)
__device__ __forceinline__ float direct_divide(float x, float s, float eps) {
    const float m = s > eps ? s : eps;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
    const float q = x * r;
    const float c = fmaf(fmaf(-q, m, x), r, q);
    // (huge divisors, whose reciprocal is 0; tiny ones and quotients beyond the float
    // range, whose correction is NaN)
    return m < 0x1p100f && q < __int_as_float(0x7f800000) ? c : __fdiv_rn(x, m);
}

// shared memory of a tile: partial-row slots, their rows, the rows finished here
__host__ __device__ constexpr size_t direct_smem() {
    return (size_t)2 * kDirectThreads * 4 * sizeof(float) + (size_t)(2 * kDirectThreads + 2) * 4;
}

// One tile (t) of one tensor (a) by a block of kDirectThreads threads; G = Rp / 4
// lanes with a float4 of ranks each.  A run's terms are summed in two
// interleaved accumulators for 16 nonzeros at a time, whose sums go to a
// compensated (Kahan) sum.
template <int NM1, int G, int OP, bool PI>
__device__ __forceinline__ void direct_tile(const PhiArgs &a, const int t, unsigned char *smem_raw, double *red) {
    static_assert(OP == OP_PHI || (OP == OP_MTTKRP && !PI), "Phi or MTTKRP");
    constexpr int THREADS = kDirectThreads, NG = THREADS / G, U = 4;
    constexpr int MAXK = PI ? 1 : (NM1 > 0 ? NM1 : kMaxNm1);
    constexpr int Rp = 4 * G;
    constexpr unsigned full = 0xffffffffu;
    constexpr int LPU = G >= U ? G / U : 1;  // lanes per finished nonzero
    constexpr int NF = G >= U ? 1 : U / G;   // nonzeros a lane finishes: u0 .. u0 + NF - 1
    float *slot_val = reinterpret_cast<float *>(smem_raw);                    // [2 * NG][Rp]
    int32_t *slot_row = reinterpret_cast<int32_t *>(slot_val + 2 * NG * Rp);  // [2 * NG]
    int32_t *slot_fin = slot_row + 2 * NG;                                    // [2]

    const int tid = threadIdx.x;
    const int g = tid / G, lane = tid % G, wlane = tid & 31;
    const int u0 = (lane / LPU) * NF;
    const int gbase = (wlane / G) * G;
    const int nm1 = (!PI && NM1 > 0) ? NM1 : a.nm1;
    const float *Bm = reinterpret_cast<const float *>(a.B);
    const float *__restrict__ val = reinterpret_cast<const float *>(a.val);
    float *out = reinterpret_cast<float *>(a.out);
    const float eps = (float)a.eps;
    // positions are below 2^31 (so is the number of nonzeros); runs start at
    // multiples of four (so do tiles)
    const int p0 = t * a.T;
    const int p1 = (int)min((int64_t)p0 + a.T, a.nnz);
    const int vlen = ((a.T + NG - 1) / NG + U - 1) & ~(U - 1);
    const int qa = (int)min((int64_t)p0 + (int64_t)g * vlen, (int64_t)p1);
    const int qb = min(qa + vlen, p1);
    auto bit_at = [&](int p) -> uint32_t { return (__ldg(a.rstart + (p >> 5)) >> (p & 31)) & 1u; };

    int kcur = run_first_row(a, t, p0, p1, qa, wlane);
    const bool run = qa < qb;
    const bool head_open = qa > 0 && !bit_at(qa);
    const bool tail_open = qb < a.nnz && !bit_at(qb);
    int32_t cur = __ldg(a.nzrow + kcur);
    int32_t nxt = __ldg(a.nzrow + kcur + 1);  // (padded past the last row)
    bool first = true;
    if (lane == 0) slot_row[2 * g] = slot_row[2 * g + 1] = -1;
    if (tid < 2) slot_fin[tid] = -1;

    float kkt = 0.f;
    float b[4], acc[2][4], ks[4], kc[4];
    auto load4 = [&](const float *row, float (&d)[4]) {
        const float4 y = __ldg(reinterpret_cast<const float4 *>(row) + lane);
        d[0] = y.x, d[1] = y.y, d[2] = y.z, d[3] = y.w;
    };
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[0][r] = acc[1][r] = ks[r] = kc[r] = 0.f;
    // the accumulators into the compensated sum
    auto fold = [&]() {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float y = (acc[0][r] + acc[1][r]) - kc[r];
            const float s = ks[r] + y;
            // (finite even where the sum is not, so that it stays infinite: its correction
            // would be infinite or NaN, and fminf returns the other operand of a NaN)
            kc[r] = fminf((s - ks[r]) - y, 0x1.fffffep127f);
            ks[r] = s;
            acc[0][r] = acc[1][r] = 0.f;
        }
    };
    if (OP == OP_PHI) load4(Bm + (int64_t)cur * Rp, b);

    auto flush = [&](bool is_last) {
        const bool before = first && head_open, after = is_last && tail_open;
        fold();
        float v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            v[r] = ks[r] - kc[r];
            ks[r] = kc[r] = 0.f;
        }
        const float4 v4 = make_float4(v[0], v[1], v[2], v[3]);
        if (!before && !after) {
            reinterpret_cast<float4 *>(out + (int64_t)cur * Rp)[lane] = v4;
            if (OP == OP_PHI && a.inner) {
#pragma unroll
                for (int r = 0; r < 4; ++r) kkt = tmax(kkt, viol_t(b[r], v[r]));
            }
        } else if (a.atomic) {
#pragma unroll
            for (int r = 0; r < 4; ++r) atomicAdd(out + (int64_t)cur * Rp + lane * 4 + r, v[r]);
        } else {
            const int s = before ? 2 * g : 2 * g + 1;
            if (lane == 0) slot_row[s] = cur;
            reinterpret_cast<float4 *>(slot_val + (int64_t)s * Rp)[lane] = v4;
        }
    };

    // what a window reads: its row starts; its counts; the materialised rows, or the
    // coordinates of the rows to form (streams are padded past the last nonzero)
    float pi[U][4];
    int4 ii[MAXK];
    uint32_t bits = 0;
    float x[NF];
    const int pmax = (p1 - 1) & ~(U - 1);
    auto load_window = [&](int w) {
        const int p = min(w, pmax);
        bits = __ldg(a.rstart + (p >> 5)) >> (p & 31);
#pragma unroll
        for (int f = 0; f < NF; ++f) x[f] = __ldg(val + p + u0 + f);
        if constexpr (PI) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float4 y = __ldcs(reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(a.pi) +
                                                                         (int64_t)min(p + u, p1 - 1) * Rp) + lane);
                pi[u][0] = y.x, pi[u][1] = y.y, pi[u][2] = y.z, pi[u][3] = y.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < MAXK; ++k)
                if (k < nm1) ii[k] = __ldg(reinterpret_cast<const int4 *>(a.idx[k] + p));
        }
    };
    int w = qa;
    load_window(w);
#pragma unroll 1
    for (int step = 1; __any_sync(full, w < qb); ++step) {
        if constexpr (!PI) {
#pragma unroll
            for (int k = 0; k < MAXK; ++k) {
                if (k < nm1) {
                    const float *A = reinterpret_cast<const float *>(a.A[k]);
                    const int32_t i4[U] = {ii[k].x, ii[k].y, ii[k].z, ii[k].w};
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        float f[4];
                        load4(A + (int64_t)i4[u] * Rp, f);
#pragma unroll
                        for (int r = 0; r < 4; ++r) pi[u][r] = k == 0 ? f[r] : pi[u][r] * f[r];
                    }
                }
            }
        }
        // the window's nonzeros [lo, hi) of the run, in passes of one row each
        int lo = 0;
        const int hi = max(min(U, qb - w), 0);
        uint32_t st = bits & ((1u << hi) - 1u);
        if (w == qa) st &= ~1u;  // the run's first row is cur
        do {
            if ((st >> lo) & 1u) {
                flush(false);
                first = false;
                cur = nxt;
                nxt = __ldg(a.nzrow + ++kcur + 1);
                if (OP == OP_PHI) load4(Bm + (int64_t)cur * Rp, b);
            }
            const uint32_t rest = (st >> lo) >> 1;
            const int end = rest ? lo + __ffs(rest) : hi;
            float v[U];
            if constexpr (OP == OP_MTTKRP) {
#pragma unroll
                for (int u = 0; u < U; ++u)
                    v[u] = G > 1 ? __shfl_sync(full, x[u % NF], gbase + (u / NF) * LPU) : x[u % NF];
            } else {
                float s[U], y[NF];
#pragma unroll
                for (int u = 0; u < U; ++u) s[u] = dot_regs<float, 4>(b, pi[u]);
                if constexpr (G == 1) {
#pragma unroll
                    for (int f = 0; f < NF; ++f) y[f] = direct_divide(x[f], s[f], eps);
                } else if constexpr (G == 2) {
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        const float send = lane ? s[f] : s[f + 2], keep = lane ? s[f + 2] : s[f];
                        y[f] = direct_divide(x[f], keep + __shfl_xor_sync(full, send, 1), eps);
                    }
                } else {
                    y[0] = direct_divide(x[0], group_reduce_scatter<float, (G >= U ? G : U), U>(s, lane, full), eps);
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    v[u] = G > 1 ? __shfl_sync(full, y[u % NF], gbase + (u / NF) * LPU) : y[u % NF];
            }
            // nonzeros of other passes stay out (they may hold infinities)
            if (__all_sync(full, end - lo == U)) {
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int r = 0; r < 4; ++r) acc[u & 1][r] = fmaf(v[u], pi[u][r], acc[u & 1][r]);
            } else {
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (u >= lo && u < end) {
#pragma unroll
                        for (int r = 0; r < 4; ++r) acc[u & 1][r] = fmaf(v[u], pi[u][r], acc[u & 1][r]);
                    }
            }
            lo = end;
        } while (__any_sync(full, lo < hi));
        if (step % 4 == 0) fold();
        w += U;
        load_window(w);
    }
    if (run) flush(true);
    if (!a.atomic) {
        // the row at the next tile's start if it goes on from this tile, else -1
        auto next_row_of = [&]() -> int32_t {
            return (p1 < a.nnz && !bit_at(p1))
                       ? __ldg(a.nzrow + __ldg(a.krow + min((int64_t)(t + 1) << a.ksh, (int64_t)a.ntab)))
                       : -1;
        };
        segmented_tail<float, OP, THREADS, NG, Rp, Rp>(a, t, slot_val, slot_row, slot_fin, next_row_of, Bm, out,
                                                       tid >> 5, wlane, kkt);
        if (OP == OP_PHI && a.inner) publish_kkt<THREADS>((double)kkt, a.inner, red);
    }
}

}  // namespace cpapr
