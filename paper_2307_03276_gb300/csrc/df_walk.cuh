// The FP64 form's Phi with the Khatri-Rao rows as float pairs (df_pair.cuh): the
// dot s = <B[i_n], pi>, the division v = x / max(s, eps) and the scale-add
// Phi[i_n] += v pi all run on the FP32 pipe with error-free transformations.
//
// What bounded it before: with only the divisor on the FP32 pipe the kernel cut
// every FP64 Pi element into two floats for the dot (13 integer operations per
// element) and issued one DFMA per element for the scale-add, 64 cycles of an
// SM quarter's FP64 pipe per warp instruction: 63 issue slots and 64 FP64 cycles
// per element.  Now the pairs are built once per mode and outer iteration and an
// element costs about 18 FP32 operations, two columns per packed instruction, and
// no FP64 one (the FP32 sums move to an FP64 accumulator every 16 nonzeros).  A
// launch on the 4-way tensor with 5e7 nonzeros (R = 16) went from 2.67 to 1.31 ms
// (0.73 of the HBM peak for its 6.45 GB), on the 3-way one with 1e7 (R = 32) from
// 0.95 to 0.58 ms (0.68); 1.37 and 0.61 before the packed instructions.  What bounds
// it now is instruction issue and the waits that too few warps (20 per SM) leave
// open: loads of the next step, and the block's slowest warp at a tile's end.
//
// Scaled quantities (all powers of two): pi' = pi 2^K (the pairs), b' = b 2^(S - K),
// eps' = eps 2^S, s' = s 2^S with S = kDfS; v' = v 2^V with V = kDfV; FP32 sums
// of v' pi' carry 2^(K + V), the FP64 accumulators nothing.  The float range then covers
//   pi' in [2^-80, 2^60], v' in [2^-20, 2^50] or 0, s' in [0, 2^100);
// a nonzero outside (a huge model value, a count outside {0} and [2^-20, 2^30), a
// quotient outside the window) is redone in FP64 by its group.  Escaped elements
// below the window add 0 to the dot: they are below 2^-80 while max(s', eps') >= eps', so the
// dropped terms stay below 2^-47 of it where b' < eps' 2^34; else the nonzero is
// redone in FP64.  They are left out of the sums as well, with a bound on what
// that leaves out; a column whose sum is not large beside it is summed again in
// FP64 (along a solve a quarter of the elements come to escape, and hardly any
// matters: with each added in FP64 as it came an outer iteration of the 3-way
// tensor grew from 21 to 55 ms within 20 of them).
//
// Error of v relative to itself, u = 2^-24, k = 4 terms per lane (all >= 0): the
// pairs' rounding (2^-49 for b, 2^-47 for a product), the dropped lo lo terms
// (u^2 each), and the FP32 sums of the two-sum errors, FMA errors and cross
// terms, each at most u of its product and rounded to u of itself: k^2 u^2 + 4 k u^2
// < 40 u^2 at worst and a few u^2 in the mean; the quotient's remainder is exact to
// 2 u^2.  That is below 3e-13 at worst.  The scale-add of n terms rounds C, at most (2 + n) u
// of the sum, three times a term: (3 n (2 + n) + n) u^2, 3e-12 for the 16 terms between two
// moves to FP64 if every rounding had one sign, some 1e-15 as they come.  Phi entries
// of the timed workloads are within 1e-14 to 3e-14 of 64-bit results, like those of
// the FP64 scale-add and the one-step quotient before (a few parts larger on the 4-way
// solve, smaller on others).
#pragma once

#include "direct.cuh"

namespace cpapr {

constexpr int kDfS = 60;
constexpr int kDfV = 10;
static_assert(30 + kDfS + kDfV <= 100, "df_bad_x: counts below 2^30 stay below df_cut's 2^100");
constexpr int kDfThreads = 128;
// Resident blocks per SM the registers are held to (96 each).  4 / 5 / 6 blocks:
// 1.43 / 1.31 / 1.36 ms a launch (4-way, 5e7 nonzeros, R = 16), 0.64 / 0.58 / 0.59 ms
// (3-way, 1e7, R = 32); six (80 registers) spill.
constexpr int kDfBlocks = 5;
constexpr int kDfSpill = 16;  // nonzeros summed in FP32 pairs before they move to FP64

// doubles from one partial-row slot to the next: two more than a row, so that
// the slots of a warp's groups start in different shared-memory banks
__host__ __device__ constexpr int df_slot_stride(int rp) { return rp + 2; }

// x 2^s (x >= 0) as hi + lo, its leading 48 bits rounded to nearest hi: integer
// operations and one integer-to-float conversion.  Below 2^-126: 0 + 0; from
// 2^100 on (and infinite or NaN): hi = inf.
__device__ __forceinline__ void df_cut(double x, int s, float &hi, float &lo) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const uint32_t H = (uint32_t)(bits >> 32), L = (uint32_t)bits;
    const int e = (int)(H >> 20) + s;  // biased exponent of x 2^s
    const bool keep = e >= 1023 - 126;
    // the first 23 fraction bits with the exponent rebased from 1023 to 127
    const float h = __uint_as_float(__funnelshift_l(L, H, 3) + ((uint32_t)(s - 896) << 23));
    // the next 29 fraction bits (24 kept) times 2^(e - 1075), in two exact steps that
    // stay in the float range for every e kept
    const float m = __uint2float_rz(L & 0x1fffffffu);
    const float l = __fmul_rn(m * __uint_as_float((uint32_t)(e - 1023 + 127) << 23), 0x1p-52f);
    const float t = h + l;
    hi = keep ? t : 0.f;
    lo = keep ? l - (t - h) : 0.f;
    if (e >= 1023 + 100) {
        hi = __uint_as_float(0x7f800000u);
        lo = 0.f;
    }
}

// S + C += a b for pairs a, b >= 0, two columns at once (.x and .y: Blackwell's
// packed FP32 instructions take two per lane and issue slot; the kernel is bound by
// issue).  t = S + a_hi b_hi is rounded once (FMA); its error is (S - (t - z)) +
// (a_hi b_hi - z) with z = t - S as in Knuth's two-sum: the first part is exact, the
// second is an FMA whose rounding is 2^-24 of it, 2^-48 of t.  The error and the
// cross terms go to C: nine operations (twelve with the product and the sum
// taken apart).  Differences are FMAs with -1, which round the same.
__device__ __forceinline__ void df_fma2(float2 ah, float2 al, float2 bh, float2 bl, float2 &S, float2 &C) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 t = __ffma2_rn(ah, bh, S);
    const float2 nz = __ffma2_rn(t, m1, S);                       // -z
    const float2 e = __ffma2_rn(__fadd2_rn(t, nz), m1, S);        // S - (t - z)
    const float2 r = __ffma2_rn(ah, bh, nz);
    C = __ffma2_rn(ah, bl, C);
    C = __ffma2_rn(al, bh, C);
    C = __fadd2_rn(C, __fadd2_rn(e, r));
    S = t;
}

// <a, b> of two rows of pairs as a renormalised pair: even and odd columns
// side by side, then their sums added (two-sum)
template <int VP>
__device__ __forceinline__ float2 df_dot(const float2 (&ah)[VP], const float2 (&al)[VP], const float2 (&bh)[VP],
                                         const float2 (&bl)[VP]) {
    const float2 m1 = make_float2(-1.f, -1.f), zero = make_float2(0.f, 0.f);
    float2 S = __fmul2_rn(ah[0], bh[0]);
    float2 C = __ffma2_rn(ah[0], bh[0], __ffma2_rn(S, m1, zero));
    C = __ffma2_rn(ah[0], bl[0], C);
    C = __ffma2_rn(al[0], bh[0], C);
#pragma unroll
    for (int v = 1; v < VP; ++v) df_fma2(ah[v], al[v], bh[v], bl[v], S, C);
    const float t = S.x + S.y;
    const float z = t - S.x;
    const float c = ((S.x - (t - z)) + (S.y - z)) + (C.x + C.y);
    const float h = t + c;
    return make_float2(h, c - (h - t));
}

// (xh + xl) / max(s, eps) as a pair: q0 from the hardware reciprocal refined by
// one Newton step, the remainder x - q0 m (the product q0 m_hi taken exactly with
// an FMA; x_hi - p is exact, p being within a factor of two of x_hi) divided
// by m_hi, and the two added.  Operands are in the ranges above.
__device__ __forceinline__ float2 df_divide(float xh, float xl, float2 s, float eh, float el) {
    const bool use_s = (s.x - eh) + (s.y - el) >= 0.f;  // s.x - eh is exact where they are close
    const float mh = use_s ? s.x : eh, ml = use_s ? s.y : el;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(mh));
    r = fmaf(r, fmaf(-mh, r, 1.f), r);
    const float q0 = __fmul_rn(xh, r);
    const float p = __fmul_rn(q0, mh);
    const float pe = fmaf(q0, mh, -p);
    const float q1 = __fmul_rn(((xh - p) - pe) + fmaf(-q0, ml, xl), r);
    const float h = q0 + q1;
    return make_float2(h, q1 - (h - q0));
}

// true unless x = 0 or 2^-20 <= x < 2^30 (x >= 0): x 2^(kDfS + kDfV) is within df_cut's range
__device__ __forceinline__ bool df_bad_x(double x) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const unsigned e = (unsigned)(bits >> 52);
    return bits != 0ull && (e < 1023u - 20u || e >= 1023u + 30u);
}

// (The paths that are rarely taken are inlined all the same: as called functions
// they cost the loop its registers, 1.53 against 1.39 ms a launch on the 4-way
// tensor.)

// this lane's columns of nonzero p's row in FP64, and its part of <B[row], pi>: the
// pairs' values, and FP64 products where there is none
template <int NM1, int RPL, int G, bool PI>
__device__ __forceinline__ double pair_row64(const PhiArgs &a, int nm1, int K, int p, int row, int lane,
                                             double (&pv)[RPL]) {
    const double *B = reinterpret_cast<const double *>(a.B) + (int64_t)row * (RPL * G);
    constexpr int Rp = RPL * G, MAXK = PI ? 1 : NM1 > 0 ? NM1 : kMaxNm1;
    int64_t at[MAXK];
    if constexpr (!PI) {
#pragma unroll
        for (int k = 0; k < MAXK; ++k) at[k] = k < nm1 ? (int64_t)__ldg(a.idx[k] + p) * Rp : 0;
    }
#pragma unroll
    for (int v = 0; v < RPL / 2; ++v) {
        float2 e0, e1;
        double2 f = make_double2(0.0, 0.0);
        if constexpr (PI) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = (v * G + lane) * 2 + h;
                const float2 e = pair_at(reinterpret_cast<const float *>(a.pi), (int64_t)p * Rp, c);
                double d = pair_value(e, K);
                if (is_escape(e)) {
                    d = 1.0;
#pragma unroll 1
                    for (int k = 0; k < nm1; ++k)
                        d *= __ldg(reinterpret_cast<const double *>(a.A[k]) + (int64_t)__ldg(a.idx[k] + p) * Rp + c);
                }
                pv[2 * v + h] = d;
            }
            continue;
        } else {
            PairProduct y0, y1;
#pragma unroll
            for (int k = 0; k < MAXK; ++k)
                if (k < nm1) {
                    const float4 y = __ldg(reinterpret_cast<const float4 *>(a.P[k] + at[k]) + v * G + lane);
                    if (k == 0) {
                        y0.start(make_float2(y.x, y.z));
                        y1.start(make_float2(y.y, y.w));
                    } else {
                        y0.mul(make_float2(y.x, y.z));
                        y1.mul(make_float2(y.y, y.w));
                    }
                }
            e0 = y0.value();
            e1 = y1.value();
            if (is_escape(e0) || is_escape(e1)) {
#pragma unroll
                for (int k = 0; k < MAXK; ++k)
                    if (k < nm1) {
                        const double2 g = __ldg(reinterpret_cast<const double2 *>(
                                                    reinterpret_cast<const double *>(a.A[k]) + at[k]) + v * G + lane);
                        f = k == 0 ? g : make_double2(f.x * g.x, f.y * g.y);
                    }
            }
        }
        pv[2 * v] = is_escape(e0) ? f.x : pair_value(e0, K);
        pv[2 * v + 1] = is_escape(e1) ? f.y : pair_value(e1, K);
    }
    double d = 0.0;
#pragma unroll
    for (int r = 0; r < RPL; ++r) d = fma(__ldg(B + ((r >> 1) * G + lane) * 2 + (r & 1)), pv[r], d);
    return d;
}

// Nonzero p in FP64: a warp's lanes all call it, those of the groups that redo
// their nonzero (`mine`) add v pi to their accumulators (Phi); returns x log m in
// lane 0 of such a group (log-likelihood).
template <int NM1, int RPL, int G, int OP, bool PI>
__device__ __forceinline__ double pair_redo(const PhiArgs &a, double2 *acc, int nm1, int K, int p, int row, int lane,
                                         bool mine) {
    double pv[RPL];
    double d = pair_row64<NM1, RPL, G, PI>(a, nm1, K, p, row, lane, pv);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if (!mine) return 0.0;
    const double x = __ldg(reinterpret_cast<const double *>(a.val) + p);
    if (OP == OP_LL) return lane == 0 ? x * log(d) : 0.0;
    const double v = phi_divide(x, d, a.eps);
#pragma unroll
    for (int k = 0; k < RPL / 2; ++k) {
        double2 t = acc[k * G + lane];
        t.x = fma(v, pv[2 * k], t.x);
        t.y = fma(v, pv[2 * k + 1], t.y);
        acc[k * G + lane] = t;
    }
    return 0.0;
}

// The columns `low` of v: the sums of v pi over one row's nonzeros from q - 1 back
// to the row's start, or to qa, in FP64.  A group's lanes call it together.
template <int NM1, int RPL, int G, bool PI>
__device__ __forceinline__ void pair_resum(const PhiArgs &a, int nm1, int K, int qa, int q, int row, int lane,
                                           unsigned gmask, uint32_t low, double (&v)[RPL]) {
#pragma unroll
    for (int r = 0; r < RPL; ++r)
        if ((low >> r) & 1u) v[r] = 0.0;
    bool more = true;
#pragma unroll 1
    for (int p = q - 1; more; --p) {
        more = p > qa && !((__ldg(a.rstart + (p >> 5)) >> (p & 31)) & 1u);
        double pv[RPL];
        double d = pair_row64<NM1, RPL, G, PI>(a, nm1, K, p, row, lane, pv);
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) d += __shfl_xor_sync(gmask, d, o);
        d = phi_divide(__ldg(reinterpret_cast<const double *>(a.val) + p), d, a.eps);
#pragma unroll
        for (int r = 0; r < RPL; ++r)
            if ((low >> r) & 1u) v[r] = fma(d, pv[r], v[r]);
    }
}

// One block per tile; a group of G lanes owns a contiguous run of the tile and
// takes U nonzeros of one row per step.  A step ends early where a row ends, so
// that a flush and the next row's B come at one place, before a step, and the
// code of the loop stays within the instruction cache (with a flush after every
// nonzero and the FP64 paths unrolled in line, a quarter of the stalls waited for
// instructions).  Every lane of a warp steps until all its groups are done, so the
// warp stays converged and exchanges over full masks; positions past a step or a
// run weigh nothing.
//
// Nothing is staged in shared memory: the next step's rows, counts and row-start
// bits are loaded into registers at the end of a step (the other warps' work
// covers their latency), so no block waits for a tile's copies, and a block holds
// little shared memory.  Four ranks per lane: a row change costs a lane half of
// what it does with eight.  A lane's element r is column ((r / 2) G + lane) 2 +
// r % 2: the lanes of a group read 16 G contiguous bytes per load, whole sectors.
template <int NM1, int RPL, int G, int OP, int U, bool PI>
__global__ void __launch_bounds__(kDfThreads, kDfBlocks) phi_pair_kernel(const __grid_constant__ PhiArgs a) {
    static_assert(RPL % 2 == 0 && RPL <= 8 && U <= 4, "pairs of columns, 8 mask bits per nonzero");
    static_assert(OP == OP_PHI || (OP == OP_LL && PI), "Phi, or the log-likelihood of materialised rows");
    constexpr int THREADS = kDfThreads, NG = THREADS / G;
    constexpr int MAXK = PI ? 1 : (NM1 > 0 ? NM1 : kMaxNm1);
    constexpr int Rp = RPL * G, SP = df_slot_stride(Rp), VP = RPL / 2;
    constexpr unsigned full = 0xffffffffu;
    constexpr int LPU = G > 1 ? G / U : 1;
    constexpr int XN = G > 1 ? 1 : U;  // counts a lane holds: its own nonzero's, or all
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[THREADS / 32];
    double *slot_val = reinterpret_cast<double *>(smem_raw);                // [2 * NG][SP]
    int32_t *slot_row = reinterpret_cast<int32_t *>(slot_val + 2 * NG * SP);  // [2 * NG]
    int32_t *slot_fin = slot_row + 2 * NG;                                  // [2]

    if (a.inner && a.inner->done) return;
    const int t = blockIdx.x, tid = threadIdx.x;
    const int g = tid / G, lane = tid % G, wlane = tid & 31;
    const int u_mine = G > 1 ? lane / LPU : 0;
    const int gbase = (wlane / G) * G;
    const unsigned gmask = G >= 32 ? full : ((1u << (G & 31)) - 1u) << gbase;
    const int nm1 = (!PI && NM1 > 0) ? NM1 : a.nm1;
    const double *__restrict__ Bm = reinterpret_cast<const double *>(a.B);
    const double *__restrict__ val = reinterpret_cast<const double *>(a.val);
    double *__restrict__ out = reinterpret_cast<double *>(a.out);
    // positions are below 2^31 (so is the number of nonzeros)
    const int p0 = t * a.T;
    const int p1 = (int)min((int64_t)p0 + a.T, a.nnz);
    const int vlen = (a.T + NG - 1) / NG;
    const int qa = (int)min((int64_t)p0 + (int64_t)g * vlen, (int64_t)p1);
    const int qb = min(qa + vlen, p1);

    int K = kPairTop;
    for (int m = 0; m <= nm1; ++m)
        if (m != a.mode) K -= __ldg(a.kexp + m);
    // the FP32 sums carry 2^(K + kDfV), the FP64 accumulator nothing, so that it has the
    // FP64 range (|K| <= 760); unit takes the one to the other, exactly
    const double unit = __hiloint2double((1023 - K - kDfV) << 20, 0);
    float eh, el;
    df_cut(a.eps, kDfS, eh, el);
    const float bmax = eh * 0x1p34f;

    auto bit_at = [&](int p) -> uint32_t { return (__ldg(a.rstart + (p >> 5)) >> (p & 31)) & 1u; };
    auto col = [&](int v) -> int { return (v * G + lane) * 2; };

    int kcur = run_first_row(a, t, p0, p1, qa, wlane);
    const bool run = qa < qb;
    const bool head_open = qa > 0 && !bit_at(qa);
    const bool tail_open = qb < a.nnz && !bit_at(qb);
    int32_t cur = __ldg(a.nzrow + kcur);
    int32_t nxt = __ldg(a.nzrow + kcur + 1);  // (padded past the last row)
    bool first = true;

    if (OP == OP_PHI) {
        if (lane == 0) slot_row[2 * g] = slot_row[2 * g + 1] = -1;
        if (tid < 2) slot_fin[tid] = -1;
    }
    // the running KKT maximum starts from the one published so far
    double kkt = 0.0, ll = 0.0;
    if (OP == OP_PHI && a.inner) {
        const int l = *((volatile int32_t *)&a.inner->l);
        kkt = __longlong_as_double((long long)*((volatile unsigned long long *)&a.inner->kkt[l & 1]));
    }

    float2 S[VP], C[VP], bh[VP], bl[VP];  // columns 2v (.x) and 2v + 1 (.y)
    float top = 0.f;  // largest b_hi of the lane's columns
    auto load_b = [&](int32_t row) {
        top = 0.f;
#pragma unroll
        for (int v = 0; v < VP; ++v) {
            const double2 b = __ldg(reinterpret_cast<const double2 *>(Bm + (int64_t)row * Rp + col(v)));
            df_cut(b.x, kDfS - K, bh[v].x, bl[v].x);
            df_cut(b.y, kDfS - K, bh[v].y, bl[v].y);
            top = fmaxf(top, fmaxf(bh[v].x, bh[v].y));
        }
    };
    load_b(cur);

    // the FP64 accumulator: this lane's columns of the group's tail slot
    double2 *acc = reinterpret_cast<double2 *>(slot_val + (int64_t)(2 * g + 1) * SP);
    if (OP == OP_PHI) {
#pragma unroll
        for (int v = 0; v < VP; ++v) acc[v * G + lane] = make_double2(0.0, 0.0);
#pragma unroll
        for (int v = 0; v < VP; ++v) S[v] = C[v] = make_float2(0.f, 0.f);
    }
    int q = qa;
    // escapes left out of the current sums: the columns that had them (low 8 bits)
    // and a float not below the sum of their nonzeros' v' (the bits above)
    uint32_t esc = 0;
    // b_hi = bh 2^(K - S) where the float range holds it; its entries below
    // 2^-126 2^(K - S) count as 0, far inside kkt_candidate's margin
    const bool b_in_regs = K >= -40 && K <= 140;
    const float b_scale = b_in_regs ? __uint_as_float((uint32_t)(K - kDfS + 127) << 23) : 0.f;
    auto flush = [&](bool is_last) {
        const bool before = first && head_open, after = is_last && tail_open;
        double v[RPL];
#pragma unroll
        for (int k = 0; k < VP; ++k) {
            const double2 t = acc[k * G + lane];
            v[2 * k] = fma(df_widen(S[k].x) + df_widen(C[k].x), unit, t.x);
            v[2 * k + 1] = fma(df_widen(S[k].y) + df_widen(C[k].y), unit, t.y);
            acc[k * G + lane] = make_double2(0.0, 0.0);
            S[k] = C[k] = make_float2(0.f, 0.f);
        }
        // escaped elements were left out: below 2^-80 of their v' in all, nothing in FP64
        // beside a sum of 2^-25 of them or more; a column with less is summed again
        uint32_t low = 0;
        if (__builtin_expect(esc != 0u, 0)) {
            const double bound = df_widen(__uint_as_float(esc & ~0xffu)) * 0x1p-25 * unit;
#pragma unroll
            for (int r = 0; r < RPL; ++r)
                if (((esc >> r) & 1u) && !(v[r] >= bound)) low |= 1u << r;
        }
        if (__builtin_expect(__any_sync(gmask, low != 0u), 0)) {
            pair_resum<NM1, RPL, G, PI>(a, nm1, K, qa, q, cur, lane, gmask, low, v);
        }
        esc = 0;
        if (!before && !after) {
            double *o = out + (int64_t)cur * Rp;
#pragma unroll
            for (int k = 0; k < VP; ++k)
                *reinterpret_cast<double2 *>(o + col(k)) = make_double2(v[2 * k], v[2 * k + 1]);
            if (a.inner) {
                // the exact FP64 term only where it could raise the running maximum
                // (flushes diverge across a warp's groups, and each FP64 warp
                // instruction costs the FP64 pipe the same with two lanes or 32)
                const float kf = float_below(kkt);
                const double *b = Bm + (int64_t)cur * Rp;
#pragma unroll
                for (int r = 0; r < RPL; ++r) {
                    const float br = r % 2 ? bh[r / 2].y : bh[r / 2].x;
                    if (!b_in_regs || !(br < 0x1p100f) || kkt_candidate(br * b_scale, v[r], kf))
                        kkt = tmax(kkt, viol_t(__ldg(b + col(r / 2) + r % 2), v[r]));
                }
            }
        } else if (a.atomic) {
#pragma unroll
            for (int r = 0; r < RPL; ++r) atomicAdd(out + (int64_t)cur * Rp + col(r / 2) + r % 2, v[r]);
        } else {
            const int s = before ? 2 * g : 2 * g + 1;
            if (lane == 0) slot_row[s] = cur;
            double *o = slot_val + (int64_t)s * SP;
#pragma unroll
            for (int k = 0; k < VP; ++k)
                *reinterpret_cast<double2 *>(o + col(k)) = make_double2(v[2 * k], v[2 * k + 1]);
        }
    };

    float2 ph[U][VP], pl[U][VP];  // rows of the step at position q: hi and lo parts, columns as above
    // what a step reads: the materialised rows, or the coordinates of the rows to
    // form; its row starts; its counts
    int32_t ii[U][MAXK];
    uint32_t starts = 0;
    double x[XN];
    auto load_step = [&](int q) {
        const uint32_t *w = a.rstart + (q >> 5);
        starts = __funnelshift_r(__ldg(w), __ldg(w + 1), q & 31);
        if constexpr (G > 1) {
            x[0] = __ldg(val + min(q + u_mine, p1 - 1));
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) x[u] = __ldg(val + min(q + u, p1 - 1));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = min(q + u, p1 - 1);
            if constexpr (PI) {
                const float4 *P = reinterpret_cast<const float4 *>(reinterpret_cast<const float2 *>(a.pi) + (int64_t)p * Rp);
#pragma unroll
                for (int v = 0; v < VP; ++v) {
                    const float4 y = __ldcs(P + v * G + lane);
                    ph[u][v] = make_float2(y.x, y.y);
                    pl[u][v] = make_float2(y.z, y.w);
                }
            } else {
#pragma unroll
                for (int k = 0; k < MAXK; ++k)
                    if (k < nm1) ii[u][k] = __ldg(a.idx[k] + p);
            }
        }
    };
    auto form_rows = [&](int q) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int v = 0; v < VP; ++v) {
                PairProduct y0, y1;
#pragma unroll
                for (int k = 0; k < MAXK; ++k) {
                    if (k < nm1) {
                        const float4 y =
                            __ldg(reinterpret_cast<const float4 *>(a.P[k] + (int64_t)ii[u][k] * Rp) + v * G + lane);
                        if (k == 0) {
                            y0.start(make_float2(y.x, y.z));
                            y1.start(make_float2(y.y, y.w));
                        } else {
                            y0.mul(make_float2(y.x, y.z));
                            y1.mul(make_float2(y.y, y.w));
                        }
                    }
                }
                const float2 e0 = y0.value(), e1 = y1.value();
                ph[u][v] = make_float2(e0.x, e1.x);
                pl[u][v] = make_float2(e0.y, e1.y);
            }
        }
    };
    load_step(q);
#pragma unroll 1
    for (int step = 1; __any_sync(full, q < qb); ++step) {
        if constexpr (!PI) form_rows(q);
        // the step takes m nonzeros, up to the next row start
        if (q < qb && q > qa && (starts & 1u)) {
            if (OP == OP_PHI) flush(false);
            first = false;
            cur = nxt;
            nxt = __ldg(a.nzrow + ++kcur + 1);
            load_b(cur);
        }
        int m = max(min(U, qb - q), 0);
        const uint32_t next = (starts >> 1) & ((1u << (U - 1)) - 1u);
        if (next) m = min(m, __ffs(next));

        // escapes (sign bit set: the largest bit patterns): out of the FP32
        // arithmetic, remembered in em (8 bits per nonzero)
        uint32_t top_bits = 0, em = 0, redo = 0;
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int v = 0; v < VP; ++v)
                top_bits = max(top_bits, max(__float_as_uint(ph[u][v].x), __float_as_uint(ph[u][v].y)));
        if (__builtin_expect((int)top_bits < 0, 0)) {
            // one above the pairs' window, or any where B is not safe, sends its
            // nonzero to FP64
            const bool unsafe = OP == OP_PHI && !(top < bmax);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                uint32_t e8 = 0, big = 0;
#pragma unroll
                for (int r = 0; r < RPL; ++r) {
                    float &h = r % 2 ? ph[u][r / 2].y : ph[u][r / 2].x;
                    if ((int)__float_as_uint(h) < 0) {
                        e8 |= 1u << r;
                        big = max(big, __float_as_uint(h));
                        h = 0.f;
                        (r % 2 ? pl[u][r / 2].y : pl[u][r / 2].x) = 0.f;
                    }
                }
                if (u < m) {
                    em |= e8 << (8 * u);
                    if (e8 && (unsafe || big >= kHighEscape)) redo |= 1u << u;
                }
            }
        }

        float2 s2[U];
#pragma unroll
        for (int u = 0; u < U; ++u) s2[u] = df_dot<VP>(bh, bl, ph[u], pl[u]);

        float vh[U], vl[U];
        double m_ll = 1.0;
        // one quotient (or model value) from a complete dot
        auto finish = [&](float2 tot, double xx, int u) -> float2 {
            const bool valid = u < m;
            if constexpr (OP == OP_PHI) {
                float xh, xl;
                df_cut(xx, kDfS + kDfV, xh, xl);
                const float2 v = df_divide(xh, xl, tot, eh, el);
                // NaN and infinite sums fail the comparisons
                const bool ok = tot.x < 0x1p100f && !df_bad_x(xx) && (xx == 0.0 || (v.x >= 0x1p-20f && v.x <= 0x1p50f));
                if (valid && !ok) redo |= 1u << u;
                return valid && ok ? v : make_float2(0.f, 0.f);
            } else {
                if (valid && !(tot.x >= 1.f && tot.x < 0x1p100f)) redo |= 1u << u;
                m_ll = scale_pow2(df_widen(tot.x) + df_widen(tot.y), -kDfS);
                return make_float2(0.f, 0.f);
            }
        };
        // log-likelihood: the dropped terms, below 2^-80 top each, are nothing beside
        // a model value of 2^-26 top or more (2^-47 of it with up to 128 columns)
        auto drop_ok = [&](float tot, int u) {
            if (((em >> (8 * u)) & 0xffu) && !(tot >= top * 0x1p-26f)) redo |= 1u << u;
        };
        if constexpr (G == 1) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (OP == OP_LL) drop_ok(s2[u].x, u);
                const float2 v = finish(s2[u], x[G > 1 ? 0 : u], u);
                vh[u] = v.x;
                vl[u] = v.y;
                if (OP == OP_LL && u < m && !((redo >> u) & 1u)) ll += x[G > 1 ? 0 : u] * log(m_ll);
            }
        } else {
            const float2 tot = group_reduce_scatter_df<G, U>(s2, lane, full);
            if (OP == OP_LL && __builtin_expect(__any_sync(full, em != 0u), 0)) {
#pragma unroll
                for (int u = 0; u < U; ++u) drop_ok(__shfl_sync(full, tot.x, gbase + u * LPU), u);
            }
            const float2 v = finish(tot, x[0], u_mine);
            if constexpr (OP == OP_PHI) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    vh[u] = __shfl_sync(full, v.x, gbase + u * LPU);
                    vl[u] = __shfl_sync(full, v.y, gbase + u * LPU);
                }
            }
        }
        // FP64, for the nonzeros outside the FP32 ranges (a warp-uniform branch)
        if (__builtin_expect(__any_sync(full, redo != 0u), 0)) {
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) redo |= __shfl_xor_sync(full, redo, o);
#pragma unroll 1
            for (int u = 0; u < U; ++u)
                if (__any_sync(full, (redo >> u) & 1u))
                    ll += pair_redo<NM1, RPL, G, OP, PI>(a, acc, nm1, K, min(q + u, p1 - 1), cur, lane, (redo >> u) & 1u);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if ((redo >> u) & 1u) {
                    vh[u] = vl[u] = 0.f;
                    em &= ~(0xffu << (8 * u));
                }
        }
        if constexpr (OP == OP_LL && G > 1) {
            if (u_mine < m && (lane % LPU) == 0 && !((redo >> u_mine) & 1u)) ll += x[0] * log(m_ll);
        }

        if constexpr (OP == OP_PHI) {
            if (__builtin_expect(em != 0u, 0)) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t e8 = (em >> (8 * u)) & 0xffu;
                    if (e8) {
                        const float sum = __uint_as_float(esc & ~0xffu) + vh[u] * 1.01f;
                        esc = ((__float_as_uint(sum) & ~0xffu) + 0x100u) | (esc & 0xffu) | e8;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float2 h2 = make_float2(vh[u], vh[u]), l2 = make_float2(vl[u], vl[u]);
#pragma unroll
                for (int v = 0; v < VP; ++v) df_fma2(h2, l2, ph[u][v], pl[u][v], S[v], C[v]);
            }
            if (step % (kDfSpill / U) == 0) {
#pragma unroll
                for (int k = 0; k < VP; ++k) {
                    double2 t = acc[k * G + lane];
                    t.x = fma(df_widen(S[k].x) + df_widen(C[k].x), unit, t.x);
                    t.y = fma(df_widen(S[k].y) + df_widen(C[k].y), unit, t.y);
                    acc[k * G + lane] = t;
                    S[k] = C[k] = make_float2(0.f, 0.f);
                }
            }
        }
        q += m;
        load_step(min(q, p1));
    }

    if constexpr (OP == OP_LL) {
        const double v = warp_sum(ll);
        if (wlane == 0) red[tid >> 5] = v;
        __syncthreads();
        if (tid == 0) {
            double sum = 0.0;
#pragma unroll
            for (int w = 0; w < THREADS / 32; ++w) sum += red[w];
            a.llpart[t] = sum;
        }
    } else {
        if (run) flush(true);
        if (!a.atomic) {
            // the row at the next tile's start if it goes on from this tile, else -1
            auto next_row_of = [&]() -> int32_t {
                return (p1 < a.nnz && !bit_at(p1))
                           ? __ldg(a.nzrow + __ldg(a.krow + min((int64_t)(t + 1) << a.ksh, (int64_t)a.ntab)))
                           : -1;
            };
            segmented_tail<double, OP, THREADS, NG, Rp, SP>(a, t, slot_val, slot_row, slot_fin, next_row_of, Bm, out,
                                                            tid >> 5, wlane, kkt);
            if (a.inner) publish_kkt<THREADS>(kkt, a.inner, red);
        }
    }
}

}  // namespace cpapr
