// Least-squares calibration of the Eq. 9 batch-time coefficients per model from a
// log of executed token batches (Sec. 4.1: the coefficients are calibrated from
// observed token-batch processing times).
//
// One kernel, one pass over the log: per model the normal equations G = sum x x^T,
// b = sum x t and the row count, as exact 128-bit integers (times in 2^-44 s fixed
// point); the last CTA to finish then solves every model's system (the paper's four
// regressors, with F1 + F2 as the token count, or the five features), scaled by
// powers of two so that its diagonal is near 1 (exact, and it restores the
// conditioning the raw feature magnitudes take away), by an LDL^T factorization,
// and clears the sums for the next call.
#include "lr_internal.cuh"

#include <algorithm>

namespace lr {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// Packed upper triangle of a 5x5 symmetric matrix.
__device__ __forceinline__ int tri(int a, int b) {
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    return lo * kCalCols - lo * (lo - 1) / 2 + (hi - lo);
}

// A 128-bit unsigned sum kept as (lo, hi) 64-bit halves.
struct U128 {
    unsigned long long lo, hi;
};
__device__ __forceinline__ void add128(U128 &a, unsigned long long lo, unsigned long long hi) {
    const unsigned long long s = a.lo + lo;
    a.hi += hi + (s < lo ? 1ull : 0ull);
    a.lo = s;
}
// Atomic version: the carry of this addition into the low word follows from the old
// value the atomic returns, so the pair is right once every addition has landed.
__device__ __forceinline__ void atomic_add128(unsigned long long *p, unsigned long long lo, unsigned long long hi) {
    if (lo == 0ull && hi == 0ull) return;
    const unsigned long long old = atomicAdd(p, lo);
    const unsigned long long c = (old + lo < old) ? 1ull : 0ull;
    if (hi + c != 0ull) atomicAdd(p + 1, hi + c);
}

__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred P;\n mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n selp.u32 %0, 1, 0, P;\n}"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

constexpr unsigned long long kTimeMaxBits = 0x4120000000000000ull;  // the bits of 2^19 (kCalTimeMax)

// floor(t * 2^44) for 0 <= t < 2^19 given the bits of t: the IEEE-754 value of t is
// m * 2^(E - 1075) with the 53-bit significand m, so the product is m shifted left by
// E - 1031 bits, or right (dropping what lies below 2^-44 s) when that is negative.
// Integer operations only.
__device__ __forceinline__ unsigned long long fixed_time(unsigned long long bits) {
    const int E = (int)(bits >> 52);
    const unsigned long long m = (bits & ((1ull << 52) - 1)) | (E != 0 ? (1ull << 52) : 0ull);
    const int sh = max(E, 1) - 1031;
    return sh >= 0 ? m << sh : m >> min(-sh, 63);  // sh <= 10 below 2^19 s
}

// acc += a * b with the 64-bit product of two 32-bit factors, one instruction
__device__ __forceinline__ void mad64(unsigned long long &acc, uint32_t a, uint32_t b) {
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// v * 2^e2 as the nearest double (ties to even) for a 128-bit unsigned v of leading bit p
// (-1: zero), assuming the result is a normal number: v shifted until its leading bit is
// the highest, of which the top 53 bits are the significand and the rest rounds it.
// Integer operations only, and none of them in a branch.
__device__ __forceinline__ int lead_bit(const U128 &v) {
    return v.hi ? 127 - __clzll((long long)v.hi) : 63 - __clzll((long long)v.lo);  // (clz of 0 is 64)
}
__device__ __forceinline__ double u128_to_double(const U128 &v, int p, int e2) {
    const int up = 127 - max(p, 0);  // 0 .. 127
    const bool far = up >= 64;
    const unsigned long long h0 = far ? v.lo : v.hi, l0 = far ? 0ull : v.lo;
    const int sh = up & 63;
    const unsigned long long h = (h0 << sh) | ((l0 >> 1) >> (63 - sh)), l = l0 << sh;
    const unsigned long long q = h >> 11, dropped = (h & 2047ull) | (l != 0ull ? 1ull : 0ull);
    // (a carry out of the significand moves the exponent, as it should)
    const unsigned long long up1 = dropped > 1024ull || (dropped == 1024ull && (q & 1ull)) ? 1ull : 0ull;
    const unsigned long long bits = ((unsigned long long)(p + e2 + 1022) << 52) + q + up1;
    return p < 0 ? 0.0 : __longlong_as_double((long long)bits);
}

// The solve of every model's system, on the last CTA: regressors, power-of-two Jacobi
// scaling, LDL^T, unscaling.  D regressors: 4 (the paper's form, F1 + F2 as one token
// count) or 5; with four, a unit fifth regressor uncoupled from the others keeps one
// code path (its weight is 0).  The regressor sums are formed exactly in 128 bits; each
// enters fp64 once, already scaled by the powers of two that bring the diagonal into
// [1, 4) (regressor p scaled by 2^-h_p with h_p half the leading-bit position of G_pp),
// so the conditioning that the raw feature magnitudes take away is restored without a
// rounding.  The solve is a chain of dependent integer and fp64 work on one CTA, and the
// fp64 pipe is narrow on this part: a warp forms the 20 scaled entries of a model,
// a lane each (integer pipes only), then a warp factors five models' systems with
// straight-line code in registers, whose only fp64 divisions are the pivot reciprocals.
constexpr int kCalSolveWords = 24;  // per model in shared memory: 15 + 5 scaled entries, 5 exponents

__device__ __forceinline__ void calib_lohi(bool four, int p, int &lo, int &hi) {  // regressor p: features lo..hi
    lo = four ? (p == 0 ? 0 : p == 1 ? 1 : p + 1) : p;
    hi = four ? (p == 0 ? 0 : p == 1 ? 2 : p + 1) : p;
}

// Entry e of a model's system from its exact sums S [kCalAcc] (U128 pairs): e < 15 is
// G_pq of the packed lower triangle, e = 15 + p is b_p.  At most two features a regressor:
// four sums, taken without a branch.
__device__ __forceinline__ U128 calib_gsum(const unsigned long long *S, bool four, int e, int &p, int &q) {
    p = e < 15 ? (e >= 1) + (e >= 3) + (e >= 6) + (e >= 10) : e - 15;
    q = e < 15 ? e - p * (p + 1) / 2 : 0;
    int pl, ph, ql, qh;
    calib_lohi(four, p, pl, ph);
    calib_lohi(four, q, ql, qh);
    const bool unit = four && (p == 4 || (e < 15 && q == 4));  // the unit regressor
    U128 g{unit && e == 14 ? 1ull : 0ull, 0ull};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int a = i & 1 ? ph : pl, c = i & 2 ? qh : ql;
        const bool on = !unit && (!(i & 1) || ph > pl) && (e < 15 ? !(i & 2) || qh > ql : !(i & 2));
        const int k = on ? (e < 15 ? tri(a, c) : 15 + a) : 0;
        const unsigned long long lo = S[2 * k], hi = S[2 * k + 1];
        add128(g, on ? lo : 0ull, on ? hi : 0ull);
    }
    return g;
}

// A model's scaled system, by one warp: entry e of W on lane e < 20 (the packed lower
// triangle of A, then b), the scale exponents h_p from the diagonal's lanes.  (The entries'
// own regressor sums serve for the exponents: an extra pass and a CTA barrier less.  With
// the conversion and the sums free of branches, 4M rows 42.2 -> 40.7 us, 20,000 14.3 -> 13.0.)
__device__ void calib_entries(int m, bool four, const unsigned long long *S, double *W) {
    const int lane = threadIdx.x & 31;
    int p, q;
    const U128 g = calib_gsum(S + (size_t)m * kCalAcc * 2, four, min(lane, 19), p, q);
    const int lead = lead_bit(g), h = max(lead, 0) >> 1;
    const int hp = __shfl_sync(kFull, h, p * (p + 3) / 2), hq = __shfl_sync(kFull, h, q * (q + 3) / 2);
    double *Wm = W + (size_t)m * kCalSolveWords;
    if (lane < 20) Wm[lane] = u128_to_double(g, lead, -(hp + (lane < 15 ? hq : 44)));  // b carries 2^-44 s
    if (lane >= 15 && lane < 20) reinterpret_cast<int *>(Wm + 20)[p] = hp;
}

// On this part the SM's fp64 unit is narrow: each fp64 instruction of a warp costs
// tens of cycles whatever the active lanes, so the solve keeps its fp64 instructions
// few and does comparisons, clamps and power-of-two scalings on the bits.

// 1/x for a positive normal double: the fp32 reciprocal of its significand truncated to
// 24 bits (built from the bits, relative error below 2^-23), rescaled by the exponent,
// then one Newton-Raphson step r <- r (2 - x r), which squares the error (2^-46).
__device__ __forceinline__ double recip_pos(double x) {
    const unsigned long long bx = (unsigned long long)__double_as_longlong(x);
    const long long e = (long long)((bx >> 52) & 0x7ff) - 1023;
    const float m = __int_as_float((int)((127u << 23) | (unsigned)((bx >> 29) & 0x7fffffu)));  // [1, 2)
    const unsigned rb = (unsigned)__float_as_int(__frcp_rn(m));                                  // (1/2, 1]
    const long long re = (long long)((rb >> 23) & 0xff) - 127 - e;
    const double r = __longlong_as_double((long long)(((unsigned long long)(re + 1023) << 52) |
                                                      ((unsigned long long)(rb & 0x7fffffu) << 29)));
    return __fma_rn(r, __fma_rn(-x, r, 1.0), r);
}

// v * 2^-h for a finite v (0 stays 0; the results here stay normal): the exponent field
__device__ __forceinline__ double scale_pow2(double v, int h) {
    const long long bv = __double_as_longlong(v);
    return (bv & 0x7ff0000000000000LL) ? __longlong_as_double(bv - ((long long)h << 52)) : v;
}

// The scaled 5x5 systems of models m0 .. m0 + 4 by LDL^T, a warp together: six lanes a
// model, a row of the packed triangle each, the right-hand side being the sixth (its
// elimination is the forward substitution).  An fp64 instruction of a warp holds the narrow
// unit for some 64 cycles whatever its lanes, and this part is bound by them: 35 here, 65
// with a lane a model (4M rows 40.7 -> 39.4 us, 20,000 13.0 -> 12.1).
__device__ void calib_factor(int m0, int M, int D, const unsigned long long *S, const double *W, double *coef) {
    const int lane = threadIdx.x & 31, gm = min(lane / 6, 4), r = lane - 6 * gm, l0 = 6 * gm;
    const int m = min(m0 + gm, M - 1);
    const double *Wm = W + (size_t)m * kCalSolveWords;
    const int *h = reinterpret_cast<const int *>(Wm + 20);
    const unsigned long long *cnt = S + ((size_t)m * kCalAcc + 20) * 2;
    bool ok = cnt[1] != 0ull || cnt[0] >= (unsigned long long)D;
    double A[5], L[5], w[5];  // this row's LD (as eliminated so far) and L
#pragma unroll
    for (int q = 0; q < 5; ++q) A[q] = q <= r && r <= 5 ? Wm[r * (r + 1) / 2 + q] : 0.0;
    constexpr long long kMinPivot = 0x3d3c25c268497682LL;  // the bits of 1e-13
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const double v = __shfl_sync(kFull, A[k], l0 + k);  // the pivot: row k's diagonal
        // v > 1e-13 on the bits (a positive double orders as its bits; NaN fails)
        const long long bv = __double_as_longlong(v);
        const bool piv = bv > kMinPivot && bv < 0x7ff0000000000000LL;
        ok = ok && piv;  // rank-deficient design (or a zero G_pp)
        L[k] = A[k] * (piv ? recip_pos(v) : 0.0);
#pragma unroll
        for (int q = k + 1; q < 5; ++q) A[q] = __fma_rn(-A[k], __shfl_sync(kFull, L[k], l0 + q), A[q]);
    }
    // back substitution from the right-hand side's row, on every lane alike
#pragma unroll
    for (int p = 4; p >= 0; --p) {
        double v = __shfl_sync(kFull, L[p], l0 + 5);
#pragma unroll
        for (int k = p + 1; k < 5; ++k) v = __fma_rn(-__shfl_sync(kFull, L[p], l0 + k), w[k], v);
        w[p] = v;
    }
    if (r != 0 || lane >= 30 || m0 + gm >= M) return;
    // the five coefficients, unscaled by 2^-h_p: with four regressors the token slope
    // serves prefill and decode
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    const bool four = D == 4;
    double out[5];
    out[0] = scale_pow2(w[0], h[0]);
    out[1] = scale_pow2(w[1], h[1]);
    out[2] = four ? out[1] : scale_pow2(w[2], h[2]);
    out[3] = four ? scale_pow2(w[2], h[2]) : scale_pow2(w[3], h[3]);
    out[4] = four ? scale_pow2(w[3], h[3]) : scale_pow2(w[4], h[4]);
#pragma unroll
    for (int k = 0; k < 5; ++k) coef[(size_t)m * 5 + k] = ok ? out[k] : nan;
}

// The share of warp `warp` of a mixed tile's rows: models [x, y), rank z among its w warps.
// c: the rows of models 4 lane .. 4 lane + 3, e0 those of the models before them, T all
// rows (at least one).  A call of its own: it runs about once a slice, and inlined it takes
// registers from the sums.
__device__ __noinline__ int4 calib_share(int4 c, int e0, int T, int M, int warp) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int e1 = e0 + c.x, e2 = e1 + c.y, e3 = e2 + c.z;
    int4 out;
    const int cc[4] = {c.x, c.y, c.z, c.w}, ee[4] = {e0, e1, e2, e3};
    int live = 0, rank = 0;  // models with rows, and those before this lane's
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const unsigned b = __ballot_sync(kFull, cc[i] > 0);
        live += __popc(b);
        rank += __popc(b & lt);
    }
    int lo = kCalMaxModels, hi = 0, r0 = 0, n0 = 0;
    const int spare = kCalConsumerWarps - live;
    if (spare >= 0) {
        // a warp each, the spare ones by the rows; a model without rows goes
        // with the one before it (the first ones with the first)
        int next = M;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (cc[i] == 0) continue;
            const int f = rank + ee[i] * spare / T, z = rank + 1 + (ee[i] + cc[i]) * spare / T;
            if (f <= warp && warp < z) {
                lo = rank == 0 ? 0 : 4 * lane + i;
                hi = 4 * lane + i;
                r0 = warp - f;
                n0 = z - f;
            }
            ++rank;
        }
        lo = __reduce_min_sync(kFull, lo);
        hi = __reduce_max_sync(kFull, hi);
#pragma unroll
        for (int i = 3; i >= 0; --i)
            if (cc[i] > 0 && 4 * lane + i > hi) next = 4 * lane + i;
        out.x = lo;
        out.y = __reduce_min_sync(kFull, next);
        out.z = __reduce_max_sync(kFull, r0);
        out.w = __reduce_max_sync(kFull, n0);
    } else {
        // more models than warps: each model whole, to the warp its middle row falls to
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int w = min(kCalConsumerWarps - 1, (2 * ee[i] + cc[i]) * kCalConsumerWarps / (2 * T));
            if (w == warp && 4 * lane + i < M) {
                lo = min(lo, 4 * lane + i);
                hi = max(hi, 4 * lane + i + 1);
            }
        }
        out.x = __reduce_min_sync(kFull, lo);
        out.y = __reduce_max_sync(kFull, hi);
        out.z = 0;
        out.w = 1;
    }
    return out;
}

// The pass over the log.  Exact integer sums: features below 2^32 make every product
// of two of them exact in 64 bits, and a time below 2^19 s becomes a 2^-44 s fixed-
// point integer below 2^63, so that feature x time fits 96 bits.  Rows whose features
// are below 2^26 and whose time is below 2^8 s (the usual case) add their 15 products,
// and the products of each feature with the two 26-bit halves of the time, into plain
// 64-bit sums in registers: every product is below 2^52, so a lane's sums of up to 128
// rows stay below 2^59 and a warp's below 2^64.  The warp flushes them into the
// 128-bit sums in shared memory when a lane's model changes (rows grouped by model are
// the usual case), before 128 rows and at the end: a reduce-scatter over the 32 lanes
// (five rounds of exchanging half of the remaining values with the partner lane) leaves
// lane k with the warp total of sum k, which it adds to the model's shared sum -- one
// shared atomic per sum, model and warp.  The warp decides together whether to flush:
// one vote per two rows a lane, one per row where those fail it.  Other rows
// add to the shared 128-bit sums directly.  Nothing uses the fp64 pipe.
//
// TMA: each CTA streams a contiguous slice of the log through a ring of `nst`
// shared-memory tiles of kCalTile rows (features, times, model ids), each filled by
// bulk copies that complete on its mbarrier.  Without it (inputs not 16-byte aligned)
// rows are read directly.
template <bool TMA>
__global__ void __launch_bounds__(kCalThreads, 1) k_calibrate(long long N, const long long *F, const int32_t *model,
                                                              const double *time, int M, int D, int nst,
                                                              unsigned long long *acc, double *coef, DevCtl *ctl) {
    extern __shared__ __align__(16) unsigned char cal_smem[];
    unsigned long long *sacc = reinterpret_cast<unsigned long long *>(cal_smem);  // [M][kCalAcc][2] (lo, hi)
    // the flushes' totals in carry-save form: [M][26][2], sum k = w0 + 2^32 w1, each flush
    // adding the low and the high 32 bits of its (below 2^64) total with a reduction that
    // returns nothing (no carry to wait for)
    unsigned long long *scs = sacc + (size_t)M * kCalAcc * 2;
    const int lane = threadIdx.x & 31;
    unsigned char *stages = cal_smem + cal_sums_bytes(M);
    __shared__ __align__(8) unsigned long long s_mbar[kCalStagesMax];
    __shared__ int s_last, s_work;
    __shared__ long long s_none[kCalCols + 1];  // a row that adds nothing: constant 1, then zeros
    unsigned int *done = reinterpret_cast<unsigned int *>(acc + 2 * (size_t)M * kCalAcc);
    for (int i = threadIdx.x; i < M * (kCalAcc + kCalFlushSums) * 2; i += blockDim.x) sacc[i] = 0ull;
    if (threadIdx.x < kCalCols + 1) s_none[threadIdx.x] = threadIdx.x == 0 ? 1 : 0;
    if (threadIdx.x == 0) s_work = 0;
    unsigned long long g[15], bl[5], bh[5];  // 64-bit sums since the last flush
    int nfast = 0, cur = -1;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 15; ++k) g[k] = 0ull;
#pragma unroll
    for (int q = 0; q < 5; ++q) bl[q] = bh[q] = 0ull;
    auto flush = [&]() {  // every lane of the warp calls it
        const int key = nfast > 0 ? cur : -1;
        unsigned pend = __ballot_sync(kFull, key >= 0);
        while (pend) {
            const int mk = __shfl_sync(kFull, key, __ffs(pend) - 1);
            const bool mine = key == mk;
            // sums 0..14: G; 15..19: x t_lo halves of b; 20..24: x t_hi halves (weight
            // 2^26); 25: the row count
            unsigned long long a[32];
#pragma unroll
            for (int k = 0; k < 15; ++k) a[k] = mine ? g[k] : 0ull;
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                a[15 + q] = mine ? bl[q] : 0ull;
                a[20 + q] = mine ? bh[q] : 0ull;
            }
            a[25] = mine ? (unsigned long long)nfast : 0ull;
#pragma unroll
            for (int k = 26; k < 32; ++k) a[k] = 0ull;
#pragma unroll
            for (int w = 16; w >= 1; w >>= 1) {  // keep the half of a[0..2w) that this lane's bit w selects
                const bool up = (lane & w) != 0;
#pragma unroll
                for (int j = 0; j < w; ++j) {
                    const unsigned long long give = up ? a[j] : a[j + w];
                    a[j] = (up ? a[j + w] : a[j]) + __shfl_xor_sync(kFull, give, w);
                }
            }
            if (lane < kCalFlushSums) {  // a[0]: the warp's total of sum `lane`
                const uint32_t sa = (uint32_t)__cvta_generic_to_shared(scs + ((size_t)mk * kCalFlushSums + lane) * 2);
                asm volatile("red.shared.add.u64 [%0], %1;" ::"r"(sa), "l"(a[0] & 0xffffffffull) : "memory");
                asm volatile("red.shared.add.u64 [%0], %1;" ::"r"(sa + 8u), "l"(a[0] >> 32) : "memory");
            }
            pend &= ~__ballot_sync(kFull, mine);
        }
#pragma unroll
        for (int k = 0; k < 15; ++k) g[k] = 0ull;
#pragma unroll
        for (int q = 0; q < 5; ++q) bl[q] = bh[q] = 0ull;
        nfast = 0;
    };
    // One row per lane, the whole warp together (`in` false: no row).  The warp first
    // flushes if a lane's model changes or its sums reach 128 rows.
    auto row = [&](bool in, int m, double t, const long long *f) {
        long long v[kCalCols];
        long long any = 0;
        unsigned long long tb = 0ull;
        if (in) {
#pragma unroll
            for (int k = 0; k < kCalCols; ++k) {
                v[k] = f[k];
                any |= v[k];
            }
            tb = (unsigned long long)__double_as_longlong(t);
        }
        // 0 <= t < 2^19 on the bits (-0 counts as 0; NaN fails), every feature in
        // [0, 2^32): no bit of any of them at 2^32 or above (nor the sign)
        const unsigned long long tmag = tb & 0x7fffffffffffffffull;
        const bool tok = (tb >> 63) == 0ull ? tb < kTimeMaxBits : tmag == 0ull;
        const bool ok = in && m >= 0 && m < M && tok && (any >> 32) == 0;
        bad |= in && !ok;
        if (__any_sync(kFull, (ok && m != cur) || nfast >= kCalFlushRows)) flush();
        if (!ok) return;
        cur = m;
        const unsigned long long tf = fixed_time(tmag);
        uint32_t x[kCalCols];
#pragma unroll
        for (int k = 0; k < kCalCols; ++k) x[k] = (uint32_t)v[k];
        if ((any >> 26) == 0 && (tf >> 52) == 0ull) {
            const uint32_t tl = (uint32_t)tf & ((1u << 26) - 1), th = (uint32_t)(tf >> 26);
            // Eq. 9's constant feature is 1 (the usual row): its products are additions
            const int q0 = x[0] == 1u ? 1 : 0;
            if (q0) {
                g[tri(0, 0)] += 1ull;
#pragma unroll
                for (int r = 1; r < kCalCols; ++r) g[tri(0, r)] += x[r];
                bl[0] += tl;
                bh[0] += th;
            }
#pragma unroll
            for (int q = 0; q < kCalCols; ++q) {
                if (q == 0 && q0) continue;
#pragma unroll
                for (int r = q; r < kCalCols; ++r) mad64(g[tri(q, r)], x[q], x[r]);
                mad64(bl[q], x[q], tl);
                mad64(bh[q], x[q], th);
            }
            ++nfast;
            return;
        }
        // rows with larger values add exactly into the shared 128-bit sums
        unsigned long long *s = sacc + (size_t)m * kCalAcc * 2;
        const uint32_t tlo = (uint32_t)tf, thi = (uint32_t)(tf >> 32);
#pragma unroll
        for (int q = 0; q < kCalCols; ++q) {
#pragma unroll
            for (int r = q; r < kCalCols; ++r) atomic_add128(s + 2 * tri(q, r), (unsigned long long)x[q] * x[r], 0ull);
            // x * t = x * t_lo + (x * t_hi) * 2^32, below 2^96
            const unsigned long long p1 = (unsigned long long)x[q] * thi;
            U128 w{(unsigned long long)x[q] * tlo, 0ull};
            add128(w, p1 << 32, p1 >> 32);
            atomic_add128(s + 2 * (15 + q), w.lo, w.hi);
        }
        atomic_add128(s + 40, 1ull, 0ull);
    };
    // Two staged rows a lane at once, when one vote finds every lane's rows of its current
    // model, with a constant feature of 1, features below 2^26 and a time in [0, 2^8) s, and
    // its sums far enough from their limit (false: nothing was added).  The pass waits for
    // memory and for the instructions it issues alike, so this path has no branch inside:
    // the constant's products of the two rows are added as one 32-bit sum each, and a lane
    // without a row reads the row of zeros at s_none (its constant is 1, and not counted).
    // 4M rows of 8 models: 51.3 -> 42.2 us a call.
    auto both = [&](auto masked, bool in0, bool in1, int m0, int m1, const long long *f0, const long long *f1, const double *t0,
                    const double *t1) {
        constexpr bool kMask = decltype(masked)::value;
        uint2 u[kCalCols], v[kCalCols];
        uint32_t lo = 0u, hi = 0u;
#pragma unroll
        for (int k = 0; k < kCalCols; ++k) {
            u[k] = reinterpret_cast<const uint2 *>(!kMask || in0 ? f0 : s_none)[k];
            v[k] = reinterpret_cast<const uint2 *>(!kMask || in1 ? f1 : s_none)[k];
            lo |= u[k].x | v[k].x;
            hi |= u[k].y | v[k].y;
        }
        const uint2 ta = *reinterpret_cast<const uint2 *>(!kMask || in0 ? (const void *)t0 : (const void *)(s_none + 1));
        const uint2 tb = *reinterpret_cast<const uint2 *>(!kMask || in1 ? (const void *)t1 : (const void *)(s_none + 1));
        m0 = !kMask || in0 ? m0 : cur;
        m1 = !kMask || in1 ? m1 : cur;
        const int two = kMask ? (int)in0 + (int)in1 : 2;
        constexpr uint32_t k256s = 0x40700000u;  // the high word of 2^8; sign or NaN is above it
        const int c = nfast == 0 ? m0 : cur;  // nothing summed yet: any model will do
        const bool fast = ((unsigned)c < (unsigned)M) & (m0 == c) & (m1 == c) & (nfast <= kCalFlushRows - 2) & (hi == 0u) &
                          (lo < (1u << 26)) & (u[0].x == 1u) & (v[0].x == 1u) & (max(ta.y, tb.y) < k256s);
        if (!__all_sync(kFull, fast)) return false;
        uint32_t tl[2], th[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            // floor(t * 2^44) as fixed_time forms it; below 2^8 s it is a right shift (a
            // subnormal's implied bit falls out with the rest)
            const uint2 t = r ? tb : ta;
            const unsigned long long mant = ((unsigned long long)((t.y & 0xfffffu) | 0x100000u) << 32) | t.x;
            const unsigned long long tf = mant >> min(1031u - (t.y >> 20), 63u);
            tl[r] = (uint32_t)tf & ((1u << 26) - 1);
            th[r] = (uint32_t)(tf >> 26);
        }
        g[0] += (unsigned long long)two;
#pragma unroll
        for (int r = 1; r < kCalCols; ++r) g[tri(0, r)] += u[r].x + v[r].x;
        bl[0] += tl[0] + tl[1];
        bh[0] += th[0] + th[1];
#pragma unroll
        for (int q = 1; q < kCalCols; ++q) {
#pragma unroll
            for (int r = q; r < kCalCols; ++r) {
                mad64(g[tri(q, r)], u[q].x, u[r].x);
                mad64(g[tri(q, r)], v[q].x, v[r].x);
            }
            mad64(bl[q], u[q].x, tl[0]);
            mad64(bh[q], u[q].x, th[0]);
            mad64(bl[q], v[q].x, tl[1]);
            mad64(bh[q], v[q].x, th[1]);
        }
        nfast += two;
        cur = c;
        return true;
    };
    // this CTA's contiguous slice, starting on a tile boundary
    const long long per = ((N + gridDim.x - 1) / gridDim.x + kCalTile - 1) / kCalTile * kCalTile;
    const long long c0 = min(N, (long long)blockIdx.x * per), c1 = min(N, c0 + per);
    long long rest = c0;
    bool ok = true;
    // per stage: `full` completes when its tile has landed, `empty` when every consumer
    // warp has read it
    __shared__ __align__(8) unsigned long long s_empty[kCalStagesMax];
    if (TMA && threadIdx.x == 0) {
        for (int st = 0; st < nst; ++st) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(&s_mbar[st]))
                         : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(&s_empty[st])),
                         "r"(kCalConsumerWarps)
                         : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();  // the sums are zero and the barriers ready
    chain_wait();
    if (TMA && c0 < c1) {
        // The last warp produces (its lane 0 issues each tile once the consumers have
        // released the stage), the others consume at their own pace: no CTA barrier in
        // the loop, so a warp that finishes a tile early starts the next one.
        const int ntiles = (int)((c1 - c0 + kCalTile - 1) / kCalTile);  // the last may be short
        constexpr uint32_t kFeat = kCalTile * kCalCols * 8, kTime = kCalTile * 8, kModel = kCalTile * 4;
        constexpr uint32_t kStage = kFeat + kTime + kModel;
        __shared__ __align__(16) int s_cnt[2][kCalMaxModels];  // the tile's rows per model
        __shared__ uint16_t s_list[kCalTile];                  // a mixed tile's rows in model order
        __shared__ __align__(16) int s_start[kCalMaxModels + 4];  // where each model's rows start in it, and their end
        __shared__ int4 s_share[kCalConsumerWarps];            // each warp's share of them (calib_share)
        __shared__ int s_redo[2];
        const int warp = threadIdx.x >> 5;
        bool failed = false;
        if (warp == kCalConsumerWarps) {
            if (lane == 0) {
                unsigned long long once;
                asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(once));
                int issued = 0;
                for (int k = 0; k < ntiles; ++k) {
                    const int st = k % nst, r = k / nst;
                    if (r > 0 && !mbar_wait((uint32_t)__cvta_generic_to_shared(&s_empty[st]), (uint32_t)((r - 1) & 1))) {
                        failed = true;  // a consumer never released the stage: stop issuing
                        break;
                    }
                    const long long r0 = c0 + (long long)k * kCalTile;
                    const uint32_t mb = (uint32_t)__cvta_generic_to_shared(&s_mbar[st]);
                    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(stages + (size_t)st * kStage);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    // bulk copies take whole 16 bytes: up to three rows at the log's end go by hand
                    const int nrow = (int)min((long long)kCalTile, c1 - r0);
                    const uint32_t n4 = (uint32_t)nrow & ~3u;
                    unsigned char *sb = stages + (size_t)st * kStage;
                    for (int j = (int)n4; j < nrow; ++j) {
                        for (int q = 0; q < kCalCols; ++q)
                            reinterpret_cast<long long *>(sb)[j * kCalCols + q] = F[(r0 + j) * kCalCols + q];
                        reinterpret_cast<double *>(sb + kFeat)[j] = time[r0 + j];
                        reinterpret_cast<int32_t *>(sb + kFeat + kTime)[j] = model[r0 + j];
                    }
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb),
                                 "r"(n4 * (kStage / kCalTile))
                                 : "memory");
                    issued = k + 1;
                    if (n4 == 0u) break;  // (the last tile, nothing to copy)
                    // the log is read once: first out of L2, ahead of the code and the sums
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, "
                        "[%3], %4;" ::"r"(dst),
                        "l"(F + r0 * kCalCols), "r"(n4 * kCalCols * 8u), "r"(mb), "l"(once)
                        : "memory");
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, "
                        "[%3], %4;" ::"r"(dst + kFeat),
                        "l"(time + r0), "r"(n4 * 8u), "r"(mb), "l"(once)
                        : "memory");
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, "
                        "[%3], %4;" ::"r"(dst + kFeat + kTime),
                        "l"(model + r0), "r"(n4 * 4u), "r"(mb), "l"(once)
                        : "memory");
                }
                // every copy has landed before the CTA moves on: only the last nst issued
                // tiles can still be in flight (bounded waits)
                for (int q = max(0, issued - nst); q < issued; ++q)
                    failed |= !mbar_wait((uint32_t)__cvta_generic_to_shared(&s_mbar[q % nst]), (uint32_t)((q / nst) & 1));
            }
        } else {
            // A log whose rows are in the order they ran mixes the models, and a lane that
            // meets another model has its warp flush, once for each model its lanes hold.  Where
            // that is much, each tile's rows are first listed by model (a counting sort of their
            // indexes; the sums are exact, so any order will do), and each warp takes the rows of
            // the models it owns: the warps are dealt out by the models' rows in a tile, again
            // when a warp's share grows fourfold.  2M rows of 8 / 12 / 40 models in random order:
            // 260 / 360 / 679 us with flushes alone, 56 / 57 / 145 this way.
            // The slice's first tile decides.  `per` is the flushes a warp would make in a tile,
            // about a microsecond each: for each of its two rows a lane as many as the models of
            // the warp's rows, if a lane's two rows differ (rows that take turns, so that each
            // lane meets one model, cost none but the last), and those of the end.  Listing costs
            // two to three, or, with more models than warps, flushes as well, of every model in
            // the tile by some warp, and the more so where one model has most rows and the others
            // crowd the last warps.  (The slowest slice sets the time, so the lines keep clear of
            // what chance moves a tile by.)  2M rows, flushes / listed: 2 models in runs of 16 rows
            // (per 2.3) 76 / 50 us, 8 in runs of 32 (2.0) 66 / 49, 12 in random runs of 64 (1.9)
            // 65 / 106; 40 models in turn (0.1) 58 / 139, runs of 8 in turn (8) 154 / 121, random runs
            // of 16 (4) 98 / 159; 64 and 128 models in runs of 8 and 4 (8, 16) 157 / 247, 279 /
            // 445, of 2 (32) 491 / 206, 501 / 359; skewed counts of 16 / 40 / 128 models (16 to
            // 18) 276 / 179, 308 / 419, 330 / 802.
            auto consumers = [&]() {
                __syncwarp();
                asm volatile("bar.sync 1, %0;" ::"n"(kCalConsumerWarps * 32) : "memory");
            };
            const unsigned lt = (1u << lane) - 1u;
            // the ring's stage of the next tile, its phase, and the rows from that tile on
            int st = 0, left = (int)(c1 - c0);
            uint32_t ph = 0u;
            auto landed = [&]() { return mbar_wait((uint32_t)__cvta_generic_to_shared(&s_mbar[st]), ph); };
            auto release = [&]() {  // this warp is done with the stage
                __syncwarp();
                if (lane == 0 && !failed)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(&s_empty[st]))
                                 : "memory");
                left -= kCalTile;
                if (++st == nst) {
                    st = 0;
                    ph ^= 1u;
                }
            };
            const int ja = threadIdx.x, jb = threadIdx.x + kCalConsumerWarps * 32;
            if (threadIdx.x < kCalMaxModels) s_cnt[0][threadIdx.x] = s_cnt[1][threadIdx.x] = 0;
            if (threadIdx.x < 2) s_redo[threadIdx.x] = 1;
            // (a tile that never lands ends the sums but not the barriers; the producer's waits
            // are bounded too)
            failed = !__all_sync(kFull, landed());
            const int32_t *m0 = reinterpret_cast<const int32_t *>(stages + kFeat + kTime);
            const bool va = !failed && ja < left;
            const int xa = va ? m0[ja] : -1, xb = va && jb < left ? m0[jb] : xa;
            const unsigned same = __match_any_sync(kFull, xa);
            const int kinds = __popc(__ballot_sync(kFull, va && (same & lt) == 0u));
            const bool moves = __any_sync(kFull, xa != xb);
            if (lane == 0) atomicAdd(&s_work, moves ? 2 * ntiles * kinds : kinds);
            consumers();
            const float per = (float)s_work / (float)(min(kCalConsumerWarps, (left + 31) / 32) * ntiles);
            bool mixed = per >= (M > kCalConsumerWarps ? 4.f : 2.5f);
            if (mixed && M > kCalConsumerWarps) {
                if (va && xa >= 0 && xa < M) atomicAdd(&s_cnt[1][xa], 1);
                if (va && jb < left && xb >= 0 && xb < M) atomicAdd(&s_cnt[1][xb], 1);
                consumers();
                const int4 c = reinterpret_cast<const int4 *>(s_cnt[1])[lane];  // (cleared with the first tile)
                const int n = __reduce_add_sync(kFull, (c.x > 0) + (c.y > 0) + (c.z > 0) + (c.w > 0));
                const int most = __reduce_max_sync(kFull, max(max(c.x, c.y), max(c.z, c.w)));
                const bool skewed = most * kCalConsumerWarps > 4 * min(left, kCalTile);
                if (n > kCalConsumerWarps) mixed = per >= (0.7f + 0.18f * (float)n) * (skewed ? 3.5f : 1.f);
            }
            if (!mixed) {
                for (; left > 0 && !failed; release()) {
                    if (!landed()) {
                        failed = true;
                        break;
                    }
                    const unsigned char *sb = stages + (size_t)st * kStage;
                    const long long *sf = reinterpret_cast<const long long *>(sb);
                    const double *stt = reinterpret_cast<const double *>(sb + kFeat);
                    const int32_t *sm = reinterpret_cast<const int32_t *>(sb + kFeat + kTime);
                    if (left < kCalTile || !both(std::false_type{}, true, true, sm[ja], sm[jb], sf + ja * kCalCols,
                                                 sf + jb * kCalCols, stt + ja, stt + jb)) {
#pragma unroll 1
                        for (int j = ja; j < ja + 2 * (jb - ja); j += jb - ja)
                            row(j < left, sm[j], stt[j], sf + j * kCalCols);
                    }
                }
            } else {
                for (int k = 0; k < ntiles; ++k) {
                    failed = failed || !__all_sync(kFull, landed());
                    const int nrow = failed ? 0 : left;
                    const unsigned char *sb = stages + (size_t)st * kStage;
                    const long long *sf = reinterpret_cast<const long long *>(sb);
                    const double *stt = reinterpret_cast<const double *>(sb + kFeat);
                    const int32_t *sm = reinterpret_cast<const int32_t *>(sb + kFeat + kTime);
                    int *cnt = s_cnt[k & 1];
                    int mm[2], pos[2];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int j = q ? jb : ja;
                        const int m = j < nrow ? sm[j] : -1;
                        const bool v = m >= 0 && m < M;
                        bad |= j < nrow && !v;
                        mm[q] = v ? m : -1;
                        const unsigned peers = __match_any_sync(kFull, mm[q]);
                        const int first = __ffs(peers) - 1;
                        int p0 = 0;
                        if (v && lane == first) p0 = atomicAdd(&cnt[m], __popc(peers));
                        pos[q] = __shfl_sync(kFull, p0, first) + __popc(peers & lt);
                    }
                    consumers();
                    // the counts of models 4 lane .. 4 lane + 3 and their exclusive sums
                    const int4 c = reinterpret_cast<const int4 *>(cnt)[lane];
                    const int own = c.x + c.y + c.z + c.w;
                    int e = own;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(kFull, e, o);
                        if (lane >= o) e += y;
                    }
                    const int T = __shfl_sync(kFull, e, 31);
                    const int e0 = e - own, e1 = e0 + c.x, e2 = e1 + c.y, e3 = e2 + c.z;
                    const int pk0 = e0 | (e1 << 16), pk1 = e2 | (e3 << 16);
                    if (warp == 0) {
                        reinterpret_cast<int4 *>(s_start)[lane] = make_int4(e0, e1, e2, e3);
                        if (lane == 0) s_start[kCalMaxModels] = T;
                    }
                    if (threadIdx.x < kCalMaxModels) s_cnt[(k + 1) & 1][threadIdx.x] = 0;
                    const bool redo = s_redo[(k + 1) & 1] != 0;
                    if (threadIdx.x == 0) s_redo[k & 1] = 0;
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int m = max(mm[q], 0);
                        const int a = __shfl_sync(kFull, pk0, m >> 2), b = __shfl_sync(kFull, pk1, m >> 2);
                        const int s0 = (((m & 2) ? b : a) >> ((m & 1) * 16)) & 0xffff;
                        if (mm[q] >= 0) s_list[s0 + pos[q]] = (uint16_t)(q ? jb : ja);
                    }
                    if (redo && T > 0) {
                        const int4 sh = calib_share(c, e0, T, M, warp);
                        if (lane == 0) s_share[warp] = sh;
                    }
                    consumers();
                    if (T == 0 && threadIdx.x == 0) s_redo[k & 1] = 1;  // nothing to share out: the next tile's rows decide
                    const int4 sh = T > 0 ? s_share[warp] : make_int4(0, 0, 0, 1);
                    const int rk = sh.z, nwp = sh.w;
                    if (lane == 0 && sh.x < sh.y && s_start[sh.y] - s_start[sh.x] > 4 * 64 * nwp) s_redo[k & 1] = 1;
                    for (int m = sh.x; m < sh.y; ++m) {
                        const int s0 = s_start[m], s1 = s_start[m + 1];
                        if (s0 + 32 * rk >= s1) continue;
                        if (__any_sync(kFull, cur != m)) {
                            flush();
                            cur = m;
                        }
                        for (int p = s0 + 32 * rk; p < s1; p += 64 * nwp) {
                            const int p0 = p + lane, p1 = p0 + 32 * nwp;
                            const bool in0 = p0 < s1, in1 = p1 < s1;
                            const int j0 = in0 ? s_list[p0] : 0, j1 = in1 ? s_list[p1] : 0;
                            if (both(std::true_type{}, in0, in1, sm[j0], sm[j1], sf + j0 * kCalCols, sf + j1 * kCalCols,
                                     stt + j0, stt + j1))
                                continue;
#pragma unroll 1
                            for (int q = 0; q < 2; ++q) {
                                const int j = q ? j1 : j0;
                                row(q ? in1 : in0, sm[j], stt[j], sf + j * kCalCols);
                            }
                        }
                    }
                    release();
                }
            }
        }
        ok = !__syncthreads_or(failed);
        rest = c1;
    }
    if (!TMA)  // row by row, every warp through the same number of steps
        for (long long i0 = rest; i0 < c1; i0 += blockDim.x) {
            const long long i = i0 + threadIdx.x;
            const bool in = i < c1;
            row(in, in ? model[i] : 0, in ? time[i] : 0.0, F + (in ? i : 0) * kCalCols);
        }
    chain_next();
    flush();
    if (__any_sync(kFull, bad) && lane == 0) record_status(ctl, kEInval);
    if (!ok && threadIdx.x == 0) record_status(ctl, kECuda);
    __syncthreads();
    // each sum: the direct adds plus the flushes' carry-save words (the x t_hi halves of b
    // weigh 2^26)
    for (int i = threadIdx.x; i < M * kCalAcc; i += blockDim.x) {
        const int mm = i / kCalAcc, k = i - mm * kCalAcc;
        U128 v{sacc[2 * i], sacc[2 * i + 1]};
        auto add_cs = [&](int f, int sh) {
            const unsigned long long *w = scs + ((size_t)mm * kCalFlushSums + f) * 2;
            // w0 + 2^32 w1, then shifted left by sh (< 32): below 2^128
            U128 c{w[0], 0ull};
            add128(c, w[1] << 32, w[1] >> 32);
            add128(v, c.lo << sh, sh ? (c.hi << sh) | (c.lo >> (64 - sh)) : c.hi);
        };
        if (k < 15) add_cs(k, 0);
        else if (k < 20) {
            add_cs(k, 0);
            add_cs(k + 5, 26);
        } else add_cs(25, 0);
        atomic_add128(acc + 2 * i, v.lo, v.hi);
    }
    // the last CTA to finish solves every model and clears the sums for the next call
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the totals into the CTA's (now free) shared sums, the scaled entries into the ring
    for (int i = threadIdx.x; i < 2 * M * kCalAcc; i += blockDim.x) sacc[i] = __ldcg(acc + i);
    __syncthreads();
    double *W = reinterpret_cast<double *>(stages);
    for (int m = threadIdx.x >> 5; m < M; m += kCalThreads / 32) calib_entries(m, D == 4, sacc, W);
    __syncthreads();
    for (int m = (threadIdx.x >> 5) * 5; m < M; m += kCalThreads / 32 * 5) calib_factor(m, M, D, sacc, W, coef);
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * M * kCalAcc; i += blockDim.x) acc[i] = 0ull;
    if (threadIdx.x == 0) *done = 0u;
}

}  // namespace

static_assert(kCalMaxModels * (kCalAcc + kCalFlushSums) * 16 + 2 * kCalStageBytes <= kCalSmemMax,
              "two stages at most models");

static_assert((size_t)kCalMaxModels * kCalSolveWords * 8 <= 2 * kCalStageBytes, "the solve's entries fit the ring");
static size_t solve_bytes(int M) { return (size_t)M * kCalSolveWords * 8; }

static int calib_stages(int M) {
    const size_t fixed = cal_sums_bytes(M);
    return (int)std::min<size_t>(kCalStagesMax, (kCalSmemMax - fixed) / kCalStageBytes);
}

cudaError_t launch_calibrate(long long N, const long long *F, const int32_t *model, const double *time, int M,
                             int shared_beta1, unsigned long long *acc, double *coef, DevCtl *ctl, int grid,
                             cudaStream_t st) {
    const int D = shared_beta1 ? 4 : 5;
    const int nst = calib_stages(M);
    const size_t fixed = cal_sums_bytes(M);
    const bool tma = ((uintptr_t)F | (uintptr_t)model | (uintptr_t)time) % 16 == 0;
    if (N <= 0) grid = 1;
    // the ring also holds the solve's scaled entries (kCalSolveWords doubles a model)
    return launch_chained(tma ? k_calibrate<true> : k_calibrate<false>, grid, kCalThreads,
                          fixed + (tma ? kCalStageBytes * nst : solve_bytes(M)), st, N, F, model, time, M, D, nst, acc, coef,
                          ctl);
}

cudaError_t set_calib_smem() {
    cudaError_t e = allow_smem(k_calibrate<true>, kCalSmemMax);
    if (e == cudaSuccess)
        e = allow_smem(k_calibrate<false>, cal_sums_bytes(kCalMaxModels) + solve_bytes(kCalMaxModels));
    return e;
}

}  // namespace lr
