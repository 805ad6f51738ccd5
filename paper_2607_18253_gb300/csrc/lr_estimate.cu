// K2: per-candidate SFS TTFT (Sec. 4.1, Eq. 7-9), utility (Eq. 2) and the
// per-query argmax (Eq. 3, Eq. 5).
//
// Each thread owns four consecutive instances of its CTA's instance tile and
// walks the CTA's query rows; the instances' summaries (written by K1) sit in
// shared memory, their scalars in registers.  For a query of prompt p:
//
//   k* = #{k : R_k < p}          cumulative budget after the admission batch;
//                                found with one bucket lookup (bucket width
//                                2^shift is below every budget increment, so a
//                                bucket holds at most one boundary)
//   F  = (la + k* + [separate first decode], F1tot + p, F2_k*,
//         F3_k* + [separate first decode] p, F4tot + p(p+1)/2)
//   TTFT = b0 F0 + b1d F2 + b1p F1 + b2 F3 + b3 F4   (fixed fp32 order)
//
// The first two terms depend on k* only and are precomputed as T_k.  The
// int64 -> fp32 roundings of F1, F3 and F4 are done exactly with fp32 adds:
// X + y with X = H + L (H a multiple of 2^20 below 2^44, L < 2^20) rounds as
// fadd(H, fadd(L, y)) because the inner sum is an exact integer below 2^24
// and the outer add rounds the exact total once.  This keeps the hot loop on
// the FMA pipe; instances whose totals reach 2^44 take an int64 path.
//
// The kernel is bound by the instructions issued per candidate (and, below some tens of
// microseconds, by its start-up: tile block, live index, first rows), so:
//   * the fp32 work of two instances goes in one packed instruction;
//   * a prompt of at most near = min_j(B_j - S_j + 1) + 1 tokens has at most one budget
//     boundary below it on every instance, so k* is p > R_0 and the two candidate entries
//     stay in registers: no bucket and no table read (98% of pool256's queries);
//   * a row of several warps describes its winner once, after the chunk.
// Warp instructions for 65,536 x 256 candidates, kernel time: estimate 11.9 M, 16.0 us ->
// 8.3 M, 15.0 us; route 20.2 M, 27.0 -> 15.1 M, 23.0 us; with the matrix 27.6 -> 24.5 us.
//
// The estimate matrix is write-only (4 bytes per candidate) and leaves as one
// 16-byte evict-first store per thread and row, the batch indices too.  Where rows are not
// whole 16-byte words (I % 4 != 0) a thread stores its four values one by one, under
// predicates (in a loop that could not be unrolled they took 27.3 us for 50,001 x 250, now
// 12.3).  The average-case sources have little else to do than to store: there each warp puts
// its 128 elements of a row in order in shared memory first (15.0 -> 10.7 us for 50,001 x 250;
// the SFS estimate, bound by issue, loses by it: 12.3 -> 13.6).
// Routing reduces each row with redux.sync over the objective (the value itself, or an
// order-preserving integer key): the lowest lane (lowest instance) among the maximal wins,
// as in a first-max scan.
#include <cooperative_groups.h>
#include <math.h>

#include "lr_internal.cuh"

namespace lr {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr long long kLowMask = (1LL << kSplitBits) - 1;
constexpr float kNaN = __builtin_nanf("");

// A staged query row: the fp32 values twice each, as the packed instructions take them.
struct __align__(16) QRec {
    float fp[2];  // p as fp32, NaN if p was out of range
    float ph[2];  // p(p+1)/2 high part (multiple of 2^20)
    float pl[2];  // p(p+1)/2 low part
    int p;        // prompt length, clamped into [1, pmax] for table lookups
    int row;      // a matrix source: the query's row
};

__device__ __forceinline__ QRec make_qrec(int p, int pmax, bool *ok) {
    QRec q;
    *ok = p >= 1 && p <= pmax;
    if (!*ok) p = 1;
    const long long pp = ((long long)p * (p + 1)) / 2;
    const long long pl = pp & kLowMask;
    q.p = p;
    q.fp[0] = q.fp[1] = *ok ? (float)p : kNaN;
    q.ph[0] = q.ph[1] = __ll2float_rn(pp - pl);
    q.pl[0] = q.pl[1] = __ll2float_rn(pl);
    q.row = 0;
    return q;
}

// Order-preserving key of a float (no NaN): larger float <-> larger key, and
// -0 and +0 share a key.  Zero is below every key.
__device__ __forceinline__ unsigned order_key(float x) {
    const unsigned u = __float_as_uint(__fadd_rn(x, 0.0f));
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// ---------------------------------------------------------------------------
// Integer features (exact, for verification): one thread per candidate.
__global__ void __launch_bounds__(256) k_features(const K2Launch a) {
    const DevConfig &c = a.cfg;
    const int active = *((volatile int32_t *)&a.ctl->active);
    const long long total = (long long)a.Q * c.I;
    const int off = (c.mode == 0) ? 1 : 0;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(idx / c.I);
        const int j = (int)(idx - (long long)i * c.I);
        long long *F = a.features + idx * 5;
        const int p = a.prompt[i];
        if (active < 0 || p < 1 || p > c.pmax) {
            record_status(a.ctl, active < 0 ? kENoState : kEInval);
            for (int f = 0; f < 5; ++f) F[f] = -1;
            continue;
        }
        const StateBuf sb = active ? a.buf1 : a.buf0;
        const InstParams ip = sb.inst[j];
        const int2 bk = sb.bkt[(size_t)(p >> ip.shift) * c.I + j];
        const int k = bk.y + (p > bk.x ? 1 : 0);
        const size_t e = (size_t)k * c.I + j;
        F[0] = ip.la + k + off;
        F[1] = ip.f1tot + p;
        F[2] = sb.f2[e];
        F[3] = sb.f3[e] + (c.mode == 0 ? p : 0);
        F[4] = ip.f4tot + ((long long)p * (p + 1)) / 2;
    }
}

// ---------------------------------------------------------------------------
// The candidate kernel.
enum : int {
    kOutMatrix = 1,   // write the TTFT matrix
    kOutIters = 2,    // write the first-token batch index
    kOutLag = 4,      // Lagrangian argmax (Eq. 5), one (lambda, mu) pair
    kOutCon = 8,      // constrained argmax (Eq. 3), one lambda
    kOutSweep = 16    // Lagrangian argmax for several pairs
};

// Two fp32 values in one 64-bit register pair: the packed fp32 instructions do the two
// IEEE operations of a pair in one issue slot, each rounded as the scalar instruction.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
    f32x2 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
    return v;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 v;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 v;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
    return v;
}

// A thread's four instances as two pairs.  Of a compact instance h1 holds the whole F1tot
// (exact in fp32, and so is F1tot + p) and l1 is unused.
struct Inst4 {
    f32x2 h1[2], l1[2], h4[2], l4[2], b1p[2], b2[2], b3[2];
};

// T: the first two terms, which depend on k* only; f3 = fp32(F3 of the candidate); F1 and F4
// by exact fp32 sums of the split totals and the query's parts.
template <bool COMPACT>
__device__ __forceinline__ f32x2 ttft_fast2(f32x2 fp, f32x2 ph, f32x2 pl, const Inst4 &r, int v, f32x2 T, f32x2 f3) {
    const f32x2 f1 = add2(r.h1[v], COMPACT ? fp : add2(r.l1[v], fp));
    const f32x2 f4 = add2(add2(r.h4[v], ph), add2(r.l4[v], pl));
    f32x2 t = fma2(r.b1p[v], f1, T);
    t = fma2(r.b2[v], f3, t);
    return fma2(r.b3[v], f4, t);
}

// Exact int64 path for instances whose totals do not split into fp32.
template <int MODE>
__device__ float ttft_exact64(const DevConfig &c, const StateBuf &sb, int qp, int j, int k, const float T) {
    const InstParams ip = sb.inst[j];
    const int m = c.moi[j];
    const long long p = qp;
    const float f1 = __ll2float_rn(ip.f1tot + p);
    const float f3 = __ll2float_rn(sb.f3[(size_t)k * c.I + j] + (MODE == 0 ? p : 0));
    const float f4 = __ll2float_rn(ip.f4tot + (p * (p + 1)) / 2);
    float t = __fmaf_rn(c.coef[m * 5 + 1], f1, T);
    t = __fmaf_rn(c.coef[m * 5 + 3], f3, t);
    t = __fmaf_rn(c.coef[m * 5 + 4], f4, t);
    return t;
}

// Reduce a key over the row's lanes; returns the winning lane's value of `v`
// (and its key) to every lane of the row group.  Rows of up to 32 groups sit in
// an aligned power-of-two lane group; wider rows use whole warps per row.
__device__ __forceinline__ unsigned group_mask(int Gp, int lane) {
    if (Gp >= 32) return kFull;
    const unsigned g = (Gp == 32) ? kFull : ((1u << Gp) - 1u);
    return g << (lane & ~(Gp - 1));
}

// A routing candidate: its key, instance, TTFT and utility.
struct Cand {
    unsigned key;  // order key of the objective, 0 = none
    int j;         // instance (the thread-local index before group_pick)
    float t, U;
};

__device__ __forceinline__ int4 pack(const Cand &c) {
    return make_int4((int)c.key, c.j, __float_as_int(c.t), __float_as_int(c.U));
}

__device__ __forceinline__ Cand unpack(const int4 v) {
    return Cand{(unsigned)v.x, v.y, __int_as_float(v.z), __int_as_float(v.w)};
}

__device__ __forceinline__ void write_pick(const K2Launch &a, size_t o, const Cand &w) {
    if (w.key == 0u) {  // invalid prompt: no instance
        a.assign[o] = -1;
        a.util[o] = kNaN;
        if (a.ttft_chosen) a.ttft_chosen[o] = kNaN;
    } else {
        a.assign[o] = w.j;
        a.util[o] = w.U;
        if (a.ttft_chosen) a.ttft_chosen[o] = w.t;
    }
}

// Table loads by 32-bit shared-memory address.  The tables are written once
// before the first barrier and only read afterwards.
__device__ __forceinline__ float2 lds_float2(uint32_t addr) {
    float2 v;
    asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint4 lds_u32x4(uint32_t addr) {
    uint4 v;
    asm("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

__device__ __forceinline__ void sts_f4(uint32_t addr, float x, float y, float z, float w) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

__device__ __forceinline__ float lds_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

// Maximum over the warp (all 32 lanes); NaN values lose, and only if all are is it NaN.
__device__ __forceinline__ float warp_max_f32(float x) {
    float m;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
    return m;
}

// The first index of x among v[0..3] (x is one of them, or nothing compares equal).
__device__ __forceinline__ int first4(const float v[4], float x) {
    return v[0] == x ? 0 : v[1] == x ? 1 : v[2] == x ? 2 : 3;
}

__device__ __forceinline__ float pick4(const float v[4], int u) {
    float x = v[0];
    x = (u == 1) ? v[1] : x;
    x = (u == 2) ? v[2] : x;
    x = (u == 3) ? v[3] : x;
    return x;
}

// Asynchronous 4-byte global -> shared copies (the staging of the next chunk of
// query rows overlaps the current chunk's compute).
__device__ __forceinline__ void cp_async4(void *smem_dst, const void *gmem_src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)),
                 "l"(gmem_src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One poll of an mbarrier's phase 0 (true once the bulk copy it tracks has landed).
__device__ __forceinline__ bool mbar_test(uint32_t mbar) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred P;\n mbarrier.try_wait.parity.shared::cta.b64 P, [%1], 0;\n selp.u32 %0, 1, 0, P;\n}"
        : "=r"(done)
        : "r"(mbar)
        : "memory");
    return done != 0;
}

template <bool B>
struct Flag {
    static constexpr bool value = B;
};

// The rows of a launch, per tile, as ranges (x, end) that a CTA works through QT rows
// at a time.  CTA b < first_ctas starts with the static range [b F, (b + 1) F)
// (F = first_rows, most of its share of the rows): those CTAs fit beside a snapshot
// load's CTAs running on another stream and start at once.  The remaining rows are
// claimed from the tile's counter, which counts the rows past the static ones: an equal
// share of those left, to route half of one (65,536 x 256 beside a load 33.0 -> 30.8 us, with
// deadlines 47 -> 40; an estimate of 16,384, with fewer and wider CTAs, takes 14.4 us with
// whole shares and 16.1 with halves), at most QT, down to a.least at the end (a claim's
// atomic still returns well within the chunk before it).  So CTAs that start late (their SM busy with the
// load) or run slower take less, and all finish at about the same time.  `seen` is
// a row index recently reached.
__device__ __forceinline__ int claim_size(const K2Launch &a, int seen) {
    const int n = (a.Q - seen) / (a.share * (int)gridDim.x);
    return min(a.QT, max(a.least, n - n % a.QS));
}
__device__ __forceinline__ int static_rows(const K2Launch &a) { return min(a.Q, a.first_ctas * a.first_rows); }
// Every row of the launch lies in a static range: no CTA claims, and the counters stay
// untouched (and zero) -- a call that runs alone takes no atomic round trip at all.
__device__ __forceinline__ bool all_static(const K2Launch &a) { return (long long)a.first_ctas * a.first_rows >= a.Q; }
__device__ __forceinline__ int claim_rows(const K2Launch &a, int seen) {
    if (all_static(a)) return a.Q;
    return static_rows(a) + (int)atomicAdd(a.work + 1 + blockIdx.y, (unsigned)claim_size(a, seen));
}
__device__ __forceinline__ int2 first_range(const K2Launch &a) {
    if ((int)blockIdx.x < a.first_ctas)
        return make_int2((int)blockIdx.x * a.first_rows, ((int)blockIdx.x + 1) * a.first_rows);
    const int seen = static_rows(a) + (int)*(volatile uint32_t *)(a.work + 1 + blockIdx.y);
    const int x = claim_rows(a, seen);
    return make_int2(x, x + claim_size(a, seen));
}
// The range left after the chunk at the head of r, if any: no claim needed.
__device__ __forceinline__ bool has_rest(const K2Launch &a, int2 r) { return r.x + a.QT < min(r.y, a.Q); }
// The range that follows the chunk at the head of r (the claim x was made for it).
__device__ __forceinline__ int2 range_after(const K2Launch &a, int2 r, int x) {
    return has_rest(a, r) ? make_int2(r.x + a.QT, r.y) : make_int2(x, x + claim_size(a, r.x));
}

// End of a candidate-kernel CTA: the last of `ctas` to finish clears the row
// counters of the `tiles` tiles and the completion count for the next launch.
__device__ __forceinline__ void k2_finish(const K2Launch &a, uint32_t *work, unsigned ctas, unsigned tiles) {
    if (all_static(a)) return;  // no counter was touched
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(work, 1u) == ctas - 1) {
            for (unsigned y = 0; y < tiles; ++y) atomicExch(work + 1 + y, 0u);
            atomicExch(work, 0u);
            __threadfence();
        }
    }
}

// MODE 0 / 1: SFS with the first output token in its own batch / with the last
// prompt chunk.  MODE 2: an average-case source (Sec. 4, App. E), affine in p:
// t = fma(p, g_j, C_j) with g_j = fp32(1/theta_j) and C_j = fp32(W_j + Tdec_j).
// Routing launches three 256-thread CTAs per SM (80 registers a thread), the estimate
// alone one 512-thread CTA (up to 128: the two-entry path of mixed models fits without
// spills; 768 threads took 17.9 us for 50,001 x 250 against 15.6).
template <int MODE, int OUT>
__global__ void __launch_bounds__((OUT & (kOutLag | kOutCon | kOutSweep)) ? kK2Block : kK2EstBlock,
                                  (OUT & (kOutLag | kOutCon | kOutSweep)) ? 3 : 1) k_cand(const K2Launch a) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool AFF = MODE == 2;
    constexpr bool ROUTE = (OUT & (kOutLag | kOutCon | kOutSweep)) != 0;
    constexpr bool CON = (OUT & kOutCon) != 0;
    constexpr bool SWEEP = (OUT & kOutSweep) != 0;
    constexpr int off = (MODE == 0) ? 1 : 0;
    const DevConfig &c = a.cfg;
    const int I = c.I, M = c.M, Gp = a.Gp, QS = a.QS, QT = a.QT;
    const int lane = threadIdx.x & 31;
    const int g = threadIdx.x % Gp;
    const int qs = threadIdx.x / Gp;
    const int j0 = blockIdx.y * Gp * 4;
    const int jb = j0 + 4 * g;                         // first instance of this thread
    const int nv = max(0, min(4, I - jb));             // instances this thread owns
    // Query rows come in ranges (first_range, range_after): a static one, then claims
    // from this tile's counter, in the no-snapshot path as in the main one.
    __shared__ int s_active;
    __shared__ int2 s_claim[2];
    __shared__ __align__(8) unsigned long long s_mbar;
    const uint32_t mbar = (uint32_t)__cvta_generic_to_shared(&s_mbar);
    const size_t tb = tile_bytes(c);
    // Shared memory: the tile block (tables and per-instance scalars, exactly as K1
    // laid it out for this tile), query records, row partials, utility inputs,
    // targets and the raw query rows (route with one pair stages (U, cost) per row
    // and model, sweeps (cost, acc)).
    const int WPR = Gp > 32 ? Gp / 32 : 1;  // warps per row
    // (an affine source needs no tables: in their place each warp has two 128-float buffers in
    // which its stores are put in order, if rows are not whole 16-byte words)
    QRec *s_q = reinterpret_cast<QRec *>(smem + k2_head_bytes(c, blockDim.x));         // [QT]
    int4 *s_part = reinterpret_cast<int4 *>(s_q + QT);                                 // [NP][QT][WPR][2]
    // a sweep keeps the chunk's times [QT][4 Gp] instead of row partials, and per thread group
    // and instance the model (s_m4: -1 if the group's four differ)
    float4 *s_t = reinterpret_cast<float4 *>(s_part);                                  // [QT][Gp]
    int32_t *s_m4 = reinterpret_cast<int32_t *>(s_t + (SWEEP ? QT * Gp : 0));          // [Gp], [Gp][4], then lambda, mu
    float2 *s_lm = reinterpret_cast<float2 *>(s_m4 + (SWEEP ? 5 * Gp + (Gp & 1) : 0));  // [kMaxPairs] (lambda, -mu)
    float2 *s_ca = SWEEP ? s_lm + kMaxPairs
                         : reinterpret_cast<float2 *>(s_part + (ROUTE && Gp > 32 ? 2 * QT * WPR : 0));  // [QT][M]
    float *s_tau = reinterpret_cast<float *>(s_ca + (ROUTE ? QT * M : 0));             // [QT]
    // raw query rows as copied from global memory, two chunks in flight:
    // prompt [2][QT], and for routing tau [2][QT], dec_hat [2][QT][M], acc [2][QT][M]
    int32_t *r_p = reinterpret_cast<int32_t *>(s_tau + (ROUTE ? QT : 0));
    float *r_t = reinterpret_cast<float *>(r_p + 2 * QT);
    int32_t *r_d = reinterpret_cast<int32_t *>(r_t + (ROUTE ? 2 * QT : 0));
    float *r_a = reinterpret_cast<float *>(r_d + (ROUTE ? 2 * QT * M : 0));
    // copies of query rows [q0, q0 + nrows) into raw buffer b
    auto issue = [&](int q0, int nrows, int b) {
        for (int t = threadIdx.x; t < nrows; t += blockDim.x) {
            cp_async4(r_p + b * QT + t, a.prompt + q0 + t);
            if (CON) cp_async4(r_t + b * QT + t, a.tau + q0 + t);
        }
        if (ROUTE) {
            const size_t g0 = (size_t)q0 * M;
            for (int idx = threadIdx.x; idx < nrows * M; idx += blockDim.x) {
                cp_async4(r_d + b * QT * M + idx, a.dec_hat + g0 + idx);
                cp_async4(r_a + b * QT * M + idx, a.acc + g0 + idx);
            }
        }
        cp_async_commit();
    };
    // The tile block arrives with one bulk copy (TMA) completing on an mbarrier:
    // every CTA reads the same few tens of KB, and one large request per CTA is far
    // cheaper than thousands of scattered loads of the same lines.
    auto tile_copy = [&](const unsigned char *src, uint32_t dst_off) {
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                (uint32_t)__cvta_generic_to_shared(smem) + dst_off),
            "l"(src), "r"((uint32_t)tb), "r"(mbar)
            : "memory");
    };
    // bounded wait for the tile block: a copy that never lands is reported, not waited out
    auto tile_wait = [&]() -> bool {
        bool landed = false;
        for (int it = 0; it < (1 << 22) && !landed; ++it) landed = mbar_test(mbar);
        return landed;
    };
    if (threadIdx.x == 0 && !AFF) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    chain_wait();
    if (threadIdx.x == 0) s_claim[0] = first_range(a);
    __syncthreads();
    const int2 first = s_claim[0];
    // the first chunk of query rows travels while the live index is read and the tile
    // block lands; one read of the live-buffer index per CTA (every thread reading the
    // same word would queue them all on one L2 line)
    if (first.x < a.Q) issue(first.x, min(QT, min(first.y, a.Q) - first.x), 0);
    if (threadIdx.x == 0) s_active = load_live(a.ctl);
    __syncthreads();
    const int active = s_active;
    // the LPS source and a given matrix need no live snapshot; every other source does
    if (active < 0 && !(AFF && (a.src == kSrcLps || a.src == kSrcMatrix))) {
        if (threadIdx.x == 0) record_status(a.ctl, kENoState);
        cp_async_wait<0>();  // nothing may still be landing when the CTA leaves
        for (int k = 0;; ++k) {
            __syncthreads();  // the previous range has been read
            if (threadIdx.x == 0 && k > 0) {
                const int2 r = s_claim[0];
                s_claim[0] = range_after(a, r, has_rest(a, r) ? 0 : claim_rows(a, r.x));
            }
            __syncthreads();
            const int rb = s_claim[0].x, re = min(min(a.Q, s_claim[0].y), rb + QT);
            if (rb >= a.Q) break;
            for (int rr = rb + qs; rr < re; rr += QS) {
                for (int u = 0; u < nv; ++u) {
                    if (OUT & kOutMatrix) a.ttft[(size_t)rr * I + jb + u] = kNaN;
                    if (OUT & kOutIters) a.first_batch[(size_t)rr * I + jb + u] = -1;
                }
                if (ROUTE && g == 0)
                    for (int pp = 0; pp < a.P; ++pp) {
                        a.assign[(size_t)pp * a.Q + rr] = -1;
                        a.util[(size_t)pp * a.Q + rr] = kNaN;
                        if (a.ttft_chosen) a.ttft_chosen[(size_t)pp * a.Q + rr] = kNaN;
                    }
            }
        }
        k2_finish(a, a.work, gridDim.x * gridDim.y, gridDim.y);
        return;
    }
    {
    const StateBuf sb = active ? a.buf1 : a.buf0;
    // (Gp == c.tgp: the tile block's sections at the offsets K1 wrote them)
    const unsigned char *tile = smem;
    const unsigned char *s_ent = tile;                                                         // entA, entB
    const unsigned char *s_bkt = tile + tile_ent_bytes(c);                                     // [nbh][4][Gp]
    const int32_t *s_scal = reinterpret_cast<const int32_t *>(s_bkt + tile_bkt_bytes(c));    // [kScal][4][Gp]
    if (threadIdx.x == 0 && !AFF) {
        // the block was written by generic stores (possibly of a load on another
        // stream, acquired above); order them before the bulk copy's reads
        asm volatile("fence.proxy.async.global;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"((uint32_t)tb) : "memory");
        tile_copy(sb.tile + (size_t)blockIdx.y * tb, 0u);
    }
    // what follows the first chunk: found now, published once the tile block has landed
    int2 second = make_int2(a.Q, a.Q);
    if (threadIdx.x == 0 && first.x < a.Q) second = range_after(a, first, has_rest(a, first) ? 0 : claim_rows(a, first.x));
    if (!AFF) {
        if (__syncthreads_or(!tile_wait())) {
            if (threadIdx.x == 0) record_status(a.ctl, kECuda);
            for (int it = 0; it < (1 << 22) && !mbar_test(mbar); ++it) {
            }
            cp_async_wait<0>();
            goto finish;
        }
    }
    int model[4];
    float ag[4], ac[4];  // average-case sources: t = fma(p, ag, ac)
    bool fast_mine = true, compact_mine = true;
    const int fs = 4 * Gp;  // scalar field stride
    auto scal = [&](int f, int u) { return s_scal[f * fs + u * Gp + g]; };
    // the bucket width of the tile's first instance
    const int shift0 = AFF ? 0 : s_scal[kScShift * fs];
    bool same_model = true, same_shift = true;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (AFF) {
            const int j = min(jb + u, I - 1);
            model[u] = c.moi[j];
            const QueueDev qd = a.qd[j];
            ag[u] = qd.g;
            // throughput source: residents' remaining prefill tokens / theta + Tdec
            ac[u] = (a.src == kSrcLps)      ? qd.clps
                    : (a.src == kSrcMatrix) ? 0.f
                                            : __double2float_rn(__dadd_rn(__ddiv_rn((double)sb.inst[j].f1tot, qd.theta), qd.tdec));
        } else {
            model[u] = scal(kScModel, u);
            same_shift = same_shift && scal(kScShift, u) == shift0;
            if (u < nv) fast_mine = fast_mine && scal(kScFast, u) != 0;
            if (u < nv) compact_mine = compact_mine && scal(kScCompact, u) != 0;
        }
        same_model = same_model && model[u] == model[0];
    }
    if (threadIdx.x == 0) s_claim[1] = second;
    const bool fast = __syncthreads_and(fast_mine);
    // every instance of the CTA compact (padding columns are)
    const bool compact = fast && __syncthreads_and(compact_mine);
    const bool vec = a.vec_ok && nv == 4;
    const unsigned gmask = group_mask(Gp, lane);
    const int wrow = g / 32;                          // warp index within a wide row
    // shared addresses of this thread's table columns: entA (k, u) at
    // ecol + u * ecst + k * erow (entB ebofs further), bucket (b, u) at
    // bcol + 4 u + b * brow (formed at each use: the kernel is at its register limit)
    const uint32_t ecol = (uint32_t)__cvta_generic_to_shared(s_ent) + 8u * (uint32_t)g;
    const uint32_t bcol = (uint32_t)__cvta_generic_to_shared(s_bkt) + 16u * (uint32_t)g;
    const uint32_t ecst = 8u * (uint32_t)Gp;
    const uint32_t erow = 8u * 4u * (uint32_t)Gp, brow = 4u * 4u * (uint32_t)Gp;
    const uint32_t ebofs = (uint32_t)tile_enta_bytes(c);
    const bool tr = AFF && I % 4 != 0 && Gp >= 32;
    const uint32_t trb = (uint32_t)__cvta_generic_to_shared(smem) + (threadIdx.x >> 5) * 1024u;
    const int ntr = min(4, max(0, (I - (jb - 4 * lane) - lane + 31) >> 5));  // of this lane's four, those in the pool
    if (SWEEP) {
        if (threadIdx.x < Gp) {
            bool one = true;
            for (int u = 0; u < 4; ++u) {
                s_m4[Gp + 4 * g + u] = model[u];
                one = one && (u >= nv || model[u] == model[0]);
            }
            s_m4[g] = one ? model[0] : -1;
        }
        for (int k = threadIdx.x; k < a.P; k += blockDim.x) s_lm[k] = make_float2(a.lam[k], -a.mu[k]);
    }
    // UNI: every thread of the CTA has four compact instances of one model and every
    // instance the same bucket width (a thread's four buckets are one 16-byte load)
    const bool uni = __syncthreads_and(compact && nv == 4 && same_model && same_shift);
    auto run = [&](auto fast_tag, auto compact_tag, auto uni_tag, auto wide_tag) {
        constexpr bool FAST = decltype(fast_tag)::value;
        constexpr bool COMPACT = decltype(compact_tag)::value;
        constexpr bool UNI = decltype(uni_tag)::value;
        constexpr bool WIDE = decltype(wide_tag)::value;  // Gp > 32: whole warps per row
        // the register path for prompts with at most one budget boundary below them (not
        // beside the routing state of threads with several models: the registers end there)
        constexpr bool NEAR = COMPACT && !AFF && (UNI || !ROUTE);
        // Lagrangian routing over threads of one model each: the winner of a row of several
        // warps is described once per row, after the chunk, instead of by a lane of every warp
        constexpr bool DEFER = ROUTE && UNI && WIDE && !CON && !SWEEP;
        Inst4 r;
        int r0[4], shift[4], la[4] = {0, 0, 0, 0};
        float T0[4], T1[4], X0[4], X1[4];  // entries 0 and 1 of the thread's instances (see the tile block)
        if (!AFF) {
            auto two = [&](int f, int v) { return pack2(__int_as_float(scal(f, 2 * v)), __int_as_float(scal(f, 2 * v + 1))); };
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                r.l1[v] = two(kScL1, v);
                r.h1[v] = COMPACT ? add2(two(kScH1, v), r.l1[v]) : two(kScH1, v);
                r.h4[v] = two(kScH4, v);
                r.l4[v] = two(kScL4, v);
                r.b1p[v] = UNI && v ? r.b1p[0] : two(kScB1p, v);
                r.b2[v] = UNI && v ? r.b2[0] : two(kScB2, v);
                r.b3[v] = UNI && v ? r.b3[0] : two(kScB3, v);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                shift[u] = scal(kScShift, u);
                if (OUT & kOutIters) la[u] = scal(kScLa, u);
                r0[u] = scal(kScR0, u);
                const float2 e0 = lds_float2(ecol + u * ecst), e1 = lds_float2(ecol + u * ecst + (c.kph > 1 ? erow : 0u));
                T0[u] = e0.x;
                X0[u] = e0.y;
                T1[u] = e1.x;
                X1[u] = e1.y;
            }
        }
        const f32x2 nmu2 = (ROUTE && !CON && !SWEEP) ? pack2(-a.mu[0], -a.mu[0]) : 0ull;
        // chunk k: the first QT rows of the range in s_claim[k & 1], staged in raw buffer k & 1
        for (int buf = 0;; buf ^= 1) {
            int q0, nrows;
            {
                const int2 cur = s_claim[buf], nxt = s_claim[buf ^ 1];
                if (cur.x >= a.Q) break;
                q0 = cur.x;
                nrows = min(QT, min(cur.y, a.Q) - q0);
                if (nxt.x < a.Q) {
                    issue(nxt.x, min(QT, min(nxt.y, a.Q) - nxt.x), buf ^ 1);
                    cp_async_wait<1>();
                } else {
                    cp_async_wait<0>();
                }
            }
            __syncthreads();  // every thread's copies of this chunk have landed
            // the range after the next chunk: claimed now if needed, published when this chunk is done
            int ahead = a.Q;
            if (threadIdx.x == 0 && s_claim[buf ^ 1].x < a.Q && !has_rest(a, s_claim[buf ^ 1]))
                ahead = claim_rows(a, s_claim[buf ^ 1].x);
            const int32_t *bp = r_p + buf * QT;
            for (int t = threadIdx.x; t < nrows; t += blockDim.x) {
                bool ok;
                s_q[t] = make_qrec(bp[t], c.pmax, &ok);
                // a given matrix: this query's row of it
                if (AFF) s_q[t].row = a.lead_order ? a.lead_order[a.lead_start[ok ? bp[t] : 0]] : q0 + t;
                if (!ok && blockIdx.y == 0) record_status(a.ctl, kEInval);
                if (CON) s_tau[t] = r_t[buf * QT + t];
            }
            if (ROUTE) {
                const int32_t *bd = r_d + buf * QT * M;
                const float *ba = r_a + buf * QT * M;
                for (int idx = threadIdx.x; idx < nrows * M; idx += blockDim.x) {
                    const int rr = idx / M;
                    const int m = idx - rr * M;
                    const float cost = __fmaf_rn((float)bd[idx], c.pout[m], __fmul_rn((float)bp[rr], c.pin[m]));
                    const float acc = ba[idx];
                    // one pair: stage U itself (x), else (cost, acc)
                    s_ca[idx] = SWEEP ? make_float2(cost, acc) : make_float2(__fmaf_rn(-a.lam[0], cost, acc), cost);
                }
            }
            __syncthreads();
            float *orow = (OUT & kOutMatrix) ? a.ttft + (size_t)(q0 + qs) * I + jb : nullptr;
            const size_t ostep = (size_t)QS * I;
            float *frow = (OUT & kOutIters) ? reinterpret_cast<float *>(a.first_batch) + (size_t)(q0 + qs) * I + jb : nullptr;
            const bool mat = AFF && a.src == kSrcMatrix;
            // a given matrix: its row is read one row ahead
            float tn[4];
            auto read_row = [&](int rr) {
                if (!mat || rr >= nrows) return;
                const float *src = a.ttft_in + (size_t)s_q[rr].row * I + jb;
                if (vec) {
                    const float4 f = __ldcs(reinterpret_cast<const float4 *>(src));
                    tn[0] = f.x;
                    tn[1] = f.y;
                    tn[2] = f.z;
                    tn[3] = f.w;
                } else {
#pragma unroll
                    for (int u = 0; u < 4; ++u) tn[u] = u < nv ? __ldcs(src + u) : kNaN;
                }
            };
            if (AFF) read_row(qs);
            uint32_t trw = trb;  // the buffer of the two that is next
            // four values of a row at p (v4: as one 16-byte word)
            auto store4 = [&](float *p, bool v4, const float v[4]) {
                if (v4) {
                    __stcs(reinterpret_cast<float4 *>(p), make_float4(v[0], v[1], v[2], v[3]));
                } else if (tr) {
                    sts_f4(trw + 16u * lane, v[0], v[1], v[2], v[3]);
                    __syncwarp();
                    p -= 3 * lane;  // element `lane` of the warp's block
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (u < ntr) __stcs(p + 32 * u, lds_f32(trw + 4u * lane + 128u * u));
                    trw ^= 512u;  // the other buffer: the next row's writes need not wait for these reads
                } else if (nv > 0) {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (u < nv) __stcs(p + u, v[u]);
                }
            };
            for (int rr = qs; rr < nrows; rr += QS) {
                struct {
                    f32x2 fp2, ph2, pl2;
                    float fp;
                    int p;
                } q;
                {
                    const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(s_q + rr);
                    const int4 y = reinterpret_cast<const int4 *>(s_q + rr)[1];
                    q.fp2 = x.x;
                    q.ph2 = x.y;
                    q.pl2 = pack2(__int_as_float(y.x), __int_as_float(y.y));
                    q.p = y.z;
                    q.fp = __uint_as_float((unsigned)x.x);
                }
                float t[4];
                int kk[4] = {0, 0, 0, 0};
                if (AFF) {
                    if (mat) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) t[u] = tn[u];
                        read_row(rr + QS);
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u) t[u] = __fmaf_rn(q.fp, ag[u], ac[u]);
                    }
                } else if (FAST) {
                    float T[4], F3[4];
                    if (NEAR && q.p <= c.near) {
                        // at most one budget boundary lies below p: k* = (p > r0), and the
                        // two candidate entries are in registers
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const bool k1 = q.p > r0[u];
                            T[u] = k1 ? T1[u] : T0[u];
                            const float x = k1 ? X1[u] : X0[u];
                            F3[u] = MODE == 0 ? __int2float_rn(__float_as_int(x) + q.p) : x;
                            kk[u] = k1 ? 1 : 0;
                        }
                    } else {
                        const uint32_t p7 = (uint32_t)q.p << 7;
                        uint4 bw4 = make_uint4(0u, 0u, 0u, 0u);
                        if (UNI) bw4 = lds_u32x4(bcol + (uint32_t)(q.p >> shift0) * brow);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            // bucket word (boundary << 7) | below: p > boundary iff (p << 7) > word
                            const uint32_t bw = UNI ? (u == 0 ? bw4.x : u == 1 ? bw4.y : u == 2 ? bw4.z : bw4.w)
                                                    : lds_u32(bcol + 4u * u + (uint32_t)(q.p >> shift[u]) * brow);
                            kk[u] = (int)(bw & 127u) + (p7 > bw ? 1 : 0);
                            const uint32_t ea = ecol + u * ecst + (uint32_t)kk[u] * erow;
                            const float2 e = lds_float2(ea);
                            T[u] = e.x;
                            F3[u] = e.y;
                            if (COMPACT && MODE == 0) {
                                // F3 + p below 2^31, one exact int -> fp32 rounding
                                F3[u] = __int2float_rn(__float_as_int(e.y) + q.p);
                            } else if (MODE == 0) {
                                const float2 hl = lds_float2(ea + ebofs);
                                F3[u] = __fadd_rn(hl.x, __fadd_rn(hl.y, q.fp));
                            }
                        }
                    }
#pragma unroll
                    for (int v = 0; v < 2; ++v)
                        unpack2(ttft_fast2<COMPACT>(q.fp2, q.ph2, q.pl2, r, v, pack2(T[2 * v], T[2 * v + 1]),
                                                    pack2(F3[2 * v], F3[2 * v + 1])),
                                t[2 * v], t[2 * v + 1]);
                } else {
                    const uint32_t p7 = (uint32_t)q.p << 7;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t bw = lds_u32(bcol + 4u * u + (uint32_t)(q.p >> shift[u]) * brow);
                        kk[u] = (int)(bw & 127u) + (p7 > bw ? 1 : 0);
                        const float2 e = lds_float2(ecol + u * ecst + (uint32_t)kk[u] * erow);
                        t[u] = q.fp != q.fp ? kNaN : (u < nv) ? ttft_exact64<MODE>(c, sb, q.p, jb + u, kk[u], e.x) : 0.f;
                    }
                }
                if (OUT & kOutMatrix) {
                    store4(orow, UNI ? a.vec_ok != 0 : vec, t);
                    orow += ostep;
                }
                if (OUT & kOutIters) {
                    const bool bad = q.fp != q.fp;
                    float f[4];  // (the indices' bits)
#pragma unroll
                    for (int u = 0; u < 4; ++u) f[u] = __int_as_float(bad ? -1 : la[u] + kk[u] + off);
                    store4(frow, UNI ? a.vec_first != 0 : a.vec_first && nv == 4, f);
                    frow += ostep;
                }
                if (SWEEP) {
                    if (!UNI) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (u >= nv) t[u] = kNaN;
                    }
                    s_t[rr * Gp + g] = make_float4(t[0], t[1], t[2], t[3]);
                } else if (ROUTE) {
                    const float2 *carow = s_ca + rr * M;
                    const float tau = CON ? s_tau[rr] : 0.f;
                    float2 ca0 = make_float2(0.f, 0.f);
                    if (UNI || same_model) ca0 = carow[model[0]];
                    float B[4];  // constrained: the times themselves, NaN beyond the pool
                    if (!UNI) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (u >= nv) t[u] = kNaN;
                    }
                    unsigned k2 = 0u;
                    float m2 = 0.f;
                    if (CON) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) B[u] = t[u];
                        m2 = fminf(fminf(t[0], t[1]), fminf(t[2], t[3]));  // NaN only if all are
                        k2 = m2 == m2 ? order_key(-m2) : 0u;
                    }
                    do {
                        float U[4];
                        if (UNI || same_model) {
                            U[0] = U[1] = U[2] = U[3] = ca0.x;
                        } else {
#pragma unroll
                            for (int u = 0; u < 4; ++u) U[u] = carow[model[u]].x;
                        }
                        // this thread's objective values; NaN (an invalid prompt, no estimate or an
                        // instance beyond the pool) is never the maximum
                        float J[4];
                        if (CON) {
#pragma unroll
                            for (int u = 0; u < 4; ++u) J[u] = t[u] <= tau ? U[u] : kNaN;
                        } else {
#pragma unroll
                            for (int v = 0; v < 2; ++v)
                                unpack2(fma2(nmu2, pack2(t[2 * v], t[2 * v + 1]), pack2(U[2 * v], U[2 * v + 1])), J[2 * v],
                                        J[2 * v + 1]);
                        }
                        const float m1 = fmaxf(fmaxf(J[0], J[1]), fmaxf(J[2], J[3]));
                        if (DEFER) {
                            // the first of the lanes with the warp's maximum leaves its times; its
                            // instance is picked when the chunk's rows are written (see below)
                            const float w = warp_max_f32(m1);
                            const unsigned best = __ballot_sync(kFull, m1 == w);
                            if (m1 == w && (best & lanemask_lt()) == 0u) {
                                float4 *part = reinterpret_cast<float4 *>(s_part + 2 * (rr * WPR + wrow));
                                part[0] = make_float4(t[0], t[1], t[2], t[3]);
                                part[1] = make_float4(w, U[0], __int_as_float(jb), 0.f);
                            } else if (best == 0u && lane == 0) {  // every objective is NaN
                                reinterpret_cast<float *>(s_part + 2 * (rr * WPR + wrow) + 1)[0] = kNaN;
                            }
                            break;
                        }
                        const unsigned k1 = m1 == m1 ? order_key(m1) : 0u;
                        // row group argmax: the lowest lane among the maximal keys
                        const unsigned w1 = __reduce_max_sync(gmask, k1);
                        const int src1 = __ffs(__ballot_sync(gmask, k1 == w1) & gmask) - 1;
                        unsigned w2 = 0u;
                        int src2 = 0;
                        if (CON) {
                            w2 = __reduce_max_sync(gmask, k2);
                            src2 = __ffs(__ballot_sync(gmask, k2 == w2) & gmask) - 1;
                        }
                        // the winner of each reduction describes itself: the first of its instances
                        // with the best value
                        if (Gp <= 32) {
                            const bool use2 = CON && w1 == 0u;
                            if (lane == (use2 ? src2 : src1)) {
                                const int u = use2 ? first4(B, m2) : first4(J, m1);
                                write_pick(a, (size_t)(q0 + rr), Cand{use2 ? w2 : w1, jb + u, pick4(t, u), pick4(U, u)});
                            }
                        } else {
                            // wide rows: each warp leaves its partial; combined once per chunk
                            int4 *part = s_part + 2 * (rr * WPR + wrow);
                            if (lane == src1) {
                                const int u = first4(J, m1);
                                part[0] = pack(Cand{w1, jb + u, pick4(t, u), pick4(U, u)});
                            }
                            if (CON && lane == src2) {
                                const int u = first4(B, m2);
                                part[1] = pack(Cand{w2, jb + u, pick4(t, u), pick4(U, u)});
                            }
                        }
                    } while (false);
                }
            }
            if (SWEEP) {
                // A lane per (row, pair), or several that split the row's instances (set_sweep_lanes):
                // each follows the pool's times of its row in instance order, so a candidate of a
                // pair costs a packed multiply-add and a running maximum, with no reduction per
                // row (a lane per four instances and one pair after the other took about 120 warp
                // instructions per row and pair).  32 pairs x 4,096 queries x 64 instances: kernel
                // 17.3 -> 12.0 us.
                __syncthreads();
                const int pg = a.pg, sp = a.sp, rw = 32 / (pg * sp), np = (a.P + pg - 1) / pg;
                const int pl = lane & (pg - 1), sl = lane / pg & (sp - 1), rs = lane / (pg * sp);
                const int nw = blockDim.x >> 5, w0 = threadIdx.x >> 5;
                const int drow = nw / np * rw, dpr = nw % np;  // the next unit: rows and blocks of pairs on
                for (int r0 = w0 / np * rw, pb = w0 % np; r0 < nrows;) {
                    const int row = r0 + rs, pp = pb * pg + pl;
                    r0 += drow;
                    pb += dpr;
                    if (pb >= np) {
                        pb -= np;
                        r0 += rw;
                    }
                    const bool act = row < nrows && pp < a.P && sl == 0;
                    const int rr = min(row, nrows - 1);
                    const float2 lm = s_lm[min(pp, a.P - 1)];
                    const f32x2 nm = pack2(lm.y, lm.y);
                    const float4 *tr4 = s_t + rr * Gp;
                    const float2 *carow = s_ca + rr * M;
                    // the best of a group of four, and the first group that has it: an objective of
                    // -inf (a product beyond fp32) is a value like any other, NaN (no estimate, or
                    // beyond the pool) is none
                    float best = -INFINITY, U = 0.f;
                    int bg = -1, cur = -1;
                    auto objectives = [&](int gg, float U4[4], float J[4]) {
                        const float4 t4 = tr4[gg];
                        const int m = s_m4[gg];
                        if (m >= 0) {
                            if (m != cur) {
                                const float2 ca = carow[m];
                                U = __fmaf_rn(-lm.x, ca.x, ca.y);
                                cur = m;
                            }
                            U4[0] = U4[1] = U4[2] = U4[3] = U;
                        } else {
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const float2 ca = carow[s_m4[Gp + 4 * gg + u]];
                                U4[u] = __fmaf_rn(-lm.x, ca.x, ca.y);
                            }
                        }
                        unpack2(fma2(nm, pack2(t4.x, t4.y), pack2(U4[0], U4[1])), J[0], J[1]);
                        unpack2(fma2(nm, pack2(t4.z, t4.w), pack2(U4[2], U4[3])), J[2], J[3]);
                    };
                    float U4[4], J[4];
                    auto walk = [&](int first, int step) {
                        for (int gg = first; 4 * gg < I; gg += step) {
                            objectives(gg, U4, J);
                            const float m1 = fmaxf(fmaxf(J[0], J[1]), fmaxf(J[2], J[3]));  // NaN only if all are
                            if (m1 > best) {
                                best = m1;
                                bg = gg;
                            }
                        }
                    };
                    if (sp == 1) {
                        walk(0, 1);  // (a step the compiler knows: 32,768 x 256 x 64 pairs 170 -> 153 us)
                    } else {
                        walk(sl, sp);
                        // the best of the lanes that share the instances, the lowest group among equals
                        for (int o = pg; o < pg * sp; o <<= 1) {
                            const float b2 = __shfl_xor_sync(kFull, best, o);
                            const int g2 = __shfl_xor_sync(kFull, bg, o);
                            if (b2 > best || (b2 == best && (unsigned)g2 < (unsigned)bg)) {
                                best = b2;
                                bg = g2;
                            }
                        }
                    }
                    if (bg < 0)  // none above -inf: the first that is not NaN, if any
                        for (int gg = 0; 4 * gg < I && bg < 0; ++gg) {
                            objectives(gg, U4, J);
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                if (J[u] == J[u]) bg = gg;
                        }
                    if (act) {
                        Cand w = {0u, 0, 0.f, 0.f};
                        if (bg >= 0) {
                            objectives(bg, U4, J);
                            const int u = first4(J, best);
                            w = Cand{1u, 4 * bg + u, reinterpret_cast<const float *>(tr4)[4 * bg + u], pick4(U4, u)};
                        }
                        write_pick(a, (size_t)pp * a.Q + q0 + row, w);
                    }
                }
            } else if (DEFER) {
                // one thread per row: the best warp of the row (the first among equals; a warp whose
                // objectives are all NaN -- an invalid prompt, or a cost that overflows times a
                // lambda of 0 -- yields to any), then the first of the winning thread's four
                // instances with that value
                __syncthreads();
                for (int r2 = threadIdx.x; r2 < nrows; r2 += blockDim.x) {
                    const float4 *part = reinterpret_cast<const float4 *>(s_part + 2 * (size_t)(r2 * WPR));
                    int wb = 0;
                    float w = part[1].x;
                    for (int wi = 1; wi < WPR; ++wi) {
                        const float x = part[2 * wi + 1].x;
                        if (x > w || w != w) {
                            w = x;
                            wb = wi;
                        }
                    }
                    const float4 tw = part[2 * wb], d = part[2 * wb + 1];
                    const float nm = -a.mu[0], tt[4] = {tw.x, tw.y, tw.z, tw.w};
                    const float J[4] = {__fmaf_rn(nm, tt[0], d.y), __fmaf_rn(nm, tt[1], d.y), __fmaf_rn(nm, tt[2], d.y),
                                        __fmaf_rn(nm, tt[3], d.y)};
                    const int u = first4(J, w);
                    // (w is NaN only if it is in every warp)
                    write_pick(a, (size_t)(q0 + r2), Cand{w == w ? 1u : 0u, __float_as_int(d.z) + u, pick4(tt, u), d.y});
                }
            } else if (ROUTE && Gp > 32) {
                // one thread per row combines the warps of the row in instance order
                __syncthreads();
                for (int r2 = threadIdx.x; r2 < nrows; r2 += blockDim.x) {
                    Cand c1 = {0u, 0, 0.f, 0.f}, c2 = {0u, 0, 0.f, 0.f};
                    for (int wi = 0; wi < WPR; ++wi) {
                        const Cand x1 = unpack(s_part[2 * (r2 * WPR + wi)]);
                        if (x1.key > c1.key) c1 = x1;
                        if (CON) {
                            const Cand x2 = unpack(s_part[2 * (r2 * WPR + wi) + 1]);
                            if (x2.key > c2.key) c2 = x2;
                        }
                    }
                    write_pick(a, (size_t)(q0 + r2), (CON && c1.key == 0u) ? c2 : c1);
                }
            }
            if (threadIdx.x == 0) {  // into the slot this chunk was read from
                const int2 nxt = s_claim[buf ^ 1];
                s_claim[buf] = nxt.x < a.Q ? range_after(a, nxt, ahead) : make_int2(a.Q, a.Q);
            }
            __syncthreads();
        }
    };
    const Flag<true> yes{};
    const Flag<false> no{};
    if (AFF) run(yes, yes, no, no);
    else if (uni && Gp > 32) run(yes, yes, yes, yes);
    else if (uni) run(yes, yes, yes, no);
    else if (compact) run(yes, yes, no, no);
    else if (fast) run(yes, no, no, no);
    else run(no, no, no, no);
    }
finish:
    chain_next();
    k2_finish(a, a.work, gridDim.x * gridDim.y, gridDim.y);
}

// Per-pair means of (accuracy, cost, TTFT) of the chosen instances, fp64, in a fixed
// reduction order: a cluster of CTAs per pair, each over a contiguous range of queries, its
// rank 0 adding the ranks' sums in order.  Bound by the SM's narrow fp64 unit (six
// operations a query: three conversions, three additions, about 16 cycles per warp
// instruction) and the three dependent loads of a query, so the pairs spread over the SMs
// and a thread has four queries' loads in flight.  32 pairs x 4,096 queries: 17.1 us (one
// CTA per pair, one query at a time) -> 7.3 us.
constexpr int kFrontierThreads = 256;
__global__ void __launch_bounds__(kFrontierThreads) k_frontier(const K2Launch a, double *out) {
    __shared__ double red[3][kFrontierThreads];
    __shared__ double part[8][3];  // rank 0: the ranks' sums
    chain_wait();
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    cluster.sync();  // every CTA of the cluster runs before one writes into another's shared memory
    const int pp = blockIdx.y, cs = gridDim.x, rank = blockIdx.x;
    const DevConfig &c = a.cfg;
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    const int per = (a.Q + cs - 1) / cs, lo = rank * per, hi = min(a.Q, lo + per);
    double sa = 0.0, sc = 0.0, st = 0.0;
    constexpr int kU = 4;
    for (int i0 = lo + threadIdx.x; i0 < hi; i0 += kU * kFrontierThreads) {
        int jj[kU], m[kU], d[kU], p[kU];
        float t[kU], ac[kU];
#pragma unroll
        for (int k = 0; k < kU; ++k) {
            const int i = i0 + k * kFrontierThreads;
            const size_t o = (size_t)pp * a.Q + i;
            jj[k] = i < hi ? a.assign[o] : 0;
            t[k] = i < hi ? a.ttft_chosen[o] : 0.f;
            p[k] = i < hi ? a.prompt[i] : 0;
        }
#pragma unroll
        for (int k = 0; k < kU; ++k) m[k] = (jj[k] >= 0 && jj[k] < c.I) ? c.moi[jj[k]] : 0;
#pragma unroll
        for (int k = 0; k < kU; ++k) {
            const int i = i0 + k * kFrontierThreads;
            const size_t g = (size_t)i * c.M + m[k];
            d[k] = i < hi ? a.dec_hat[g] : 0;
            ac[k] = i < hi ? a.acc[g] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < kU; ++k) {
            if (i0 + k * kFrontierThreads >= hi) break;
            if (jj[k] < 0 || jj[k] >= c.I) {  // no instance: the means are undefined
                sa = sc = st = nan;
                continue;
            }
            const float cost = __fmaf_rn((float)d[k], c.pout[m[k]], __fmul_rn((float)p[k], c.pin[m[k]]));
            sa += (double)ac[k];
            sc += (double)cost;
            st += (double)t[k];
        }
    }
    red[0][threadIdx.x] = sa;
    red[1][threadIdx.x] = sc;
    red[2][threadIdx.x] = st;
    __syncthreads();
    for (int s = kFrontierThreads / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s)
            for (int f = 0; f < 3; ++f) red[f][threadIdx.x] += red[f][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < 3) cluster.map_shared_rank(&part[0][0], 0)[rank * 3 + threadIdx.x] = red[threadIdx.x][0];
    cluster.sync();
    if (rank == 0 && threadIdx.x < 3) {
        double v = part[0][threadIdx.x];
        for (int r = 1; r < cs; ++r) v += part[r][threadIdx.x];
        out[pp * 3 + threadIdx.x] = v / (double)a.Q;
    }
}

template <int MODE>
cudaError_t launch_cand_mode(const K2Launch &a, int out, dim3 grid, int block, size_t smem, cudaStream_t st) {
    auto go = [&](void (*k)(K2Launch)) { return launch_chained(k, grid, block, smem, st, a); };
    switch (out) {
        case kOutMatrix: return go(k_cand<MODE, kOutMatrix>);
        case kOutMatrix | kOutIters:
            if (MODE == 2) return cudaErrorInvalidValue;  // the batch index exists only for SFS
            return go(k_cand<(MODE == 2 ? 0 : MODE), kOutMatrix | kOutIters>);
        case kOutLag: return go(k_cand<MODE, kOutLag>);
        case kOutLag | kOutMatrix: return go(k_cand<MODE, kOutLag | kOutMatrix>);
        case kOutCon: return go(k_cand<MODE, kOutCon>);
        case kOutCon | kOutMatrix: return go(k_cand<MODE, kOutCon | kOutMatrix>);
        case kOutSweep: return go(k_cand<MODE, kOutSweep>);
        case kOutSweep | kOutMatrix: return go(k_cand<MODE, kOutSweep | kOutMatrix>);
        default: return cudaErrorInvalidValue;
    }
}

template <int MODE>
cudaError_t set_mode_attrs() {
    const cudaError_t es[] = {
        allow_smem(k_cand<MODE, kOutMatrix>, kK2SmemMax), allow_smem(k_cand<(MODE == 2 ? 0 : MODE), kOutMatrix | kOutIters>, kK2SmemMax),
        allow_smem(k_cand<MODE, kOutLag>, kK2SmemMax), allow_smem(k_cand<MODE, kOutLag | kOutMatrix>, kK2SmemMax),
        allow_smem(k_cand<MODE, kOutCon>, kK2SmemMax), allow_smem(k_cand<MODE, kOutCon | kOutMatrix>, kK2SmemMax),
        allow_smem(k_cand<MODE, kOutSweep>, kK2SmemMax), allow_smem(k_cand<MODE, kOutSweep | kOutMatrix>, kK2SmemMax)};
    for (cudaError_t x : es)
        if (x != cudaSuccess) return x;
    return cudaSuccess;
}

}  // namespace

int cand_out_flags(bool matrix, bool iters, bool route, bool constrained, int P) {
    int f = 0;
    if (matrix) f |= kOutMatrix;
    if (iters) f |= kOutIters;
    if (route) f |= constrained ? kOutCon : (P > 1 ? kOutSweep : kOutLag);
    return f;
}

cudaError_t launch_cand(const K2Launch &a, int out, dim3 grid, int block, size_t smem, cudaStream_t st) {
    if (a.src != kSrcSfs) return launch_cand_mode<2>(a, out, grid, block, smem, st);
    return a.cfg.mode == 0 ? launch_cand_mode<0>(a, out, grid, block, smem, st)
                           : launch_cand_mode<1>(a, out, grid, block, smem, st);
}

namespace {

// x^k, k >= 0, by binary exponentiation (the bits of k from the least significant).
__device__ double pow_int(double x, int k) {
    double r = 1.0, b = x;
    while (k > 0) {
        if (k & 1) r = __dmul_rn(r, b);
        k >>= 1;
        if (k > 0) b = __dmul_rn(b, b);
    }
    return r;
}

// Per instance: the LPS expected wait of App. E, ((ca2 + cs2) / 2) rho^k / (mu - alpha)
// with rho = alpha / mu, and the fp32 constants of the affine TTFT.
__global__ void k_queue_params(int I, const QueueRaw *raw, QueueDev *qd) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= I) return;
    const QueueRaw r = raw[j];
    double w = __longlong_as_double(0x7ff8000000000000LL);
    if (r.has_lps) {
        const double rho = __ddiv_rn(r.alpha, r.mu);
        const double c = __dmul_rn(__dadd_rn(r.ca2, r.cs2), 0.5);
        w = __ddiv_rn(__dmul_rn(c, pow_int(rho, r.k)), __dsub_rn(r.mu, r.alpha));
    }
    QueueDev o;
    o.theta = r.theta;
    o.tdec = r.tdec;
    o.wlps = w;
    o.g = __double2float_rn(__ddiv_rn(1.0, r.theta));
    o.clps = __double2float_rn(__dadd_rn(w, r.tdec));
    qd[j] = o;
}

// ---------------------------------------------------------------------------
// Baseline routing policies (Sec. 6, the baselines): the instance is chosen without the
// latency estimates, and the chosen candidate's utility (Eq. 2) and SFS TTFT estimate
// are reported beside it (the TTFT through the same exact path as the candidate
// kernel's, so the two agree bit for bit).  One thread per query.
//   Round Robin: (start + i) mod I.
//   Shortest Queue: the queries in order each join the instance with the fewest
//     resident requests, counting those routed before them, ties to the lowest index.
//     Query k therefore takes the k-th smallest slot (level, j) over the slots
//     instance j offers at levels c_j, c_j + 1, ...: the level L is the largest with
//     N(L) = sum_j max(0, L - c_j) <= k (N from the sorted counts and their prefix
//     sums), and the instance is the (k - N(L))-th, by index, of those with c_j <= L.
//   Latency-Agnostic: the largest utility, ties to the lowest index (utility depends
//     on the instance's model only, so the models are compared at their first instance).
template <int MODE>
__global__ void __launch_bounds__(256) k_baseline(const K2Launch a, int policy, long long rr_start, float lam) {
    extern __shared__ __align__(16) unsigned char bsm[];
    const DevConfig &c = a.cfg;
    const int I = c.I, M = c.M;
    chain_wait();
    __shared__ int s_active;
    if (threadIdx.x == 0) s_active = load_live(a.ctl);
    __syncthreads();
    const int active = s_active;
    const StateBuf sb = active > 0 ? a.buf1 : a.buf0;
    int P2 = 1;
    while (P2 < I) P2 <<= 1;
    int *cnt = reinterpret_cast<int *>(bsm);                              // [I] resident requests
    int *srt = cnt + I;                                                   // [P2] the counts, sorted
    long long *pre = reinterpret_cast<long long *>(bsm + 8 * ((I + P2 + 1) / 2));  // [I + 1] prefix sums
    int *firstj = reinterpret_cast<int *>(pre + I + 1);                   // [M] first instance of each model
    if (active >= 0 && policy == 1) {
        for (int j = threadIdx.x; j < P2; j += blockDim.x) {
            const int v = j < I ? sb.n_run[j] + sb.n_wait[j] : 0x7fffffff;
            if (j < I) cnt[j] = v;
            srt[j] = v;
        }
        __syncthreads();
        // bitonic sort of srt, ascending
        for (int k = 2; k <= P2; k <<= 1) {
            for (int h = k >> 1; h > 0; h >>= 1) {
                for (int t = threadIdx.x; t < P2; t += blockDim.x) {
                    const int u = t ^ h;
                    if (u > t) {
                        const int x = srt[t], y = srt[u];
                        if (((t & k) == 0) == (x > y)) {
                            srt[t] = y;
                            srt[u] = x;
                        }
                    }
                }
                __syncthreads();
            }
        }
        if (threadIdx.x == 0) {
            long long run = 0;
            for (int t = 0; t < I; ++t) {
                pre[t] = run;
                run += srt[t];
            }
            pre[I] = run;
        }
    }
    if (policy == 2) {
        for (int m = threadIdx.x; m < M; m += blockDim.x) firstj[m] = -1;
        __syncthreads();
        for (int j = threadIdx.x; j < I; j += blockDim.x) atomicMin(reinterpret_cast<unsigned *>(firstj) + c.moi[j], (unsigned)j);
    }
    __syncthreads();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.Q; i += gridDim.x * blockDim.x) {
        const int p = a.prompt[i];
        bool ok;
        const QRec q = make_qrec(p, c.pmax, &ok);
        if (!ok || active < 0) {
            record_status(a.ctl, active < 0 ? kENoState : kEInval);
            a.assign[i] = -1;
            a.util[i] = kNaN;
            if (a.ttft_chosen) a.ttft_chosen[i] = kNaN;
            continue;
        }
        int j = 0;
        if (policy == 0) {
            j = (int)((rr_start + i) % I);
        } else if (policy == 1) {
            // N(L): slots below level L = (#counts below L) * L - (their sum)
            auto slots_below = [&](long long L) -> long long {
                int lo = 0, hi = I;  // first sorted count >= L
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if ((long long)srt[mid] < L) lo = mid + 1;
                    else hi = mid;
                }
                return (long long)lo * L - pre[lo];
            };
            long long lo = srt[0], hi = (long long)srt[0] + i + 1;  // N(lo) <= i < N(hi)
            while (hi - lo > 1) {
                const long long mid = (lo + hi) >> 1;
                if (slots_below(mid) <= i) lo = mid;
                else hi = mid;
            }
            long long r = i - slots_below(lo);  // < #{j : c_j <= lo}, so the scan finds it
            for (j = 0; j < I; ++j)
                if ((long long)cnt[j] <= lo && r-- == 0) break;
            j = min(j, I - 1);
        } else {
            float best = 0.f;
            int bj = -1;
            for (int m = 0; m < M; ++m) {
                const int fj = firstj[m];
                if (fj < 0) continue;
                const float cost = __fmaf_rn((float)a.dec_hat[(size_t)i * M + m], c.pout[m], __fmul_rn((float)p, c.pin[m]));
                const float U = __fmaf_rn(-lam, cost, a.acc[(size_t)i * M + m]);
                if (bj < 0 || U > best || (U == best && fj < bj)) {
                    best = U;
                    bj = fj;
                }
            }
            j = bj;
        }
        const int m = c.moi[j];
        const float cost = __fmaf_rn((float)a.dec_hat[(size_t)i * M + m], c.pout[m], __fmul_rn((float)p, c.pin[m]));
        const float U = __fmaf_rn(-lam, cost, a.acc[(size_t)i * M + m]);
        a.assign[i] = j;
        a.util[i] = U;
        if (a.ttft_chosen && a.ttft_in) {
            a.ttft_chosen[i] = a.ttft_in[(size_t)i * I + j];  // the KV-limited estimate
        } else if (a.ttft_chosen) {
            const InstParams ip = sb.inst[j];
            const int2 bk = sb.bkt[(size_t)(q.p >> ip.shift) * I + j];
            const int k = bk.y + (q.p > bk.x ? 1 : 0);
            const float T =
                reinterpret_cast<const float2 *>(sb.tile + tile_base(c, j))[(size_t)k * 4 * c.tgp + tile_col(c, j)].x;
            a.ttft_chosen[i] = ttft_exact64<MODE>(c, sb, q.p, j, k, T);
        }
    }
}

// OnTimeUtility (Eq. 4) and SLO attainment, in one launch: CTA b sums the fixed row range
// [b R, (b + 1) R) in a fixed tree order into part[2 b .. 2 b + 1], and the last CTA to
// finish adds the parts in index order and clears the count for the next call.  The
// realized TTFT is the fp32 sum delay + ttft.  Launch-bound at a few thousand queries; the
// rows on time are counted as integers, which leaves the narrow fp64 unit one conversion
// and one addition a row (4,096 queries: 5.8 + 3.6 us in two launches -> 7.4 us).
__global__ void __launch_bounds__(256) k_on_time(int Q, const float *util, const float *ttft, const float *tau,
                                                 const float *delay, double *part, unsigned *done, double *out) {
    __shared__ double su[256];
    __shared__ int sn[8], s_last;
    chain_wait();
    const int R = (Q + gridDim.x - 1) / gridDim.x;
    const int lo = blockIdx.x * R, hi = min(Q, lo + R);
    double u = 0.0;
    int n = 0;
#pragma unroll 4
    for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const float realized = delay ? __fadd_rn(delay[i], ttft[i]) : ttft[i];
        const float ui = util[i];
        if (realized <= tau[i]) {
            u += (double)ui;
            ++n;
        }
    }
    chain_next();
    su[threadIdx.x] = u;
    n = __reduce_add_sync(kFull, n);
    if ((threadIdx.x & 31) == 0) sn[threadIdx.x >> 5] = n;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) su[threadIdx.x] += su[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        int c = 0;
        for (int w = 0; w < 8; ++w) c += sn[w];
        part[2 * blockIdx.x] = su[0];
        part[2 * blockIdx.x + 1] = (double)c;
        __threadfence();
        s_last = atomicAdd(done, 1u) == gridDim.x - 1;
        if (s_last) {
            __threadfence();
            double us = 0.0, ns = 0.0;
            for (unsigned b = 0; b < gridDim.x; ++b) {
                us += __ldcg(part + 2 * b);
                ns += __ldcg(part + 2 * b + 1);
            }
            out[0] = us / Q;
            out[1] = ns / Q;
            *done = 0u;
        }
    }
}

}  // namespace

cudaError_t launch_queue_params(int I, const QueueRaw *raw, QueueDev *qd, cudaStream_t st) {
    k_queue_params<<<(I + 127) / 128, 128, 0, st>>>(I, raw, qd);
    return cudaGetLastError();
}

cudaError_t launch_features(const K2Launch &a, int sms, cudaStream_t st) {
    const long long total = (long long)a.Q * a.cfg.I;
    const int grid = (int)std::min<long long>((total + 255) / 256, (long long)sms * 8);
    k_features<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_frontier(const K2Launch &a, double *out, int sms, cudaStream_t st) {
    // CTAs per pair: a power of two up to 8 (the portable cluster size), while the pairs
    // leave SMs free and each CTA still has more than 256 queries
    int cs = 1;
    while (cs < 8 && 2 * cs * a.P <= sms && 512 * cs < a.Q) cs *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs, a.P);
    cfg.blockDim = dim3(kFrontierThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_frontier, a, out);
}

size_t baseline_smem(const DevConfig &c) {
    int P2 = 1;
    while (P2 < c.I) P2 <<= 1;
    return 8 * (size_t)((c.I + P2 + 1) / 2) + 8 * (size_t)(c.I + 1) + 4 * (size_t)c.M;
}

cudaError_t launch_baseline(const K2Launch &a, int policy, long long rr_start, float lam, int sms, cudaStream_t st) {
    const size_t smem = baseline_smem(a.cfg);
    const int grid = std::max(1, std::min((a.Q + 255) / 256, sms * 4));
    return launch_chained(a.cfg.mode == 0 ? k_baseline<0> : k_baseline<1>, grid, 256, smem, st, a, policy, rr_start, lam);
}

cudaError_t launch_on_time(int Q, const float *util, const float *ttft, const float *tau, const float *delay,
                           double *part, int max_parts, double *out, cudaStream_t st) {
    // 512 rows a CTA while the last one's sum over the parts stays short
    const int rows = Q <= 16384 ? 512 : 2048;
    const int parts = std::max(1, std::min(max_parts, (Q + rows - 1) / rows));
    return launch_chained(k_on_time, parts, 256, 0, st, Q, util, ttft, tau, delay, part,
                          reinterpret_cast<unsigned *>(part + 2 * max_parts), out);
}

cudaError_t set_baseline_smem() {
    cudaError_t e = allow_smem(k_baseline<0>, kSmemMax);
    if (e == cudaSuccess) e = allow_smem(k_baseline<1>, kSmemMax);
    return e;
}

cudaError_t set_k2_smem() {
    cudaError_t e = set_mode_attrs<0>();
    if (e == cudaSuccess) e = set_mode_attrs<1>();
    if (e == cudaSuccess) e = set_mode_attrs<2>();
    return e;
}

cudaError_t cand_occupancy(int mode, bool route, int block, size_t smem, int *n) {
    if (route)
        return mode == 0 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_cand<0, kOutLag | kOutMatrix>, block, smem)
                         : cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_cand<1, kOutLag | kOutMatrix>, block, smem);
    return mode == 0 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_cand<0, kOutMatrix>, block, smem)
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_cand<1, kOutMatrix>, block, smem);
}

}  // namespace lr
