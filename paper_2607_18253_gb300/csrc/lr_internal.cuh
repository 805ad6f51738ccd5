// Library-internal layout shared by the host API and the kernels.
//
// Data layout in HBM (all per-instance tables are [row][I], instance-minor, so
// that consecutive threads of a CTA -- which own consecutive instances -- read
// consecutive words):
//
//   config      : model_of_instance[I], B[I], S[I], shift[I], nb[I], coef[M][5],
//                 price_in[M], price_out[M]
//   buffer 0/1  : a snapshot copy (SoA, row stride cap) plus its summary:
//                 inst[I]           InstParams (admission batch, totals, splits)
//                 bkt[NBH][I]       int2 (in-bucket boundary, boundaries below)
//                 f2[KPH][I], f3[KPH][I], rcum[KPH][I]
//                 tile[T]           per tile of 4*tgp instances, the candidate
//                                   kernel's shared-memory image (see below)
//   control     : live buffer index, sticky status word, load error, CTA counter
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace lr {

constexpr int kKMax = 64;               // table entries per instance (k = 0..kp-1)
constexpr int kNBMax = 2 * kKMax + 2;   // prompt-length buckets per instance
constexpr int kBig = 0x7fffffff;        // "never" / "no boundary"
constexpr int kSplitBits = 20;          // low part of the exact fp32 splits
constexpr long long kFastLimit = 1LL << 44;  // integers below this split exactly
constexpr int kMaxPairs = 64;

// Return codes (mirror include/latency_router.h).
enum : int { kOk = 0, kEInval = 1, kENoMem = 2, kECuda = 3, kECapacity = 4, kETraj = 5, kEState = 6,
             kENoState = 7 };

struct InstParams {      // 64 bytes
    int32_t la;          // batch at which a query appended now is admitted
    int32_t kp;          // number of table entries
    int32_t shift;       // log2 of the bucket width
    int32_t fast;        // 1: every feature of this instance splits exactly into fp32
    long long f1tot;     // prefill tokens of all residents
    long long f4tot;     // prefill attention pairs of all residents
    float h1, l1, h4, l4;  // exact fp32 high/low parts of f1tot and f4tot
    int32_t r0;          // budget left to the query in its admission batch
    int32_t pad[3];
};

struct DevConfig {
    int32_t I, M, capR, capW;
    int32_t pmax, mode, max_iters, tgp;     // tgp: thread groups per instance tile of the candidate kernel
    int32_t kph, nbh;                       // table row counts (host bounds over instances)
    int32_t near;                           // k* <= 1 on every instance for a prompt up to this
    const int32_t *moi, *B, *S, *shift, *nb;
    const float *coef, *pin, *pout;
};

// KV-limited simulation (App. F): one batch of an instance's residents alone, from
// the first batch in which a query could be admitted (the waiting queue empty after
// admissions, budget and a seat left).  64 bytes.
// The walk's fields are clamped to 32 bits, which no comparison with a query's own blocks
// or prompt (at most 2^20 + 1) can tell.
struct __align__(16) KvRec {
    long long cf[4];             // residents' features 1..4 summed from the first record through this one
    int32_t slack;               // least (free blocks - blocks needed) over the running scan; < 0: a preemption
    int32_t far;                 // free blocks after the running scan
    int32_t thr;                 // a waiting query with prompt p is admitted in this batch iff p <= thr
    int32_t bar, bl;             // budget left after the running scan, after admissions
    int32_t pad[3];
};
// Per instance: the residents' features before the first record, and the records' extent.
struct __align__(16) KvInst {
    long long fcum[5];
    int32_t la0;   // batch of record 0
    int32_t nrec;  // records written
    int32_t done;  // 1: no resident is left after the last record (later batches are empty)
    int32_t pad;
};
struct KvLimits {
    const int32_t *bs;     // [I] block size (tokens), at most kKvMaxBlock
    const long long *nb;   // [I] blocks
    const long long *mctx; // [I] context limit
    int32_t horizon;       // records per instance
    int32_t hist;          // the largest block size: entries of the load's residue histogram
};
constexpr int kKvMaxBlock = 4096;
constexpr int kKvCal = 1024;  // batches covered by the load's end calendar

struct StateBuf {
    int32_t *n_run, *run_ctx, *run_pre, *run_dec, *n_wait, *wait_pre, *wait_dec;
    double *clock;  // [I] end time of the instance's last completed batch (s)
    InstParams *inst;
    int2 *bkt;
    unsigned char *tile;  // candidate-kernel tile blocks
    long long *f2, *f3;
    int32_t *rcum;
    KvInst *kvi;   // [I], with KV limits
    KvRec *kvr;    // [I][horizon], with KV limits
    int32_t *kvp;  // [I][horizon] running maximum of the records' thr (clamped to int32), with KV limits
    // first-token tracking (lr_track_first_tokens): each request's id until its first output
    // token, else -1; written by the stream step only (a snapshot load makes every request -1)
    int32_t *run_id, *wait_id;  // [I][capR], [I][capW]
};

// Copies of the live-buffer index, each in its own 128-byte line: the CTAs of a
// candidate-kernel launch (hundreds, all starting at once) read different copies
// instead of queueing on one line.
constexpr int kLiveReps = 64;
struct __align__(128) DevCtl {
    int32_t active;      // live buffer, -1 before the first successful load
    int32_t status;      // first error since the last lr_status
    int32_t load_err;    // error of the load in progress
    uint32_t done_ctas;  // K1 completion counter
    int32_t pad[28];
    int32_t live[kLiveReps][32];  // live[r][0]: copies of active
};

struct StateIn {
    const int32_t *n_run, *run_ctx, *run_pre, *run_dec, *n_wait, *wait_pre, *wait_dec;
    const double *clock;  // may be null: clocks start at 0
};

// Programmatic dependent launch between the library's kernels: a kernel launched with
// launch_chained may be scheduled while its predecessor in the stream finishes, and waits
// in chain_wait -- every thread's first statement that touches global memory written after
// lr_create comes after it -- until the predecessor has completed and its writes are
// visible, exactly as without it (so a chain of such launches stays ordered).  chain_next
// lets the successor be scheduled; it stands near a kernel's end, so that the successor's
// CTAs take no room on the SMs for longer than the launch itself takes.  What it hides is
// launch latency: about a microsecond between two of the library's kernels (a 64-instance
// decision, three launches: 36 -> 30 us; 50,001 x 250 estimates back to back 16.2 -> 12.9 us).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
cudaError_t launch_chained(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const A &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, P(args)...);
}

// Lets kernel f be launched with up to `most` bytes of dynamic shared memory.  The limit belongs
// to the process's kernel, not to one lr_ctx, so `most` is a constant, the most that lr_create or
// lr_set_kv_limits lets any context need: no context takes away what another launches with.
constexpr size_t kSmemMax = 200 * 1024;    // the loads, the stream steps, the baselines
constexpr size_t kK2SmemMax = 224 * 1024;  // the candidate kernel
template <typename F>
cudaError_t allow_smem(F *f, size_t most) {
    return cudaFuncSetAttribute((const void *)f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// K1 asks for the whole shared-memory carve-out as well: with one that fits its own CTAs alone, an
// SM could not take a larger CTA of a call on another stream before it was idle (routes beside a
// load, 16,384 x 61 / 256 / 640: 12.4 / 17.6 / 55 -> 11.5 / 14.1 / 44 us).  Not the KV load, whose
// few warps are the longer part and lose more to company (65,536 x 256 186 -> 200 us).
template <typename F>
cudaError_t beside_smem(F *f, size_t most) {
    cudaError_t e = allow_smem(f, most);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return e;
}

// The live-buffer index with acquire ordering: reads of the buffer it names see
// everything the load that published it wrote (it may have finished on another stream).
__device__ __forceinline__ int32_t load_acquire(const int32_t *p) {
    int32_t v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The end of a load's CTA (every thread calls it): the last CTA to finish publishes the
// new live buffer if every instance succeeded -- the index and its copies, which readers
// take with acquire loads -- and resets the load's control words.  One fence and one
// atomic a CTA; the copies are stored by a warp, two a lane (one thread storing 64 words
// between four atomics cost a load about a microsecond).
__device__ __forceinline__ void finish_load(DevCtl *ctl, int dst, unsigned ctas) {
    __shared__ int s_publish;
    __syncthreads();
    chain_next();
    if (threadIdx.x == 0) {
        __threadfence();
        int v = -1;
        if (atomicAdd(&ctl->done_ctas, 1u) == ctas - 1) {
            __threadfence();
            if (*(volatile int32_t *)&ctl->load_err == 0) v = dst;
            *(volatile int32_t *)&ctl->load_err = 0;
            *(volatile uint32_t *)&ctl->done_ctas = 0u;
        }
        s_publish = v;
    }
    __syncthreads();
    const int v = s_publish;
    if (v >= 0 && threadIdx.x < 32) {
        __threadfence();  // what this CTA's thread 0 acquired precedes the stores
        if (threadIdx.x == 0) asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(&ctl->active), "r"(v) : "memory");
        for (int r = threadIdx.x; r < kLiveReps; r += 32)
            asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(&ctl->live[r][0]), "r"(v) : "memory");
    }
}

// The live-buffer index from this CTA's copy, with acquire ordering.
__device__ __forceinline__ int32_t load_live(const DevCtl *ctl) {
    return load_acquire(&ctl->live[blockIdx.x % kLiveReps][0]);
}

__device__ __forceinline__ void record_status(DevCtl *ctl, int code) {
    atomicCAS(&ctl->status, 0, code);
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Sum over the warp, modulo 2^64, on every lane: three reductions of 22-bit pieces (each
// sum stays below 2^32) instead of five rounds of two shuffles and a 64-bit addition.
__device__ __forceinline__ long long warp_sum64(long long v) {
    const unsigned long long u = (unsigned long long)v;
    const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)u & 0x3fffffu);
    const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 22) & 0x3fffffu);
    const unsigned s2 = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 44));
    return (long long)(s0 + ((unsigned long long)s1 << 22) + ((unsigned long long)s2 << 44));
}

// Division by an instance's block size, which the KV kernels repeat many times a batch:
// unsigned n / d for any 32-bit n as a multiply-high and shifts (Granlund and
// Montgomery's method for invariant divisors: l = ceil(log2 d), m = floor(2^32 (2^l - d)
// / d) + 1, q = (t + ((n - t) >> 1)) >> (l - 1) with t = mulhi(m, n); d = 1 takes
// shifts of 0).
struct Div32 {
    unsigned d, m;
    int s1, s2;
};
__device__ __forceinline__ Div32 make_div32(int d) {
    const unsigned ud = (unsigned)d;
    const int l = ud <= 1u ? 0 : 32 - __clz((int)(ud - 1u));
    Div32 v;
    v.d = ud;
    v.m = (unsigned)((((1ull << 32) * ((1ull << l) - ud)) / ud) + 1ull);
    v.s1 = min(l, 1);
    v.s2 = max(l - 1, 0);
    return v;
}
__device__ __forceinline__ unsigned udiv32(const Div32 &v, unsigned n) {
    const unsigned t = __umulhi(v.m, n);
    return (t + ((n - t) >> v.s1)) >> v.s2;
}
// ceil(c / d) for 0 <= c < 2^31
__device__ __forceinline__ int dblk(const Div32 &v, int c) { return (int)udiv32(v, (unsigned)c + v.d - 1u); }
// x mod d in [0, d) for any int x
__device__ __forceinline__ int dres(const Div32 &v, int x) {
    if (x >= 0) return (int)((unsigned)x - udiv32(v, (unsigned)x) * v.d);
    const unsigned ax = (unsigned)(-(long long)x);
    const unsigned r = ax - udiv32(v, ax) * v.d;
    return r == 0u ? 0 : (int)(v.d - r);
}

// Candidate-kernel tile block: everything one CTA of the candidate kernel needs about
// its tile of 4 * tgp instances, laid out as that CTA's shared memory so that a single
// bulk copy brings it in.  Instance j0 + 4g + u of the tile sits in column u * tgp + g:
//   entA [kph][4][tgp]    8 bytes: T_k (fp32) and X_k, which is f3_k (fp32) when the
//                         first token comes with the last chunk, else F3_k as an int32
//                         (valid when the instance is compact: F3_k + pmax < 2^31 and
//                         F1tot + pmax <= 2^24)
//   entB [kph][4][tgp]    8 bytes: H3_k, L3_k, the exact fp32 split of F3_k
//   bkt  [nbh][tgp][4]    uint32: (in-bucket boundary << 7) | boundaries below, the
//                         boundary 2^24 - 1 when the bucket holds none; a thread's four
//                         instances are adjacent (one 16-byte load when they share the
//                         bucket width)
//   scal [kScal][4][tgp]  32-bit scalars, fields kSc*
// A warp reads a table as one dense 4- or 8-byte word per lane (1 or 2 shared-memory
// wavefronts); a compact CTA reads only entA.
constexpr int kScal = 13;
enum : int { kScShift = 0, kScH1, kScL1, kScH4, kScL4, kScB1p, kScB2, kScB3, kScModel, kScLa, kScFast, kScCompact, kScR0 };
constexpr uint32_t kBktNone = (1u << 24) - 1;  // bucket boundary field of a bucket without one
__host__ __device__ inline size_t tile_enta_bytes(const DevConfig &c) { return (size_t)c.kph * 4 * c.tgp * 8; }
__host__ __device__ inline size_t tile_ent_bytes(const DevConfig &c) { return 2 * tile_enta_bytes(c); }
__host__ __device__ inline size_t tile_bkt_bytes(const DevConfig &c) {
    return ((size_t)c.nbh * 4 * c.tgp * 4 + 15) & ~(size_t)15;
}
__host__ __device__ inline size_t tile_bytes(const DevConfig &c) {
    return tile_ent_bytes(c) + tile_bkt_bytes(c) + (size_t)kScal * 4 * c.tgp * 4;
}
// The head of the candidate kernel's shared memory: the tile block, or (an affine source with
// rows that are not whole 16-byte words) 1 KB a warp in which stores are put in order.
__host__ __device__ inline size_t k2_head_bytes(const DevConfig &c, int block) {
    const size_t tb = tile_bytes(c), ord = c.I % 4 != 0 && c.tgp >= 32 ? (size_t)block * 32 : 0;
    return tb > ord ? tb : ord;
}
__host__ __device__ inline int tile_count(const DevConfig &c) { return (c.I + 4 * c.tgp - 1) / (4 * c.tgp); }
// Byte offset of instance j's column within its tile block, and the tile's base.
__host__ __device__ inline size_t tile_base(const DevConfig &c, int j) { return (size_t)(j / (4 * c.tgp)) * tile_bytes(c); }
__host__ __device__ inline int tile_col(const DevConfig &c, int j) {
    const int jj = j % (4 * c.tgp);
    return (jj & 3) * c.tgp + (jj >> 2);
}
// Columns past the last instance, written once so that they read as empty instances.
cudaError_t launch_tile_pad(const DevConfig &c, unsigned char *tile, cudaStream_t st);

// Calibration of the batch-time coefficients (lr_calibrate.cu).
constexpr int kCalCols = 5;
constexpr int kCalAcc = 21;        // per model: 15 sums of the upper triangle of G, 5 of b, the row count
constexpr int kCalMaxModels = 128;  // shared-memory sums of one CTA (128-bit each)
constexpr double kCalTimeScale = 17592186044416.0;  // 2^44: times in 2^-44 s fixed point
constexpr double kCalTimeMax = 524288.0;            // 2^19 s
constexpr int kCalThreads = 512;                    // one CTA per SM
constexpr int kCalConsumerWarps = kCalThreads / 32 - 1;  // the last warp issues the copies
constexpr int kCalTile = 2 * 32 * kCalConsumerWarps;     // rows per staged tile, two a consumer lane (16-byte copies)
constexpr int kCalStagesMax = 3;                    // tiles in flight per CTA
constexpr int kCalFlushRows = 128;                  // rows a lane sums in 64 bits between flushes
constexpr size_t kCalSmemMax = 223 * 1024;           // (the kernel's static words need 4 KB)
constexpr size_t kCalStageBytes = (size_t)kCalTile * (kCalCols * 8 + 8 + 4);
constexpr int kCalFlushSums = 26;  // a warp flush's sums: 15 of G, 5 + 5 halves of b, the row count
// the CTA's shared sums: 128-bit [M][kCalAcc] and the flushes' carry-save words [M][kCalFlushSums]
__host__ __device__ inline size_t cal_sums_bytes(int M) { return (size_t)M * (kCalAcc + kCalFlushSums) * 16; }
// the calibration's device words: the sums [M][kCalAcc][2] and the CTA counter of the
// last-CTA solve (zero between calls)
__host__ __device__ inline size_t cal_acc_words(int M) { return (size_t)M * kCalAcc * 2 + 2; }
cudaError_t launch_calibrate(long long N, const long long *F, const int32_t *model, const double *time, int M,
                             int shared_beta1, unsigned long long *acc, double *coef, DevCtl *ctl, int grid,
                             cudaStream_t st);
cudaError_t set_calib_smem();

// Launch helpers implemented in the kernel translation units.
struct K1Launch {
    DevConfig cfg;
    StateBuf buf0, buf1;
    DevCtl *ctl;
    StateIn in;
};
cudaError_t launch_trajectory(const K1Launch &a, int grid, int block, size_t smem, cudaStream_t st);
cudaError_t set_k1_smem();
constexpr int kK1Warps = 4;

// KV-limited load (residents alone, records) and estimate (per-candidate walk).
struct KvLoad {
    DevConfig cfg;
    KvLimits kv;
    StateBuf buf0, buf1;
    DevCtl *ctl;
    StateIn in;
};
constexpr int kKvWarps = 4;
// shared memory per warp of the KV load: the running list (context, prefill, decode,
// blocks) and the waiting ring (prefill, decode) over capR + capW requests, the end
// calendar (links and blocks at the end per request, kKvCal heads) and the residue
// histogram, 16-byte aligned
__host__ __device__ inline size_t kv_smem_per_warp(const DevConfig &c, int hist) {
    return (sizeof(int32_t) * (8 * (size_t)(c.capR + c.capW) + kKvCal + hist + 16) + 15) & ~(size_t)15;
}
// warps: instances per CTA, 1 .. kKvWarps
cudaError_t launch_kv_load(const KvLoad &a, int grid, int warps, size_t smem, cudaStream_t st);
cudaError_t set_kv_smem();
struct KvEst {
    DevConfig cfg;
    KvLimits kv;
    StateBuf buf0, buf1;
    DevCtl *ctl;
    int32_t Q;
    const int32_t *prompt;
    float *ttft;
    int32_t *first_batch;
    long long *features;
    // the call's queries sorted by prompt length (counting sort over kKvBuckets
    // buckets: invalid lengths, then valid ones >> shift); with shift 0 one
    // query per length is estimated and the others copy its rows
    int32_t *cnt, *start, *run, *uid;  // [kKvBuckets]
    int32_t *nu;                       // [1] distinct lengths
    int32_t *tsum;                     // [2][kKvScanTiles] per-tile bucket sums of the scan
    int32_t *order, *leaders;          // [max_queries]
    int32_t *claim;                    // [ceil(I / 8)] the estimate's block counters per instance group
};
constexpr int kKvBuckets = 1 << 16;
constexpr int kKvScanTiles = kKvBuckets / 4096;  // the bucket scan's tiles, one CTA each
// expand: every query's row is written; else, when the call is sorted (*leaders set), only the
// row of the first query of each length, order[start[p]]
cudaError_t launch_kv_estimate(const KvEst &a, int sms, bool expand, bool *leaders, cudaStream_t st);

// Batches covered by K1's completion calendar; decoders ending later are
// tracked by scanning the decoder list.
constexpr int kCalendar = 2048;

// Shared memory of one K1 warp (in int32 words, a multiple of 4): calendar and
// its bitmap, the decoder list (first batch, last batch, context offset, pad),
// the waiting queue's prompt prefix sums and decode lengths, and the budgets.
__host__ __device__ inline size_t trajectory_smem_per_warp(const DevConfig &c) {
    const size_t words = (size_t)kCalendar + kCalendar / 32 + 4 * (size_t)(c.capR + c.capW) +
                         (size_t)(c.capW + 2) + (size_t)(c.capW + 1) + (size_t)c.kph + 32;
    return sizeof(int32_t) * ((words + 3) & ~(size_t)3);
}

// Average-case TTFT sources (Sec. 4, App. E): per-instance parameters as given
// and the derived constants of t = fma(p, g, C).
// kSrcMatrix (internal): the times come from a [Q][I] matrix already computed (the
// KV-limited estimate), read by the candidate kernel's affine mode
enum : int { kSrcSfs = 0, kSrcThroughput = 1, kSrcLps = 2, kSrcMatrix = 3 };
struct QueueRaw {      // 64 bytes, copied from the caller's arrays
    double theta, tdec, alpha, mu, ca2, cs2;
    int32_t k, has_lps;
    int32_t pad[2];
};
struct QueueDev {      // 32 bytes
    double theta, tdec;
    double wlps;       // LPS expected wait (NaN without queue rates)
    float g;           // fp32(1 / theta)
    float clps;        // fp32(wlps + tdec)
};
cudaError_t launch_queue_params(int I, const QueueRaw *raw, QueueDev *qd, cudaStream_t st);

struct K2Launch {
    DevConfig cfg;
    StateBuf buf0, buf1;
    DevCtl *ctl;
    int32_t Q;
    const int32_t *prompt;
    // estimate outputs
    float *ttft;
    int32_t *first_batch;
    long long *features;
    // route inputs / outputs
    const int32_t *dec_hat;
    const float *acc;
    const float *tau;
    int32_t P;
    float lam[kMaxPairs];
    float mu[kMaxPairs];
    int32_t *assign;
    float *util;
    float *ttft_chosen;
    // launch shape: Gp thread groups of four instances per row (a power of two up
    // to 32, else a multiple of 32), QS rows in flight, QT rows per staged chunk
    int32_t Gp, QS, QT, vec_ok;
    int32_t vec_first;  // first_batch rows are whole, aligned 16-byte words
    int32_t least, share;  // a claim: the fewest rows, and 1 / share of an equal part of those left
    int32_t pg, sp;  // sweep: lanes by pair and lanes that share a row's instances (powers of two)
    // TTFT source (kSrc*) and, for the average-case ones, the instance constants
    int32_t src;
    const QueueDev *qd;
    const float *ttft_in;  // kSrcMatrix: [Q][I]
    // kSrcMatrix, or null: the row of a query of p tokens is lead_order[lead_start[p]] (0 for an
    // invalid length), not its own
    const int32_t *lead_start, *lead_order;
    // [0]: CTAs finished; [1 + tile]: query rows of the tile claimed past the static
    // ones.  Zero before a launch; the last CTA to finish clears them for the next.
    uint32_t *work;
    // CTAs (per tile) that start with a static chunk of first_rows query rows
    int32_t first_ctas, first_rows;
};
// Entries of the candidate kernel's work counters for I instances.
inline int k2_work_words(int I) { return (I + 1023) / 1024 + 2; }
int cand_out_flags(bool matrix, bool iters, bool route, bool constrained, int P);
cudaError_t launch_cand(const K2Launch &a, int out, dim3 grid, int block, size_t smem, cudaStream_t st);
cudaError_t launch_features(const K2Launch &a, int sms, cudaStream_t st);
cudaError_t launch_frontier(const K2Launch &a, double *out, int sms, cudaStream_t st);
// Baseline routing policies (0 Round Robin, 1 Shortest Queue, 2 Latency-Agnostic) and
// the stream metrics (OnTimeUtility, SLO attainment) over routed queries.
size_t baseline_smem(const DevConfig &c);
cudaError_t set_baseline_smem();
cudaError_t launch_baseline(const K2Launch &a, int policy, long long rr_start, float lam, int sms, cudaStream_t st);
constexpr int kOnTimeParts = 1024;
cudaError_t launch_on_time(int Q, const float *util, const float *ttft, const float *tau, const float *delay,
                           double *part, int max_parts, double *out, cudaStream_t st);
cudaError_t cand_occupancy(int mode, bool route, int block, size_t smem, int *blocks_per_sm);
cudaError_t set_k2_smem();
constexpr int kK2Block = 256;                // route: three CTAs per SM, one fits beside a load's CTA
constexpr size_t kK2SmemTarget = 72 * 1024;  // three CTAs per SM
constexpr int kK2EstBlock = 512;             // estimate alone: one CTA per SM, one tile copy per SM
constexpr size_t kK2EstSmemTarget = 120 * 1024;

// K3: append routed queries and advance every instance to t_now (online stream).
struct K3Launch {
    DevConfig cfg;
    StateBuf buf0, buf1;  // the live one is read
    StateBuf scratch;     // receives the advanced snapshot (then summarized by K1)
    DevCtl *ctl;
    int32_t Q;
    int32_t dec_cols;  // 1: dec[i]; M: dec[i][model of the chosen instance]
    const int32_t *assign, *prompt, *dec;
    double t_now;
    // first-token tracking: the appended query i gets id id_base + i (id_base < 0: -1);
    // ftt[id] receives the end time of the batch with its first output token
    int32_t track;
    long long id_base;
    double *ftt;
    KvLimits kv;  // the KV stream step (launch_advance_kv) only
};
constexpr int kK3Warps = 4;
// Shared memory of one K3 warp: a window's ends by batch, the decoders (context and decode
// offsets, id) and the waiting queue (prompt, decode, id); 16-byte aligned.
__host__ __device__ inline size_t advance_smem_per_warp(const DevConfig &c) {
    return (sizeof(int32_t) * ((size_t)3 * c.capR + (size_t)3 * c.capW + 96) + 15) & ~(size_t)15;
}
// The KV stream step's waiting queue is a ring of capW + capR entries: preempted
// requests return to its front.  (A window's words, the decoders, the ring; 16-byte aligned.)
__host__ __device__ inline size_t advance_kv_smem_per_warp(const DevConfig &c) {
    return (sizeof(int32_t) * ((size_t)3 * c.capR + (size_t)3 * ((size_t)c.capW + c.capR) + 160) + 15) & ~(size_t)15;
}
cudaError_t launch_advance(const K3Launch &a, int grid, size_t smem, cudaStream_t st);
cudaError_t launch_advance_kv(const K3Launch &a, int grid, size_t smem, cudaStream_t st);
cudaError_t set_k3_kv_smem();
cudaError_t set_k3_smem();
struct StateOut {
    int32_t *n_run, *run_ctx, *run_pre, *run_dec, *n_wait, *wait_pre, *wait_dec;
    double *clock;
};
cudaError_t launch_read_state(const DevConfig &c, const StateBuf &b0, const StateBuf &b1, DevCtl *ctl,
                              const StateOut &o, cudaStream_t st);

}  // namespace lr
