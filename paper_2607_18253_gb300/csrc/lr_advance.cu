// K3: online stream step (Sec. 5: queries arrive by a Poisson process and are
// routed as they come; App. F: every instance keeps executing token batches
// and publishes its state after each one).
//
// One warp per instance: the queries routed to it join its waiting tail in
// query order (a stable ballot compaction over the assignment vector), then
// the instance executes whole token batches -- the same scheduler step the
// estimator simulates -- as long as each ends by t_now.  Each batch takes the
// Eq. 9 time of its own composition, evaluated in the same fp32 order as the
// estimate and accumulated into an fp64 clock.  An instance with nothing to
// run jumps to t_now.  The advanced snapshot goes to a scratch buffer, which
// K1 then summarizes and publishes like any snapshot.
//
// A published snapshot has at most one request in prefill, its last, and at most
// S_j <= B_j requests running (K1 refuses any other), and batches keep it so: every
// decoder gets its token in every batch.  The list therefore holds what decoding does
// not change -- context - G and decode + G, G batches done -- and a batch touches it
// only where requests end or join.  Batches that only decode are taken up to 32 at a
// time, a lane each (see below).
//
// Under KV-cache limits a second kernel (k_advance_kv) executes the KV step rule
// and hands its snapshot to the KV load instead of K1.
#include "lr_internal.cuh"

namespace lr {

namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ long long warp_incl_sum64(long long x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

__device__ void fail3(DevCtl *ctl, int code, int lane) {
    if (lane == 0) {
        atomicCAS(&ctl->load_err, 0, code);
        record_status(ctl, code);
    }
}

// First-token tracking (Sec. 4.1: the TTFT ends with the first output token; Eq. 4
// scores the realized TTFT): a tracked request (id >= 0) that emits its first output
// token in an executed batch -- its first decode token, or the token sampled with its
// last prompt chunk in that mode -- records the batch's end time and drops its id.
__device__ __forceinline__ int emit_first(const K3Launch &a, int id, bool emitted, double t_end) {
    if (emitted && id >= 0) {
        a.ftt[id] = t_end;
        return -1;
    }
    return id;
}

// The fp32 Eq. 9 time of a batch, in the estimator's order.
struct BatchTime {
    float b0, b1p, b1d, b2, b3;
    __device__ __forceinline__ float operator()(long long f1, long long f2, long long f3, long long f4) const {
        float T = __fmul_rn(b0, 1.0f);
        T = __fmaf_rn(b1d, __ll2float_rn(f2), T);
        T = __fmaf_rn(b1p, __ll2float_rn(f1), T);
        T = __fmaf_rn(b2, __ll2float_rn(f3), T);
        return __fmaf_rn(b3, __ll2float_rn(f4), T);
    }
};

__device__ __forceinline__ int warp_incl_sum32(int x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// The end times of consecutive batches by lane.  The clock adds the batch times one after
// the other in fp64; while those sums are exact their order does not matter, so an integer
// prefix sum in units of the clock's last bit gives every partial sum at once.  It is exact
// from the first lane on as long as a lane's time is a multiple of that unit and the sum
// stays in the clock's binade (below 2^53 units).
struct ClockScan {
    long long end;  // the batch's end, in units of 2^(e - 1075)
    int e;          // the clock's exponent field
    unsigned exact; // lanes whose partial sums are exact (a prefix of the warp's)
    __device__ __forceinline__ double time() const {  // of an exact lane
        // 2^52 <= end < 2^53: the clock's own exponent
        return __longlong_as_double(((long long)e << 52) | (end & ((1LL << 52) - 1)));
    }
};
__device__ __forceinline__ ClockScan clock_scan(double t, float T, int lane) {
    ClockScan c;
    const long long tb = __double_as_longlong(t);
    c.e = (int)(tb >> 52);  // t >= 0
    const unsigned Tb = __float_as_uint(T);
    const int Te = (int)(Tb >> 23);  // T >= 0, and not subnormal here
    const int sh = (Te - 150) - (c.e - 1075);  // T = m 2^(Te - 150)
    const bool fits = c.e > 0 && ((Te > 0 && sh >= 0 && sh <= 28) || Tb == 0u);
    const long long Ti = (fits && Tb != 0u) ? (long long)((Tb & 0x7fffffu) | 0x800000u) << sh : 0;
    const long long sum = warp_incl_sum64(Ti, lane);  // 32 times of less than 2^52 units
    c.end = ((tb & ((1LL << 52) - 1)) | (1LL << 52)) + sum;
    const unsigned bad = __ballot_sync(kFull, !fits || c.end >= (1LL << 53));
    c.exact = bad ? (1u << (__ffs(bad) - 1)) - 1u : kFull;
    return c;
}

// src: the live snapshot; idst: the buffer K1 publishes next (it receives the ids)
__device__ void advance_instance(const K3Launch &a, const StateBuf &src, const StateBuf &idst, int j, int lane,
                                 int32_t *wbase) {
    const DevConfig &c = a.cfg;
    const StateBuf &dst = a.scratch;
    const int B = c.B[j];
    const int S = c.S[j];
    const int capR = c.capR, capW = c.capW;
    long long *ends = reinterpret_cast<long long *>(wbase);  // [32] a window's ends: offsets summed
    int32_t *endc = wbase + 64;                              // [32] and counted
    int32_t *rx = endc + 32, *rz = rx + capR, *ri = rz + capR;  // decoders: context - G, decode + G, id
    int32_t *wp = ri + capR, *wd = wp + capW, *wi = wd + capW;  // waiting: prompt, decode, id
    const bool track = a.track != 0;
    const size_t rrow = (size_t)j * capR, wrow = (size_t)j * capW;
    const int nr0 = src.n_run[j];
    int nw = src.n_wait[j];
    // the request in prefill, if any, is the last running one
    int pP = 0, pC = 0, pD = 0, pI = -1;
    if (nr0 > 0) {
        pP = src.run_pre[rrow + nr0 - 1];
        pC = src.run_ctx[rrow + nr0 - 1];
        pD = src.run_dec[rrow + nr0 - 1];
        if (track) pI = src.run_id[rrow + nr0 - 1];
    }
    bool pf = pP > 0;
    int nd = nr0 - (pf ? 1 : 0);  // decoders
    long long csx = 0;            // their context offsets summed
    int zmin = kBig;              // the least decode + G
    for (int t = lane; t < nd; t += 32) {
        const int x = src.run_ctx[rrow + t], z = src.run_dec[rrow + t];
        rx[t] = x;
        rz[t] = z;
        if (track) ri[t] = src.run_id[rrow + t];
        csx += x;
        zmin = min(zmin, z);
    }
    for (int t = lane; t < nw; t += 32) {
        wp[t] = src.wait_pre[wrow + t];
        wd[t] = src.wait_dec[wrow + t];
        if (track) wi[t] = src.wait_id[wrow + t];
    }
    // routed queries join the waiting tail in query order (256 assignments in flight at once)
    for (int base = 0; base < a.Q; base += 256) {
        int as[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) as[k] = base + 32 * k + lane < a.Q ? a.assign[base + 32 * k + lane] : -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int i = base + 32 * k + lane;
            const bool mine = as[k] == j;
            const unsigned bal = __ballot_sync(kFull, mine);
            if (bal == 0u) continue;
            if (mine) {
                const int pos = nw + __popc(bal & lanemask_lt());
                if (pos < capW) {
                    wp[pos] = a.prompt[i];
                    wd[pos] = a.dec[(size_t)i * a.dec_cols + (a.dec_cols == 1 ? 0 : c.moi[j])];
                    if (track) wi[pos] = a.id_base >= 0 ? (int)(a.id_base + i) : -1;
                }
            }
            nw += __popc(bal);
        }
    }
    const bool over = nw > capW;
    bool bad = false;
    for (int t = lane; t < min(nw, capW); t += 32)
        bad |= wp[t] < 1 || wp[t] > (1 << 24) || wd[t] < 1 || wd[t] > (1 << 24);
    if (over) {
        fail3(a.ctl, kECapacity, lane);
        return;
    }
    if (__any_sync(kFull, bad)) {
        fail3(a.ctl, kEInval, lane);
        return;
    }
    csx = warp_sum64(csx);
    zmin = __reduce_min_sync(kFull, zmin);
    __syncwarp();

    const float *cf = c.coef + 5 * c.moi[j];
    const BatchTime bt = {cf[0], cf[1], cf[2], cf[3], cf[4]};
    double t = src.clock[j];
    int wh = 0, iters = 0;
    int G = 0;        // batches executed
    int fresh = 0;    // decoders from this one on may still owe their first token's time
    bool ok = true;
    // first tokens with a batch of their own: every decoder that has not emitted one does so
    // at the end of the next executed batch
    auto emit_fresh = [&](double t_end) {
        if (!track) return;
        if (c.mode == 0)
            for (int r = fresh + lane; r < nd; r += 32) ri[r] = emit_first(a, ri[r], true, t_end);
        __syncwarp();
        fresh = nd;
    };
    // the decoders that end by batch g (their last batch is decode + G - 1) leave, in place
    auto drop_ended = [&](int g) {
        int kept = 0, zm = kBig;
        long long cs = 0;
        for (int base = 0; base < nd; base += 32) {
            const int r = base + lane;
            const bool live = r < nd;
            const int x = live ? rx[r] : 0, z = live ? rz[r] : 0;
            const int id = (live && track) ? ri[r] : -1;
            const bool keep = live && z > g + 1;
            const unsigned bal = __ballot_sync(kFull, keep);
            __syncwarp();
            if (keep) {
                const int pos = kept + __popc(bal & lanemask_lt());
                rx[pos] = x;
                rz[pos] = z;
                if (track) ri[pos] = id;
                cs += x;
                zm = min(zm, z);
            }
            kept += __popc(bal);
        }
        nd = kept;
        csx = warp_sum64(cs);
        zmin = __reduce_min_sync(kFull, zm);
        fresh = min(fresh, nd);
        __syncwarp();
    };
    while (true) {
        if (nd == 0 && !pf && wh == nw) {  // nothing to run: idle until t_now (never backwards)
            t = fmax(t, a.t_now);
            break;
        }
        if (iters >= c.max_iters) {
            ok = false;
            break;
        }
        if (!pf && (wh == nw || nd >= S)) {
            // Only decoding: up to 32 batches, lane k taking batch G + k.  Batch k runs the
            // decoders that have not ended before it, each at its context, so its features
            // follow from the ends in the window, counted and summed by batch; with requests
            // waiting for a seat the window ends at the first end.  The clock's partial sums
            // come from an integer scan; where they are not exact (the clock enters another
            // binade) one batch is timed alone.  The time is then that of a few warp
            // operations for the window, where batch by batch a chain of five fp32 and one
            // fp64 operation and a pass over the list wherever a request ended set it.  With
            // the list held by offsets, a 256-query micro-batch on 64 instances (about 100
            // batches an instance): kernel 92 -> 28 us.
            int W = min(32, c.max_iters - iters);
            int cnt = 0;
            long long sx = 0;
            if (zmin - 1 - G < W) {
                ends[lane] = 0;
                endc[lane] = 0;
                __syncwarp();
                for (int r = lane; r < nd; r += 32) {
                    const int k = rz[r] - 1 - G;
                    if (k < 32) {
                        atomicAdd(&endc[k], 1);
                        atomicAdd(reinterpret_cast<unsigned long long *>(&ends[k]), (unsigned long long)(long long)rx[r]);
                    }
                }
                __syncwarp();
                cnt = endc[lane];
                sx = ends[lane];
                __syncwarp();  // read before the next window clears them
                if (wh < nw) W = min(W, zmin - G);  // through the batch with the first end
            }
            const int ndk = nd - (warp_incl_sum32(cnt, lane) - cnt);
            const long long csk = csx - (warp_incl_sum64(sx, lane) - sx);
            const float T = bt(0, ndk, csk + (long long)ndk * (G + lane), 0);
            const ClockScan cs = clock_scan(t, T, lane);
            const double te = cs.time();
            // batches that run: exact, within the window, something left to run, ending by t_now
            const unsigned in = W == 32 ? kFull : (1u << W) - 1u;
            const unsigned can = __ballot_sync(kFull, ndk > 0) & in;
            const unsigned run = __ballot_sync(kFull, te <= a.t_now) & can & cs.exact;
            const int n = run == kFull ? 32 : __ffs(~run) - 1;
            double t_first = 0.0;
            int done = n;
            if (n > 0) {
                t_first = __shfl_sync(kFull, te, 0);
                t = __shfl_sync(kFull, te, n - 1);
            } else if (!(cs.exact & 1u)) {
                const double t1 = t + (double)__shfl_sync(kFull, T, 0);
                if (t1 > a.t_now) break;  // still running at t_now
                t = t_first = t1;
                done = 1;
            } else {
                break;  // the next batch would end after t_now
            }
            emit_fresh(t_first);
            iters += done;
            G += done;
            if (zmin <= G) drop_ended(G - 1);
            // an exact batch inside the window that does not end by t_now ends the step
            if (n > 0 && n < 32 && ((can & cs.exact) >> n & 1u)) break;
            continue;
        }
        ++iters;
        // Plan the batch: every decoder one token, the prefill request its chunk, then FCFS
        // admission while budget and a slot remain (the k-th waiting request is admitted if
        // its prompt starts inside the budget and a sequence slot is free).
        const int px = pf ? min(pP, B - nd) : 0;
        const int budget = B - nd - px, nr = nd + (pf ? 1 : 0);
        long long f1 = px, f4 = (long long)px * pC + (long long)px * (px + 1) / 2;
        const long long f3 = csx + (long long)nd * G;
        int na = 0, wused = 0;
        for (int base = 0; budget - wused > 0 && wh + base < nw && nr + base < S; base += 32) {
            const int k = base + lane;
            const bool cand = wh + k < nw && nr + k < S;
            const int p = cand ? wp[wh + k] : 0;
            const int incl = wused + warp_incl_sum32(p, lane);  // below 2^24 + 32 prompts of at most 2^24
            const int st = incl - p;
            const bool adm = cand && st < budget;
            const long long x = adm ? min(p, budget - st) : 0;
            f1 += warp_sum64(x);
            f4 += warp_sum64(x * (x + 1) / 2);
            const int nadm = __popc(__ballot_sync(kFull, adm));
            na += nadm;
            if (nadm < 32) break;
            wused = __shfl_sync(kFull, incl, 31);
        }
        const float T = bt(f1, nd, f3, f4);
        const double t1 = t + (double)T;
        if (t1 > a.t_now) break;  // still running at t_now
        if (nr + na > capR) {
            ok = false;
            break;
        }
        // Execute it.
        emit_fresh(t1);
        t = t1;
        if (zmin == G + 1) drop_ended(G);
        const int off = c.mode == 1 ? 1 : 0;  // the first token comes with the last chunk
        if (pf) {
            pC += px;
            pP -= px;
            if (pP == 0) {
                pf = false;
                const int dec = pD - off;
                if (track && off) pI = lane == 0 ? emit_first(a, pI, true, t1) : -1;
                if (dec > 0) {
                    if (lane == 0) {
                        rx[nd] = pC - (G + 1);
                        rz[nd] = dec + (G + 1);
                        if (track) ri[nd] = pI;
                    }
                    csx += pC - (G + 1);
                    zmin = min(zmin, dec + G + 1);
                    ++nd;
                }
            }
        }
        int left = budget;
        for (int base = 0; base < na; base += 32) {
            const int k = base + lane;
            const bool in = k < na;
            const int p = in ? wp[wh + k] : 0, d = in ? wd[wh + k] : 0;
            int id = (in && track) ? wi[wh + k] : -1;
            const int incl = warp_incl_sum32(p, lane);
            const bool whole = in && incl <= left;
            if (track && off && whole) id = emit_first(a, id, true, t1);
            const bool keep = whole && d - off > 0;
            const unsigned bal = __ballot_sync(kFull, keep);
            if (keep) {
                const int pos = nd + __popc(bal & lanemask_lt());
                rx[pos] = p - (G + 1);
                rz[pos] = d - off + (G + 1);
                if (track) ri[pos] = id;
            }
            if (bal) {
                csx += warp_sum64(keep ? (long long)(p - (G + 1)) : 0);
                zmin = min(zmin, __reduce_min_sync(kFull, keep ? d - off + G + 1 : kBig));
                nd += __popc(bal);
            }
            // the last admitted prompt may continue in later batches
            const unsigned part = __ballot_sync(kFull, in && !whole);
            if (part) {
                const int l = __ffs(part) - 1;
                pf = true;
                pC = left - (__shfl_sync(kFull, incl, l) - __shfl_sync(kFull, p, l));
                pP = __shfl_sync(kFull, p, l) - pC;
                pD = __shfl_sync(kFull, d, l);
                pI = __shfl_sync(kFull, id, l);
            }
            left -= __shfl_sync(kFull, incl, 31);
        }
        __syncwarp();
        wh += na;
        ++G;
    }
    if (!ok) {
        fail3(a.ctl, kETraj, lane);
        return;
    }
    const int nw2 = nw - wh, nr = nd + (pf ? 1 : 0);
    for (int q = lane; q < capR; q += 32) {
        const bool d = q < nd, p = pf && q == nd;
        dst.run_ctx[rrow + q] = d ? rx[q] + G : p ? pC : 0;
        dst.run_pre[rrow + q] = p ? pP : 0;
        dst.run_dec[rrow + q] = d ? rz[q] - G : p ? pD : 0;
        if (track) idst.run_id[rrow + q] = d ? ri[q] : p ? pI : -1;
    }
    for (int q = lane; q < capW; q += 32) {
        dst.wait_pre[wrow + q] = q < nw2 ? wp[wh + q] : 0;
        dst.wait_dec[wrow + q] = q < nw2 ? wd[wh + q] : 0;
        if (track) idst.wait_id[wrow + q] = q < nw2 ? wi[wh + q] : -1;
    }
    if (lane == 0) {
        dst.n_run[j] = nr;
        dst.n_wait[j] = nw2;
        dst.clock[j] = t;
    }
}

// ---- The stream step under KV-cache limits (App. F: KV-cache allocation, context
// limits and preemption; the same step rule as the KV estimate) ----
//
// One warp per instance, as above: the decoders are held by offsets, the prefill request in
// registers, the waiting queue in a ring to whose front preempted requests return.  The
// free blocks are a running total; a batch needs a block for each decoder whose context is
// a multiple of the block size.  If they do not suffice, requests leave from the list's
// tail until what the leavers would hold after the batch reaches the excess (which leaves
// the longest prefix of the list that fits, as serving it in order does); their whole
// context becomes prefill again.  A request whose context reaches the limit ends.  Each
// batch takes the Eq. 9 time of its own composition in the estimator's fp32 order, and runs
// only if it ends by t_now: a plan touches no state but free ring slots until then.

__device__ void advance_instance_kv(const K3Launch &a, const StateBuf &src, const StateBuf &idst, int j, int lane,
                                    int32_t *wbase) {
    const DevConfig &c = a.cfg;
    const StateBuf &dst = a.scratch;
    const int B = c.B[j];
    const int S = c.S[j];
    const int bs = a.kv.bs[j];
    const long long nbk = a.kv.nb[j], mctx = a.kv.mctx[j];
    const int capR = c.capR, capW = c.capW;
    const int Wc = capW + capR;  // the waiting ring
    const Div32 dv = make_div32(bs);
    long long *wsx = reinterpret_cast<long long *>(wbase);  // [32] a window's ends: offsets summed,
    int32_t *wcnt = wbase + 64, *weblk = wcnt + 32;         // [32] counted, and their blocks;
    int32_t *wneed = weblk + 32;                            // [32] and the blocks its batches need
    int32_t *rx = wneed + 32, *rz = rx + capR, *ri = rz + capR;  // decoders: context - G, decode + G, id
    int32_t *wp = ri + capR, *wd = wp + Wc, *wi = wd + Wc;
    const bool track = a.track != 0;
    const size_t rrow = (size_t)j * capR, wrow = (size_t)j * capW;
    const int nr0 = src.n_run[j];
    int nw = src.n_wait[j];
    // the request in prefill, if any, is the last running one
    int pP = 0, pC = 0, pD = 0, pI = -1;
    if (nr0 > 0) {
        pP = src.run_pre[rrow + nr0 - 1];
        pC = src.run_ctx[rrow + nr0 - 1];
        pD = src.run_dec[rrow + nr0 - 1];
        if (track) pI = src.run_id[rrow + nr0 - 1];
    }
    bool pf = pP > 0;
    int nd = nr0 - (pf ? 1 : 0);  // decoders
    // a decoder's last batch: its decode count or the context limit
    auto last_batch = [&](int x, int z) { return (int)min((long long)z - 1, mctx - 1 - x); };
    long long csx = 0, freeb = 0;  // the decoders' context offsets summed; free blocks
    int emin = kBig;               // the first last batch
    for (int t = lane; t < nd; t += 32) {
        const int x = src.run_ctx[rrow + t], z = src.run_dec[rrow + t];
        rx[t] = x;
        rz[t] = z;
        ri[t] = track ? src.run_id[rrow + t] : -1;
        csx += x;
        freeb -= dblk(dv, x);
        emin = min(emin, last_batch(x, z));
    }
    csx = warp_sum64(csx);
    int pH = pf ? dblk(dv, pC) : 0;  // the prefill request's blocks
    freeb = nbk + warp_sum64(freeb) - pH;
    emin = __reduce_min_sync(kFull, emin);
    for (int t = lane; t < nw; t += 32) {
        wp[t] = src.wait_pre[wrow + t];
        wd[t] = src.wait_dec[wrow + t];
        wi[t] = track ? src.wait_id[wrow + t] : -1;
    }
    // routed queries join the waiting tail in query order; one that could never run
    // (its prompt at the context limit, or its whole context capped at the limit needing
    // more blocks than the instance has) is refused
    bool bad = false;
    for (int base = 0; base < a.Q; base += 32) {
        const int i = base + lane;
        const bool mine = i < a.Q && a.assign[i] == j;
        const unsigned bal = __ballot_sync(kFull, mine);
        if (mine) {
            const int pos = nw + __popc(bal & lanemask_lt());
            const int p = a.prompt[i];
            const int d = a.dec[(size_t)i * a.dec_cols + (a.dec_cols == 1 ? 0 : c.moi[j])];
            bad |= p < 1 || p > (1 << 24) || d < 1 || d > (1 << 24);
            bad |= (long long)p >= mctx;
            bad |= (long long)(((unsigned long long)min((long long)p + d, mctx) + bs - 1) / bs) > nbk;
            if (pos < capW) {
                wp[pos] = p;
                wd[pos] = d;
                wi[pos] = (track && a.id_base >= 0) ? (int)(a.id_base + i) : -1;
            }
        }
        nw += __popc(bal);
    }
    if (nw > capW) {
        fail3(a.ctl, kECapacity, lane);
        return;
    }
    if (__any_sync(kFull, bad)) {
        fail3(a.ctl, kEInval, lane);
        return;
    }
    __syncwarp();

    const float *cf = c.coef + 5 * c.moi[j];
    const BatchTime bt = {cf[0], cf[1], cf[2], cf[3], cf[4]};
    double t = src.clock[j];
    int wh = 0, iters = 0;  // the waiting ring holds nw requests from wh on
    int G = 0, fresh = 0;   // batches executed; decoders from `fresh` on may owe their first token's time
    int err = kOk;
    const int off = c.mode == 1 ? 1 : 0;  // the first token comes with the last chunk
    auto emit_fresh = [&](double t_end) {
        if (!track) return;
        if (c.mode == 0)
            for (int r = fresh + lane; r < nd; r += 32) ri[r] = emit_first(a, ri[r], true, t_end);
        __syncwarp();
        fresh = nd;
    };
    // the decoders whose last batch is g or before leave, in place; returns the blocks they held
    auto drop_ended = [&](int g) -> long long {
        int kept = 0, em = kBig;
        long long cs = 0, back = 0;
        for (int base = 0; base < nd; base += 32) {
            const int r = base + lane;
            const bool live = r < nd;
            const int x = live ? rx[r] : 0, z = live ? rz[r] : 0, id = live ? ri[r] : -1;
            const int E = live ? last_batch(x, z) : -1;
            const bool keep = live && E > g;
            const unsigned bal = __ballot_sync(kFull, keep);
            __syncwarp();
            if (keep) {
                const int pos = kept + __popc(bal & lanemask_lt());
                rx[pos] = x;
                rz[pos] = z;
                ri[pos] = id;
                cs += x;
                em = min(em, E);
            } else if (live) {
                back += dblk(dv, x + E + 1);
            }
            kept += __popc(bal);
        }
        nd = kept;
        csx = warp_sum64(cs);
        emin = __reduce_min_sync(kFull, em);
        fresh = min(fresh, nd);
        __syncwarp();
        return warp_sum64(back);
    };
    while (true) {
        if (nd == 0 && !pf && nw == 0) {  // nothing to run: idle until t_now (never backwards)
            t = fmax(t, a.t_now);
            break;
        }
        if (iters >= c.max_iters) {
            err = kETraj;
            break;
        }
        // 1. the running scan: every decoder one token, the prefill request its chunk
        int need_d = 0;
        for (int r = lane; r < nd; r += 32) need_d += dres(dv, rx[r] + G) == 0 ? 1 : 0;
        need_d = __reduce_add_sync(kFull, need_d);
        const int hp = nw > 0 ? wp[wh] : 0;
        if (!pf && nd > 0 && need_d <= freeb &&
            (nw == 0 || nd >= S || B <= nd || dblk(dv, min(hp, B - nd)) > freeb - need_d)) {
            // Only decoding: up to 32 batches, lane k taking batch G + k, as in the plain step.
            // Batch k runs if the blocks suffice -- those its decoders need, and those the
            // window's ends return, are counted by batch -- and the head, if one waits, still
            // cannot be admitted.  With the list held by offsets, 16-query micro-batches on 64
            // instances: kernel 42 -> 32 us.
            wsx[lane] = 0;
            wcnt[lane] = weblk[lane] = wneed[lane] = 0;
            __syncwarp();
            for (int r = lane; r < nd; r += 32) {
                const int x = rx[r];
                const int e = last_batch(x, rz[r]) - G;  // its last batch of the window
                const int g = dres(dv, x + G);
                for (int k = g == 0 ? 0 : bs - g; k < 32 && k <= e; k += bs) atomicAdd(&wneed[k], 1);
                if (e < 32) {
                    atomicAdd(&wcnt[e], 1);
                    atomicAdd(reinterpret_cast<unsigned long long *>(&wsx[e]), (unsigned long long)(long long)x);
                    atomicAdd(&weblk[e], dblk(dv, x + G + e + 1));
                }
            }
            __syncwarp();
            const int cnt = wcnt[lane], eb = weblk[lane], need = wneed[lane];
            const long long sx = wsx[lane];
            __syncwarp();  // read before the next window clears them
            const int ndk = nd - (warp_incl_sum32(cnt, lane) - cnt);
            const long long csk = csx - (warp_incl_sum64(sx, lane) - sx);
            const long long gain = warp_incl_sum64((long long)eb - need, lane);  // through batch k
            const long long fb = freeb + gain - eb;                              // after its scan
            const float T = bt(0, ndk, csk + (long long)ndk * (G + lane), 0);
            const ClockScan cs = clock_scan(t, T, lane);
            const double te = cs.time();
            const bool blocked = nw == 0 || ndk >= S || B <= ndk || dblk(dv, min(hp, B - ndk)) > fb;
            const int W = min(32, c.max_iters - iters);
            const unsigned in = W == 32 ? kFull : (1u << W) - 1u;
            const unsigned bad = ~__ballot_sync(kFull, ndk > 0 && fb >= 0 && blocked);
            const unsigned can = (bad ? (1u << (__ffs(bad) - 1)) - 1u : kFull) & in;  // (lane 0 always)
            const unsigned run = __ballot_sync(kFull, te <= a.t_now) & can & cs.exact;
            const int n = run == kFull ? 32 : __ffs(~run) - 1;
            double t_first;
            int done = n;
            if (n > 0) {
                t_first = __shfl_sync(kFull, te, 0);
                t = __shfl_sync(kFull, te, n - 1);
            } else if (!(cs.exact & 1u)) {
                const double t1 = t + (double)__shfl_sync(kFull, T, 0);
                if (t1 > a.t_now) break;  // still running at t_now
                t = t_first = t1;
                done = 1;
            } else {
                break;  // the next batch would end after t_now
            }
            emit_fresh(t_first);
            freeb += __shfl_sync(kFull, gain, done - 1);  // less what the batches needed, and the ends' blocks
            iters += done;
            G += done;
            if (emin < G) drop_ended(G - 1);
            // an admissible exact batch that does not end by t_now ends the step
            if (n > 0 && n < 32 && ((can & cs.exact) >> n & 1u)) break;
            continue;
        }
        ++iters;
        const int px = pf ? min(pP, B - nd) : 0;
        const int pnew = pf ? dblk(dv, pC + px) : 0;
        const int need_all = need_d + (pnew - pH);
        // the plan: what the batch would leave of the list and of the blocks
        int pnd = nd, kq = 0;  // decoders left, requests preempted
        bool ppf = pf;
        long long pcsx = csx, fb = freeb - need_all;
        if (fb < 0) {
            long long acc = 0;  // post-batch blocks of those gone
            const long long excess = -fb;
            if (pf) {
                acc = pnew;
                ppf = false;
                kq = 1;
            }
            while (acc < excess && pnd > 0) {
                const int x = rx[--pnd];
                acc += dblk(dv, x + G + 1);
                pcsx -= x;
                ++kq;
            }
            fb = acc - excess;
        }
        int wh2 = wh - kq;
        if (wh2 < 0) wh2 += Wc;
        // (in running order, before the head: decoders, then the prefill request)
        for (int i = lane; i < nd - pnd; i += 32) {
            int pos = wh2 + i;
            if (pos >= Wc) pos -= Wc;
            wp[pos] = rx[pnd + i] + G;
            wd[pos] = rz[pnd + i] - G;
            wi[pos] = ri[pnd + i];
        }
        if (pf && !ppf && lane == 0) {
            int pos = wh2 + kq - 1;
            if (pos >= Wc) pos -= Wc;
            wp[pos] = pC + pP;
            wd[pos] = pD;
            wi[pos] = pI;
        }
        __syncwarp();
        const int nw2 = nw + kq, qx = ppf ? px : 0;
        const int pnr = pnd + (ppf ? 1 : 0);
        const int budget = B - pnd - qx;
        long long f1 = qx, f4 = (long long)qx * pC + (long long)qx * (qx + 1) / 2;
        const long long f3 = pcsx + (long long)pnd * G;
        // 2. admission from the ring's head while the budget, a seat and the first chunk's
        //    blocks allow (each condition holds for a prefix of the queue)
        int na = 0, wused = 0;
        long long bused = 0, ablk = 0;  // blocks up to the round; of the admitted
        for (int base = 0; budget - wused > 0 && base < nw2 && pnr + base < S; base += 32) {
            const int q = base + lane;
            int pos = wh2 + q;
            if (pos >= Wc) pos -= Wc;
            const bool in = q < nw2 && pnr + q < S;
            const int p = in ? wp[pos] : 0;
            // (a preempted context can reach 2^28 tokens)
            const long long incl = wused + warp_incl_sum64(p, lane);
            const long long st = incl - p;
            const bool cand = in && st < budget;
            const long long x = cand ? min((long long)p, budget - st) : 0;
            const int nb1 = cand ? dblk(dv, (int)x) : 0;
            const long long binc = bused + warp_incl_sum64(nb1, lane);
            const bool adm = cand && binc <= fb;
            f1 += warp_sum64(adm ? x : 0);
            f4 += warp_sum64(adm ? x * (x + 1) / 2 : 0);
            ablk += warp_sum64(adm ? (long long)nb1 : 0);
            const int nadm = __popc(__ballot_sync(kFull, adm));
            na += nadm;
            if (nadm < 32) break;
            wused = (int)__shfl_sync(kFull, incl, 31);  // all admitted: below the budget, or the last
            bused = __shfl_sync(kFull, binc, 31);
        }
        const float T = bt(f1, pnd, f3, f4);
        const double t1 = t + (double)T;
        if (t1 > a.t_now) break;  // still running at t_now
        if (pnr + na > capR) {
            err = kETraj;
            break;
        }
        // 3. execute it: a request with no decode token left, or whose context reached the
        //    limit, ends
        nd = pnd;
        csx = pcsx;
        pf = ppf;
        fresh = min(fresh, nd);
        freeb = fb - ablk;
        emit_fresh(t1);
        t = t1;
        if (emin <= G || kq > 0) freeb += drop_ended(G);
        if (pf) {
            pC += px;
            pP -= px;
            pH = pnew;
            if (pP == 0) {
                pf = false;
                const int dec = pD - off;
                if (track && off) pI = lane == 0 ? emit_first(a, pI, true, t1) : -1;
                if (dec > 0 && (long long)pC < mctx) {
                    const int x = pC - (G + 1), z = dec + (G + 1);
                    if (lane == 0) {
                        rx[nd] = x;
                        rz[nd] = z;
                        ri[nd] = pI;
                    }
                    csx += x;
                    emin = min(emin, last_batch(x, z));
                    ++nd;
                } else {
                    freeb += pH;
                }
                pH = 0;
            }
        } else {
            pH = 0;
        }
        long long left = budget;
        for (int base = 0; base < na; base += 32) {
            const int q = base + lane;
            int pos = wh2 + q;
            if (pos >= Wc) pos -= Wc;
            const bool in = q < na;
            const int p = in ? wp[pos] : 0, d = in ? wd[pos] : 0;
            int id = in ? wi[pos] : -1;
            const long long incl = warp_incl_sum64(p, lane);
            const bool whole = in && incl <= left;
            if (track && off && whole) id = emit_first(a, id, true, t1);
            const bool keep = whole && d - off > 0 && (long long)p < mctx;
            const unsigned bal = __ballot_sync(kFull, keep);
            const int x = p - (G + 1), z = d - off + (G + 1);
            if (keep) {
                const int r = nd + __popc(bal & lanemask_lt());
                rx[r] = x;
                rz[r] = z;
                ri[r] = id;
            }
            if (bal) {
                csx += warp_sum64(keep ? (long long)x : 0);
                emin = min(emin, __reduce_min_sync(kFull, keep ? last_batch(x, z) : kBig));
                nd += __popc(bal);
            }
            freeb += warp_sum64(whole && !keep ? (long long)dblk(dv, p) : 0);  // ended with its prompt
            // the last admitted prompt may continue in later batches
            const unsigned part = __ballot_sync(kFull, in && !whole);
            if (part) {
                const int l = __ffs(part) - 1;
                pf = true;
                pC = (int)(left - (__shfl_sync(kFull, incl, l) - __shfl_sync(kFull, p, l)));
                pP = __shfl_sync(kFull, p, l) - pC;
                pD = __shfl_sync(kFull, d, l);
                pI = __shfl_sync(kFull, id, l);
                pH = dblk(dv, pC);
            }
            left -= __shfl_sync(kFull, incl, 31);
        }
        __syncwarp();
        wh = wh2 + na;
        if (wh >= Wc) wh -= Wc;
        nw = nw2 - na;
        ++G;
        if (nw > capW) {
            err = kECapacity;
            break;
        }
    }
    if (err != kOk) {
        fail3(a.ctl, err, lane);
        return;
    }
    const int nr = nd + (pf ? 1 : 0);
    for (int q = lane; q < capR; q += 32) {
        const bool d = q < nd, p = pf && q == nd;
        dst.run_ctx[rrow + q] = d ? rx[q] + G : p ? pC : 0;
        dst.run_pre[rrow + q] = p ? pP : 0;
        dst.run_dec[rrow + q] = d ? rz[q] - G : p ? pD : 0;
        if (track) idst.run_id[rrow + q] = d ? ri[q] : p ? pI : -1;
    }
    for (int q = lane; q < capW; q += 32) {
        int pos = wh + q;
        if (pos >= Wc) pos -= Wc;
        dst.wait_pre[wrow + q] = q < nw ? wp[pos] : 0;
        dst.wait_dec[wrow + q] = q < nw ? wd[pos] : 0;
        if (track) idst.wait_id[wrow + q] = q < nw ? wi[pos] : -1;
    }
    if (lane == 0) {
        dst.n_run[j] = nr;
        dst.n_wait[j] = nw;
        dst.clock[j] = t;
    }
}

__global__ void __launch_bounds__(kK3Warps * 32) k_advance(const K3Launch a) {
    extern __shared__ __align__(16) int32_t k3_smem[];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    const int j = blockIdx.x * kK3Warps + wid;
    chain_wait();
    const int active = *((volatile int32_t *)&a.ctl->active);
    if (j >= a.cfg.I) return;
    if (active < 0) {
        fail3(a.ctl, kENoState, lane);
        return;
    }
    const StateBuf src = active ? a.buf1 : a.buf0;
    // the buffer the summary (K1) publishes next, as K1 chooses it from the same index
    const StateBuf idst = active ? a.buf0 : a.buf1;
    const size_t per_warp = advance_smem_per_warp(a.cfg) / sizeof(int32_t);
    advance_instance(a, src, idst, j, lane, k3_smem + wid * per_warp);
    chain_next();
}

__global__ void __launch_bounds__(kK3Warps * 32) k_advance_kv(const K3Launch a) {
    extern __shared__ __align__(16) int32_t k3_smem[];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    const int j = blockIdx.x * kK3Warps + wid;
    chain_wait();
    const int active = *((volatile int32_t *)&a.ctl->active);
    if (j >= a.cfg.I) return;
    if (active < 0) {
        fail3(a.ctl, kENoState, lane);
        return;
    }
    const StateBuf src = active ? a.buf1 : a.buf0;
    // the buffer the KV load publishes next, as it chooses it from the same index
    const StateBuf idst = active ? a.buf0 : a.buf1;
    const size_t per_warp = advance_kv_smem_per_warp(a.cfg) / sizeof(int32_t);
    advance_instance_kv(a, src, idst, j, lane, k3_smem + wid * per_warp);
    chain_next();
}

// Copy of the live snapshot into caller arrays (the live buffer is known only on
// the device).
__global__ void k_read_state(const DevConfig c, const StateBuf b0, const StateBuf b1, const DevCtl *ctl,
                             const StateOut o) {
    chain_wait();
    const int active = *((volatile const int32_t *)&ctl->active);
    const StateBuf s = active == 1 ? b1 : b0;
    const size_t R = (size_t)c.I * c.capR, W = (size_t)c.I * c.capW;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < R + W + c.I;
         i += (size_t)gridDim.x * blockDim.x) {
        if (i < R) {
            if (o.run_ctx) o.run_ctx[i] = s.run_ctx[i];
            if (o.run_pre) o.run_pre[i] = s.run_pre[i];
            if (o.run_dec) o.run_dec[i] = s.run_dec[i];
        } else if (i < R + W) {
            if (o.wait_pre) o.wait_pre[i - R] = s.wait_pre[i - R];
            if (o.wait_dec) o.wait_dec[i - R] = s.wait_dec[i - R];
        } else {
            const size_t k = i - R - W;
            if (o.n_run) o.n_run[k] = s.n_run[k];
            if (o.n_wait) o.n_wait[k] = s.n_wait[k];
            if (o.clock) o.clock[k] = s.clock[k];
        }
    }
}

}  // namespace

cudaError_t launch_read_state(const DevConfig &c, const StateBuf &b0, const StateBuf &b1, DevCtl *ctl,
                              const StateOut &o, cudaStream_t st) {
    return launch_chained(k_read_state, 128, 256, 0, st, c, b0, b1, (const DevCtl *)ctl, o);
}

cudaError_t launch_advance(const K3Launch &a, int grid, size_t smem, cudaStream_t st) {
    return launch_chained(k_advance, grid, kK3Warps * 32, smem, st, a);
}

cudaError_t set_k3_smem() {
    return allow_smem(k_advance, kSmemMax);
}

cudaError_t launch_advance_kv(const K3Launch &a, int grid, size_t smem, cudaStream_t st) {
    return launch_chained(k_advance_kv, grid, kK3Warps * 32, smem, st, a);
}

cudaError_t set_k3_kv_smem() {
    return allow_smem(k_advance_kv, kSmemMax);
}

}  // namespace lr
