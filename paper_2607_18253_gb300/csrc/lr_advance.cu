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
// One warp per instance, every batch planned in two warp passes: the running list in
// order (each request's tokens within the budget, its new blocks, the blocks it holds),
// then FCFS admission from the waiting head while the budget, a seat and the first
// chunk's blocks allow.  When the running scan's new blocks exceed the free ones, lane
// 0 replays the scan request by request, preempting the last running request (possibly
// the one being served) until each finds its blocks; that case is rare and keeps the
// exact order of the rule.  A preempted request returns its blocks, its whole context
// becomes prefill again and it goes to the front of the waiting ring, in running order.
// A request whose context reaches the limit ends.  Each batch takes the Eq. 9 time of
// its own composition in the estimator's fp32 order, and runs only if it ends by t_now.

__device__ __forceinline__ int kv_blk(int c, int bs) { return (int)(((unsigned)c + (unsigned)bs - 1u) / (unsigned)bs); }

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
    int32_t *rc0 = wbase, *rp0 = rc0 + capR, *rd0 = rp0 + capR;
    int32_t *rc1 = rd0 + capR, *rp1 = rc1 + capR, *rd1 = rp1 + capR;
    int32_t *ri0 = rd1 + capR, *ri1 = ri0 + capR;
    int32_t *wp = ri1 + capR, *wd = wp + Wc, *wi = wd + Wc;
    const bool track = a.track != 0;
    const size_t rrow = (size_t)j * capR, wrow = (size_t)j * capW;
    int nr = src.n_run[j];
    int nw = src.n_wait[j];
    for (int t = lane; t < nr; t += 32) {
        rc0[t] = src.run_ctx[rrow + t];
        rp0[t] = src.run_pre[rrow + t];
        rd0[t] = src.run_dec[rrow + t];
        ri0[t] = track ? src.run_id[rrow + t] : -1;
    }
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
    const float b0 = cf[0], b1p = cf[1], b1d = cf[2], b2 = cf[3], b3 = cf[4];
    double t = src.clock[j];
    int wh = 0, iters = 0;  // the waiting ring holds nw requests from wh on
    int err = kOk;
    int32_t *rc = rc0, *rp = rp0, *rd = rd0, *ri = ri0, *nc = rc1, *np = rp1, *nd = rd1, *ni = ri1;
    while (true) {
        if (nr == 0 && nw == 0) {  // nothing to run: idle until t_now (never backwards)
            t = fmax(t, a.t_now);
            break;
        }
        if (++iters > c.max_iters) {
            err = kETraj;
            break;
        }
        // 1. the running scan: each request's tokens within the budget (a prefix of the
        //    list is served), the new blocks they need and the blocks every request holds
        long long used = 0, held = 0, nblk = 0;
        long long f1 = 0, f2 = 0, f3 = 0, f4 = 0;
        int rend = 0;
        for (int base = 0; base < nr; base += 32) {
            const int r = base + lane;
            const bool live = r < nr;
            const int ctx = live ? rc[r] : 0, pre = live ? rp[r] : 0;
            const int need = live ? (pre > 0 ? pre : 1) : 0;
            const long long incl = used + warp_incl_sum64(need, lane);
            const long long x = live ? max(0LL, min((long long)need, (long long)B - (incl - need))) : 0;
            if (live) held += kv_blk(ctx, bs);
            if (x > 0) {
                nblk += kv_blk(ctx + (int)x, bs) - kv_blk(ctx, bs);
                if (pre > 0) {
                    f1 += x;
                    f4 += x * ctx + x * (x + 1) / 2;
                } else {
                    f2 += 1;
                    f3 += ctx;
                }
            }
            rend += __popc(__ballot_sync(kFull, x > 0));
            used = __shfl_sync(kFull, incl, 31);
        }
        held = warp_sum64(held);
        nblk = warp_sum64(nblk);
        long long freeb = nbk - held;
        long long budget = max(0LL, (long long)B - used);
        int pnr = nr;  // running requests left after preemptions
        if (nblk > freeb) {
            // Not every served request finds its blocks: lane 0 replays the scan in the
            // rule's order, preempting from the tail, and the served prefix's features
            // are summed again.
            long long pf = freeb, bud = B;
            int r = 0, n = nr;
            if (lane == 0) {
                while (r < n && bud > 0) {
                    const long long x = rp[r] > 0 ? min((long long)rp[r], bud) : 1LL;
                    const int nb1 = kv_blk(rc[r] + (int)x, bs) - kv_blk(rc[r], bs);
                    while (pf < nb1 && n - 1 >= r) {
                        --n;
                        pf += kv_blk(rc[n], bs);
                    }
                    if (r >= n) break;  // r preempted itself
                    pf -= nb1;
                    bud -= x;
                    ++r;
                }
            }
            rend = __shfl_sync(kFull, r, 0);
            pnr = __shfl_sync(kFull, n, 0);
            freeb = __shfl_sync(kFull, pf, 0);
            budget = __shfl_sync(kFull, bud, 0);
            f1 = f2 = f3 = f4 = 0;
            used = 0;
            for (int base = 0; base < rend; base += 32) {
                const int r2 = base + lane;
                const bool live = r2 < rend;
                const int ctx = live ? rc[r2] : 0, pre = live ? rp[r2] : 0;
                const int need = live ? (pre > 0 ? pre : 1) : 0;
                const long long incl = used + warp_incl_sum64(need, lane);
                const long long x = live ? max(0LL, min((long long)need, (long long)B - (incl - need))) : 0;
                if (x > 0) {
                    if (pre > 0) {
                        f1 += x;
                        f4 += x * ctx + x * (x + 1) / 2;
                    } else {
                        f2 += 1;
                        f3 += ctx;
                    }
                }
                used = __shfl_sync(kFull, incl, 31);
            }
        } else {
            freeb -= nblk;
        }
        // the preempted tail [pnr, nr) goes to the ring's front in running order, its
        // whole context prefill again (the slots before the head are free; the head
        // moves only if the batch runs)
        const int k = nr - pnr;
        int wh2 = wh - k;
        if (wh2 < 0) wh2 += Wc;
        for (int i = lane; i < k; i += 32) {
            int pos = wh2 + i;
            if (pos >= Wc) pos -= Wc;
            wp[pos] = rc[pnr + i] + rp[pnr + i];
            wd[pos] = rd[pnr + i];
            wi[pos] = ri[pnr + i];
        }
        __syncwarp();
        const int nw2 = nw + k;
        // 2. admission from the ring's head while the budget, a seat and the first
        //    chunk's blocks allow (each condition holds for a prefix of the queue)
        int na = 0;
        long long wused = 0, bused = 0;
        for (int base = 0; budget - wused > 0 && base < nw2 && pnr + base < S; base += 32) {
            const int q = base + lane;
            int pos = wh2 + q;
            if (pos >= Wc) pos -= Wc;
            const bool in = q < nw2 && pnr + q < S;
            const int p = in ? wp[pos] : 0;
            const long long incl = wused + warp_incl_sum64(p, lane);
            const long long st = incl - p;
            const bool cand = in && st < budget;
            const long long x = cand ? min((long long)p, budget - st) : 0;
            const int nb1 = cand ? kv_blk((int)x, bs) : 0;
            const long long binc = bused + warp_incl_sum64(nb1, lane);
            const bool adm = cand && binc <= freeb;
            if (adm) {
                f1 += x;
                f4 += x * (x + 1) / 2;
            }
            const int nadm = __popc(__ballot_sync(kFull, adm));
            na += nadm;
            wused = __shfl_sync(kFull, incl, 31);
            bused = __shfl_sync(kFull, binc, 31);
            if (nadm < 32) break;
        }
        f1 = warp_sum64(f1);
        f2 = warp_sum64(f2);
        f3 = warp_sum64(f3);
        f4 = warp_sum64(f4);
        // Eq. 9 for this batch, in the estimator's fp32 order
        float T = __fmul_rn(b0, 1.0f);
        T = __fmaf_rn(b1d, __ll2float_rn(f2), T);
        T = __fmaf_rn(b1p, __ll2float_rn(f1), T);
        T = __fmaf_rn(b2, __ll2float_rn(f3), T);
        T = __fmaf_rn(b3, __ll2float_rn(f4), T);
        if (t + (double)T > a.t_now) break;  // still running at t_now
        if (pnr + na > capR) {
            err = kETraj;
            break;
        }
        // 3. execute it: the served prefix and the admitted requests advance; a request
        //    with no decode token left, or whose context reached the limit, ends
        int kept = 0;
        long long rused = 0, wst = 0;
        const int total = pnr + na;
        for (int base = 0; base < total; base += 32) {
            const int r = base + lane;
            const bool isr = r < pnr, isw = r >= pnr && r < total;
            int ctx = 0, pre = 0, dec = 0, id = -1;
            if (isr) {
                ctx = rc[r];
                pre = rp[r];
                dec = rd[r];
                id = ri[r];
            } else if (isw) {
                int pos = wh2 + (r - pnr);
                if (pos >= Wc) pos -= Wc;
                pre = wp[pos];
                dec = wd[pos];
                id = wi[pos];
            }
            const long long inr = isr ? (pre > 0 ? pre : 1) : 0;
            const long long incl_r = rused + warp_incl_sum64(inr, lane);
            const long long inw = isw ? pre : 0;
            const long long incl_w = wst + warp_incl_sum64(inw, lane);
            long long x = 0;
            if (isr && r < rend) x = max(0LL, min(inr, (long long)B - (incl_r - inr)));
            if (isw) x = min(inw, budget - (incl_w - inw));
            if (x > 0) {
                if (pre > 0) {
                    ctx += (int)x;
                    pre -= (int)x;
                    if (pre == 0 && c.mode == 1) {
                        dec -= 1;  // first token with the last chunk
                        if (track) id = emit_first(a, id, true, t + (double)T);
                    }
                } else {
                    ctx += 1;
                    dec -= 1;
                    if (track) id = emit_first(a, id, c.mode == 0, t + (double)T);
                }
            }
            if (pre == 0 && (long long)ctx >= mctx) dec = 0;  // the context limit
            const bool keep = (isr || isw) && dec > 0;
            const unsigned bal = __ballot_sync(kFull, keep);
            if (keep) {
                const int pos = kept + __popc(bal & lanemask_lt());
                nc[pos] = ctx;
                np[pos] = pre;
                nd[pos] = dec;
                ni[pos] = id;
            }
            kept += __popc(bal);
            rused = __shfl_sync(kFull, incl_r, 31);
            wst = __shfl_sync(kFull, incl_w, 31);
        }
        __syncwarp();
        int32_t *x0 = rc, *x1 = rp, *x2 = rd, *x3 = ri;
        rc = nc;
        rp = np;
        rd = nd;
        ri = ni;
        nc = x0;
        np = x1;
        nd = x2;
        ni = x3;
        nr = kept;
        wh = wh2 + na;
        if (wh >= Wc) wh -= Wc;
        nw = nw2 - na;
        t += (double)T;
        if (nw > capW) {
            err = kECapacity;
            break;
        }
    }
    if (err != kOk) {
        fail3(a.ctl, err, lane);
        return;
    }
    for (int q = lane; q < capR; q += 32) {
        dst.run_ctx[rrow + q] = q < nr ? rc[q] : 0;
        dst.run_pre[rrow + q] = q < nr ? rp[q] : 0;
        dst.run_dec[rrow + q] = q < nr ? rd[q] : 0;
        if (track) idst.run_id[rrow + q] = q < nr ? ri[q] : -1;
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

cudaError_t set_k3_smem(size_t bytes) {
    return cudaFuncSetAttribute(k_advance, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t launch_advance_kv(const K3Launch &a, int grid, size_t smem, cudaStream_t st) {
    return launch_chained(k_advance_kv, grid, kK3Warps * 32, smem, st, a);
}

cudaError_t set_k3_kv_smem(size_t bytes) {
    return cudaFuncSetAttribute(k_advance_kv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace lr
