// KV-limited Serving Framework Simulation (Sec. 4.1; App. F names context limits,
// the KV-cache allocation state and preemption among what the simulation models).
//
// Reading of the step rule: instance j has nb_j blocks of bs_j tokens and a request
// with c tokens in the cache holds ceil(c / bs_j) of them.  The running list is
// served in order; a request whose tokens of the batch need blocks that are not
// free preempts the last running request (its blocks return, its whole context
// becomes prefill again and it goes to the front of the waiting queue), itself if it
// is the last.  The waiting head is admitted only if its first chunk's blocks are
// free.  A request whose context reaches mctx_j ends there.
//
// The query q appended at the waiting tail never changes the residents' batches:
// it is admitted only once no resident waits, and while it runs it is the last
// running request, so it is the first preemption victim and no resident ever waits
// for its blocks.  So the load (k_kv_load) simulates each instance's residents
// alone, once, and records for every batch from the first in which q could be
// admitted what q's fate depends on: the budget left to it, the largest prompt it
// could be admitted with, the free blocks and the least block slack of the
// residents' scan (q, holding h blocks, is preempted in a batch whose slack is
// below h), and the residents' Eq. 9 features summed so far.  The estimate
// (k_kv_estimate) then finds each (query, instance) candidate's admission batch by
// a binary search over the running maximum of the admission bounds and follows it
// from there, record by record, through prefill chunks, preemptions and
// readmissions, to its first token.  A candidate depends only on the instance and
// the prompt length, so each call first counting-sorts its queries by length
// (k_kv_count, k_kv_scan, k_kv_scatter), walks once per distinct length, and
// copies those rows to the other queries of the same length (k_kv_expand; a route that
// returns no matrix reads the first query's row instead).  A call of few
// queries walks each of them directly instead, in the one launch.
#include "lr_internal.cuh"

namespace lr {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr long long kHuge = 1LL << 62;
constexpr int kBigKv = 0x7fffffff;
// A condition that is the same on every lane, as a vote: the compiler then knows it and
// branches without setting up a reconvergence point (which costs the scalar code of a warp
// more than the vote).
__device__ __forceinline__ bool uni(bool c) { return __any_sync(kFull, c) != 0; }
__device__ __forceinline__ int clamp32(long long x) { return (int)min(x, (long long)kBigKv); }

__device__ __forceinline__ long long kv_blocks(long long c, long long bs) { return (c + bs - 1) / bs; }
// ceil(c / bs) for 0 <= c < 2^31 (32-bit division)
__device__ __forceinline__ int kv_blocks32(int c, int bs) {
    return (int)(((unsigned)c + (unsigned)bs - 1u) / (unsigned)bs);
}

__device__ void kv_fail(DevCtl *ctl, int code, int lane) {
    if (lane == 0) {
        atomicCAS(&ctl->load_err, 0, code);
        record_status(ctl, code);
    }
}

__device__ __forceinline__ long long warp_incl_sum64(long long x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    return x;
}
__device__ __forceinline__ int warp_incl_sum32(int x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    return x;
}
__device__ __forceinline__ int warp_sum32(int x) { return __reduce_add_sync(kFull, x); }

// End calendar of the KV load: a decoder that ends in batch E (>= the current
// batch G) waits in list E mod kKvCal if E < G + kKvCal, else in the overflow list,
// whose nodes are re-filed at every multiple of kKvCal.  Pushes from several lanes
// at once are safe.
__device__ __forceinline__ void kv_cal_push(int32_t *head, int32_t *nxt, int32_t *ovf, int s, long long E, int G) {
    int32_t *h = E < (long long)G + kKvCal ? &head[E & (kKvCal - 1)] : ovf;
    nxt[s] = atomicExch(h, s);
}
// the batch (as a value of G) in which a decoder held as (context - G, decode + G) ends
__device__ __forceinline__ long long kv_end(const int4 &q, long long mctx) {
    return min((long long)q.z - 1, mctx - 1 - q.x);
}
// One instance's residents alone, batch by batch, from the snapshot.  Every lane
// holds the same scalar state.
//
// Running request in slot s: rq[s] = (context - G, 0, decode + G, context residue mod
// bs) for a decoder, whose blocks at its end wait in eb[s].  Slots keep the list's
// order; a request that leaves becomes a hole (second word -1) until a compaction.  Only
// the last running request may be in prefill (slot pfs, second word 1, its state in
// registers).  The others decode one token
// a batch (G = batches done), so no word of theirs changes until they end.  The
// decoders crossing into a new block in batch G are those whose context is a
// multiple of bs, counted by a histogram of stored contexts mod bs; their context
// sum (Eq. 9's F3 term) is a running total; the batch each one ends in (decode
// count or context limit) waits in the end calendar.  A request that ends frees
// ceil(context / bs) blocks after its last batch.
template <int MODE>
__device__ void kv_instance(const KvLoad &a, const StateBuf &out, int j, int lane, int32_t *wb) {
    const DevConfig &c = a.cfg;
    const int B = c.B[j];
    const int S = c.S[j];
    const long long nbk = a.kv.nb[j], mctx = a.kv.mctx[j];
    const int bs = a.kv.bs[j];
    const Div32 dv = make_div32(bs);
    const int C = c.capR + c.capW;  // at most this many residents
    int4 *rq = reinterpret_cast<int4 *>(wb);               // running list slots
    int2 *wq = reinterpret_cast<int2 *>(rq + C);           // waiting ring (prefill, decode)
    int32_t *nxt = reinterpret_cast<int32_t *>(wq + C);    // [C] calendar links
    int32_t *eb = nxt + C;                                 // [C] a decoder's blocks at its end
    int32_t *head = eb + C;                                // [kKvCal] calendar lists
    int32_t *hist = head + kKvCal;                         // [bs] residue histogram
    int32_t *ovf = hist + a.kv.hist;                       // overflow list head
    const int nr0 = a.in.n_run[j];
    const int nw0 = a.in.n_wait[j];
    if (lane == 0) {
        out.n_run[j] = nr0;
        out.n_wait[j] = nw0;
        out.clock[j] = a.in.clock ? a.in.clock[j] : 0.0;
    }
    if (!(nr0 >= 0 && nr0 <= c.capR && nr0 <= S && nw0 >= 0 && nw0 <= c.capW)) {
        kv_fail(a.ctl, kEState, lane);
        return;
    }
    for (int b = lane; b < kKvCal; b += 32) head[b] = -1;
    for (int b = lane; b < bs; b += 32) hist[b] = 0;
    if (lane == 0) *ovf = -1;
    // file decoder slot s, held as q (fourth word: residue) at batch G
    auto file = [&](int s, const int4 &q, int G_) {
        const long long E = kv_end(q, mctx);
        eb[s] = dblk(dv, (int)(q.x + E + 1));
        kv_cal_push(head, nxt, ovf, s, E, G_);
    };
    // Copy and validate the snapshot: only the last running request may still be in
    // prefill, no context reaches the limit, every request's whole context fits the
    // instance's blocks, and the running requests' blocks fit together.
    const size_t rrow = (size_t)j * c.capR, wrow = (size_t)j * c.capW;
    bool bad = false;
    long long held = 0, wsum = 0, src = 0;
    int nd = 0;
    for (int t = lane; t < c.capR; t += 32) {
        const int ctx = a.in.run_ctx[rrow + t], pre = a.in.run_pre[rrow + t], dec = a.in.run_dec[rrow + t];
        out.run_ctx[rrow + t] = ctx;
        out.run_pre[rrow + t] = pre;
        out.run_dec[rrow + t] = dec;
        if (t < nr0) {
            const bool ok = ctx >= 0 && ctx <= (1 << 28) && pre >= 0 && pre <= (1 << 24) && dec >= 1 &&
                            dec <= (1 << 24);
            bad |= !ok;
            bad |= pre > 0 && t != nr0 - 1;
            bad |= (long long)ctx + pre >= mctx;
            bad |= ok && kv_blocks(min((long long)ctx + pre + dec, mctx), bs) > nbk;
            const int h = ok ? dblk(dv, ctx) : 0;
            held += h;
            if (pre == 0) {
                src += ctx;
                ++nd;
            }
            rq[t] = pre > 0 ? make_int4(ctx, pre, dec, h) : make_int4(ctx, 0, dec, dres(dv, ctx));
        }
    }
    for (int t = lane; t < c.capW; t += 32) {
        const int pre = a.in.wait_pre[wrow + t], dec = a.in.wait_dec[wrow + t];
        out.wait_pre[wrow + t] = pre;
        out.wait_dec[wrow + t] = dec;
        if (t < nw0) {
            bad |= pre < 1 || pre > (1 << 24) || dec < 1 || dec > (1 << 24);
            bad |= (long long)pre >= mctx;
            bad |= kv_blocks(min((long long)pre + dec, mctx), bs) > nbk;
            wsum += pre;
            wq[t] = make_int2(pre, dec);
        }
    }
    held = warp_sum64(held);
    wsum = warp_sum64(wsum);
    src = warp_sum64(src);
    nd = warp_sum32(nd);
    if (__any_sync(kFull, bad) || held > nbk || wsum > (1LL << 30)) {
        kv_fail(a.ctl, kEState, lane);
        return;
    }
    __syncwarp();
    // the decoders into the histogram and the calendar (G = 0)
    for (int t = lane; t < nr0; t += 32) {
        const int4 q = rq[t];
        if (q.y == 0) {
            atomicAdd(&hist[q.w], 1);
            file(t, q, 0);
        }
    }
    __syncwarp();

    long long freeb = nbk - held;
    int nr = nr0, ne = nr0;                             // running requests; slots in use
    int tl = nr0;                                       // past the last running request's slot (holes follow it)
    int pfs = (nr0 > 0 && rq[nr0 - 1].y > 0) ? nr0 - 1 : -1;  // the prefill request's slot
    int pC = 0, pP = 0, pD = 0, pH = 0;                       // its context, prefill, decode and blocks
    if (pfs >= 0) {
        const int4 q = rq[pfs];
        pC = q.x;
        pP = q.y;
        pD = q.z;
        pH = q.w;
    }
    int wh = 0, wc = nw0;                               // waiting ring head and count
    int G = 0, gr = 0;                                  // batches done; G mod bs
    long long fcum[5] = {0, 0, 0, 0, 0};
    long long cf1 = 0, cf2 = 0, cf3 = 0, cf4 = 0;  // features summed over the records
    int la0 = 0, nrec = 0, done = 0, pmx = 0;
    // Where the records may end.  In a "clear" record a query of any allowed length that has
    // no first token yet is admitted if it waits, is not preempted (the slack and the free
    // blocks reach a whole query's, hq) and prefills `bl` tokens.  So after consecutive
    // clear records whose budgets sum to max_prompt_len every query has its prompt done, and
    // one clear record later its first token: no walk passes that record, and the
    // simulation stops there (`clear` is the budget sum of the current stretch).  A load
    // that the batches up to the horizon could still take past max_iters keeps going, so
    // the same snapshots are refused.  On the 64- and 256-instance pools the records end
    // after 42 batches in the mean, 227 at most, where up to 4,096 used to be simulated and
    // written: load 403 -> 370 us (64 instances), 456 -> 405 us (256).
    const int hq = dblk(dv, c.pmax + 1);
    int clear = 0;
    auto stops = [&](int l_) -> bool { return (long long)l_ + (a.kv.horizon - nrec) <= c.max_iters; };
    KvRec *rec = out.kvr + (size_t)j * a.kv.horizon;
    int32_t *pmxo = out.kvp + (size_t)j * a.kv.horizon;

    // live slots to [0, nr) in order, and the calendar rebuilt
    auto compact = [&]() {
        int kept = 0;
        for (int base = 0; base < ne; base += 32) {
            const int s = base + lane;
            const int4 q = s < ne ? rq[s] : make_int4(0, -1, 0, 0);
            const int e = s < ne ? eb[s] : 0;
            const bool live = q.y >= 0;
            const unsigned m = __ballot_sync(kFull, live);
            __syncwarp();
            if (live) {
                const int d = kept + __popc(m & ((1u << lane) - 1u));
                rq[d] = q;
                eb[d] = e;
            }
            kept += __popc(m);
            __syncwarp();
        }
        ne = tl = kept;
        for (int b = lane; b < kKvCal; b += 32) head[b] = -1;
        if (lane == 0) *ovf = -1;
        __syncwarp();
        for (int s = lane; s < ne; s += 32) {
            const int4 q = rq[s];
            if (q.y == 0) kv_cal_push(head, nxt, ovf, s, kv_end(q, mctx), G);
        }
        pfs = (ne > 0 && rq[ne - 1].y > 0) ? ne - 1 : -1;
        __syncwarp();
    };

    // Up to 32 batches at once, lane k taking batch G + k, while no resident waits
    // (after the first record): then a batch admits nobody, and all it depends on is
    // known at the window's start -- the decoders ending in it (the calendar), those
    // crossing into a new block (the histogram, less the earlier ends of the
    // window), the prefill request's chunk (the budget the decoders leave, summed)
    // and the free blocks (needs and returns, summed).  The window stops before a
    // batch that preempts or in which the prefill request finishes (both taken by
    // the batch step), at a re-file boundary, at the horizon, and after the batch
    // that empties the instance.  The window's ends are listed in the idle waiting
    // ring.  Returns the batches done (0: none).
    int32_t *evn = ovf + 1;  // the window's ends
    bool wstop = false;      // the window's last record may be the last one
    auto window = [&]() -> int {
        const int W = min(min(32, a.kv.horizon - nrec), kKvCal - (G & (kKvCal - 1)));
        if (lane == 0) *evn = 0;
        __syncwarp();
        const int k = lane;
        int cntk = 0;
        long long rck = 0, ebk = 0;
        if (k < W) {
            for (int s = head[(G + k) & (kKvCal - 1)]; s >= 0;) {
                const int ns = nxt[s];
                const int4 q = rq[s];
                if (q.y == 0) {
                    ++cntk;
                    rck += q.x;
                    ebk += eb[s];
                    wq[atomicAdd(evn, 1)] = make_int2(k, s);
                }
                s = ns;
            }
        }
        __syncwarp();
        const int nev = *evn;
        const int endsb = warp_incl_sum32(cntk, lane) - cntk;  // ends before batch k
        const long long rcb = warp_incl_sum64(rck, lane) - rck;
        const int ndk = nd - endsb, nrk = nr - endsb;
        const long long srck = src - rcb;
        // decoders at a block boundary in batch G + k, the window's earlier ends removed
        const int gk = dres(dv, gr + k);
        const int rk = gk == 0 ? 0 : bs - gk;
        int sub = 0;
        for (int e = 0; e < nev; ++e) {
            const int2 ev = wq[e];
            if (ev.x < k && rq[ev.y].w == rk) ++sub;
        }
        const int need_d = ndk > 0 ? hist[rk] - sub : 0;
        // the prefill request's chunk: what the decoders leave, until it finishes
        int x = 0, pneed = 0, ctxp = 0, remk = 0;
        bool pf_ends = false;
        if (pfs >= 0) {
            const int avail = B - ndk;
            const int before = warp_incl_sum32(k < W ? avail : 0, lane) - (k < W ? avail : 0);
            remk = max(0, pP - before);
            x = min(remk, avail);
            pf_ends = remk - x == 0;
            ctxp = pC + (pP - remk);
            pneed = dblk(dv, ctxp + x) - dblk(dv, ctxp);
        }
        const int need_all = need_d + pneed;
        const long long dl = k < W ? ebk - need_all : 0;       // free blocks gained over batch k
        const long long fb = freeb + warp_incl_sum64(dl, lane) - dl;  // free blocks before batch k
        const unsigned okm = __ballot_sync(kFull, k < W && !pf_ends && need_all <= fb);
        int n = okm == kFull ? 32 : __ffs(~okm) - 1;
        const unsigned em = __ballot_sync(kFull, k < n && nrk - cntk == 0);  // the instance empties
        if (em) n = __ffs(em);
        if (n == 0) return 0;
        const bool in = k < n;
        const long long fa = fb - need_all;
        const int bar = B - ndk - x;
        const long long c1 = cf1 + warp_incl_sum64(in ? x : 0, lane);
        const long long c2 = cf2 + warp_incl_sum64(in ? ndk : 0, lane);
        const long long c3 = cf3 + warp_incl_sum64(in ? srck + (long long)ndk * (G + k) : 0, lane);
        const long long c4 = cf4 + warp_incl_sum64(in ? (long long)x * ctxp + (long long)x * (x + 1) / 2 : 0, lane);
        long long thr = 0;
        if (in && bar > 0 && nrk < S) thr = ((long long)bar <= fa * bs) ? kHuge : fa * bs;
        int pm = max(pmx, (int)min(thr, (long long)INT32_MAX));
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, pm, o);
            if (lane >= o) pm = max(pm, y);
        }
        if (in) {
            KvRec R;
            R.cf[0] = c1;
            R.cf[1] = c2;
            R.cf[2] = c3;
            R.cf[3] = c4;
            R.slack = clamp32(fa);  // nrk > 0: the window never starts on an empty instance
            R.far = clamp32(fa);
            R.thr = clamp32(thr);
            R.bar = bar;
            R.bl = bar;
            rec[nrec + k] = R;
            pmxo[nrec + k] = pm;
        }
        // the state after batch n - 1
        const int L = n - 1;
        const int ndL = __shfl_sync(kFull, ndk, L), nrL = __shfl_sync(kFull, nrk, L), cntL = __shfl_sync(kFull, cntk, L);
        const long long srcL = __shfl_sync(kFull, srck, L), rckL = __shfl_sync(kFull, rck, L);
        const long long fbL = __shfl_sync(kFull, fb, L), dlL = __shfl_sync(kFull, dl, L);
        const int xL = __shfl_sync(kFull, x, L), ctxpL = __shfl_sync(kFull, ctxp, L), remL = __shfl_sync(kFull, remk, L);
        cf1 = __shfl_sync(kFull, c1, L);
        cf2 = __shfl_sync(kFull, c2, L);
        cf3 = __shfl_sync(kFull, c3, L);
        cf4 = __shfl_sync(kFull, c4, L);
        pmx = __shfl_sync(kFull, pm, L);
        // the stretch of clear records: all of this window's, or none of it counts (a later
        // end of the records is only longer)
        const bool ck = in && thr >= c.pmax && fa >= hq;
        if (__ballot_sync(kFull, ck) == (n == 32 ? kFull : (1u << n) - 1u)) {
            const int before = clear + __reduce_add_sync(kFull, k < n - 1 ? bar : 0);  // through the record before the last
            wstop = before >= c.pmax;
            clear = min(before + __shfl_sync(kFull, bar, L), 1 << 29);
        } else {
            clear = 0;
        }
        __syncwarp();
        for (int e = lane; e < nev; e += 32) {  // the window's ends leave
            const int2 ev = wq[e];
            if (ev.x < n) {
                atomicSub(&hist[rq[ev.y].w], 1);
                reinterpret_cast<int *>(rq + ev.y)[1] = -1;
            }
        }
        if (in) head[(G + k) & (kKvCal - 1)] = -1;
        if (pfs >= 0) {
            pC = ctxpL + xL;
            pP = remL - xL;
            pH = dblk(dv, pC);
        }
        nd = ndL - cntL;
        nr = nrL - cntL;
        src = srcL - rckL;
        freeb = fbL + dlL;
        nrec += n;
        G += n;
        gr = dres(dv, G);
        if (nr == 0) done = 1;
        __syncwarp();
        return n;
    };

    // The batch step, in two forms.  Both are bound by the chain of shared-memory reads,
    // divisions and branches of one warp (no bandwidth or issue limit is near), and most
    // batches admit, preempt or end one or two requests, so every lane runs them as scalar
    // code on the same values and requests are taken one by one: scans over 32 candidates
    // cost several times what they saved (about 1,900 cycles for a batch with an admission).
    // The prefill request and the waiting head stay in registers.
    int ridx = 0;        // residue of the stored contexts at a block boundary in batch G
    int hp = 0, hd = 0;  // the waiting head (prompt, decode), if any waits
    if (wc > 0) {
        hp = wq[wh].x;
        hd = wq[wh].y;
    }
    // Counts change by reductions that return nothing: a load, an addition and a store by one
    // lane would hold the whole (in-order) warp for a shared-memory round trip.
    auto hist_add = [&](int res, int d) {
        if (lane == 0) asm volatile("red.shared.add.s32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(hist + res)), "r"(d) : "memory");
    };
    // a decoder from batch G + 1 on, in slot s, with context ctx (of residue rem) and dec tokens to go
    auto decode_from_next = [&](int s, int ctx, int rem, int dec) {
        const int x = ctx - (G + 1), z = dec + (G + 1);
        int res = rem - (gr + 1);  // x mod bs
        if (res < 0) res += bs;
        const int4 q = make_int4(x, 0, z, res);
        const long long E = kv_end(q, mctx);
        const int ebv = dblk(dv, (int)(x + E + 1));
        int32_t *h = E < (long long)G + kKvCal ? &head[E & (kKvCal - 1)] : ovf;
        const int hv = *h;
        if (lane == 0) {
            rq[s] = q;
            eb[s] = ebv;
            nxt[s] = hv;
            *h = s;
        }
        hist_add(res, 1);
        __syncwarp();  // the next filing of this batch reads the list's head
        src += x;
        ++nd;
    };
    const int mctx_i = (int)min(mctx, 1LL << 30);  // no context reaches 2^30 tokens
    const int bB = dblk(dv, B - S + 1);            // the least blocks of a whole batch's budget with a seat free
    const bool small = nbk < (1LL << 30);
    for (;;) {
        int l = G + 1;  // this batch
        if (l > c.max_iters) {
            kv_fail(a.ctl, kETraj, lane);
            return;
        }
        if (G > 0 && (G & (kKvCal - 1)) == 0) {
            // re-file the overflow list
            if (lane == 0) {
                int s = *ovf, keep = -1;
                while (s >= 0) {
                    const int ns = nxt[s];
                    const int4 q = rq[s];
                    if (q.y == 0) {
                        const long long E = kv_end(q, mctx);
                        int32_t *h = E < (long long)G + kKvCal ? &head[E & (kKvCal - 1)] : &keep;
                        nxt[s] = *h;
                        *h = s;
                    }
                    s = ns;
                }
                *ovf = keep;
            }
            __syncwarp();
        }
        if (la0 != 0 && wc == 0) {
            const int n = window();
            if (n > 0) {
                if (done || nrec == a.kv.horizon || (wstop && stops(G))) break;
                ridx = gr == 0 ? 0 : bs - gr;
                continue;
            }
        }
        int s_end = 0, budget = 0, ndb = 0;  // (ndb: decoders of this batch)
        int dying = 0;                       // requests leaving after this batch
        long long back = 0;                  // and their blocks
        long long slack = 0, far = 0;        // block slack of the running scan; free blocks after it
        int bar = 0;                         // budget after it
        long long f1 = 0, f3 = 0, f4 = 0;
        bool scanned = false;                // the running scan of this batch is done
        // The lean form, while requests wait and only decoders run: batch after batch until
        // one needs the general form below (a prompt taken in chunks, the last waiting
        // request, no slot left: from after its running scan on) or the calendar, the
        // iteration bound or the horizon is reached.  A batch without any event costs one
        // histogram and one calendar word: it is told by the free blocks staying below
        // `hm`, under which the head cannot get in, and no end.  With it, load 241 -> 144 us
        // on the 64-instance pool (370 before any of this), 255 -> 184 us on 256 instances
        // (405), whose slowest instance steps 455 batches with 129 admissions and 55
        // preemptions.
        if (small && pfs < 0 && wc > 0) {
            int fb = (int)freeb;
            int hb = 0, hrem = 0, hfin = 0, hm = 0;  // the head's blocks, residue and last context; the blocks it needs
            auto derive = [&]() {
                const int qt = (int)udiv32(dv, (unsigned)hp);
                hrem = hp - qt * bs;
                hb = qt + (hrem > 0 ? 1 : 0);
                hfin = min(hp + hd - (MODE == 1 ? 1 : 0), mctx_i);
                hm = nr < S ? min(hb, bB) : kBigKv;
            };
            derive();
            int Gstop = (G | (kKvCal - 1)) + 1;  // the next re-file
            Gstop = min(Gstop, c.max_iters);
            if (la0 != 0) Gstop = min(Gstop, G + (a.kv.horizon - nrec));
            long long r1 = 0, r2 = 0, r3 = 0, r4 = 0;  // features summed here
            long long t3 = src + (long long)nd * G;    // F3 of batch G
            const int G0 = G;
            auto record = [&](long long sl, int fa_, int bar_, int bl_) {
                if (lane == 0) {
                    KvRec R;
                    R.cf[0] = cf1 + r1;
                    R.cf[1] = cf2 + r2;
                    R.cf[2] = cf3 + r3;
                    R.cf[3] = cf4 + r4;
                    R.slack = clamp32(sl);
                    R.far = fa_;
                    R.thr = 0;  // requests wait: no query is admitted
                    R.bar = bar_;
                    R.bl = bl_;
                    rec[nrec] = R;
                    pmxo[nrec] = pmx;
                }
                ++nrec;
            };
            while (G < Gstop) {
                int need = hist[ridx];
                int s = head[G & (kKvCal - 1)];
                int fa = fb - need;
                // decoding only: the next batch's words are read while this one is judged
                while (G < Gstop) {
                    const int rn = ridx == 0 ? bs - 1 : ridx - 1;
                    const int need_n = hist[rn], s_n = head[(G + 1) & (kKvCal - 1)];
                    if (__any_sync(kFull, (fa < 0) | (fa >= hm) | (s >= 0))) break;
                    fb = fa;
                    r2 += nd;
                    r3 += t3;
                    t3 += nd;
                    if (la0 != 0) record(fa, fa, B - nd, B - nd);
                    ++G;
                    ridx = rn;
                    s = s_n;
                    fa = fb - need_n;
                }
                if (G >= Gstop) break;
                slack = nr > 0 ? fa : kHuge;
                if (uni(fa < 0)) {
                    // preemption from the tail (see the general form)
                    const int excess = -fa;
                    int acc = 0;
                    for (int top = tl - 1; uni((top >= 0) & (acc < excess)); top -= 32) {
                        const int s2 = top - lane;
                        unsigned live = __ballot_sync(kFull, s2 >= 0 && reinterpret_cast<const int *>(rq + s2)[1] >= 0);
                        while (uni((live != 0u) & (acc < excess))) {
                            const int r = top - (__ffs(live) - 1);
                            live &= live - 1u;
                            const int4 q = rq[r];
                            wh = wh == 0 ? C - 1 : wh - 1;
                            hp = q.x + G;
                            hd = q.z - G;
                            acc += dblk(dv, hp + 1);
                            src -= q.x;
                            hist_add(q.w, -1);
                            if (lane == 0) {
                                wq[wh] = make_int2(hp, hd);
                                reinterpret_cast<int *>(rq + r)[1] = -1;
                            }
                            ++wc;
                            --nr;
                            tl = r;
                        }
                    }
                    nd = nr;
                    fa = acc - excess;
                    slack = -1;
                    t3 = src + (long long)nd * G;
                    derive();
                    __syncwarp();
                }
                ndb = nd;
                budget = B - nd;
                const int bar_ = budget, far_ = fa;
                f1 = f4 = 0;
                if (uni(fa >= hm)) {
                    do {
                        const int x = min(hp, budget);
                        const bool fits = (x == hp ? hb : dblk(dv, x)) <= fa;
                        // (the general form admits it)
                        scanned = fits & ((x < hp) | (wc == 1) | (hfin <= hp) | (ne == C));
                        if (uni(!fits | scanned)) break;
                        // whole: a decoder from the next batch on, ending in batch G + hfin - hp
                        const int xs = hp - (G + 1), E = G + (hfin - hp);
                        int res = hrem + ridx - 1;  // xs mod bs
                        if (res < 0) res += bs;
                        if (res >= bs) res -= bs;
                        int32_t *h = hfin - hp < kKvCal ? &head[E & (kKvCal - 1)] : ovf;
                        const int hv = *h;
                        wh = wh + 1 == C ? 0 : wh + 1;
                        const int2 wv = wq[wh];  // the next head
                        const int ebv = dblk(dv, hfin), slot = ne++;
                        if (lane == 0) {
                            rq[slot] = make_int4(xs, 0, hd - (MODE == 1 ? 1 : 0) + (G + 1), res);
                            eb[slot] = ebv;
                            nxt[slot] = hv;
                            *h = slot;
                        }
                        hist_add(res, 1);
                        __syncwarp();  // a further admission reads the list's head
                        tl = ne;
                        src += xs;
                        ++nd;
                        ++nr;
                        fa -= hb;
                        budget -= x;
                        f1 += x;
                        f4 += (long long)x * (x + 1) / 2;
                        --wc;
                        hp = wv.x;
                        hd = wv.y;
                        derive();
                    } while (uni((budget > 0) & (nr < S)));
                }
                if (uni(scanned)) {  // this batch goes on below
                    fb = fa;
                    s_end = s;
                    f3 = t3;
                    bar = bar_;
                    far = far_;
                    break;
                }
                fb = fa;
                r1 += f1;
                r2 += ndb;
                r3 += t3;
                r4 += f4;
                if (uni(la0 != 0)) record(slack, far_, bar_, budget);
                if (uni(s >= 0)) {  // the decoders whose last batch this is return their blocks
                    do {
                        const int ns = nxt[s];
                        const int4 q = rq[s];
                        const int ebs = eb[s];
                        if (uni(q.y == 0)) {  // a hole is a request preempted after it was filed
                            fb += ebs;
                            src -= q.x;
                            --nd;
                            hist_add(q.w, -1);
                            if (lane == 0) reinterpret_cast<int *>(rq + s)[1] = -1;
                        }
                        s = ns;
                    } while (uni(s >= 0));
                    if (lane == 0) head[G & (kKvCal - 1)] = -1;
                    nr = nd;
                }
                hm = nr < S ? min(hb, bB) : kBigKv;
                ++G;
                ridx = ridx == 0 ? bs - 1 : ridx - 1;
                t3 = src + (long long)nd * G;
                __syncwarp();
            }
            if (la0 != 0) {
                cf1 += r1;
                cf2 += r2;
                cf3 += r3;
                cf4 += r4;
                if (G != G0) clear = 0;
            } else {
                fcum[0] += G - G0;
                fcum[1] += r1;
                fcum[2] += r2;
                fcum[3] += r3;
                fcum[4] += r4;
            }
            gr = ridx == 0 ? 0 : bs - ridx;
            freeb = fb;
            l = G + 1;
            if (!scanned) {
                if (la0 != 0 && nrec == a.kv.horizon) break;
                continue;
            }
        }
        // A prompt that outruns the free blocks: its first chunk takes a batch's whole budget,
        // the next batch's chunk does not fit, so the request is preempted and, first in the
        // queue again, admitted with the same chunk -- batch after batch, until enough blocks
        // are free or a decoder ends.  Such a batch changes the free blocks alone, and costs
        // the words of a batch without events (the general form took 1,200 cycles; on the
        // 64-instance pool, where 8% of the prompts exceed the budget, half of the slowest
        // instance's time: load 138 -> 80 us).
        if (small && !scanned && pfs >= 0 && pC == B - nd && pP > 0) {
            int F = (int)freeb + pH;                        // the blocks free without this request
            const int more = dblk(dv, pC + min(pP, B - nd));  // what its second chunk would hold
            int Gstop = min((G | (kKvCal - 1)) + 1, c.max_iters);
            if (la0 != 0) Gstop = min(Gstop, G + (a.kv.horizon - nrec));
            const int G0 = G;
            long long t3 = src + (long long)nd * G, r3 = 0;
            const long long tri = (long long)pC * (pC + 1) / 2;
            int s = head[G & (kKvCal - 1)];
            int F1 = F - hist[ridx];
            while (G < Gstop) {
                const int rn = ridx == 0 ? bs - 1 : ridx - 1;
                const int need_n = hist[rn], s_n = head[(G + 1) & (kKvCal - 1)];
                if (__any_sync(kFull, (F1 < pH) | (F1 >= more) | (s >= 0))) break;
                F = F1;
                r3 += t3;
                if (la0 != 0) {
                    if (lane == 0) {
                        const long long k = G - G0 + 1;
                        KvRec R;
                        R.cf[0] = cf1 + k * pC;
                        R.cf[1] = cf2 + k * nd;
                        R.cf[2] = cf3 + r3;
                        R.cf[3] = cf4 + k * tri;
                        R.slack = -1;
                        R.far = F;
                        R.thr = 0;  // no budget is left
                        R.bar = B - nd;
                        R.bl = 0;
                        rec[nrec] = R;
                        pmxo[nrec] = pmx;
                    }
                    ++nrec;
                }
                t3 += nd;
                ++G;
                ridx = rn;
                s = s_n;
                F1 = F - need_n;
            }
            if (G != G0) {
                const long long k = G - G0;
                if (la0 != 0) {
                    cf1 += k * pC;
                    cf2 += k * nd;
                    cf3 += r3;
                    cf4 += k * tri;
                    clear = 0;
                } else {
                    fcum[0] += k;
                    fcum[1] += k * pC;
                    fcum[2] += k * nd;
                    fcum[3] += r3;
                    fcum[4] += k * tri;
                }
                gr = ridx == 0 ? 0 : bs - ridx;
                freeb = F - pH;
                l = G + 1;
                if (la0 != 0 && nrec == a.kv.horizon) break;
                if (G >= Gstop) continue;
            }
        }
        // 1. The running scan.  n_run <= S <= B and only the last request may be in
        //    prefill, so every request gets its tokens if the blocks suffice: one per
        //    decoder, and the last one's chunk from what the decoders leave.
        if (!scanned) {
            int need_all = hist[ridx];  // decoders at a block boundary
            s_end = head[G & (kKvCal - 1)];
            int px = 0, pneed = 0;
            if (pfs >= 0) {
                px = min(pP, B - nd);
                pneed = dblk(dv, pC + px) - pH;
                need_all += pneed;
            }
            f1 = px;
            f4 = (long long)px * pC + (long long)px * (px + 1) / 2;
            if (need_all <= freeb) {
                freeb -= need_all;
                slack = nr > 0 ? freeb : kHuge;
                budget = B - nd - px;
            } else {
                // a request runs out of blocks.  Preempting the tail until each request, in
                // order, has its blocks leaves the longest prefix of the list whose blocks
                // after the batch fit in the instance (what the rest held is what was free
                // to them): those run, the rest go, in order, to the front of the waiting
                // queue.  The prefill request, last, goes first, so the survivors are
                // decoders.  Every request's blocks after the batch sum to what is held plus
                // what the batch needs, so requests leave from the tail until their post-batch
                // blocks reach the excess over nb_j, usually one or two.
                const int excess = need_all - (int)freeb;  // need_all > freeb >= 0
                long long acc = 0;                         // post-batch blocks of those gone
                for (int top = tl - 1; top >= 0 && acc < excess; top -= 32) {
                    const int s = top - lane;
                    unsigned live = __ballot_sync(kFull, s >= 0 && reinterpret_cast<const int *>(rq + s)[1] >= 0);
                    while (live != 0u && acc < excess) {
                        const int r = top - (__ffs(live) - 1);
                        live &= live - 1u;
                        wh = wh == 0 ? C - 1 : wh - 1;
                        if (r != pfs) {
                            const int4 q = rq[r];
                            acc += dblk(dv, q.x + G + 1);
                            src -= q.x;
                            --nd;
                            hp = q.x + G;
                            hd = q.z - G;
                            hist_add(q.w, -1);
                        } else {
                            acc += dblk(dv, pC + px);
                            hp = pC + pP;
                            hd = pD;
                            pfs = -1;
                        }
                        if (lane == 0) {
                            wq[wh] = make_int2(hp, hd);
                            reinterpret_cast<int *>(rq + r)[1] = -1;
                        }
                        ++wc;
                        --nr;
                        tl = r;
                    }
                }
                freeb = acc - excess;
                budget = B - nr;
                f1 = f4 = 0;
                slack = -1;
                __syncwarp();
            }
            ndb = nd;
            f3 = src + (long long)nd * G;
            if (pfs >= 0) {
                // the prefill request's chunk; at its last chunk it turns decoder
                pC += px;
                pP -= px;
                pH += pneed;
                if (pP == 0) {
                    const int dec = pD - (MODE == 1 ? 1 : 0);
                    if (dec <= 0 || (long long)pC >= mctx) {
                        if (lane == 0) reinterpret_cast<int *>(rq + pfs)[1] = -1;
                        back += pH;
                        ++dying;
                    } else {
                        decode_from_next(pfs, pC, dres(dv, pC), dec);
                    }
                    pfs = -1;
                }
            }
            bar = budget;
            far = freeb;
        }
        // slots for every request this batch could admit, those it preempted among them
        // (residents never outnumber the slots)
        if (ne + min(wc, S - nr) > C) {
            __syncwarp();
            compact();
            s_end = head[G & (kKvCal - 1)];
        }
        // 2. Admission from the waiting front while budget, a seat and the first chunk's
        //    blocks allow; one that prefills whole decodes from the next batch.
        while ((budget > 0) & (wc > 0) & (nr < S)) {
            const int x = min(hp, budget);
            const int qt = (int)udiv32(dv, (unsigned)x), rem = x - qt * bs;
            const int nb1 = qt + (rem > 0 ? 1 : 0);
            if (nb1 > freeb) break;
            const int left = hp - x, dec = hd;
            budget -= x;
            freeb -= nb1;
            f1 += x;
            f4 += (long long)x * (x + 1) / 2;
            ++nr;
            const int s = ne++;
            tl = ne;
            wh = wh + 1 == C ? 0 : wh + 1;
            if (--wc > 0) {
                const int2 h = wq[wh];
                hp = h.x;
                hd = h.y;
            }
            if (left > 0) {
                pfs = s;
                pC = x;
                pP = left;
                pD = dec;
                pH = nb1;
                if (lane == 0) rq[s] = make_int4(0, 1, 0, 0);
                break;
            }
            const int dec_a = dec - (MODE == 1 ? 1 : 0);
            if (dec_a <= 0 || (long long)x >= mctx) {
                if (lane == 0) reinterpret_cast<int *>(rq + s)[1] = -1;
                back += nb1;
                ++dying;
            } else {
                decode_from_next(s, x, rem, dec_a);
            }
        }
        const bool qcan = wc == 0;
        if (la0 == 0 && qcan && budget > 0 && nr < S) la0 = l;
        // 3. The batch's record, or the features before the first record.
        bool rstop = false;
        if (la0 != 0) {
            cf1 += f1;
            cf2 += ndb;
            cf3 += f3;
            cf4 += f4;
            // the largest prompt p admitted now: min(p, bl) tokens need at most fa blocks
            long long thr = 0;
            if (qcan && budget > 0 && nr < S) thr = ((long long)budget <= freeb * bs) ? kHuge : freeb * bs;
            pmx = (int)max((long long)pmx, min(thr, (long long)INT32_MAX));
            if (lane == 0) {
                KvRec R;
                R.cf[0] = cf1;
                R.cf[1] = cf2;
                R.cf[2] = cf3;
                R.cf[3] = cf4;
                R.slack = clamp32(slack);
                R.far = clamp32(far);
                R.thr = clamp32(thr);
                R.bar = bar;
                R.bl = budget;
                rec[nrec] = R;
                pmxo[nrec] = pmx;
            }
            ++nrec;
            if (thr >= c.pmax && far >= hq && slack >= hq) {
                rstop = clear >= c.pmax;
                clear = min(clear + budget, 1 << 29);
            } else {
                clear = 0;
            }
        } else {
            fcum[0] += 1;
            fcum[1] += f1;
            fcum[2] += ndb;
            fcum[3] += f3;
            fcum[4] += f4;
        }
        // 4. The decoders whose last batch this is leave and return their blocks.
        if (s_end >= 0) {
            do {
                const int ns = nxt[s_end];
                const int4 q = rq[s_end];
                if (q.y == 0) {  // a hole is a request preempted after it was filed
                    back += eb[s_end];
                    ++dying;
                    src -= q.x;
                    --nd;
                    hist_add(q.w, -1);
                    if (lane == 0) reinterpret_cast<int *>(rq + s_end)[1] = -1;
                }
                s_end = ns;
            } while (s_end >= 0);
            if (lane == 0) head[G & (kKvCal - 1)] = -1;
        }
        nr -= dying;
        freeb += back;
        ++G;
        gr = gr + 1 == bs ? 0 : gr + 1;
        ridx = ridx == 0 ? bs - 1 : ridx - 1;
        __syncwarp();
        if (nr == 0 && wc == 0) {  // no resident left: every later batch is empty
            if (la0 == 0) la0 = l + 1;
            done = 1;
            break;
        }
        if (nrec == a.kv.horizon || (rstop && stops(l))) break;
    }
    if (lane == 0) {
        KvInst hd;
        for (int k = 0; k < 5; ++k) hd.fcum[k] = fcum[k];
        hd.la0 = la0;
        hd.nrec = nrec;
        hd.done = done;
        hd.pad = 0;
        out.kvi[j] = hd;
    }
}

template <int MODE>
__global__ void __launch_bounds__(kKvWarps * 32) k_kv_load(const KvLoad a) {
    extern __shared__ __align__(16) int32_t kv_smem[];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    const int j = blockIdx.x * (int)(blockDim.x >> 5) + wid;
    chain_wait();
    __shared__ int s_active;
    if (threadIdx.x == 0) s_active = load_acquire(&a.ctl->active);
    __syncthreads();
    const int dst = (s_active == 0) ? 1 : 0;
    const StateBuf out = dst ? a.buf1 : a.buf0;
    const size_t per_warp = kv_smem_per_warp(a.cfg, a.kv.hist) / sizeof(int32_t);
    if (j < a.cfg.I) kv_instance<MODE>(a, out, j, lane, kv_smem + wid * per_warp);
    finish_load(a.ctl, dst, gridDim.x);
}

constexpr float kNaN = __builtin_nanf("");
constexpr int kEstWarps = 8;    // warps per CTA
// The two shapes of the estimate.  Sorted: 32 instances per CTA, whose leading records'
// walk fields are staged in shared memory: on pool256, 99.3% of the candidates reach
// their first token within 64 records (88% within 16).  Direct (few queries): an instance
// per warp, so that the walks of a call spread over as many warps as it has (instance,
// 32 queries) units.
template <bool DIRECT>
struct EstShape {
    static constexpr int kGroup = DIRECT ? kEstWarps : 32;  // instances per CTA
    static constexpr int kStage = DIRECT ? 128 : 78;        // leading records staged
    // the staged fields of the walk: (slack, far, thr, bar), bl and the admission maximum
    static constexpr size_t kStageBytes = (size_t)kGroup * kStage * (16 + 2 * 4);
    // and each warp's tile of 32 later records; sorted, three CTAs with their views fit an SM
    static constexpr size_t kTileBytes = 32 * (16 + 4);
    static constexpr size_t kSmem = kStageBytes + kEstWarps * kTileBytes;
};

// The walk's fields of an instance's leading records, in shared memory.
struct KvStage {
    int4 *q;  // slack, far, thr, bar
    int32_t *bl, *pmx;
};
template <typename SH>
__device__ __forceinline__ KvStage kv_stage(unsigned char *smem, int g) {
    constexpr int n = SH::kStage;
    KvStage st;
    st.q = reinterpret_cast<int4 *>(smem) + (size_t)g * n;
    st.bl = reinterpret_cast<int32_t *>(reinterpret_cast<int4 *>(smem) + (size_t)SH::kGroup * n) + (size_t)g * 2 * n;
    st.pmx = st.bl + n;
    return st;
}

// One instance as the estimate reads it: the first `ns` records (with their admission
// maxima) from shared memory; later records through the warp's tile, and their
// admission maxima and the residents' features from global memory.
struct KvView {
    const KvRec *rec;
    const int32_t *pmx;
    long long fcum[5];
    long long nb, mctx;
    float b[5];
    int la0, nrec, ns, done, B, bs;
    Div32 dv;  // division by bs
};

// A warp's tile of 32 consecutive records past the staged ones (the walk's fields).
struct KvTile {
    int4 *q;
    int32_t *bl;
};
template <typename SH>
__device__ __forceinline__ KvTile kv_tile(unsigned char *smem, int w) {
    KvTile tl;
    tl.q = reinterpret_cast<int4 *>(smem + SH::kStageBytes + (size_t)w * SH::kTileBytes);
    tl.bl = reinterpret_cast<int32_t *>(tl.q + 32);
    return tl;
}

// first index in [lo, lo + n) whose value is >= p, in a nondecreasing array
__device__ __forceinline__ int kv_lower_bound(const int32_t *a, int lo, int n, int p) {
    while (n > 0) {
        const int half = n >> 1;
        if (a[lo + half] < p) {
            lo += half + 1;
            n -= half + 1;
        } else {
            n = half;
        }
    }
    return lo;
}

// A candidate's walk: whether it runs, its context and the blocks it holds.  Its own Eq. 9
// features need no sum along the way: the chunks that build a context of c tokens from
// nothing sum to c prefill tokens and c (c + 1) / 2 attention pairs whatever their sizes,
// so only what preemptions discard is kept (lost1, lost4), the whole prompt is added at
// the end, and its one decode token comes at context p.
struct KvWalk {
    bool run;
    int ctx, held;
    long long lost1, lost4;
};

// One batch (record) of the walk of a query of p tokens; true if its first token falls in
// it.  A running query is preempted if the residents' scan leaves a slack below its blocks,
// or if its own tokens need more blocks than are free to it (it is the last running
// request: it preempts itself); a preempted query recomputes its whole context and may be
// readmitted in the same batch.
template <int MODE>
__device__ __forceinline__ bool kv_step(KvWalk &w, const Div32 &dv, int p, const int4 &q, int bl) {
    // Without branches: the lanes of a warp are in different states, a long walk (a query
    // that is admitted, runs out of blocks and is admitted again, batch after batch) takes
    // every case in every record, and the two block counts overlap.
    const int slack = q.x, far = q.y, thr = q.z, bar = q.w;
    const int rem = p - w.ctx;  // 0 only while it waits for its decode token
    const int x = rem > 0 ? min(rem, bar) : 1;
    const int y = min(p, bl);
    const int nh = dblk(dv, w.ctx + x), hy = dblk(dv, y);
    const bool stays = w.run & (slack >= w.held) & ((nh <= far) | (bar <= 0));
    const bool goes = stays & (bar > 0);
    const bool lost = w.run & !stays;
    const bool adm = !stays & (p <= thr);
    if (lost) {
        w.lost1 += w.ctx;
        w.lost4 += (long long)w.ctx * (w.ctx + 1) / 2;
    }
    const bool fin = goes & (MODE == 1 ? x == rem : rem == 0);
    w.held = adm ? hy : goes ? nh : w.held;
    w.ctx = adm ? y : goes ? w.ctx + x : w.ctx;
    w.run = stays | adm;
    return fin | (MODE == 1 && adm && y == p);
}

// The (query, instance) candidates of a warp's lanes (one instance, `live`: the lane
// has one), called by all 32 lanes: each candidate's features and first-token record,
// or an error.  The query waits (pre = p) until the first record whose admission bound
// reaches p, found by binary search over the bounds' running maximum (the staged part
// in shared memory, the rest in global memory), and is followed from there record by
// record to its first token: through the staged records alone, then through the warp's
// tile, which holds the 32 records from the least one a lane still needs (one load of
// 32 records for the warp instead of one dependent load per record and lane).
template <int MODE>
__device__ int kv_candidate(const KvView &v, const KvStage &st, const KvTile &tl, int lane, bool live, int p,
                            long long F[5], int &lt) {
    int err = 0, t = 0;
    KvWalk w = {false, 0, 0, 0, 0};
    bool fin = !live;
    if (live) {
        int lo;
        if (v.ns > 0 && st.pmx[v.ns - 1] >= p) lo = kv_lower_bound(st.pmx, 0, v.ns, p);
        else lo = kv_lower_bound(v.pmx, v.ns, v.nrec - v.ns, p);
        if (lo == v.nrec && !v.done) {
            err = kETraj;
            fin = true;
        }
        for (t = lo; !fin && t < v.ns;) {
            if (kv_step<MODE>(w, v.dv, p, st.q[t], st.bl[t])) fin = true;
            else ++t;
        }
    }
    // after the records the instance is empty; the query then needs at most
    // ceil(p / B) + 2 batches
    const int limit = live ? v.nrec + (v.done ? (p / v.B + 3) : 0) : 0;
    for (;;) {
        if (__ballot_sync(kFull, !fin) == 0u) break;
        const int base = __reduce_min_sync(kFull, fin ? 0x7fffffff : t);  // >= ns
        {
            const int r = base + lane;
            int4 q = make_int4(kBigKv, clamp32(v.nb), kBigKv, v.B);  // past the records: an empty batch
            int bb = v.B;
            if (r < v.nrec) {
                q = __ldg(reinterpret_cast<const int4 *>(&v.rec[r].slack));
                bb = __ldg(&v.rec[r].bl);
            }
            tl.q[lane] = q;
            tl.bl[lane] = bb;
        }
        __syncwarp();
        while (!fin && t < base + 32) {
            if (t >= limit) {
                err = kETraj;
                fin = true;
                break;
            }
            const int k = t - base;
            if (kv_step<MODE>(w, v.dv, p, tl.q[k], tl.bl[k])) fin = true;
            else ++t;
        }
        __syncwarp();  // the tile is read before the next one is written
    }
    if (!live || err) return err;
    lt = t;
    const int tc = min(t, v.nrec - 1);
    long long cf[4] = {0, 0, 0, 0};
    if (tc >= 0) {
        const longlong2 *r = reinterpret_cast<const longlong2 *>(v.rec[tc].cf);
        const longlong2 x = __ldg(r), y = __ldg(r + 1);
        cf[0] = x.x;
        cf[1] = x.y;
        cf[2] = y.x;
        cf[3] = y.y;
    }
    F[0] = v.fcum[0] + t + 1;
    F[1] = v.fcum[1] + cf[0] + w.lost1 + p;
    F[2] = v.fcum[2] + cf[1] + (MODE == 0 ? 1 : 0);
    F[3] = v.fcum[3] + cf[2] + (MODE == 0 ? p : 0);
    F[4] = v.fcum[4] + cf[3] + w.lost4 + (long long)p * (p + 1) / 2;
    return 0;
}

// The call's queries sorted by prompt length, by a counting sort over buckets:
// bucket 0 holds the invalid lengths, bucket 1 + ((p - 1) >> shift) the valid ones.
// A candidate depends on the instance and p alone, so with shift 0 (one bucket per
// length) the estimate runs once per distinct length, on the bucket's first query
// (its leader), and k_kv_expand copies the leader's rows to the bucket's other
// queries; with a coarser shift every query is estimated, in sorted order, which
// keeps the lanes of a warp on near-equal walks through the records.
__device__ __forceinline__ int kv_bucket(int p, int pmax, int shift) {
    return (p >= 1 && p <= pmax) ? 1 + ((p - 1) >> shift) : 0;
}

__global__ void __launch_bounds__(256) k_kv_count(const int32_t *prompt, int Q, int pmax, int shift, int32_t *cnt) {
    chain_wait();
    chain_next();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Q; i += gridDim.x * blockDim.x) {
        const int b = kv_bucket(prompt[i], pmax, shift);
        const unsigned m = __match_any_sync(__activemask(), b);
        if ((threadIdx.x & 31) == __ffs(m) - 1) atomicAdd(&cnt[b], __popc(m));
    }
}

// One CTA: start = run = exclusive prefix sums of the counts, uid = the number of
// non-empty buckets before each one, nu = their total; the counts are cleared for
// the next call, and the estimate's block counters too.  Tiles of 4096 buckets,
// four per thread as one 16-byte word.
constexpr int kScanThreads = 1024;
static_assert(kKvBuckets == kKvScanTiles * 4 * kScanThreads, "scan tiles cover the buckets");
// The bucket scan in two launches, one CTA per tile of 4,096 buckets: the tiles'
// sums (count and non-empty buckets), then each tile's exclusive scan from the sums of
// the tiles before it.  (One CTA over every bucket was bound by one SM's bandwidth.)
__global__ void __launch_bounds__(kScanThreads) k_kv_tile_sums(const int32_t *cnt, int32_t *tsum, int32_t *claim,
                                                               int groups) {
    chain_wait();
    chain_next();
    __shared__ int ws[2][kScanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (blockIdx.x == 0)
        for (int g = tid; g < groups; g += kScanThreads) claim[g] = 0;
    const int4 v = reinterpret_cast<const int4 *>(cnt)[blockIdx.x * kScanThreads + tid];
    int sc = v.x + v.y + v.z + v.w;
    int su = (v.x > 0) + (v.y > 0) + (v.z > 0) + (v.w > 0);
    sc = warp_sum32(sc);
    su = warp_sum32(su);
    if (lane == 0) {
        ws[0][w] = sc;
        ws[1][w] = su;
    }
    __syncthreads();
    if (w == 0) {
        const int xc = warp_sum32(ws[0][lane]), xu = warp_sum32(ws[1][lane]);
        if (lane == 0) {
            tsum[2 * blockIdx.x] = xc;
            tsum[2 * blockIdx.x + 1] = xu;
        }
    }
}

__global__ void __launch_bounds__(kScanThreads) k_kv_scan(int32_t *cnt, int32_t *start, int32_t *run, int32_t *uid,
                                                          int32_t *nu, const int32_t *tsum) {
    __shared__ int ws[2][kScanThreads / 32];
    __shared__ int base[2];
    chain_wait();
    chain_next();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) {  // the tiles before this one
        int c = 0, u = 0;
        for (int t = 0; t < (int)blockIdx.x; ++t) {
            c += tsum[2 * t];
            u += tsum[2 * t + 1];
        }
        base[0] = c;
        base[1] = u;
        if (blockIdx.x == gridDim.x - 1) *nu = u + tsum[2 * blockIdx.x + 1];
    }
    const int b = (blockIdx.x * kScanThreads + tid) * 4;
    const int4 v = reinterpret_cast<const int4 *>(cnt)[b / 4];
    const int sc = v.x + v.y + v.z + v.w;
    const int su = (v.x > 0) + (v.y > 0) + (v.z > 0) + (v.w > 0);
    const int ic = warp_incl_sum32(sc, lane), iu = warp_incl_sum32(su, lane);
    if (lane == 31) {
        ws[0][w] = ic;
        ws[1][w] = iu;
    }
    __syncthreads();
    if (w == 0) {
        const int xc = ws[0][lane], xu = ws[1][lane];
        const int yc = warp_incl_sum32(xc, lane), yu = warp_incl_sum32(xu, lane);
        ws[0][lane] = yc - xc;
        ws[1][lane] = yu - xu;
    }
    __syncthreads();
    int oc = base[0] + ws[0][w] + ic - sc, ou = base[1] + ws[1][w] + iu - su;
    int4 so, uo;
    so.x = oc;
    uo.x = ou;
    oc += v.x;
    ou += v.x > 0;
    so.y = oc;
    uo.y = ou;
    oc += v.y;
    ou += v.y > 0;
    so.z = oc;
    uo.z = ou;
    oc += v.z;
    ou += v.z > 0;
    so.w = oc;
    uo.w = ou;
    reinterpret_cast<int4 *>(start)[b / 4] = so;
    reinterpret_cast<int4 *>(run)[b / 4] = so;
    reinterpret_cast<int4 *>(uid)[b / 4] = uo;
    reinterpret_cast<int4 *>(cnt)[b / 4] = make_int4(0, 0, 0, 0);
}

__global__ void __launch_bounds__(256) k_kv_scatter(const int32_t *prompt, int Q, int pmax, int shift, int32_t *run,
                                                    const int32_t *start, const int32_t *uid, int32_t *order,
                                                    int32_t *leaders) {
    chain_wait();
    chain_next();
    const int lane = threadIdx.x & 31;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Q; i += gridDim.x * blockDim.x) {
        const int b = kv_bucket(prompt[i], pmax, shift);
        const unsigned act = __activemask();
        const unsigned m = __match_any_sync(act, b);
        const int lead = __ffs(m) - 1;
        int base = 0;
        if (lane == lead) base = atomicAdd(&run[b], __popc(m));
        base = __shfl_sync(m, base, lead);
        const int pos = base + __popc(m & ((1u << lane) - 1u));
        order[pos] = i;
        if (pos == start[b]) leaders[uid[b]] = i;
    }
}

// One warp per query row: a query that is not its bucket's leader copies the
// leader's rows (times, and first batches and features if asked for).
__global__ void __launch_bounds__(256) k_kv_expand(const KvEst a) {
    chain_wait();
    const int I = a.cfg.I, lane = threadIdx.x & 31;
    const int warps = gridDim.x * (blockDim.x >> 5);
    const bool v4 = I % 4 == 0 && (reinterpret_cast<uintptr_t>(a.ttft) & 15) == 0;
    const bool f2 = I % 2 == 0 && (reinterpret_cast<uintptr_t>(a.features) & 15) == 0;
    for (int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < a.Q; i += warps) {
        const int L = a.order[a.start[kv_bucket(a.prompt[i], a.cfg.pmax, 0)]];
        if (L == i) continue;
        const size_t ri = (size_t)i * I, rl = (size_t)L * I;
        if (a.ttft) {
            if (v4) {
                const float4 *src = reinterpret_cast<const float4 *>(a.ttft + rl);
                float4 *dst = reinterpret_cast<float4 *>(a.ttft + ri);
                for (int c = lane; c < I / 4; c += 32) dst[c] = src[c];
            } else {
                for (int c = lane; c < I; c += 32) a.ttft[ri + c] = a.ttft[rl + c];
            }
        }
        if (a.first_batch)
            for (int c = lane; c < I; c += 32) a.first_batch[ri + c] = a.first_batch[rl + c];
        if (a.features) {
            if (f2) {
                const int4 *src = reinterpret_cast<const int4 *>(a.features + rl * 5);
                int4 *dst = reinterpret_cast<int4 *>(a.features + ri * 5);
                for (int c = lane; c < I * 5 / 2; c += 32) dst[c] = src[c];
            } else {
                for (int c = lane; c < I * 5; c += 32) a.features[ri * 5 + c] = a.features[rl * 5 + c];
            }
        }
    }
}

// CTA: SH::kGroup instances (strided over the pool), the walk's fields of their leading
// records staged in shared memory.  Sorted: the CTAs of a group claim units of (32
// queries, one instance), the longest prompts first, so the longest walks start first and
// no warp holds more than one instance's walks of one block.  Direct: warp w walks
// instance w of the group, for the query blocks x, x + gridDim.x, ..., in the call's order.
template <int MODE, bool DIRECT>
__global__ void __launch_bounds__(kEstWarps * 32, 3) k_kv_estimate(const KvEst a, bool exact) {
    using SH = EstShape<DIRECT>;
    constexpr int kEstGroup = SH::kGroup, kEstStage = SH::kStage;
    extern __shared__ __align__(16) unsigned char est_smem[];
    __shared__ KvView sv[kEstGroup];
    const DevConfig &c = a.cfg;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // group y holds instances y, y + gy, y + 2 gy, ... (gy groups): every group mixes the
    // pool's models, whose walks differ in length, so the groups' work is alike
    const int gy = gridDim.y;
    const int ng = min(kEstGroup, (c.I - (int)blockIdx.y + gy - 1) / gy);
    chain_wait();
    const int active = load_acquire(&a.ctl->active);
    // the group's views, a thread each
    if ((int)threadIdx.x < ng) {
        const int gw = threadIdx.x;
        const int j = gw * gy + blockIdx.y;
        KvView v;
        v.nb = a.kv.nb[j];
        v.mctx = a.kv.mctx[j];
        v.bs = a.kv.bs[j];
        v.dv = make_div32(v.bs);
        v.B = c.B[j];
        const float *cf = c.coef + 5 * c.moi[j];
        for (int k = 0; k < 5; ++k) v.b[k] = cf[k];
        v.ns = 0;
        v.nrec = 0;
        if (active >= 0) {
            const StateBuf sb = active ? a.buf1 : a.buf0;
            const KvInst hd = sb.kvi[j];
            for (int k = 0; k < 5; ++k) v.fcum[k] = hd.fcum[k];
            v.la0 = hd.la0;
            v.nrec = hd.nrec;
            v.done = hd.done;
            v.rec = sb.kvr + (size_t)j * a.kv.horizon;
            v.pmx = sb.kvp + (size_t)j * a.kv.horizon;
            v.ns = min(v.nrec, kEstStage);
        }
        sv[gw] = v;
    }
    __syncthreads();
    // the walk's fields of the instances' leading records, staged by every thread of the
    // CTA in rounds whose loads are all issued before their stores
    if (active >= 0) {
        constexpr int kRound = 4;
        constexpr int kAll = kEstGroup * kEstStage;
        for (int r0 = 0; r0 < kAll; r0 += kRound * kEstWarps * 32) {
            int4 f_q[kRound];
            int f_bl[kRound], f_pm[kRound];
#pragma unroll
            for (int k = 0; k < kRound; ++k) {
                const int idx = r0 + (int)threadIdx.x + k * kEstWarps * 32;
                const int gw = idx / kEstStage, t = idx - gw * kEstStage;
                if (gw < ng && t < sv[gw].ns) {
                    const KvRec *r = sv[gw].rec + t;
                    f_q[k] = __ldg(reinterpret_cast<const int4 *>(&r->slack));
                    f_bl[k] = __ldg(&r->bl);
                    f_pm[k] = __ldg(sv[gw].pmx + t);
                }
            }
#pragma unroll
            for (int k = 0; k < kRound; ++k) {
                const int idx = r0 + (int)threadIdx.x + k * kEstWarps * 32;
                const int gw = idx / kEstStage, t = idx - gw * kEstStage;
                if (gw < ng && t < sv[gw].ns) {
                    const KvStage st = kv_stage<SH>(est_smem, gw);
                    st.q[t] = f_q[k];
                    st.bl[t] = f_bl[k];
                    st.pmx[t] = f_pm[k];
                }
            }
        }
    }
    __syncthreads();
    // the work: one query per distinct prompt length, or every query, by length
    const int nwork = DIRECT ? a.Q : exact ? *a.nu : a.Q;
    const int32_t *work = exact ? a.leaders : a.order;
    const int nitems = DIRECT ? (w < ng ? (nwork + 31) / 32 : 0) : (nwork + 31) / 32 * ng;
    // Software-pipelined: the claim of the next item and its query's prompt are in
    // flight while the current item is walked.
    int own = blockIdx.x;  // direct: this warp's next query block
    auto claim = [&]() {
        if (DIRECT) {
            const int b = own;
            own += gridDim.x;
            return b;
        }
        int v = 0;
        if (lane == 0) v = atomicAdd(&a.claim[blockIdx.y], 1);
        return __shfl_sync(kFull, v, 0);
    };
    auto fetch = [&](int it_, int &i_, int &p_) {  // this lane's query of item it_ (i_ < 0: none)
        i_ = -1;
        p_ = 0;
        if (DIRECT && it_ < nitems) {
            const int pos_ = it_ * 32 + lane;
            if (pos_ < nwork) {
                i_ = pos_;
                p_ = a.prompt[pos_];
            }
        } else if (it_ < nitems) {
            const int pos_ = nwork - 1 - ((it_ / ng) * 32 + lane);
            if (pos_ >= 0) {
                i_ = work[pos_];
                p_ = a.prompt[i_];
            }
        }
    };
    int it = claim();
    int i_cur, p_cur;
    fetch(it, i_cur, p_cur);
    for (;;) {
        if (it >= nitems) break;
        const int it_next = claim();
        const int g = DIRECT ? w : it - it / ng * ng;
        const int i = i_cur, p = p_cur;
        int i_nx, p_nx;
        fetch(it_next, i_nx, p_nx);
        // every lane of the warp takes part in the walks (their record tiles)
        const KvView &v = sv[g];
        long long F[5] = {-1, -1, -1, -1, -1};
        int lt = -1;
        int err = 0;
        // a query with one output token: its prompt below the context limit and
        // its first token within the instance's blocks
        if (i >= 0) {
            if (active < 0) err = kENoState;
            else if (!(p >= 1 && p <= c.pmax && (long long)p < v.mctx && kv_blocks32(p + 1, v.bs) <= v.nb))
                err = kEInval;
        }
        const int werr = kv_candidate<MODE>(v, kv_stage<SH>(est_smem, g), kv_tile<SH>(est_smem, w), lane,
                                            i >= 0 && err == 0, p, F, lt);
        if (err == 0) err = werr;
        if (i >= 0) {
            float tt = kNaN;
            if (err) {
                record_status(a.ctl, err);
                for (int k = 0; k < 5; ++k) F[k] = -1;
            } else {
                tt = __fmul_rn(v.b[0], __ll2float_rn(F[0]));
                tt = __fmaf_rn(v.b[2], __ll2float_rn(F[2]), tt);
                tt = __fmaf_rn(v.b[1], __ll2float_rn(F[1]), tt);
                tt = __fmaf_rn(v.b[3], __ll2float_rn(F[3]), tt);
                tt = __fmaf_rn(v.b[4], __ll2float_rn(F[4]), tt);
            }
            const size_t idx = (size_t)i * c.I + g * gy + blockIdx.y;
            if (a.ttft) a.ttft[idx] = tt;
            if (a.first_batch) a.first_batch[idx] = err ? -1 : v.la0 + lt;
            if (a.features)
                for (int k = 0; k < 5; ++k) a.features[idx * 5 + k] = F[k];
        }
        it = it_next;
        i_cur = i_nx;
        p_cur = p_nx;
    }
    chain_next();
}

}  // namespace

cudaError_t launch_kv_load(const KvLoad &a, int grid, int warps, size_t smem, cudaStream_t st) {
    return launch_chained(a.cfg.mode == 0 ? k_kv_load<0> : k_kv_load<1>, grid, warps * 32, smem, st, a);
}

cudaError_t set_kv_smem() {
    cudaError_t e = allow_smem(k_kv_load<0>, kSmemMax);
    if (e == cudaSuccess) e = allow_smem(k_kv_load<1>, kSmemMax);
    auto est = [&](auto f, size_t n) {
        if (e == cudaSuccess) e = allow_smem(f, n);
    };
    est(k_kv_estimate<0, false>, EstShape<false>::kSmem);
    est(k_kv_estimate<1, false>, EstShape<false>::kSmem);
    est(k_kv_estimate<0, true>, EstShape<true>::kSmem);
    est(k_kv_estimate<1, true>, EstShape<true>::kSmem);
    return e;
}

cudaError_t launch_kv_estimate(const KvEst &a, int sms, bool expand, bool *leaders, cudaStream_t st) {
    *leaders = false;
    constexpr int thr = kEstWarps * 32;
    // Few queries are walked directly, in one launch.  The sort by prompt length, the walks
    // of distinct lengths alone and the copies of their rows pay for their five further
    // launches once a warp would take several units: while the units make one wave (three
    // CTAs an SM), or up to 1,024 queries at four units a warp, direct is faster.  Event-timed
    // calls, direct / sorted: 24 instances x 4,096 queries 31 / 58 us, 8,192 54 / 52; 64 x
    // 1,024 49 / 87, 2,048 88 / 83; 256 x 1,024 31 / 86, 4,096 95 / 68; 64 x 16 13 / 39.
    const int gd = (a.cfg.I + EstShape<true>::kGroup - 1) / EstShape<true>::kGroup;
    const int qb = (a.Q + 31) / 32, wave = std::max(1, sms * 3 / gd);
    if (qb <= std::max(wave, std::min(32, 4 * wave))) {
        const dim3 grid(std::min(qb, wave), gd);
        return launch_chained(a.cfg.mode == 0 ? k_kv_estimate<0, true> : k_kv_estimate<1, true>, grid, thr,
                              EstShape<true>::kSmem, st, a, false);
    }
    const int gy = (a.cfg.I + EstShape<false>::kGroup - 1) / EstShape<false>::kGroup;
    const int blocks = (a.Q + 32 * kEstWarps - 1) / (32 * kEstWarps);
    const int gx = std::max(1, std::min(blocks, (sms * 3 + gy - 1) / gy));  // three CTAs fit an SM
    const dim3 grid(gx, gy);
    int shift = 0;
    while (2 + ((a.cfg.pmax - 1) >> shift) > kKvBuckets) ++shift;
    const int nbk = 2 + ((a.cfg.pmax - 1) >> shift);
    const bool exact = shift == 0;
    const int g1 = std::max(1, std::min((a.Q + 255) / 256, sms * 4));
    const int tiles = (nbk + 4095) / 4096;
    cudaError_t e = launch_chained(k_kv_count, g1, 256, 0, st, a.prompt, a.Q, a.cfg.pmax, shift, a.cnt);
    if (e == cudaSuccess)
        e = launch_chained(k_kv_tile_sums, tiles, kScanThreads, 0, st, (const int32_t *)a.cnt, a.tsum, a.claim, gy);
    if (e == cudaSuccess)
        e = launch_chained(k_kv_scan, tiles, kScanThreads, 0, st, a.cnt, a.start, a.run, a.uid, a.nu, (const int32_t *)a.tsum);
    if (e == cudaSuccess)
        e = launch_chained(k_kv_scatter, g1, 256, 0, st, a.prompt, a.Q, a.cfg.pmax, shift, a.run, (const int32_t *)a.start,
                           (const int32_t *)a.uid, a.order, a.leaders);
    if (e == cudaSuccess)
        e = launch_chained(a.cfg.mode == 0 ? k_kv_estimate<0, false> : k_kv_estimate<1, false>, grid, thr,
                           EstShape<false>::kSmem, st, a, exact);
    *leaders = exact && !expand;
    if (e == cudaSuccess && exact && expand)
        e = launch_chained(k_kv_expand, std::max(1, std::min((a.Q + 7) / 8, sms * 8)), 256, 0, st, a);
    return e;
}

}  // namespace lr
