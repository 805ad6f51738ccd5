"""Performance cases of the latency-aware router, through its Python entry points.

Every case is one unit of work that a routing service asks of the library:

  route      a fresh snapshot of the pool is loaded and a batch of queries is routed on it
             (Lagrangian or constrained objective, or a sweep of trade-off pairs), without or
             with KV-cache limits
  estimate   the time-to-first-token matrix of a batch of queries on a snapshot that is loaded
             already (or from the average-case sources, which need none)
  stream     a snapshot is loaded, then a run of arrivals is served decision by decision: the
             pool advances to the arrival with the previous micro-batch appended, and the new
             one is routed; at the end the state is read back
  calibrate  the batch-time coefficients are fitted to a log of executed batches
  evaluate   the baseline policies route a trace and each is scored by OnTimeUtility

Sizes follow the repository's workloads (8, 64 and 256 instances, 3 for the evaluation pool;
16 to 65,536 queries; prompts up to 32,768 tokens), and odd sizes between them.
"""
import math

import numpy as np
import torch

from paper_2607_18253_gb300 import router as R
from paper_2607_18253_gb300 import workloads as W

QPS_PER_INSTANCE = 2.5  # what one instance of the 64-instance pool completes per second when saturated


# ---------------------------------------------------------------------------------------------
# The cases

def _pool(instances, models, run_max, wait_max, median, cap, budget, seqs, beta_acc=False, mode=0):
    return {"instances": instances, "models": models, "run_max": run_max, "wait_max": wait_max, "median": median,
            "cap": cap, "budget": budget, "seqs": seqs, "beta_acc": beta_acc, "mode": mode}


TINY = _pool(8, 2, 32, 16, 512, 4096, 2048, 64)
POOL64 = _pool(64, 4, 64, 64, 1024, 8192, 4096, 64)
POOL256 = _pool(256, 8, 256, 256, 1024, 32768, 8192, 256, beta_acc=True)
PAPER3 = _pool(3, 3, 64, 64, 1024, 8192, 4096, 64)
ROUTE = {"kind": "route", "objective": "lagrangian", "pairs": 1, "matrix": False, "frontier": False, "kv": False}
ESTIMATE = {"kind": "estimate", "source": "sfs", "first_batch": False}
STREAM = {"kind": "stream", "arrivals": "poisson", "load": 0.8, "tracked": False, "kv": False}


def listed():
    return [
        # a handful of queries on a small pool: latency and launches
        dict(ROUTE, name="route_tiny", queries=16, **TINY),
        # one routing tick of a mid-size service: deadlines (Eq. 3), first token with the last chunk
        dict(ROUTE, name="route_pool64_deadlines", queries=4096, **dict(POOL64, mode=1, instances=61), **{
            "objective": "constrained"}),
        # an operator choosing a trade-off: 32 (lambda, mu) pairs and their frontier
        dict(ROUTE, name="sweep_pool64", queries=4096, **POOL64, **{"objective": "sweep", "pairs": 32, "frontier": True}),
        # the large step: 65,536 queries on 256 instances with deep queues, matrix written out
        dict(ROUTE, name="step_pool256", queries=65536, **POOL256, **{"matrix": True}),
        # estimates alone for a ragged pool and batch
        dict(ESTIMATE, name="estimate_pool250", queries=50001, **dict(POOL256, instances=250, models=7)),
        # the average-case (LPS) estimates a service falls back on without snapshots
        dict(ESTIMATE, name="estimate_lps_pool256", queries=16384, **POOL256, **{"source": "lps"}),
        # per-arrival routing of a Poisson stream, 24 arrivals
        dict(STREAM, name="stream_each_arrival", batch=1, decisions=24, **POOL64),
        # bursts: six micro-batches of 256 of an MMPP-2 stream, first tokens tracked
        dict(STREAM, name="stream_bursts_256", batch=256, decisions=6, **POOL64, **{"arrivals": "mmpp2", "tracked": True}),
        # the large step when the engines' KV caches limit admission
        dict(ROUTE, name="step_kv_pool256", queries=65536, **POOL256, **{"kv": True}),
        # a stream under KV-cache limits
        dict(STREAM, name="stream_kv", batch=16, decisions=8, **POOL64, **{"kv": True, "load": 0.5}),
        # refitting the coefficients from the pool's log of executed batches
        dict(kind="calibrate", name="calibrate_4m", rows=4_000_000, models=8, grouped=True, shared=True),
        # a recorded trace scored under the three baselines on the three-instance pool
        dict(kind="evaluate", name="evaluate_paper3", queries=4096, **PAPER3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_pool(rng, most):
    """A pool of up to `most` instances, with the queue depths and limits of a pool of its size."""
    instances = min(most, _log_int(rng, 4, most))
    models = rng.randint(2, min(8, instances))
    depth = rng.choice([16, 32, 64]) if instances <= 64 else rng.choice([64, 128, 256])
    budget = rng.choice([2048, 4096]) if depth <= 64 else 8192
    cap = {2048: 4096, 4096: 8192, 8192: 32768}[budget]
    pool = _pool(instances, models, depth, rng.choice([depth // 2, depth]), rng.choice([512, 1024]), cap, budget,
                 max(64, depth), beta_acc=rng.random() < 0.5, mode=rng.randint(0, 1))
    return pool


def draw(rng):
    kind = rng.choice(["route", "route", "route_kv", "estimate", "stream", "stream_kv", "calibrate", "evaluate"])
    if kind == "calibrate":
        return dict(kind="calibrate", rows=_log_int(rng, 10_000, 3_900_000), models=rng.randint(1, 12),
                    grouped=rng.random() < 0.6, shared=rng.random() < 0.5)
    if kind == "evaluate":
        return dict(kind="evaluate", queries=_log_int(rng, 100, 4096), **_draw_pool(rng, 64))
    if kind in ("stream", "stream_kv"):
        pool = _draw_pool(rng, 64)
        batch = _log_int(rng, 1, 4 * pool["instances"])
        kv = kind == "stream_kv"
        return dict(STREAM, batch=batch, decisions=rng.randint(4, 6 if kv or batch > 16 else 24), **pool, **{
            "kv": kv, "load": rng.choice([0.2, 0.4]) if kv else rng.choice([0.4, 0.6, 0.8]),
            "arrivals": rng.choice(["poisson", "mmpp2"]), "tracked": rng.random() < 0.4})
    pool = _draw_pool(rng, 256)
    if kind == "estimate":
        source = rng.choice(["sfs", "sfs", "lps", "throughput"])
        return dict(ESTIMATE, queries=_log_int(rng, 1, 60_000), **pool, **{
            "source": source, "first_batch": source == "sfs" and rng.random() < 0.3})
    if kind == "route_kv":
        return dict(ROUTE, queries=_log_int(rng, 1, 60_000), **pool, **{
            "kv": True, "objective": rng.choice(["lagrangian", "constrained"])})
    objective = rng.choice(["lagrangian", "constrained", "sweep"])
    pairs = rng.choice([4, 8, 32]) if objective == "sweep" else 1
    return dict(ROUTE, queries=_log_int(rng, 1, 60_000 if pairs == 1 else 8192), **pool, **{
        "objective": objective, "pairs": pairs, "frontier": pairs > 1 or rng.random() < 0.2,
        "matrix": rng.random() < 0.3})


# ---------------------------------------------------------------------------------------------
# Inputs, from the seed alone

def _up(x, m=32):
    return (x + m - 1) // m * m


def _lognormal(g, median, cap, size):
    return np.clip(np.rint(median * np.exp(g.standard_normal(size))), 1, cap).astype(np.int32)


def _workload(case, seed):
    """The pool, its snapshot and the queries: the repository's recipes (decoding requests at
    contexts 128..2048, lognormal prompts and responses) with this case's sizes."""
    I, M, stream = case["instances"], case["models"], case["kind"] == "stream"
    n = case["batch"] * case["decisions"] if stream else case["queries"]
    g, gq = (np.random.default_rng(s) for s in np.random.SeedSequence([seed, 0x0CA5]).spawn(2))
    alpha, beta, gamma, price = W.model_pool(M)
    price = (price * 1e-6).astype(np.float32)
    capR = _up(max(case["run_max"], case["seqs"] if stream else 1))
    # a stream's queues also take what a run of micro-batches sends to one instance
    capW = _up(case["wait_max"] + (min(448, n) if stream else 0))
    n_run = g.integers(0, case["run_max"] + 1, I).astype(np.int32)
    n_wait = g.integers(0, case["wait_max"] + 1, I).astype(np.int32)
    run, wait = np.arange(capR)[None, :] < n_run[:, None], np.arange(capW)[None, :] < n_wait[:, None]
    pairs = case.get("pairs", 1)
    lam, mu = np.array([1.0], np.float32), np.array([0.1], np.float32)
    if pairs > 1:
        L, U = np.meshgrid(np.logspace(-1, 1, max(1, pairs // 8)), np.logspace(-2, 0, min(8, pairs)), indexing="ij")
        lam, mu = L.ravel().astype(np.float32), U.ravel().astype(np.float32)
    prompt = _lognormal(gq, case["median"], case["cap"], n)
    return W.Workload(
        name="case", model_of_instance=(np.arange(I) * M // I).astype(np.int32), coef=W.coefficients(alpha, beta, gamma),
        price_in=price.copy(), price_out=price.copy(), max_batched_tokens=np.full(I, case["budget"], np.int32),
        max_seqs=np.full(I, case["seqs"], np.int32), cap_running=capR, cap_waiting=capW, n_run=n_run,
        run_ctx=np.where(run, g.integers(128, 2049, (I, capR)), 0).astype(np.int32),
        run_pre=np.zeros((I, capR), np.int32),
        run_dec=np.where(run, _lognormal(g, 128, 2048, (I, capR)), 0).astype(np.int32), n_wait=n_wait,
        wait_pre=np.where(wait, _lognormal(g, case["median"], case["cap"], (I, capW)), 0).astype(np.int32),
        wait_dec=np.where(wait, _lognormal(g, 256, 2048, (I, capW)), 0).astype(np.int32), prompt_len=prompt,
        dec_hat=_lognormal(gq, 256, 2048, (n, M)),
        acc=(gq.beta(2.0, 2.0, (n, M)) if case["beta_acc"] else gq.uniform(0.0, 1.0, (n, M))).astype(np.float32),
        tau=W.ttft_targets(gq, prompt), lam=lam, mu=mu, max_prompt_len=case["cap"], first_token_mode=case["mode"], seed=seed)


def _limits(case, wl, seed):
    # a stream runs its queries to their end, an estimate to their first token
    return W.kv_limits(wl, seed, block_sizes=(16,), max_new=2048 if case["kind"] == "stream" else 1)


def _queues(case, seed):
    """Average-case parameters per instance: measured throughputs, loads below saturation."""
    g, I = np.random.default_rng(np.random.SeedSequence([seed, 0x0A7E])), case["instances"]
    service = g.uniform(2.0, 4.0, I)
    return {"prefill_tput": g.uniform(5e3, 5e4, I), "decode_batch_time": g.uniform(0.01, 0.05, I),
            "arrival_rate": service * g.uniform(0.3, 0.95, I), "service_rate": service,
            "parallelism": g.integers(8, 65, I).astype(np.int32)}


def _times(case, wl):
    n, rate = wl.num_queries, case["load"] * QPS_PER_INSTANCE * case["instances"]
    if case["arrivals"] == "mmpp2":
        return W.mmpp2_arrivals(n, rate, 6.0, wl.seed)
    return W.poisson_arrivals(n, rate, wl.seed)


def _log(case, seed):
    """A log of executed batches on the GPU: up to 256 decode tokens at contexts 128..4096 and up to
    two prefill chunks of 1..2048 tokens at contexts 0..8192; times with 4% noise."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n, M = case["rows"], case["models"]

    def integers(lo, hi):
        return torch.randint(lo, hi, (n,), generator=g, device="cuda", dtype=torch.int64)

    model = integers(0, M)
    if case["grouped"]:
        model = model.sort().values
    F = torch.zeros((n, 5), dtype=torch.int64, device="cuda")
    F[:, 0] = 1
    F[:, 2] = integers(0, 257)
    F[:, 3] = F[:, 2] * integers(128, 4097)
    for _ in range(2):
        x, c = integers(0, 2) * integers(1, 2049), integers(0, 8193)
        F[:, 1] += x
        F[:, 4] += x * c + x * (x + 1) // 2
    coef = torch.from_numpy(W.coefficients(*W.model_pool(max(2, M))[:3]).astype(np.float64)).cuda()[model]
    t = (coef * F).sum(1) * (1.0 + 0.04 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
    return F, model.to(torch.int32), t


# ---------------------------------------------------------------------------------------------
# What a user's program holds before the call, and the call

def prepare(case, seed):
    kind = case["kind"]
    if kind == "calibrate":
        F, model, t = _log(case, seed)
        M = case["models"]
        rt = R.LatencyRouter(model_of_instance=np.arange(M), coef=np.ones((M, 5)), price_in=np.ones(M),
                             price_out=np.ones(M), max_batched_tokens=np.full(M, 4096), max_seqs=np.full(M, 64),
                             cap_running=64, cap_waiting=64, max_queries=1, max_prompt_len=8192)
        return {"kind": kind, "rt": rt, "args": (F, model, t), "shared": case["shared"],
                "out": torch.empty((M, 5), dtype=torch.float64, device="cuda")}
    wl = _workload(case, seed)
    p, dh, acc, tau = R.query_tensors(wl)
    rt = R.LatencyRouter.from_workload(wl, max_queries=case["batch"] if kind == "stream" else None)
    if case.get("kv"):
        rt.set_kv_limits(*_limits(case, wl, seed))
    st = {"kind": kind, "rt": rt, "state": R.state_tensors(wl), "wl": wl, "p": p, "dh": dh, "acc": acc, "tau": tau}
    Q, I = wl.num_queries, wl.num_instances
    new = lambda shape, dt=torch.float32: torch.empty(shape, dtype=dt, device="cuda")  # noqa: E731
    if kind == "route":
        st.update(constrained=case["objective"] == "constrained", frontier=case["frontier"],
                  matrix=new((Q, I)) if case["matrix"] else None, out={})
    elif kind == "estimate":
        if case["source"] != "sfs":
            rt.set_queue_params(**_queues(case, seed))
            rt.set_ttft_source(R.LR_TTFT_LPS if case["source"] == "lps" else R.LR_TTFT_THROUGHPUT)
        rt.load_state(*st["state"])
        st.update(out=new((Q, I)), first=new((Q, I), torch.int32) if case["first_batch"] else None)
    elif kind == "stream":
        m, D = case["batch"], case["decisions"]
        t = _times(case, wl)
        st["all"] = {"assign": new((D, m), torch.int32), "util": new((D, m)), "ttft_chosen": new((D, m))}
        cut = [slice(k * m, (k + 1) * m) for k in range(D)]
        st["steps"] = [(float(t[c.stop - 1]), p[c], dh[c], acc[c], {n: v[k:k + 1] for n, v in st["all"].items()})
                       for k, c in enumerate(cut)]
        st["none"] = (new((0,), torch.int32), new((0,), torch.int32), new((0, wl.num_models), torch.int32))
        if case["tracked"]:
            st["first_token"] = torch.full((Q,), float("nan"), dtype=torch.float64, device="cuda")
            rt.track_first_tokens(st["first_token"])
    elif kind == "evaluate":
        rt.load_state(*st["state"])
        st["delay"] = torch.rand(Q, generator=torch.Generator().manual_seed(int(seed))).mul_(0.05).cuda()
        st["outs"] = [{"assign": new((Q,), torch.int32), "util": new((Q,)), "ttft_chosen": new((Q,)),
                       "score": new((2,), torch.float64)} for _ in range(3)]
    return st


def run(s):
    rt, kind = s["rt"], s["kind"]
    if kind == "calibrate":
        return rt.calibrate(*s["args"], shared_beta1=s["shared"], out=s["out"])
    if kind == "estimate":
        rt.estimate_ttft(s["p"], out=s["out"], first_batch=s["first"])
        return {"ttft": s["out"], "first_batch": s["first"]}
    wl = s["wl"]
    if kind == "route":
        rt.load_state(*s["state"])
        return rt.route(s["p"], s["dh"], s["acc"], wl.lam, None if s["constrained"] else wl.mu,
                        tau=s["tau"] if s["constrained"] else None, frontier=s["frontier"], ttft_matrix=s["matrix"],
                        out=s["out"])
    if kind == "stream":
        rt.load_state(*s["state"])
        assign, p, dec, first = *s["none"], 0
        tracked = "first_token" in s
        for t, p1, dh1, acc1, out in s["steps"]:
            rt.advance(assign, p, dec, t, id_base=first if tracked else None)
            first += p.numel()
            rt.route(p1, dh1, acc1, wl.lam, wl.mu, out=out)
            assign, p, dec = out["assign"].view(-1), p1, dh1
        return {"routed": s["all"], "state": rt.read_state(), "first_token": s.get("first_token")}
    for policy, o in enumerate(s["outs"]):  # evaluate
        rt.route_baseline(policy, s["p"], s["dh"], s["acc"], 1.0, rr_start=0, out=o)
        rt.on_time_utility(o["util"], o["ttft_chosen"], s["tau"], s["delay"], out=o["score"])
    return s["outs"]


def work(case):
    """Inputs read once and outputs written once; the arithmetic of one candidate is about 12
    operations (five fused multiply-adds of Eq. 9, the utility and a comparison)."""
    kind = case["kind"]
    if kind == "calibrate":
        return {"bytes": case["rows"] * 52 + case["models"] * 40, "flops": case["rows"] * 50}
    I, M = case["instances"], case["models"]
    snapshot = 4 * I * (2 + 3 * case["run_max"] + 2 * case["wait_max"]) // 2  # half of the slots are taken
    if kind == "stream":
        n = case["batch"] * case["decisions"]
        return {"bytes": 2 * snapshot + n * (16 + 8 * M), "flops": 12 * n * I}
    Q = case["queries"]
    if kind == "estimate":
        return {"bytes": 4 * Q + Q * I * (8 if case["first_batch"] else 4), "flops": 10 * Q * I}
    if kind == "evaluate":
        return {"bytes": 3 * Q * (16 + 8 * M + 12), "flops": 3 * 20 * Q}
    P = case["pairs"]
    return {"bytes": snapshot + Q * (4 + 8 * M) + 12 * P * Q + (4 * Q * I if case["matrix"] else 0),
            "flops": Q * I * (10 + 4 * P)}


def tolerance(case):
    # calibration: exact integer sums, then one 4x4 or 5x5 solve in fp64 (6e-12 off a least-squares
    # solver on the rows at 4,000,000 rows; fewer rows are conditioned worse)
    if case["kind"] == "calibrate":
        return {"rel": 1e-10}
    # fp32 times and utilities of five terms, one rounding per operation: 3e-8 to 4.6e-8 off 64 bits in
    # the norm, a few units of 6e-8 at most for one value; whole numbers (assignments, batch
    # indices, states) agree
    return {"rel": 2e-7, "max": 8e-7, "differ": 0.0}


# ---------------------------------------------------------------------------------------------
# The same results in plain numpy, 64 bits

def _blocks(c, bs):
    return -(-c // bs)


class _Residents:
    """One instance's resident requests, stepped batch by batch (chunked prefill, FCFS)."""

    def __init__(self, wl, j, limits=None):
        nr, nw = int(wl.n_run[j]), int(wl.n_wait[j])
        self.ctx, self.pre, self.dec = (a[j, :nr].astype(np.int64) for a in (wl.run_ctx, wl.run_pre, wl.run_dec))
        self.wait = [(int(a), int(b)) for a, b in zip(wl.wait_pre[j, :nw], wl.wait_dec[j, :nw])]
        self.B, self.S, self.mode = int(wl.max_batched_tokens[j]), int(wl.max_seqs[j]), wl.first_token_mode
        self.bs, self.nb, self.mctx = (int(a[j]) for a in limits) if limits else (1, 1 << 60, 1 << 60)
        self.F = np.zeros(5, np.int64)  # features summed over the batches done

    def step(self):
        """One batch.  Returns (budget after the running scan, budget left, whether a request at the
        tail would be admitted, block slack of the scan, free blocks after it, free blocks left)."""
        ctx, pre, dec = self.ctx, self.pre, self.dec
        need = np.where(pre > 0, pre, 1)
        x = np.clip(self.B - (np.cumsum(need) - need), 0, need)
        free = self.nb - int(_blocks(ctx, self.bs).sum())
        want = _blocks(ctx + x, self.bs) - _blocks(ctx, self.bs)
        slack = free - int(want.sum()) if ctx.size else 1 << 62
        if slack < 0:  # in order, the last running request gives way
            n, i, budget, got = ctx.size, 0, self.B, []
            while i < n and budget > 0:
                xi = min(int(need[i]), budget)
                wi = int(_blocks(ctx[i] + xi, self.bs) - _blocks(ctx[i], self.bs))
                while free < wi and n > i:
                    n -= 1
                    free += int(_blocks(ctx[n], self.bs))
                if i >= n:
                    break
                free -= wi
                budget -= xi
                got.append(xi)
                i += 1
            self.wait[:0] = [(int(ctx[k] + pre[k]), int(dec[k])) for k in range(n, ctx.size)]
            ctx, pre, dec, x = ctx[:n], pre[:n], dec[:n], np.zeros(n, np.int64)
            x[:len(got)] = got
            slack = -1
        else:
            free -= int(want.sum())
            budget = self.B - int(x.sum())
        after_scan, far = budget, free
        chunk = np.where(pre > 0, x, 0)
        token = (pre == 0) & (x > 0)
        f = [1, int(chunk.sum()), int(token.sum()), int(ctx[token].sum()), int((chunk * ctx + chunk * (chunk + 1) // 2).sum())]
        new = []
        while self.wait and budget > 0 and ctx.size + len(new) < self.S:
            p, d = self.wait[0]
            c = min(p, budget)
            if int(_blocks(c, self.bs)) > free:
                break
            self.wait.pop(0)
            new.append((c, p - c, d - (1 if p == c and self.mode == 1 else 0)))
            budget -= c
            free -= int(_blocks(c, self.bs))
            f[1] += c
            f[4] += c * (c + 1) // 2
        joins = not self.wait and budget > 0 and ctx.size + len(new) < self.S
        left = free
        self.F = self.F + np.array(f, np.int64)
        done = (pre > 0) & (pre == x)
        dec = dec - token - (done if self.mode == 1 else 0)
        ctx, pre = ctx + x, pre - chunk
        if new:
            a = np.array(new, np.int64)
            ctx, pre, dec = (np.concatenate([u, a[:, k]]) for k, u in enumerate((ctx, pre, dec)))
        keep = (dec > 0) & ((pre > 0) | (ctx < self.mctx))
        self.ctx, self.pre, self.dec = ctx[keep], pre[keep], dec[keep]
        return after_scan, budget, joins, slack, far, left


def _times_plain(wl, j, lengths):
    """Features of a query of each length (ascending) on instance j up to its first token."""
    r, off = _Residents(wl, j), 1 - wl.first_token_mode
    while True:
        _, budget, joins, *_ = r.step()
        if joins:
            break
    la, reach, at = int(r.F[0]), [budget], [r.F]
    while reach[-1] < lengths[-1]:
        _, budget, *_ = r.step()
        reach.append(reach[-1] + budget)
        at.append(r.F)
    r.step()
    at.append(r.F)
    k = np.searchsorted(np.array(reach), lengths, "left")
    F = np.array(at)[k + off].copy()
    F[:, 1] += lengths
    F[:, 2] += off
    F[:, 3] += off * lengths
    F[:, 4] += lengths * (lengths + 1) // 2
    return F, la + k + off


def _times_kv(wl, j, lengths, limits):
    """The same under KV-cache limits: the query, last in the list, is followed batch by batch."""
    r = _Residents(wl, j, limits)
    n = lengths.size
    pre, ctx, held = lengths.copy(), np.zeros(n, np.int64), np.zeros(n, np.int64)
    on, out, own = np.zeros(n, bool), np.zeros((n, 5), np.int64), np.zeros((n, 5), np.int64)
    todo = np.arange(n)
    while todo.size:
        scan, budget, joins, slack, far, left = r.step()
        if not joins and not on[todo].any():
            continue
        t = todo
        p, c, run, o = pre[t], ctx[t], on[t], own[t]
        first = np.zeros(t.size, bool)
        x = np.where(p > 0, np.minimum(p, scan), 1)
        # waits to be admitted again if a resident needs its blocks, or its own tokens do not fit
        lost = run & ((slack < held[t]) | ((scan > 0) & (_blocks(c + x, r.bs) > far)))
        go = run & ~lost & (scan > 0)
        chunk = go & (p > 0)
        o[chunk, 1] += x[chunk]
        o[chunk, 4] += (x * c + x * (x + 1) // 2)[chunk]
        token = go & (p == 0)
        o[token, 2] += 1
        o[token, 3] += c[token]
        first |= token
        p = np.where(lost, p + c, np.where(chunk, p - x, p))
        c = np.where(lost, 0, np.where(go, c + x, c))
        h = np.where(lost, 0, np.where(go, _blocks(c, r.bs), held[t]))
        run = run & ~lost
        if joins:
            y = np.minimum(p, budget)
            adm = ~run & ~first & (_blocks(y, r.bs) <= left)
            o[adm, 1] += y[adm]
            o[adm, 4] += (y * (y + 1) // 2)[adm]
            c, p, h = np.where(adm, y, c), np.where(adm, p - y, p), np.where(adm, _blocks(y, r.bs), h)
            run = run | adm
            chunk = chunk | adm
        if wl.first_token_mode == 1:
            first |= chunk & run & (p == 0)
        pre[t], ctx[t], held[t], on[t], own[t] = p, c, h, run, o
        out[t[first]] = r.F + o[first]
        todo = t[~first]
    return out, out[:, 0].copy()


def _matrix(case, wl, seed):
    """[Q][I] times to first token in 64 bits, and first-token batch indices."""
    lengths, back = np.unique(wl.prompt_len.astype(np.int64), return_inverse=True)
    limits = _limits(case, wl, seed) if case.get("kv") else None
    T, N = np.empty((lengths.size, wl.num_instances)), np.empty((lengths.size, wl.num_instances), np.int64)
    coef = wl.coef.astype(np.float64)
    for j in range(wl.num_instances):
        F, N[:, j] = _times_kv(wl, j, lengths, limits) if limits else _times_plain(wl, j, lengths)
        T[:, j] = F.astype(np.float64) @ coef[wl.model_of_instance[j]]
    return T[back], N[back]


def exact(case, seed):
    kind = case["kind"]
    if kind == "stream":
        # every batch is a decision on the fp32 batch times the library defines (whether it ends by
        # the arrival), so wider times give another stream, not the same one more exactly
        return None
    if kind == "calibrate":
        F, model, t = (a.cpu().numpy() for a in _log(case, seed))
        out = np.full((case["models"], 5), np.nan)
        for m in range(case["models"]):
            X = F[model == m].astype(np.float64)
            if case["shared"]:
                X = np.stack([X[:, 0], X[:, 1] + X[:, 2], X[:, 3], X[:, 4]], 1)
            size = np.sqrt((X * X).mean(0))
            w = np.linalg.lstsq(X / size, t[model == m], rcond=None)[0] / size
            out[m] = w[[0, 1, 1, 2, 3]] if case["shared"] else w
        return out
    wl = _workload(case, seed)
    p, moi = wl.prompt_len.astype(np.float64), wl.model_of_instance
    if kind == "estimate" and case["source"] != "sfs":
        q = _queues(case, seed)
        if case["source"] == "lps":
            wait = (q["arrival_rate"] / q["service_rate"]) ** q["parallelism"] / (q["service_rate"] - q["arrival_rate"])
        else:
            wait = (wl.run_pre.sum(1, dtype=np.int64) + wl.wait_pre.sum(1, dtype=np.int64)) / q["prefill_tput"]
        return {"ttft": wait + q["decode_batch_time"] + p[:, None] / q["prefill_tput"], "first_batch": None}
    T, _ = _matrix(case, wl, seed)
    if kind == "estimate":
        return {"ttft": T, "first_batch": None}
    cost = wl.dec_hat * wl.price_out.astype(np.float64) + p[:, None] * wl.price_in.astype(np.float64)
    acc, rows = wl.acc.astype(np.float64), np.arange(wl.num_queries)
    if kind == "evaluate":
        level, outs = (wl.n_run + wl.n_wait).astype(np.int64), []
        delay = torch.rand(wl.num_queries, generator=torch.Generator().manual_seed(int(seed))).mul_(0.05).numpy()
        U = (acc - cost)[:, moi]
        for policy in range(3):
            j = rows % wl.num_instances if policy == 0 else U.argmax(1)
            if policy == 1:
                queue = level.copy()
                for i in rows:
                    j[i] = queue.argmin()
                    queue[j[i]] += 1
            ok = T[rows, j] + delay <= wl.tau
            outs.append({"assign": None, "util": U[rows, j], "ttft_chosen": T[rows, j],
                         "score": np.array([(U[rows, j] * ok).mean(), ok.mean()])})
        return outs
    picks, front = [], []
    for lam, mu in zip(wl.lam.astype(np.float64), wl.mu.astype(np.float64)):
        U = (acc - lam * cost)[:, moi]
        if case["objective"] == "constrained":
            fits = T <= wl.tau[:, None]
            j = np.where(fits.any(1), np.where(fits, U, -np.inf).argmax(1), T.argmin(1))
        else:
            j = (U - mu * T).argmax(1)
        picks.append((U[rows, j], T[rows, j]))
        front.append([acc[rows, moi[j]].mean(), cost[rows, moi[j]].mean(), T[rows, j].mean()])
    out = {"assign": None, "util": np.array([u for u, _ in picks]), "ttft_chosen": np.array([t for _, t in picks])}
    if case["frontier"]:
        out["frontier"] = np.array(front)
    if case["matrix"]:
        out["ttft_matrix"] = T
    return out
