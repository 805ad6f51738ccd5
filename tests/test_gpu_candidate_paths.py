"""The candidate kernel's paths against the CPU oracle, bit for bit: instance counts around the
warp and tile edges (rows that are not whole 16-byte words: stored value by value, by the
average-case sources in order through shared memory), prompts around the bound up to which a
candidate's two table entries stay in registers, sweeps with every lane split, and instances
whose prefill total is not exact in fp32.

Times, utilities and assignments are compared exactly (both sides evaluate the same sequence
of IEEE operations)."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2607_18253_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def R():
    from paper_2607_18253_gb300 import router
    return router


def bits(a):
    return np.ascontiguousarray(a, np.float32).view(np.uint32)


def check(wl, sweep=5):
    rt = R().LatencyRouter.from_workload(wl, max_pairs=max(1, sweep))
    rt.load_state(*R().state_tensors(wl))
    p, dh, acc, tau = R().query_tensors(wl)
    Q, I = wl.num_queries, wl.num_instances
    _, lt, t32, _ = oracle.estimate_matrix(wl)
    # estimates, into a buffer whose rows start at any 4-byte word, guarded at both ends
    for shift in (0, 1):
        guard = torch.full((Q * I + 8,), -7.0, device="cuda")
        out = guard[4 + shift:4 + shift + Q * I]
        rt.estimate_ttft(p, out=out)
        np.testing.assert_array_equal(bits(out.cpu().numpy()), bits(t32).ravel())
        assert (guard[:4 + shift] == -7.0).all() and (guard[4 + shift + Q * I:] == -7.0).all()
    for shift in (0, 1):
        guard = torch.full((Q * I + 8,), -7, dtype=torch.int32, device="cuda")
        fb = guard[4 + shift:4 + shift + Q * I]
        rt.estimate_ttft(p, first_batch=fb)
        np.testing.assert_array_equal(fb.cpu().numpy(), lt.ravel())
        assert (guard[:4 + shift] == -7).all() and (guard[4 + shift + Q * I:] == -7).all()
    if I > 1024:
        rt.close()
        return
    # routes, with and without the matrix
    for tt in (None, tau):
        for matrix in (None, torch.empty((Q, I), device="cuda")):
            o = rt.route(p, dh, acc, wl.lam[:1], None if tt is not None else wl.mu[:1], tau=tt, ttft_matrix=matrix)
            a, u, tc = oracle.route(wl, t32, tau=wl.tau if tt is not None else None)
            np.testing.assert_array_equal(o["assign"].cpu().numpy(), a)
            np.testing.assert_array_equal(bits(o["util"].cpu().numpy()), bits(u))
            np.testing.assert_array_equal(bits(o["ttft_chosen"].cpu().numpy()), bits(tc))
            if matrix is not None:
                np.testing.assert_array_equal(bits(matrix.cpu().numpy()), bits(t32))
    if sweep > 1:
        lam, mu = np.linspace(0.0, 3.0, sweep).astype(np.float32), np.geomspace(1e-3, 1.0, sweep).astype(np.float32)
        matrix = torch.empty((Q, I), device="cuda")
        o = rt.route(p, dh, acc, lam, mu, frontier=True, ttft_matrix=matrix)
        a, u, tc = oracle.route(wl, t32, lam=lam, mu=mu)
        np.testing.assert_array_equal(o["assign"].cpu().numpy(), a)
        np.testing.assert_array_equal(bits(o["util"].cpu().numpy()), bits(u))
        np.testing.assert_array_equal(bits(o["ttft_chosen"].cpu().numpy()), bits(tc))
        np.testing.assert_array_equal(bits(matrix.cpu().numpy()), bits(t32))
        np.testing.assert_allclose(o["frontier"].cpu().numpy(), oracle.frontier(wl, a, tc), rtol=1e-12)
    assert rt.status() == R().LR_OK
    rt.close()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("I", [1, 3, 5, 31, 33, 125, 128, 129, 131, 250, 257, 510, 1023, 1025])
def test_instance_counts(I, mode):
    # (a wide pool's tables hold fewer budget boundaries)
    wl = W.small_workload(1000 + I, num_instances=I, num_models=3, num_queries=37, first_token_mode=mode,
                          budget_range=(16, 96) if I < 500 else (64, 128), min_gap=8 if I < 500 else 48)
    gap = wl.max_batched_tokens - wl.max_seqs + 1
    near = int(gap.min()) + 1  # at most one budget boundary lies below a prompt up to this
    wl.prompt_len[:8] = np.clip([1, near - 1, near, near + 1, near + 2, 2 * near, 159, 160], 1, 160)
    check(wl)


@pytest.mark.parametrize("I,Q", [(33, 9000), (257, 5000), (384, 4001), (513, 3000), (640, 2500), (1000, 1500), (1023, 700),
                                 (1024, 65), (3001, 300)])
def test_chunks_and_claims_of_wide_pools(I, Q):
    # calls of several chunks of rows a CTA and of less than one, on the load's stream (equal
    # parts) and on another one (parts and claims): the same results, those of the oracle where
    # sampled, and the average-case source's, whose ragged rows are put in order in shared memory
    wl = W.small_workload(7 + I, num_instances=I, num_models=3, num_queries=Q, budget_range=(64, 128), min_gap=48)
    rt = R().LatencyRouter.from_workload(wl)
    rt.load_state(*R().state_tensors(wl))
    p, dh, acc, tau = R().query_tensors(wl)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()

    def calls(stream):
        with torch.cuda.stream(stream):
            fb = torch.empty((Q, I), dtype=torch.int32, device="cuda")
            o = [rt.estimate_ttft(p, first_batch=fb), fb]
            if I <= 1024:
                for mu, tt, m in ((wl.mu, None, None), (wl.mu, None, torch.empty((Q, I), device="cuda")), (None, tau, None)):
                    r = rt.route(p, dh, acc, wl.lam, mu, tau=tt, ttft_matrix=m)
                    o += [r[k] for k in sorted(r)]
        torch.cuda.synchronize()
        return [x.cpu().numpy() for x in o]

    one, two = calls(torch.cuda.current_stream()), calls(side)
    for a, b in zip(one, two):
        np.testing.assert_array_equal(a.view(np.uint8), b.view(np.uint8))
    t = one[0]
    rng = np.random.default_rng(I)
    cq, cj = rng.integers(0, Q, 2000), rng.integers(0, I, 2000)
    _, lt, t32, _ = oracle.estimate_candidates(wl, cq, cj)
    np.testing.assert_array_equal(bits(t[cq, cj]), bits(t32))
    np.testing.assert_array_equal(one[1][cq, cj], lt)
    if I <= 1024:
        for k, tt in ((2, None), (5, None), (9, wl.tau)):
            a, u, tc = oracle.route(wl, t, tau=tt)
            got = dict(zip(("assign", "ttft_chosen", "util") if k != 5 else ("assign", "ttft_chosen", "ttft_matrix", "util"),
                           one[k:k + 4]))
            np.testing.assert_array_equal(got["assign"], a)
            np.testing.assert_array_equal(bits(got["util"]), bits(u))
            np.testing.assert_array_equal(bits(got["ttft_chosen"]), bits(tc))
            if k == 5:
                np.testing.assert_array_equal(bits(got["ttft_matrix"]), bits(t))
    service = rng.uniform(2.0, 4.0, I)
    theta, tdec, alpha = rng.uniform(3e3, 4e4, I), rng.uniform(0.004, 0.06, I), service * rng.uniform(0.3, 0.95, I)
    k = rng.integers(1, 64, I).astype(np.int32)
    rt.set_queue_params(theta, tdec, alpha, service, k)
    rt.set_ttft_source(R().LR_TTFT_LPS)
    want = oracle.avgcase_matrix(wl, np.array([oracle.lps_wait(*x) for x in zip(alpha, service, k.tolist())]), theta, tdec)[0]
    guard = torch.full((Q * I + 8,), -7.0, device="cuda")
    rt.estimate_ttft(p, out=guard[4:4 + Q * I])
    assert rt.status() == R().LR_OK and (guard[:4] == -7.0).all() and (guard[4 + Q * I:] == -7.0).all()
    np.testing.assert_array_equal(bits(guard[4:4 + Q * I].cpu().numpy()), bits(want).ravel())
    rt.close()


@pytest.mark.parametrize("I", [12, 128, 256])
@pytest.mark.parametrize("grouped", [False, True])
def test_models_of_a_thread(I, grouped):
    # four instances of one model a thread and equal budgets (one bucket width), or mixed models
    wl = W.small_workload(5, num_instances=I, num_models=4, num_queries=300, budget_range=(64, 64), min_gap=8)
    moi = np.arange(I) * 4 // I if grouped else wl.model_of_instance
    wl = dataclasses.replace(wl, model_of_instance=moi.astype(np.int32), max_seqs=np.full(I, 8, np.int32),
                             n_run=np.minimum(wl.n_run, 8))
    # replicas with equal states: ties go to the lowest instance
    for a in (wl.n_run, wl.run_ctx, wl.run_pre, wl.run_dec, wl.n_wait, wl.wait_pre, wl.wait_dec):
        a[1::2] = a[0::2][:a[1::2].shape[0]]
    check(wl)


@pytest.mark.parametrize("P", [2, 3, 8, 31, 32, 33, 64])
def test_sweep_lane_splits(P):
    check(W.small_workload(40 + P, num_instances=45, num_models=3, num_queries=101, budget_range=(16, 96), min_gap=8),
          sweep=P)


@pytest.mark.parametrize("I", [1, 9, 66, 130, 256, 700, 1024])
@pytest.mark.parametrize("Q", [3, 300, 4000])
def test_sweep_splits_the_instances(I, Q):
    # calls of few and many pairs and rows, whose warps split rows, pairs and a row's instances in
    # different ways; equal replicas (ties go to the lowest instance, across lanes too) and an
    # invalid prompt
    if I * Q > 1_200_000:
        Q = 1100
    wl = W.small_workload(9 + I, num_instances=I, num_models=3, num_queries=Q, budget_range=(64, 64), min_gap=48)
    wl = dataclasses.replace(wl, max_seqs=np.full(I, 8, np.int32), n_run=np.minimum(wl.n_run, 8),
                             model_of_instance=(np.arange(I) // 2 * 2 % 3).astype(np.int32))
    for a in (wl.n_run, wl.run_ctx, wl.run_pre, wl.run_dec, wl.n_wait, wl.wait_pre, wl.wait_dec):
        a[1::2] = a[0::2][:a[1::2].shape[0]]
    wl.prompt_len[Q // 2] = 0
    rt = R().LatencyRouter.from_workload(wl, max_pairs=64)
    rt.load_state(*R().state_tensors(wl))
    p, dh, acc, _ = R().query_tensors(wl)
    t = rt.estimate_ttft(p).cpu().numpy()
    assert rt.status() == R().LR_EINVAL and np.isnan(t[Q // 2]).all()
    for P in (2, 3, 16, 64):
        lam, mu = np.linspace(0.0, 3.0, P).astype(np.float32), np.geomspace(1e-3, 1.0, P).astype(np.float32)
        o = rt.route(p, dh, acc, lam, mu)
        a, u, tc = oracle.route(wl, t, lam=lam, mu=mu)
        assert rt.status() == R().LR_EINVAL
        np.testing.assert_array_equal(o["assign"].cpu().numpy(), a)
        ok = a >= 0
        np.testing.assert_array_equal(bits(o["util"].cpu().numpy()[ok]), bits(u[ok]))
        np.testing.assert_array_equal(bits(o["ttft_chosen"].cpu().numpy()[ok]), bits(tc[ok]))
        assert np.isnan(o["util"].cpu().numpy()[~ok]).all() and np.isnan(o["ttft_chosen"].cpu().numpy()[~ok]).all()
    rt.close()


@pytest.mark.parametrize("I", [5, 45, 200])
@pytest.mark.parametrize("P", [1, 2, 5, 33])
def test_objectives_beyond_fp32(I, P):
    # a finite mu or lambda whose product with the time or the cost overflows: the objective is
    # -inf on some instances or on all, and the lowest instance wins the tie, alone or in a sweep
    wl = W.small_workload(50 + P, num_instances=I, num_models=3, num_queries=101, budget_range=(16, 96), min_gap=8)
    wl = dataclasses.replace(wl, coef=wl.coef * np.float32(100.0), price_in=(wl.price_in * 1e6).astype(np.float32))
    rt = R().LatencyRouter.from_workload(wl, max_pairs=P)
    rt.load_state(*R().state_tensors(wl))
    p, dh, acc, _ = R().query_tensors(wl)
    _, _, t32, _ = oracle.estimate_matrix(wl)
    mid = np.float32(np.finfo(np.float32).max / np.median(t32))  # overflows on about half of the candidates
    for lam1, mu1 in ((1.0, 3e38), (1.0, mid), (3e38, 0.0)):
        lam, mu = np.linspace(0.5, 2.0, P).astype(np.float32), np.geomspace(1e-2, 1.0, P).astype(np.float32)
        lam[P // 2], mu[P // 2] = lam1, mu1
        a, u, tc = oracle.route(wl, t32, lam=lam, mu=mu)
        o = rt.route(p, dh, acc, lam, mu, frontier=True)
        np.testing.assert_array_equal(o["assign"].cpu().numpy(), a)
        np.testing.assert_array_equal(bits(o["util"].cpu().numpy()), bits(u))
        np.testing.assert_array_equal(bits(o["ttft_chosen"].cpu().numpy()), bits(tc))
        np.testing.assert_allclose(o["frontier"].cpu().numpy(), oracle.frontier(wl, a, tc), rtol=1e-12)
    assert rt.status() == R().LR_OK
    rt.close()


@pytest.mark.parametrize("I", [64, 256, 512])
@pytest.mark.parametrize("first", [0, 1])
def test_a_model_without_objective(I, first):
    # a cost that overflows times a lambda of 0 is no objective (NaN) on every instance of one
    # model, here whole warps of a wide pool, the first of a row's or its last: the others compete
    wl = W.small_workload(6, num_instances=I, num_models=2, num_queries=200, budget_range=(64, 64), min_gap=8)
    moi = (np.arange(I) * 2 // I).astype(np.int32)
    wl = dataclasses.replace(wl, model_of_instance=moi, max_seqs=np.full(I, 8, np.int32), n_run=np.minimum(wl.n_run, 8),
                             prompt_len=np.maximum(wl.prompt_len, 2))
    wl.price_in[first] = np.finfo(np.float32).max
    rt = R().LatencyRouter.from_workload(wl, max_pairs=2)
    rt.load_state(*R().state_tensors(wl))
    p, dh, acc, _ = R().query_tensors(wl)
    t32 = oracle.estimate_matrix(wl)[2]
    mine = np.flatnonzero(moi != first)
    zero, mu = np.zeros(2, np.float32), np.float32(0.1)
    # U = acc (lambda 0), J = U - mu t (rounded to 64 bits, then to 32: no winner hangs on it here)
    J = (wl.acc[:, 1 - first, None].astype(np.float64) - np.float64(mu) * t32[:, mine]).astype(np.float32)
    want = mine[np.argmax(J, 1)]
    for lam, m in ((zero[:1], [mu]), (zero, [mu, mu])):
        o = rt.route(p, dh, acc, lam, np.array(m, np.float32))
        for k in range(len(lam)):
            np.testing.assert_array_equal(o["assign"][k].cpu().numpy(), want)
            np.testing.assert_array_equal(bits(o["util"][k].cpu().numpy()), bits(wl.acc[:, 1 - first]))
            np.testing.assert_array_equal(bits(o["ttft_chosen"][k].cpu().numpy()), bits(t32[np.arange(len(want)), want]))
    rt.close()


@pytest.mark.parametrize("mode", [0, 1])
def test_prefill_totals_beyond_fp32(mode):
    # one instance whose residents hold more than 2^24 prompt tokens: the whole tile leaves the
    # single-sum path
    I = 40
    wl = W.small_workload(77, num_instances=I, num_models=3, num_queries=33, first_token_mode=mode,
                          budget_range=(1 << 20, 1 << 20), min_gap=1 << 19, max_prompt_len=4000)
    wl.wait_pre[7, :] = (1 << 22) + 12345
    wl.wait_dec[7, :] = 3
    wl.n_wait[7] = wl.cap_waiting
    check(wl)


def test_one_token_prompts():
    # max_prompt_len 1: the tables have a single row
    check(W.small_workload(3, num_instances=9, num_models=2, num_queries=5, max_prompt_len=1))


@pytest.mark.parametrize("P,Q", [(1, 1), (1, 511), (1, 513), (1, 5000), (3, 2048), (19, 2049), (64, 1025)])
def test_frontier_splits(P, Q):
    # one to eight CTAs per pair, ranges that end inside a thread's four queries, and queries
    # without an instance
    wl = W.small_workload(60, num_instances=11, num_models=3, num_queries=Q, budget_range=(16, 64), min_gap=8)
    rt = R().LatencyRouter.from_workload(wl, max_pairs=P)
    rt.load_state(*R().state_tensors(wl))
    p, dh, acc, _ = R().query_tensors(wl)
    lam, mu = np.linspace(0.5, 2.0, P).astype(np.float32), np.geomspace(1e-2, 1.0, P).astype(np.float32)
    o = rt.route(p, dh, acc, lam, mu, frontier=True)
    want = oracle.frontier(wl, o["assign"].cpu().numpy(), o["ttft_chosen"].cpu().numpy())
    np.testing.assert_allclose(o["frontier"].cpu().numpy(), want, rtol=1e-12)
    again = rt.route(p, dh, acc, lam, mu, frontier=True)
    assert torch.equal(o["frontier"].view(torch.int64), again["frontier"].view(torch.int64))
    p[Q // 2] = 0
    bad = rt.route(p, dh, acc, lam, mu, frontier=True)
    assert torch.isnan(bad["frontier"]).all() and rt.status() == R().LR_EINVAL
    rt.close()
