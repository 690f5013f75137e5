"""The eviction where its pieces meet the rest of a request: the first block in row panels, wide pooling, launches."""
import numpy as np
import pytest
import torch

from oracle import a3_oracle as O
from paper_2511_17560_b200 import workloads as W
from tests.helpers import oracle_model, oracle_weights
from tests.test_gpu_steps import a3mod, f64, make_engine, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu

TWO_BLOCKS = W.ModelShape("two_blocks", 2, 128, 2, 2, 64, 128, 1000, 1e4, 1e-5)


def check_kept(kept, votes, n_system, n_ctx, nq, tol=2e-3):
    """System prompt and question whole, between them ascending slots whose votes are the largest.  Votes are sums of fp32
    exponentials, 1e-3 relative as for the scores, so which of two candidates nearer than twice that is kept is open."""
    k = len(kept) - n_system - nq
    assert kept[:n_system].tolist() == list(range(n_system)) and kept[n_system + k:].tolist() == list(range(n_ctx, n_ctx + nq))
    sel = kept[n_system:n_system + k]
    assert (np.diff(sel) > 0).all() and sel[0] >= n_system and sel[-1] < n_ctx
    v = votes[n_system:n_ctx]
    thr = np.sort(v)[-k]
    inside = np.isin(np.arange(n_system, n_ctx), sel)
    assert (v[inside] >= thr * (1 - tol)).all() and (v[~inside] <= thr * (1 + tol)).all()


@pytest.mark.parametrize("nq", [4096, 4097, 5000])
def test_votes_of_a_question_longer_than_the_last_panel(a3mod, nq):
    """16 384 rows: the first block walks four panels, the last of them rows 12 288 and on.  A question that begins there, one
    slot before it and far before it: block 0's eviction takes the votes of all of its rows.  The host entry agrees."""
    m, n = TWO_BLOCKS, 16384
    n_ctx, capacity = n - nq, nq + 300
    eng, layers, dev = make_engine(a3mod, m, seed=nq, w_std=0.1)
    g = torch.Generator(device=dev)
    g.manual_seed(nq)
    ck, cv = (torch.randn(m.n_layers, n_ctx, m.n_kv_heads, m.head_dim, device=dev, generator=g).bfloat16() for _ in range(2))
    x0 = torch.randn(n, m.d_model, device=dev, generator=g).bfloat16()
    tab = a3mod.chunk_table([ck], [cv], [0])
    res = []
    for host in (False, True):
        K, V = (torch.zeros(m.n_layers, n, m.n_kv_heads, m.head_dim, device=dev, dtype=torch.bfloat16) for _ in range(2))
        rq, out = eng.make_request(None if host else tab, 1, n_ctx, n_ctx, nq, None if host else x0, K, V, ratio=0.01, evict_capacity=capacity)
        if host:
            rows = torch.empty(out["p"] + nq, dtype=torch.int32).pin_memory()
            x = torch.empty((out["p"] + nq, m.d_model), dtype=torch.bfloat16).pin_memory()
            staging = torch.empty(eng.host_staging_bytes(n_ctx, n), dtype=torch.uint8, device=dev)
            eng.fuse_request_host(rq, [ck.cpu().pin_memory()], [cv.cpu().pin_memory()], x0.cpu().pin_memory(), rows, x, staging)
        else:
            eng.fuse_request(rq)
        assert eng.device_status() == 0
        res.append((K, V, out["kept"], out["k_evicted"], out["v_evicted"]))
    for a, b in zip(*res):
        assert torch.equal(a, b)
    K, _, kept, k_evicted, _ = res[0]
    # block 0 sees the embeddings themselves: its question queries are one norm and one projection away
    model, w = oracle_model(m), oracle_weights(layers)[0]
    pos = np.arange(n_ctx, n)
    a = O.round_bf16(O.rmsnorm(f64(x0[n_ctx:]), w.attn_norm.astype(np.float64), m.rms_eps))
    q, _, _ = O.project_qkv(a, w, model, pos, rnd=O.round_bf16)
    votes = O.eviction_scores(q, pos, f64(K[0]), model, 0, n_ctx)
    for h in range(m.n_kv_heads):
        check_kept(kept[0, h].cpu().numpy(), votes[h], 0, n_ctx, nq)
        assert torch.equal(k_evicted[0, :, h], K[0][kept[0, h].long(), h])
    eng.close()


def evict_setup(a3mod, m, n_ctx, nq, seed):
    eng, _, dev = make_engine(a3mod, m, seed=seed)
    rng = np.random.default_rng(seed)
    K, V = (W.bf16_round(rng.standard_normal((n_ctx + nq, m.n_kv_heads, m.head_dim), dtype=np.float32)) for _ in range(2))
    q = W.bf16_round(rng.standard_normal((nq, m.n_q_heads, m.head_dim), dtype=np.float32))
    pos = np.arange(n_ctx, n_ctx + nq)
    s = np.einsum("jhd,ihd->jhi", q.astype(np.float64), np.repeat(K, m.n_q_heads // m.n_kv_heads, axis=1).astype(np.float64)) / np.sqrt(m.head_dim)
    s[np.broadcast_to(np.arange(n_ctx + nq)[None, None, :] > pos[:, None, None], s.shape)] = -np.inf
    lse = torch.from_numpy(np.log(np.exp(s).sum(axis=2)).astype(np.float32)).to(dev)
    return eng, q, pos, K, (to_dev(q, dev), torch.from_numpy(pos.astype(np.int32)).to(dev), lse, to_dev(K, dev), to_dev(V, dev))


@pytest.mark.parametrize("n_cand,pool,launches", [(95, 1001, 3), (700, 2001, 4), (900, 255, 3), (1024, 249, 3), (1024, 251, 4), (5120, 49, 3),
                                                  (5120, 51, 4), (8192, 31, 3), (8192, 33, 4), (8193, 3, 4), (20000, 7, 4)])
def test_wide_pooling(a3mod, n_cand, pool, launches):
    """Windows as wide as the candidates and wider, both sides of the line between pooling inside the selection and apart."""
    m, nq, n_system = W.TINY_GQA, 9, 5
    n_ctx = n_system + n_cand
    eng, q, pos, K, args = evict_setup(a3mod, m, n_ctx, nq, n_cand + pool)
    k = n_cand // 3
    a3mod.launch_count(reset=True)
    k_out, v_out, kept = eng.evict_layer(*args, n_system, n_ctx, n_system + nq + k, pool)
    assert a3mod.launch_count() == launches
    assert eng.device_status() == 0
    votes = O.pool_scores(O.eviction_scores(q.astype(np.float64), pos, K.astype(np.float64), oracle_model(m), n_system, n_ctx), n_system, n_ctx, pool)
    for h in range(m.n_kv_heads):
        check_kept(kept[h].cpu().numpy(), votes[h], n_system, n_ctx, nq)
        assert torch.equal(k_out[:, h], args[3][kept[h].long(), h]) and torch.equal(v_out[:, h], args[4][kept[h].long(), h])
    eng.close()


@pytest.mark.parametrize("n_cand,pool", [(3073, 3), (4000, 3), (4000, 5), (4000, 7), (5120, 3), (5121, 3), (5121, 5), (5121, 7), (6000, 7), (8191, 5),
                                         (8192, 3), (8192, 7), (8192, 9)])
def test_narrow_windows(a3mod, n_cand, pool):
    """Windows narrower than the five or eight slots of a thread, at both ends of these sizes and beside the first wider one."""
    m, nq, n_system = W.TINY_GQA, 9, 5
    n_ctx, k = n_system + n_cand, n_cand // 5
    eng, q, pos, K, args = evict_setup(a3mod, m, n_ctx, nq, n_cand + pool)
    k_out, _, kept = eng.evict_layer(*args, n_system, n_ctx, n_system + nq + k, pool)
    assert eng.device_status() == 0
    votes = O.pool_scores(O.eviction_scores(q.astype(np.float64), pos, K.astype(np.float64), oracle_model(m), n_system, n_ctx), n_system, n_ctx, pool)
    for h in range(m.n_kv_heads):
        check_kept(kept[h].cpu().numpy(), votes[h], n_system, n_ctx, nq)
        assert torch.equal(k_out[:, h], args[3][kept[h].long(), h])
    eng.close()


@pytest.mark.parametrize("n_cand,pool", [(900, 1), (900, 3), (2000, 5), (4000, 3), (5121, 7), (8192, 7), (8192, 9), (9000, 3)])
def test_votes_that_are_no_numbers(a3mod, n_cand, pool):
    """Infinite votes win their windows, NaN votes are passed over where a window has others and come last where it has not, and either
    is flagged.  Alone, at the ends of the candidates and in a run as wide as a window."""
    m, nq, n_system = W.TINY_GQA, 9, 5
    n_ctx, k, group = n_system + n_cand, n_cand // 5, m.n_q_heads // m.n_kv_heads
    eng, q, pos, K, (dq, dpos, lse, dK, dV) = evict_setup(a3mod, m, n_ctx, nq, n_cand * 3 + pool)
    votes = O.eviction_scores(q.astype(np.float64), pos, K.astype(np.float64), oracle_model(m), n_system, n_ctx)
    nan = [n_system, n_system + 333] + list(range(n_system + 600, n_system + 600 + pool))
    inf = [n_system + 100, n_system + 334, n_ctx - 1]
    dK[nan] = float("nan")
    for g in range(m.n_kv_heads):
        dK[inf, g] = 300 * dq[0, g * group]  # a logit in the thousands
    votes[:, nan], votes[:, inf] = np.nan, np.inf
    k_out, _, kept = eng.evict_layer(dq, dpos, lse, dK, dV, n_system, n_ctx, n_system + nq + k, pool)
    assert eng.device_status() == 2  # A3_DEV_NONFINITE_SCORE
    for h in range(m.n_kv_heads):
        v = np.full(n_ctx, np.nan)
        for i in range(n_system, n_ctx):
            v[i] = np.fmax.reduce(votes[h, max(n_system, i - pool // 2):min(n_ctx, i + pool // 2 + 1)])
        rank = np.where(np.isnan(v), -1.0, np.where(np.isinf(v), 1e30, v))  # infinity before the rest before NaN
        check_kept(kept[h].cpu().numpy(), rank, n_system, n_ctx, nq)
        assert torch.equal(k_out[:, h].view(torch.int16), dK[kept[h].long(), h].view(torch.int16))
    eng.close()


@pytest.mark.parametrize("n_cand,pool", [(8, 31999), (40, 6399), (128, 1999), (300, 853)])
def test_windows_reach_no_further_than_the_candidates(a3mod, n_cand, pool):
    """A window wider than the candidates costs what one that just covers them costs (a walk along its whole width takes 3 to 100
    times as long), and keeps the same."""
    m, nq = W.TINY_GQA, 9
    eng, _, _, _, args = evict_setup(a3mod, m, n_cand, nq, n_cand)
    kept, us = [], []
    for width in (2 * n_cand - 1, pool):
        call = lambda: eng.evict_layer(*args, 0, n_cand, nq + n_cand // 2, width)
        kept.append(call())
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=stream):
            for _ in range(20):
                call()
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            graph.replay()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        us.append(min(times))
    assert eng.device_status() == 0
    for a, b in zip(*kept):
        assert torch.equal(a, b)
    assert us[1] < 1.5 * us[0], us
    eng.close()


@pytest.mark.parametrize("n_system,n_cand,nq,more", [(0, 300, 9, 0), (5, 95, 9, 40), (7, 1, 0, 0), (0, 33, 0, 5)])
def test_everything_fits(a3mod, n_system, n_cand, nq, more):
    """Capacity for the whole cache, or for more: a copy, in one launch (the header promises at most four)."""
    m = W.TINY_GQA
    n_ctx = n_system + n_cand
    eng, _, _, _, (q, pos, lse, K, V) = evict_setup(a3mod, m, n_ctx, nq, n_cand)
    a3mod.launch_count(reset=True)
    k_out, v_out, kept = eng.evict_layer(q, pos, lse, K, V, n_system, n_ctx, n_ctx + nq + more, 7)
    assert a3mod.launch_count() == 1
    assert eng.device_status() == 0
    assert torch.equal(k_out, K) and torch.equal(v_out, V)
    assert torch.equal(kept, torch.arange(n_ctx + nq, dtype=torch.int32, device=kept.device).expand(m.n_kv_heads, -1))
    eng.close()
