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
