"""The paths that only launches of few rows take: GEMMs whose k-loop is cut into slices, added up by the kernel that follows
(output and down projection) or within a cluster (QKV projection), and attention whose keys are shared out to a cluster of CTAs.

The models here are the smallest whose matrices are deep enough to be cut (at least two slices of 1 024).  Gates as in
tests/test_gpu_steps.py: the slices are fp32 sums of the same products, so the bounds derived there hold unchanged.
"""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import a3_oracle as O
from paper_2511_17560_b200 import workloads as W
from tests.helpers import oracle_model, oracle_weights
from tests.test_gpu_steps import a3mod, check_kv, f64, hidden_rows_scale, make_engine, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu

# d_model 896: the last 256-feature block is half empty; d_ff 2176 = 17 ring stages: slices of 8 and 9
DEEP = W.ModelShape("deep", 2, 896, 16, 4, 128, 2176, 32000, 5e5, 1e-5)


# QKV: 17 ring stages in halves of 8 and 9; 15 heads, so the last pair of CTAs has one without a head
BROAD = W.ModelShape("broad", 1, 2176, 9, 3, 128, 640, 32000, 5e5, 1e-5)


# two layers are 243 MB, more than L2: every weight of a launch of one token tile leaves L2 first; down projection in 8 slices,
# which the adding kernel takes in its loop
BEYOND_L2 = W.ModelShape("beyond_l2", 2, 2048, 16, 4, 128, 8192, 32000, 5e5, 1e-5)


def layer_parity(a3mod, m, M, seed):
    eng, layers, dev = make_engine(a3mod, m, seed=seed, w_std=0.05 * (512 / m.d_model) ** 0.5)
    model, weights = oracle_model(m), oracle_weights(layers)
    rng = np.random.default_rng(300 + seed)
    kv_len, layer = M + 37, m.n_layers - 1
    pos = np.sort(rng.choice(kv_len, size=M, replace=False))
    pos[-1] = kv_len - 1
    X = W.bf16_round(rng.standard_normal((M, m.d_model), dtype=np.float32))
    Kc, Vc = W.make_cache_like(m, kv_len, seed, 9, std=1.0)
    dpos = torch.from_numpy(pos.astype(np.int32)).to(dev)
    outs = []
    for _ in range(2):
        dX, dK, dV = to_dev(X, dev), to_dev(Kc[layer], dev), to_dev(Vc[layer], dev)
        eng.recompute_layer(layer, dX, dpos, dK, dV)
        assert eng.device_status() == 0
        outs.append((dX, dK, dV))
    for a, b in zip(*outs):
        assert torch.equal(a, b)  # the slices are added in a fixed order
    Ko, Vo = Kc[layer].astype(np.float64), Vc[layer].astype(np.float64)
    _, parts = O.recompute_layer(X.astype(np.float64), pos, weights[layer], model, Ko, Vo, rnd=O.round_bf16, return_parts=True)
    gX, gK, gV = (f64(t) for t in outs[0])
    check_kv(gK[pos], parts["k_exact"], "recomputed K rows")
    check_kv(gV[pos], parts["v_exact"], "recomputed V rows")
    keep = np.ones(kv_len, bool)
    keep[pos] = False
    np.testing.assert_array_equal(gK[keep], Kc[layer][keep])
    np.testing.assert_array_equal(gV[keep], Vc[layer][keep])
    check_kv(gX, parts["x_exact"], "hidden rows", scale=hidden_rows_scale(parts["x_exact"]))
    eng.close()


@pytest.mark.parametrize("M", [1, 16, 17, 255, 256, 257, 470])
def test_residual_gemm_in_slices(a3mod, M):
    """Output and down projection of few rows: one token, ragged and full token tiles, two tiles."""
    layer_parity(a3mod, DEEP, M, seed=M)


@pytest.mark.parametrize("M", [1, 16, 17, 75, 255, 256, 257])
def test_qkv_projection_in_halves(a3mod, M):
    """Two pairs of CTAs per two heads, up to one full token tile: one token, warp sets with and without tokens."""
    layer_parity(a3mod, BROAD, M, seed=M + 1)


@pytest.mark.parametrize("M", [1, 75, 256, 257])
def test_layer_of_a_stack_beyond_l2(a3mod, M):
    """One token tile (the instances that mark the weights) and two (those that do not)."""
    layer_parity(a3mod, BEYOND_L2, M, seed=M + 2)


# one layer that L2 holds; 38 feature blocks of SwiGLU, 8 of the down projection (38 ring stages in four slices)
TWO_TILES = W.ModelShape("two_tiles", 1, 2048, 16, 4, 128, 4864, 32000, 5e5, 1e-5)


@pytest.mark.parametrize("m", [BEYOND_L2, TWO_TILES], ids=lambda m: m.name)
@pytest.mark.parametrize("M", [257, 289, 320, 321, 471])
def test_two_token_tiles_on_one_stream_of_weights(a3mod, m, M):
    """Row counts around those at which units take two token tiles, on widths that keep one tile per unit (the widths that take two:
    test_accumulators_of_two_token_tiles_take_turns, test_slices_of_two_token_tiles): the oracle's layer, and the gate/up product bit
    for bit whatever the tiling."""
    layer_parity(a3mod, m, M, seed=M + 4)
    eng, _, dev = make_engine(a3mod, m, seed=M, w_std=0.05)
    g = torch.Generator(device=dev)
    g.manual_seed(M)
    x = torch.randn(M, m.d_model, device=dev, generator=g).bfloat16()
    both = eng.swiglu_rows(0, x)
    eng.set_option(a3mod.OPT_GEMM_TILING, 1)
    assert torch.equal(both, eng.swiglu_rows(0, x))
    assert eng.device_status() == 0
    eng.close()


# gate/up product: one, two and three units per pair of CTAs (64, 148 and 222 feature blocks, 74 pairs), the smallest depths at which a
# unit takes two token tiles
SWIGLU_UNITS = {units: W.ModelShape(f"units_{units}", 1, d_model, 1, 1, 128, d_ff, 1000, 1e4, 1e-5)
                for units, d_model, d_ff in ((1, 2560, 8192), (2, 2560, 18944), (3, 2688, 28416))}


@pytest.mark.parametrize("units", [1, 2, 3])
@pytest.mark.parametrize("M", [257, 272, 288])
def test_accumulators_of_two_token_tiles_take_turns(a3mod, units, M):
    """Two, four and six accumulators in three slots of tensor memory: slots that are used once, that are taken again (behind a drained
    accumulator, a unit astride the last and the first slot), all of them.  Bit for bit the product of one tile per unit."""
    m, dev = SWIGLU_UNITS[units], torch.device("cuda:0")
    assert a3mod.plan_layer(m, M)["swiglu_tiles"] == 2 and -(-m.d_ff // 128 // 74) == units
    eng = a3mod.A3(m, W.make_weights_device(m, dev, units), M)
    g = torch.Generator(device=dev)
    g.manual_seed(M)
    x = torch.randn(M, m.d_model, device=dev, generator=g).bfloat16()
    both = eng.swiglu_rows(0, x)
    again = eng.swiglu_rows(0, x)
    eng.set_option(a3mod.OPT_GEMM_TILING, 1)
    one = eng.swiglu_rows(0, x)
    assert eng.device_status() == 0
    assert torch.equal(both, one) and torch.equal(both, again)
    w = eng._weights[0]
    rows = torch.tensor([0, M // 2, 143, 144, M - 1], device=dev)
    gate, up = (x[rows].double() @ w[name].double().T for name in ("w_gate", "w_up"))
    want = torch.nn.functional.silu(gate) * up
    # one bf16 rounding (2^-9 of the value) besides fp32 sums of d_model products, silu_mul's 2^-21 and its cancellation near zero
    assert ((both[rows].double() - want).abs() <= 2 ** -8 * want.abs() + 1e-5 * want.abs().max()).all()
    eng.close()


# the widths at which a slice of the down projection takes two token tiles: five slices of Qwen-7B's to 352 rows, of 3 200 x 13 440 at 257
QWEN_LAYER = replace(W.QWEN7B, n_layers=1)
TWO_TILE_SLICES = W.ModelShape("two_tile_slices", 1, 3200, 16, 4, 128, 13440, 32000, 5e5, 1e-5)


@pytest.mark.parametrize("m,M", [(QWEN_LAYER, M) for M in (257, 270, 289, 320, 321, 352)] + [(TWO_TILE_SLICES, 257)])
def test_slices_of_two_token_tiles(a3mod, m, M):
    """The same slices with one token tile each: bit for bit, since neither their number nor the cuts of the k-loop depend on it.
    Undivided sums: within what one rounding of the hidden row leaves (hidden_rows_scale's gates)."""
    assert a3mod.plan_layer(m, M)["down_tiles"] == 2
    dev = torch.device("cuda:0")
    eng = a3mod.A3(m, W.make_weights_device(m, dev, M), M)
    g = torch.Generator(device=dev)
    g.manual_seed(M)
    x0 = torch.randn(M, m.d_model, device=dev, generator=g).bfloat16()
    pos = torch.arange(M, dtype=torch.int32, device=dev)
    outs = {}
    for residual in (1, 3, 2):
        eng.set_option(a3mod.OPT_RESIDUAL_T, residual)
        x, K, V = x0.clone(), *(torch.zeros(M, m.n_kv_heads, m.head_dim, device=dev, dtype=torch.bfloat16) for _ in range(2))
        eng.recompute_layer(0, x, pos, K, V)
        assert eng.device_status() == 0
        outs[residual] = x
    assert torch.equal(outs[1], outs[3])
    exact = f64(outs[2])
    check_kv(f64(outs[1]), exact, "hidden rows", scale=hidden_rows_scale(exact))
    eng.close()


def test_two_token_tiles_of_a_slice_against_the_oracle(a3mod):
    layer_parity(a3mod, TWO_TILE_SLICES, 257, seed=11)


# rows of more than 4 096 values: what the threads of the adding kernel do not keep in registers is read again; both of a layer's
# residual products in two slices
LONG_ROWS = W.ModelShape("long_rows", 1, 4224, 16, 4, 128, 2176, 32000, 5e5, 1e-5)


@pytest.mark.parametrize("M", [1, 17])
def test_slices_added_to_long_rows(a3mod, M):
    layer_parity(a3mod, LONG_ROWS, M, seed=M + 3)


@pytest.mark.parametrize("d_model", [4224, 8448])
def test_long_rows_enter_a_request(a3mod, d_model):
    """Copied, gathered and normed by one kernel: the request that recomputes everything is the layer-by-layer prefill, bit for
    bit, and its first keys are the oracle's."""
    m = W.ModelShape("long_rows", 2, d_model, 2, 1, 128, 256, 1000, 1e4, 1e-5)
    eng, layers, dev = make_engine(a3mod, m, seed=d_model, w_std=0.05 * (512 / d_model) ** 0.5)
    n_ctx, nq = 61, 9
    n = n_ctx + nq
    g = torch.Generator(device=dev)
    g.manual_seed(d_model)
    ck, cv = (torch.randn(m.n_layers, n_ctx, m.n_kv_heads, m.head_dim, device=dev, generator=g).bfloat16() for _ in range(2))
    x0 = torch.randn(n, d_model, device=dev, generator=g).bfloat16()
    K, V = (torch.zeros(m.n_layers, n, m.n_kv_heads, m.head_dim, device=dev, dtype=torch.bfloat16) for _ in range(2))
    rq, out = eng.make_request(a3mod.chunk_table([ck], [cv], [0]), 1, n_ctx, n_ctx, nq, x0, K, V, ratio=1.0)
    eng.fuse_request(rq)
    x, Kp, Vp = x0.clone(), torch.zeros_like(K), torch.zeros_like(V)
    pos = torch.arange(n, dtype=torch.int32, device=dev)
    for layer in range(m.n_layers):
        eng.recompute_layer(layer, x, pos, Kp[layer], Vp[layer])
    assert eng.device_status() == 0
    assert torch.equal(K, Kp) and torch.equal(V, Vp) and torch.equal(out["x"], x)
    Ko, Vo, _ = O.full_prefill(f64(x0), oracle_weights(layers), oracle_model(m), rnd=O.round_bf16)
    check_kv(f64(K[0]), Ko[0], "first layer's K")
    check_kv(f64(V[0]), Vo[0], "first layer's V")
    eng.close()


@pytest.mark.parametrize("shape,kv_len,M", [(W.TINY_GQA, 768, 60), (W.TINY_GQA, 1023, 41), (W.TINY_GQA, 1024, 64), (W.TINY_GQA, 1153, 7),
                                            (W.TINY_GQA, 3000, 300), (W.TINY_G7, 1200, 55), (W.TINY, 700, 33), (W.TINY, 770, 128)])
def test_attention_keys_shared_by_a_cluster(a3mod, shape, kv_len, M):
    """Two and four CTAs per row tile (from six and eight key tiles on, head dimension 64 and 128): segments of equal and
    unequal length, a last segment that starts behind the cache (1 153 slots), early rows that see no key of the later
    segments.  Against the oracle, against one CTA per row tile, reproducibly; and invalid positions give finite rows."""
    m = shape
    eng, layers, dev = make_engine(a3mod, m, seed=M, w_std=0.05)
    model, weights = oracle_model(m), oracle_weights(layers)
    rng = np.random.default_rng(700 + M)
    pos = np.sort(rng.choice(kv_len, size=M, replace=False))
    pos[0], pos[-1] = 0, kv_len - 1
    X = W.bf16_round(rng.standard_normal((M, m.d_model), dtype=np.float32))
    Kc, Vc = W.make_cache_like(m, kv_len, M, 9, std=1.0)
    layer = m.n_layers - 1
    dpos = torch.from_numpy(pos.astype(np.int32)).to(dev)
    outs = []
    try:
        for split in (0, 0, 1):
            eng.set_option(a3mod.OPT_ATTN_SPLIT, split)
            dX, dK, dV = to_dev(X, dev), to_dev(Kc[layer], dev), to_dev(Vc[layer], dev)
            lse = torch.empty((M, m.n_q_heads), dtype=torch.float32, device=dev)
            eng.recompute_layer(layer, dX, dpos, dK, dV, lse_out=lse)
            assert eng.device_status() == 0
            outs.append((dX, lse))
    finally:
        eng.set_option(a3mod.OPT_ATTN_SPLIT, 0)
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    np.testing.assert_allclose(outs[0][1].cpu().numpy(), outs[2][1].cpu().numpy(), atol=1e-4)  # fp32 sums in another order
    Ko, Vo = Kc[layer].astype(np.float64), Vc[layer].astype(np.float64)
    _, parts = O.recompute_layer(X.astype(np.float64), pos, weights[layer], model, Ko, Vo, rnd=O.round_bf16, return_parts=True)
    check_kv(f64(outs[0][0]), parts["x_exact"], "hidden rows", scale=hidden_rows_scale(parts["x_exact"]))
    np.testing.assert_allclose(outs[0][1].cpu().numpy(), parts["lse"], atol=5e-3)
    bad = dpos.clone()
    bad[-1] = kv_len + 5
    bad[0] = -3
    dX = to_dev(X, dev)
    eng.recompute_layer(layer, dX, bad, to_dev(Kc[layer], dev), to_dev(Vc[layer], dev))
    assert eng.device_status() & a3mod.DEV_BAD_POSITION
    assert torch.isfinite(dX.float()).all()
    eng.close()


@pytest.mark.parametrize("n", [1023, 1024, 3071, 3072, 3073, 5119, 5121, 8192, 8193])
def test_topk_at_the_register_sizes(a3mod, n):
    """Candidate counts around those at which a thread holds one key more, with ties across the threshold and k = 1, n - 1."""
    eng, _, dev = make_engine(a3mod, W.TINY)
    s = (np.random.default_rng(n).integers(0, 37, size=n) / 32.0).astype(np.float32)
    for k in (1, n // 7, n - 1):
        got = eng.topk_select(torch.from_numpy(s).to(dev), 0, n, k).cpu().numpy()
        assert got.tolist() == O.topk_select(s.astype(np.float64), 0, n, k).tolist()
    assert eng.device_status() == 0
    eng.close()


@pytest.mark.parametrize("n,near", [(1, 1), (128, 128), (129, 129), (3000, 128), (3000, 129), (8192, 127)])
def test_topk_threshold_among_few_keys(a3mod, n, near):
    """`near` keys that agree in their first 16 bits, some of them equal, around the threshold: what is ranked in a list and what is not."""
    eng, _, dev = make_engine(a3mod, W.TINY)
    rng = np.random.default_rng(n + near)
    s = rng.uniform(2.0, 3.0, size=n).astype(np.float32) * rng.choice([1.0, 0.01], size=n).astype(np.float32)
    at = rng.permutation(n)[:near]
    s[at] = 1.0 + rng.integers(0, 2000, size=near).astype(np.float32) * 2.0 ** -23
    above = int((s >= 2.0).sum())
    for k in {max(above, 1), above + 1, above + near // 2, above + near}:
        if 0 < k <= n:
            got = eng.topk_select(torch.from_numpy(s).to(dev), 0, n, k).cpu().numpy()
            assert got.tolist() == O.topk_select(s.astype(np.float64), 0, n, k).tolist(), k
    assert eng.device_status() == 0
    eng.close()


@pytest.mark.parametrize("n_ctx,pool", [(900, 3), (3073, 7), (5120, 5), (8200, 7)])
def test_pooled_selection_of_the_eviction(a3mod, n_ctx, pool):
    """Pooling inside the selection, and (8 200 candidates) by the kernel of its own."""
    m = W.TINY_GQA
    eng, _, dev = make_engine(a3mod, m, seed=n_ctx)
    model, nq, n_system, capacity = oracle_model(m), 9, 5, 300
    rng = np.random.default_rng(n_ctx)
    K, V = (W.bf16_round(rng.standard_normal((n_ctx + nq, m.n_kv_heads, m.head_dim), dtype=np.float32)) for _ in range(2))
    q = W.bf16_round(rng.standard_normal((nq, m.n_q_heads, m.head_dim), dtype=np.float32))
    pos = np.arange(n_ctx, n_ctx + nq)
    dq, dK, dpos = to_dev(q, dev), to_dev(K, dev), torch.from_numpy(pos.astype(np.int32)).to(dev)
    s = np.einsum("jhd,ihd->jhi", q.astype(np.float64), np.repeat(K, m.n_q_heads // m.n_kv_heads, axis=1).astype(np.float64)) / np.sqrt(m.head_dim)
    s[np.broadcast_to(np.arange(n_ctx + nq)[None, None, :] > pos[:, None, None], s.shape)] = -np.inf
    lse = np.log(np.exp(s).sum(axis=2)).astype(np.float32)
    k_out, v_out, kept = eng.evict_layer(dq, dpos, torch.from_numpy(lse).to(dev), dK, to_dev(V, dev), n_system, n_ctx, capacity, pool)
    assert eng.device_status() == 0
    votes = O.pool_scores(O.eviction_scores(q, pos, K, model, n_system, n_ctx), n_system, n_ctx, pool)
    k = capacity - n_system - nq
    for g in range(m.n_kv_heads):
        idx = kept[g].cpu().numpy()
        assert idx[:n_system].tolist() == list(range(n_system)) and idx[-nq:].tolist() == list(range(n_ctx, n_ctx + nq))
        sel = idx[n_system:n_system + k]
        assert (np.diff(sel) > 0).all()
        v = votes[g][n_system:n_ctx]
        thr = np.sort(v)[-k]
        inside = np.isin(np.arange(n_system, n_ctx), sel)
        # votes are sums of fp32 exponentials: 1e-3 relative, as for the scores
        assert (v[inside] >= thr * (1 - 2e-3)).all() and (v[~inside] <= thr * (1 + 2e-3)).all()
        assert torch.equal(k_out[:, g], dK[kept[g].long(), g])
    eng.close()


@pytest.mark.parametrize("shape,n_ctx,nq", [(W.TINY_GQA, 300, 1), (W.TINY_GQA, 511, 40), (W.TINY_GQA, 100, 300), (W.TINY_G7, 7, 5),
                                            (W.TINY_G7, 250, 33)])
def test_late_queries_ride_along(a3mod, shape, n_ctx, nq):
    """Selection layer: the question rows' queries in the launch of everybody's keys and values (one or more token tiles of
    them, an odd number of heads) against launches of their own on the tile kernel: the same bits."""
    m, dev, n = shape, torch.device("cuda:0"), n_ctx + nq
    eng = a3mod.A3(m, W.make_weights_device(m, dev, 0), n + 8)
    g = torch.Generator(device=dev)
    g.manual_seed(n)
    ck, cv = (torch.randn(m.n_layers, n_ctx, m.n_kv_heads, m.head_dim, device=dev, generator=g).bfloat16() for _ in range(2))
    x0 = torch.randn(n, m.d_model, device=dev, generator=g).bfloat16()
    tab = a3mod.chunk_table([ck], [cv], [0])
    res = []
    for qkv_t in (1, 0):
        eng.set_option(a3mod.OPT_QKV_T, qkv_t)
        K, V = (torch.zeros(m.n_layers, n, m.n_kv_heads, m.head_dim, device=dev, dtype=torch.bfloat16) for _ in range(2))
        rq, out = eng.make_request(tab, 1, n_ctx, n_ctx, nq, x0, K, V, ratio=0.0, select_layer=0)
        eng.fuse_request(rq)
        assert eng.device_status() == 0
        res.append((K[0, :n_ctx], V[0, :n_ctx], out["scores"][:n_ctx]))
    eng.set_option(a3mod.OPT_QKV_T, 1)
    for a, b in zip(*res):
        assert torch.equal(a, b)
    assert float(res[0][2].abs().max()) > 0
    eng.close()


HEADS_32_8 = W.ModelShape("heads_32_8", 1, 128, 32, 8, 128, 128, 1000, 5e5, 1e-5)
HEADS_28_4 = W.ModelShape("heads_28_4", 1, 128, 28, 4, 128, 128, 1000, 1e6, 1e-6)
HEADS_4_2 = W.ModelShape("heads_4_2", 1, 128, 4, 2, 128, 128, 1000, 5e5, 1e-5)


@pytest.mark.parametrize("m,n_ctx,nq,launches", [(HEADS_32_8, 805, 8, 3), (HEADS_32_8, 805, 9, 3), (HEADS_32_8, 805, 17, 4), (HEADS_32_8, 1200, 9, 4),
                                                 (HEADS_32_8, 5120, 32, 4), (HEADS_32_8, 18930, 8, 3), (HEADS_32_8, 18960, 8, 3), (HEADS_32_8, 32768, 32, 4),
                                                 (HEADS_28_4, 17871, 9, 3), (HEADS_28_4, 17871, 64, 4), (HEADS_28_4, 19000, 9, 4),
                                                 (HEADS_4_2, 356, 13, 3), (HEADS_4_2, 18800, 64, 3), (HEADS_4_2, 19000, 64, 4)])
def test_statistics_merged_where_that_is_shorter(a3mod, m, n_ctx, nq, launches):
    """Position check, statistics and scores, and a merge between the last two unless the score kernel merges the segments in one
    round (or a second one over few segments): the same scores as the warp-level kernel's, which always has them merged before."""
    eng, n = a3mod.A3(m, W.make_weights_device(m, torch.device("cuda:0"), 0), n_ctx + nq), n_ctx + nq
    g = torch.Generator(device=eng.device)
    g.manual_seed(n)
    q = torch.randn(nq, m.n_q_heads, m.head_dim, device=eng.device, generator=g).bfloat16()
    k = torch.randn(n, m.n_kv_heads, m.head_dim, device=eng.device, generator=g).bfloat16()
    pos = torch.arange(n_ctx, n, dtype=torch.int32, device=eng.device)
    a3mod.launch_count(reset=True)
    scores = eng.query_scores(q, pos, k, 3, n_ctx)
    assert a3mod.launch_count() == launches
    eng.set_option(a3mod.OPT_SCORES_KERNEL, 2)
    other = eng.query_scores(q, pos, k, 3, n_ctx)
    assert eng.device_status() == 0
    # A logit (up to 2^6 before its scale of 2^-3.5) is summed in fp32 in eight steps, each off by at most 2^-23 of it: 5.4e-6 in the
    # exponent; ex2.approx 2^-22, the log-sum-exp no more.  Both kernels: below 2e-5, and the sums add terms of one sign.
    assert torch.allclose(scores, other, rtol=2e-5, atol=0)
    assert float(scores[3:n_ctx].min()) > 0 and float(scores[:3].abs().max()) == 0 == float(scores[n_ctx:].abs().max())
    eng.close()
