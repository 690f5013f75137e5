"""The paths that only launches of few rows take: GEMMs whose k-loop is cut into slices, added up by the kernel that follows,
and attention whose keys are shared out to a cluster of CTAs.

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
