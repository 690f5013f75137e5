"""The host-buffer entry copies chunk caches several layers at a time: the device entry's result, bit for bit, wherever the
groups end."""
from dataclasses import replace

import pytest
import torch

from paper_2511_17560_b200 import workloads as W
from tests.test_gpu_steps import a3mod  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_layers,select_layer,lens", [(2, 1, (40, 30)), (3, 0, (1, 64)), (4, 1, (33, 70, 5)), (9, 1, (48, 16)),
                                                        (14, 2, (20, 31, 12)), (12, 1, ())])
def test_groups_of_layers_match_the_device_entry(a3mod, n_layers, select_layer, lens):
    compare_entries(a3mod, replace(W.TINY_GQA, n_layers=n_layers), select_layer, lens)


# 2 KB of keys a token: slices of 4.1 MB, 2.1, 1.4, 1.0 and 0.7 are copied one, one, three, four and five layers at a time
@pytest.mark.parametrize("n_layers,lens", [(5, (2007,)), (6, (1025, 1030)), (9, (650, 700)), (13, (512, 512)), (12, (400, 300))])
def test_large_slices_are_copied_in_smaller_groups(a3mod, n_layers, lens):
    compare_entries(a3mod, W.ModelShape("broad_cache", n_layers, 128, 8, 8, 128, 128, 1000, 1e4, 1e-5), 1, lens)


def compare_entries(a3mod, m, select_layer, lens):
    dev, n_layers, n_ctx, nq = torch.device("cuda:0"), m.n_layers, sum(lens), 9
    n = n_ctx + nq
    eng = a3mod.A3(m, W.make_weights_device(m, dev, 0), n + 8)
    g = torch.Generator(device=dev)
    g.manual_seed(n_layers)
    cache = lambda t: torch.randn(n_layers, t, m.n_kv_heads, m.head_dim, device=dev, generator=g).bfloat16()  # noqa: E731
    ck, cv = [cache(t) for t in lens], [cache(t) for t in lens]
    x0 = torch.randn(n, m.d_model, device=dev, generator=g).bfloat16()
    offsets = [sum(lens[:i]) for i in range(len(lens))]
    tab = a3mod.chunk_table(ck, cv, offsets)
    res = []
    for host in (False, True):
        K = torch.zeros(n_layers, n, m.n_kv_heads, m.head_dim, device=dev, dtype=torch.bfloat16)
        V = torch.zeros_like(K)
        rq, out = eng.make_request(None if host else tab, len(lens), 0 if host else max(lens, default=0), n_ctx, nq, None if host else x0, K, V,
                                   ratio=0.3, select_layer=select_layer)
        if host:
            rows = torch.empty(out["p"] + nq, dtype=torch.int32).pin_memory()
            x = torch.empty((out["p"] + nq, m.d_model), dtype=torch.bfloat16).pin_memory()
            staging = torch.empty(eng.host_staging_bytes(n_ctx, n), dtype=torch.uint8, device=dev)
            eng.fuse_request_host(rq, [t.cpu().pin_memory() for t in ck], [t.cpu().pin_memory() for t in cv], x0.cpu().pin_memory(), rows, x, staging)
            res.append((K, V, rows, x))
        else:
            eng.fuse_request(rq)
            res.append((K, V, out["rows"].cpu(), out["x"].cpu()))
        assert eng.device_status() == 0
    for a, b in zip(*res):
        assert torch.equal(a, b)
    eng.close()
