"""evict_layer's outputs do not take after the positions: with no question rows nothing reads those, so any tensor may stand
there.  The library call itself is replaced; nothing here needs a GPU."""
import pytest
import torch

from paper_2511_17560_b200 import a3
from paper_2511_17560_b200 import workloads as W


class Recorder:
    def __init__(self, lib):
        self._lib, self.calls = lib, []

    def __getattr__(self, name):
        return getattr(self._lib, name)

    def a3_evict_workspace_bytes(self, h, kv_len):
        return 64

    def a3_evict_layer(self, *args):
        self.calls.append(args)
        return 0


@pytest.mark.parametrize("q_pos", [torch.empty(0, dtype=torch.int32), torch.empty(0, dtype=torch.int64), torch.empty(0)])
def test_outputs_are_the_caches_whatever_the_positions(monkeypatch, q_pos):
    m = W.TINY_GQA
    lib = Recorder(a3._load())
    monkeypatch.setattr(a3, "_load", lambda: lib)
    monkeypatch.setattr(a3, "_stream", lambda: 0)
    eng = a3.A3.__new__(a3.A3)
    eng.shape, eng._h, eng._ws, eng.device = m, None, None, torch.device("cpu")
    cache = torch.empty((50, m.n_kv_heads, m.head_dim), dtype=torch.bfloat16, device="meta")  # another device than the positions'
    k, v, kept = eng.evict_layer(None, q_pos, None, cache, cache, 5, 50, 20)
    assert len(lib.calls) == 1
    assert kept.dtype == torch.int32 and kept.device == cache.device and kept.shape == (m.n_kv_heads, 20)
    for t in (k, v):
        assert t.dtype == torch.bfloat16 and t.device == cache.device and t.shape == (20, m.n_kv_heads, m.head_dim)
