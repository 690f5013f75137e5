"""The work that users of the library have it do, as measurable cases.

Kinds of case (`case["kind"]`), all through the public binding `paper_2511_17560_b200.a3`:

  fuse        one request up to its first token: `fuse_request` (or the replay of a captured `graph`) and `first_token`
  batch       several requests on one stream (`fuse_batch`), as a server with a queue issues them
  host        `fuse_request_host`: chunk caches and embeddings in pinned host memory, results back in host memory
  precompute  `precompute_chunk`: one document prefilled alone, which fills the store the other kinds read from
  evict       `evict_layer`: the compaction of one layer's fused cache to a fixed capacity

Chunk lengths are a text: "512x64", or "100,37,128"; the requests of a batch are separated by ";".  Weights are
N(0, 0.02^2) with the two matrices that write to the residual stream scaled by 1/sqrt(2 layers), embeddings have unit
RMS, and chunk caches have the spread that such weights give normalised rows.  Relevance is planted: the question and
exactly as many context tokens as the request recomputes, in spans of 16 spread over the chunks, share a direction of
the hidden space that the selection layer's query and key projections map onto their slowest rotation pairs.  Relevant
tokens then stand clear of the others, as they do in trained models, and every correct implementation selects the same.
"""
import math
from dataclasses import replace

import numpy as np
import torch

from paper_2511_17560_b200 import a3
from paper_2511_17560_b200 import workloads as W

MODELS = {"llama8b": W.LLAMA8B, "qwen7b": W.QWEN7B, "tiny_gqa": W.TINY_GQA, "tiny_g7": W.TINY_G7}
SELECT_LAYER = 1
COSINE = 0.5   # of a relevant row with the shared direction
SPAN = 16      # tokens of one relevant passage
LOGIT = 8.0    # what relevance adds to a question-context logit at the selection layer


def listed():
    fuse = dict(kind="fuse", ratio=0.15, n_system=0, cached_keys=False, graph=False)
    return [
        # a handful of short passages on a small model: launches and host work are all there is
        dict(fuse, name="tiny_passages", model="tiny_gqa", lens="100,37,128,1,90", nq=13),
        # one or a few retrieved paragraphs behind a short system prompt: the weights are read for a hundred rows
        dict(fuse, name="llama_3_passages", model="llama8b", lens="61,256,301,187", nq=21, n_system=61),
        # the common retrieval request: ten chunks of 512, replayed from a graph as a server with fixed shapes does
        dict(fuse, name="llama_10x512_graph", model="llama8b", lens="512x10", nq=32, graph=True),
        # a middling request whose scores are taken against the stored keys, the cheaper of the two readings
        dict(fuse, name="qwen_6_cached_keys", model="qwen7b", lens="333,512,47,700,256,419", nq=40, ratio=0.1, cached_keys=True),
        # long documents of uneven length
        dict(fuse, name="qwen_16_ragged", model="qwen7b",
             lens="1837,412,1290,705,988,1513,300,2048,1101,871,633,1999,257,1340,790,1787", nq=64),
        # the longest context
        dict(fuse, name="llama_64x512", model="llama8b", lens="512x64", nq=32),
        # a server's queue: requests of different sizes over stored chunks of 256 to 1024 tokens
        dict(kind="batch", name="llama_batch_4", model="llama8b", ratio=0.15, nq=33,
             lens="300,911,256,640,1024,433,777,512;260,350,333,420;512,1000,700,813,299,640,581,903,450,377,610,280;600,256,444,381,290"),
        # chunk store in host memory
        dict(kind="host", name="llama_host_10x512", model="llama8b", ratio=0.15, lens="512x10", nq=32),
        # filling the store: the usual chunk, a short note, a long document
        dict(kind="precompute", name="llama_chunk_512", model="llama8b", tokens=512),
        dict(kind="precompute", name="qwen_note_75", model="qwen7b", tokens=75),
        dict(kind="precompute", name="qwen_document_1931", model="qwen7b", tokens=1931),
        # one layer's cache cut to 1024 entries per head, votes pooled over 7 neighbours
        dict(kind="evict", name="llama_evict_1024", model="llama8b", n_ctx=5120, nq=32, n_system=0, capacity=1024, pool=7),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _drawn_lens(rng, most_chunks, lo, hi):
    mean = _log_uniform(rng, lo, hi)
    return ",".join(str(rng.randint(mean // 2, mean + mean // 2)) for _ in range(_log_uniform(rng, 1, most_chunks)))


def draw(rng):
    largest = work(next(c for c in listed() if c["name"] == "llama_64x512"))
    while True:
        kind = rng.choices(("fuse", "batch", "host", "precompute", "evict"), (6, 1, 1, 3, 1))[0]
        model = rng.choices(("llama8b", "qwen7b", "tiny_gqa", "tiny_g7"), (5, 4, 1, 1) if kind == "fuse" else (1, 1, 0, 0))[0]
        case = dict(kind=kind, model=model)
        if kind == "fuse":
            case.update(lens=_drawn_lens(rng, 64, 32, 1024), nq=_log_uniform(rng, 4, 96), ratio=round(rng.uniform(0.04, 0.3), 3),
                        n_system=0, cached_keys=rng.random() < 0.2, graph=rng.random() < 0.3)
            lens = _lens(case["lens"])
            if len(lens) > 2 and rng.random() < 0.25:
                case["n_system"] = lens[0]
        elif kind == "batch":
            case.update(lens=";".join(_drawn_lens(rng, 16, 128, 768) for _ in range(rng.randint(2, 6))), nq=_log_uniform(rng, 8, 64),
                        ratio=round(rng.uniform(0.05, 0.25), 3))
        elif kind == "host":
            case.update(lens=_drawn_lens(rng, 16, 128, 768), nq=_log_uniform(rng, 8, 64), ratio=round(rng.uniform(0.05, 0.25), 3))
            if sum(_lens(case["lens"])) > 6144:  # pinned memory is slow to get
                continue
        elif kind == "precompute":
            case.update(tokens=_log_uniform(rng, 24, 2048))
        else:
            n_ctx = _log_uniform(rng, 1500, 32768)
            case.update(n_ctx=n_ctx, nq=_log_uniform(rng, 8, 64), n_system=rng.choice((0, 100)), capacity=_log_uniform(rng, 256, n_ctx // 2),
                        pool=rng.choice((1, 5, 7)))
        w = work(case)
        if w["flops"] <= largest["flops"] and w["bytes"] <= largest["bytes"]:
            return case


# ------------------------------------------------------------------ inputs


def _lens(text):
    out = []
    for item in text.split(","):
        t, _, times = item.partition("x")
        out += [int(t)] * int(times or 1)
    return out


def _count(case, lens):
    n_ctx, n_system = sum(lens), case.get("n_system", 0)
    return int(math.floor(case["ratio"] * (n_ctx + case["nq"]) + 1e-9)), n_ctx, n_system


def _slow_dims(m):
    """The first halves of the slowest eighth of a head's rotation pairs (pairs (i, i + D/2))."""
    half = m.head_dim // 2
    return slice(half - half // 8, half)


class _Inputs:
    def __init__(self, case, seed):
        self.dev = torch.device("cuda")
        self.m = MODELS[case["model"]]
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(seed * 977 + 13)
        u = self.normal((self.m.d_model,))
        self.u = u / u.norm()

    def normal(self, shape, std=1.0, dtype=torch.float32):
        return torch.randn(shape, generator=self.g, device=self.dev, dtype=dtype) * std

    def weights(self, seed):
        m = self.m
        layers = W.make_weights_device(m, self.dev, seed)
        for w in layers:
            w["wo"] *= (2 * m.n_layers) ** -0.5
            w["w_down"] *= (2 * m.n_layers) ** -0.5
            for name in ("attn_norm", "mlp_norm"):
                w[name] = (1 + self.normal((m.d_model,), 0.1)).to(torch.bfloat16)
        # the shared direction of the hidden space onto the slow dimensions of every head of the selection layer
        dims = _slow_dims(m)
        direction = torch.zeros(m.head_dim, device=self.dev)
        direction[dims] = (dims.stop - dims.start) ** -0.5
        self.slow = direction
        gain = math.sqrt(LOGIT * math.sqrt(m.head_dim)) / (COSINE * math.sqrt(m.d_model))
        for name, heads in (("wq", m.n_q_heads), ("wk", m.n_kv_heads)):
            layers[SELECT_LAYER][name] += (gain * torch.outer(direction.repeat(heads), self.u)).to(torch.bfloat16)
        return layers

    def embeddings(self, n, relevant):
        e = self.normal((n, self.m.d_model))
        e[relevant] = COSINE * math.sqrt(self.m.d_model) * self.u + math.sqrt(1 - COSINE ** 2) * e[relevant]
        return e.to(torch.bfloat16)

    def relevant(self, first, end, p):
        """p slots of [first, end): whole spans in a random order, then what is left of the next one."""
        slots = torch.arange(first, end, device=self.dev)
        order = torch.randperm((end - first + SPAN - 1) // SPAN, generator=self.g, device=self.dev)
        key = order[(slots - first) // SPAN] * SPAN + (slots - first) % SPAN
        return slots[torch.argsort(key)[:p]]

    def chunk(self, t, offset, relevant):
        """A stored chunk [L][T][Hkv][D]: keys and values, the relevant tokens' keys marked at the selection layer."""
        m = self.m
        shape, std = (m.n_layers, t, m.n_kv_heads, m.head_dim), 0.02 * math.sqrt(m.d_model)
        k, v = self.normal(shape, std, torch.bfloat16), self.normal(shape, std, torch.bfloat16)
        rows = relevant[(relevant >= offset) & (relevant < offset + t)] - offset
        k[SELECT_LAYER, rows] += (self.slow * math.sqrt(LOGIT * math.sqrt(m.head_dim))).to(torch.bfloat16)
        return k, v

    def request(self, case, lens):
        """Chunks, embeddings and empty fused caches of one request."""
        m = self.m
        p, n_ctx, n_system = _count(case, lens)
        n = n_ctx + case["nq"]
        p = min(p, n_ctx - n_system)
        rel = self.relevant(n_system, n_ctx, p)
        x0 = self.embeddings(n, torch.cat([rel, torch.arange(n_ctx, n, device=self.dev)]))
        offsets = [int(o) for o in np.cumsum([0] + lens[:-1])]
        chunks = [self.chunk(t, o, rel) for t, o in zip(lens, offsets)]
        k = torch.zeros((m.n_layers, n, m.n_kv_heads, m.head_dim), dtype=torch.bfloat16, device=self.dev)
        return dict(x0=x0, offsets=offsets, ck=[c[0] for c in chunks], cv=[c[1] for c in chunks], k=k, v=torch.zeros_like(k), n_ctx=n_ctx)

    def vocabulary(self):
        """Final norm and output head; one token answers to the shared direction, so that the greedy choice is clear."""
        m = self.m
        head = self.normal((m.vocab, m.d_model), 0.02, torch.bfloat16)
        token = int(torch.randint(m.vocab, (1,), generator=self.g, device=self.dev))
        head[token] += (20.0 / (COSINE * math.sqrt(m.d_model)) * self.u).to(torch.bfloat16)
        return torch.ones(m.d_model, dtype=torch.bfloat16, device=self.dev), head


def prepare(case, seed):
    return {"fuse": _prepare_fuse, "batch": _prepare_batch, "host": _prepare_host, "precompute": _prepare_precompute,
            "evict": _prepare_evict}[case["kind"]](case, seed)


def run(state):
    return state["run"](state)


# ------------------------------------------------------------------ one request and its first token


def _prepare_fuse(case, seed):
    i = _Inputs(case, seed)
    lens = _lens(case["lens"])
    eng = a3.A3(i.m, i.weights(seed), sum(lens) + case["nq"])
    r = i.request(case, lens)
    norm, head = i.vocabulary()
    chunks = a3.chunk_table(r["ck"], r["cv"], r["offsets"])
    req, out = eng.make_request(chunks, len(lens), max(lens), r["n_ctx"], case["nq"], r["x0"], r["k"], r["v"], ratio=case["ratio"],
                                select_layer=SELECT_LAYER, n_system=case["n_system"], score_source=int(case["cached_keys"]))
    state = dict(run=_run_fuse, eng=eng, req=req, out=out, r=r, norm=norm, head=head, graph=None)
    if case["graph"]:
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            state["graph"] = eng.graph_capture(req)
        torch.cuda.current_stream().wait_stream(stream)
    return state


def _run_fuse(s):
    if s["graph"] is not None:
        s["graph"].launch()
    else:
        s["eng"].fuse_request(s["req"])
    logits, token = s["eng"].first_token(s["out"]["x"][-1], s["norm"], s["head"])
    return dict(k=s["r"]["k"], v=s["r"]["v"], rows=s["out"]["rows"], scores=s["out"]["scores"], x=s["out"]["x"], logits=logits, token=token)


# ------------------------------------------------------------------ several requests


def _prepare_batch(case, seed):
    i = _Inputs(case, seed)
    all_lens = [_lens(t) for t in case["lens"].split(";")]
    eng = a3.A3(i.m, i.weights(seed), max(sum(lens) for lens in all_lens) + case["nq"])
    reqs, outs = [], []
    for lens in all_lens:
        r = i.request(case, lens)
        chunks = a3.chunk_table(r["ck"], r["cv"], r["offsets"])
        req, out = eng.make_request(chunks, len(lens), max(lens), r["n_ctx"], case["nq"], r["x0"], r["k"], r["v"], ratio=case["ratio"],
                                    select_layer=SELECT_LAYER)
        out.update(r=r)
        reqs.append(req)
        outs.append(out)
    return dict(run=_run_batch, eng=eng, reqs=reqs, outs=outs)


def _run_batch(s):
    s["eng"].fuse_batch(s["reqs"])
    return [dict(k=o["r"]["k"], v=o["r"]["v"], rows=o["rows"], scores=o["scores"], x=o["x"]) for o in s["outs"]]


# ------------------------------------------------------------------ chunk store in host memory


def _prepare_host(case, seed):
    i = _Inputs(case, seed)
    lens = _lens(case["lens"])
    eng = a3.A3(i.m, i.weights(seed), sum(lens) + case["nq"])
    r = i.request(case, lens)
    n = r["n_ctx"] + case["nq"]

    def pinned(tensors):
        flat = torch.empty(sum(t.numel() for t in tensors), dtype=torch.bfloat16, pin_memory=True)
        views, at = [], 0
        for t in tensors:
            views.append(flat[at:at + t.numel()].view(t.shape))
            views[-1].copy_(t)
            at += t.numel()
        return views

    host = pinned(r.pop("ck") + r.pop("cv") + [r["x0"]])
    req, out = eng.make_request(None, len(lens), max(lens), r["n_ctx"], case["nq"], r["x0"], r["k"], r["v"], ratio=case["ratio"],
                                select_layer=SELECT_LAYER)
    rows = torch.empty(out["rows"].shape, dtype=torch.int32, pin_memory=True)
    x = torch.empty(out["x"].shape, dtype=torch.bfloat16, pin_memory=True)
    staging = torch.empty(eng.host_staging_bytes(r["n_ctx"], n), dtype=torch.uint8, device=i.dev)
    return dict(run=_run_host, eng=eng, req=req, out=out, r=r, ck=host[:len(lens)], cv=host[len(lens):-1], x0=host[-1], rows=rows, x=x,
                staging=staging)


def _run_host(s):
    s["eng"].fuse_request_host(s["req"], s["ck"], s["cv"], s["x0"], s["rows"], s["x"], s["staging"])
    return dict(k=s["r"]["k"], v=s["r"]["v"], scores=s["out"]["scores"], rows=s["rows"], x=s["x"])


# ------------------------------------------------------------------ one document alone


def _prepare_precompute(case, seed):
    i = _Inputs(case, seed)
    m, t = i.m, case["tokens"]
    eng = a3.A3(m, i.weights(seed), t)
    k = torch.zeros((m.n_layers, t, m.n_kv_heads, m.head_dim), dtype=torch.bfloat16, device=i.dev)
    x0 = i.embeddings(t, torch.arange(0, device=i.dev))
    return dict(run=_run_precompute, eng=eng, x0=x0, x=torch.empty_like(x0), k=k, v=torch.zeros_like(k))


def _run_precompute(s):
    s["x"].copy_(s["x0"])  # the call works in place; the embeddings are looked up anew for every document
    s["eng"].precompute_chunk(s["x"], s["k"], s["v"])
    return dict(x=s["x"], k=s["k"], v=s["v"])


# ------------------------------------------------------------------ one layer's eviction


def _prepare_evict(case, seed):
    i = _Inputs(case, seed)
    m, nq, n_ctx, n_system, pool = i.m, case["nq"], case["n_ctx"], case["n_system"], case["pool"]
    n, std, group = n_ctx + nq, 0.02 * math.sqrt(m.d_model), m.n_q_heads // m.n_kv_heads
    layer = W.make_weights_device(replace(m, n_layers=1), i.dev, seed)
    eng = a3.A3(replace(m, n_layers=1), layer, n)
    slow = torch.zeros(m.head_dim, device=i.dev)
    slow[_slow_dims(m)] = (m.head_dim // 16) ** -0.5
    mark = slow * math.sqrt(LOGIT * math.sqrt(m.head_dim))
    q = (i.normal((nq, m.n_q_heads, m.head_dim), std) + mark).to(torch.bfloat16)
    k = i.normal((n, m.n_kv_heads, m.head_dim), std)
    # Each head keeps its own slots: the middles of enough pooling windows, the last of them marked less, so that the
    # capacity ends inside a window of equal votes (lower slots first) and not between two that are nearly alike.
    keep = max(0, min(case["capacity"] - n_system - nq, n_ctx - n_system))
    whole, part = divmod(keep, pool)
    for head in range(m.n_kv_heads):
        windows = torch.randperm((n_ctx - n_system) // pool, generator=i.g, device=i.dev)
        at = n_system + windows * pool + pool // 2
        k[at[:whole], head] += 1.3 * mark
        if part:
            k[at[whole:whole + 1], head] += 0.65 * mark
    k = k.to(torch.bfloat16)
    v = i.normal(k.shape, std, torch.bfloat16)
    pos = torch.arange(n_ctx, n, dtype=torch.int32, device=i.dev)
    lse = torch.empty((nq, m.n_q_heads), dtype=torch.float32, device=i.dev)
    hidden = torch.arange(n, device=i.dev)[None, :] > pos[:, None]
    for h in range(m.n_q_heads):
        s = q[:, h].float() @ k[:, h // group].float().T / math.sqrt(m.head_dim)
        lse[:, h] = torch.logsumexp(s.masked_fill(hidden, -math.inf), dim=1)
    return dict(run=_run_evict, eng=eng, q=q, pos=pos, lse=lse, k=k, v=v, args=(n_system, n_ctx, case["capacity"], pool))


def _run_evict(s):
    k, v, kept = s["eng"].evict_layer(s["q"], s["pos"], s["lse"], s["k"], s["v"], *s["args"])
    return dict(k=k, v=v, kept=kept)


# ------------------------------------------------------------------ what a pass cannot do without


def _layer_params(m):
    return m.d_model * ((2 * m.n_q_heads + 2 * m.n_kv_heads) * m.head_dim + 3 * m.d_ff)


def _request_work(case, lens):
    m = MODELS[case["model"]]
    p, n_ctx, n_system = _count(case, lens)
    nq, L, d, kvd, qd = case["nq"], m.n_layers, m.d_model, m.n_kv_heads * m.head_dim, m.n_q_heads * m.head_dim
    n, rows = n_ctx + nq, min(p, n_ctx - n_system) + nq
    sparse_keys = (rows - nq) * (n_ctx + n_system + 1) / 2 + nq * (n_ctx + (nq + 1) / 2)  # relevant tokens lie anywhere
    question_keys = nq * (n_ctx + (nq + 1) / 2)
    if case.get("cached_keys"):
        flops = 2.0 * _layer_params(m) * (rows * L + nq * SELECT_LAYER) + 2.0 * nq * d * (qd + 2 * kvd)
        flops += 4.0 * qd * (L * sparse_keys + SELECT_LAYER * question_keys)
        stored = L
    else:
        flops = 2.0 * _layer_params(m) * (rows * (L - SELECT_LAYER) + n * SELECT_LAYER) + 2.0 * d * (2 * kvd * n + qd * nq)
        flops += 4.0 * qd * ((L - SELECT_LAYER) * sparse_keys + SELECT_LAYER * n * (n + 1) / 2)
        stored = L - SELECT_LAYER - 1
    flops += 4.0 * qd * question_keys  # row statistics and scores
    byts = 4.0 * kvd * (stored * n_ctx + L * n) + 2.0 * d * (n + rows) + 4.0 * (n + rows)
    return byts, flops


def work(case):
    m = MODELS[case["model"]]
    d, kvd, qd = m.d_model, m.n_kv_heads * m.head_dim, m.n_q_heads * m.head_dim
    weights = 2.0 * m.n_layers * _layer_params(m)
    if case["kind"] == "precompute":
        t = case["tokens"]
        return {"bytes": weights + 4.0 * d * t + 4.0 * kvd * m.n_layers * t,
                "flops": m.n_layers * (2.0 * _layer_params(m) * t + 4.0 * qd * t * (t + 1) / 2)}
    if case["kind"] == "evict":
        n, nq = case["n_ctx"] + case["nq"], case["nq"]
        kept = case["n_system"] + nq + max(0, min(case["capacity"] - case["n_system"] - nq, case["n_ctx"] - case["n_system"]))
        return {"bytes": 2.0 * kvd * (n + 3 * kept) + 4.0 * kept * m.n_kv_heads + 2.0 * nq * qd, "flops": 2.0 * nq * qd * n}
    requests = [_request_work(case, _lens(t)) for t in case["lens"].split(";")]
    byts, flops = weights + sum(r[0] for r in requests), sum(r[1] for r in requests)
    if case["kind"] == "fuse":
        byts += 2.0 * m.vocab * d + 4.0 * m.vocab
        flops += 2.0 * m.vocab * d
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    if case["kind"] == "evict":
        return "exact"  # the kept rows are copies, and which are kept is planted
    # against the same stack in torch operators: 0.021 in the hidden rows after 32 layers of bf16 residuals, 0.12 in one value;
    # with the sums of the attention in another order 0.019 and 0.11
    return {"rel": 0.03, "max": 0.45, "differ": 0.0}
