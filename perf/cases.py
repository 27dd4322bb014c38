"""The work users of this library have it do: what is timed, on which inputs, and how exact its results have to be.

A pass goes through the public calls of the ctypes binding, which are those of include/lsa.h:

  prefill        cache upkeep for the queries' own keys (lsa_block_means), then one layer group (lsa_layer_group): indexer
                 once, sparse attention for each of the group's layers
  prefill_host   the same group with its per-query tensors in pinned host memory (lsa_layer_group_host)
  decode         one layer group for a batch of sequences with paged caches, one new query each
  decode_append  lsa_append of every sequence's new token (indexer key, mean key, latent rows), then that layer group

Shapes, distributions and parameters are those of configs.py, of the sweeps and of the parity tests.
"""
from __future__ import annotations

import math

import torch

from paper_2608_01662_b200 import binding, inputs
from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload, PrefillWorkload

# The parameter sets in use (page, sub-block, kept pages, sink, window, heads, dims, key type): configs.py.
_MLA_PREFILL = ("cfg2", "cfg3", "cfg5")
_MAX_TOKENS = 4_700_000        # paged caches of a decode batch, all sequences together (64 x 16K-128K)


def _prefill(name, base, n_query, n_key, layers, flat=False, keep_pages=0, host_pass=0):
    return {"name": name, "kind": "prefill_host" if host_pass else "prefill", "base": base, "n_query": n_query, "n_key": n_key,
            "layers": layers, "flat": flat, "keep_pages": keep_pages or CONFIGS[base].M, "host_pass": host_pass}


def _decode(name, batch, ctx_lo, ctx_hi, layers, keys="e4m3", flat=False, append=False):
    return {"name": name, "kind": "decode_append" if append else "decode", "base": "cfg4", "batch": batch, "ctx_lo": ctx_lo,
            "ctx_hi": ctx_hi, "layers": layers, "keys": keys, "flat": flat}


def listed():
    return [
        # a short whole prompt on the small 8-head indexer and 16-head attention: launches and latency
        _prefill("prompt_2k_small_heads", "cfg1", 2048, 2048, 1),
        # a short whole prompt of odd length on the MLA shapes: ragged tiles, most queries see less than their budget
        _prefill("prompt_1k_ragged", "cfg3", 1237, 1237, 4),
        # a whole 32K prompt, bf16 indexer keys, two layers per group
        _prefill("prompt_32k_bf16", "cfg2", 32768, 32768, 2),
        # the last chunk of a 128K prompt prefilled in chunks, e4m3 keys, four layers per group
        _prefill("chunk_16k_of_128k", "cfg3", 16384, 131072, 4),
        # a chunk at the end of a million cached tokens: coarse scoring of the whole cache
        _prefill("chunk_4k_of_1m", "cfg5", 4096, 1048576, 4),
        # 2048 queries with the large recall budget (1024 pages of 128) the method was published with
        _prefill("chunk_2k_recall_128k", "cfg3", 2048, 262144, 4, keep_pages=1024),
        # 1000 queries on the flat indexer (every cached token scored)
        _prefill("chunk_1k_flat_64k", "cfg3", 1000, 65536, 4, flat=True),
        # the group fed from pinned host buffers in passes, as a caller without device-resident activations runs it
        _prefill("host_2k_of_32k", "cfg3", 2048, 32768, 4, host_pass=512),
        # one user's decode step at a moderate context: latency of every kernel in the chain
        _decode("decode_1_seq", 1, 20_000, 24_000, 4),
        # a serving batch, contexts between 16K and 128K
        _decode("decode_64_seq", 64, 16384, 131072, 4),
        # a decode step of a growing batch: append, then the group; odd batch, short and long contexts, bf16 keys
        _decode("decode_append_23_seq", 23, 900, 40_000, 3, keys="bf16", append=True),
        # a serving batch on the flat indexer
        _decode("decode_flat_16_seq", 16, 16384, 131072, 4, flat=True),
    ]


def draw(rng):
    """One more case: the kinds in the proportions of the list above, sizes over their whole ranges (mostly odd)."""

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("prefill", "prefill", "prefill", "small", "recall", "flat", "host", "decode", "decode", "append", "decode_flat"))
    layers = rng.randint(1, 4)
    if kind == "small":
        n_key = log_int(300, 16384)
        case = _prefill("", "cfg1", rng.choice((n_key, log_int(64, n_key))), n_key, layers)
    elif kind == "prefill":
        n_query = log_int(200, 8192)
        case = _prefill("", rng.choice(_MLA_PREFILL), n_query, max(n_query, log_int(1000, 1_048_576)), layers)
    elif kind == "recall":
        case = _prefill("", "cfg3", log_int(100, 2048), log_int(16384, 524_288), layers, keep_pages=rng.choice((128, 256, 512, 1024)))
    elif kind == "flat":
        case = _prefill("", rng.choice(("cfg2", "cfg3")), log_int(100, 1500), log_int(8192, 131_072), layers, flat=True)
    elif kind == "host":
        n_query = log_int(300, 2048)
        case = _prefill("", rng.choice(("cfg2", "cfg3")), n_query, max(n_query, log_int(4096, 131_072)), layers,
                        host_pass=rng.choice((256, 512, 1024)))
    else:
        batch = log_int(1, 40 if kind == "append" else 128)
        lo = log_int(700, 40_000 if kind == "append" else 65_536)
        lo = min(lo, _MAX_TOKENS // batch)
        hi = max(lo, min(1_048_576 // (20 if kind == "append" else 1), int(lo * rng.uniform(1.0, 8.0)), 2 * _MAX_TOKENS // batch - lo))
        case = _decode("", batch, lo, hi, layers, keys=rng.choice(("e4m3", "e4m3", "bf16")), flat=kind == "decode_flat",
                       append=kind == "append")
    del case["name"]
    return case


class _GrowingBatch(DecodeWorkload):
    """A decode batch whose pools hold what every sequence may grow to, as an engine sizes them once: the pages in use lie
    anywhere in them, whatever the sequences' present lengths."""

    def __init__(self, cfg):
        super().__init__(cfg, make_ctx=False)
        dev, used = self.device, self.n_pg
        self.n_pg = cfg.batch * -(-(cfg.ctx_hi + cfg.ctx_grow) // cfg.kv_page)
        place = torch.randperm(self.n_pg, generator=torch.Generator().manual_seed(cfg.seed))[:used].to(device=dev, dtype=torch.int32)
        self.page_table = torch.where(self.page_table >= 0, place[self.page_table.clamp(min=0).long()], -1)
        n_rows = self.n_pg * cfg.kv_page
        self.keys = inputs.indexer_keys(cfg, n_rows, dev)
        self.kmean = torch.zeros((n_rows // cfg.B, cfg.d_I), dtype=torch.bfloat16, device=dev)
        for r in range(cfg.R):
            self.k[r], self.v[r] = inputs.attn_kv(cfg, r, n_rows, dev)
        self.ctx = binding.Context(self.params, cfg.batch, self.page_table.shape[1] * cfg.kv_page, cfg.batch, device=dev)


def _config(case, seed):
    base = CONFIGS[case["base"]]
    change = {"seed": int(seed), "R": case["layers"], "hi_enable": not case["flat"], "q_chunk": 0}
    if case["kind"].startswith("decode"):
        change.update(batch=case["batch"], ctx_lo=case["ctx_lo"], ctx_hi=case["ctx_hi"], key_dtype=case["keys"],
                      ctx_grow=1 if case["kind"] == "decode_append" else 0)
    else:
        change.update(L=case["n_key"], M=case["keep_pages"])
    return base.replace(**change)


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def prepare(case, seed):
    cfg = _config(case, seed)
    state = {"kind": case["kind"], "cfg": cfg}
    if case["kind"].startswith("decode"):
        wl = _GrowingBatch(cfg) if case["kind"] == "decode_append" else DecodeWorkload(cfg)
        wl.prepare()                                    # the mean keys of the tokens cached so far
        state["wl"] = wl
        if case["kind"] == "decode_append":
            g = torch.Generator(device=wl.device).manual_seed(int(seed) * 1_000_003 + 999_331)
            new = lambda d, std: torch.randn((cfg.batch, d), generator=g, device=wl.device).mul_(std).to(torch.bfloat16)  # noqa: E731
            state["k_new"] = new(cfg.d_I, 1.0 / math.sqrt(cfg.d_I))
            state["kv_new"] = [new(cfg.d_qk, 1.0) for _ in range(cfg.R)]
            state["ctx_now"] = torch.empty_like(wl.ctx_len)
        return state
    wl = PrefillWorkload(cfg, q_pos0=case["n_key"] - case["n_query"], n_query=case["n_query"], n_key=case["n_key"])
    wl.prepare()
    state["wl"] = wl
    # the sub-block that holds the chunk's first key, and everything after it, is what a chunk adds to the mean keys
    state["first_key"] = wl.q_pos0 // cfg.B * cfg.B
    if case["kind"] == "prefill_host":
        stage_queries = case["host_pass"]
        state["stage_queries"] = stage_queries
        nbytes = binding.host_stage_bytes(wl.params, stage_queries)
        state["stage"] = [torch.empty(nbytes, dtype=torch.uint8, device=wl.device) for _ in range(2)]
        state["q_idx"], state["w"], state["q"] = _pinned(wl.q_idx), _pinned(wl.w), [_pinned(q) for q in wl.q]
        state["out"] = [torch.empty(o.shape, dtype=o.dtype, pin_memory=True) for o in wl.out]
        wl.q_idx = wl.w = None
        wl.q, wl.out, wl.lse = [], [], []
    return state


def run(state):
    wl, cfg = state["wl"], state["cfg"]
    keys, scale = wl.keys["k"], wl.keys.get("scale")
    if state["kind"].startswith("decode"):
        ctx_len = wl.ctx_len
        grown = {}
        if state["kind"] == "decode_append":
            wl.ctx.append(state["k_new"], keys, scale, wl.kmean, wl.page_table, ctx_len, state["ctx_now"], state["kv_new"], wl.k)
            ctx_len = state["ctx_now"]
            grown = {"keys": keys, "scale": scale, "kmean": wl.kmean, "caches": wl.k, "ctx_len": ctx_len}
        wl.ctx.layer_group(wl.q_idx, wl.w, keys, scale, wl.kmean, 0, cfg.batch, 0, wl.q, wl.k, wl.v, wl.out, wl.lse, wl.sparse_idx,
                           wl.n_sparse, wl.page_table, ctx_len)
        return {"out": wl.out, "lse": wl.lse, "sparse_idx": wl.sparse_idx, "n_sparse": wl.n_sparse, **grown}
    if state["kind"] == "prefill_host":
        wl.ctx.layer_group_host(state["q_idx"], state["w"], keys, scale, wl.kmean, wl.q_pos0, wl.n_query, wl.n_key, state["q"], wl.k,
                                wl.v, state["out"], state["stage_queries"], state["stage"])
        return {"out": state["out"]}
    a = state["first_key"]
    wl.ctx.block_means(keys[a:], None if scale is None else scale[a:], wl.n_key - a, wl.kmean[a // cfg.B:])
    wl.ctx.layer_group(wl.q_idx, wl.w, keys, scale, wl.kmean, wl.q_pos0, wl.n_query, wl.n_key, wl.q, wl.k, wl.v, wl.out, wl.lse,
                       wl.sparse_idx, wl.n_sparse)
    return {"out": wl.out, "lse": wl.lse, "sparse_idx": wl.sparse_idx, "n_sparse": wl.n_sparse, "kmean": wl.kmean}


def _per_query(cfg, t):
    """(mean keys scored, tokens scored, rows attended) of the query at position t."""
    cand = max(0, t - cfg.W - cfg.S + 1)
    first, last = cfg.S // cfg.P, (t - cfg.W) // cfg.P
    pages = last - first + 1 if cand > 0 else 0
    kept = pages if not cfg.hi_enable else min(pages, cfg.M)
    sub = pages * (cfg.P // cfg.B) if cfg.hi_enable and pages > cfg.M else 0
    scored = min(cand, kept * cfg.P)
    return sub, scored, min(t + 1, cfg.S + cfg.W) + min(cfg.Ksp, scored)


def work(case):
    """What the method cannot do without: each query scored against the mean keys of its eligible pages and the tokens of the
    kept ones, its rows attended in every layer; each input read once and each output written once."""
    cfg = _config(case, 0)
    key_bytes = cfg.d_I + 4 if cfg.key_dtype == "e4m3" else 2 * cfg.d_I
    row_bytes = cfg.d_qk * 2 if cfg.mla else (cfg.d_qk + cfg.d_v) * 2
    per_query_bytes = cfg.H_I * (2 * cfg.d_I + 4) + cfg.R * cfg.H * (2 * cfg.d_qk + 2 * cfg.d_v + 4) + 4 * cfg.Ksp + 4
    if case["kind"].startswith("decode"):
        n, weight, positions = cfg.batch, cfg.batch / 64.0, [cfg.ctx_lo + (cfg.ctx_hi - cfg.ctx_lo) * (i + 0.5) / 64 for i in range(64)]
        positions = [int(p) - 1 for p in positions]
    else:
        n, weight, step = case["n_query"], 1.0, max(1, case["n_query"] // 512)
        positions = list(range(case["n_key"] - n, case["n_key"], step))
        weight = n / len(positions)
    sub = scored = rows = 0.0
    for t in positions:
        s, c, r = _per_query(cfg, t)
        sub, scored, rows = sub + weight * s, scored + weight * c, rows + weight * r
    flops = 2.0 * cfg.H_I * cfg.d_I * (sub + scored) + 2.0 * cfg.R * cfg.H * (cfg.d_qk + cfg.d_v) * rows
    if case["kind"].startswith("decode"):               # every sequence reads its own caches
        cache = sub * cfg.d_I * 2 + scored * key_bytes + rows * row_bytes * cfg.R
        if case["kind"] == "decode_append":
            per_query_bytes += 2 * (2 * cfg.d_I + cfg.R * row_bytes)
    else:                                               # the queries of a chunk share the caches
        n_key = case["n_key"]
        reach = min(n_key, rows, n + cfg.W + cfg.S + min(scored, n_key))
        cache = min(sub, n_key / cfg.B) * cfg.d_I * 2 + min(scored, n_key) * key_bytes + reach * row_bytes * cfg.R
        if case["kind"] == "prefill":                   # the chunk's own keys into mean keys
            cache += n * key_bytes + n / cfg.B * cfg.d_I * 2
    return {"bytes": n * per_query_bytes + cache, "flops": flops}


def tolerance(case):
    """Attention: bf16 probabilities and bf16 results of fp32 sums; two kernels that sum in different orders are 2.2e-3 apart (both are
    2.0e-3 from fp64).  A selection is decided on fp32 sums, so a candidate at the very edge of its budget may change places with the
    next one when the sums are taken in another order: that moves the entries between the two in its query's ascending list, and
    changes that query's output.  Seen with the flat scores of 1000 queries summed in another order: one query of the 1000, 8e-4 of
    all list entries, at most 0.14 of the output's root mean square.  Stated: four times these."""
    return {"rel": 9e-3, "max": 0.5, "differ": 3e-3}
