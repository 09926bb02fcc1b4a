"""Timed cases of the eviction path, each a call sequence that a user's program makes.

A case is a dict of plain values; `kind` says which part of the library it exercises:

  prefill  one batch (or two batches in turn, through one context) of prompts: score, allocate and
           evict every layer, then one gather-compaction.  `calls` is "run" (Cake.run, every layer
           in hand) or "layers" (the per-layer calls, as a model's prefill makes them between its
           layers); `lse` hands over the window rows' log-sum-exps, as a fused attention forward
           leaves them.
  decode   tokens of decode-time eviction after a finished prefill, all layers, then the state is
           read back; with `begin` the pass also builds the decode cache (one prompt's answer).
  int4     4-bit compaction of a finished prefill.
  select   the stand-alone per-head selection that allocates nothing.

Inputs are random with the structure of the library's own synthetic workloads: a temperature per
layer, sink, heavy-hitter, recent and needle keys along the mean window query.  The stages after
the scoring start from supplied indicators and preferences, so that their inputs do not depend on
how the scores are computed.
"""
import math
import random

import torch

from paper_2503_12491_b200 import binding, harness, profile_case, synth


# ------------------------------------------------------------------ the cases
def _prefill(**kw):
    c = dict(kind="prefill", layers=32, q_heads=32, kv_heads=8, head_dim=128, dtype="bf16", window=32, pool=7,
             pool_mode="max", gamma=200.0, budget=2048, requests=1, shortest=4096, longest=4096, batches=1,
             lse=False, calls="layers")
    c.update(kw)
    return c


def _after(kind, **kw):
    c = dict(kind=kind, layers=32, q_heads=32, kv_heads=8, head_dim=128, dtype="bf16", window=32, pool=7,
             pool_mode="max", budget=2048, requests=1, shortest=16384, longest=16384)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest configuration: four fp32 layers of 512 tokens; launches and host time count
        _prefill(name="tiny-fp32", layers=4, q_heads=4, kv_heads=4, head_dim=64, dtype="fp32", window=16, pool=5,
                 gamma=1.0, budget=128, shortest=512, longest=512, calls="run"),
        # multi-head attention at 4K: many short (request, head) pairs per layer
        _prefill(name="mha-4k", kv_heads=32, budget=1024, calls="run"),
        # a long-document prompt of a grouped-query model
        _prefill(name="gqa-32k", shortest=32768, longest=32768),
        # the 128K prompt the headline benchmark uses
        _prefill(name="gqa-128k", budget=4096, shortest=131072, longest=131072),
        # a ragged batch: eight requests of 8K to 64K
        _prefill(name="ragged-8x8k-64k", requests=8, shortest=8192, longest=65536, calls="run"),
        # a server between long prompts: short prompts of odd lengths, one after the other, a new batch each
        _prefill(name="serve-odd", budget=512, shortest=1501, longest=7919, batches=2),
        # scoring behind a fused attention forward that hands over its log-sum-exps; odd lengths
        _prefill(name="lse-2x24k-odd", requests=2, shortest=20011, longest=28657, lse=True),
        # fp32 inputs with average pooling: research use and the numerics baseline
        _prefill(name="fp32-gqa-6k", layers=8, q_heads=16, kv_heads=4, dtype="fp32", pool_mode="avg",
                 budget=512, shortest=6001, longest=6001, calls="run"),
        # generation after a 128K-class prompt: large heads (budgets of 4096 on average, uneven over layers)
        _after("decode", name="decode-4096", budget=4096, shortest=65536, longest=65536, tokens=8, begin=False),
        # short answers for a batch of four requests, cache set-up included
        _after("decode", name="decode-batch4", layers=16, budget=768, requests=4, shortest=3000, longest=9000,
               tokens=8, begin=True),
        # the quantised cache of a 32K-class batch
        _after("int4", name="int4-2048", requests=2, shortest=12000, longest=40000, group=32),
        # one layer's selection for a caller with its own scores and its own memory plan
        dict(kind="select", name="select-8x128k", heads=8, n=131040, keep=4064),
    ]


def _log_int(rng, lo, hi):
    """An integer spread evenly over the logarithm of lo..hi."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# (query heads, KV heads, head_dim, window) in use: grouped-query and multi-head models
_HEADS_BF16 = [(32, 8, 128, 32), (32, 32, 128, 32), (32, 8, 128, 16), (16, 2, 128, 16), (16, 8, 128, 32), (16, 16, 64, 32)]
_HEADS_FP32 = [(4, 4, 64, 16), (16, 4, 128, 32), (8, 8, 64, 32), (8, 2, 128, 16)]


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "prefill", "prefill-fp32", "decode", "int4", "select"])
    if kind == "select":
        heads = _log_int(rng, 1, 64)
        n = _log_int(rng, 256, min(262144, 32768 // heads * 32))
        return dict(kind="select", heads=heads, n=n, keep=min(n, _log_int(rng, 16, max(16, n // 4))))
    fp32 = kind == "prefill-fp32"
    q_heads, kv_heads, head_dim, window = rng.choice(_HEADS_FP32 if fp32 else _HEADS_BF16)
    pool, pool_mode = rng.choice([(7, "max"), (7, "max"), (5, "max"), (7, "avg")])
    shape = dict(q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim, window=window, pool=pool, pool_mode=pool_mode)
    if kind.startswith("prefill"):
        layers = rng.choice([4, 8]) if fp32 else rng.choice([8, 16, 32])
        requests = rng.choice([1, 1, 1, 2, 4, 8])
        # fp32: at most 8K tokens in all; bf16: no more K than the ragged batch has
        most = 8192 // requests if fp32 else min(131072, 12_000_000_000 // (layers * kv_heads * head_dim * 2 * requests))
        longest = _log_int(rng, 512, most)
        shortest = longest if requests == 1 else max(256, longest // rng.choice([1, 2, 8]))
        batches = 2 if longest <= 8192 and rng.random() < 0.3 else 1
        if batches == 2:
            shortest = max(256, longest // rng.choice([2, 3, 5]))
        lse = rng.random() < 0.25
        return _prefill(layers=layers, dtype="fp32" if fp32 else "bf16", gamma=rng.choice([1.0, 200.0]),
                        budget=_log_int(rng, 128, max(256, min(4096, longest // 4))), requests=requests, shortest=shortest,
                        longest=longest, batches=batches, lse=lse, calls="layers" if lse else rng.choice(["run", "layers"]),
                        **shape)
    layers, requests = rng.choice([(8, 1), (8, 4), (16, 1), (16, 2), (16, 4), (32, 1), (32, 2)])
    budget = _log_int(rng, 128, 4096 if layers * kv_heads * requests <= 256 else 1024)
    longest = _log_int(rng, 4 * budget, 16 * budget)
    more = dict(tokens=4 if layers * requests > 32 else rng.choice([4, 8]), begin=rng.random() < 0.5) if kind == "decode" else \
        dict(group=rng.choice([g for g in (32, 64, 128) if g <= head_dim]))
    return _after(kind, layers=layers, budget=budget, requests=requests, shortest=longest // rng.choice([1, 2]),
                  longest=longest, **more, **shape)


# ------------------------------------------------------------------ inputs
def _lengths(case, batch=0):
    """Prompt lengths of a batch: a property of the case, not of the seed."""
    lo, hi = case["shortest"], case["longest"]
    if case["requests"] == 1:                        # a second batch brings the other end of the range
        return (hi if batch == 0 else lo,)
    r = random.Random(lo * 1000003 + hi * 101 + batch)
    return tuple(r.randint(lo, hi) for _ in range(case["requests"]))


def _workload(case, batch=0):
    return synth.Workload("case", case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"], _lengths(case, batch),
                          case["window"], case["pool"], case.get("gamma", 1.0), case["layers"] * case["budget"],
                          case["dtype"], 1)


def _context(case, works):
    mode = binding.CAKE_POOL_AVG if case["pool_mode"] == "avg" else binding.CAKE_POOL_MAX
    return harness.cake_for(works[0], pool_mode=mode, max_total_tokens=max(w.total_tokens for w in works))


def _layer(w, gen, temperature):
    """Q_win, K and V of one layer: a few keys lie along the mean window query of their KV head."""
    dev, dt, d = "cuda", w.torch_dtype, w.head_dim
    q = torch.randn(len(w.seq_lens), w.n_q_heads, w.window, d, generator=gen, device=dev) * temperature
    k = torch.randn(w.n_kv_heads, w.total_tokens, d, generator=gen, device=dev, dtype=dt)
    v = torch.randn(w.n_kv_heads, w.total_tokens, d, generator=gen, device=dev, dtype=dt)
    beta = (torch.rand(w.n_kv_heads, w.total_tokens, generator=gen, device=dev) < 0.01).float() * 2.0
    cu = w.cu_seqlens
    for r, n_tok in enumerate(w.seq_lens):
        mean = q[r].view(w.n_kv_heads, -1, d).mean(dim=1)
        u = mean * (temperature * math.sqrt(d)) / (mean * mean).sum(dim=1, keepdim=True)
        b = beta[:, cu[r]:cu[r + 1]]
        n = n_tok - w.window
        b[:, max(0, n - 256):n].clamp_(min=1.0)
        b[:, :4] = 3.0
        b[:, torch.randint(0, max(n, 1), (16,), generator=gen, device=dev)] = 4.0
        b[:, n:] = 0.0
        k[:, cu[r]:cu[r + 1]] += (b[:, :, None] * u[:, None, :]).to(dt)
    return q.to(dt), k, v


def _evicted(case, gen):
    """A context whose prefill cascade is finished, on supplied indicators and preferences; its K and V."""
    w = _workload(case)
    cake = _context(case, [w])
    cake.begin(w.cu_seqlens)
    pref = torch.randn(len(w.seq_lens), w.n_layers, generator=gen, device="cuda", dtype=torch.float64).mul_(0.7).exp_()
    cake.set_preferences(pref)
    ks, vs = [], []
    for l in range(w.n_layers):
        x = torch.randn(w.n_kv_heads, w.total_tokens, generator=gen, device="cuda").exp_() * (1.0 / case["longest"])
        x = torch.nn.functional.max_pool1d(x, w.pool_kernel, 1, w.pool_kernel // 2).contiguous()
        cake.set_indicators(l, x)
        cake.allocate(l)
        cake.evict(l)
        ks.append(torch.randn(w.n_kv_heads, w.total_tokens, w.head_dim, generator=gen, device="cuda", dtype=w.torch_dtype))
        vs.append(torch.randn(w.n_kv_heads, w.total_tokens, w.head_dim, generator=gen, device="cuda", dtype=w.torch_dtype))
    return w, cake, ks, vs


def _bits(t):
    """The rows as whole numbers: the compaction moves bytes and computes nothing on them."""
    return t.view(torch.int16 if t.dtype == torch.bfloat16 else torch.int32)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "select":
        x = torch.randn(case["heads"], case["n"], generator=gen, device="cuda").exp_()
        x = torch.nn.functional.max_pool1d(x, 7, 1, 3).contiguous()
        return dict(kind=kind, values=x, keep=case["keep"],
                    out=torch.empty(case["heads"], case["keep"], dtype=torch.int32, device="cuda"))
    if kind == "prefill":
        works = [_workload(case, b) for b in range(case["batches"])]
        cake = _context(case, works)
        temps = random.Random(seed)
        batches = []
        for w in works:
            layers = [_layer(w, gen, math.exp(temps.uniform(math.log(0.5), math.log(4.0)))) for _ in range(w.n_layers)]
            qs, ks, vs = (list(x) for x in zip(*layers))
            lses = [profile_case.window_lse(w, q, k) for q, k in zip(qs, ks)] if case["lse"] else None
            cake.begin(w.cu_seqlens)
            rows = cake.packed_rows_bound()
            bufs = dict(k_out=torch.zeros(rows, w.head_dim, dtype=w.torch_dtype, device="cuda"),
                        v_out=torch.zeros(rows, w.head_dim, dtype=w.torch_dtype, device="cuda"),
                        row_offsets=torch.zeros(len(w.seq_lens) * w.n_layers + 1, dtype=torch.int64, device="cuda"),
                        positions=torch.zeros(rows, dtype=torch.int32, device="cuda"))
            out = [_bits(bufs["k_out"]), _bits(bufs["v_out"]), bufs["row_offsets"], bufs["positions"]]
            batches.append(dict(cu=w.cu_seqlens, qs=qs, ks=ks, vs=vs, lses=lses, bufs=bufs, out=out))
        return dict(kind=kind, cake=cake, batches=batches, layers=case["layers"], calls=case["calls"])
    w, cake, ks, vs = _evicted(case, gen)
    st = dict(kind=kind, cake=cake, ks=ks, vs=vs, layers=w.n_layers, requests=len(w.seq_lens))
    if kind == "int4":
        return dict(st, group=case["group"])
    dt, lead = w.torch_dtype, (case["tokens"], w.n_layers, len(w.seq_lens))
    q = (torch.randn(*lead, w.n_q_heads, w.head_dim, generator=gen, device="cuda") * 1.5).to(dt)
    k = torch.randn(*lead, w.n_kv_heads, w.head_dim, generator=gen, device="cuda").to(dt)
    v = torch.randn(*lead, w.n_kv_heads, w.head_dim, generator=gen, device="cuda").to(dt)
    st["new"] = [[(q[t, l], k[t, l], v[t, l]) for l in range(w.n_layers)] for t in range(case["tokens"])]
    st["lengths"] = cake.get_budgets().cpu().tolist()
    st["cache"] = None if case["begin"] else cake.decode_begin(ks, vs)
    return st


# ------------------------------------------------------------------ one pass
def run(state):
    kind = state["kind"]
    if kind == "prefill":
        cake, out = state["cake"], []
        for b in state["batches"]:
            if state["calls"] == "run" and b["lses"] is None:
                cake.run(b["qs"], b["ks"], b["vs"], b["cu"], **b["bufs"])
            else:
                cake.begin(b["cu"])
                for l in range(state["layers"]):
                    cake.score_layer(l, b["qs"][l], b["ks"][l], lse=b["lses"][l] if b["lses"] else None)
                    cake.allocate(l)
                    cake.evict(l)
                cake.compact(b["ks"], b["vs"], **b["bufs"])
            out += b["out"]
        return out
    if kind == "select":
        return binding.select_positions_static(state["values"], state["keep"], out=state["out"])
    cake = state["cake"]
    if kind == "int4":
        return cake.compact_int4(state["ks"], state["vs"], group=state["group"])
    k_cache, v_cache, offsets = state["cache"] or cake.decode_begin(state["ks"], state["vs"])
    for token in state["new"]:
        for l, (q, k, v) in enumerate(token):
            cake.decode_step(l, q, k, v, k_cache, v_cache)
    got = [cake.decode_get_state(r, l, state["lengths"][r][l]) for r in range(state["requests"]) for l in range(state["layers"])]
    pos, score, slot = (torch.cat([x.view(-1) for x in part]) for part in zip(*got))
    return [_bits(k_cache), _bits(v_cache), offsets, pos, score, slot]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    if case["kind"] == "select":
        return {"bytes": 4 * case["heads"] * (case["n"] + case["keep"]), "flops": 0}
    esize = 4 if case["dtype"] == "fp32" else 2
    L, hq, hkv, d, sw = (case[x] for x in ("layers", "q_heads", "kv_heads", "head_dim", "window"))
    row = d * esize
    total = dict(bytes=0, flops=0)
    for b in range(case.get("batches", 1)):
        lens = _lengths(case, b)
        kept = hkv * sum(min(L * case["budget"], L * n) for n in lens)          # packed rows
        if case["kind"] == "prefill":
            # K and the window queries in; the retained V rows in; K^, V^ and positions out
            total["bytes"] += L * hkv * sum(lens) * row + L * len(lens) * hq * sw * row + kept * (3 * row + 4)
            total["flops"] += L * hq * sw * sum(lens) * (2 * d + 8)
        elif case["kind"] == "int4":
            groups = d // case["group"]
            total["bytes"] += kept * (2 * row + d + 8 * groups + 4) + 8 * d * (kept // case["group"])
            total["flops"] += kept * d * 2 * 6
        else:
            # per token: every cached key, its score in and out, the rank list; the new rows
            tokens = case["tokens"]
            total["bytes"] += tokens * (kept * (row + 8 + 4) + L * len(lens) * (hq + 4 * hkv) * row)
            total["flops"] += tokens * kept * (hq // hkv) * (2 * d + 8)
            total["bytes"] += kept * (12 + (4 * row if case["begin"] else 0))
    return total


def tolerance(case):
    if case["kind"] in ("int4", "select"):
        return "exact"
    if case["kind"] == "decode":
        # scores are sums of fp32 softmax values; an entry whose score ties with the lowest one to within
        # their rounding may go in its place, which moves the entries of its head between the two
        return {"rel": 1e-4, "max": 1e-3, "differ": 0.005}
    # whole numbers only: a key whose indicator lies within fp32 rounding of a head's threshold may be kept
    # in place of its neighbour, which moves that head's packed rows between the two by one
    return {"rel": 0.0, "differ": 0.01}
