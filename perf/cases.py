"""The work users of this framework have it do, as cases that can be timed and compared.

A case is one sequence (or, with `caches`, several decoded or folded together) whose cache already
holds `prefix` tokens: a pass folds `tokens` more in chunks of `chunk`, then `decode` tokens one at a
time, through the public binding, and hands back every output row and the rows it appended.  At the
start of a pass the cache is set back to `prefix` rows (`set_len`, the way several questions are asked
about one folded haystack), so a pass can be repeated.  Inputs are i.i.d. Gaussian, as everywhere in
this repository (no trained weights and no text corpus are at hand).

Fields: q_heads, kv_heads, head_dim; dtype "bf16" / "f32"; cache "plain" / "int8" / "int4" (storage of
the rows); scale (of the inputs); prefix, tokens, chunk, decode; sinks, window (0 = full prefix);
caches (0 = one contiguous cache, else a batch of that many paged caches); ragged (batch members of
different length); behind (the merge kernel behind the step, closed by a flush); host (inputs and
results in pinned host memory, copies inside the call).
"""
import math

import torch

from paper_2605_12471_b200 import binding

_BASE = dict(q_heads=32, kv_heads=8, head_dim=128, dtype="bf16", cache="plain", scale=1.0, prefix=0, tokens=0, chunk=256,
             decode=0, sinks=0, window=0, caches=0, ragged=False, behind=False, host=False)
_PAGE = 128


def _case(**kw):
    return dict(_BASE, **kw)


def listed():
    return [
        # the smallest calls: eight steps of 64 tokens of a toy model, fp32, head_dim 64 (latency and launches)
        _case(name="tiny_fold", q_heads=4, kv_heads=1, head_dim=64, dtype="f32", tokens=512, chunk=64),
        # a medium document in large chunks: 16K tokens at an 8B model's attention shape, trained-like logits
        _case(name="prefill_16k_c2048", scale=128 ** -0.5, tokens=16384, chunk=2048),
        # the deep chain the framework is named for: 128K tokens, 256 at a time
        _case(name="deep_chain_128k_c256", tokens=131072, chunk=256, behind=True),
        # the precision ablation: the same fold on an fp32 cache
        _case(name="fold_f32_64k_c512", dtype="f32", tokens=65536, chunk=512),
        # a 7B model's heads (groups of 7), a document of no round length, a question and an answer behind it
        _case(name="qwen_ragged_15k", q_heads=28, kv_heads=4, tokens=15077, chunk=256, decode=30),
        # a question about a long folded context: a short chunk and thirty decoded tokens, latency per token
        _case(name="question_128k_bf16", prefix=129024, tokens=32, chunk=32, decode=30),
        # the same on a cache stored as int8 codes
        _case(name="question_128k_int8", cache="int8", prefix=129024, tokens=32, chunk=32, decode=30),
        # a long fold into a quantised cache
        _case(name="fold_int8_64k_c256", cache="int8", tokens=65536, chunk=256),
        # attention sinks and a sliding window: constant work per step
        _case(name="window_32k_c256", tokens=32768, chunk=256, sinks=4, window=1020),
        # serving: 32 sequences of different length decoded together, token by token
        _case(name="batch_decode_32x16k", prefix=16384, decode=16, caches=32, ragged=True),
        # a whole model's layers per chunk: 32 layer caches advance by 1024 tokens with one launch of each kernel
        _case(name="layer_stack_32x8k_c1024", prefix=7168, tokens=1024, chunk=1024, caches=32),
        # end to end from pinned host buffers, copies beside the compute
        _case(name="host_chain_16k_c256", tokens=16384, chunk=256, behind=True, host=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: shapes of the models in this repository's tests, sizes spread over the whole range."""
    while True:
        case = _draw(rng)
        w = work(case)
        # (fp32 takes three tensor-core products for one, head_dim 64 the CUDA cores)
        cost = w["flops"] * (40 if case["head_dim"] == 64 else 3 if case["dtype"] == "f32" else 1)
        steps = -(-case["tokens"] // case["chunk"]) + case["decode"]
        if cost <= 1.4e14 and steps <= 512 and w["bytes"] <= 2e11:
            return case


def _draw(rng):
    kind = rng.choice(["tiny", "fold", "fold", "f32", "quant", "question", "question", "window", "batch_decode", "batch_fold", "host"])
    heads = rng.choice([(32, 8), (32, 8), (28, 4), (16, 16), (12, 2)])
    shape = dict(q_heads=heads[0], kv_heads=heads[1])
    cache = rng.choice(["plain", "int8", "int4"])
    if kind == "tiny":
        q, kv = rng.choice([(4, 1), (8, 2), (2, 2)])
        chunk = _log(rng, 8, 256)
        return _case(q_heads=q, kv_heads=kv, head_dim=64, dtype=rng.choice(["f32", "f32", "bf16"]), tokens=chunk * rng.randint(2, 16) + rng.randint(0, 7), chunk=chunk)
    if kind == "fold":
        return _case(**shape, scale=rng.choice([1.0, 128 ** -0.5]), prefix=rng.choice([0, 0, _log(rng, 100, 40000)]), tokens=_log(rng, 512, 100000),
                     chunk=_log(rng, 64, 8192), behind=rng.random() < 0.5)
    if kind == "f32":
        return _case(**shape, dtype="f32", tokens=_log(rng, 512, 65536), chunk=_log(rng, 64, 4096), decode=rng.choice([0, 8]))
    if kind == "quant":
        return _case(**shape, cache=rng.choice(["int8", "int4"]), tokens=_log(rng, 512, 65536), chunk=_log(rng, 64, 4096), decode=rng.choice([0, 30]))
    if kind == "question":
        tokens = _log(rng, 1, 128)
        return _case(**shape, cache=cache, prefix=_log(rng, 1000, 130000), tokens=tokens, chunk=tokens, decode=rng.randint(1, 30))
    if kind == "window":
        return _case(**shape, tokens=_log(rng, 2048, 65536), chunk=_log(rng, 64, 1024), sinks=4, window=_log(rng, 250, 4000))
    if kind == "batch_decode":
        return _case(**shape, cache=cache, prefix=_log(rng, 500, 24000), decode=rng.randint(2, 16), caches=_log(rng, 2, 40), ragged=rng.random() < 0.7)
    if kind == "batch_fold":
        chunk = _log(rng, 128, 1024)
        return _case(**shape, cache=cache, prefix=_log(rng, 256, 12000), tokens=chunk, chunk=chunk, caches=_log(rng, 2, 40))
    return _case(**shape, tokens=_log(rng, 1024, 16384), chunk=_log(rng, 64, 2048), behind=True, host=True)


def _member_prefixes(case):
    """Rows the members of a batch hold (ragged: spread over half the range below `prefix`)."""
    n, p = case["caches"], case["prefix"]
    return [p - (i * 37 % n) * p // (2 * n) if case["ragged"] else p for i in range(n)]


def _chunks(case):
    full, rest = divmod(case["tokens"], case["chunk"])
    return [case["chunk"]] * full + ([rest] if rest else []) + [1] * case["decode"]


def _seen(case, prefix, n):
    """(visible query-key pairs of a step of n tokens, cache rows it reads)."""
    rows = prefix
    if case["window"] and prefix - case["window"] > case["sinks"]:
        rows = case["sinks"] + case["window"]
    return n * rows + n * (n + 1) // 2, rows + n


def work(case):
    h, kv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    eb = 4 if case["dtype"] == "f32" else 2
    row = {"plain": d * eb, "int8": d + 4, "int4": d // 2 + 4}[case["cache"]]
    flops = moved = 0
    for prefix in (_member_prefixes(case) if case["caches"] else [case["prefix"]]):
        for n in _chunks(case):
            pairs, rows = _seen(case, prefix, n)
            flops += 4 * h * d * pairs
            # the step's own rows are read as inputs and written to the cache; earlier rows are read from it
            moved += 2 * kv * (rows - n) * row + 2 * kv * n * row + n * (2 * h + 2 * kv) * d * eb
            prefix += n
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    # Against the same fold in 64 bits, deep rows of a chain are off by 1e-6 (fp32) and 3.5e-3 (bf16), whole chains
    # by 1.5e-7 and 1.3e-3.  Codes and stored keys are whole values: a last-bit difference in a sine may flip a rounding.
    return {"rel": 4e-6 if case["dtype"] == "f32" else 1e-2, "differ": 1e-5}


def _draws(case, gen, shape):
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    x = torch.randn(shape, generator=gen, device="cuda", dtype=dtype)
    return x if case["scale"] == 1.0 else x.mul_(case["scale"])


def _inputs(case, gen, n, lead=()):
    return [_draws(case, gen, (*lead, n, heads, case["head_dim"])) for heads in (case["q_heads"], case["kv_heads"], case["kv_heads"])]


def _config(case, capacity, max_chunk):
    flags = {"plain": 0, "int8": binding.KVF_CACHE_INT8, "int4": binding.KVF_CACHE_INT4}[case["cache"]]
    if case["behind"]:
        flags |= binding.KVF_COMBINE_BEHIND
    if case["host"]:
        flags |= binding.KVF_HOST_UPLOAD_AHEAD | binding.KVF_HOST_DOWNLOAD_BEHIND
    return binding.make_config(case["q_heads"], case["kv_heads"], case["head_dim"], case["dtype"], capacity, max_chunk,
                               rope_base=10000.0 if case["head_dim"] == 64 else 500000.0, flags=flags)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return _prepare_batch(case, gen) if case["caches"] else _prepare_one(case, gen)


def _prepare_one(case, gen):
    chunks = _chunks(case)
    end = case["prefix"] + sum(chunks)
    fill = min(2048, case["prefix"])
    cache = binding.Cache(_config(case, end, max(chunks + [fill])))
    cache.storage.zero_()
    if case["window"]:
        cache.set_window(case["sinks"], case["window"])
    for at in range(0, case["prefix"], 2048):
        cache.fold_step(*_inputs(case, gen, min(2048, case["prefix"] - at)))
    cache.flush()
    q, k, v = _inputs(case, gen, sum(chunks))
    out = torch.zeros_like(q)
    if case["host"]:
        q, k, v, out = (x.cpu().pin_memory() for x in (q, k, v, out))
    steps = list(zip(*(x.split(chunks) for x in (q, k, v, out))))
    # the rows a pass appends, as views of the cache
    heads, new = case["kv_heads"], slice(case["prefix"], end)
    if case["cache"] == "int4":
        planes = cache.storage[:heads * end * case["head_dim"]].view(2, heads, end, case["head_dim"] // 2)
        rows = [planes[0, :, new], planes[1, :, new]]
    else:
        rows = [cache.k_plane()[:, new], cache.v_plane()[:, new]]
    if case["cache"] != "plain":
        rows += [cache.scales(0)[:, new], cache.scales(1)[:, new]]
    return {"case": case, "cache": cache, "steps": steps, "out": out, "rows": rows}


def _prepare_batch(case, gen):
    chunks, lens = _chunks(case), _member_prefixes(case)
    n, end = case["caches"], case["prefix"] + sum(_chunks(case))
    cfg = _config(case, end, max(chunks + [min(1024, case["prefix"])]))
    per = -(-end // _PAGE)
    pool = torch.zeros(binding.paged_pool_bytes(cfg, n * per), dtype=torch.uint8, device="cuda")
    tables = torch.randperm(n * per, generator=gen, device="cuda").to(torch.int32).view(n, per)     # pages in no order
    shared = torch.empty(binding.workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    caches = [binding.PagedCache(cfg, pool, n * per, tables[i], workspace=shared) for i in range(n)]
    for cache, rows in zip(caches, lens):
        for at in range(0, rows, 1024):
            cache.fold_step(*_inputs(case, gen, min(1024, rows - at)))
    batch = binding.Batch(caches)
    steps = [[*x, torch.zeros_like(x[0])] for x in (_inputs(case, gen, m, (n,)) for m in chunks)]
    return {"case": case, "caches": caches, "lens": lens, "batch": batch, "steps": steps, "pool": pool}


def run(state):
    case = state["case"]
    if case["caches"]:
        for cache, rows in zip(state["caches"], state["lens"]):
            cache.set_len(rows)
        for q, k, v, out in state["steps"]:
            state["batch"].fold_step(q, k, v, out=out, ragged=case["ragged"])
        return {"out": [s[3] for s in state["steps"]], "pool": state["pool"]}
    cache = state["cache"]
    cache.set_len(case["prefix"])
    step = cache.fold_step_host if case["host"] else cache.fold_step
    for q, k, v, out in state["steps"]:
        step(q, k, v, out=out)
    if case["behind"]:
        cache.flush()
    return {"out": state["out"], "rows": state["rows"]}


def _rotated(case, x, pos0):
    """x [n, heads, d] rotated at positions pos0, pos0 + 1, ..., in 64 bits."""
    d = case["head_dim"]
    base = 10000.0 if d == 64 else 500000.0
    inv = base ** (-2.0 * torch.arange(d // 2, device="cuda", dtype=torch.float64) / d)
    theta = (pos0 + torch.arange(x.shape[0], device="cuda", dtype=torch.float64))[:, None, None] * inv
    lo, hi = x.double().split(d // 2, dim=-1)
    return torch.cat([lo * theta.cos() - hi * theta.sin(), hi * theta.cos() + lo * theta.sin()], dim=-1)


def _stored(case, x):
    """(rows [n, heads, d] as the attention reads them, their scales or None): what a quantised cache keeps of them."""
    if case["cache"] == "plain":
        return x.double(), None
    levels = 127 if case["cache"] == "int8" else 7
    top = x.double().abs().amax(-1, keepdim=True)
    return (x.double() * (levels / top.clamp(min=1e-300))).round().clamp(-levels, levels) * (top / levels), (top / levels)[..., 0]


class _Fold:
    """One sequence's fold in 64 bits."""

    def __init__(self, case, capacity):
        shape = (case["kv_heads"], capacity, case["head_dim"])
        self.case, self.len = case, 0
        self.k, self.v = (torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(2))
        self.scales = [torch.zeros(shape[:2], dtype=torch.float64, device="cuda") for _ in range(2)]

    def append(self, k, v):
        new = slice(self.len, self.len + k.shape[0])
        for plane, scales, rows in ((self.k, self.scales[0], _rotated(self.case, k, self.len)), (self.v, self.scales[1], v)):
            rows, s = _stored(self.case, rows)
            plane[:, new] = rows.transpose(0, 1)
            if s is not None:
                scales[:, new] = s.T
        self.len = new.stop

    def step(self, q, k, v):
        case, first, n = self.case, self.len, q.shape[0]
        self.append(k, v)
        heads, d, group = case["kv_heads"], case["head_dim"], case["q_heads"] // case["kv_heads"]
        keys = torch.arange(self.len, device="cuda")
        lo = max(first - case["window"], 0) if case["window"] else 0
        out = torch.empty((n, heads, group, d), dtype=torch.float64, device="cuda")
        q = _rotated(case, q, first).view(n, heads, group, d) / math.sqrt(d)
        some = max(1, (1 << 28) // (group * self.len))
        for a in range(0, n, some):
            b = min(n, a + some)
            hidden = keys[None] > first + torch.arange(a, b, device="cuda")[:, None]
            hidden |= (keys >= case["sinks"]) & (keys < lo)
            hidden = hidden[:, None].expand(b - a, group, self.len).reshape(-1, self.len)
            for h in range(heads):
                p = (q[a:b, h].reshape(-1, d) @ self.k[h, :self.len].T).masked_fill_(hidden, -math.inf)
                p = p.sub_(p.amax(-1, keepdim=True)).exp_()
                out[a:b, h] = ((p @ self.v[h, :self.len]) / p.sum(-1, keepdim=True)).view(b - a, group, d)
        return out.view(n, heads * group, d)


def exact(case, seed):
    """The outputs of run in 64 bits, from the statement of the fold alone; codes and pages of a pool are whole values and have none."""
    if work(case)["flops"] > 6e13:
        return None
    gen = torch.Generator(device="cuda").manual_seed(seed)
    chunks = _chunks(case)
    end = case["prefix"] + sum(chunks)
    if case["caches"]:
        n, lens = case["caches"], _member_prefixes(case)
        torch.randperm(n * -(-end // _PAGE), generator=gen, device="cuda")
        held = [[_inputs(case, gen, min(1024, rows - at))[1:] for at in range(0, rows, 1024)] for rows in lens]
        steps = [_inputs(case, gen, m, (n,)) for m in chunks]
        outs = [torch.empty(s[0].shape, dtype=torch.float64, device="cuda") for s in steps]
        for i in range(n):
            fold = _Fold(case, end)
            for k, v in held[i]:
                fold.append(k, v)
            for (q, k, v), out in zip(steps, outs):
                out[i] = fold.step(q[i], k[i], v[i])
        return {"out": outs, "pool": None}
    fold = _Fold(case, end)
    for at in range(0, case["prefix"], 2048):
        fold.append(*_inputs(case, gen, min(2048, case["prefix"] - at))[1:])
    steps = zip(*(x.split(chunks) for x in _inputs(case, gen, sum(chunks))))
    out = torch.cat([fold.step(q, k, v) for q, k, v in steps])
    new = slice(case["prefix"], end)
    rows = [fold.k[:, new], fold.v[:, new]] if case["cache"] == "plain" else [None, None] + [s[:, new] for s in fold.scales]
    return {"out": out.cpu() if case["host"] else out, "rows": rows}
