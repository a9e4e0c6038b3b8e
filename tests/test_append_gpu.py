"""Rotate + append of long chunks, several tokens per CTA or four CTAs on an SM (297 tokens of a launch on): the cache bits, row
scales included, are those of short chunks, which take one token per CTA and two CTAs on an SM, and the outputs those of the same
rows folded in short chunks, within the bounds of tests/chain.py (a wrong rotation of a query would show: inputs are N(0, 1))."""
import pytest
import torch

from paper_2605_12471_b200 import binding
from tests.chain import TOL

pytestmark = pytest.mark.gpu

KINDS = {"bf16": ("bf16", 0), "bf16_interleaved": ("bf16", binding.KVF_ROPE_INTERLEAVED), "f32": ("f32", 0),
         "f32_interleaved": ("f32", binding.KVF_ROPE_INTERLEAVED), "int8": ("bf16", binding.KVF_CACHE_INT8),
         "int4_interleaved": ("bf16", binding.KVF_CACHE_INT4 | binding.KVF_ROPE_INTERLEAVED)}


def _inputs(lead, n, h, kv, d, dtype):
    return [torch.randn(*lead, n, heads, d, device="cuda").to(torch.float32 if dtype == "f32" else torch.bfloat16) for heads in (h, kv, kv)]


# both sides of each line of the dispatch, remainders of 2 and 4 tokens; 7 / 1 heads leave threads of a CTA without an item
@pytest.mark.parametrize("heads", [(8, 2), (7, 1)], ids=["8_2", "7_1"])
@pytest.mark.parametrize("kind", KINDS)
def test_long_chunks_append_the_bits_of_short_ones(kind, heads):
    dtype, flags = KINDS[kind]
    torch.manual_seed(len(kind))
    for d in (128, 64) if not flags & (binding.KVF_CACHE_INT8 | binding.KVF_CACHE_INT4) else (128,):
        for n in (296, 297, 300, 513, 1023, 1024, 1027, 1030):
            first = 77
            x = _inputs((), first + n, *heads, d, dtype)
            got, scales = [], []
            for cuts in ([first, n], [first] + [250] * (n // 250) + [n % 250]):
                c = binding.Cache(binding.make_config(*heads, d, dtype, first + n + 50, n, rope_base=10000.0, flags=flags))
                c.storage.fill_(0x5A)
                out = torch.cat([c.fold_step(*(t.contiguous() for t in step)) for step in zip(*(t.split(cuts) for t in x))])
                assert c.status() == binding.KVF_OK
                got.append((out.float(), c.storage))
                if flags & (binding.KVF_CACHE_INT8 | binding.KVF_CACHE_INT4):
                    scales.append([c.scales(kv) for kv in (0, 1)])
            rows = slice(0, first + n)
            if flags & (binding.KVF_CACHE_INT8 | binding.KVF_CACHE_INT4):
                assert all(torch.equal(*(s[:, rows] for s in pair)) for pair in zip(scales[-2], scales[-1]))
            assert torch.equal(*(_held(s, heads[1], first + n + 50, d, dtype, flags)[:, :, rows] for _, s in got))
            assert (got[0][0] - got[1][0]).abs().max().item() <= 2 * TOL[dtype][0]


# the lines of the dispatch in tokens per SM: one CTA of one token becomes four to an SM (fp32, quantised rows: two tokens) behind 2,
# four tokens from 7 (quantised: 6) on; remainders behind them
@pytest.mark.parametrize("kind", KINDS)
def test_the_lines_between_one_and_several_tokens_per_cta(kind):
    dtype, flags = KINDS[kind]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    quant = flags & (binding.KVF_CACHE_INT8 | binding.KVF_CACHE_INT4)
    lines = [2 * sms] + ([6 * sms - 1] if quant else [7 * sms - 1] if dtype == "bf16" else [])
    torch.manual_seed(len(kind))
    for n in (line + more for line in lines for more in (0, 1, 2, 3)):
        x = _inputs((), n, 8, 2, 128, dtype)
        got = []
        for cuts in ([n], [250] * (n // 250) + [n % 250]):
            c = binding.Cache(binding.make_config(8, 2, 128, dtype, n, n, rope_base=10000.0, flags=flags))
            out = torch.cat([c.fold_step(*(t.contiguous() for t in step)) for step in zip(*(t.split(cuts) for t in x))])
            assert c.status() == binding.KVF_OK
            got.append((out.float(), c.k_plane(), c.v_plane(), *((c.scales(0), c.scales(1)) if quant else ())))
        assert (got[0][0] - got[1][0]).abs().max().item() <= 2 * TOL[dtype][0]
        assert all(torch.equal(*pair) for pair in list(zip(*got))[1:])


@pytest.mark.parametrize("flags", [0, binding.KVF_CACHE_INT8, binding.KVF_CACHE_INT4], ids=["bf16", "int8", "int4"])
@pytest.mark.parametrize("members,n", [(300, 1), (310, 2), (200, 3), (160, 4), (1100, 3)])
def test_many_members_of_a_few_tokens(members, n, flags):
    """A CTA takes tokens of one member only."""
    torch.manual_seed(members)
    cfg = binding.make_config(4, 1, 128, "bf16", 128, 20, rope_base=10000.0, flags=flags)
    x, first = _inputs((members,), n, 4, 1, 128, "bf16"), _inputs((members,), 20, 4, 1, 128, "bf16")
    ws = torch.empty(binding.workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    pools, outs = [], []
    for together in (True, False):
        pool = torch.zeros(binding.paged_pool_bytes(cfg, members), dtype=torch.uint8, device="cuda")
        tables = torch.arange(members, device="cuda").flip(0).to(torch.int32).view(members, 1)
        caches = [binding.PagedCache(cfg, pool, members, tables[i], workspace=ws) for i in range(members)]
        for c, step in zip(caches, zip(*first)):
            c.fold_step(*(t.contiguous() for t in step))
        if together:
            outs.append(binding.Batch(caches).fold_step(*x))
        else:
            outs.append(torch.stack([c.fold_step(*(t.contiguous() for t in step)) for c, step in zip(caches, zip(*x))]))
        torch.cuda.synchronize()
        pools.append(pool)
    assert torch.equal(*pools)
    assert (outs[0].float() - outs[1].float()).abs().max().item() <= 2 * TOL["bf16"][0]


def _held(storage, kv, capacity, d, dtype, flags):
    """[K and V, KV head, row, bytes of codes or elements]"""
    row = d // 2 if flags & binding.KVF_CACHE_INT4 else d if flags & binding.KVF_CACHE_INT8 else d * (4 if dtype == "f32" else 2)
    return storage[:2 * kv * capacity * row].view(2, kv, capacity, row)


@pytest.mark.parametrize("flags", [0, binding.KVF_CACHE_INT8, binding.KVF_CACHE_INT4], ids=["bf16", "int8", "int4"])
def test_batches_append_the_bits_of_single_caches(flags):
    torch.manual_seed(3)
    for n in (33, 57, 114, 129):              # 9 members: 297, 513, 1026 and 1161 tokens to a launch
        cfg = binding.make_config(8, 2, 128, "bf16", 300, n, rope_base=10000.0, flags=flags)
        pools = []
        x = _inputs((9,), n, 8, 2, 128, "bf16")
        for together in (True, False):
            pool = torch.zeros(binding.paged_pool_bytes(cfg, 27), dtype=torch.uint8, device="cuda")
            tables = torch.arange(27, device="cuda").flip(0).to(torch.int32).view(9, 3)
            caches = [binding.PagedCache(cfg, pool, 27, tables[i]) for i in range(9)]
            if together:
                binding.Batch(caches).fold_step(*x)
            else:
                for c, step in zip(caches, zip(*x)):
                    c.fold_step(*(t.contiguous() for t in step))
            torch.cuda.synchronize()
            pools.append(pool)
        assert torch.equal(*pools)


# Rotate + append calls its inputs' lines into L2, and every kernel sets itself up, while the kernel before still runs: inputs that this
# kernel is writing are read as it leaves them, in buffers that hold the step before's until then.
@pytest.mark.parametrize("dtype,flags,chunk", [("bf16", 0, 1), ("bf16", 0, 256), ("bf16", 0, 2048), ("bf16", binding.KVF_CACHE_INT8, 256),
                                               ("bf16", binding.KVF_ROPE_INTERLEAVED, 300), ("f32", 0, 512)])
def test_inputs_written_by_the_kernel_ahead_of_the_step(dtype, flags, chunk):
    steps, kind = 8, torch.float32 if dtype == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(chunk)
    ins = [[torch.randn(chunk, h, 128, generator=gen, device="cuda").to(kind) for h in (32, 8, 8)] for _ in range(steps)]
    total = steps * chunk
    outs = []
    for own_buffers in (True, False):
        cache = binding.Cache(binding.make_config(32, 8, 128, dtype, total, chunk, rope_base=10000.0, flags=flags))
        cache.storage.zero_()
        x, out = [torch.zeros_like(y) for y in ins[0]], []
        torch.cuda.synchronize()
        for y in ins:
            if own_buffers:
                out.append(cache.fold_step(*y))
                torch.cuda.synchronize()
            else:
                torch._foreach_copy_(x, y)
                out.append(cache.fold_step(*x))
        torch.cuda.synchronize()
        assert cache.status() == binding.KVF_OK
        outs.append((out, cache.storage))
    assert all(torch.equal(a, b) for a, b in zip(outs[0][0], outs[1][0])) and torch.equal(outs[0][1], outs[1][1])
