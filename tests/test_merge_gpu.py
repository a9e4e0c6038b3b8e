"""The merge of partial results: its kernels for few rows and for few parts against the general one, bit for bit."""
import pytest
import torch

from paper_2605_12471_b200 import binding

pytestmark = pytest.mark.gpu

MANY, FEW = [5, 9, 18, 33, 48, 65, 96], [2, 3, 4, 5, 8]


@pytest.mark.parametrize("h,kv", [(32, 8), (28, 4), (12, 2), (16, 16)])
@pytest.mark.parametrize("flags", [0, binding.KVF_OUT_F32, binding.KVF_CACHE_INT4], ids=["bf16", "f32", "int4"])
def test_merge_kernels_give_the_same_bits(h, kv, flags):
    """Up to four parts of a row, nine and more parts of few rows: the bits of the general merge kernel, which a batch of members
    of different length (here one) takes for the same cut."""
    gen = torch.Generator(device="cuda").manual_seed(h)
    prefix = 96 * 128 + 17
    cfg = binding.make_config(h, kv, 128, "bf16", prefix + 320, 2048, rope_base=10000.0, flags=flags)
    pages = -(-cfg.capacity // 128)
    pool = torch.zeros(binding.paged_pool_bytes(cfg, pages), dtype=torch.uint8, device="cuda")
    c = binding.PagedCache(cfg, pool, pages, torch.arange(pages, device="cuda", dtype=torch.int32))
    for at in range(0, prefix, 2048):
        c.fold_step(*(torch.randn(min(2048, prefix - at), heads, 128, generator=gen, device="cuda").bfloat16() for heads in (h, kv, kv)))
    batch, compared = binding.Batch([c]), set()
    gp = 1 << (h // kv - 1).bit_length()                        # rows of a token in a partial slot
    # the decode kernel; two streams (two parts a range); row pairs with a short second tile, a short last pair
    for n, cuts in ((1, MANY), (2, MANY), (3, MANY), (17, [1, 2, *MANY]), (40, FEW), (300, FEW)):
        x = [torch.randn(n, heads, 128, generator=gen, device="cuda").bfloat16() for heads in (h, kv, kv)]
        for splits in cuts:
            c.set_splits(splits)
            c.set_len(prefix)
            lse, lse_b = torch.empty(n, h, device="cuda"), torch.empty(1, n, h, device="cuda")
            alone = c.plan(n)
            if batch.plan(n, prefix)[:3] != alone[:3]:          # (a cut the batch's partial area does not hold)
                continue
            # two parts to a range where one row tile is dealt to two streams (not in the decode kernel)
            parts = alone[1] * (2 if n * (h // kv) > 16 and n * gp <= 128 else 1)
            rows = n * h <= 8 * torch.cuda.get_device_properties(0).multi_processor_count
            compared.add("small" if parts <= 4 else "eight" if parts <= 8 else "general" if not rows or parts > 96 else
                         "rows_24" if parts <= 24 else "rows_48" if parts <= 48 else "rows_96")
            want = batch.fold_step(*(t[None].contiguous() for t in x), ragged=True, lse=lse_b)[0]
            c.set_len(prefix)
            got = c.fold_step(*x, lse=lse)
            assert torch.equal(got, want) and torch.equal(lse, lse_b[0])
    assert c.status() == binding.KVF_OK and batch.status_word() == 0
    assert compared >= {"small", "eight", "rows_24", "rows_48", "rows_96"}, compared
