"""The cuts of the (KV head, key tile) line at sizes where a finer or a coarser one is measurably slower (us per step in
the comments: the cut asserted, the cut it must not be).  kvf_cache_plan launches nothing; the figures are of 148 SMs."""
import pytest
import torch

from paper_2605_12471_b200 import binding

pytestmark = pytest.mark.gpu


def _plan(h, kv, n, rows, flags=0, window=0):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("measured on 148 SMs")
    c = binding.Cache(binding.make_config(h, kv, 128, "bf16", rows + n, n, rope_base=10000.0, flags=flags))
    if window:
        c.set_window(4, window)
    return c.plan(n, rows)


@pytest.mark.parametrize("h,kv,n,rows,flags,lo,hi", [
    (28, 4, 64, 4000, 0, 2, 8),                             # 22 us with eight ranges per head, 31 with 18
    (12, 2, 32, 16000, 0, 8, 32),                           # 35 with 31, 56 with 72
    (16, 16, 96, 839, 0, 4, 4),                             # 15.9 with four, 17.5 with two and with three
    (28, 4, 200, 500, 0, 1, 1),                             # 19.7 uncut, 21.6 with three
    (32, 8, 512, 250, binding.KVF_CACHE_INT8, 1, 1),        # 30.3 uncut, 31.8 with two
    (32, 8, 64, 700, binding.KVF_CACHE_INT8, 3, 8),         # 25.4 uncut, 20.3 with three
    (32, 8, 256, 768, 0, 3, 4),                             # 20.1 with four, 24.6 uncut
])
def test_ranges_per_head_of_steps_that_leave_sms_idle(h, kv, n, rows, flags, lo, hi):
    assert lo <= _plan(h, kv, n, rows, flags)[1] <= hi


def test_ranges_under_a_window():
    assert 3 <= _plan(32, 8, 256, 8192, window=1020)[1] <= 4       # 25.1 us with four, 30.7 with two
    # 13 row pairs, 11 ranges over four heads: 62.5 us; two per head: 70.8
    assert _plan(28, 4, 416, 5860, binding.KVF_CACHE_INT8, window=2860)[2] == 13 * 11


@pytest.mark.parametrize("n,rows,flags,groups", [(1783, 44202, 0, 10),                            # 1052 us; 11: 1366, uncut ~1190
                                                 (1777, 20337, binding.KVF_CACHE_INT8, 10),       # 760; 11: 986
                                                 (2048, 2000, 0, 8), (2048, 30000, 0, 9),         # 115 / 145 with 9; 906 / 1002 uncut
                                                 (2048, 4000, binding.KVF_CACHE_INT8, 8)])        # 255 / 274 with 9
def test_ranges_of_steps_that_fill_the_sms(n, rows, flags, groups):
    assert _plan(32, 8, n, rows, flags)[2] == groups * -(-n // 64)


# few rows: a block per row merges any number of parts up to 96 in ~2 us, so the ranges are short
@pytest.mark.parametrize("h,kv,n,rows,flags,lo,hi", [
    (12, 2, 45, 7027, 0, 16, 48),                           # 16.6 us with 28, 26.5 with eight
    (32, 4, 21, 6264, 0, 16, 37),                           # 17.2 with 25, 26.4 with eight
    (12, 2, 18, 4663, binding.KVF_CACHE_INT4, 12, 48),      # 17.2 with 19, 26.0 with eight
])
def test_ranges_per_head_where_rows_are_merged_a_block_each(h, kv, n, rows, flags, lo, hi):
    assert lo <= _plan(h, kv, n, rows, flags)[1] <= hi


def test_ranges_of_ragged_steps_are_priced_with_their_own_merge():
    """The kernel that merges many parts of few rows needs the ranges from the host, which does not have them for members of different
    length: those keep to ranges that one trip to memory merges, eight a head.  Told from the bits, as the order of the sums is the cut's."""
    h, kv, n, prefix, pages = 12, 2, 45, 7027, 56
    cfg = binding.make_config(h, kv, 128, "bf16", pages * 128, 1024, rope_base=10000.0, flags=binding.KVF_OUT_F32)
    pool = torch.zeros(binding.paged_pool_bytes(cfg, 2 * pages), dtype=torch.uint8, device="cuda")
    tables = torch.arange(2 * pages, dtype=torch.int32, device="cuda").view(2, pages)
    caches = [binding.PagedCache(cfg, pool, 2 * pages, tables[i]) for i in range(2)]
    gen = torch.Generator(device="cuda").manual_seed(8)
    draw = lambda *lead: [torch.randn(*lead, heads, 128, generator=gen, device="cuda").bfloat16() for heads in (h, kv, kv)]
    for c in caches:
        for at in range(0, prefix, 1024):
            c.fold_step(*draw(min(1024, prefix - at)))
    batch, x = binding.Batch(caches), draw(2, n)

    def step(splits):
        for c in caches:
            c.set_len(prefix)
        caches[0].set_splits(splits)
        return batch.fold_step(*x, ragged=True)

    out, lock_step = step(0), batch.plan(n, prefix)[1]
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert lock_step > 8                                # members that advance together
        assert torch.equal(out, step(8)) and not torch.equal(out, step(lock_step))
    assert batch.status_word() == 0
