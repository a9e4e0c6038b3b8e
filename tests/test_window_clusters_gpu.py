"""Small bf16 steps under a window (clusters of one, two or four CTAs per 128-row tile merge their key ranges): against the
CUDA-core kernel on the same rows.

Both read the same bf16 cache.  What the tensor-core kernel rounds are the probabilities, to bf16: an output element moves by at most
2^-8 of sum p |v|, which the CUDA-core kernel gives when it is run on |v|.  Scores differ by fp32 sums of 128 products, up to ~60
in the growing case (5e-4, as in test_early_issue_gpu.py): the same for a log-sum-exp, twice that of sum p |v| for an output.
bf16 outputs are rounded by both, 2^-8 of the element each."""
import pytest
import torch

from paper_2605_12471_b200 import binding

pytestmark = pytest.mark.gpu


def _run(h, kv, prefix, n, sinks, window, growing, out_f32, gen):
    rows = prefix + n
    q, k, v = (torch.randn(rows, heads, 128, generator=gen, device="cuda") for heads in (h, kv, kv))
    if growing:
        k *= torch.linspace(0.1, 12.0, rows, device="cuda")[:, None, None]
    q, k, v = (x.bfloat16() for x in (q, k, v))

    def fold(flags, values):
        c = binding.Cache(binding.make_config(h, kv, 128, "bf16", rows, rows, rope_base=10000.0, flags=flags))
        c.storage.zero_()
        c.fold_step(q[:prefix].contiguous(), k[:prefix].contiguous(), values[:prefix].contiguous())
        c.set_window(sinks, window)
        lse = torch.empty(n, h, device="cuda")
        before = c.launch_count()
        out = c.fold_step(q[prefix:].contiguous(), k[prefix:].contiguous(), values[prefix:].contiguous(), lse=lse)
        assert c.status() == binding.KVF_OK
        return out.float(), lse, c.launch_count() - before, c.plan(n, prefix)

    kind = binding.KVF_OUT_F32 if out_f32 else 0
    a, la, launches, plan = fold(kind, v)
    b, lb, _, _ = fold(kind | binding.KVF_FORCE_SIMT, v)
    weight = fold(binding.KVF_OUT_F32 | binding.KVF_FORCE_SIMT, v.abs())[0]
    bound = (2.0 ** -8 + 2 * 5e-4) * weight + (0.0 if out_f32 else 2 * 2.0 ** -8) * torch.maximum(a.abs(), b.abs())
    assert ((a - b).abs() <= bound).all()
    assert (la - lb).abs().max().item() <= 5e-4
    assert launches == plan[3]
    return plan


# rows at the edges of a 128-row tile; one key tile (fewer than the CTAs of a cluster), a window inside it, many; padded groups
@pytest.mark.parametrize("out_f32", [False, True], ids=["bf16", "f32"])
@pytest.mark.parametrize("h,kv", [(8, 2), (7, 1), (3, 3)])
@pytest.mark.parametrize("prefix,sinks,window", [(130, 1, 3), (300, 4, 20), (600, 0, 129), (900, 64, 300), (1500, 4, 1300)])
def test_small_windowed_steps_against_the_cuda_core_kernel(h, kv, prefix, sinks, window, out_f32):
    gen = torch.Generator(device="cuda").manual_seed(prefix + h)
    for n in (17, 31, 32, 33, 65, 190):
        _run(h, kv, prefix, n, sinks, window, n & 1, out_f32, gen)


# clusters of four, two and one CTA (two streams each), and the 256-row CTAs beyond
@pytest.mark.parametrize("n,window,parts", [(64, 1020, 8), (256, 1020, 4), (400, 500, 2), (700, 500, None)])
def test_one_two_and_four_ctas_per_row_tile(n, window, parts):
    plan = _run(32, 8, 2000, n, 4, window, False, False, torch.Generator(device="cuda").manual_seed(n))
    if parts and torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert plan[1] == parts and plan[3] == 2


# A NaN, or an infinity that makes one, reaches the rows that see it and no others, as with the CUDA-core kernel.  `where`: a query
# element, a key of the chunk (seen from its token on), a key of an earlier step inside the window, one outside (seen by nobody).
@pytest.mark.parametrize("bad", [float("nan"), float("inf")], ids=["nan", "inf"])
@pytest.mark.parametrize("where", ["query", "own key", "earlier key", "hidden key"])
@pytest.mark.parametrize("n,window", [(64, 1020), (256, 1020), (400, 500), (700, 500)])
def test_not_a_number_reaches_the_rows_that_see_it(n, window, where, bad):
    h, kv, prefix = 32, 8, 2000
    rows, gen = prefix + n, torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn(rows, heads, 128, generator=gen, device="cuda").bfloat16() for heads in (h, kv, kv))
    q2, k2 = q.clone(), k.clone()
    if where == "query":
        q2[prefix + n // 2, 9, 77] = bad
    else:
        k2[{"own key": prefix + n // 3, "earlier key": prefix - 10, "hidden key": prefix - window - 300}[where], 2, 5] = bad

    def fold(flags, q, k):
        c = binding.Cache(binding.make_config(h, kv, 128, "bf16", rows, rows, rope_base=10000.0, flags=flags))
        c.storage.zero_()
        c.fold_step(q[:prefix].contiguous(), k[:prefix].contiguous(), v[:prefix].contiguous())
        c.set_window(4, window)
        if flags:
            c.set_splits(1)          # (the CUDA-core kernel's merge leaves out a part whose sum is a NaN)
        lse = torch.empty(n, h, device="cuda")
        out = c.fold_step(q[prefix:].contiguous(), k[prefix:].contiguous(), v[prefix:].contiguous(), lse=lse)
        assert c.status() == binding.KVF_OK
        return out, lse

    clean, clean_lse = fold(0, q, k)
    out, lse = fold(0, q2, k2)
    simt, _ = fold(binding.KVF_FORCE_SIMT, q2, k2)
    assert torch.equal(out.isnan(), simt.isnan())
    seen = torch.zeros(n, h, dtype=torch.bool, device="cuda")
    if where == "query":
        seen[n // 2, 9] = True
    elif where != "hidden key":
        seen[n // 3 if where == "own key" else 0:, 8:12] = True
    assert torch.equal(out[~seen], clean[~seen]) and torch.equal(lse[~seen], clean_lse[~seen])
    if bad != bad:
        assert out[seen].isnan().all()


# paged caches (pages in no order), alone and advancing together: clusters of four, two and one CTA
@pytest.mark.parametrize("members,n,window,parts", [(1, 64, 1020, 8), (2, 64, 1020, 8), (3, 64, 1020, 4), (3, 100, 400, 2), (2, 33, 150, 4)])
def test_paged_caches_and_batches_under_a_window(members, n, window, parts):
    h, kv, prefix = 32, 8, 1500
    rows, gen = prefix + n, torch.Generator(device="cuda").manual_seed(members + n)
    cfg = lambda flags: binding.make_config(h, kv, 128, "bf16", rows, rows, rope_base=10000.0, flags=binding.KVF_OUT_F32 | flags)
    pages = 4 * (-(-rows // 512))
    tables = torch.randperm(members * pages, generator=gen, device="cuda").to(torch.int32).view(members, pages)
    pool = torch.full((binding.paged_pool_bytes(cfg(0), members * pages) // 2,), 0x7FC0, dtype=torch.int16, device="cuda").view(torch.uint8)
    caches = [binding.PagedCache(cfg(0), pool, members * pages, t) for t in tables]
    x = [torch.randn(members, rows, heads, 128, generator=gen, device="cuda").bfloat16() for heads in (h, kv, kv)]
    chunk = lambda y: y[:, prefix:].contiguous()
    for i, c in enumerate(caches):
        c.fold_step(*(y[i, :prefix].contiguous() for y in x))
        c.set_window(4, window)
    lse = torch.empty(members, n, h, device="cuda")
    if members == 1:
        plan = caches[0].plan(n, prefix)
        out = caches[0].fold_step(*(chunk(y)[0] for y in x), lse=lse[0])[None]
        assert caches[0].status() == binding.KVF_OK
    else:
        batch = binding.Batch(caches)
        plan = batch.plan(n, prefix)
        out = batch.fold_step(*(chunk(y) for y in x), lse=lse)
        assert batch.status_word() == 0
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert plan[1] == parts and plan[3] == 2
    for i in range(members):
        def simt(values):
            c = binding.Cache(cfg(binding.KVF_FORCE_SIMT))
            c.storage.zero_()
            c.fold_step(*(y[i, :prefix].contiguous() for y in (x[0], x[1], values)))
            c.set_window(4, window)
            want_lse = torch.empty(n, h, device="cuda")
            return c.fold_step(*(y[i, prefix:].contiguous() for y in (x[0], x[1], values)), lse=want_lse), want_lse

        want, want_lse = simt(x[2])
        weight, _ = simt(x[2].abs())
        assert ((out[i] - want).abs() <= (2.0 ** -8 + 2 * 5e-4) * weight).all()
        assert (lse[i] - want_lse).abs().max().item() <= 5e-4
