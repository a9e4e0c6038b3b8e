"""Small steps of head_dim 64 take one launch (fold_small.cu): against the three-launch path (KVF_FORCE_SIMT) with every
bit of the cache, and against the oracle through the chains of test_fold_gpu.py.

Tolerance: both paths compute in fp32 and differ in the order of their sums: 64-term scores up to ~|s| = 8 (2^-21
each), exponentials and output sums of unit size: a few 1e-6; a bf16 output may round the other way (one ulp, 2^-8
relative, at |out| up to 4)."""
import pytest
import torch

from paper_2605_12471_b200 import binding

pytestmark = pytest.mark.gpu


def _caches(h, kv, dtype, capacity, max_chunk, flags=0):
    made = []
    for extra in (0, binding.KVF_FORCE_SIMT):
        c = binding.Cache(binding.make_config(h, kv, 64, dtype, capacity, max_chunk, rope_base=10000.0, flags=flags | extra))
        c.storage.fill_(7)                 # (the value rows up to the tile boundary are cleared by both)
        made.append(c)
    return made


def _inputs(h, kv, n, dtype, gen):
    t = torch.float32 if dtype == "f32" else torch.bfloat16
    return [torch.randn(n, heads, 64, generator=gen, device="cuda", dtype=t) for heads in (h, kv, kv)]


def _compare(a, b, dtype):
    (oa, la), (ob, lb) = a, b
    tol = 1e-5 if dtype == "f32" else 2.0 ** -6
    assert (oa.float() - ob.float()).abs().max().item() <= tol
    assert (la - lb).abs().max().item() <= 1e-5


# chunks at the edges of the 32-row tile, the 64-key tile and the slices; groups of 1, 3, 4, 7
@pytest.mark.parametrize("h,kv", [(4, 1), (2, 2), (6, 2), (7, 1)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("flags", [0, binding.KVF_ROPE_INTERLEAVED], ids=["half", "interleaved"])
def test_one_launch_against_three(h, kv, dtype, flags):
    chunks = [1, 7, 8, 48, 63, 1, 64, 65, 3, 130, 250, 1, 33]
    gen = torch.Generator(device="cuda").manual_seed(h * 10 + kv)
    small, general = _caches(h, kv, dtype, 1000, 250, flags)
    for n in chunks:
        assert small.plan(n)[3] == 1 and general.plan(n)[3] >= 2
        q, k, v = _inputs(h, kv, n, dtype, gen)
        got = []
        for c in (small, general):
            lse = torch.empty(n, h, device="cuda")
            got.append((c.fold_step(q, k, v, lse=lse), lse))
        _compare(*got, dtype)
        assert torch.equal(small.storage, general.storage), n
        la, lb = torch.empty(n, h, device="cuda"), torch.empty(n, h, device="cuda")
        _compare((small.attend(q, lse=la), la), (general.attend(q, lse=lb), lb), dtype)
    assert small.status() == binding.KVF_OK


def test_one_launch_under_a_window_and_with_wide_clusters():
    gen = torch.Generator(device="cuda").manual_seed(3)
    for window, chunks in ((100, [64, 64, 50, 64, 1, 64]), (0, [250] * 4 + [8, 1, 32, 64])):
        small, general = _caches(4, 1, "f32", 1500, 250)
        if window:
            small.set_window(4, window)
            general.set_window(4, window)
        for n in chunks:
            q, k, v = _inputs(4, 1, n, "f32", gen)
            got = []
            for c in (small, general):
                lse = torch.empty(n, 4, device="cuda")
                got.append((c.fold_step(q, k, v, lse=lse), lse))
            _compare(*got, "f32")
            assert torch.equal(small.storage, general.storage)


def test_results_over_the_inputs_take_the_three_launches():
    """Output rows over the queries' own rows, and over the new keys' (2 / 2 heads: the same shape)."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = [_inputs(2, 2, 200, "f32", gen) for _ in range(2)]
    for over in (0, 1, 2):
        small, general = _caches(2, 2, "f32", 400, 200)
        for ins in x:
            want = general.fold_step(*ins)
            mine = [t.clone() for t in ins]
            launches = small.launch_count()
            small.fold_step(*mine, out=mine[over])
            assert (small.launch_count() - launches == 1) == (over == 0)
            assert (mine[over] - want).abs().max().item() <= 1e-5
        assert torch.equal(small.storage, general.storage)


# (n, heads, 64-row key tiles, kernels): slices of up to 7 (one row tile) and 4 (eight) key tiles take one launch, up to two
# more where the three launches' splits take a fifth tile (no multiple of four); far beyond never
@pytest.mark.parametrize("n,h,kv,tiles,kernels", [(1, 4, 1, 112, 1), (1, 4, 1, 113, 1), (1, 4, 1, 116, 3), (1, 4, 1, 513, 3),
                                                  (8, 2, 2, 513, 3), (4, 14, 2, 132, 3), (64, 4, 1, 64, 1), (64, 4, 1, 68, 3)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_long_prefixes_take_the_launches_that_split_them(n, h, kv, tiles, kernels, dtype):
    prefix = 64 * tiles - n
    gen = torch.Generator(device="cuda").manual_seed(prefix)
    small, general = _caches(h, kv, dtype, prefix + n, n)
    held = torch.randn(small.storage.numel() // (4 if dtype == "f32" else 2), generator=gen, device="cuda", dtype=small.torch_dtype)
    q, k, v = _inputs(h, kv, n, dtype, gen)
    got = []
    for c in (small, general):
        c.storage.copy_(held.view(torch.uint8))
        c.set_len(prefix)
        lse = torch.empty(n, h, device="cuda")
        before = c.launch_count()
        got.append((c.fold_step(q, k, v, lse=lse), lse))
        assert c.launch_count() - before == (kernels if c is small else 3)
    assert small.plan(n, prefix)[3] == kernels
    _compare(*got, dtype)
    assert torch.equal(small.storage, general.storage)


# tiles of 32 keys: prefixes around their edges and around every number of slices, chunks within one and across two of them
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("flags", [0, binding.KVF_ROPE_INTERLEAVED], ids=["half", "interleaved"])
def test_short_slices(dtype, flags):
    gen = torch.Generator(device="cuda").manual_seed(7)
    slices = set()
    for prefix in (0, 1, 31, 32, 33, 63, 64, 97, 128, 130, 191, 255, 256, 400, 480):
        for n in (1, 5, 32, 33, 64):
            small, general = _caches(4, 1, dtype, prefix + n, prefix + n, flags)
            got = []
            held, new = _inputs(4, 1, max(prefix, 1), dtype, gen), _inputs(4, 1, n, dtype, gen)
            for c in (small, general):
                c.storage.fill_(0x5A)
                if prefix:
                    general.set_len(0)
                    general.fold_step(*held)
                    c.storage.copy_(general.storage)
                c.set_len(prefix)
                lse = torch.empty(n, 4, device="cuda")
                got.append((c.fold_step(*new, lse=lse), lse))
            slices.add(small.plan(n, prefix)[1])
            assert small.plan(n, prefix)[3] == 1 and small.status() == binding.KVF_OK
            _compare(*got, dtype)
            assert torch.equal(small.storage, general.storage)
    assert slices == {1, 2, 4, 8, 16}


def test_chunks_of_two_key_tiles_on_bf16_rows_have_shorter_slices():
    for dtype, kernels in (("f32", 1), ("bf16", 3)):
        c, _ = _caches(2, 2, dtype, 4096, 160)
        assert c.plan(160, 4096 - 160)[3] == kernels          # bf16: 34.5 us in three launches, 37.4 in one


@pytest.mark.parametrize("h,kv", [(4, 1), (7, 1), (2, 2)])
def test_fp32_results_of_bf16_rows(h, kv):
    gen = torch.Generator(device="cuda").manual_seed(h)
    small, general = _caches(h, kv, "bf16", 400, 130, binding.KVF_OUT_F32)
    for n in (1, 64, 130, 33):
        q, k, v = _inputs(h, kv, n, "bf16", gen)
        got = []
        for c in (small, general):
            lse = torch.empty(n, h, device="cuda")
            got.append((c.fold_step(q, k, v, lse=lse), lse))
            assert got[-1][0].dtype == torch.float32
        assert small.plan(n, len(small) - n)[3] == 1
        _compare(*got, "f32")                  # (nothing is rounded to bf16 behind the sums)
        assert torch.equal(small.storage, general.storage)
    # fp32 rows over bf16 queries are not "exactly over them": the three launches
    buf = torch.empty(64 * h * 64, dtype=torch.float32, device="cuda")
    over = buf.view(torch.bfloat16)[:64 * h * 64].view(64, h, 64)
    q, k, v = _inputs(h, kv, 64, "bf16", gen)
    over.copy_(q)
    want, before = general.fold_step(q, k, v), small.launch_count()
    got = small.fold_step(over, k, v, out=buf.view(64, h, 64))
    assert small.launch_count() - before > 1
    assert (got - want).abs().max().item() <= 1e-5


def test_lse_and_cache_rows_over_the_inputs_take_the_three_launches():
    gen = torch.Generator(device="cuda").manual_seed(9)
    n, h = 64, 4
    for over in (0, 1, 2):                     # the log-sum-exp over the first rows of the queries, keys and values
        small, general = _caches(h, 1, "f32", 400, n)
        ins = _inputs(h, 1, n, "f32", gen)
        lse = torch.empty(n, h, device="cuda")
        want = (general.fold_step(*ins, lse=lse), lse)
        mine = [t.clone() for t in ins]
        inside = mine[over].view(-1)[:n * h].view(n, h)
        before = small.launch_count()
        _compare((small.fold_step(*mine, lse=inside), inside), want, "f32")
        assert small.launch_count() - before > 1
        assert torch.equal(small.storage, general.storage)
    for kv in (0, 1):                          # keys and values that lie in rows of the cache no one holds yet
        small, general = _caches(h, 1, "f32", 400, n)
        ins = _inputs(h, 1, n, "f32", gen)
        want = general.fold_step(*ins)
        inside = (small.v_plane() if kv else small.k_plane())[0, 200:200 + n].view(n, 1, 64)
        inside.copy_(ins[1 + kv])
        mine = [ins[0], inside, ins[2]] if kv == 0 else [ins[0], ins[1], inside]
        before = small.launch_count()
        got = small.fold_step(*mine)
        assert small.launch_count() - before > 1
        assert (got - want).abs().max().item() <= 1e-5
        rows = slice(0, n)
        assert torch.equal(small.k_plane()[:, rows], general.k_plane()[:, rows]) and torch.equal(small.v_plane()[:, rows], general.v_plane()[:, rows])
