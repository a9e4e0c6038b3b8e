"""bf16 chunks of two row tiles (the early issue of Q K^T): against the CUDA-core kernel on the same rows.

Both read the same bf16 cache (checked bit for bit).  What the tensor-core kernel rounds are the probabilities: to bf16, whose
8 significant bits put the nearest value at most 2^-8 of a number away (half of the last bit, 2^-7 of a number just above a power
of two), so an output element by at most 2^-8 of sum p |v|, which the CUDA-core kernel gives when it is run on |v|.  Scores
differ by fp32 sums of 128 products, up to ~60 in the growing case (2^-24 * 60 * 128 = 5e-4): the same for a log-sum-exp,
twice that of sum p |v| for an output.  bf16 outputs are rounded by both, 2^-8 of the element each."""
import pytest
import torch

from paper_2605_12471_b200 import binding

pytestmark = pytest.mark.gpu


def _run(prefix, n, splits, growing, out_f32, gen):
    h, kv = 8, 2
    rows = prefix + n
    q, k, v = (torch.randn(rows, heads, 128, generator=gen, device="cuda") for heads in (h, kv, kv))
    if growing:      # the running maximum moves by more than the rescale threshold in many tiles
        k *= torch.linspace(0.1, 12.0, rows, device="cuda")[:, None, None]
    q, k, v = (x.bfloat16() for x in (q, k, v))

    def fold(flags, values, splits=0):
        c = binding.Cache(binding.make_config(h, kv, 128, "bf16", rows, rows, rope_base=10000.0, flags=flags))
        c.storage.zero_()
        if prefix:
            c.fold_step(q[:prefix].contiguous(), k[:prefix].contiguous(), values[:prefix].contiguous())
        c.set_splits(splits)
        if not flags & binding.KVF_FORCE_SIMT:
            assert c.plan(n)[0] == 1
        lse = torch.empty(n, h, device="cuda")
        out = c.fold_step(q[prefix:].contiguous(), k[prefix:].contiguous(), values[prefix:].contiguous(), lse=lse)
        assert c.status() == binding.KVF_OK
        return out.float(), lse, c.storage

    kind = binding.KVF_OUT_F32 if out_f32 else 0
    a, la, sa = fold(kind, v, splits)
    b, lb, sb = fold(kind | binding.KVF_FORCE_SIMT, v)
    weight, _, _ = fold(binding.KVF_OUT_F32 | binding.KVF_FORCE_SIMT, v.abs())
    assert torch.equal(sa, sb)
    bound = (2.0 ** -8 + 2 * 5e-4) * weight + (0.0 if out_f32 else 2 * 2.0 ** -8) * torch.maximum(a.abs(), b.abs())
    assert ((a - b).abs() <= bound).all()
    assert (la - lb).abs().max().item() <= 5e-4


# key tiles of 128 rows: one, two, three, many; the second row tile from one valid row on; one to many ranges
@pytest.mark.parametrize("out_f32", [False, True], ids=["bf16", "f32"])
@pytest.mark.parametrize("growing", [False, True], ids=["plain", "growing_maxima"])
@pytest.mark.parametrize("prefix", [0, 1, 127, 129, 1000])
def test_two_row_tiles_against_the_cuda_core_kernel(prefix, growing, out_f32):
    gen = torch.Generator(device="cuda").manual_seed(prefix + growing)
    for n in (33, 64, 65, 190):
        for splits in (0, 1, 3):
            _run(prefix, n, splits, growing, out_f32, gen)


# pairs of CTAs on quantised rows: the last key tile ends in the half of either CTA, at its edge, or before the second half
@pytest.mark.parametrize("flags", [binding.KVF_CACHE_INT8, binding.KVF_CACHE_INT4], ids=["int8", "int4"])
def test_pairs_of_ctas_at_the_end_of_the_planes(flags):
    gen = torch.Generator(device="cuda").manual_seed(5)
    for n in (128, 256):
        for prefix in (0, 44, 64, 65, 100, 172, 1000):
            rows = prefix + n
            x = [torch.randn(rows, heads, 128, generator=gen, device="cuda").bfloat16() for heads in (8, 2, 2)]
            outs = []
            for capacity in (rows, rows + 777):
                c = binding.Cache(binding.make_config(8, 2, 128, "bf16", capacity, rows, rope_base=10000.0, flags=flags))
                c.storage.fill_(0xFF)                # scales of rows nobody wrote: NaN
                if prefix:
                    c.fold_step(*(t[:prefix].contiguous() for t in x))
                outs.append(c.fold_step(*(t[prefix:].contiguous() for t in x)))
                assert c.status() == binding.KVF_OK
            assert torch.isfinite(outs[0]).all() and torch.equal(*outs)


@pytest.mark.parametrize("flags", [binding.KVF_CACHE_INT8, binding.KVF_CACHE_INT4], ids=["int8", "int4"])
def test_pairs_of_ctas_repeat_their_bits(flags):
    """A raw tile given back before its codes were read would show as another tile's codes now and then."""
    gen = torch.Generator(device="cuda").manual_seed(6)
    n = 256
    for prefix in (2048, 8448, 20000):
        c = binding.Cache(binding.make_config(32, 8, 128, "bf16", prefix + n, 2048, rope_base=10000.0, flags=flags))
        for at in range(0, prefix, 2048):
            c.fold_step(*(torch.randn(min(2048, prefix - at), heads, 128, generator=gen, device="cuda").bfloat16() for heads in (32, 8, 8)))
        x = [torch.randn(n, heads, 128, generator=gen, device="cuda").bfloat16() for heads in (32, 8, 8)]
        first = c.fold_step(*x)
        outs = [torch.empty_like(first) for _ in range(50)]
        for _ in range(8):
            for out in outs:
                c.set_len(prefix)
                c.fold_step(*x, out=out)
            assert all(torch.equal(first, out) for out in outs)
        assert c.status() == binding.KVF_OK
