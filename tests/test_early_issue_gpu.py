"""bf16 chunks of two row tiles (the early issue of Q K^T): against the CUDA-core kernel on the same rows.

Both read the same bf16 cache (checked bit for bit).  Rounding to bf16 (8 significant bits) is off by at most 2^-8 of a
value: the tensor-core kernel rounds the probabilities, which sum to one, and both round the outputs - together at most
3 * 2^-8 of the largest |v|.  Log-sum-exp differs by fp32 sums of 128 products per score, scores up to ~60 in the
growing case (2^-24 * 60 * 128 = 5e-4)."""
import pytest
import torch

from paper_2605_12471_b200 import binding

pytestmark = pytest.mark.gpu


def _run(prefix, n, splits, growing, gen):
    outs = []
    h, kv = 8, 2
    rows = prefix + n
    q, k, v = (torch.randn(rows, heads, 128, generator=gen, device="cuda") for heads in (h, kv, kv))
    if growing:      # the running maximum moves by more than the rescale threshold in many tiles
        k *= torch.linspace(0.1, 12.0, rows, device="cuda")[:, None, None]
    q, k, v = (x.bfloat16() for x in (q, k, v))
    for flags in (0, binding.KVF_FORCE_SIMT):
        c = binding.Cache(binding.make_config(h, kv, 128, "bf16", rows, rows, rope_base=10000.0, flags=flags))
        c.storage.zero_()
        if prefix:
            c.fold_step(q[:prefix].contiguous(), k[:prefix].contiguous(), v[:prefix].contiguous())
        if not flags:
            c.set_splits(splits)
            assert c.plan(n)[0] == 1
        lse = torch.empty(n, h, device="cuda")
        out = c.fold_step(q[prefix:].contiguous(), k[prefix:].contiguous(), v[prefix:].contiguous(), lse=lse)
        assert c.status() == binding.KVF_OK
        outs.append((out, lse, c.storage.clone()))
    (a, la, sa), (b, lb, sb) = outs
    assert torch.equal(sa, sb)
    assert (a.float() - b.float()).abs().max().item() <= 3 * 2.0 ** -8 * v.float().abs().max().item()
    assert (la - lb).abs().max().item() <= 5e-4


# key tiles of 128 rows: one, two, three, many; the second row tile from one valid row on; one to many ranges
@pytest.mark.parametrize("growing", [False, True], ids=["plain", "growing_maxima"])
@pytest.mark.parametrize("prefix", [0, 1, 127, 129, 1000])
def test_two_row_tiles_against_the_cuda_core_kernel(prefix, growing):
    gen = torch.Generator(device="cuda").manual_seed(prefix + growing)
    for n in (33, 64, 65, 190):
        for splits in (0, 1, 3):
            _run(prefix, n, splits, growing, gen)
