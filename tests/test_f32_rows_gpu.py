"""fp32 caches on the tensor cores, with running maxima that move at most steps: against the CUDA-core kernel on the same rows.

Operands are split into two fp16 halves (22 bits; what is below 2^-3 to an absolute 2^-25), so a score is off by at most
3 * 2^-22 of |q| |k| scale (two roundings and the dropped small term, Cauchy) plus fp32 sums, 2^-22 of the same: e = 2^-20 |q| |k|
scale.  The same for a log-sum-exp; an output element by 2 e sum p |v| plus 2^-20 of it for the split of p and v, and for
small values and small probabilities (whose sum is 1 or more before they are normalised) 2^-25 (1 + sum |v|)."""
import pytest
import torch

from paper_2605_12471_b200 import binding

pytestmark = pytest.mark.gpu


def _run(h, kv, prefix, n, splits, window, gen):
    rows = prefix + n
    q, k, v = (torch.randn(rows, heads, 128, generator=gen, device="cuda") for heads in (h, kv, kv))
    k *= torch.linspace(0.1, 8.0, rows, device="cuda")[:, None, None]       # the reference moves by more than its threshold

    def fold(flags, values, splits=0):
        c = binding.Cache(binding.make_config(h, kv, 128, "f32", rows, rows, rope_base=10000.0, flags=flags))
        c.storage.zero_()
        if prefix:
            c.fold_step(q[:prefix].contiguous(), k[:prefix].contiguous(), values[:prefix].contiguous())
        if window:
            c.set_window(4, window)
        c.set_splits(splits)
        lse = torch.empty(n, h, device="cuda")
        out = c.fold_step(q[prefix:].contiguous(), k[prefix:].contiguous(), values[prefix:].contiguous(), lse=lse)
        assert c.status() == binding.KVF_OK
        return out, lse, c.plan(n, prefix)

    a, la, plan = fold(0, v, splits)
    b, lb, _ = fold(binding.KVF_FORCE_SIMT, v)
    weight, _, _ = fold(binding.KVF_FORCE_SIMT, v.abs())
    e = 2.0 ** -20 * (q.norm(dim=-1).max() * k.norm(dim=-1).max()).item() * 128 ** -0.5
    small = 2.0 ** -25 * (1 + v.abs().sum(0)).repeat_interleave(h // kv, dim=0)
    assert ((a - b).abs() <= (2 * e + 2.0 ** -20) * weight + small).all()
    assert (la - lb).abs().max().item() <= e
    return plan


# one step of 64 keys, two, three, many; pairs of row blocks and single ones; padded groups; one to many ranges
@pytest.mark.parametrize("h,kv", [(8, 2), (7, 1)])
@pytest.mark.parametrize("prefix", [0, 1, 63, 129, 700])
def test_moving_maxima(h, kv, prefix):
    gen = torch.Generator(device="cuda").manual_seed(prefix + h)
    for n in (1, 31, 64, 65, 190):
        for splits in (0, 1, 3):
            _run(h, kv, prefix, n, splits, 0, gen)


def test_moving_maxima_under_a_window():
    gen = torch.Generator(device="cuda").manual_seed(5)
    for n in (33, 64):
        _run(8, 2, 900, n, 0, 300, gen)


def test_moving_maxima_in_ranges_that_run_into_the_next_head():
    gen = torch.Generator(device="cuda").manual_seed(6)
    plan = _run(32, 8, 4096, 512, 0, 0, gen)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert plan[2] % (16 * 8) != 0          # nine ranges over eight KV heads
