"""Short steps on quantised rows (at most 16 query rows: the decode kernel) over the range of bf16: rows and query elements that
differ by many powers of two, rows that a query must not see.  Against the oracle's fold on code * scale.

RoPE is switched off (frequencies of zero), so that queries reach the kernel as given.  Bound per element, with A = sum p |v| / l (the
oracle's fold of |v|): a product of probability and scale is rounded once to fp16 (2^-11 of it; 2^-25 where the row's largest is
2^14 or more, 127 codes, a few thousand keys: below 2^-20 of the row's largest A), the rest is fp32 (scores of up to ~60 in log2
units: 2^-16)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_12471_b200 import binding
from tests.chain import to_f64

pytestmark = pytest.mark.gpu

D, KV = 128, 2
FLAGS = {8: binding.KVF_CACHE_INT8, 4: binding.KVF_CACHE_INT4}
BITS = pytest.mark.parametrize("bits", [8, 4], ids=["int8", "int4"])
# (query heads per KV head, tokens): one block of query rows (up to 8) and two
SHAPES = pytest.mark.parametrize("group,n", [(4, 1), (4, 2), (4, 3), (4, 4), (1, 16), (7, 2)])


def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen)


def _cache(bits, group, capacity):
    cfg = binding.make_config(KV * group, KV, D, "bf16", capacity, capacity, inv_freq=np.zeros(D // 2), flags=FLAGS[bits] | binding.KVF_OUT_F32)
    return binding.Cache(cfg)


def _oracle(bits, group, capacity):
    c = oracle.OracleCache(KV * group, KV, D, capacity, inv_freq_table=np.zeros(D // 2))
    c.set_quant(bits)
    c.set_unrounded(True)
    return c


def _close(got, want, mean_abs):
    bound = 2.0 ** -11 * 1.1 * mean_abs + 2.0 ** -20 * mean_abs.max(-1, keepdims=True)
    assert np.isfinite(got).all() and (np.abs(got - want) <= bound).all(), float((np.abs(got - want) / bound).max())


def _check(bits, group, prefix, chunk):
    """Folds `prefix` (q, k, v) as one chunk, then `chunk` as the step under test."""
    total = chunk[0].shape[0] + (prefix[0].shape[0] if prefix else 0)
    steps = [[x.bfloat16() for x in s] for s in ([prefix] if prefix else []) + [chunk]]
    c, oc, oa = _cache(bits, group, total + 200), _oracle(bits, group, total), _oracle(bits, group, total)
    c.storage.fill_(0x5A)
    for q, k, v in steps[:-1]:
        c.fold_step(q.cuda(), k.cuda(), v.cuda())
        for o, w in ((oc, v), (oa, v.abs())):
            o.fold_step(to_f64(q), to_f64(k), to_f64(w), rows=[])
    q, k, v = steps[-1]
    lse = torch.empty(q.shape[:2], device="cuda")
    got = to_f64(c.fold_step(q.cuda(), k.cuda(), v.cuda(), lse=lse))
    want, want_lse, _ = oc.fold_step(to_f64(q), to_f64(k), to_f64(v), want_stats=True)
    _close(got, want, oa.fold_step(to_f64(q), to_f64(k), to_f64(v.abs())))
    assert np.abs(to_f64(lse) - want_lse).max() <= 1e-4 * (1 + np.abs(want_lse).max())
    assert c.status() == binding.KVF_OK


@BITS
@SHAPES
@pytest.mark.parametrize("prefix", [0, 70, 700])
def test_rows_later_in_the_chunk_do_not_reach_earlier_tokens(bits, group, n, prefix):
    gen = torch.Generator().manual_seed(prefix + n)
    chunk = [_normal(gen, n, h, D) for h in (KV * group, KV, KV)]
    chunk[2] *= 2.0 ** (45 * torch.arange(n).clamp(max=2)).view(n, 1, 1)       # 1, 2^45, 2^90, 2^90 ...
    _check(bits, group, [_normal(gen, prefix, h, D) for h in (KV * group, KV, KV)] if prefix else None, chunk)


@BITS
@pytest.mark.parametrize("held", [1, 63, 64, 130])
def test_rows_behind_the_length_do_not_reach_attend(bits, held):
    gen = torch.Generator().manual_seed(held)
    group, total = 4, held + 300
    x = [_normal(gen, total, h, D) for h in (KV * group, KV, KV)]
    x[2][held:] *= 2.0 ** 60
    x = [t.bfloat16() for t in x]
    c, oc, oa = _cache(bits, group, total), _oracle(bits, group, total), _oracle(bits, group, total)
    c.fold_step(*(t.cuda() for t in x))
    c.set_len(held)
    got = to_f64(c.attend(x[0][held - 1:held].cuda()))
    q, k, v = (to_f64(t[:held]) for t in x)
    want, mean_abs = (o.fold_step(q, k, w, rows=[held - 1]) for o, w in ((oc, v), (oa, np.abs(v))))
    _close(got, want, mean_abs)
    assert c.status() == binding.KVF_OK


@BITS
@SHAPES
@pytest.mark.parametrize("order", ["growing", "shrinking", "mixed"])
def test_values_of_very_different_size_that_weigh_the_same(bits, group, n, order):
    """Row i of size 2^e_i, e_i from -40 to 40 within and across key tiles; scores make up for it (or add to it) in some heads."""
    gen = torch.Generator().manual_seed(n)
    prefix = 2500
    rows = prefix + n
    e = torch.linspace(-40, 40, rows).round()
    e = {"growing": e, "shrinking": e.flip(0), "mixed": e[torch.randperm(rows, generator=gen)]}[order].view(rows, 1, 1)
    k = torch.zeros(rows, KV, D)
    k[:, :, :1] = -e * np.log(2.0) * D ** 0.5 / 8
    v = _normal(gen, rows, KV, D) * 2.0 ** e
    q = _normal(gen, rows, KV * group, D)
    q[:, :, 0] = torch.tensor([8.0, 4.0, 16.0, -8.0])[torch.arange(KV * group) % 4]
    x = (q, k, v)
    _check(bits, group, [t[:prefix] for t in x], [t[prefix:] for t in x])


@BITS
@SHAPES
def test_a_large_value_row_that_hardly_counts(bits, group, n):
    gen = torch.Generator().manual_seed(11)
    prefix = 600
    q, k, v = (_normal(gen, prefix + n, h, D) for h in (KV * group, KV, KV))
    q[:, :, 0], k[:, :, 0] = 32.0, 0.0
    for row in (3, 200, 599):                      # scores ~85 below the others: probabilities of 2^-120
        k[row, :, 0] = -30.0
        v[row] *= 2.0 ** 45
    x = (q, k, v)
    _check(bits, group, [t[:prefix] for t in x], [t[prefix:] for t in x])


@BITS
@SHAPES
@pytest.mark.parametrize("large,small", [(2.0 ** 45, 1.0), (2.0 ** 33, 1.0), (2.0 ** 100, 2.0 ** 60), (1.0, 2.0 ** -50)])
def test_queries_with_one_large_element(bits, group, n, large, small):
    """... where the keys have a zero: the scores come from the small elements alone."""
    gen = torch.Generator().manual_seed(12)
    prefix = 300
    q, k, v = (_normal(gen, prefix + n, h, D) for h in (KV * group, KV, KV))
    q *= small
    k /= small
    q[:, ::2, 5] = large
    k[:, :, 5] = 0.0
    x = (q, k, v)
    _check(bits, group, [t[:prefix] for t in x], [t[prefix:] for t in x])


@BITS
@SHAPES
def test_ordinary_rows(bits, group, n):
    """The value seen is code * scale, not that rounded to bf16: a token that sees one or two rows shows the difference."""
    gen = torch.Generator().manual_seed(13)
    for prefix in (0, 1, 900):
        x = [_normal(gen, prefix + n, h, D) for h in (KV * group, KV, KV)]
        _check(bits, group, [t[:prefix] for t in x] if prefix else None, [t[prefix:] for t in x])


@BITS
def test_empty_values_and_scores_that_rise(bits):
    """Rows of zeros (scale 0) first, then rows whose scores and sizes rise by powers of two from tile to tile."""
    gen = torch.Generator().manual_seed(14)
    group, n, prefix = 4, 2, 2000
    q, k, v = (_normal(gen, prefix + n, h, D) for h in (KV * group, KV, KV))
    q[:, :, 0] = 16.0
    k[:, :, 0] = torch.linspace(-20, 20, prefix + n).view(-1, 1)
    v *= 2.0 ** torch.linspace(-30, 10, prefix + n).round().view(-1, 1, 1)
    v[:1000] = 0.0
    x = (q, k, v)
    _check(bits, group, [t[:prefix] for t in x], [t[prefix:] for t in x])
    _check(bits, group, [t[:900] for t in x], [t[900:900 + n] for t in x])
