"""More row pairs than a grid's y has room for: 262 144 queries of 64 heads on one KV head are 65 536 pairs of 128-row
tiles.  Queries only (kvf_attend) against 200 rows, so the work is small; sampled tokens against fp32 attention over the
rotated rows the cache holds."""
import math

import pytest
import torch

from paper_2605_12471_b200 import binding

pytestmark = pytest.mark.gpu


def test_more_row_pairs_than_a_grid_has_in_y():
    n, h, d, held = 262144, 64, 128, 200
    gen = torch.Generator(device="cuda").manual_seed(11)
    c = binding.Cache(binding.make_config(h, 1, d, "bf16", n, n, rope_base=10000.0))
    q, k, v = (torch.randn(held, x, d, generator=gen, device="cuda", dtype=torch.bfloat16) for x in (h, 1, 1))
    c.fold_step(q, k, v)
    q = torch.empty(n, h, d, device="cuda", dtype=torch.bfloat16).normal_(generator=gen)
    out = c.attend(q, pos0=held)
    assert c.status() == binding.KVF_OK and len(c) == held
    keys, values = c.k_plane()[0, :held].float(), c.v_plane()[0, :held].float()
    toks = torch.tensor([0, 1, 3, 4, 131071, 262139, 262140, 262143], device="cuda")
    theta = (held + toks.double())[:, None, None] * 10000.0 ** (-2.0 * torch.arange(d // 2, device="cuda", dtype=torch.float64) / d)
    lo, hi = q[toks].double().split(d // 2, dim=-1)
    rot = torch.cat([lo * theta.cos() - hi * theta.sin(), hi * theta.cos() + lo * theta.sin()], dim=-1).bfloat16().float()
    p = torch.softmax(rot @ keys.T / math.sqrt(d), dim=-1)
    want = p @ values
    # probabilities and outputs are rounded to bf16 (2^-8 of each: of sum p |v| and of |out|); a query element may round
    # the other way from 64-bit angles (2^-8 of one of 128 terms of a score: 2e-3 of an output of unit size)
    bound = 2.0 ** -8 * (p @ values.abs() + want.abs()) + 2e-3
    assert ((out[toks].float() - want).abs() <= bound).all()
