"""kvf_fold_step_host with uploads ahead and results behind, enqueued without any synchronisation: the bits of the device entry point."""
import pytest
import torch
from cuda.bindings import runtime

from paper_2605_12471_b200 import binding

pytestmark = pytest.mark.gpu

AHEAD, BEHIND = binding.KVF_HOST_UPLOAD_AHEAD, binding.KVF_HOST_DOWNLOAD_BEHIND


def _chain(shape, dtype, chunks, flags, seed):
    """A cache for host steps, pinned inputs of every chunk, and the device entry point's results on the host."""
    h, kv, d = shape
    total, kind = sum(chunks), torch.float32 if dtype == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(seed)
    make = lambda f: binding.Cache(binding.make_config(h, kv, d, dtype, total, max(chunks), rope_base=10000.0, flags=f))
    dev, host = make(0), make(flags)
    ins, want = [], []
    for n in chunks:
        x = [torch.randn(n, heads, d, generator=gen, device="cuda").to(kind) for heads in (h, kv, kv)]
        lse = torch.empty(n, h, device="cuda")
        want.append((dev.fold_step(*x, lse=lse).cpu(), lse.cpu()))
        ins.append([y.cpu().pin_memory() for y in x])
    torch.cuda.synchronize()
    return host, ins, want


def _waits_for(graph, first, second):
    """Does node `second` of a captured graph run behind node `first`?"""
    count = runtime.cudaGraphGetEdges_v2(graph)[4]
    err, begin, end, _, count = runtime.cudaGraphGetEdges_v2(graph, count)
    behind = {}
    for a, b in zip(begin[:count], end[:count]):
        behind.setdefault(int(a), []).append(int(b))
    todo, seen = [int(first)], set()
    while todo:
        x = todo.pop()
        if x not in seen:
            seen.add(x)
            todo += behind.get(x, [])
    return int(second) in seen


# Copies of one direction happen to run one after the other on this GPU; what makes sure of it is read off a captured chain.
@pytest.mark.parametrize("at,lse_at,ordered", [(0, 2, True), (2 * 40 - 1, 2, True), (2 * 40, 2, False), (100, 0, True), (100, 1, True)])
def test_copies_into_the_same_host_memory_are_ordered(at, lse_at, ordered):
    """Two steps (40 and 3 tokens): the second's rows begin at half-row `at` behind the first's begin, its log-sum-exps at block `lse_at`."""
    host, ins, _ = _chain((32, 8, 128), "bf16", [40, 3], BEHIND, 4)
    out, lse = torch.zeros(200 * 32 * 64, dtype=torch.bfloat16).pin_memory(), torch.zeros(4 * 40 * 32).pin_memory()
    half = 32 * 64
    views = [(out[:40 * 2 * half].view(40, 32, 128), lse[:40 * 32].view(40, 32)),
             (out[at * half:(at + 6) * half].view(3, 32, 128), lse[lse_at * 20 * 32:][:3 * 32].view(3, 32))]
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        for x, (o, l) in zip(ins, views):
            host.fold_step_host(*x, o, lse=l)
        host.flush()
    raw = runtime.cudaGraph_t(graph.raw_cuda_graph())
    err, nodes, count = runtime.cudaGraphGetNodes(raw)
    err, nodes, count = runtime.cudaGraphGetNodes(raw, count)
    copies = {}                                  # by their size
    for node in nodes[:count]:
        if runtime.cudaGraphNodeGetType(node)[1] == runtime.cudaGraphNodeType.cudaGraphNodeTypeMemcpy:
            copies[runtime.cudaGraphMemcpyNodeGetParams(node)[1].extent.width] = node
    for x in views[0]:
        for y in views[1]:
            assert _waits_for(raw, copies[x.nbytes], copies[y.nbytes]) == ordered


# a copy of 16 MB beside a step of 1 - 64 tokens: whoever keeps one result buffer has the later call's rows, on top of the earlier one's
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("flags", [BEHIND, BEHIND | AHEAD], ids=["behind", "ahead_and_behind"])
def test_results_of_steps_that_share_a_buffer_come_in_order(flags, offset):
    chunks = [2048, 32, 2048, 1, 64, 2048, 5]
    host, ins, want = _chain((32, 8, 128), "bf16", chunks, flags, 3)
    out, lse = torch.zeros(2048 + 64, 32, 128, dtype=torch.bfloat16), torch.zeros(2048 + 64, 32)
    at = [0 if n == 2048 else offset * (2048 - n // 2) for n in chunks]          # the same rows, or across the end of the large block
    for n, a, (o, l) in zip(chunks, at, want):
        out[a:a + n], lse[a:a + n] = o, l
    got, got_lse = torch.zeros_like(out).pin_memory(), torch.zeros_like(lse).pin_memory()
    for _ in range(20):
        got.zero_()
        got_lse.zero_()
        host.set_len(0)
        for n, a, x in zip(chunks, at, ins):
            host.fold_step_host(*x, got[a:a + n], lse=got_lse[a:a + n])
        host.flush()
        torch.cuda.current_stream().synchronize()
        assert torch.equal(got.view(torch.int16), out.view(torch.int16)) and torch.equal(got_lse, lse)
    assert host.status() == binding.KVF_OK


# Staging sets are written again as soon as their last reader is done: rotate + append, or the one launch of a small step.  Large and
# small steps in turn, so that copies and kernels of several steps lie side by side in every order.
@pytest.mark.parametrize("flags", [AHEAD, BEHIND, AHEAD | BEHIND, AHEAD | BEHIND | binding.KVF_COMBINE_BEHIND],
                         ids=["ahead", "behind", "both", "both_and_merge_behind"])
@pytest.mark.parametrize("shape,dtype,chunks", [
    ((4, 1, 64), "f32", [64] * 6),                                   # one launch each
    ((4, 1, 64), "bf16", [64, 2000, 1, 2000, 300, 64, 64, 1, 1]),    # one launch and three in turn
    ((32, 8, 128), "bf16", [2048, 1, 32, 2048, 3, 2048, 2048, 64, 1, 1]),
    ((32, 8, 128), "f32", [512, 1, 512, 32, 32, 512]),
], ids=["small", "small_and_large", "bf16", "f32"])
def test_host_steps_of_different_size_in_turn(shape, dtype, chunks, flags):
    host, ins, want = _chain(shape, dtype, chunks, flags, 5)
    got = [(torch.zeros_like(o).pin_memory(), torch.zeros_like(l).pin_memory()) for o, l in want]
    for _ in range(5):
        for o, l in got:
            o.zero_()
            l.zero_()
        host.set_len(0)
        for x, (o, l) in zip(ins, got):
            host.fold_step_host(*x, o, lse=l)
        host.flush()
        torch.cuda.current_stream().synchronize()
        for t, ((o, l), (wo, wl)) in enumerate(zip(got, want)):
            assert torch.equal(o, wo) and torch.equal(l, wl), t
    assert host.status() == binding.KVF_OK
