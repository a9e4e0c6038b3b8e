"""Rules of the kernels' mbarrier protocols whose breach could only show as a hang, checked without a GPU.

A wait asks for a phase by its parity, so it is sound only while its thread is never two phases behind the barrier."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_12471_b200", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


# An issuing warp: all lanes wait, one issues, and only what it issues lets the barriers move on.  The other lanes keep up only where a
# vote stands between a wait and the next thing issued.
@pytest.mark.parametrize("name,end", [("attn_tc.cu", "softmax, one thread per row"), ("attn_tc32.cu", "converters: fp32 rows")])
def test_waits_of_issuing_warps_end_in_a_vote(name, end):
    text = _source(name)
    start = text.index("leader = elect_one()")
    lines = text[start:text.index(end, start)].splitlines()
    waits = [i for i, line in enumerate(lines) if re.search(r"\bmbar_wait\w*\(", line) and "mbar_wait_drain(" not in line]
    assert len(waits) >= 4
    for i in waits:
        voted = re.search(r"\bmbar_wait4?_warp\(", lines[i]) or any("__all_sync" in line for line in lines[i:i + 4])
        assert voted, lines[i]
        if not re.search(r"\bmbar_wait4?_warp\(", lines[i]):
            until = next(k for k in range(i, i + 4) if "__all_sync" in lines[k])
            assert not any("leader" in line for line in lines[i:until])


# .aligned instructions want all lanes of a warp together, which only a warp-wide instruction makes sure of behind a branch of some of
# them.  Read down the text of a role; __syncthreads and votes count as much as __syncwarp.
@pytest.mark.parametrize("name", ["attn_tc.cu", "attn_tc32.cu", "fold_small.cu"])
def test_aligned_instructions_stand_behind_a_reconvergence(name):
    apart = None
    for number, line in enumerate(_source(name).splitlines(), 1):
        code = line.split("//")[0]
        if "// -----" in line or "tcgen05.alloc" in code or code.startswith(("__global__", "}")) or code.strip() == "continue;":
            apart = None                         # (another role, warps that the branch before did not hold, a branch that ends here)
        if re.search(r"KVF_TMEM_(LD|ST)\d+\(|\.aligned;|cluster_sync_all\(\)", code):
            assert apart is None, f"{name}:{number}: behind the branch in line {apart}"
        if re.search(r"\b(if|for) \(.*\b(lane == 0|tid == 0|threadIdx\.x == 0|clocked\)|valid\)|gi1? >= a\.G|i = tid;)", code):
            apart = number
        if re.search(r"__syncwarp|__syncthreads|_sync\(0xffffffffu|mbar_wait4?_warp\(", code):
            apart = None
    for kernel in ("attn_tc.cu", "attn_tc32.cu"):          # (the roles begin with setmaxnreg)
        assert re.search(r"ns0 = global_ns\(\);\n    }\n    __syncwarp\(\);", _source(kernel))


class _Overtaken(Exception):
    pass


def _explore(programs, counts):
    """Every interleaving of `programs` (lists of ("wait", barrier, phase) and ("arrive", barrier, weight)): raises if a barrier completes a
    phase while somebody has yet to see the one before it, or if everybody waits for ever."""
    after = []                                   # of each program, at each position: the next wait on a barrier
    for ops in programs:
        table, nxt = [], {}
        for op in reversed(ops):
            if op[0] == "wait":
                nxt = {**nxt, op[1]: op[2]}
            table.append(nxt)
        after.append([{}] + table)
    todo, seen = [(0,) * len(programs)], set()
    while todo:
        at = todo.pop()
        if at in seen:
            continue
        seen.add(at)
        arrived = {}
        for ops, i in zip(programs, at):
            for op in ops[:i]:
                if op[0] == "arrive":
                    arrived[op[1]] = arrived.get(op[1], 0) + op[2]
        done = {b: n // counts[re.sub(r"\d+$", "", b)] for b, n in arrived.items()}
        for p, i in enumerate(at):
            for b, phase in after[p][len(programs[p]) - i].items():
                if done.get(b, 0) > phase + 1:
                    raise _Overtaken(f"program {p} waits for phase {phase} of {b}, which has completed {done[b]}")
        moved = False
        for p, i in enumerate(at):
            if i < len(programs[p]):
                op = programs[p][i]
                if op[0] == "arrive" or done.get(op[1], 0) > op[2]:
                    moved = True
                    todo.append(at[:p] + (i + 1,) + at[p + 1:])
        assert moved or all(i == len(ops) for i, ops in zip(at, programs)), "all wait"
    return len(seen)


def _f32_programs(pieces, output_arrives):
    """The roles of the fp32 tensor-core kernel over pieces of so many steps (the K and V rings left out: each has one writer and one
    reader that wait for one another)."""
    softmax, scores, products, output = [], [], [], []
    g = 0
    for p, steps in enumerate(pieces):
        if p:
            softmax += [("wait", "OFREE", g - 1), ("wait", "QEMPTY", p - 1)]
        softmax.append(("arrive", "QFULL", 4))
        scores.append(("wait", "QFULL", p))
        for j in range(steps):
            buf, use = str(g & 1), g >> 1
            softmax += [("wait", "SFULL", g), ("arrive", "SFREE", 4)]
            softmax += [("wait", "PFREE" + buf, use - 1)] if g > 1 else []
            softmax.append(("arrive", "PFULL" + buf, 4))
            scores += [("wait", "SFREE", g - 1)] if g else []
            scores.append(("arrive", "SFULL", 1))
            products.append(("wait", "PFULL" + buf, use))
            products += [("wait", "OFREE", g - 1)] if g else []
            products += [("arrive", "OFULL", 1), ("arrive", "PFREE" + buf, 1)]
            output.append(("wait", "PFULL" + buf, use))
            output += [("arrive", "PFREE" + buf, 4)] if output_arrives else []
            output.append(("wait", "OFULL", g))
            if j == steps - 1:
                softmax += [("wait", "PFREE" + buf, use), ("arrive", "ROWDONE", 4)]
                output.append(("wait", "ROWDONE", p))
            output.append(("arrive", "OFREE", 4))
            g += 1
        scores.append(("arrive", "QEMPTY", 1))
    return [softmax, scores, products, output]


# ranges that run across KV heads: pieces of one and more steps, whatever the delay of a role
@pytest.mark.parametrize("pieces", [[5], [1, 1, 1, 4], [2, 5], [3, 1, 4]])
def test_no_role_of_the_f32_kernel_falls_two_phases_behind(pieces):
    text = _source("attn_tc32.cu")
    counts = {name: eval(count) for name, count in re.findall(r"mbar_init\(bar\(B_([A-Z]+)0?(?: \+ i)?\), ([\d +]+)\)", text)}
    start = text.index("output rows, one thread per row\n        // The running")
    arrives = "mbar_arrive(bar(B_PFREE0" in text[start:text.index("softmax, one thread per row", start)]
    _explore(_f32_programs(pieces, arrives), counts)
    with pytest.raises(_Overtaken):              # what the output warps' arrival is for
        _explore(_f32_programs(pieces, False), {**counts, "PFREE": 1})


# A cluster whose CTAs store into one another: each arrives once more behind its last store and waits for the others ahead of its end, on
# every way out.
@pytest.mark.parametrize("name,begin", [("attn_tc.cu", "if constexpr (kRanks > 0) {"), ("fold_small.cu", "if (ranks > 1) cluster_wait();")])
def test_no_cta_leaves_a_cluster_that_may_still_store_into_it(name, begin):
    text = re.sub(r"//.*", "", _source(name))
    start = text.index(begin)
    end = text.index("\n}\n", start)
    merge = text[start:end]
    last_store = merge.rindex("peer_store")
    assert merge.index("cluster_wait()") < merge.index("peer_store")                # the partners' barriers exist
    assert last_store < merge.index("cluster_arrive_relaxed()") < merge.rindex("cluster_wait()")
    assert not re.search(r"\breturn;", merge)
