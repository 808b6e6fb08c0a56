"""The hand-off of work items between the warps of a forward block (forward_loop
in forward.cu), played through with the slots and the order that the source
has.  Thread 0 may be ahead of every other warp up to the next barrier: a late
warp makes its reads of an interval only after thread 0 has made all of its
writes of that interval, and must still find its own item."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_02350_gb300", "csrc", "forward.cu")


def _protocol():
    """(first slot written, first slot read, start of par, write before the barrier) for records and fields."""
    src = open(SRC).read()
    loop = src[src.index("void forward_loop("):src.index("#define SERBF_FWD_BOUNDS")]
    names = {k: int(v) for k, v in re.findall(r"constexpr int (\w+) = (\d+);", loop)}
    value = lambda expr: eval(expr, {}, names)
    many = loop[loop.index("} else {", loop.index("if constexpr (G == 1)")):]  # several warps
    barrier = many.index("__syncthreads();")
    out = []
    for name, first in (("s_rec", r"s_rec\[(\w+)\] = resolve\(a1"), ("s_field", r"s_field\[(\w+)\] = f;")):
        head = loop[:loop.index("while (rec.x")]
        store = value(re.search(first, head).group(1))
        load = value(re.search(r"= (?:BATCH \? )?%s\[(\w+)\]" % name, head[head.index("__syncthreads();"):]).group(1))
        at = many.index("%s[par] = " % name)
        assert many.index("= %s[par]" % name if name == "s_rec" else "field = s_field[par]") > barrier
        out.append((store, load, value(re.search(r"int par = ([^;]+);", head).group(1)), at < barrier))
    return out


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("items", [1, 2, 3, 7])
def test_a_late_warp_finds_its_own_items(which, items):
    store, load, par, before = _protocol()[which]
    slot = [None, None]
    slot[store] = 0                      # thread 0, then the first barrier
    taken, late, read = [], load, load   # late: the slot the late warps have yet to read
    for k in range(items):
        if before:                       # thread 0 stores the next record, then waits at the barrier
            slot[par] = k + 1
        taken.append(slot[late])         # the late warps catch up: their read of item k
        if not before:
            slot[par] = k + 1
        late = par                       # past the barrier: the next record is read here
        par ^= 1
    assert taken == list(range(items))
