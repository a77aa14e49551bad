"""The two buffers through which the warps of a pivoted Cholesky CTA exchange their pivot candidates
(csrc/gramqr.cu): with one block barrier a step, a buffer may be written again only after a barrier that
follows the last read of it. The kernels' picks, barriers and buffer indexes are read from the source in
their order and played for the first search and a few steps (no GPU needed)."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_11004_gb300", "csrc",
                   "gramqr.cu")


def _body(kernel):
    """Source of the kernel from its first search on, without comments: (before the loop, loop)."""
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    at = re.search(r"\b%s\(const double" % kernel, text).start()
    text = text[text.index("const int steps =", at):text.index("*rank_out = j", at)]
    loop = re.search(r"for \(; go && j < steps; \+\+j\)", text).start()
    return text[:loop], text[loop:]


def _events(text, forced):
    """(write | read, index expression) and barriers, in order."""
    write = r"s_next\[([^\]]+)\] = " if forced else r"\bwarp_pick\(([^)]+)\)"
    read = r"s_next\[([^\]]+)\](?! = )" if forced else r"\bblock_pick\(([^,]+),"
    found = [(m.start(), "barrier", None) for m in re.finditer(r"__syncthreads\(\)", text)]
    found += [(m.start(), "write", m.group(1)) for m in re.finditer(write, text)]
    found += [(m.start(), "read", m.group(1)) for m in re.finditer(read, text)]
    return [e[1:] for e in sorted(found)]


@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("kernel", ["k_pchol_cluster", "k_pchol_grid_reg"])
def test_no_buffer_is_written_before_its_readers_are_past_a_barrier(kernel, forced):
    first, loop = _body(kernel)
    played = [("first search", e, 0) for e in _events(first, forced)]
    for j in range(4):
        played += [("step %d" % j, e, j & 1) for e in _events(loop, forced)]
    kinds = [e[0] for _, e, _ in played]
    assert kinds.count("write") == kinds.count("read") == 5 and kinds.count("barrier") >= 5
    read, written = set(), set()                           # buffers used since the last barrier
    for where, (kind, index), b in played:
        if kind == "barrier":
            read, written = set(), set()
            continue
        buf = eval(index, {"b": b})
        if kind == "write":
            assert buf not in read, "%s writes buffer %d, which other warps may still read" % (where, buf)
            written.add(buf)
        else:
            assert buf not in written, "%s reads buffer %d before a barrier" % (where, buf)
            read.add(buf)
