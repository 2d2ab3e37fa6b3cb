"""Rings of shared words that a CTA's loop rewrites while its warps run on: no
word is written between the two barriers between which another warp may still
be reading it.

The loops are read from the kernel sources.  What stands after the body's
barrier falls into the same interval between barriers as what stands before it
in the next iteration."""
import os
import re

import pytest

from paper_2608_15764_gb300 import build

LOOPS = [("k_batch.cuh", "for (uint32_t j = 0;; ++j)", ("vidx", "slot", "wp")),
         ("k_cpasync_dyn.cu", "for (uint32_t it = 0; clen; ++it)", ("vs",)),
         ("k_ldg.cuh", "for (uint32_t j = 0; cur < total; ++j)", ("vslot",)),
         ("k_ldg32.cu", "for (uint32_t j = 0; cur < total; ++j)", ("vslot",))]


def _body(name, head):
    with open(os.path.join(build.CSRC, name), encoding="utf-8") as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    assert text.count(head) == 1
    begin = at = text.index("{", text.index(head))
    depth = 0
    while True:
        depth += {"{": 1, "}": -1}.get(text[at], 0)
        at += 1
        if depth == 0:
            return text[begin:at]


def _accesses(body, ring):
    """(index expression, is a write, stands after the barrier) of each access."""
    assert body.count("__syncthreads()") == 1
    barrier = body.index("__syncthreads()")
    out = []
    for m in re.finditer(r"\b%s\[([^][]*)\]" % ring, body):
        copied_to = body[:m.start()].endswith("smem_addr(&")
        assigned = re.match(r"(\[[^;=]*\])?\s*=(?!=)", body[m.end():]) is not None
        out.append((m.group(1), copied_to or assigned, m.start() > barrier))
    return out


@pytest.mark.parametrize("name,head,rings", LOOPS)
def test_no_word_is_written_while_it_may_be_read(name, head, rings):
    var = re.search(r"uint32_t (\w+) = 0;", head).group(1)
    body = _body(name, head)
    for ring in rings:
        found = _accesses(body, ring)
        reads, writes = set(), set()
        for index, write, after in found:
            for i in range(24):
                if write:
                    writes.add((i + after, eval(index, {var: i})))
                elif after:  # (what stands before the barrier is read back by its own writer)
                    reads.add((i + 1, eval(index, {var: i})))
        assert reads and writes, found
        assert not reads & writes, f"{name}: (interval, word) of {ring} both written and read"
