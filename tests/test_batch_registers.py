"""Registers of the batched form's class kernels, from the compiler's report of
the build: no spills (a kernel with them is refused), enough registers for the
loads in flight, and resident CTAs that the streaming loops need.  The numbers
of CTAs are those of the loops without the item claims and merges around them."""
import glob
import os
import re

import pytest

from paper_2608_15764_gb300 import build

U32, F32, BF16, FP8 = 0, 1, 2, 3


@pytest.fixture(scope="module")
def report():
    build.build()
    out = {}
    for name in glob.glob(os.path.join(build.BUILD, "k_batch*.ptxas.log")):
        with open(name, encoding="utf-8") as f:
            for part in f.read().split("Compiling entry function '")[1:]:
                regs, stack = re.search(r"Used (\d+) registers", part), re.search(r"(\d+) bytes stack frame", part)
                out[part.split("'")[0]] = (int(regs.group(1)), int(stack.group(1)))
    assert out
    return out


def _resident(regs, threads):
    return min(2048 // threads, 32, 65536 // (-(-regs // 8) * 8 * threads))


def _find(report, pattern):
    hits = [v for k, v in report.items() if re.search(pattern, k)]
    assert len(hits) == 1, pattern
    return hits[0]


def test_no_spills_and_room_for_the_loads(report):
    for name, (regs, stack) in report.items():
        assert stack == 0, name
        m = re.search(r"kb_ldg(?:_any)?ILi(\d+)E", name)
        if m:
            assert regs >= 4 * int(m.group(1)) + 14, name


@pytest.mark.parametrize("k,cta,dtype,ctas", [(2, 256, U32, 8), (4, 256, U32, 8), (8, 256, U32, 4), (16, 256, U32, 2),
                                              (4, 512, U32, 4), (8, 512, U32, 2), (8, 128, U32, 9), (1, 256, F32, 6),
                                              (2, 256, F32, 6), (4, 256, F32, 4), (6, 512, F32, 2), (2, 256, BF16, 6),
                                              (3, 256, BF16, 5), (16, 256, BF16, 2), (8, 128, BF16, 6),
                                              (2, 512, FP8, 3), (6, 512, FP8, 2), (12, 128, FP8, 5)])
def test_ldg_classes(report, k, cta, dtype, ctas):
    assert _resident(_find(report, rf"kb_ldgILi{k}ELi{cta}ELi{dtype}E")[0], cta) >= ctas


@pytest.mark.parametrize("d,dtype,ctas", [(4, U32, 8), (6, U32, 8), (8, U32, 8), (4, F32, 8), (6, F32, 5), (1, BF16, 8),
                                          (4, BF16, 6), (6, BF16, 5), (4, FP8, 8), (6, FP8, 6)])
def test_cpasync_classes_of_256_threads(report, d, dtype, ctas):
    assert _resident(_find(report, rf"kb_cpasyncILi{d}ELi{dtype}E")[0], 256) >= ctas
