"""Batches with TMA classes of different ring sizes: classes of one kernel in one
table, larger ring first and last, and a batch run after another was created with
a smaller ring (the kernel's shared-memory limit is shared by all of them)."""
import pytest

import oracle
from paper_2608_15764_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MIB = 1 << 20
RINGS = [(65536, 3), (16384, 2)]


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    sl.load()
    return sl


def _buffers(sizes):
    host = [workloads.splitmix_u32(i + 1, s // 4) for i, s in enumerate(sizes)]
    return [torch.from_numpy(h.view("uint8").copy()).cuda() for h in host], [oracle.checksum(h) for h in host]


def _check(sl, batch, want):
    assert [(r.sum_u32, r.xor_u64, r.status) for r in sl.sl_batch_run(batch)[0]] == [(*w, 0) for w in want]


def _tma(sl, lo, hi, ring):
    return sl.tune_entry(lo, hi, sl.config("tma", cta=256, stage_bytes=ring[0], stages=ring[1]))


@pytest.mark.parametrize("rings", [RINGS, RINGS[::-1]])
def test_two_rings_in_one_table(sl, rings):
    dev, want = _buffers([3 * MIB, 80, 5 * MIB + 16, 2 * MIB, 64 * 1024])
    table = [_tma(sl, 3 * MIB, 1 << 62, rings[0]), _tma(sl, 0, 3 * MIB - 1, rings[1])]
    b = sl.sl_batch_create([(d, d.numel(), sl.SL_U32) for d in dev], table)
    for _ in range(2):
        _check(sl, b, want)
    sl.sl_batch_destroy(b)


def test_a_batch_after_one_with_a_smaller_ring(sl):
    dev, want = _buffers([3 * MIB, MIB + 48])
    made = [sl.sl_batch_create([(d, d.numel(), sl.SL_U32) for d in dev], [_tma(sl, 0, 1 << 62, r)]) for r in RINGS]
    for b in (*made, *made):
        _check(sl, b, want)
    for b in made:
        sl.sl_batch_destroy(b)
