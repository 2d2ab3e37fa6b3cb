"""Work items of the batched form: sizes around an item's unit and around the
numbers of items at which a class gets fewer CTAs than its grid, a second and
later items per CTA, empty buffers among others, and repeated runs (every run
leaves the counters as it found them)."""
import numpy as np
import pytest

import oracle
from paper_2608_15764_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ARENA = 8 << 20
POINTS = [("ldg", dict(k=1, cta=128), 2048), ("ldg", dict(k=16, cta=512), 131072), ("cpasync", dict(k=3, cta=96), 4608),
          ("cpasync", dict(k=8, cta=256), 32768), ("tma", dict(cta=256, stage_bytes=4096, stages=2), 131072),
          ("tma", dict(cta=96, stage_bytes=16384, stages=3), 131072)]


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    sl.load()
    return sl


@pytest.fixture(scope="module")
def arena(sl):
    dev = torch.empty(ARENA, dtype=torch.uint8, device="cuda")
    sl.sl_fill_splitmix64(dev, seed=1)
    return dev, workloads.splitmix_u32(1, ARENA // 4)


@pytest.mark.parametrize("mech,kw,unit", POINTS)
@pytest.mark.parametrize("grid", [0, 1, 3])
def test_item_sizes(sl, arena, mech, kw, unit, grid):
    dev, host = arena
    sizes = [16, 0, unit - 16, unit, unit + 16, 0, 3 * unit + 32, 16, 7 * unit, 2 << 20, 16]
    bufs, spans, off = [], [], 0
    for s in sizes:
        bufs.append((dev[off:off + s], s, sl.SL_U32))
        spans.append((off, s))
        off += s
    assert off <= ARENA
    b = sl.sl_batch_create(bufs, [sl.tune_entry(0, 1 << 62, sl.config(mech, grid=grid, **kw))])
    for _ in range(3):
        res, _ = sl.sl_batch_run(b)
        for (o, s), r in zip(spans, res):
            want = oracle.checksum(host[o // 4:(o + s) // 4]) if s else (0, 0)
            assert (r.sum_u32, r.xor_u64, r.issued_loads, r.status) == (*want, s // 16, 0), (o, s)
        sl.sl_batch_run(b, results=False)
    sl.sl_batch_destroy(b)


@pytest.mark.parametrize("dtype", [workloads.F32, workloads.BF16, workloads.FP8_E4M3])
@pytest.mark.parametrize("mech,kw,unit", POINTS)
def test_item_sums(sl, dtype, mech, kw, unit):
    """Float sums of a buffer cut into many items: within 2e-6 of sum|x|, the
    same in every run."""
    eb = workloads.ELEM_BYTES[dtype]
    sizes = [16, unit + 16, 5 * unit - 16, 3 << 20]
    x = workloads.payload(dtype, sum(sizes) // eb)
    dev = torch.from_numpy(x.view(np.uint8).copy()).cuda()
    bufs, spans, off = [], [], 0
    for s in sizes:
        bufs.append((dev[off:off + s], s, dtype))
        spans.append((off, s))
        off += s
    b = sl.sl_batch_create(bufs, [sl.tune_entry(0, 1 << 62, sl.config(mech, **kw))])
    runs = [[(r.fsum, r.sum_u32, r.xor_u64) for r in sl.sl_batch_run(b)[0]] for _ in range(3)]
    assert runs[0] == runs[1] == runs[2]
    for (o, s), (f, su, xo) in zip(spans, runs[0]):
        part = x[o // eb:(o + s) // eb]
        ref, _ = oracle.fsum(dtype, part)
        if dtype == workloads.F32:
            v = part.astype(np.float64)
        elif dtype == workloads.BF16:
            v = workloads.bf16_as_f32_bits(part).astype(np.float64)
        else:
            v = torch.from_numpy(part.copy()).view(torch.float8_e4m3fn).to(torch.float32).numpy().astype(np.float64)
        assert abs(f - ref) <= 2e-6 * float(np.abs(v).sum())
        assert (su, xo) == oracle.checksum(part.view(np.uint32))
    sl.sl_batch_destroy(b)


@pytest.mark.parametrize("k,cta", [(1, 512), (2, 128), (8, 256), (16, 128)])
@pytest.mark.parametrize("scale", [1, 24])
def test_mixed_types_of_one_entry(sl, k, cta, scale):
    """Four types under one LDG entry: few items (one launch for all types) and
    many (a launch per type); every result as that of its own buffer, in every
    run."""
    unit = k * cta * 16
    kinds = [workloads.U32, workloads.F32, workloads.BF16, workloads.FP8_E4M3]
    bufs, want = [], []
    for i in range(16):
        dt = kinds[i % 4]
        nbytes = [16, unit - 16, unit + 16, 3 * unit * scale, 0][i % 5]
        if dt == workloads.U32:
            x = workloads.splitmix_u32(i + 1, nbytes // 4)
        else:
            x = workloads.payload(dt, nbytes // workloads.ELEM_BYTES[dt], seed=i + 1)
        dev = torch.from_numpy(x.view(np.uint8).copy()).cuda()
        ref = 0.0 if dt == workloads.U32 else oracle.fsum(dt, x)[0] if nbytes else 0.0
        bufs.append((dev, nbytes, dt))
        want.append((*(oracle.checksum(x.view(np.uint32)) if nbytes else (0, 0)), nbytes // 16, ref, nbytes))
    b = sl.sl_batch_create(bufs, [sl.tune_entry(0, 1 << 62, sl.config("ldg", k=k, cta=cta))])
    assert sl.sl_batch_info(b)[0] == 4
    for _ in range(3):
        for r, (s, x, n, f, nbytes) in zip(sl.sl_batch_run(b)[0], want):
            assert (r.sum_u32, r.xor_u64, r.issued_loads, r.status) == (s, x, n, 0)
            assert abs(r.fsum - f) <= 2e-6 * 448.0 * max(nbytes, 1)
            assert abs(r.fsum - f) <= 2e-6 * max(abs(f), 1e-3 * 36.0 * max(nbytes, 1) ** 0.5)
    sl.sl_batch_destroy(b)
