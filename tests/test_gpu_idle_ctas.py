"""Launches with more CTAs than tiles: CTAs without a tile leave at once and
the last of the others combines, around one tile per CTA, one tile in all and
one tile less or more than the grid, alone and in back-to-back passes."""
import numpy as np
import pytest

import oracle
from paper_2608_15764_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LARGEST = 4 << 20
# (mechanism, configuration, bytes of a tile, tiles a CTA takes at a time)
POINTS = [("ldg", dict(k=2, cta=32), 1024, 1), ("ldg", dict(k=2, cta=256, order="desc"), 8192, 1),
          ("ldg", dict(k=3, cta=128, order="dyn"), 6144, 1), ("ldg32", dict(k=1, cta=128), 4096, 1),
          ("ldg4", dict(k=4, cta=256), 4096, 1), ("cpasync", dict(k=2, cta=128), 4096, 1),
          ("cpasync", dict(k=2, copies=2, cta=128, order="dyn"), 8192, 1), ("ldsts", dict(k=2, cta=128), 4096, 1),
          ("tma", dict(cta=128, stage_bytes=4096, stages=2), 4096, 1),
          ("tma", dict(cta=128, stage_bytes=4096, stages=4, ring="warp"), 4096, 4)]


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    sl.load()
    return sl


@pytest.fixture(scope="module")
def data(sl):
    dev = torch.empty(LARGEST, dtype=torch.uint8, device="cuda")
    sl.sl_fill_splitmix64(dev, seed=1)
    return dev, workloads.splitmix_u32(1, LARGEST // 4)


@pytest.mark.parametrize("mech,kw,tile,per", POINTS)
@pytest.mark.parametrize("grid", [1, 2, 33, 200])
def test_more_ctas_than_tiles(sl, data, mech, kw, tile, per, grid):
    dev, host = data
    sizes = {16, tile, tile + 16, grid * per * tile - 16, grid * per * tile, grid * per * tile + 16}
    for nbytes in sorted(b for b in sizes if b <= LARGEST):
        want = oracle.checksum(host[: nbytes // 4])
        for _ in range(2):  # the counters are left clean for the next launch
            r = sl.sl_run(dev, nbytes=nbytes, dtype=sl.SL_U32, cfg=sl.config(mech, grid=grid, **kw))
            assert (r.sum_u32, r.xor_u64, r.grid, r.status) == (*want, grid, 0), nbytes
            assert r.window_ns > 0


@pytest.mark.parametrize("mech,kw,tile,per", POINTS)
def test_idle_ctas_in_overlapped_passes(sl, data, mech, kw, tile, per):
    dev, host = data
    n = 6
    out = torch.zeros(n * sl.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    for nbytes in (16, tile + 16, 20 * tile + 16):
        want = oracle.checksum(host[: nbytes // 4])
        sl.sl_enqueue_steps(dev, out, n, nbytes=nbytes, dtype=sl.SL_U32, cfg=sl.config(mech, **kw))
        raw = out.cpu().numpy().tobytes()
        for i in range(n):
            r = sl.sl_result.from_buffer_copy(raw[i * sl.RESULT_BYTES:(i + 1) * sl.RESULT_BYTES])
            assert (r.sum_u32, r.xor_u64, r.status) == (*want, 0), (nbytes, i)


@pytest.mark.parametrize("dtype", [workloads.F32, workloads.BF16, workloads.FP8_E4M3])
def test_noalloc_with_idle_ctas(sl, dtype):
    for nvec in (1, 257, 1025, 40_000):
        x = workloads.payload(dtype, nvec * 16 // workloads.ELEM_BYTES[dtype])
        ref, _ = oracle.fsum(dtype, x)
        dev = torch.from_numpy(x.view(np.uint8).copy()).cuda()
        out = torch.zeros(sl.RESULT_BYTES, dtype=torch.uint8, device="cuda")
        for _ in range(2):
            sl.sl_run_noalloc(dev, out, dtype=dtype, cfg=sl.config("ldg", k=4, cta=256))
            r = sl.sl_result.from_buffer_copy(out.cpu().numpy().tobytes())
            assert (r.sum_u32, r.xor_u64) == oracle.checksum(x.view(np.uint32))
            assert r.issued_loads == nvec
            absum = float(np.abs(_values(dtype, x)).sum())
            assert abs(r.fsum - ref) <= 2e-6 * absum


def _values(dtype, x):
    if dtype == workloads.F32:
        return x.astype(np.float64)
    if dtype == workloads.BF16:
        return workloads.bf16_as_f32_bits(x).astype(np.float64)
    return torch.from_numpy(x.copy()).view(torch.float8_e4m3fn).to(torch.float32).numpy().astype(np.float64)
