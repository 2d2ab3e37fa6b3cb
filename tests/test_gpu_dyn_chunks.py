"""The SL_DYN traversal's chunk sizes: from one tile per claim (small buffers,
many CTAs) to the largest chunk, around the sizes where the chunk grows by a
tile, with fewer claims than CTAs, several passes and coverage of every
vector exactly once per pass."""
import numpy as np
import pytest

import oracle
from paper_2608_15764_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LARGEST = (24 << 20) + 16 * 1237
POINTS = [("ldg", dict(k=2, cta=128)), ("ldg", dict(k=12, cta=256)), ("ldg32", dict(k=2, cta=256)),
          ("cpasync", dict(k=4, cta=256)), ("cpasync", dict(k=2, copies=8, cta=128))]


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


def _tile(mech, kw):
    return kw["cta"] * kw["k"] * kw.get("copies", 1) * (32 if mech == "ldg32" else 16)


@pytest.mark.parametrize("mech,kw", POINTS)
@pytest.mark.parametrize("grid", [1, 5, 152, 1000, 3000])
def test_chunk_sizes(sl, data, mech, kw, grid):
    dev, host = data
    tile = _tile(mech, kw)
    edges = {16, tile - 16, tile, tile + 16, 6 * 5 * tile - 16, 12 * 5 * tile, 12 * 5 * tile + 16, LARGEST}
    for nbytes in sorted(b for b in edges if b <= LARGEST):
        s, x = oracle.checksum(host[: nbytes // 4])
        for passes in (1, 3):
            r = sl.sl_run(dev, nbytes=nbytes, dtype=sl.SL_U32,
                          cfg=sl.config(mech, order="dyn", grid=grid, passes=passes, **kw))
            unit = 32 if mech == "ldg32" else 16
            assert (r.sum_u32, r.xor_u64) == ((s * passes) & 0xFFFFFFFF, x), (nbytes, passes)
            assert r.issued_loads == passes * (-(-nbytes // unit)), (nbytes, passes)


@pytest.mark.parametrize("mech,kw", [("ldg", dict(k=2, cta=256)), ("ldg32", dict(k=3, cta=256)),
                                     ("cpasync", dict(k=2, copies=4, cta=256))])
@pytest.mark.parametrize("nbytes", [16 * 5, (1 << 20) + 16, LARGEST])
def test_every_vector_once_per_pass(sl, data, mech, kw, nbytes):
    dev, _ = data
    counts = torch.empty(nbytes // 16, dtype=torch.int32, device="cuda")
    for passes in (1, 2):
        sl.sl_coverage(dev, counts, nbytes=nbytes, cfg=sl.config(mech, order="dyn", passes=passes, **kw))
        got = counts.cpu().numpy()
        assert np.all(got == passes)


def test_many_passes_stay_accepted(sl):
    """Passes whose small chunks would overrun the 32-bit claim counter fall
    back to larger chunks; beyond those the launch is refused."""
    cfg = sl.config("ldg", k=4, cta=256, order="dyn", passes=200_000)
    assert sl.sl_plan(4 << 30, sl.SL_U32, cfg).grid > 0
    cfg.passes = 2_000_000
    with pytest.raises(sl.SLError) as e:
        sl.sl_plan(4 << 30, sl.SL_U32, cfg)
    assert e.value.status == sl.SL_ERR_ARG
