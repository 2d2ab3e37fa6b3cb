"""sl_enqueue on what a dependent launch must treat with care: page-locked host
memory (not prefetched before the wait) that a kernel of the same stream has just
rewritten, and the load flavours, the non-coherent one among them (an ordinary
launch)."""
import pytest

import oracle
from paper_2608_15764_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    sl.load()
    return sl


def _fields(sl, out, n):
    w = out.view(torch.int64).view(n, sl.RESULT_BYTES // 8).cpu()
    sums = out.view(torch.int32).view(n, sl.RESULT_BYTES // 4)[:, 12].cpu()
    return [(int(s) & 0xFFFFFFFF, int(x) & 0xFFFFFFFFFFFFFFFF) for s, x in zip(sums, w[:, 0])]


@pytest.mark.parametrize("where", ["pinned", "device"])
@pytest.mark.parametrize("mech,kw", [("ldg", dict(k=8, cta=256)), ("ldg", dict(k=4, cta=256, order="dyn")),
                                     ("cpasync", dict(k=2, copies=8, cta=256)),
                                     ("tma", dict(cta=256, stage_bytes=65536, stages=2))])
def test_rewritten_between_enqueues(sl, where, mech, kw):
    n, nbytes = 6, (1 << 20) + 16 * 37
    buf = torch.zeros(nbytes, dtype=torch.uint8)
    buf = buf.pin_memory() if where == "pinned" else buf.cuda()
    out = torch.zeros(n * sl.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    cfg = sl.config(mech, **kw)
    for i in range(n):
        sl.sl_fill_splitmix64(buf, seed=i + 1)
        sl.sl_enqueue(buf, out[i * sl.RESULT_BYTES:], dtype=sl.SL_U32, cfg=cfg)
    torch.cuda.synchronize()
    assert _fields(sl, out, n) == [oracle.checksum(workloads.splitmix_u32(i + 1, nbytes // 4)) for i in range(n)]


@pytest.mark.parametrize("cop", [0, 1, 2])
@pytest.mark.parametrize("nbytes", [16, (1 << 20) + 16 * 37, 24 << 20])
def test_load_flavours_in_stream_order(sl, cop, nbytes):
    """The same configuration reads the buffer before and after each rewrite, so
    that its lines have been in every cache."""
    n = 12
    buf = torch.zeros(nbytes // 4, dtype=torch.int32, device="cuda")
    out = torch.zeros(n * sl.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    cfg = sl.config("ldg", k=8, cta=256, cop=cop)
    for i in range(n):
        if i % 2 == 0:
            buf.fill_(i + 1)
        sl.sl_enqueue(buf, out[i * sl.RESULT_BYTES:], dtype=sl.SL_U32, cfg=cfg)
    torch.cuda.synchronize()
    assert [s for s, _ in _fields(sl, out, n)] == [((i // 2 * 2 + 1) * (nbytes // 4)) & 0xFFFFFFFF for i in range(n)]
