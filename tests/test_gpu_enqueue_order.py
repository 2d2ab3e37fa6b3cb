"""Stream order of sl_enqueue: the load kernel is a programmatic dependent
launch whose CTAs wait for the work before it, so a buffer written by any
earlier kernel on the stream is read complete, a later kernel may overwrite
it, and a captured graph holds plain launches."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

POINTS = [("ldg", dict(k=2, cta=256)), ("ldg", dict(k=8, cta=512, order="desc")), ("ldg", dict(k=4, cta=256, order="dyn")),
          ("ldg32", dict(k=2, cta=256)), ("ldg32", dict(k=2, cta=256, order="dyn")), ("ldg4", dict(k=4, cta=256)),
          ("cpasync", dict(k=4, cta=256)), ("cpasync", dict(k=2, copies=8, cta=256, order="dyn")), ("ldsts", dict(k=4, cta=256)),
          ("tma", dict(cta=256, stage_bytes=16384, stages=4)),
          ("tma", dict(cta=256, stage_bytes=4096, stages=8, ring="warp"))]


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    sl.load()
    return sl


def _sums(sl, out, n):
    return [int(v) & 0xFFFFFFFF for v in out[: n * sl.RESULT_BYTES].view(torch.int32).view(n, sl.RESULT_BYTES // 4)[:, 12].cpu()]


@pytest.mark.parametrize("mech,kw", POINTS)
@pytest.mark.parametrize("nbytes", [16, (1 << 20) + 16 * 37, 48 << 20])
def test_enqueue_reads_what_the_stream_wrote(sl, mech, kw, nbytes):
    """Rewrite the buffer between enqueues, with a kernel of another library
    and with this library's own; every result is that of its own contents."""
    n = 24
    buf = torch.zeros(nbytes // 4, dtype=torch.int32, device="cuda")
    out = torch.zeros(n * sl.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    cfg = sl.config(mech, **kw)
    for i in range(n):
        buf.fill_(i + 1)
        sl.sl_enqueue(buf, out[i * sl.RESULT_BYTES:], dtype=sl.SL_U32, cfg=cfg)
    want = [((i + 1) * (nbytes // 4)) & 0xFFFFFFFF for i in range(n)]
    assert _sums(sl, out, n) == want
    for i in range(n):  # two readers in a row, then a writer
        if i % 2 == 0:
            buf.fill_(i + 3)
        sl.sl_enqueue(buf, out[i * sl.RESULT_BYTES:], dtype=sl.SL_U32, cfg=cfg)
    want = [((i // 2 * 2 + 3) * (nbytes // 4)) & 0xFFFFFFFF for i in range(n)]
    assert _sums(sl, out, n) == want


@pytest.mark.parametrize("mech,kw", [POINTS[0], POINTS[2], POINTS[9]])
def test_enqueue_under_capture(sl, mech, kw):
    nbytes, n = (1 << 20) + 16 * 37, 4
    buf = torch.zeros(nbytes // 4, dtype=torch.int32, device="cuda")
    out = torch.zeros(n * sl.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream()
    cfg = sl.config(mech, stream=stream, **kw)
    with torch.cuda.stream(stream):
        sl.sl_enqueue(buf, out, dtype=sl.SL_U32, cfg=cfg)  # scratch and kernel loaded before the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for i in range(n):
            buf.add_(i + 1)
            sl.sl_enqueue(buf, out[i * sl.RESULT_BYTES:], dtype=sl.SL_U32, cfg=cfg)
    total = 0
    for _ in range(3):
        g.replay()
        torch.cuda.synchronize()
        want = []
        for i in range(n):
            total += i + 1
            want.append((total * (nbytes // 4)) & 0xFFFFFFFF)
        assert _sums(sl, out, n) == want


@pytest.mark.parametrize("passes", [1, 2])
@pytest.mark.parametrize("nbytes", [16, (1 << 20) + 16 * 37])
def test_noalloc_order_and_capture(sl, nbytes, passes):
    """sl_run_noalloc clears its control block and reads the buffer in stream
    order, back to back, between writers, and replayed from a graph."""
    n = 16
    buf = torch.zeros(nbytes // 4, dtype=torch.int32, device="cuda")
    out = torch.zeros(n * sl.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    cfg = sl.config("ldg", k=2, cta=128, passes=passes)
    for i in range(n):
        if i % 2 == 0:
            buf.fill_(i + 1)
        sl.sl_run_noalloc(buf, out[i * sl.RESULT_BYTES:], dtype=sl.SL_U32, cfg=cfg)
    assert _sums(sl, out, n) == [(passes * (i // 2 * 2 + 1) * (nbytes // 4)) & 0xFFFFFFFF for i in range(n)]
    stream = torch.cuda.Stream()
    cfg = sl.config("ldg", k=2, cta=128, passes=passes, stream=stream)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for i in range(2):
            buf.fill_(i + 7)
            sl.sl_run_noalloc(buf, out[i * sl.RESULT_BYTES:], dtype=sl.SL_U32, cfg=cfg)
    for _ in range(3):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert _sums(sl, out, 2) == [(passes * (i + 7) * (nbytes // 4)) & 0xFFFFFFFF for i in range(2)]
