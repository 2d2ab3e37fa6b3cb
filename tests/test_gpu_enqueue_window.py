"""window_ns of launches enqueued back to back covers everything they read, what
they prefetch while the launch before them ends included: a launch in a chain
does the same reads as one on an idle stream, beside another's last ones, so its
window is not the shorter one (two steps of the 32 ns timer allowed)."""
import statistics

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BYTES, NBUF, CHAIN = 48 << 20, 48, 16  # 48 buffers: none is in L2 when its turn comes


@pytest.mark.parametrize("mech,kw", [("cpasync", dict(k=2, copies=8, cta=256)), ("ldg", dict(k=8, cta=256, order="dyn")),
                                     ("tma", dict(cta=256, stage_bytes=16384, stages=4))])
def test_window_of_a_chain(mech, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    arena = torch.zeros(NBUF * BYTES, dtype=torch.uint8, device="cuda")
    bufs = [arena[i * BYTES:(i + 1) * BYTES] for i in range(NBUF)]
    size = sl.RESULT_BYTES
    out = torch.zeros(CHAIN * size, dtype=torch.uint8, device="cuda")
    cfg = sl.config(mech, **kw)

    def windows():
        torch.cuda.synchronize()
        return out.view(torch.int64).view(CHAIN, size // 8)[:, 3].tolist()

    chain, alone = [], []
    for rep in range(3):
        for i in range(CHAIN):
            sl.sl_enqueue(bufs[(rep * CHAIN + i) % NBUF], out[i * size:], dtype=sl.SL_U32, cfg=cfg)
        chain += windows()[1:]
    for i in range(CHAIN):
        sl.sl_enqueue(bufs[i], out, dtype=sl.SL_U32, cfg=cfg)
        alone.append(windows()[0])
    assert statistics.median(chain) >= min(alone) - 64
