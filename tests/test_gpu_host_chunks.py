"""The staged host-buffer form around the size at which the payload is cut
into chunks, and with a ragged last chunk."""
import numpy as np
import pytest

import oracle
from paper_2608_15764_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MIB = 1 << 20
ONE = 64 * MIB  # up to here: one piece


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    sl.load()
    return sl


@pytest.fixture(scope="module")
def host():
    t = torch.empty(300 * MIB, dtype=torch.uint8).pin_memory()
    a = t.numpy().view(np.uint32)
    workloads.splitmix_u32(1, a.size, out=a)
    return t, a


@pytest.mark.parametrize("mech,kw", [("ldg", dict(k=4, cta=512, order="dyn")), ("ldg", dict(k=2, cta=256)),
                                     ("ldg32", dict(k=2, cta=256, order="dyn")), ("ldg4", dict(k=8, cta=256)),
                                     ("cpasync", dict(k=2, copies=8, cta=256, order="dyn")),
                                     ("tma", dict(cta=256, stage_bytes=16384, stages=4))])
@pytest.mark.parametrize("nbytes", [0, 16, MIB + 48, ONE - 16, ONE, ONE + 16, 4 * ONE + 16 * 5, 300 * MIB - 16])
def test_staged_sizes(sl, host, mech, kw, nbytes):
    t, a = host
    want = oracle.checksum(a[: nbytes // 4]) if nbytes else (0, 0)
    unit = {"ldg32": 32, "ldg4": 4}.get(mech, 16)
    for passes in (1, 2):
        r = sl.sl_run_host(t, nbytes=nbytes, dtype=sl.SL_U32, cfg=sl.config(mech, passes=passes, **kw))
        assert (r.sum_u32, r.xor_u64) == ((passes * want[0]) & 0xFFFFFFFF, want[1] if passes & 1 else 0)
        assert r.issued_loads == passes * (-(-nbytes // unit)) and r.status == 0


@pytest.mark.parametrize("nbytes", [ONE, ONE + 16])
def test_staged_float(sl, nbytes):
    x = workloads.payload(workloads.F32, nbytes // 4)
    ref, _ = oracle.fsum(workloads.F32, x)
    t = torch.from_numpy(x).pin_memory()
    r = sl.sl_run_host(t, dtype=sl.SL_F32, cfg=sl.config("ldg", k=8, cta=256))
    assert abs(r.fsum - ref) <= 2e-6 * float(np.abs(x.astype(np.float64)).sum())
    assert (r.sum_u32, r.xor_u64) == oracle.checksum(x.view(np.uint32))
