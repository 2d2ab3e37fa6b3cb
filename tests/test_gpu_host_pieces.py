"""The staged host-buffer form around the sizes at which the payload is copied in
one, two, three or four pieces, and in more than a staging buffer holds four of."""
import numpy as np
import pytest

import oracle
from paper_2608_15764_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MIB = 1 << 20


@pytest.mark.parametrize("nbytes", [112 * MIB - 16, 112 * MIB, 112 * MIB + 16, 144 * MIB - 16, 144 * MIB, 192 * MIB + 48,
                                    256 * MIB + 16, 1024 * MIB + 16])
def test_pieces(nbytes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    t = torch.empty(nbytes, dtype=torch.uint8).pin_memory()
    a = t.numpy().view(np.uint32)
    workloads.splitmix_u32(1, a.size, out=a)
    want = oracle.checksum(a)
    for mech, kw, unit in (("ldg", dict(k=4, cta=512, order="dyn"), 16), ("ldg32", dict(k=2, cta=256), 32)):
        r = sl.sl_run_host(t, dtype=sl.SL_U32, cfg=sl.config(mech, **kw))
        assert (r.sum_u32, r.xor_u64, r.issued_loads, r.status) == (*want, -(-nbytes // unit), 0)
