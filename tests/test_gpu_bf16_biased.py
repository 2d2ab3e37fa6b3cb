"""The biased BF16 sum (kernels that fold four or more vectors at a time):
payloads that make a thread take its bias, raise it as the sum grows, give it
up (a value too large, values of mixed sizes, infinities, NaN) or start it on
zeros; against the FP64 oracle and against a kernel that folds by TwoSum."""
import math

import numpy as np
import pytest

import oracle
from paper_2608_15764_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (1 << 19) + 8 * 37  # values: several tiles per thread at a grid of 4, ragged at the end
POINTS = [("ldg", dict(k=4, cta=128)), ("ldg", dict(k=8, cta=256)), ("ldg", dict(k=16, cta=128, order="desc")),
          ("ldg", dict(k=8, cta=256, order="dyn")), ("ldg32", dict(k=2, cta=128)), ("ldg32", dict(k=8, cta=128, order="dyn")),
          ("cpasync", dict(k=2, copies=8, cta=128)), ("cpasync", dict(k=2, copies=8, cta=128, order="dyn"))]


def _bf16(x):
    return workloads.f32_to_bf16(np.asarray(x, dtype=np.float32))


def _payload(kind):
    rng = np.random.default_rng(11)
    x = rng.standard_normal(N)
    if kind == "zeros_then_normal":
        x[: N // 2] = 0.0
    elif kind == "ones":
        x[:] = 1.0
    elif kind == "growing":
        x = np.abs(x) * np.exp2(np.arange(N) * (20.0 / N))
    elif kind == "outliers":
        x[rng.integers(0, N, 40)] *= 1e5
    elif kind == "mixed_sizes":
        x *= np.exp2(rng.integers(-20, 20, N))
    elif kind == "tiny":
        x *= 1e-38
    elif kind == "huge":
        x *= 1e30
    elif kind == "sparse":
        x[rng.random(N) < 0.9] = 0.0
    return _bf16(x)


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    sl.load()
    return sl


@pytest.fixture(scope="module", params=["normal", "zeros_then_normal", "ones", "growing", "outliers", "mixed_sizes",
                                        "tiny", "huge", "sparse"])
def case(request):
    c = _payload(request.param)
    ref, _ = oracle.fsum(workloads.BF16, c)
    absum = float(np.abs(workloads.bf16_as_f32_bits(c).astype(np.float64)).sum())
    return torch.from_numpy(c.view(np.uint8).copy()).cuda(), ref, absum, oracle.checksum(c.view(np.uint32))


@pytest.mark.parametrize("mech,kw", POINTS)
@pytest.mark.parametrize("grid,passes", [(1, 1), (4, 2)])
def test_biased_sum(sl, case, mech, kw, grid, passes):
    """A thread adds fewer than 2^15 values; what Fast2Sum leaves in the error
    sum is below 2^-13 of the largest of them each, and that sum's own rounding
    2^-24 of it: 2^15 * 2^-37 = 2^-22 of sum|x| at the very worst, where every
    value is as large as its bias allows; 1e-9 with the values here."""
    dev, ref, absum, ck = case
    r = sl.sl_run(dev, dtype=sl.SL_BF16, cfg=sl.config(mech, grid=grid, passes=passes, **kw))
    assert abs(r.fsum - passes * ref) <= 1e-9 * passes * absum
    assert r.sum_u32 == (passes * ck[0]) & 0xFFFFFFFF and r.xor_u64 == (ck[1] if passes & 1 else 0)


@pytest.mark.parametrize("cfg", [dict(mech="ldg", k=8, cta=256), dict(mech="tma", cta=256, stage_bytes=16384, stages=2),
                                 dict(mech="tma", cta=96, stage_bytes=16384, stages=3)])
def test_biased_sum_in_a_batch(sl, case, cfg):
    dev, ref, absum, ck = case
    b = sl.sl_batch_create([(dev, dev.numel(), sl.SL_BF16)], [sl.tune_entry(0, 1 << 62, sl.config(grid=2, **cfg))])
    r = sl.sl_batch_run(b)[0][0]
    assert abs(r.fsum - ref) <= 1e-9 * absum and (r.sum_u32, r.xor_u64) == ck
    sl.sl_batch_destroy(b)


@pytest.mark.parametrize("mech,kw", POINTS)
@pytest.mark.parametrize("bad", [0x7F80, 0xFF80, 0x7FC0])
@pytest.mark.parametrize("where", [0, N // 3, N - 1])
def test_infinities_and_nan_as_by_twosum(sl, mech, kw, bad, where):
    c = _payload("normal")
    c[where] = bad
    dev = torch.from_numpy(c.view(np.uint8)).cuda()
    want = sl.sl_run(dev, dtype=sl.SL_BF16, cfg=sl.config("ldg", k=2, cta=256, grid=4)).fsum
    got = sl.sl_run(dev, dtype=sl.SL_BF16, cfg=sl.config(mech, grid=4, **kw)).fsum
    assert math.isnan(want) == math.isnan(got) and (math.isnan(want) or want == got)
