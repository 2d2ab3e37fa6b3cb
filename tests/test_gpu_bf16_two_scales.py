"""BF16 sums of a thread whose first vectors are large and whose later values are
tiny: nothing of the later values is lost beside what the first ones left.

The first tile holds values of two sizes, multiples of 2^-21 whose running sums
stay below 8, so a thread's FP32 sum of them is exact; every later value is
2^-42, fewer than 2^13 to a packed lane, so that a thread's two-word sum holds all of
them exactly.  What is left are the at most 1,024 additions of pairs that merge a CTA's
threads (two lanes each), every one rounded below 2^-37 while the sums stay below 2^12."""
import math

import numpy as np
import pytest

from paper_2608_15764_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TILE = 1 << 15        # bytes of a tile of every point below
TILES = 64
LATER = 2.0 ** -42
BOUND = 1024 * 2.0 ** -37
POINTS = [("ldg", dict(k=16, cta=128)), ("ldg", dict(k=8, cta=256)), ("ldg", dict(k=4, cta=512)),
          ("ldg", dict(k=8, cta=256, order="desc")), ("ldg", dict(k=8, cta=256, order="dyn")),
          ("ldg32", dict(k=4, cta=256)), ("ldg32", dict(k=4, cta=256, order="dyn")),
          ("cpasync", dict(k=2, copies=8, cta=128)), ("cpasync", dict(k=2, copies=8, cta=128, order="dyn"))]


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_15764_gb300 as sl
    sl.load()
    return sl


def _payload(every, last=False):
    """Codes, exact sum, and the sum of the later values; a large tile every
    ``every`` tiles (the last tile instead of the first: ``last``)."""
    rng = np.random.default_rng(3)
    vals = np.full((TILES, TILE // 16, 4, 2), LATER)
    large = np.zeros(TILES, bool)
    large[::every] = True
    if last:
        large = large[::-1]
    shape = (int(large.sum()), TILE // 16, 4, 2)
    x = 1.0 + rng.integers(0, 128, shape) / 128.0
    x[:, :, 1::2] *= 2.0 ** -14
    x[:, :, 2] = -x[:, :, 0] + rng.integers(-1, 2, x[:, :, 0].shape) / 128.0  # a vector's large values nearly cancel
    x[:, :, 2] = np.clip(x[:, :, 2], -1.9921875, -1.0)
    vals[large] = x
    codes = workloads.f32_to_bf16(vals.astype(np.float32).ravel())
    assert np.array_equal(workloads.bf16_as_f32_bits(codes).astype(np.float64), vals.ravel())
    later = LATER * 8.0 * (TILE // 16) * int((~large).sum())
    return codes, math.fsum(vals[large].ravel().tolist() + [later]), later


@pytest.mark.parametrize("mech,kw", POINTS)
def test_later_values_are_not_lost(sl, mech, kw):
    codes, ref, later = _payload(TILES, last=kw.get("order") == "desc")
    dev = torch.from_numpy(codes.view(np.uint8).copy()).cuda()
    r = sl.sl_run(dev, dtype=sl.SL_BF16, cfg=sl.config(mech, grid=1, **kw))
    assert abs(r.fsum - ref) <= BOUND < later / 16


def test_later_values_are_not_lost_in_a_batch(sl):
    """One CTA; items of at most eight tiles, each starting with a large one."""
    codes, ref, later = _payload(8)
    dev = torch.from_numpy(codes.view(np.uint8).copy()).cuda()
    b = sl.sl_batch_create([(dev, dev.numel(), sl.SL_BF16)],
                           [sl.tune_entry(0, 1 << 62, sl.config("ldg", k=8, cta=256, grid=1))])
    r = sl.sl_batch_run(b)[0][0]
    sl.sl_batch_destroy(b)
    assert abs(r.fsum - ref) <= TILES // 8 * BOUND < later / 2
