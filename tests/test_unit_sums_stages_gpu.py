"""Sums in units of 2^40 where a launch has whole code stages of workers (eight up to four bits, four above), with and without
workers beyond them: the (min, max) update and the downlink at the ends of the scales, tiles whose scales all fit the units next
to tiles with one that does not.  Against the CPU checker bit for bit."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from tests.gpu_util import Guarded, bits_equal
from tests.test_unit_sums_gpu import BUCKET, N, _codes, _compare, _dev

pytestmark = pytest.mark.gpu


def _scales(rng, bits, W, nb):
    """A tile of 32 rows is a bucket (of 1024): all workers' scales inside in every other one, a random worker's outside in the rest."""
    L = (1 << bits) - 1
    lo, hi = np.float32(L * 2.0 ** -85), np.float32(L * 2.0 ** 18)     # twice the smallest half step, half the largest
    inside = np.array([lo, hi, np.nextafter(lo, np.float32(1)), np.nextafter(hi, np.float32(0)), 0.0, 1e-3, 3e-5], np.float32)
    outside = np.array([L * 2.0 ** -87, L * 2.0 ** 20, np.nextafter(np.float32(L * 2.0 ** -86), np.float32(0)), 2.0 ** -96, 1e30],
                       np.float32)
    scales = rng.choice(inside, (W, nb))
    for b in range(1, nb, 2):
        scales[rng.integers(W), b] = rng.choice(outside)
    return scales


@pytest.mark.parametrize("W", [8, 9])
@pytest.mark.parametrize("bits", range(1, 9))
def test_server_minmax(bits, W):
    rng = np.random.default_rng(100 + bits)
    nb = O.num_buckets(N, BUCKET)
    step = _scales(rng, bits, W, nb)
    lows = np.array([0.0, -1e-3, 2.0 ** -85, -(2.0 ** -85), -(2.0 ** 17), 1e-3], np.float32)
    ranges = []
    for w in range(W):
        lo = rng.choice(lows, nb)
        lo[3::4] = rng.choice(np.array([2.0 ** -87, 1e-30, 2.0 ** 19], np.float32), len(lo[3::4]))
        ranges.append(np.stack([lo, (lo + step[w]).astype(np.float32)], 1).reshape(-1))
    codes = _codes(rng, W, bits)
    for lr in (0.1, 2.0 ** 79, 2.0 ** 80):       # the last one is too large for the units
        _compare(mqg.mqg_server_step_minmax, mqg.mqg_dequant_accumulate_minmax, O.server_step_minmax,
                 O.dequant_accumulate_minmax, codes, ranges, bits, W, BUCKET, lr)


@pytest.mark.parametrize("bucket", [1024, 8192, 768])            # CTAs of four, eight and three warps
@pytest.mark.parametrize("W", [8, 9])
@pytest.mark.parametrize("bits", range(2, 9))
def test_downlink(bits, W, bucket):
    n = 48 * bucket
    rng = np.random.default_rng(200 + bits)
    codes, scales = _codes(rng, W, bits, n), list(_scales(rng, bits, W, n // bucket))
    small = [np.minimum(s, np.float32(1e-3)) for s in scales]        # the sum times a large mean stays finite
    dev = _dev(codes)
    for mean, sc in ((0.2, scales), (1e-30, scales), (2.0 ** 79, small), (2.0 ** 81, small)):
        c_ref, s_ref = O.server_requantize(codes, sc, bits, n, bucket, mean, 7)
        c, s = Guarded(O.code_words(n, bits), torch.int32), Guarded(n // bucket, torch.float32)
        mqg.mqg_server_requantize(dev, _dev(sc), W, bits, n, bucket, mean, 7, c.view, s.view)
        torch.cuda.synchronize()
        c.check_guards(), s.check_guards()
        assert bits_equal(s.numpy(np.float32), s_ref) == 0
        assert np.array_equal(c.numpy(np.uint32), c_ref)
