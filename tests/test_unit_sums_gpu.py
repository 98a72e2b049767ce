"""Sums of de-quantized buffers at the ends of the scales that the bulk-copy server kernels and the downlink kernel sum in
units of 2^40: the largest and smallest ones they take, the ones just outside, zero, tiles that hold both kinds, and a
factor (learning rate, mean) that is too large for it.  Against the CPU checker bit for bit."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu

N, BUCKET = 40 * 1024 + 5, 1024         # a tile of 32 rows lies in one bucket; 512 below: in two


def _step_edges(L):
    """Scales whose step s / L is at, just inside and just outside the limits, and far away on either side."""
    lo, hi = np.float32(L * 2.0 ** -86), np.float32(L * 2.0 ** 18)
    near = [np.nextafter(v, np.float32(d)) for v in (lo, hi) for d in (0, np.inf)]
    return np.array([1e-3, lo, hi, *near, 0.0, 2.0 ** -96, 1e30, 3e-5, L * 2.0 ** -86], np.float32)


def _codes(rng, W, bits, n=N):
    return [rng.integers(0, 1 << 32, O.code_words(n, bits), dtype=np.uint32) for _ in range(W)]


def _dev(arrays):
    return [to_dev(a.view(np.int32) if a.dtype == np.uint32 else a) for a in arrays]


def _compare(step, total, ref_step, ref_total, codes, scales, bits, W, bucket, lr):
    dc, ds = _dev(codes), _dev(scales)
    p0 = wl.params(N, 0.05, config=1)
    p, acc = Guarded(N, torch.float32, fill=p0), Guarded(N, torch.float32)
    step(dc, ds, W, bits, N, bucket, p.view, lr)
    total(dc, ds, W, bits, N, acc.view, bucket)
    torch.cuda.synchronize()
    p.check_guards(), acc.check_guards()
    assert bits_equal(p.numpy(np.float32), ref_step(codes, scales, bits, N, bucket, p0.copy(), lr)[0]) == 0
    assert bits_equal(acc.numpy(np.float32), ref_total(codes, scales, bits, N, bucket)) == 0


@pytest.mark.parametrize("bucket,W", [(BUCKET, 3), (512, 9), (BUCKET, 8)])
@pytest.mark.parametrize("bits", range(2, 9))
def test_server(bits, bucket, W):
    rng = np.random.default_rng(bits)
    edges = _step_edges((1 << bits) - 1)
    nb = O.num_buckets(N, bucket)
    scales = [rng.choice(edges[:1] if w % 3 == 2 else edges, nb) for w in range(W)]
    codes = _codes(rng, W, bits)
    for lr in (0.1, 1e26, 2.0 ** -140):
        _compare(mqg.mqg_server_step, mqg.mqg_dequant_accumulate, O.server_step, O.dequant_accumulate, codes, scales, bits, W,
                 bucket, lr)


@pytest.mark.parametrize("bits", range(1, 9))
def test_server_minmax(bits):
    rng = np.random.default_rng(bits)
    W, nb = 5, O.num_buckets(N, BUCKET)
    step = _step_edges((1 << bits) - 1)
    lows = np.array([0.0, -1e-3, 2.0 ** -86, -(2.0 ** -86), 2.0 ** -87, 1e-30, -(2.0 ** 18), 2.0 ** 19, 1e-3], np.float32)
    ranges = []
    for w in range(W):
        lo = rng.choice(lows, nb)
        hi = (lo + rng.choice(step, nb)).astype(np.float32)        # a step that is lost in lo is a constant bucket
        lo[0], hi[0] = -1e-3, 2e-3
        ranges.append(np.stack([lo, hi], 1).reshape(-1))
    _compare(mqg.mqg_server_step_minmax, mqg.mqg_dequant_accumulate_minmax, O.server_step_minmax, O.dequant_accumulate_minmax,
             _codes(rng, W, bits), ranges, bits, W, BUCKET, 0.1)


@pytest.mark.parametrize("bits", range(2, 9))
def test_downlink(bits):
    n, W = 40 * 1024, 5
    rng = np.random.default_rng(bits)
    edges = _step_edges((1 << bits) - 1)
    scales = [rng.choice(edges[:1] if w % 3 == 2 else edges, n // BUCKET) for w in range(W)]
    codes = _codes(rng, W, bits, n)
    for mean in (0.2, 1e-30, 2.0 ** 81):
        c_ref, s_ref = O.server_requantize(codes, scales, bits, n, BUCKET, mean if mean < 1 else 1.0, 7)
        if mean > 1:                     # only small scales: the mean stays finite
            small = [np.minimum(s, np.float32(1e-3)) for s in scales]
            c_ref, s_ref = O.server_requantize(codes, small, bits, n, BUCKET, mean, 7)
        c, s = Guarded(O.code_words(n, bits), torch.int32), Guarded(n // BUCKET, torch.float32)
        mqg.mqg_server_requantize(_dev(codes), _dev(small if mean > 1 else scales), W, bits, n, BUCKET, mean, 7, c.view, s.view)
        torch.cuda.synchronize()
        assert bits_equal(s.numpy(np.float32), s_ref) == 0
        assert np.array_equal(c.numpy(np.uint32), c_ref)
