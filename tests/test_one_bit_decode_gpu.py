"""Decoding one-bit buffers at the ends of the scale's range, on every kernel of the server side: a scale above 2^127
(2s is no finite float), the largest float, a zero scale added to a sum that holds -0.  Against the CPU checker bit for bit."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu

FLT_MAX = np.finfo(np.float32).max
# scales of worker 0 by bucket; the other workers' are small, so that no sum overflows.  Zero in every worker's
# buffer: the sum keeps what it started from.
EDGES = np.array([1e-3, 2e38, FLT_MAX, np.float32(2.0 ** 127), np.nextafter(np.float32(2.0 ** 127), np.float32(np.inf)), 0.0],
                 np.float32)


def _buffers(n, nscales, W, words=None):
    rng = np.random.default_rng(n + W)
    codes = [rng.integers(0, 1 << 32, words or O.code_words(n, 1), dtype=np.uint32) for _ in range(W)]
    scales = [np.full(nscales, 1e-3, np.float32) for _ in range(W)]
    edge = EDGES[(np.arange(nscales) + nscales) % len(EDGES)]
    edge[-1] = FLT_MAX                                     # the bucket of a ragged last row
    scales[0][:] = edge
    for s in scales[1:]:
        s[edge == 0] = 0.0
    return codes, scales, [to_dev(c.view(np.int32)) for c in codes], [to_dev(s) for s in scales]


@pytest.mark.parametrize("n,bucket,W", [
    (1000, 96, 3),                        # direct kernel, buckets inside a warp's elements
    (4000 + 9, 256, 9),                   # direct kernel, a bucket per warp
    (40 * 1024 + 5, 2048, 3),             # bulk-copy kernel with a ragged last row
    (40 * 1024 + 31, 2048, 9),
    ((1 << 25) // 12 + 37, 96, 8),        # row kernel
])
def test_uniform_buckets(n, bucket, W):
    nb = O.num_buckets(n, bucket)
    codes, scales, dc, ds = _buffers(n, nb, W)
    p0 = wl.params(n, 0.05, config=1)
    p_ref, acc_ref = O.server_step(codes, scales, 1, n, bucket, p0.copy(), 0.1, want_acc=True)
    assert np.isfinite(p_ref).all()
    for with_acc in (False, True):
        p, acc = Guarded(n, torch.float32, fill=p0), Guarded(n, torch.float32) if with_acc else None
        mqg.mqg_server_step(dc, ds, W, 1, n, bucket, p.view, 0.1, acc.view if with_acc else None)
        torch.cuda.synchronize()
        p.check_guards()
        assert bits_equal(p.numpy(np.float32), p_ref) == 0
        if with_acc:
            assert bits_equal(acc.numpy(np.float32), acc_ref) == 0
    start = np.where(np.arange(n) % 3 == 0, np.float32(-0.0), p0).astype(np.float32)
    for add in (False, True):
        ref = O.dequant_accumulate(codes, scales, 1, n, bucket, start if add else None)
        acc = Guarded(n, torch.float32, fill=start)
        mqg.mqg_dequant_accumulate(dc, ds, W, 1, n, acc.view, bucket, add_into_acc=add)
        torch.cuda.synchronize()
        acc.check_guards()
        assert bits_equal(acc.numpy(np.float32), ref) == 0, add


@pytest.mark.parametrize("W", [2, 9])
def test_segments(W):
    sizes = [40_008, 100, 70_032, 17, 33_000, 8_191, 50_024, 64]      # bulk copies with ragged rows, and short ones
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    code = np.concatenate([[0], np.cumsum([-(-O.code_words(s, 1) // 4) * 4 for s in sizes])]).astype(np.uint64)
    n = int(seg[-1])
    codes, scales, dc, ds = _buffers(n, len(sizes), W, int(code[-1]))
    p0 = wl.params(n, 0.05, config=3)
    p_ref, acc_ref = O.server_step_segments(codes, scales, 1, seg, code, p0.copy(), 0.1, want_acc=True)
    assert np.isfinite(p_ref).all()
    for with_acc in (False, True):
        p, acc = Guarded(n, torch.float32, fill=p0), Guarded(n, torch.float32) if with_acc else None
        mqg.mqg_server_step_segments(dc, ds, W, 1, seg, code, p.view, 0.1, acc.view if with_acc else None)
        torch.cuda.synchronize()
        p.check_guards()
        assert bits_equal(p.numpy(np.float32), p_ref) == 0
        if with_acc:
            assert bits_equal(acc.numpy(np.float32), acc_ref) == 0


@pytest.mark.parametrize("n,bucket", [(64 * 1024, 2048), (10_001, 96)])
def test_requantize(n, bucket):
    """The downlink's decode half: a mean that is small again although the scales are not."""
    codes, scales, dc, ds = _buffers(n, O.num_buckets(n, bucket), 3)
    c_ref, s_ref = O.server_requantize(codes, scales, 1, n, bucket, 2.0 ** -10, 7)
    c, s = Guarded(O.code_words(n, 1), torch.int32), Guarded(O.num_buckets(n, bucket), torch.float32)
    mqg.mqg_server_requantize(dc, ds, 3, 1, n, bucket, 2.0 ** -10, 7, c.view, s.view)
    torch.cuda.synchronize()
    assert bits_equal(s.numpy(np.float32), s_ref) == 0
    assert np.array_equal(c.numpy(np.uint32), c_ref)
