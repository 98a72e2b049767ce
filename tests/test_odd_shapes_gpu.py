"""Shapes outside the bulk-copy kernels: the (min, max) server step on the row kernel, several workers on a CTA per bucket
or a launch per worker, and buckets of an odd number of rows in the variants whose scale is a sum.  Against the CPU
checker bit for bit."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev
from tests.test_server_dispatch_gpu import test_server_step_at_the_dispatch_lines as _step_at_the_lines

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,W,bits", [
    ((1 << 25) // 12 + 37, 8, 3), ((1 << 25) // 12 + 32, 8, 7), ((1 << 25) // 5 + 1, 1, 1), ((1 << 25) // 36 + 31, 32, 8),
    ((27 << 20) // 24, 8, 4), ((27 << 20) // 24 - 1, 8, 4), ((27 << 20) // 17 + 1, 1, 6),      # at the line of the rule
])
def test_range_server_rows(n, W, bits):
    bucket = 96
    rng = np.random.default_rng(n)
    codes = [rng.integers(0, 1 << 32, O.code_words(n, bits), dtype=np.uint32) for _ in range(W)]
    ranges = [np.sort(rng.standard_normal((O.num_buckets(n, bucket), 2), dtype=np.float32) * np.float32(1e-3), axis=1).ravel()
              for _ in range(W)]
    ranges[0][-2:] = 1e-3                                                  # a constant bucket, the ragged one
    dc, dr = [to_dev(c.view(np.int32)) for c in codes], [to_dev(r) for r in ranges]
    p0 = wl.params(n, 0.05, config=21)
    p_ref, acc_ref = O.server_step_minmax(codes, ranges, bits, n, bucket, p0.copy(), 0.1, want_acc=True)
    for with_acc in (False, True):
        p, acc = Guarded(n, torch.float32, fill=p0), Guarded(n, torch.float32) if with_acc else None
        mqg.mqg_server_step_minmax(dc, dr, W, bits, n, bucket, p.view, 0.1, acc.view if with_acc else None)
        torch.cuda.synchronize()
        p.check_guards()
        assert bits_equal(p.numpy(np.float32), p_ref) == 0
        if with_acc:
            acc.check_guards()
            assert bits_equal(acc.numpy(np.float32), acc_ref) == 0
    acc = Guarded(n, torch.float32, fill=p0)
    mqg.mqg_dequant_accumulate_minmax(dc, dr, W, bits, n, acc.view, bucket, add_into_acc=True)
    torch.cuda.synchronize()
    assert bits_equal(acc.numpy(np.float32), O.dequant_accumulate_minmax(codes, ranges, bits, n, bucket, p0)) == 0


@pytest.mark.parametrize("n,bucket,W,bits,with_acc", [
    ((27 << 20) // 24, 96, 8, 3, False), ((27 << 20) // 24 - 1, 96, 8, 5, False),              # row kernel, direct kernel
    ((1 << 21), 2048, 2, 4, True), ((1 << 21) - 1, 2048, 2, 4, True), ((1 << 21) + 9, 2048, 3, 4, True),
])
def test_server_rows_at_the_line(n, bucket, W, bits, with_acc):
    _step_at_the_lines(n, bucket, W, bits, with_acc)


@pytest.mark.parametrize("n,bucket", [
    (512 * 32, 32), (512 * 32 + 1, 32),            # as many spans as one launch takes, one more
    (65_535, 128), (65_536, 128),
])
@pytest.mark.parametrize("norm", [False, True])
def test_several_workers_with_draws_off_a_block_boundary(n, bucket, norm):
    W, bits, off = 3, 5, 3
    xs = [wl.normal(n, 1e-3, config=1, worker=w) for w in range(W)]
    codes = [Guarded(O.code_words(n, bits), torch.int32) for _ in range(W)]
    scales = [Guarded(O.num_buckets(n, bucket), torch.float32) for _ in range(W)]
    call, ref = (mqg.mqg_quantize_workers_l2, O.quantize_l2) if norm else (mqg.mqg_quantize_workers, O.quantize)
    call([to_dev(x) for x in xs], W, n, bits, bucket, 7, [c.view for c in codes], [s.view for s in scales],
         first_worker=2, step=1, elem_offset=off)
    torch.cuda.synchronize()
    for w in range(W):
        codes[w].check_guards(), scales[w].check_guards()
        c_ref, s_ref = ref(xs[w], bits, bucket, 7, worker=2 + w, step=1, elem_offset=off)
        assert bits_equal(scales[w].numpy(np.float32), s_ref) == 0
        assert np.array_equal(codes[w].numpy(np.uint32), c_ref)


@pytest.mark.parametrize("rows", [3, 7, 9, 17, 31, 33, 65, 127, 129, 255])
def test_sums_over_an_odd_number_of_rows(rows):
    """1, 2, 4 .. 32 lanes on a bucket's tree; the last bucket is short."""
    bucket = 32 * rows
    n = 9 * bucket + bucket // 2 + 5
    rng = np.random.default_rng(rows)
    x = (rng.standard_normal(n, dtype=np.float32) * np.exp2(rng.integers(-12, 12, n))).astype(np.float32)
    c, s = Guarded(O.code_words(n, 4), torch.int32), Guarded(O.num_buckets(n, bucket), torch.float32)
    mqg.mqg_quantize_l2(to_dev(x), n, 4, bucket, 5, c.view, s.view, elem_offset=3)
    e0 = rng.standard_normal(n, dtype=np.float32)
    e, c1, r = Guarded(n, torch.float32, fill=e0), Guarded(O.code_words(n, 1), torch.int32), \
        Guarded(2 * O.num_buckets(n, bucket), torch.float32)
    mqg.mqg_quantize_1bit_ef(to_dev(x), e.view, n, bucket, c1.view, r.view)
    torch.cuda.synchronize()
    c_ref, s_ref = O.quantize_l2(x, 4, bucket, 5, elem_offset=3)
    assert bits_equal(s.numpy(np.float32), s_ref) == 0 and np.array_equal(c.numpy(np.uint32), c_ref)
    want = O.quantize_1bit_ef(x, e0.copy(), bucket)
    for got, ref in zip((c1.numpy(np.uint32), r.numpy(np.float32), e.numpy(np.float32)), want):
        assert bits_equal(got, np.asarray(ref).ravel()) == 0
    for b in (c, s, e, c1, r):
        b.check_guards()


@pytest.mark.parametrize("bf16,longest", [(True, 512 * 8192), (True, 512 * 8192 + 1), (False, 2048 * 8192 + 1)])
def test_spans_beside_the_max_pass_and_before_it(bf16, longest):
    """16 workers: 8192 tiles (bf16) or 32,768 in the max pass, with which the short segment shares a launch, and more."""
    W, bits = 16, 3
    seg = np.cumsum([0, 504, longest]).astype(np.uint64)
    code = np.cumsum([0] + [O.code_words(int(b - a), bits) for a, b in zip(seg, seg[1:])]).astype(np.uint64)
    x = wl.normal(int(seg[-1]), 1e-3, config=3, worker=0)
    x = wl.f32_to_bf16_bits(x) if bf16 else x
    g = to_dev(x.view(np.int16)).view(torch.bfloat16) if bf16 else to_dev(x)
    codes = [Guarded(int(code[-1]), torch.int32) for _ in range(W)]
    scales = [Guarded(2, torch.float32) for _ in range(W)]
    mqg.mqg_quantize_segments_workers([g] * W, W, seg, code, bits, 7, [c.view for c in codes], [s.view for s in scales])
    torch.cuda.synchronize()
    for w in range(W):
        codes[w].check_guards(), scales[w].check_guards()
        if w in (0, W - 1):
            c_ref, s_ref = O.quantize_segments(x, seg, code, bits, seed=7, worker=w, dtype="bf16" if bf16 else "f32")
            assert np.array_equal(codes[w].numpy(np.uint32), c_ref)
        assert bits_equal(scales[w].numpy(np.float32), s_ref) == 0
