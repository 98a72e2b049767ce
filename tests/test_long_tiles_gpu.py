"""Buckets of 8193 to 16384 elements in the bulk-copy kernels (tiles of more rows than one copy's box holds), fp32, bf16 in
rows of 32 and of 64, one worker and several, whole and ragged ends, and buckets of 8192 in launches long enough for two stages:
bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bucket,W,bits", [
    (3 * 16384, 16384, 1, 4),
    (5 * 16384 + 31, 16384, 2, 3),
    (4 * 12288 + 12288 - 1, 12288, 1, 8),            # 384 of 512 rows
    (9216 * 6 + 33, 9216, 3, 1),                     # 288 rows (of 64: 144, no whole warps)
    (16384, 16384, 2, 5),                            # one bucket
    (16384 * 700 + 17, 16384, 2, 4),                 # more tiles than CTAs; bf16: rows of 64
    (8192 * 2305, 8192, 1, 4),                       # from 18 M elements on
    (8192 * 1160 + 17, 8192, 2, 5),
])
@pytest.mark.parametrize("bf16", [False, True])
def test_long_tiles(n, bucket, W, bits, bf16):
    xs = [wl.student_t_bf16(n, config=5, worker=w) if bf16 else wl.laplace(n, 1e-4, config=13, worker=w) for w in range(W)]
    xs[0][:min(bucket, n)] = 0                       # a flushed bucket
    grads = [to_dev(x.view(np.int16)).view(torch.bfloat16) if bf16 else to_dev(x) for x in xs]
    dt, nb = "bf16" if bf16 else "f32", mqg.mqg_num_buckets(n, bucket)
    codes = [Guarded(mqg.mqg_code_words(n, bits), torch.int32) for _ in range(W)]
    scales = [Guarded(nb, torch.float32) for _ in range(W)]
    ranges = [Guarded(2 * nb, torch.float32) for _ in range(W)]
    if W == 1:
        mqg.mqg_quantize(grads[0], n, bits, bucket, 9, codes[0].view, scales[0].view, worker=2, step=1, elem_offset=40)
    else:
        mqg.mqg_quantize_workers(grads, W, n, bits, bucket, 9, [c.view for c in codes], [s.view for s in scales],
                                 first_worker=2, step=1, elem_offset=40)
    torch.cuda.synchronize()
    for w in range(W):
        codes[w].check_guards(), scales[w].check_guards()
        c_ref, s_ref = O.quantize(xs[w], bits, bucket, 9, worker=2 + w, step=1, elem_offset=40, dtype=dt)
        assert bits_equal(scales[w].numpy(np.float32), s_ref) == 0
        assert np.array_equal(codes[w].numpy(np.uint32), c_ref)
    if W == 1:
        mqg.mqg_quantize_minmax(grads[0], n, bits, bucket, codes[0].view, ranges[0].view)
    else:
        mqg.mqg_quantize_workers_minmax(grads, W, n, bits, bucket, [c.view for c in codes], [r.view for r in ranges])
    torch.cuda.synchronize()
    for w in range(W):
        codes[w].check_guards(), ranges[w].check_guards()
        c_ref, r_ref = O.quantize_minmax(xs[w], bits, bucket, dtype=dt)
        assert bits_equal(ranges[w].numpy(np.float32), r_ref.reshape(-1)) == 0
        assert np.array_equal(codes[w].numpy(np.uint32), c_ref)
    assert mqg.mqg_device_timeouts() == 0


@pytest.mark.parametrize("n", [8192 * 2305, 8192 * 2305 + 5])
def test_norm_in_two_stages(n):
    bits, bucket = 6, 8192
    x = wl.laplace(n, 1e-4, config=13, worker=1)
    codes, scales = Guarded(mqg.mqg_code_words(n, bits), torch.int32), Guarded(mqg.mqg_num_buckets(n, bucket), torch.float32)
    mqg.mqg_quantize_l2(to_dev(x), n, bits, bucket, 9, codes.view, scales.view, worker=1)
    torch.cuda.synchronize()
    codes.check_guards(), scales.check_guards()
    c_ref, s_ref = O.quantize_l2(x, bits, bucket, 9, worker=1)
    assert bits_equal(scales.numpy(np.float32), s_ref) == 0
    assert np.array_equal(codes.numpy(np.uint32), c_ref)
