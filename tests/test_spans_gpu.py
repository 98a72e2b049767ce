"""Buckets and segments that one CTA quantizes as a whole, at the lines where the CTA grows, where two passes take
over and where rows, words and 16-byte boundaries end: bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bucket,W,bits", [
    (8193, 8193, 1, 3),                       # one bucket, the shortest span
    (3 * 16384 + 33, 16384, 3, 4),            # 512 rows, a short last bucket
    (2 * 16416 + 1, 16416, 2, 7),             # 513 rows: the larger CTA; a last bucket of one element
    (2 * 49152, 49152, 2, 8),                 # the longest span
    (2 * 49184 + 5, 49184, 2, 2),             # one row more: two passes
])
@pytest.mark.parametrize("bf16", [False, True])
def test_long_buckets_of_several_workers(n, bucket, W, bits, bf16):
    xs = [wl.student_t_bf16(n, config=5, worker=w) if bf16 else wl.laplace(n, 1e-4, config=13, worker=w) for w in range(W)]
    xs[0][:min(bucket, n)] = 0                # a flushed bucket
    grads = [to_dev(x.view(np.int16)).view(torch.bfloat16) if bf16 else to_dev(x) for x in xs]
    dt = "bf16" if bf16 else "f32"
    codes = [Guarded(mqg.mqg_code_words(n, bits), torch.int32) for _ in range(W)]
    scales = [Guarded(mqg.mqg_num_buckets(n, bucket), torch.float32) for _ in range(W)]
    ranges = [Guarded(2 * mqg.mqg_num_buckets(n, bucket), torch.float32) for _ in range(W)]
    for offset in (0, 8 * 5, 3):
        mqg.mqg_quantize_workers(grads, W, n, bits, bucket, 9, [c.view for c in codes], [s.view for s in scales],
                                 first_worker=2, step=1, elem_offset=offset)
        torch.cuda.synchronize()
        for w in range(W):
            codes[w].check_guards(), scales[w].check_guards()
            c_ref, s_ref = O.quantize(xs[w], bits, bucket, 9, worker=2 + w, step=1, elem_offset=offset, dtype=dt)
            assert bits_equal(scales[w].numpy(np.float32), s_ref) == 0
            assert np.array_equal(codes[w].numpy(np.uint32), c_ref)
    mqg.mqg_quantize_workers_minmax(grads, W, n, bits, bucket, [c.view for c in codes], [r.view for r in ranges])
    torch.cuda.synchronize()
    for w in range(W):
        codes[w].check_guards(), ranges[w].check_guards()
        c_ref, r_ref = O.quantize_minmax(xs[w], bits, bucket, dtype=dt)
        assert bits_equal(ranges[w].numpy(np.float32), r_ref.reshape(-1)) == 0
        assert np.array_equal(codes[w].numpy(np.uint32), c_ref)


@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("bits", [1, 5, 8])
def test_segments_around_the_span_limit(bits, norm):
    """Aligned and unaligned, empty, one element, spans of one and two rows per thread, just beyond a span, a norm of
    more than 1024 tile sums, more than 64 segments (several tables)."""
    sizes = [16384, 16385, 0, 1, 8192, 8193, 33, 16383, 20_000, 70_001, 31] + ([9_000_000, 8] if norm else []) + [96] * 60 + [17_000]
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    code = np.concatenate([[0], np.cumsum([O.code_words(s, bits) for s in sizes])]).astype(np.uint64)
    x = wl.layered(sizes, config=3, worker=1)
    x[:16384] = 0.0
    codes, scales = Guarded(int(code[-1]), torch.int32), Guarded(len(sizes), torch.float32)
    if norm:
        ws = torch.empty(mqg.mqg_l2_workspace_floats(seg), dtype=torch.float32, device="cuda")
        mqg.mqg_quantize_segments_l2(to_dev(x), seg, code, bits, 4, codes.view, scales.view, ws, worker=3, step=2)
        c_ref, s_ref = O.quantize_segments_l2(x, seg, code, bits, 4, worker=3, step=2)
    else:
        mqg.mqg_quantize_segments(to_dev(x), seg, code, bits, 4, codes.view, scales.view, worker=3, step=2)
        c_ref, s_ref = O.quantize_segments(x, seg, code, bits, seed=4, worker=3, step=2)
    torch.cuda.synchronize()
    codes.check_guards(), scales.check_guards()
    assert bits_equal(scales.numpy(np.float32), s_ref) == 0
    assert np.array_equal(codes.numpy(np.uint32), c_ref)
    assert mqg.mqg_device_timeouts() == 0
