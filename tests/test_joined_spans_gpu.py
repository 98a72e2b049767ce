"""Segments that a cluster of CTAs quantizes as a whole, at the lines where the part of a CTA grows (256, 512, 1024 rows),
where the cluster does, where it ends and two passes take over, and off every boundary: bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu

SIZES = {
    "two_of_256_rows": [16385, 0, 1, 8193, 8192],
    "eight_of_256_rows": [65536, 40_000, 31, 16384, 57_344],
    "longer": [65537, 16384, 16385, 100],
    "eight_of_512_rows": [131_072, 8, 131_071],
    "of_1024_rows": [131_073, 32_768, 32_769],
    "the_longest": [262_144, 7, 262_143, 196_609],
    "one_more": [262_145, 100, 30_000],
    "two_tables": [20_000, 96] * 40,
    "shared_clusters": [20_000, 17_000, 60_000, 9_000, 12_000, 33_000, 41_000, 0, 5, 8193],
    "two_rows_per_thread": [9_000, 16_384, 8193, 100] * 12 + [20_000, 60_001, 33_000] * 5,
}


@pytest.mark.parametrize("name", SIZES)
@pytest.mark.parametrize("bits,bf16,W", [(4, False, 3), (1, True, 1), (7, True, 2)])
def test_max_abs(name, bits, bf16, W):
    sizes = SIZES[name]
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    code = np.concatenate([[0], np.cumsum([O.code_words(s, bits) for s in sizes])]).astype(np.uint64)
    xs = [wl.layered(sizes, config=3, worker=w) for w in range(W)]
    xs[0][:sizes[0]] = 0.0                                        # a flushed segment
    xs[-1][sizes[0] - 1] = 1.0                                    # the maximum in the last CTA's last row
    if bf16:
        xs = [wl.f32_to_bf16_bits(x) for x in xs]
    grads = [to_dev(x.view(np.int16)).view(torch.bfloat16) if bf16 else to_dev(x) for x in xs]
    for offset in (64, 3):
        codes = [Guarded(int(code[-1]), torch.int32) for _ in range(W)]
        scales = [Guarded(len(sizes), torch.float32) for _ in range(W)]
        mqg.mqg_quantize_segments_workers(grads, W, seg, code, bits, 5, [c.view for c in codes], [s.view for s in scales],
                                          first_worker=1, step=2, elem_offset=offset)
        torch.cuda.synchronize()
        for w in range(W):
            codes[w].check_guards(), scales[w].check_guards()
            c_ref, s_ref = O.quantize_segments(xs[w], seg, code, bits, seed=5, worker=1 + w, step=2, elem_offset=offset,
                                               dtype="bf16" if bf16 else "f32")
            assert bits_equal(scales[w].numpy(np.float32), s_ref) == 0
            assert np.array_equal(codes[w].numpy(np.uint32), c_ref)


@pytest.mark.parametrize("name", SIZES)
def test_norm(name):
    sizes, bits = SIZES[name], 5
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    code = np.concatenate([[0], np.cumsum([O.code_words(s, bits) for s in sizes])]).astype(np.uint64)
    x = wl.layered(sizes, config=3, worker=1)
    codes, scales = Guarded(int(code[-1]), torch.int32), Guarded(len(sizes), torch.float32)
    ws = torch.empty(max(1, mqg.mqg_l2_workspace_floats(seg)), dtype=torch.float32, device="cuda")
    mqg.mqg_quantize_segments_l2(to_dev(x), seg, code, bits, 4, codes.view, scales.view, ws, worker=3, step=2)
    torch.cuda.synchronize()
    codes.check_guards(), scales.check_guards()
    c_ref, s_ref = O.quantize_segments_l2(x, seg, code, bits, 4, worker=3, step=2)
    assert bits_equal(scales.numpy(np.float32), s_ref) == 0
    assert np.array_equal(codes.numpy(np.uint32), c_ref)
