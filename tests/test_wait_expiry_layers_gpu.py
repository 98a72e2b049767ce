"""Bounded waits that run out (see test_wait_expiry_gpu.py for how) in the kernels where every warp gives up by itself, or
whose rows hold 64 elements: the encode of the per-layer quantizer's long segments, and long bf16 gradients."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.test_wait_expiry_gpu import SENTINEL, _expect_timeout

pytestmark = pytest.mark.gpu

BITS = 4


def _dev(x, bf16):
    return torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) if bf16 else torch.from_numpy(x).cuda()


@pytest.fixture
def waits_run_out():
    assert mqg.mqg_check_timeouts(reset=True) == 0
    yield lambda: mqg.mqg_test_wait_override(1024, True)
    mqg.mqg_test_wait_override(0, False)
    mqg.mqg_device_timeouts()


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("longest", [70_000, 6_000_000])             # a tile or less per CTA, several
def test_per_layer_encode(waits_run_out, bf16, longest):
    W, sizes = 2, [longest + 9, 500, 40_000]
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    seg[1:] = (seg[1:] + 7) // 8 * 8                                 # every start aligned for bulk copies
    coff = np.concatenate([[0], np.cumsum([O.code_words(int(b - a), BITS) for a, b in zip(seg, seg[1:])])]).astype(np.uint64)
    xs = [wl.normal(int(seg[-1]), 1e-3, config=3, worker=w) for w in range(W)]
    if bf16:
        xs = [wl.f32_to_bf16_bits(x) for x in xs]
    grads = [_dev(x, bf16) for x in xs]

    def run():
        codes = [torch.full((int(coff[-1]),), SENTINEL, dtype=torch.int32, device="cuda") for _ in range(W)]
        scales = [torch.full((len(sizes),), -7.0, device="cuda") for _ in range(W)]
        mqg.mqg_quantize_segments_workers(grads, W, seg, coff, BITS, 3, codes, scales)
        return [c.cpu().numpy().view(np.uint32) for c in codes], [s.cpu().numpy() for s in scales]

    refs = [O.quantize_segments(x, seg, coff, BITS, seed=3, worker=w, dtype="bf16" if bf16 else "f32")
            for w, x in enumerate(xs)]
    waits_run_out()
    codes, scales = run()
    _expect_timeout()
    for w in range(W):
        assert np.array_equal(scales[w], refs[w][1])                 # the passes before it read with plain loads
        for j in (0, 2):                                             # the long segments: not a word written
            assert (codes[w][int(coff[j]):int(coff[j + 1])] == SENTINEL).all()
        assert np.array_equal(codes[w][int(coff[1]):int(coff[2])], refs[w][0][int(coff[1]):int(coff[2])])
    mqg.mqg_test_wait_override(0, False)
    codes, scales = run()
    for w in range(W):
        assert np.array_equal(codes[w], refs[w][0]) and np.array_equal(scales[w], refs[w][1])
    assert mqg.mqg_check_timeouts(reset=True) == 0


@pytest.mark.parametrize("W", [1, 2])
def test_long_bf16(waits_run_out, W):
    n, bucket = (20 << 20) // W + 77, 2048
    x = wl.f32_to_bf16_bits(wl.normal(n, 1e-3, config=5, worker=0))
    g = _dev(x, True)

    def run():
        codes = [torch.full((mqg.mqg_code_words(n, BITS),), SENTINEL, dtype=torch.int32, device="cuda") for _ in range(W)]
        scales = [torch.full((mqg.mqg_num_buckets(n, bucket),), -7.0, device="cuda") for _ in range(W)]
        if W == 1:
            mqg.mqg_quantize(g, n, BITS, bucket, 3, codes[0], scales[0])
        else:
            mqg.mqg_quantize_workers([g] * W, W, n, BITS, bucket, 3, codes, scales)
        return codes, scales

    waits_run_out()
    codes, scales = run()
    _expect_timeout()
    assert all(bool((c == SENTINEL).all()) for c in codes) and all(bool((s == -7.0).all()) for s in scales)
    mqg.mqg_test_wait_override(0, False)
    codes, scales = run()
    for w in range(W):
        c_ref, s_ref = O.quantize(x, BITS, bucket, 3, worker=w, dtype="bf16")
        assert np.array_equal(codes[w].cpu().numpy().view(np.uint32), c_ref)
        assert np.array_equal(scales[w].cpu().numpy(), s_ref)
    assert mqg.mqg_check_timeouts(reset=True) == 0
