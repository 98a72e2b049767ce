"""Bounded waits that run out (see test_wait_expiry_gpu.py for how) in the kernels for segments that start off the 16-byte
boundaries and in the quantizers whose tile is a bucket of up to 16,384 elements."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.test_wait_expiry_gpu import SENTINEL, _expect_timeout
from tests.test_wait_expiry_layers_gpu import _dev, waits_run_out  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("longest", [70_000, 6_000_000])             # a tile or less per CTA, several
def test_per_layer_encode(waits_run_out, bf16, longest):  # noqa: F811
    W, bits, sizes = 2, 5, [501, longest + 9, 40_000]                # the long ones start at 501 and beyond an odd length
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    coff = np.concatenate([[0], np.cumsum([O.code_words(s, bits) for s in sizes])]).astype(np.uint64)
    xs = [wl.normal(int(seg[-1]), 1e-3, config=3, worker=w) for w in range(W)]
    if bf16:
        xs = [wl.f32_to_bf16_bits(x) for x in xs]
    grads = [_dev(x, bf16) for x in xs]

    def run():
        codes = [torch.full((int(coff[-1]),), SENTINEL, dtype=torch.int32, device="cuda") for _ in range(W)]
        scales = [torch.full((len(sizes),), -7.0, device="cuda") for _ in range(W)]
        mqg.mqg_quantize_segments_workers(grads, W, seg, coff, bits, 3, codes, scales)
        return [c.cpu().numpy().view(np.uint32) for c in codes], [s.cpu().numpy() for s in scales]

    refs = [O.quantize_segments(x, seg, coff, bits, seed=3, worker=w, dtype="bf16" if bf16 else "f32")
            for w, x in enumerate(xs)]
    waits_run_out()
    codes, scales = run()
    _expect_timeout()
    short = int(coff[1])
    for w in range(W):
        assert np.array_equal(scales[w], refs[w][1])                 # the passes before it read with plain loads
        assert np.array_equal(codes[w][:short], refs[w][0][:short])
        assert (codes[w][short:] == SENTINEL).all()                  # the long segments: not a word written
    mqg.mqg_test_wait_override(0, False)
    codes, scales = run()
    for w in range(W):
        assert np.array_equal(codes[w], refs[w][0]) and np.array_equal(scales[w], refs[w][1])
    assert mqg.mqg_check_timeouts(reset=True) == 0


@pytest.mark.parametrize("bits,W", [(4, 8), (5, 3)])
def test_server_step(waits_run_out, bits, W):  # noqa: F811
    lr, sizes = 0.05, [501, 1_100_003, 40_002, 77]
    rng = np.random.default_rng(bits)
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    coff = np.concatenate([[0], np.cumsum([O.code_words(s, bits) for s in sizes])]).astype(np.uint64)
    codes = [rng.integers(0, 1 << 32, int(coff[-1]), dtype=np.uint32) for _ in range(W)]
    scales = [rng.random(len(sizes), dtype=np.float32) * np.float32(1e-3) for _ in range(W)]
    p0 = wl.params(int(seg[-1]), 0.05, config=1)
    dev = [torch.from_numpy(c.view(np.int32)).cuda() for c in codes], [torch.from_numpy(s).cuda() for s in scales]
    ref, _ = O.server_step_segments(codes, scales, bits, seg, coff, p0.copy(), lr)

    def run():
        p = torch.from_numpy(p0.copy()).cuda()
        mqg.mqg_server_step_segments(*dev, W, bits, seg, coff, p, lr)
        return p.cpu().numpy()

    waits_run_out()
    got = run()
    _expect_timeout()
    want = ref.copy()                                                # plain loads: short tensors, first and last rows
    for j in (1, 2):
        first, last = (int(seg[j]) + 31) // 32 * 32, int(seg[j + 1])
        last -= (last - first) % 32
        want[first:last] = p0[first:last]                            # the rows of the bulk copies: as they were
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
    mqg.mqg_test_wait_override(0, False)
    assert np.array_equal(run().view(np.uint32), ref.view(np.uint32))
    assert mqg.mqg_check_timeouts(reset=True) == 0


@pytest.mark.parametrize("W", [1, 2])
@pytest.mark.parametrize("n", [16384 * 9, 16384 * 40 + 77, (20 << 20) + 64])   # a tile per CTA, a ragged last bucket, several tiles
def test_tiles_of_512_rows(waits_run_out, n, W):  # noqa: F811
    bits, bucket = 4, 16384
    x = wl.normal(n, 1e-3, config=5, worker=0)
    g = _dev(x, False)

    def run():
        codes = [torch.full((mqg.mqg_code_words(n, bits),), SENTINEL, dtype=torch.int32, device="cuda") for _ in range(W)]
        scales = [torch.full((mqg.mqg_num_buckets(n, bucket),), -7.0, device="cuda") for _ in range(W)]
        if W == 1:
            mqg.mqg_quantize(g, n, bits, bucket, 3, codes[0], scales[0])
        else:
            mqg.mqg_quantize_workers([g] * W, W, n, bits, bucket, 3, codes, scales)
        return codes, scales

    waits_run_out()
    codes, scales = run()
    _expect_timeout()
    assert all(bool((c == SENTINEL).all()) for c in codes) and all(bool((s == -7.0).all()) for s in scales)
    mqg.mqg_test_wait_override(0, False)
    codes, scales = run()
    for w in range(W):
        c_ref, s_ref = O.quantize(x, bits, bucket, 3, worker=w)
        assert np.array_equal(codes[w].cpu().numpy().view(np.uint32), c_ref)
        assert np.array_equal(scales[w].cpu().numpy(), s_ref)
    assert mqg.mqg_check_timeouts(reset=True) == 0
