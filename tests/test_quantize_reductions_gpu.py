"""The one-pass quantizers' three ways to reduce a bucket (lane shuffles, whole warps, row by row) and both CTA sizes,
for one worker and for several in one launch, in every scale mode: bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bucket", [
    (2048, 96), (148 * 5 * 126 * 32 + 77, 96),       # 3 rows, 42 buckets per tile; more tiles than CTAs, ragged row
    (50_000 + 5, 768), (20_000, 5 * 32),             # 24 and 5 rows
    (40_000 + 31, 127 * 32), (127 * 32 * 2, 127 * 32),   # one bucket of an odd number of rows per tile
    (100_003, 8192), (3 * 8192, 8192), (50_000, 5120), (30_000 + 1, 7168),     # 256, 160, 224 rows: the larger CTA
    (4000, 1 << 20), (8000, 8192),                   # a single bucket: 125 rows, 250 rows (neither way: general kernel)
])
@pytest.mark.parametrize("mode,bits,bf16", [("max", 3, False), ("max", 8, True), ("norm", 5, False), ("norm", 2, True),
                                            ("range", 4, False), ("range", 1, True)])
def test_bucket_reductions(n, bucket, mode, bits, bf16):
    if mode == "norm" and bucket < n and bucket > 8192:
        pytest.skip("longer buckets of the norm variant are segments")
    dt = "bf16" if bf16 else "f32"
    rng = np.random.default_rng(n)
    for W in (1, 3):
        xs = [rng.standard_normal(n, dtype=np.float32) * np.float32(1e-3) for _ in range(W)]
        xs[0][: min(bucket, n)] = 0.0                # a flushed bucket
        if bf16:
            xs = [wl.f32_to_bf16_bits(x) for x in xs]
        grads = [to_dev(x.view(np.int16)).view(torch.bfloat16) if bf16 else to_dev(x) for x in xs]
        per = 2 if mode == "range" else 1
        codes = [Guarded(mqg.mqg_code_words(n, bits), torch.int32) for _ in range(W)]
        scales = [Guarded(per * mqg.mqg_num_buckets(n, bucket), torch.float32) for _ in range(W)]
        cv, sv = [c.view for c in codes], [s.view for s in scales]
        if mode == "range":
            mqg.mqg_quantize_workers_minmax(grads, W, n, bits, bucket, cv, sv)
            ref = [O.quantize_minmax(x, bits, bucket, dtype=dt) for x in xs]
        else:
            f, o = ((mqg.mqg_quantize_workers, O.quantize) if mode == "max" else (mqg.mqg_quantize_workers_l2, O.quantize_l2))
            f(grads, W, n, bits, bucket, 7, cv, sv, first_worker=4, step=3, elem_offset=64)
            ref = [o(x, bits, bucket, 7, worker=4 + w, step=3, elem_offset=64, dtype=dt) for w, x in enumerate(xs)]
        torch.cuda.synchronize()
        for w in range(W):
            codes[w].check_guards(), scales[w].check_guards()
            assert bits_equal(scales[w].numpy(np.float32), np.asarray(ref[w][1]).reshape(-1)) == 0
            assert np.array_equal(codes[w].numpy(np.uint32), ref[w][0])
    assert mqg.mqg_device_timeouts() == 0


@pytest.mark.parametrize("n,bucket,W,bits", [
    ((20 << 20) // 3 + 64 + 1, 2048, 3, 4),          # rows of 64 bf16 elements; a last row of one element
    ((20 << 20) // 3 + 64 + 63, 768, 3, 3),          # 12 rows per bucket, a last row of 63
    ((20 << 20) // 2 + 4096 + 33, 8192, 2, 7),       # 128 rows per bucket
    ((20 << 20) // 2 + 32, 256, 2, 1), ((20 << 20) // 2, 64, 2, 8), ((20 << 20) // 2 + 96, 32, 2, 2),   # 4, 1 rows; narrow
    ((20 << 20) + 5, 4096, 1, 6),
])
def test_long_bf16_gradients(n, bucket, W, bits):
    """Every bucket near the ends and a sample of the others, each encoded by the checker on its own."""
    gen = torch.Generator(device="cuda").manual_seed(n)
    grads = [(torch.randn(n, generator=gen, device="cuda") * 1e-3).to(torch.bfloat16) for _ in range(W)]
    nb = mqg.mqg_num_buckets(n, bucket)
    codes = [Guarded(mqg.mqg_code_words(n, bits), torch.int32) for _ in range(W)]
    scales = [Guarded(nb, torch.float32) for _ in range(W)]
    mqg.mqg_quantize_workers(grads, W, n, bits, bucket, 7, [c.view for c in codes], [s.view for s in scales],
                             first_worker=4, step=3, elem_offset=64)
    torch.cuda.synchronize()
    rng = np.random.default_rng(n)
    some = np.unique(np.concatenate([np.arange(3), np.arange(max(0, nb - 70), nb), rng.integers(0, nb, 200)]))
    for w in range(W):
        codes[w].check_guards(), scales[w].check_guards()
        got_c, got_s = codes[w].numpy(np.uint32), scales[w].numpy(np.float32)
        x = grads[w].view(torch.int16).cpu().numpy().view(np.uint16)
        for b in some.tolist():
            lo, hi = b * bucket, min(n, (b + 1) * bucket)
            c_ref, s_ref = O.quantize(x[lo:hi], bits, bucket, 7, worker=4 + w, step=3, elem_offset=64 + lo, dtype="bf16")
            assert got_s[b] == s_ref[0]
            at = lo * bits // 32
            assert np.array_equal(got_c[at:at + c_ref.size], c_ref), (w, b)
    assert mqg.mqg_device_timeouts() == 0
