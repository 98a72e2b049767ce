"""A gradient's NaN elements do not count for the scale of their bucket, in bf16 as in fp32 and whichever kernel takes the
shape: a bucket that is NaN throughout has the scale 0, any other the largest magnitude of its other elements.  (What
code a NaN element gets is not defined.)"""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg

pytestmark = pytest.mark.gpu


def _scales(g, n, bucket, W):
    codes = [torch.zeros(mqg.mqg_code_words(n, 4), dtype=torch.int32, device="cuda") for _ in range(W)]
    scales = [torch.full((mqg.mqg_num_buckets(n, bucket),), -7.0, device="cuda") for _ in range(W)]
    if W == 1:
        mqg.mqg_quantize(g, n, 4, bucket, 0, codes[0], scales[0])
    else:
        mqg.mqg_quantize_workers([g] * W, W, n, 4, bucket, 0, codes, scales)
    return scales


@pytest.mark.parametrize("n,bucket,W", [
    (1000, 96, 1),                     # plain loads
    (20_001, 2048, 1),                 # rows of 32: whole warps, lane shuffles, rows
    (20_001, 512, 2),
    (20_001, 768, 2),
    (40_000, 16_384, 1),               # a CTA per bucket
    ((20 << 20) + 100, 2048, 1),       # rows of 64 in bf16
    ((20 << 20) + 100, 1024, 1),
    ((10 << 20) + 100, 960, 2),
])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_scales_ignore_nan(n, bucket, W, dtype):
    gen = torch.Generator(device="cuda").manual_seed(n)
    g = torch.randn(n, device="cuda", generator=gen).to(dtype)
    g[:bucket] = float("nan")                                        # a bucket, and from there rows of each kind
    for row in range(bucket // 32 + 1, min(n // 32, 40 + bucket // 32), 3):
        g[32 * row:32 * row + 32] = float("nan")
    g[-50:] = float("nan")
    g[bucket + 5] = float("nan")
    pad = torch.zeros(-(-n // bucket) * bucket, device="cuda")
    pad[:n] = torch.nan_to_num(g.float(), nan=0.0).abs()
    want = pad.view(-1, bucket).amax(1)
    assert want[0] == 0
    for s in _scales(g, n, bucket, W):
        assert np.array_equal(s.cpu().numpy(), want.cpu().numpy())
