"""The downlink's persistent kernel on ragged gradients and on buckets of three and of eight warps: the last row alone in its
tile, in a tile with others, words that end inside 16 bytes, buckets that begin inside a warp's rows; bit for bit."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bucket", [
    (16384 + 1, 2048), (128 * 32 * 5 + 31, 4096), (128 * 32 * 5 - 1, 1024), (17_000, 256), (20_011, 512), (16384 + 64 * 32 + 7, 2048),
    (8192 * 3 + 1, 8192), (8192 * 4, 8192), (8192 * 2 + 5000, 8192), (3072 * 8 + 33, 3072), (3072 * 700, 3072), (1536 * 12 - 5, 1536),
    (768 * 30 + 770, 768), (768 * 4000, 768),
])
@pytest.mark.parametrize("bits,W", [(1, 8), (2, 3), (3, 9), (4, 16), (5, 1), (7, 4), (8, 8)])
def test_downlink(n, bucket, bits, W):
    if bucket == 256:
        W = min(W, 8)
    rng = np.random.default_rng(n + bits)
    words, nb = O.code_words(n, bits), O.num_buckets(n, bucket)
    codes = [rng.integers(0, 1 << 32, words, dtype=np.uint32) for _ in range(W)]
    scales = [rng.random(nb, dtype=np.float32) * np.float32(1e-3) for _ in range(W)]
    for s in scales:
        s[nb // 2] = 0.0                          # a flushed bucket
    c_ref, s_ref = O.server_requantize(codes, scales, bits, n, bucket, 1.0 / W, 5, worker=W, step=2)
    # the streams end at the end of their buffers
    dev = [Guarded(words, torch.int32, fill=c.view(np.int32)) for c in codes]
    co, so = Guarded(words, torch.int32), Guarded(nb, torch.float32)
    mqg.mqg_server_requantize([d.view for d in dev], [to_dev(s) for s in scales], W, bits, n, bucket, 1.0 / W, 5, co.view,
                              so.view, worker=W, step=2)
    torch.cuda.synchronize()
    co.check_guards(), so.check_guards()
    assert bits_equal(so.numpy(np.float32), s_ref) == 0
    assert np.array_equal(co.numpy(np.uint32), c_ref)
