"""The downlink's general kernel on tiles of fewer than 256 rows (staged code words, whole and short last tiles) and
the several-workers quantizers on shapes that go to a CTA per bucket, against the CPU checker bit for bit."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bucket,W", [
    (240 * 32 * 5 + 17, 768, 3), (240 * 32 * 3, 768, 8),          # 24 rows: tiles of 240
    (192 * 32 * 4 + 96 * 32, 3072, 2), (3072 * 9 + 1, 3072, 16),  # 96 rows: tiles of 192
    (255 * 32 * 2 + 5, 96, 2), (250 * 32 * 3 + 64, 320, 4),       # 255 and 250 rows: words off 16 bytes at odd widths
    (2047, 2048, 32),
])
@pytest.mark.parametrize("bits", [1, 2, 3, 4, 5, 8])
def test_downlink_general_tiles(n, bucket, W, bits):
    rng = np.random.default_rng(n + bits)
    codes = [rng.integers(0, 1 << 32, O.code_words(n, bits), dtype=np.uint32) for _ in range(W)]
    scales = [rng.random(O.num_buckets(n, bucket), dtype=np.float32) for _ in range(W)]
    c_ref, s_ref = O.server_requantize(codes, scales, bits, n, bucket, 1.0 / W, 5, worker=W, step=2)
    co, so = Guarded(O.code_words(n, bits), torch.int32), Guarded(O.num_buckets(n, bucket), torch.float32)
    mqg.mqg_server_requantize([to_dev(c.view(np.int32)) for c in codes], [to_dev(s) for s in scales], W, bits, n, bucket,
                              1.0 / W, 5, co.view, so.view, worker=W, step=2)
    torch.cuda.synchronize()
    co.check_guards(), so.check_guards()
    assert bits_equal(so.numpy(np.float32), s_ref) == 0
    assert np.array_equal(co.numpy(np.uint32), c_ref)


@pytest.mark.parametrize("n,bucket,offset", [(6581, 8192, 0), (1000, 96, 0), (40_000, 1024, 3), (50_000, 4160, 8)])
@pytest.mark.parametrize("norm", [False, True])
def test_workers_outside_the_one_pass_kernel(n, bucket, offset, norm):
    W, bits = 5, 3
    rng = np.random.default_rng(n)
    xs = [rng.standard_normal(n, dtype=np.float32) for _ in range(W)]
    codes = [Guarded(O.code_words(n, bits), torch.int32) for _ in range(W)]
    scales = [Guarded(O.num_buckets(n, bucket), torch.float32) for _ in range(W)]
    call, ref = (mqg.mqg_quantize_workers_l2, O.quantize_l2) if norm else (mqg.mqg_quantize_workers, O.quantize)
    call([to_dev(x) for x in xs], W, n, bits, bucket, 3, [c.view for c in codes], [s.view for s in scales], first_worker=1,
         elem_offset=offset)
    torch.cuda.synchronize()
    for w in range(W):
        codes[w].check_guards(), scales[w].check_guards()
        c_ref, s_ref = ref(xs[w], bits, bucket, 3, worker=1 + w, elem_offset=offset)
        assert bits_equal(scales[w].numpy(np.float32), s_ref) == 0
        assert np.array_equal(codes[w].numpy(np.uint32), c_ref)
