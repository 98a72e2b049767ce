"""The persistent one-bit kernel: one tile and many per CTA, tiles of fewer rows than threads, a ragged row alone in its tile
and with others, the lines to the kernel of a CTA per tile, and a wait that runs out; bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


def _inputs(n, bf16):
    x = wl.student_t_bf16(n, config=5, worker=1) if bf16 else wl.laplace(n, 1e-4, config=13, worker=1)
    return x, (to_dev(x.view(np.int16)).view(torch.bfloat16) if bf16 else to_dev(x)), wl.normal(n, 1e-4, config=2, worker=3)


@pytest.mark.parametrize("n,bucket", [
    (2047, 512), (2048, 512), (2049, 2048), (128 * 32 * 3, 4096), (128 * 32 * 3 + 1, 4096), (128 * 32 * 2 - 1, 1024),
    (120 * 32 * 4 + 5, 768), (96 * 32 * 3 + 31, 3072), (125 * 32 * 2 + 7, 160), (40_001, 32), (5000, 8192), (3_000_001, 2048),
    (8192 * 5 + 1, 8192),
])
@pytest.mark.parametrize("bf16", [False, True])
def test_tiles(n, bucket, bf16):
    x, g, e = _inputs(n, bf16)
    res = Guarded(n, torch.float32, fill=e)
    for _ in range(2):                                  # the second pass starts from the first one's residual
        codes, ranges = Guarded(O.code_words(n, 1), torch.int32), Guarded(2 * O.num_buckets(n, bucket), torch.float32)
        mqg.mqg_quantize_1bit_ef(g, res.view, n, bucket, codes.view, ranges.view)
        torch.cuda.synchronize()
        codes.check_guards(), ranges.check_guards(), res.check_guards()
        c_ref, r_ref, e = O.quantize_1bit_ef(x, e, bucket, dtype="bf16" if bf16 else "f32")
        assert np.array_equal(codes.numpy(np.uint32), c_ref)
        assert bits_equal(ranges.numpy(np.float32), r_ref.reshape(-1)) == 0
        assert bits_equal(res.numpy(np.float32), e) == 0
    assert mqg.mqg_device_timeouts() == 0


def test_a_wait_that_runs_out():
    n, bucket = 3_000_001, 2048
    _, g, e = _inputs(n, False)
    res = Guarded(n, torch.float32, fill=e)
    codes, ranges = Guarded(O.code_words(n, 1), torch.int32), Guarded(2 * O.num_buckets(n, bucket), torch.float32)
    try:
        mqg.mqg_test_wait_override(1024, True)
        mqg.mqg_quantize_1bit_ef(g, res.view, n, bucket, codes.view, ranges.view)
        with pytest.raises(mqg.MqgError) as err:
            mqg.mqg_check_timeouts(reset=True)
        assert err.value.status == mqg.MQG_ERR_TIMEOUT
        assert bits_equal(res.numpy(np.float32), e) == 0 and (codes.numpy(np.uint32) == 0x7FC0DEAD).all()
    finally:
        mqg.mqg_test_wait_override(0, False)
    assert mqg.mqg_check_timeouts(reset=True) == 0
