"""The encode's extreme values, where its integer form touches the ends of its range: elements at +-s, +-0 and next to
the levels, scales from the flush limit to the largest float, every width and both input types, against the CPU
checker bit for bit."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", range(1, 9))
@pytest.mark.parametrize("bf16", [False, True])
def test_extreme_elements_and_scales(bits, bf16):
    bucket, L = 4096, (1 << bits) - 1
    rng = np.random.default_rng(bits)
    parts = []
    for s in (2.0 ** -96, 1.0000001 * 2.0 ** -96, 3e-20, 1e-4, 1.0, 1.5, 7.3e11, 1.6e38):
        s = np.float32(s)
        grid = (2 * rng.integers(0, L + 1, bucket).astype(np.float64) - L) / L * np.float64(s)    # the levels
        x = grid.astype(np.float32)
        k = rng.integers(0, 6, bucket)
        x = np.where(k == 1, np.nextafter(x, np.float32(0)), x)
        x = np.where(k == 2, s, x)
        x = np.where(k == 3, -s, x)
        x = np.where(k == 4, np.float32(0.0) * np.sign(x), x)
        x[0] = s
        parts.append(np.clip(x, -s, s).astype(np.float32))
    parts.append(np.full(bucket, 2.0 ** -97, np.float32))              # flushed
    x = np.concatenate(parts)
    if bf16:
        x = wl.f32_to_bf16_bits(x)
    n = x.size
    g = to_dev(x.view(np.int16)).view(torch.bfloat16) if bf16 else to_dev(x)
    codes, scales = Guarded(mqg.mqg_code_words(n, bits), torch.int32), Guarded(mqg.mqg_num_buckets(n, bucket), torch.float32)
    for seed in range(12):                                             # many draws per value
        mqg.mqg_quantize(g, n, bits, bucket, seed, codes.view, scales.view, worker=seed)
        torch.cuda.synchronize()
        c_ref, s_ref = O.quantize(x, bits, bucket, seed, worker=seed, dtype="bf16" if bf16 else "f32")
        assert bits_equal(scales.numpy(np.float32), s_ref) == 0
        assert np.array_equal(codes.numpy(np.uint32), c_ref)
