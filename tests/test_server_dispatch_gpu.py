"""The server step at the lines of its dispatch: direct kernel / row kernel for shapes the bulk-copy kernel does not
take, sum as an extra output in one pass / in two, one tile per warp / several, ragged last rows with many workers.
Every element is compared bit for bit with the CPU checker on codes and scales drawn at random (a scale of zero
among them), so a result does not depend on the quantizer."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bucket,W,bits,with_acc", [
    ((1 << 25) // 12 + 37, 96, 8, 3, True),        # row kernel, ragged last row and bucket
    ((1 << 25) // 12 - 37, 96, 8, 5, True),        # direct kernel just below the line
    ((1 << 25) // 5 + 32, 640, 1, 7, False),       # row kernel, one worker
    ((1 << 22) + 5, 2048, 8, 4, True),             # the sum by the bulk-copy kernel, then the update
    ((1 << 22) - 3, 2048, 8, 2, True),             # both in one pass
    (4 * 1024 + 1, 2048, 32, 6, False),            # the bulk-copy kernel's shortest gradient, ragged, 32 workers
    (4 * 1024 - 1, 2048, 9, 7, True),              # one below: direct kernel, a second batch of one worker
    (148 * 16 * 1024 + 1024 + 9, 1024, 2, 1, False),   # more tiles than warps in the grid
])
def test_server_step_at_the_dispatch_lines(n, bucket, W, bits, with_acc):
    rng = np.random.default_rng(n)
    codes = [rng.integers(0, 1 << 32, O.code_words(n, bits), dtype=np.uint32) for _ in range(W)]
    scales = [rng.random(O.num_buckets(n, bucket), dtype=np.float32) * np.float32(1e-3) for _ in range(W)]
    scales[W - 1][-1] = 0.0
    p0 = wl.params(n, 0.05, config=21)
    p_ref, acc_ref = O.server_step(codes, scales, bits, n, bucket, p0.copy(), 0.1 / W, want_acc=True)
    p = Guarded(n, torch.float32, fill=p0)
    acc = Guarded(n, torch.float32) if with_acc else None
    mqg.mqg_server_step([to_dev(c.view(np.int32)) for c in codes], [to_dev(s) for s in scales], W, bits, n, bucket,
                        p.view, 0.1 / W, acc.view if with_acc else None)
    torch.cuda.synchronize()
    p.check_guards()
    assert bits_equal(p.numpy(np.float32), p_ref) == 0
    if with_acc:
        acc.check_guards()
        assert bits_equal(acc.numpy(np.float32), acc_ref) == 0
    assert mqg.mqg_device_timeouts() == 0


@pytest.mark.parametrize("W", [1, 9, 16])
def test_segments_with_ragged_rows_and_short_segments(W):
    """Bulk-copy segments with ragged last rows (more of them than workers' batches hold), unaligned short ones."""
    bits = 3
    sizes = [40_008, 1, 70_032, 17, 33_000, 8_191, 50_024, 32]
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    code = np.concatenate([[0], np.cumsum([-(-O.code_words(s, bits) // 4) * 4 for s in sizes])]).astype(np.uint64)
    rng = np.random.default_rng(W)
    n = int(seg[-1])
    codes = [rng.integers(0, 1 << 32, int(code[-1]), dtype=np.uint32) for _ in range(W)]
    scales = [rng.random(len(sizes), dtype=np.float32) for _ in range(W)]
    p0 = wl.params(n, 0.05, config=3)
    for with_acc in (False, True):
        p_ref, acc_ref = O.server_step_segments(codes, scales, bits, seg, code, p0.copy(), 0.02, want_acc=True)
        p = Guarded(n, torch.float32, fill=p0)
        acc = Guarded(n, torch.float32) if with_acc else None
        mqg.mqg_server_step_segments([to_dev(c.view(np.int32)) for c in codes], [to_dev(s) for s in scales], W, bits,
                                     seg, code, p.view, 0.02, acc.view if with_acc else None)
        torch.cuda.synchronize()
        p.check_guards()
        assert bits_equal(p.numpy(np.float32), p_ref) == 0
        if with_acc:
            acc.check_guards()
            assert bits_equal(acc.numpy(np.float32), acc_ref) == 0
