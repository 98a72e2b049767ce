"""Segment tables are read once, when the call begins: what happens to the caller's array afterwards does not matter."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded

pytestmark = pytest.mark.gpu


class Seed:
    """An integer whose conversion changes the tables that stand before it in the argument list."""

    def __init__(self, *tables):
        self.tables = tables

    def __index__(self):
        for t in self.tables:
            t[1:] = 0
        return 5

    def __and__(self, mask):
        return int(self.__index__()) & mask


def test_offset_arrays_are_copied():
    bits, sizes = 3, [1000, 33, 20_000]
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    code = np.concatenate([[0], np.cumsum([O.code_words(s, bits) for s in sizes])]).astype(np.uint64)
    x = wl.normal(int(seg[-1]), 1e-3, config=3, worker=0)
    c_ref, s_ref = O.quantize_segments(x, seg, code, bits, seed=5)
    codes, scales = Guarded(int(code[-1]), torch.int32), Guarded(len(sizes), torch.float32)
    a, b = seg.copy(), code.copy()
    mqg.mqg_quantize_segments(torch.from_numpy(x).cuda(), a, b, bits, Seed(a, b), codes.view, scales.view)
    torch.cuda.synchronize()
    assert not a[1:].any()
    codes.check_guards(), scales.check_guards()
    assert np.array_equal(scales.numpy(np.float32), s_ref)
    assert np.array_equal(codes.numpy(np.uint32), c_ref)


def test_worker_counts_outside_the_range_are_the_library_s_to_reject():
    with pytest.raises(mqg.MqgError) as err:
        mqg.mqg_server_step([], [], 40, 4, 0, 32, None, 0.1)
    assert err.value.status == mqg.MQG_ERR_TOO_MANY_WORKERS
