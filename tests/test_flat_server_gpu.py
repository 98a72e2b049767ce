"""The layered server step on tensors that start anywhere - rows of the whole parameter buffer, codes that start at any bit -
with every remainder, whole and partial stages of workers, first and last rows of every length, more tensors than a launch
holds, scales outside the range that is summed in units of 2^40; bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


def _run(sizes, bits, W, gaps=0, lr=0.05, wild=False):
    rng = np.random.default_rng(len(sizes) + bits)
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    code = np.concatenate([[0], np.cumsum([O.code_words(s, bits) + gaps for s in sizes])]).astype(np.uint64)
    n, words = int(seg[-1]), int(code[-1]) - gaps              # the last stream ends with its buffer
    codes = [rng.integers(0, 1 << 32, words, dtype=np.uint32) for _ in range(W)]
    scales = [rng.random(len(sizes), dtype=np.float32) * np.float32(1e-3) for _ in range(W)]
    if wild:
        scales[0][0], scales[-1][-1], scales[W // 2][0] = 1e30, 2.0 ** -95, 0.0
    code[-1] = words
    p0 = wl.params(n, 0.05, config=1)
    dev = [Guarded(words, torch.int32, fill=c.view(np.int32)) for c in codes]
    p = Guarded(n, torch.float32, fill=p0)
    mqg.mqg_server_step_segments([d.view for d in dev], [to_dev(s) for s in scales], W, bits, seg, code, p.view, lr)
    torch.cuda.synchronize()
    p.check_guards()
    ref, _ = O.server_step_segments(codes, scales, bits, seg, code, p0.copy(), lr)
    assert bits_equal(p.numpy(np.float32), ref) == 0
    assert mqg.mqg_device_timeouts() == 0


@pytest.mark.parametrize("bits", range(1, 9))
@pytest.mark.parametrize("W", [1, 4, 8, 9, 16])
def test_widths_and_workers(bits, W):
    _run([40_001, 33, 50_031, 32_768, 900_002, 7, 32_799], bits, W, gaps=bits % 3)


@pytest.mark.parametrize("first", range(0, 33))
def test_every_remainder(first):
    _run([first, 33_000, 32_768 + first, 470_000 - first], 3 + first % 5, 4, gaps=first % 2)


@pytest.mark.parametrize("bits", [2, 4, 5, 8])
def test_scales_outside_the_range(bits):
    _run([40_001, 50_031, 1_060_003], bits, 8, wild=True)


def test_more_tensors_than_a_launch_holds():
    _run([32_769 + 2 * j for j in range(20)] + [5, 200], 6, 3)
    _run([32_769, 70_001, 8, 9], 6, 3)              # too few elements in all: the table-driven launch


def test_many_tiles_per_warp():
    _run([3_000_001, 5_000_003], 4, 8)


def test_only_those_off_the_boundaries():
    """So many codes on the 16-byte boundaries that they keep their own launch, and the short tensors ride along with it."""
    _run([8_388_608, 6, 40_002, 33_000, 500, 1_000_005, 9], 8, 8)
    _run([300, 33_000, 8_388_600 + 32_768] + [32_769] * 17, 8, 8)
