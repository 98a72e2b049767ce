"""Long segments that start off a 16-byte boundary, encoded by rows of the whole gradient: every remainder of the start, ends
inside and at the end of a row and of the gradient, neighbours that hold infinities and NaN, streams at odd words, more pairs
than a launch holds, and the calls that keep the table kernel; bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import paper_1804_08066_b200 as mqg
from oracle import mqg_oracle as O
from paper_1804_08066_b200 import workloads as wl
from tests.gpu_util import Guarded, bits_equal, to_dev

pytestmark = pytest.mark.gpu


def _run(sizes, bits, W, bf16, offset=0, gap=0, begin=0, norm=False, poison=False):
    seg = np.concatenate([[begin], begin + np.cumsum(sizes)]).astype(np.uint64)
    code = np.concatenate([[0], np.cumsum([O.code_words(s, bits) + gap for s in sizes])]).astype(np.uint64)
    xs = [np.concatenate([np.zeros(begin, np.float32), wl.layered(sizes, config=3, worker=w)]) for w in range(W)]
    for x in xs:
        for j in range(0, len(sizes), 3):                          # the maxima in the first and in the last element
            x[int(seg[j])] = 1.0
            x[int(seg[j + 1]) - 1] = -1.0
    if bf16:
        xs = [wl.f32_to_bf16_bits(x) for x in xs]
    dt = "bf16" if bf16 else "f32"
    grads = [to_dev(x.view(np.int16)).view(torch.bfloat16) if bf16 else to_dev(x) for x in xs]
    codes = [Guarded(int(code[-1]), torch.int32) for _ in range(W)]
    scales = [Guarded(len(sizes), torch.float32) for _ in range(W)]
    if norm:
        ws = torch.empty(max(1, mqg.mqg_l2_workspace_floats(seg)), dtype=torch.float32, device="cuda")
        mqg.mqg_quantize_segments_l2(grads[0], seg, code, bits, 5, codes[0].view, scales[0].view, ws, worker=2, step=1,
                                     elem_offset=offset)
    else:
        mqg.mqg_quantize_segments_workers(grads, W, seg, code, bits, 5, [c.view for c in codes], [s.view for s in scales],
                                          first_worker=2, step=1, elem_offset=offset)
    torch.cuda.synchronize()
    ref = O.quantize_segments_l2 if norm else O.quantize_segments
    for w in range(W):
        codes[w].check_guards(), scales[w].check_guards()
        c_ref, s_ref = ref(xs[w], seg, code, bits, seed=5, worker=2 + w, step=1, elem_offset=offset, dtype=dt)
        assert bits_equal(scales[w].numpy(np.float32), s_ref) == 0
        got = codes[w].numpy(np.uint32)
        for j, s in enumerate(sizes):
            lo, nw = int(code[j]), O.code_words(s, bits)
            assert np.array_equal(got[lo:lo + nw], c_ref[lo:lo + nw]), (w, j)
            assert (got[lo + nw:int(code[j + 1])] == 0x7FC0DEAD).all()
    assert mqg.mqg_device_timeouts() == 0


@pytest.mark.parametrize("bits", range(1, 9))
@pytest.mark.parametrize("bf16", [False, True])
def test_starts_and_ends(bits, bf16):
    # 124 rows of 32 (64) elements to a tile; sums to starts at many remainders, ends in the middle and at row ends
    sizes = [100_001, 124 * 64 * 3 + 1, 33, 124 * 64 * 4 - 2, 70_031, 31 * 64 * 5 + 17, 20_000, 99_999]
    _run(sizes, bits, 2, bf16)


@pytest.mark.parametrize("first", range(1, 64, 3))
def test_every_remainder(first):
    _run([first, 70_000, 66_000 - first, 65_541], 5, 1, first % 2 == 0, gap=first % 3)


@pytest.mark.parametrize("bits,bf16", [(8, False), (3, True), (8, True)])
def test_neighbours_do_not_matter(bits, bf16):
    """A segment between two that hold infinities and NaN next to it."""
    sizes = [70_003, 70_001, 70_002]
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    code = np.concatenate([[0], np.cumsum([O.code_words(s, bits) for s in sizes])]).astype(np.uint64)
    x = wl.layered(sizes, config=3, worker=0)
    clean = wl.f32_to_bf16_bits(x) if bf16 else x.copy()
    x[70_003 - 40:70_003] = np.inf
    x[140_004:140_050] = np.nan
    dirty = wl.f32_to_bf16_bits(x) if bf16 else x
    out = []
    for v in (clean, dirty):
        g = to_dev(v.view(np.int16)).view(torch.bfloat16) if bf16 else to_dev(v)
        c, s = Guarded(int(code[-1]), torch.int32), Guarded(3, torch.float32)
        mqg.mqg_quantize_segments(g, seg, code, bits, 5, c.view, s.view)
        torch.cuda.synchronize()
        c.check_guards()
        out.append((c.numpy(np.uint32)[int(code[1]):int(code[2])].copy(), s.numpy(np.float32)[1]))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


def test_more_pairs_than_a_launch_and_both_kinds():
    _run([65_537, 70_000, 65_600, 65_601] * 3, 4, 8, False)          # 96 pairs, some aligned


def test_norm():
    _run([65_537, 70_000, 130_001, 9], 6, 1, False, norm=True)


@pytest.mark.parametrize("offset,begin", [(8, 0), (3, 0), (64, 64), (0, 5), ((1 << 35) - 8 * 1000, 0)])
def test_offsets_and_first_segments(offset, begin):
    _run([65_537, 70_001], 4, 2, False, offset=offset, begin=begin)
    _run([65_537, 70_001], 4, 1, True, offset=offset, begin=begin)
