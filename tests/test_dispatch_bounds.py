"""What the library's host code decides before it launches, asked of its own functions (no GPU): the shapes that the one-pass
quantizers take (the L2-norm kernels have tiles of at most 256 rows, the others of 512), and the CTAs of a table's tensors."""
import ctypes as C
import random

import pytest

import paper_1804_08066_b200 as mqg

N = 1 << 20


def _applies(symbol, *args):
    f = getattr(C.CDLL(mqg.LIB_PATH), symbol)
    f.restype, f.argtypes = C.c_bool, [t for t, _ in args]
    return f(*(v for _, v in args))


def _one(name, *u64):
    return _applies("_ZN3mqg%d%sE%s" % (len(name), name, "m" * len(u64)), *((C.c_uint64, v) for v in u64))


def _workers(n, bucket, mode, offset=0):
    return _applies("_ZN3mqg24quantize_workers_appliesEimmmi", (C.c_int, 8), (C.c_uint64, n), (C.c_uint64, bucket),
                    (C.c_uint64, offset), (C.c_int, mode))


@pytest.mark.parametrize("n,bucket,norm,others", [
    (N, 8192, True, True), (N, 7168, True, True), (8192, 8192, True, True), (8160, N, False, False), (8192, N, True, True),
    (N, 9216, False, True), (N, 16384, False, True), (16384, 16384, False, True), (9216, N, False, True),
    (N, 17408, False, False), (17408, N, False, False)])
def test_bucket_bounds(n, bucket, norm, others):
    assert _one("quantize_norm_fused_applies", n, bucket, 0) == norm
    assert _workers(n, bucket, 2) == norm
    assert _one("quantize_long_fused_applies", n, bucket, 0) == others
    assert _one("quantize_range_fused_applies", n, bucket) == others
    assert _workers(n, bucket, 0) == _workers(n, bucket, 1) == others
    assert not _workers(n, bucket, 0, offset=3) and not _one("quantize_norm_fused_applies", n, bucket, 3)


class _Spans(C.Structure):
    _fields_ = [("bucket", C.c_uint64), ("n", C.c_uint64), ("nspan", C.c_int), ("first", C.c_int), ("clear", C.c_uint32 * 2),
                ("scale_idx", C.c_uint32 * 64), ("elem0", C.c_uint64 * 64), ("len", C.c_uint64 * 64), ("code0", C.c_uint64 * 64)]


class _Joined(C.Structure):
    _fields_ = [("spans", _Spans), ("cta", C.c_uint16 * 512), ("parts", C.c_uint8 * 64)]


def _random_sizes(seed):
    rng = random.Random(seed)
    return [rng.choice((0, 1, 8192, 8193, 16384, 16385, 65536, rng.randrange(65537))) for _ in range(rng.randint(1, 64))]


@pytest.mark.parametrize("alone", [8192, 16384])
@pytest.mark.parametrize("sizes", [[9000] * 63 + [60000], [17000] * 63 + [60000], [9000] * 32 + [33000] * 32, [20000], [65536] * 64,
                                   [100, 40000, 0], *map(_random_sizes, range(20))])
def test_ctas_of_joined_tensors(sizes, alone):
    """Every tensor once, in CTAs of one cluster, none of them shared, and no more CTAs than the parts and what fills clusters up."""
    spans, tab, cluster = _Spans(nspan=len(sizes)), _Joined(), C.c_uint()
    for j, n in enumerate(sizes):
        spans.len[j] = n
    place = C.CDLL(mqg.LIB_PATH)["_ZN3mqg18place_joined_spansERKNS_9SpanTableEmRNS_11JoinedTableERj"]
    place.restype, place.argtypes = C.c_uint, [C.c_void_p, C.c_uint64, C.c_void_p, C.c_void_p]
    ctas = place(C.byref(spans), alone, C.byref(tab), C.byref(cluster))
    need = [1 if n <= alone else -(-n // 8192) for n in sizes]
    size = cluster.value
    assert size == max(need) and ctas % size == 0 and list(tab.parts[:len(sizes)]) == need
    seen = []
    for first in range(0, ctas, size):
        placed = [divmod(c, 256)[::-1] for c in tab.cta[first:first + size] if c != 0xFFFF]
        seen += placed
        spans_here = [j for j, part in placed if part == 0]
        assert placed == [(j, part) for j in spans_here for part in range(need[j])]       # whole tensors, parts in order
        assert len({need[j] == 1 for j in spans_here}) == 1                               # none that waits for a lone one
    assert sorted(seen) == [(j, part) for j in range(len(sizes)) for part in range(need[j])]
    assert ctas <= 2 * sum(need) + 2 * size                                               # half of every cluster but the last


@pytest.mark.parametrize("on,off,W,bits,form", [
    (50_000_000, 40_000, 8, 4, 1), (50_000_000, 40_000, 8, 8, 1), (16_777_216, 40_000, 16, 4, 1),
    (8_388_608, 40_000, 8, 4, 2), (8_388_607, 2_000_000, 8, 8, 2), (100_000_000, 40_000, 4, 8, 2), (0, 50_000_000, 8, 8, 2),
    (50_000_000, 0, 8, 8, 0), (0, 0, 1, 1, 0), (400_000, 600_000, 8, 8, 0), (400_000, 700_000, 8, 8, 2), (0, 524_288, 4, 2, 2),
    (0, 524_287, 4, 2, 0)])
def test_tensors_off_the_boundaries(on, off, W, bits, form):
    """A few elements off the 16-byte boundaries do not take many away from the kernel for those on them."""
    f = C.CDLL(mqg.LIB_PATH)["_ZN3mqg16flat_server_formEmmii"]
    f.argtypes = [C.c_uint64, C.c_uint64, C.c_int, C.c_int]
    assert f(on, off, W, bits) == form


@pytest.mark.parametrize("n,bucket,W,bits,warps", [
    (1_100_000, 2048, 8, 2, True), (1_500_000, 1024, 1, 3, True), (1_100_000, 1024, 1, 6, False), (1_600_000, 1024, 1, 3, False),
    (25_000_000, 2048, 8, 4, True), (25_000_000, 2048, 4, 2, False), (9_000_000, 2048, 8, 2, True), (25_000_000, 2048, 8, 2, False),
    (6_000_000, 8192, 4, 4, False), (6_000_000, 8192, 16, 4, False), (4_000_000, 8192, 8, 4, True), (8_000_000, 8192, 8, 4, True),
    (8_000_000, 8192, 4, 8, False), (700_000, 768, 1, 4, False), (700_000, 768, 8, 4, True), (700_000, 3072, 1, 4, True),
    (4_000_000, 1536, 8, 4, True), (4_000_000, 1536, 8, 3, False), (25_000_000, 1056, 8, 4, False)])
def test_kernel_of_the_requantization(n, bucket, W, bits, warps):
    f = C.CDLL(mqg.LIB_PATH)["_ZN3mqg23requantize_warp_appliesEmmii"]
    f.restype, f.argtypes = C.c_bool, [C.c_uint64, C.c_uint64, C.c_int, C.c_int]
    assert f(n, bucket, W, bits) == warps
