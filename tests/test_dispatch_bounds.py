"""Which shapes the one-pass quantizers take, asked of the library's own predicates (no GPU): the L2-norm kernels have tiles of
at most 256 rows, the others of 512."""
import ctypes as C

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
