"""Per-layer calls whose longest tensor needs a cluster of two, four or eight CTAs, with shorter ones of every need beside it:
bit for bit against the CPU checker (see test_joined_spans_gpu.py)."""
import pytest

from tests import test_joined_spans_gpu as joined

pytestmark = pytest.mark.gpu

SIZES = {
    "clusters_of_two": [16_384, 8193, 9_001, 16_383, 100],
    "clusters_of_four": [32_768, 16_385, 24_577, 8193, 31, 32_767, 24_576],
    "clusters_of_eight": [32_769, 40_961, 65_535, 57_345, 16_385, 8192, 1],
}


@pytest.mark.parametrize("name", SIZES)
@pytest.mark.parametrize("bits,bf16,W", [(4, False, 3), (2, True, 2), (8, False, 1)])
def test_max_abs(monkeypatch, name, bits, bf16, W):
    monkeypatch.setitem(joined.SIZES, name, SIZES[name])
    joined.test_max_abs(name, bits, bf16, W)


@pytest.mark.parametrize("name", SIZES)
def test_norm(monkeypatch, name):
    monkeypatch.setitem(joined.SIZES, name, SIZES[name])
    joined.test_norm(name)
