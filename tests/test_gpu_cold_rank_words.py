"""The index-only calls on both sides of the sizes at which a thread of the cold-row ranking takes eight words of the bitmap
instead of four (2^24 rows with at most 65 536 lookups, 2^25 with more), and where the last tile of such threads is full or has
one word."""
import pytest
import test_gpu_index_shapes as shapes

pytestmark = pytest.mark.gpu

FULL = 257 * 2048 * 32                                       # 257 tiles of 2 048 words
CASES = {
    "full_tiles": ([1 << 23, FULL - (1 << 23)], 3000, 1, 1, 1, 0.005),
    "one_word_more": ([1 << 23, FULL + 1 - (1 << 23)], 3000, 1, 1, 1, 0.005),
    "2^25_rows_65538_lookups": ([1 << 24] * 2, 32769, 1, 1, 1, 0.005),
    "2^25_and_1_rows_65538_lookups": ([1 << 24, (1 << 24) + 1], 32769, 1, 1, 1, 0.005),
    "2^25_rows_65536_lookups": ([1 << 24] * 2, 32768, 1, 1, 1, 0.005),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_index_calls(case, monkeypatch):
    monkeypatch.setitem(shapes.CASES, case, CASES[case])
    shapes.test_index_calls(case)
