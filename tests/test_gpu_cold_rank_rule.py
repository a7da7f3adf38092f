"""The index-only calls on both sides of the sizes at which the cold-row ranking reads the bitmap through its summary: 2^24 rows
with at most 4 096 lookups, 2^26 with more."""
import pytest
import test_gpu_index_shapes as shapes

pytestmark = pytest.mark.gpu

CASES = {
    "16777216_rows_4096_lookups": ([1 << 23] * 2, 2048, 1, 1, 1, 0.005),
    "16777217_rows_4096_lookups": ([1 << 23, (1 << 23) + 1], 2048, 1, 1, 1, 0.005),
    "16777217_rows_4098_lookups": ([1 << 23, (1 << 23) + 1], 2049, 1, 1, 1, 0.005),
    "67108864_rows_4098_lookups": ([1 << 25] * 2, 2049, 1, 1, 1, 0.005),
    "67108865_rows_4098_lookups": ([1 << 25, (1 << 25) + 1], 2049, 1, 1, 1, 0.005),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_index_calls(case, monkeypatch):
    monkeypatch.setitem(shapes.CASES, case, CASES[case])
    shapes.test_index_calls(case)
