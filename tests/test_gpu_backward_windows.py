"""The backward call on runs at the borders of the sum kernel's windows (256 lookups, a CTA's): runs that end at a window's last
lookup, start at its first, go on for up to 32 lookups of the next one (finished there), for more (partial sums), over whole
windows, and for more windows than the sum kernel looks ahead; and lists of random runs.  Integer data, so the updated rows
must equal the oracle's bit for bit."""
import numpy as np
import pytest

from oracle import hotline_oracle as orc
from test_gpu_backward_runs import _backward, _lookups

pytestmark = pytest.mark.gpu

RNG = np.random.default_rng(5)
CASES = {
    "whole_windows": [256, 256, 512, 1, 255, 768, 256],
    "one_more_or_less": [255, 2, 255, 257, 255, 511, 2, 513, 3],
    "into_the_first_chunk": [250, 6 + 31, 219 + 32, 5, 219 + 33, 200, 56 + 32, 224 + 1, 300, 7],
    "ends_at_the_chunk_behind": [200, 88, 224, 256 + 32, 224, 256 + 33, 223, 256 + 31, 3],
    "from_a_window_before_the_last": [100, 600, 44, 300, 20, 1000, 8],
    "chunks_of_a_window": [10, 54, 30, 34, 64, 96, 95, 97, 33, 31, 1, 127, 129, 160],
    "known_and_searched_end": [5, 31 * 256 + 200, 40, 32 * 256, 3, 33 * 256 + 1, 9],
    "random_short": RNG.integers(1, 90, 400).tolist(),
    "random_long": np.minimum(RNG.zipf(1.3, 500), 5000).tolist(),
}


@pytest.mark.parametrize("dim", [4, 20, 64, 128, 256, 512, 1024])
@pytest.mark.parametrize("case", sorted(CASES))
def test_backward_on_runs_at_the_borders_of_windows(case, dim):
    import paper_2204_05436_b200 as hl
    if dim > 256 and sum(CASES[case]) > 10_000:
        pytest.skip("the same path at narrower rows")
    ids, offsets, rows = _lookups(CASES[case], seed=dim)
    rng = np.random.default_rng(dim + 1)
    cache = rng.integers(-8, 9, (rows, dim)).astype(np.float32)
    grad = rng.integers(-4, 5, (len(ids), dim)).astype(np.float32)
    want1 = cache.copy()
    orc.embbag_bwd_sgd(want1, ids, offsets, grad, 0.5)
    want2 = want1.copy()
    orc.embbag_bwd_sgd(want2, ids, offsets, grad, 0.5)
    got1, got2 = _backward(hl, ids, offsets, cache, grad, 0.5)
    assert np.array_equal(got1, want1), f"{int((got1 != want1).any(axis=1).sum())} rows differ"
    assert np.array_equal(got2, want2), "second call on the same context differs"
