"""The backward call on runs at the length where it changes how a run is finished: up to 32 chunks on, the sum kernel
finds a run's last chunk itself and one warp adds its pieces; from there on a CTA searches the end and adds them.
Integer data, so the updated rows must equal the oracle's bit for bit."""
import numpy as np
import pytest

from oracle import hotline_oracle as orc
from test_gpu_backward_runs import _backward, _lookups

pytestmark = pytest.mark.gpu

CASES = {
    "last_with_known_end": [1024, 5],
    "first_searched": [7, 1025 + 24, 1057, 3],
    "whole_list": [33 * 32],
    "several": [1100, 3, 2000, 1100, 40, 5000, 64, 1],
    "across_many_ctas": [9, 70_000, 2],
}


@pytest.mark.parametrize("dim", [4, 32, 36, 128, 512])
@pytest.mark.parametrize("case", sorted(CASES))
def test_backward_on_runs_of_many_chunks(case, dim):
    import paper_2204_05436_b200 as hl
    if dim == 512 and case == "across_many_ctas":
        pytest.skip("the same path at a quarter of the row width")
    ids, offsets, rows = _lookups(CASES[case], seed=dim)
    rng = np.random.default_rng(dim + 1)
    cache = rng.integers(-8, 9, (rows, dim)).astype(np.float32)
    grad = rng.integers(-4, 5, (len(ids), dim)).astype(np.float32)
    want1 = cache.copy()
    orc.embbag_bwd_sgd(want1, ids, offsets, grad, 0.5)
    want2 = want1.copy()
    orc.embbag_bwd_sgd(want2, ids, offsets, grad, 0.5)
    got1, got2 = _backward(hl, ids, offsets, cache, grad, 0.5)
    assert np.array_equal(got1, want1)
    assert np.array_equal(got2, want2), "second call on the same context differs"
