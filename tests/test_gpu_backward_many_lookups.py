"""The backward call on both sides of the number of lookups from which rows of 36 to 64 fp32 are summed with four CTAs per
multiprocessor (a chunk of 32 lookups for every warp of three): the run lengths that hit the chunk borders, over and over, at
that number, one more, and a ragged end.  Integer data, so the updated rows must equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

from oracle import hotline_oracle as orc
from test_gpu_backward_runs import CASES, _backward, _lookups

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [32, 36, 52, 64])
@pytest.mark.parametrize("more", [0, 1, 26_341])
def test_backward_of_many_lookups(dim, more):
    import paper_2204_05436_b200 as hl
    n = 3 * 8 * 32 * torch.cuda.get_device_properties(0).multi_processor_count + more
    rng = np.random.default_rng(n + dim)
    lengths = []
    while sum(lengths) < n:
        lengths += CASES[sorted(CASES)[int(rng.integers(len(CASES)))]]
    while sum(lengths) > n:
        lengths[-1] -= min(lengths[-1], sum(lengths) - n)
        lengths = [x for x in lengths if x]
    ids, offsets, rows = _lookups(lengths, seed=dim)
    cache = rng.integers(-8, 9, (rows, dim)).astype(np.float32)
    grad = rng.integers(-4, 5, (len(ids), dim)).astype(np.float32)
    want1 = cache.copy()
    orc.embbag_bwd_sgd(want1, ids, offsets, grad, 0.5)
    want2 = want1.copy()
    orc.embbag_bwd_sgd(want2, ids, offsets, grad, 0.5)
    got1, got2 = _backward(hl, ids, offsets, cache, grad, 0.5)
    assert np.array_equal(got1, want1)
    assert np.array_equal(got2, want2), "second call on the same context differs"
