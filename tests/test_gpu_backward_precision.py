"""How exact the backward's sums are: runs whose gradient rows nearly cancel, over several chunks of a window of 256 lookups or into
the next window's first chunk.  Such a run is summed in fp64 throughout, whatever the width of a row, so the gradient that
reaches the row is the exact sum, rounded once."""
import numpy as np
import pytest

from test_gpu_backward_runs import _backward, _lookups

pytestmark = pytest.mark.gpu

# (256 lookups a window; none of the runs has more than 32 in the window behind the one it starts in)
RUNS = [33, 64, 63, 40, 56, 96, 160, 34, 62, 33, 64, 63, 20, 236 + 20, 180, 56 + 32, 224, 5]


@pytest.mark.parametrize("dim", [4, 20, 64, 128, 132, 256, 260, 512, 516, 1024])
def test_runs_inside_a_window_are_rounded_once(dim):
    import paper_2204_05436_b200 as hl
    ids, offsets, rows = _lookups(RUNS, seed=dim)
    rng = np.random.default_rng(dim)
    grad = (1e4 * rng.standard_normal((len(ids), dim))).astype(np.float32)
    for r in range(len(RUNS)):               # the second half of a run takes back the first, but for about one
        at = np.flatnonzero(ids == 3 * r + 1)
        half = len(at) // 2
        grad[at[half:2 * half]] = rng.standard_normal((half, dim)).astype(np.float32) - grad[at[:half]]
    cache = np.zeros((rows, dim), dtype=np.float32)
    got, _ = _backward(hl, ids, offsets, cache, grad, 0.5)
    for r in range(len(RUNS)):
        g = grad[ids == 3 * r + 1].astype(np.float64)
        want = g.sum(0)
        # one rounding to fp32 (2^-24), and those of an fp64 sum of so many numbers (2^-53 of all of them each)
        bound = np.abs(want) * 2.0 ** -24 + np.abs(g).sum(0) * len(g) * 2.0 ** -53
        error = np.abs(got[3 * r + 1].astype(np.float64) / -0.5 - want)
        assert (error <= bound).all(), (r, RUNS[r], float((error / bound).max()))
