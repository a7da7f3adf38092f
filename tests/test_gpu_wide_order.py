"""The wide-id cold-row search at the sizes where it changes its launch: rows of up to 32 bits sorted as they are, more by
their lower and then their upper part; the sort in one cluster (at most 32 768 lookups) or in tiles; rank tiles of 1 024
lookups.  Against a direct computation on 64-bit rows (no table of that size is allocated, nor an array over its rows)."""
import numpy as np
import pytest
import torch

from test_gpu_wide import _t, _Wide

pytestmark = pytest.mark.gpu

# rows of each table, batch, share of lookups on hot rows, distinct rows looked up per table
CASES = {
    "no_cold_lookup": ([2_000_000_000, 50], 64, 1.0, 1000),
    "one_tile": ([2_147_483_647, 2_147_483_647, 1], 341, 0.0, 1 << 30),          # 2^32 - 1 rows, 1 023 lookups
    "tile_and_one": ([2_147_483_647, 2_147_483_647, 2], 342, 0.0, 100),          # 2^32 rows: the last of 32 bits
    "upper_bits_cluster": ([2_147_483_647, 2_147_483_647, 3], 2000, 0.3, 4000),  # 2^32 + 1 rows
    "upper_bits_tiles": ([2_000_000_000] * 9, 4097, 0.2, 20_000),
    "lower_bits_tiles": ([500_000_000] * 8, 4097, 0.2, 20_000),
    "one_a_lane_last": ([500_000_000] * 8, 10_240, 0.3, 20_000),                 # classified: one lookup a lane up to 81 920
    "four_a_lane_first": ([500_000_000] * 8, 10_241, 0.3, 20_000),
    "four_a_lane": ([2_000_000_000] * 3, 65_537, 0.1, 1 << 30),
    "many_upper_values": ([2_147_483_647] * 255, 300, 0.1, 500),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_cold_rows_and_slots(case):
    import paper_2204_05436_b200 as hl
    rows, B, hot_share, distinct = CASES[case]
    T = len(rows)
    base = np.concatenate([[0], np.cumsum(np.asarray(rows, dtype=np.int64))])
    rng = np.random.default_rng(len(case))
    pool = [np.unique(np.concatenate([rng.integers(0, r, min(distinct, 40_000)), [0, r - 1]])) for r in rows]
    hot = np.sort(np.concatenate([base[t] + rng.choice(p, (len(p) + 1) // 2, replace=False) for t, p in enumerate(pool)]))
    indices = np.empty((T, B), dtype=np.int32)
    for t, p in enumerate(pool):
        is_hot = np.isin(base[t] + p, hot)
        cold_p = p[~is_hot] if (~is_hot).any() else p
        indices[t] = np.where(rng.random(B) < hot_share, rng.choice(p[is_hot], B), rng.choice(cold_p, B))
    indices = indices.reshape(-1)
    offsets = np.arange(T * B + 1, dtype=np.int32)
    nnz = T * B
    wd = _Wide(hl, rows, 1, B, nnz, len(hot), nnz, counter_slots=1 << 10)
    try:
        wd.hot_rows.copy_(_t(hot))
        wd.n_hot.fill_(len(hot))
        hl.hl_wide_build_remap(wd.w, wd.hot_rows, wd.n_hot, wd.stream)
        g = base[np.repeat(np.arange(T), B)] + indices
        slot = np.searchsorted(hot, g)
        is_hot = hot[np.minimum(slot, len(hot) - 1)] == g
        non = np.flatnonzero(~is_hot.reshape(T, B).all(axis=0))
        X = g.reshape(T, B)[:, non].reshape(-1)
        x_hot = is_hot.reshape(T, B)[:, non].reshape(-1)
        C = np.unique(X[~x_hot])
        want = np.where(x_hot, np.searchsorted(hot, X), len(hot) + np.searchsorted(C, X))

        class Batch:
            pass
        b = Batch()
        b.indices, b.offsets = indices, offsets
        for _ in range(2):
            wd.index(b)
            assert int(wd.n_cold) == len(C)
            assert np.array_equal(wd.non_rows[:len(X)].cpu().numpy(), X)
            assert np.array_equal(wd.cold_rows[:len(C)].cpu().numpy(), C)
            assert np.array_equal(wd.non_slots[:len(X)].cpu().numpy(), want)
    finally:
        wd.close()
