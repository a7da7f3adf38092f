"""The schedules' sort of every table's pairs by themselves, at the sizes where it changes: pairs of a table for a cluster of 4,
8 and 16 CTAs, of CTAs with 512 threads, and for the chained passes; tables that hold more lookups than their cluster, in mini-batches of
as many lookups as bags (sorted through memory, in one to four passes), and others of uneven tables, which the chained passes or one
cluster sort; tables without any lookup; mini-batches that go one way and the other in turn.  Whole pipelines with both orders of a
step, integer data, so that every row must equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

from oracle import hotline_oracle as orc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# name: (rows of each table, batch, lookups per bag of each table (low, high), share of hot rows)
CASES = {
    "avg_8192": ([40_000, 50, 3000], 8192, [(1, 1)] * 3, 0.8),
    "avg_8193": ([40_000, 50, 3000], 8193, [(1, 1)] * 3, 0.8),
    "avg_16385": ([90_000, 700], 16385, [(1, 1)] * 2, 0.9),
    "avg_32769": ([90_000, 700], 32769, [(1, 1)] * 2, 0.9),
    "avg_65537": ([90_000, 700], 65537, [(1, 1)] * 2, 0.9),
    "bags_of_several": ([5000] * 5, 1000, [(0, 6)] * 5, 0.95),                 # (the chained passes)
    "one_large_table_one_pass": ([3] * 20, 2000, [(0, 1), (8, 14)] + [(0, 0)] * 16 + [(0, 1)] * 2, 0.9),
    "one_large_table_two_passes": ([700, 6000] + [10] * 20, 2000, [(1, 1), (8, 14), (0, 1)] + [(0, 0)] * 19, 0.99),
    "one_large_table_three_passes": ([90_000] + [500] * 19, 2000, [(8, 14), (1, 1)] + [(0, 0)] * 17 + [(0, 1)], 0.5),
    "one_large_table_8_ctas": ([50_000, 5], 16_384, [(2, 2), (0, 0)], 0.9),
    "one_large_table_16_ctas": ([50_000, 5], 20_001, [(2, 2), (0, 0)], 0.95),
    # (as many lookups as bags, all of them in one table: through memory, one to four digits, CTAs of 256 and of 512 threads)
    "one_full_table_one_pass": ([3] * 20, 2000, [(20, 20)] + [(0, 0)] * 19, 0.9),
    "one_full_table_two_passes": ([700, 6000] + [10] * 18, 2000, [(0, 0), (20, 20)] + [(0, 0)] * 18, 0.99),
    "one_full_table_three_passes": ([90_000] + [500] * 19, 2001, [(20, 20)] + [(0, 0)] * 19, 0.5),
    "one_full_table_four_passes": ([30] * 3 + [17_000_000] + [30] * 4, 2000, [(0, 0)] * 3 + [(8, 8)] + [(0, 0)] * 4, 1.0),
    "one_full_table_512_threads": ([90_000, 700], 33_000, [(2, 2), (0, 0)], 0.9),
    "one_full_table_512_threads_last": ([700, 90_000], 65_536, [(0, 0), (2, 2)], 0.6),
    "all_popular": ([9000] + [10] * 15, 3000, [(5, 9), (1, 1), (0, 1)] + [(0, 0)] * 13, 1.0),
    "one_table": ([20_000], 5000, [(1, 1)], 0.5),
    # (mini-batches in turn: as many lookups as bags, and fewer, which the chained passes or one cluster sort)
    "both_ways_short": ([4000, 60, 900], 3000, [[(1, 1)] * 3, [(3, 5), (0, 0), (0, 0)]], 0.9),
    "both_ways_long": ([40_000, 50, 3000], 14_000, [[(0, 1), (1, 1), (0, 1)], [(1, 1)] * 3], 0.8),
}


@pytest.mark.parametrize("order", ["fig8", "eq5"])
@pytest.mark.parametrize("case", sorted(CASES))
def test_pipeline_over_tables_of_many_sizes(case, order):
    import paper_2204_05436_b200 as hl
    rows, B, spans, hot = CASES[case]
    T, N, D, lr, steps = len(rows), int(sum(rows)), 4, 0.125, 4
    rng = np.random.default_rng(len(case))
    base = np.concatenate([[0], np.cumsum(rows)])
    batches = []
    for k in range(steps):
        lengths = np.concatenate([rng.integers(lo, hi + 1, B) for lo, hi in (spans[k % 2] if isinstance(spans[0], list) else spans)])
        offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
        r = np.repeat(np.repeat(rows, B), lengths)
        limit = np.where(rng.random(len(r)) < 0.5, np.minimum(r, 20), r)          # half of them on a few rows
        batches.append(((rng.random(len(r)) * limit).astype(np.int32), offsets))
    hot_rows = np.sort(rng.choice(N, max(1, int(N * hot)), replace=False))
    remap = orc.build_remap(hot_rows, N)
    hot_cap, max_nnz = len(hot_rows), max(len(b[0]) for b in batches)
    window = max(1, min(N, max_nnz))
    table0 = rng.integers(-8, 9, (N, D)).astype(np.float32)
    table_o, cache_o = table0.copy(), np.zeros((hot_cap + window, D), dtype=np.float32)
    cache_o[:hot_cap] = table0[hot_rows]
    grads, pooled = [], []
    for idx, off in batches:
        perm, n_pop, O, X, _ = orc.fragment(idx, off, B, rows, remap, 1)
        g = rng.integers(-3, 4, (T * B, D)).astype(np.float32)
        g_pop, g_non = g[:T * n_pop], g[T * n_pop:]
        if order == "fig8":
            out = orc.hotline_step(table_o, cache_o, hot_cap, remap, idx, off, B, rows, 1, g_pop, g_non, lr)
            pooled.append(out[5:7])
        else:
            C, x = orc.gather_cold(X.ids, remap, hot_cap)
            cache_o[hot_cap:hot_cap + len(C)] = orc.stage_cold_rows(table_o, C)
            pooled.append((orc.embbag_fwd(cache_o, O.ids, O.offsets), orc.embbag_fwd(cache_o, x, X.offsets)))
            orc.embbag_bwd_sgd(cache_o, np.concatenate([O.ids, x]), np.concatenate([O.offsets, X.offsets[1:] + len(O.ids)]),
                               g, lr)
            orc.scatter_cold(table_o, C, cache_o[hot_cap:hot_cap + len(C)])
        zeros = np.zeros((T * B, D), dtype=np.float32)
        if order == "fig8":
            gp, gn = zeros.copy(), zeros.copy()
            gp[:len(g_pop)], gn[:len(g_non)] = g_pop, g_non
        else:
            gp, gn = g, None
        grads.append((torch.from_numpy(gp).to(DEV), None if gn is None else torch.from_numpy(gn).to(DEV)))
    assert base[-1] == N
    host = torch.from_numpy(table0.copy()).pin_memory()
    p = hl.NativePipelinedHotline(rows, D, 1, B, max_nnz, hot_cap, window, host, order=order)
    try:
        with torch.cuda.stream(p.main):
            p.set_hot_rows(torch.from_numpy(hot_rows.astype(np.int32)).to(DEV))
            p.build_remap(load_rows=True)
            d = [(torch.from_numpy(i).to(DEV), torch.from_numpy(o).to(DEV), B, None) for i, o in batches]
            torch.cuda.synchronize()
            p.start(*d[0], more=d[1:p.lookahead])
            for k in range(steps):
                nxt = d[k + p.lookahead] if k + p.lookahead < steps else None
                s = p.sets[p.step(*grads[k], lr, next_batch=nxt)]
                p.drain()
                want_pop, want_non = pooled[k]
                assert np.array_equal(s.pooled_pop.cpu().numpy()[:len(want_pop)], want_pop), k
                assert np.array_equal(s.pooled_non.cpu().numpy()[:len(want_non)], want_non), k
        p.status()
        assert np.array_equal(p.cache[:hot_cap].cpu().numpy(), cache_o[:hot_cap])
        assert np.array_equal(host.numpy(), table_o)
    finally:
        p.close()
