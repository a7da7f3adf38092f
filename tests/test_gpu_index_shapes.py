"""The index-only calls (fragment, cold-row search, sort) at the sizes where they change their launch: bags per tile (512
once there is a 256-bag tile per multiprocessor, 1 024 once there is one of those), lists of lookups for bags of several, long bags in the popularity test,
words per thread and the summary bitmap of the cold-row ranking, and the sort in one cluster (up to 32 768 lookups) or in
tiles.  All outputs are integers and must equal the oracle's."""
import numpy as np
import pytest
import torch

from oracle import hotline_oracle as orc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# name: (rows of each table, batch, bags per sample, bag length low / high, share of hot rows)
CASES = {
    "one_input_one_lookup": ([50], 1, 1, 1, 1, 0.5),
    "inputs_33_ragged": ([100, 7, 3000], 33, 1, 0, 3, 0.8),
    "tiles_of_256_last_full": ([997] * 37, 1024, 1, 1, 1, 0.97),        # 37 888 bags: 148 tiles of 256
    "tiles_of_1024": ([997] * 37, 1025, 1, 0, 2, 0.97),
    "tiles_of_512_last_full": ([997] * 37, 4096, 1, 1, 1, 0.97),         # 151 552 bags: 148 tiles of 1 024
    "tiles_of_1024_from_here": ([997] * 37, 4097, 1, 0, 2, 0.97),
    "tiles_of_1024_mostly_popular": ([997] * 37, 4099, 1, 1, 1, 0.9999),
    "tiles_of_256_some_longer": ([997] * 3, 1025, 1, 0, 2, 0.9),
    "lists_short": ([997] * 20, 2049, 1, 0, 9, 0.98),
    "lists_of_up_to_129": ([997] * 2, 333, 2, 0, 4, 0.98),
    "lists_long": ([997], 40_000, 1, 0, 20, 0.95),
    "few_tables_long_bags": ([100_003] * 2, 65, 1, 0, 700, 0.999),
    "sort_32768": ([5000] * 8, 4096, 1, 1, 1, 0.9),
    "sort_32776": ([5000] * 8, 4097, 1, 1, 1, 0.9),
    "rank_four_words": ([1_300_000] * 4, 700, 1, 0, 4, 0.3),
    "rank_67108864_rows": ([1 << 25] * 2, 500, 1, 1, 2, 0.005),
    "rank_summary": ([1 << 25, (1 << 25) + 1], 500, 1, 1, 2, 0.005),
    "rank_summary_four_words": ([60_000_001] * 2, 3000, 1, 0, 3, 0.001),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_index_calls(case):
    import paper_2204_05436_b200 as hl
    rows, B, S, lo, hi, hot = CASES[case]
    T, N = len(rows), int(sum(rows))
    rng = np.random.default_rng(len(case))
    lengths = rng.integers(lo, hi + 1, T * B * S)
    offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    nnz = int(offsets[-1])
    table = np.repeat(np.arange(T * B * S) // (B * S), lengths)
    # half of the lookups on a table's first rows, so that they repeat
    limit = np.where(rng.random(nnz) < 0.5, np.minimum(40, np.asarray(rows)[table]), np.asarray(rows)[table])
    indices = (rng.random(nnz) * limit).astype(np.int32)
    n_hot = max(1, int(N * hot))
    hot_rows = np.unique(np.concatenate([rng.choice(N, n_hot, replace=False) if N < 1 << 22 else rng.integers(0, N, n_hot)]))
    remap = orc.build_remap(hot_rows, N)
    hot_cap, staging = len(hot_rows), max(1, min(N, nnz))
    perm, n_pop, O, X, _ = orc.fragment(indices, offsets, B, rows, remap, S)
    C, slots = orc.gather_cold(X.ids, remap, hot_cap)

    geom = hl.make_geometry(rows, 4, S)
    n_ws = hl.hl_workspace_bytes(geom, B, nnz, hot_cap, staging)
    ws = torch.empty(n_ws, dtype=torch.uint8, device=DEV)
    ctx = hl.hl_create(geom, B, nnz, hot_cap, staging, ws, n_ws)
    i32 = dict(dtype=torch.int32, device=DEV)
    try:
        st = torch.cuda.current_stream().cuda_stream
        d_hot, d_n_hot = torch.from_numpy(hot_rows.astype(np.int32)).to(DEV), torch.tensor([hot_cap], device=DEV)
        hl.hl_build_remap(ctx, d_hot, d_n_hot, None, None, None, st)
        d_idx, d_off = torch.from_numpy(indices).to(DEV), torch.from_numpy(offsets).to(DEV)
        d_perm, d_counts = torch.empty(B, **i32), torch.empty(2, **i32)
        off = [torch.empty(T * B * S + 1, **i32) for _ in range(2)]
        ids = [torch.empty(nnz, **i32) for _ in range(2)]
        pop, non = (hl.make_ubatch(o, i, nnz) for o, i in zip(off, ids))
        d_cold, d_n_cold = torch.empty(staging, **i32), torch.empty(1, dtype=torch.int64, device=DEV)
        for _ in range(2):                                   # the second time: the scratch was left as it has to be
            hl.hl_fragment(ctx, hl.make_batch(d_idx, d_off, B, nnz), None, 0, d_perm, d_counts, pop, non, None, st)
            assert np.array_equal(d_perm.cpu().numpy(), perm)
            assert d_counts.tolist() == [n_pop, B - n_pop]
            for mu, o, i in ((O, off[0], ids[0]), (X, off[1], ids[1])):
                assert np.array_equal(o[:len(mu.offsets)].cpu().numpy(), mu.offsets)
                assert np.array_equal(i[:len(mu.ids)].cpu().numpy(), mu.ids)
            hl.hl_index_cold(ctx, non, d_counts[1:], 0, staging, d_cold, d_n_cold, None, None, None, st)
            assert int(d_n_cold) == len(C)
            assert np.array_equal(d_cold[:len(C)].cpu().numpy(), C)
            assert np.array_equal(ids[1][:len(X.ids)].cpu().numpy(), slots)
            # the sorts: stable by slot, O before X where both form one run
            bags = [np.repeat(np.arange(len(mu.offsets) - 1), np.diff(mu.offsets)) for mu in (O, X)]
            for merged in (False, True):
                d_slots, d_bags, d_n = torch.empty(nnz, **i32), torch.empty(nnz, **i32), torch.empty(3, **i32)
                call = hl.hl_embbag_bwd_prepare_merged if merged else hl.hl_embbag_bwd_prepare2
                call(ctx, pop, d_counts, non, d_counts[1:], d_slots, d_bags, d_n, st)
                if merged:
                    key = np.concatenate([O.ids, slots])
                    bag = np.concatenate([bags[0], bags[1] + len(O.offsets) - 1])
                    order = np.argsort(key, kind="stable")
                    key, bag = key[order], bag[order]
                else:
                    a, b = np.argsort(O.ids, kind="stable"), np.argsort(slots, kind="stable")
                    key = np.concatenate([O.ids[a], slots[b] + hot_cap + staging + 1])      # X's keys behind O's
                    bag = np.concatenate([bags[0][a], bags[1][b]])
                    assert d_n[:2].tolist() == [len(O.ids), nnz - len(O.ids)]
                assert np.array_equal(d_slots.cpu().numpy(), key)
                assert np.array_equal(d_bags.cpu().numpy(), bag)
        hl.hl_status(ctx)
    finally:
        torch.cuda.synchronize()
        hl.hl_destroy(ctx)
