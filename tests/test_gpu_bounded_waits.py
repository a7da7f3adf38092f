"""The bounded waits of the chained tiles that rank cold rows (32-bit and 64-bit row ids) and that select the popular rows,
made to run out: one tile publishes nothing and the tiles behind it give up after a few polls.  The call ends with
HL_ETIMEOUT in the status word and nothing out of range; the same call on the same context is exact afterwards."""
import numpy as np
import pytest
import torch

import gen
from oracle import hotline_oracle as orc
from test_gpu_robustness import _t, _tiny_hotline
from test_gpu_wide import _check_index, _Wide

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stall_tile", [0, 1, 8])
def test_cold_row_ranks(stall_tile):
    """80 000 rows: ten tiles of 256 bitmap words, of which the last is the only one nobody waits for."""
    import paper_2204_05436_b200 as hl
    spec, geom, table0, h = _tiny_hotline(hl)
    try:
        with torch.cuda.stream(h.main):
            hot = np.sort(np.random.default_rng(5).choice(geom.total_rows, 3000, replace=False)).astype(np.int64)
            h.set_hot_rows(_t(hot))
            h.build_remap(load_rows=True)
            b = gen.make_batch(spec, geom, 3)
            d_idx, d_off = _t(b.indices), _t(b.offsets)

            def search():
                h.fragment(d_idx, d_off, spec.batch)
                assert h.status() == hl.HL_OK
                hl.hl_test_bounded_waits(h.ctx, limit, stall_tile)
                hl.hl_index_cold(h.ctx, h.non, h.counts_non, 0, h.staging_cap, h.cold_rows, h.n_cold, None, None, None,
                                 h.main.cuda_stream)
                hl.hl_test_bounded_waits(h.ctx, 0, -1)

            limit = 200
            search()
            assert h.status(raise_on_error=False) == hl.HL_ETIMEOUT
            limit = 0
            search()
            assert h.status() == hl.HL_OK
            remap = orc.build_remap(hot, geom.total_rows)
            _, _, _, X, _ = orc.fragment(b.indices, b.offsets, spec.batch, geom.table_rows, remap, 1)
            C, slots = orc.gather_cold(X.ids, remap, h.hot_cap)
            assert int(h.n_cold.item()) == len(C)
            assert np.array_equal(h.cold_rows[:len(C)].cpu().numpy(), C.astype(np.int32))
            assert np.array_equal(h.non_ids[:len(slots)].cpu().numpy(), slots)
    finally:
        h.close()


@pytest.mark.parametrize("stall_tile", [0, 1, 8])
def test_selection_of_the_popular_rows(stall_tile):
    """80 000 counters: ten tiles of 8 192."""
    import paper_2204_05436_b200 as hl
    spec, geom, table0, h = _tiny_hotline(hl)
    try:
        with torch.cuda.stream(h.main):
            batches = [gen.make_batch(spec, geom, i) for i in range(4)]
            for i, b in enumerate(batches):
                h.profile(_t(b.indices), _t(b.offsets), spec.batch, reset=(i == 0))
            select = dict(finalize=True, policy=hl.HL_HOT_TOPK_ROWS, p_num=2500)
            hl.hl_test_bounded_waits(h.ctx, 200, stall_tile)
            h.profile(None, None, **select)
            assert h.status(raise_on_error=False) == hl.HL_ETIMEOUT
            hl.hl_test_bounded_waits(h.ctx, 0, -1)
            h.profile(None, None, **select)
            assert h.status() == hl.HL_OK
            cnt = orc.access_counts([(b.indices, b.offsets) for b in batches], spec.batch, geom.table_rows, 1)
            hot = orc.select_hot(cnt, 2500)
            assert int(h.n_hot.item()) == len(hot)
            assert np.array_equal(h.hot_rows[:len(hot)].cpu().numpy(), hot.astype(np.int32))
    finally:
        h.close()


@pytest.mark.parametrize("table_rows, cold", [((6000, 9000, 20_000), 3000),                     # rows of up to 32 bits
                                              ((2 ** 31 - 9, 2 ** 31 - 1, 2 ** 31 - 5), 3000),  # the upper bits sorted too
                                              ((6000, 9000, 20_000), 1800)])                    # one tile of the sort,
def test_wide_cold_row_ranks(table_rows, cold):                                                 # two of the ranks
    import paper_2204_05436_b200 as hl
    rng = np.random.default_rng(cold)
    T, B = len(table_rows), cold // len(table_rows)
    wd = _Wide(hl, table_rows, 1, B, cold, 50, cold, 1 << 12)
    try:
        class batch:
            indices = np.concatenate([rng.integers(0, r, B) for r in table_rows]).astype(np.int32)
            offsets = np.arange(T * B + 1, dtype=np.int32)
        base = np.concatenate([[0], np.cumsum(table_rows)[:-1]]).astype(np.int64)
        hot = np.unique(np.repeat(base, B)[:: T * B // 40] + batch.indices[:: T * B // 40])[:50]
        wd.hot_rows[:len(hot)] = _t(hot)
        wd.n_hot.fill_(len(hot))
        hl.hl_wide_build_remap(wd.w, wd.hot_rows, wd.n_hot, wd.stream)
        hb = hl.make_batch(_t(batch.indices), _t(batch.offsets), B, len(batch.indices))
        hl.hl_wide_fragment(wd.w, hb, wd.perm, wd.counts, wd.pop, wd.non_off, wd.non_rows, wd.max_nnz, wd.stream)
        assert hl.hl_wide_status(wd.w) == hl.HL_OK
        hl.hl_wide_test_bounded_waits(wd.w, 200, 0)
        hl.hl_wide_index_cold(wd.w, wd.non_off, wd.non_rows, wd.max_nnz, wd.counts[1:], wd.non_slots, wd.cold_rows,
                              wd.n_cold, wd.stream)
        assert hl.hl_wide_status(wd.w, raise_on_error=False) == hl.HL_ETIMEOUT
        hl.hl_wide_test_bounded_waits(wd.w, 0, -1)
        wd.index(batch)
        n_non = int(wd.counts[1].item())
        rows = wd.non_rows[:int(wd.counts[3].item())].cpu().numpy()
        is_hot = np.isin(rows, hot)
        want = np.unique(rows[~is_hot])
        assert n_non > 0 and int(wd.n_cold.item()) == len(want)
        assert np.array_equal(wd.cold_rows[:len(want)].cpu().numpy(), want)
        slots = np.where(is_hot, np.searchsorted(hot, rows), 50 + np.searchsorted(want, rows))
        assert np.array_equal(wd.non_slots[:len(rows)].cpu().numpy(), slots)
    finally:
        wd.close()


@pytest.mark.parametrize("counted", [3000, 30_000])
def test_wide_selection(counted):
    """Two sorts and a selection over the hashed counter; with 30 000 rows all of them have several tiles in use."""
    import paper_2204_05436_b200 as hl
    rows = 50_000
    wd = _Wide(hl, (rows,), 1, counted, counted, 700, 10, 1 << 16)
    try:
        class batch:
            indices = np.random.default_rng(counted).permutation(rows)[:counted].astype(np.int32)
            offsets = np.arange(counted + 1, dtype=np.int32)
        batch.indices[: counted // 3] = batch.indices[counted // 3: 2 * (counted // 3)]
        want = wd.learn([batch], hl.HL_HOT_TOPK_ROWS, 700, 1, 16)
        hl.hl_wide_test_bounded_waits(wd.w, 200, 0)
        hl.hl_wide_profile_hot(wd.w, None, False, True, hl.HL_HOT_TOPK_ROWS, 700, 1, 16, wd.hot_rows, wd.n_hot, wd.stream)
        assert hl.hl_wide_status(wd.w, raise_on_error=False) == hl.HL_ETIMEOUT
        hl.hl_wide_test_bounded_waits(wd.w, 0, -1)
        hl.hl_wide_profile_hot(wd.w, None, False, True, hl.HL_HOT_TOPK_ROWS, 700, 1, 16, wd.hot_rows, wd.n_hot, wd.stream)
        assert hl.hl_wide_status(wd.w) == hl.HL_OK
        assert np.array_equal(wd.hot_rows[:int(wd.n_hot.item())].cpu().numpy(), want)
        cnt = np.bincount(batch.indices, minlength=rows)
        assert np.array_equal(want, orc.select_hot(cnt, 700))
    finally:
        wd.close()
