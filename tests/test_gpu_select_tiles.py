"""The hot-set selection at the edges of its tiles (8 192 rows, four counts per load) and digits (8 bits of the count; digits
that no count reaches are not looked at): ties cut by the quota, more rows wanted than were counted, none wanted."""
import numpy as np
import pytest
import torch

from oracle import hotline_oracle as orc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("top", [1, 255, 256, 70_000])
@pytest.mark.parametrize("rows", [1, 3, 511, 1023, 1025, 8191, 8192, 8193, 16_382, 1_300_001])
def test_selected_rows(rows, top):
    import paper_2204_05436_b200 as hl
    rng = np.random.default_rng(rows + top)
    seen = np.unique(np.concatenate([rng.integers(0, rows, min(rows, 5000)), [0, rows - 1]]))
    counts = rng.integers(1, 4, len(seen))
    counts[rng.integers(0, len(seen), 3)] = top
    lookups = np.repeat(seen, counts).astype(np.int32)
    rng.shuffle(lookups)
    n = len(lookups)
    offsets = np.arange(n + 1, dtype=np.int32)
    cnt = orc.access_counts([(lookups, offsets)], n, [rows], 1)
    geom = hl.make_geometry([rows], 4, 1)
    n_ws = hl.hl_workspace_bytes(geom, n, n, rows, 1)
    ws = torch.empty(n_ws, dtype=torch.uint8, device=DEV)
    ctx = hl.hl_create(geom, n, n, rows, 1, ws, n_ws)
    try:
        st = torch.cuda.current_stream().cuda_stream
        d_idx, d_off = torch.from_numpy(lookups).to(DEV), torch.from_numpy(offsets).to(DEV)
        d_hot, d_n = torch.empty(rows, dtype=torch.int32, device=DEV), torch.empty(1, dtype=torch.int64, device=DEV)
        hl.hl_profile_hot(ctx, hl.make_batch(d_idx, d_off, n, n), True, False, 0, 0, 1, d_hot, d_n, st)
        for k in sorted({0, 1, 2, len(seen) // 2, len(seen) - 1, len(seen), rows}):
            want = orc.select_hot(cnt, k)
            hl.hl_profile_hot(ctx, None, False, True, hl.HL_HOT_TOPK_ROWS, k, 1, d_hot, d_n, st)
            hl.hl_status(ctx)
            assert int(d_n) == len(want)
            assert np.array_equal(d_hot[:len(want)].cpu().numpy(), want)
    finally:
        torch.cuda.synchronize()
        hl.hl_destroy(ctx)
