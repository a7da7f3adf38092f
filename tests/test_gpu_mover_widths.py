"""The row movers inside a schedule on both sides of the numbers of rows at which they change how many CTAs work and whether
the transfer is paced: staged rows and written-back rows are bit copies, and nothing else changes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("dim", [4, 36, 128])
def test_stage_and_write_back(dim):
    import paper_2204_05436_b200 as hl
    N, cap = 90_000, 70_000
    lines = -(-dim * 4 // 128)
    rng = np.random.default_rng(dim)
    table0 = rng.standard_normal((N, dim)).astype(np.float32)
    table = torch.from_numpy(table0.copy()).pin_memory()
    h = hl.Hotline([N], dim, 1, 64, 64, 1, cap, table)
    try:
        rows = torch.zeros(cap, dtype=torch.int32, device=DEV)
        n_rows = torch.zeros(1, dtype=torch.int64, device=DEV)
        s = h.main.cuda_stream
        for n in [0, 1, 10_239, 10_240, 10_241, 65536 // lines, 65536 // lines + 1, cap]:
            pick = np.sort(rng.choice(N, n, replace=False))
            rows[:n] = torch.from_numpy(pick.astype(np.int32)).to(DEV)
            n_rows.fill_(n)
            h.cache.zero_()
            table.copy_(torch.from_numpy(table0))
            torch.cuda.synchronize()
            hl.hl_stage_cold(h.ctx, table, h.cache, 0, cap, rows, n_rows, None, s)
            assert h.status() == hl.HL_OK
            got = h.cache.cpu().numpy()
            assert np.array_equal(got[1:1 + n], table0[pick]) and not got[1 + n:].any(), n
            h.cache.neg_()
            torch.cuda.synchronize()
            hl.hl_scatter_cold_at(h.ctx, h.cache, 0, cap, rows, n_rows, table, s)
            assert h.status() == hl.HL_OK
            want = table0.copy()
            want[pick] = -want[pick]
            assert np.array_equal(table.numpy(), want), n
    finally:
        h.close()
