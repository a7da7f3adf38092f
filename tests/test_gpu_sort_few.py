"""The backward's sort of fewer pairs than its cluster has CTAs, and of a few more: slots of one to four digits, against a
stable sort."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("rows", [200, 60_000, 1 << 22, 1 << 25])
def test_few_pairs(rows):
    import paper_2204_05436_b200 as hl
    rng = np.random.default_rng(rows)
    most = 100
    geom = hl.make_geometry([rows], 4, 1)
    n_ws = hl.hl_workspace_bytes(geom, most, most, rows, 0)
    ws = torch.empty(n_ws, dtype=torch.uint8, device=DEV)
    ctx = hl.hl_create(geom, most, most, rows, 0, ws, n_ws)
    slots, bags, n_out = (torch.zeros(k, dtype=torch.int32, device=DEV) for k in (most, most, 4))
    offsets = torch.arange(most + 1, dtype=torch.int32, device=DEV)
    try:
        for n in [*range(1, 35), 63, 64, 65, 100]:
            ids = rng.integers(0, rows, n).astype(np.int32)
            ids[n // 2:] = np.where(rng.random(n - n // 2) < 0.5, ids[0], ids[n // 2:])
            d_ids = torch.from_numpy(ids).to(DEV)
            ub = hl.make_ubatch(offsets, d_ids, n)
            d_n = torch.tensor([n], dtype=torch.int32, device=DEV)
            hl.hl_embbag_bwd_prepare(ctx, ub, d_n, slots, bags, n_out, torch.cuda.current_stream().cuda_stream)
            hl.hl_status(ctx)
            order = np.argsort(ids, kind="stable")
            assert int(n_out[0]) == n
            assert np.array_equal(slots.cpu().numpy()[:n], ids[order]), n
            assert np.array_equal(bags.cpu().numpy()[:n], order), n
    finally:
        torch.cuda.synchronize()
        hl.hl_destroy(ctx)
