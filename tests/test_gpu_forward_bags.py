"""The pooling forward with several lookups per bag: a group of lanes per run of bags, one to four lookups at a time.  Bag
lengths around 32 and 4, empty bags, skipped lookups, every row width class, runs of no bag, of one and of more bags than
a group has lanes; integer data, so the pooled vectors must equal the oracle's."""
import numpy as np
import pytest
import torch

from oracle import hotline_oracle as orc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LENGTHS = [0, 1, 2, 3, 4, 5, 31, 32, 33, 0, 0, 63, 64, 65, 7, 100, 28, 36, 0]


@pytest.mark.parametrize("bags", [1, 2, 19, 5000])
@pytest.mark.parametrize("dim", [4, 16, 20, 32, 36, 64, 68, 128, 132, 256, 260, 512, 1024])
def test_forward_of_long_bags(dim, bags):
    import paper_2204_05436_b200 as hl
    lengths = np.resize(LENGTHS, bags) if bags > 2 else np.full(bags, 35)
    _check(hl, dim, bags, lengths)


@pytest.mark.parametrize("dim,bags", [(4, 170_000), (12, 100_001), (32, 160_000), (128, 155_000)])
def test_more_bags_than_lanes(dim, bags):
    import paper_2204_05436_b200 as hl
    _check(hl, dim, bags, np.resize([0, 3, 1, 2, 0, 4, 1], bags))


def _check(hl, dim, bags, lengths):
    rng = np.random.default_rng(dim + bags)
    rows = 300
    offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    nnz = int(offsets[-1])
    ids = rng.integers(0, rows, nnz).astype(np.int32)
    cache = rng.integers(-8, 9, (rows, dim)).astype(np.float32)
    geom = hl.make_geometry([rows], dim, 1)
    n_ws = hl.hl_workspace_bytes(geom, bags, nnz, rows, 0)
    ws = torch.empty(n_ws, dtype=torch.uint8, device=DEV)
    ctx = hl.hl_create(geom, bags, nnz, rows, 0, ws, n_ws)
    try:
        d_cache, d_off = torch.from_numpy(cache).to(DEV), torch.from_numpy(offsets).to(DEV)
        d_n = torch.tensor([bags], dtype=torch.int32, device=DEV)
        for skipped in (0.0, 0.2):
            skip = rng.random(nnz) < skipped
            use = np.where(skip, -1, ids).astype(np.int32)
            bag_of = np.repeat(np.arange(bags), lengths)[~skip]
            want = orc.embbag_fwd(cache, ids[~skip], np.concatenate([[0], np.cumsum(np.bincount(bag_of, minlength=bags))]))
            d_ids, out = torch.from_numpy(use).to(DEV), torch.full((bags, dim), 7.0, device=DEV)
            hl.hl_embbag_fwd(ctx, d_cache, hl.make_ubatch(d_off, d_ids, nnz), d_n, out,
                             torch.cuda.current_stream().cuda_stream)
            hl.hl_status(ctx)
            assert np.array_equal(out.cpu().numpy(), want)
    finally:
        torch.cuda.synchronize()
        hl.hl_destroy(ctx)
