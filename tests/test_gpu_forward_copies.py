"""The pooling forward on bags of one lookup, beside bags of several: up to 64 floats a row they are copies, bit for bit, with the
signs of zeros and the bits of NaNs; wider rows are added to zero.  Empty bags, and those of a skipped lookup, are +0."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dim", [4, 12, 16, 32, 36, 64, 68, 128])
def test_bags_of_one_lookup_keep_their_bits(dim):
    import paper_2204_05436_b200 as hl
    rng = np.random.default_rng(dim)
    rows, lengths = 50, np.resize([1, 0, 3, 1, 1, 2, 1, 5, 0, 1, 1, 1, 1, 2], 3001)
    bags, nnz = len(lengths), int(lengths.sum())
    offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    ids = rng.integers(0, rows, nnz).astype(np.int32)
    ids[rng.random(nnz) < 0.1] = -1
    bits = rng.choice(np.array([0x80000000, 0, 0x7fc12345, 0xffa00001, 0x80000001, 0x3f800000, 0xff800000], dtype=np.uint32),
                      (rows, dim))
    geom = hl.make_geometry([rows], dim, 1)
    n_ws = hl.hl_workspace_bytes(geom, bags, 2 * bags, rows, 0)
    ws = torch.empty(n_ws, dtype=torch.uint8, device=DEV)
    ctx = hl.hl_create(geom, bags, 2 * bags, rows, 0, ws, n_ws)
    try:
        d_off, d_ids = torch.from_numpy(offsets).to(DEV), torch.from_numpy(ids).to(DEV)
        cache, out = torch.from_numpy(bits.view(np.float32)).to(DEV), torch.full((bags, dim), 7.0, device=DEV)
        d_n = torch.tensor([bags], dtype=torch.int32, device=DEV)
        hl.hl_embbag_fwd(ctx, cache, hl.make_ubatch(d_off, d_ids, nnz), d_n, out, torch.cuda.current_stream().cuda_stream)
        hl.hl_status(ctx)
        got = out.cpu().numpy().view(np.uint32)
    finally:
        torch.cuda.synchronize()
        hl.hl_destroy(ctx)
    one = np.flatnonzero(lengths == 1)
    one_id = ids[offsets[one]]
    want = np.where((one_id < 0)[:, None], 0, bits[one_id]).astype(np.uint32)
    if dim > 64:                                 # added to +0: no -0, and a NaN is some NaN
        nan = np.isnan(want.view(np.float32))
        assert np.isnan(got[one].view(np.float32))[nan].all()
        want = np.where(want == 0x80000000, 0, want)
        assert np.array_equal(got[one][~nan], want[~nan])
    else:
        assert np.array_equal(got[one], want)
    assert (got[lengths == 0] == 0).all()
    several = np.flatnonzero(lengths > 1)
    with np.errstate(invalid="ignore"):
        values = bits.view(np.float32).astype(np.float64)
        sums = np.array([sum((values[i] for i in ids[offsets[b]:offsets[b + 1]] if i >= 0), np.zeros(dim)) for b in several])
        sums = sums.astype(np.float32)
    assert np.array_equal(np.isnan(got[several].view(np.float32)), np.isnan(sums))
    fine = ~np.isnan(sums)
    assert np.array_equal(got[several][fine], sums.view(np.uint32)[fine])
