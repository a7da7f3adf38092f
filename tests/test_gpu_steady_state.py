"""What a program does thousands of times: the pipeline over so many mini-batches that every slot has launched its kernels
plainly, has built its graphs and launches them with changed arguments (mini-batches of different numbers of lookups among
them), and calls recorded into the caller's own graph by stream capture, before and after the library has graphs of them.
Integer data: every sum is exact, results must equal the oracle's bit for bit."""
import dataclasses

import numpy as np
import pytest
import torch

import gen
from oracle import hotline_oracle as orc
from tests.harness import run_pipelined_check

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("lookahead, order", [(2, "fig8"), (1, "eq5")])
def test_pipeline_over_many_mini_batches(lookahead, order):
    spec = dataclasses.replace(gen.CONFIGS["tiny"], batch=200, rows=("fixed", 700), hot_policy=("fraction", 20, 100),
                               profile_batches=4)
    stats = run_pipelined_check(spec, steps=240, integer=True, native=True, lookahead=lookahead, order=order)
    assert stats["shared_cold_rows"] > 1000


def test_pipeline_over_many_mini_batches_of_changing_size():
    spec = dataclasses.replace(gen.CONFIGS["multi_hot"], batch=60, dim=16, rows=("fixed", 900),
                               hot_policy=("fraction", 40, 100), profile_batches=2)
    run_pipelined_check(spec, steps=160, integer=True, native=True)


def test_calls_captured_into_the_callers_graph():
    import paper_2204_05436_b200 as hl
    rng = np.random.default_rng(4)
    rows, dim, n_bags, lr = 3000, 32, 40_000, 0.5
    ids = np.minimum((rng.pareto(1.2, n_bags) * 40).astype(np.int64), rows - 1).astype(np.int32)
    offsets = np.arange(n_bags + 1, dtype=np.int32)
    cache = rng.integers(-8, 9, (rows, dim)).astype(np.float32)
    grad = rng.integers(-4, 5, (n_bags, dim)).astype(np.float32)
    geom = hl.make_geometry([rows], dim, 1)
    ws_bytes = hl.hl_workspace_bytes(geom, n_bags, n_bags, rows, 0)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=DEV)
    ctx = hl.hl_create(geom, n_bags, n_bags, rows, 0, ws, ws_bytes)
    try:
        d_cache, d_off, d_ids, d_grad = (torch.from_numpy(x).to(DEV) for x in (cache, offsets, ids, grad))
        d_n = torch.tensor([n_bags], dtype=torch.int32, device=DEV)
        out = torch.zeros((n_bags, dim), device=DEV)
        ub = hl.make_ubatch(d_off, d_ids, n_bags)

        def calls():
            s = torch.cuda.current_stream().cuda_stream
            hl.hl_embbag_fwd(ctx, d_cache, ub, d_n, out, s)
            hl.hl_embbag_bwd_sgd(ctx, d_cache, ub, d_n, d_grad, lr, s)

        want = cache.copy()
        calls()
        for warm in (0, 100):
            for _ in range(warm):
                calls()
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                calls()
            d_cache.copy_(torch.from_numpy(cache))
            want = cache.copy()
            for _ in range(3):
                pooled = want[ids]
                orc.embbag_bwd_sgd(want, ids, offsets, grad, lr)
                graph.replay()
            assert hl.hl_status(ctx) == hl.HL_OK
            assert np.array_equal(out.cpu().numpy(), pooled)
            assert np.array_equal(d_cache.cpu().numpy(), want)
            calls()                                              # and the library's own launches still work
            pooled = want[ids]
            orc.embbag_bwd_sgd(want, ids, offsets, grad, lr)
            assert hl.hl_status(ctx) == hl.HL_OK
            assert np.array_equal(out.cpu().numpy(), pooled) and np.array_equal(d_cache.cpu().numpy(), want)
            del graph
    finally:
        torch.cuda.synchronize()
        hl.hl_destroy(ctx)
