"""The workloads whose speed counts: what a training or serving program has this library do, one call or one mini-batch
at a time, through the package's public classes and calls.

Kinds of work (``case["kind"]``):

* ``train``  one mini-batch through the library's own pipelined schedule (NativePipelinedHotline.step): what a training
             loop does thousands of times per second, with its cold rows in host memory;
* ``step``   one mini-batch without pipelining (Hotline.step): small trainers, debugging, irregular input arrival;
* ``infer``  fragment, cold gather and both forwards, no update: serving and evaluation;
* ``pool``   forward and backward of an embedding bag whose rows all live in HBM (hl_embbag_fwd, hl_embbag_bwd_sgd);
* ``learn``  a re-calibration: popular rows flushed, a window of mini-batches counted, a new set selected and loaded;
* ``track``  a mini-batch presented to the approximate access logger (hl_tracker_update);
* ``wide``   the index path of models with 64-bit row ids (hl_wide_fragment, hl_wide_index_cold).

A state holds several mini-batches and a pass takes the next one, as a program's data loader would give it.  Inputs are
power-law draws per table, scattered over the table by an affine bijection, the popular set is learned from such draws
by the library itself, and the host table is memory from hl_host_alloc.
"""
from __future__ import annotations

import ctypes
import functools
import math
import random
import weakref

import numpy as np
import torch

import paper_2204_05436_b200 as hl

DEVICE = "cuda:0"
LR = 0.01


# ---- the cases ------------------------------------------------------------------------------------------------------
def _case(kind, tables, rows, dim, batch, steps=1, bag=1, cap=1, alpha=1.1, dense=0, hot=0.05, order="fig8", even=False,
          profile=16, ways=0):
    """``rows``: of all tables together, spread over them log-uniformly (``even``: equally); ``steps``: bags per input
    and table; ``bag`` / ``cap``: lookups per bag, exactly one or min(Poisson(bag), cap); ``hot``: popular rows as a
    share of all rows; ``profile``: mini-batches the popular set is learned from; ``ways``: of the access logger."""
    return dict(kind=kind, tables=tables, rows=rows, dim=dim, batch=batch, steps=steps, bag=bag, cap=cap, alpha=alpha,
                dense=dense, hot=hot, order=order, even=even, profile=profile, ways=ways)


def listed():
    cases = {
        # the Tiny configuration: 8 tables of 10 000 rows, dim 16, batch 1 024 -- every call is short, launches count
        "train tiny": _case("train", 8, 80_000, 16, 1024, alpha=1.05, hot=0.05, even=True, profile=10),
        # a time-series model: 21 steps x 3 tables, dim 16, 129 K one-lookup bags per mini-batch
        "train time series": _case("train", 3, 5_010_000, 16, 2048, steps=21, alpha=1.2, hot=0.2, profile=48),
        # the Avazu-like configuration: 21 tables, 9.3 M rows, dim 16, batch 4 096
        "train click log": _case("train", 21, 9_300_000, 16, 4096, dense=1, alpha=1.1, hot=0.22, profile=32),
        # the benchmark's workload (26 tables, dim 64, batch 16 384, 13 dense features) at three hundredths of its rows,
        # where the share of popular inputs is the paper's 3:1
        "train large": _case("train", 26, 7_725_000, 64, 16384, dense=13, alpha=1.2, hot=0.5, profile=64),
        # multi-hot model: bags of min(Poisson(20), 64) lookups, dim 128, much of the working set in host memory
        "train multi-hot": _case("train", 8, 2_000_000, 128, 8192, bag=20, cap=64, alpha=1.05, hot=0.25, even=True,
                                 profile=8),
        # ragged: 37 tables, row width that fills no power of two, odd batch, short bags, one update per row (Eq. 5)
        "train ragged": _case("train", 37, 400_003, 36, 3001, bag=3, cap=12, alpha=1.15, dense=7, hot=0.1, order="eq5",
                              profile=12),
        # the DLRM-small shape at a tenth of its rows, one mini-batch after the other
        "step small": _case("step", 26, 3_383_000, 16, 4096, dense=13, alpha=1.1, hot=0.3, profile=32),
        # serving a thousand inputs of the large model
        "infer large": _case("infer", 26, 7_725_000, 64, 1000, dense=13, alpha=1.2, hot=0.5, profile=64),
        # all rows resident, multi-hot, the largest forward and backward
        "pool multi-hot": _case("pool", 8, 4_000_000, 128, 16384, bag=20, cap=64, alpha=1.05, hot=1.0, even=True),
        # periodic re-calibration of the Avazu-like configuration
        "learn click log": _case("learn", 21, 9_300_000, 16, 4096, alpha=1.1, hot=0.05, profile=16),
        # the logger at the paper's size (2 M blocks) on the large model's mini-batches
        "track large": _case("track", 26, 25_750_000, 64, 16384, alpha=1.2, profile=4, ways=16),
        # a model beyond 2^31 rows
        "wide large": _case("wide", 26, 2_600_000_000, 64, 16384, alpha=1.2, hot=0.0005, profile=16),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["train"] * 6 + ["step", "infer", "pool", "learn", "track", "wide"])
    alpha = round(rng.uniform(1.05, 1.25), 3)
    dim = 4 * _log_int(rng, 2, 32)
    tables = _log_int(rng, 3, 40)
    bag, cap, steps = 1, 1, 1
    shape = rng.random()
    if shape < 0.3:
        bag = _log_int(rng, 2, 20)
        cap = 3 * bag + 4
    elif shape < 0.4:
        steps = rng.randint(2, 21)
    most = {"train": 900_000, "pool": 2_000_000}.get(kind, 400_000)              # lookups of a mini-batch
    most = max(3000, min(most, 100_000_000 // dim // (1 if bag > 1 else 2)))
    batch = _log_int(rng, 64, 16384) | rng.randint(0, 1)
    batch = max(16, min(batch, most // (tables * steps * bag)))
    rows = _log_int(rng, 60_000, 8_000_000)
    rows = min(rows, 400_000_000 // dim)
    if kind == "wide":
        rows = _log_int(rng, 100_000_000, 4_000_000_000)
    elif kind == "track":
        rows = _log_int(rng, 200_000, 30_000_000)
    hot = 1.0 if kind == "pool" else round(math.exp(rng.uniform(math.log(0.03), math.log(0.5))), 4)
    if kind == "wide":
        hot = min(hot, 1_000_000 / rows)
    return _case(kind, tables, rows, dim, batch, steps=steps, bag=bag, cap=cap, alpha=alpha,
                 dense=rng.choice([0, 1, 7, 13]) if kind in ("train", "step", "infer") else 0, hot=hot,
                 order=rng.choice(["fig8", "fig8", "eq5"]) if kind == "train" else "fig8", even=rng.random() < 0.3,
                 profile=4 if kind == "track" else 12, ways=rng.choice([4, 8, 16]) if kind == "track" else 0)


# ---- inputs ---------------------------------------------------------------------------------------------------------
def _table_rows(case):
    T, N = case["tables"], case["rows"]
    if case["even"]:
        rows = [N // T] * T
    else:
        r = random.Random(f"{T}/{N}")
        w = [math.exp(r.uniform(0.0, math.log(1e5))) for _ in range(T)]
        rows = [max(4, int(N * x / sum(w))) for x in w]
    return [min(x, (1 << 31) - 1) for x in rows]


def _bags(case):
    return case["tables"] * case["batch"] * case["steps"]


def _max_nnz(case):
    return _bags(case) * case["cap"]


class _Loader:
    """Mini-batches drawn on the device: table-major CSR of power-law row ids."""

    def __init__(self, case, seed):
        self.case, self.rows = case, _table_rows(case)
        self.g = torch.Generator(device=DEVICE)
        self.g.manual_seed(seed)
        r = random.Random(seed)
        mult, add = [], []
        for n in self.rows:
            m = r.randrange(n // 3, n) | 1
            while math.gcd(m, n) != 1:
                m += 1
            mult.append(m)
            add.append(r.randrange(n))
        self.R, self.M, self.A = (torch.tensor(x, dtype=torch.int64, device=DEVICE) for x in (self.rows, mult, add))

    def ids(self, table):
        """Table-local row ids of one lookup per entry of ``table``: rank k with probability close to k ** -alpha."""
        e = 1.0 - self.case["alpha"]
        R = self.R[table]
        u = torch.rand(table.shape[0], dtype=torch.float64, device=DEVICE, generator=self.g)
        rank = (1.0 + u * ((R + 1).double() ** e - 1.0)) ** (1.0 / e)
        rank = torch.minimum(rank.long(), R) - 1
        # rank * M + A mod R, with the product kept below 2^63 by splitting the rank
        hi, lo = rank >> 15, rank & 32767
        m = self.M[table]
        return ((((hi * m) % R) * 32768 + lo * m + self.A[table]) % R).to(torch.int32)

    def batch(self):
        c = self.case
        bags = _bags(c)
        per_table = c["batch"] * c["steps"]
        offsets = torch.zeros(bags + 1, dtype=torch.int32, device=DEVICE)
        if c["bag"] == 1:
            offsets[1:] = torch.arange(1, bags + 1, device=DEVICE)
            table = torch.arange(c["tables"], device=DEVICE).repeat_interleave(per_table)
        else:
            mean = torch.full((bags,), float(c["bag"]), device=DEVICE)
            size = torch.poisson(mean, generator=self.g).clamp_(max=c["cap"]).long()
            offsets[1:] = torch.cumsum(size, 0)
            table = torch.arange(c["tables"], device=DEVICE).repeat_interleave(size.view(c["tables"], per_table).sum(1))
        dense = None
        if c["dense"]:
            dense = torch.randn((c["batch"], c["dense"]), device=DEVICE, generator=self.g)
        return self.ids(table), offsets, c["batch"], dense

    def randn(self, *shape):
        return torch.randn(shape, device=DEVICE, generator=self.g)


def _host_table(rows, dim, g):
    """fp32 [rows, dim] in memory from hl_host_alloc, given back when the last tensor over it is gone."""
    ptr = hl.hl_host_alloc(rows * dim * 4)
    buf = (ctypes.c_float * (rows * dim)).from_address(ptr)
    weakref.finalize(buf, hl.hl_host_free, ptr)
    t = torch.from_numpy(np.frombuffer(buf, dtype=np.float32).reshape(rows, dim))
    step = max(1, (1 << 26) // dim)
    for r in range(0, rows, step):
        n = min(step, rows - r)
        t[r:r + n].copy_(torch.rand((n, dim), device=DEVICE, generator=g) - 0.5)
    return t


class _State:
    pass


def _learn(h, loader, n):
    """The library's learning phase over ``n`` mini-batches, popular rows loaded."""
    with torch.cuda.stream(h.main):
        for i in range(n):
            idx, off, B, _ = loader.batch()
            h.profile(idx, off, B, reset=(i == 0))
        h.profile(None, None, finalize=True, policy=hl.HL_HOT_TOPK_ROWS, p_num=h.hot_cap)
        h.build_remap()
    h.main.synchronize()


def prepare(case, seed):
    st = _State()
    st.kind, st.i = case["kind"], 0
    ld = _Loader(case, seed)
    rows, D, S, B = _table_rows(case), case["dim"], case["steps"], case["batch"]
    N, nnz, bags = sum(rows), _max_nnz(case), _bags(case)
    hot = max(1, min(N, int(N * case["hot"])))
    n_batches = 2 if case["bag"] > 1 else 8
    kind = case["kind"]
    if kind in ("train", "step", "infer", "learn"):
        staging = min(N, nnz)
        table = _host_table(N, D, ld.g)
        if kind == "train":
            n_batches = 6
            st.h = hl.NativePipelinedHotline(rows, D, S, B, nnz, hot, staging, table, n_dense=case["dense"],
                                             order=case["order"])
        else:
            st.h = hl.Hotline(rows, D, S, B, nnz, hot, staging, table, n_dense=case["dense"])
        _learn(st.h, ld, case["profile"])
        if kind == "learn":      # two windows of traffic whose popular rows differ
            st.windows = []
            for _ in range(2):
                w = _Loader(case, ld.g.initial_seed() + 1 + len(st.windows))
                st.windows.append([w.batch() for _ in range(case["profile"])])
            torch.cuda.synchronize()
            return st
        st.batches = [ld.batch() for _ in range(n_batches)]
        if kind != "infer":
            st.grad_pop = ld.randn(bags, D)
            st.grad_non = None if case["order"] == "eq5" else ld.randn(bags, D)
        torch.cuda.synchronize()
        if kind == "train":
            st.h.start(*st.batches[0], more=st.batches[1:st.h.lookahead], inputs_ready="resident")
    elif kind == "pool":
        st.geom = hl.make_geometry(rows, D, S)
        st.ws_bytes = hl.hl_workspace_bytes(st.geom, B, nnz, N, 0)
        st.ws = torch.empty(st.ws_bytes, dtype=torch.uint8, device=DEVICE)
        st.cache = torch.rand((N, D), device=DEVICE, generator=ld.g) - 0.5
        base = torch.tensor(np.concatenate([[0], np.cumsum(rows)[:-1]]), dtype=torch.int64, device=DEVICE)
        st.bags = []
        for _ in range(n_batches):
            idx, off, _, _ = ld.batch()
            table = torch.searchsorted(off[:: B * S][1:].long(), torch.arange(idx.shape[0], device=DEVICE), right=True)
            slots = (idx.long() + base[table]).to(torch.int32)
            st.bags.append((off, slots, hl.make_ubatch(off, slots, nnz)))
        st.n = torch.tensor([B], dtype=torch.int32, device=DEVICE)
        st.pooled = torch.zeros((bags, D), device=DEVICE)
        st.grad = ld.randn(bags, D)
        torch.cuda.synchronize()
        st.ctx = hl.hl_create(st.geom, B, nnz, N, 0, st.ws, st.ws_bytes)
        weakref.finalize(st, hl.hl_destroy, st.ctx)
    elif kind == "track":
        st.h = hl.Hotline(rows, D, S, B, nnz, 1, 1, torch.zeros((1, 1), device=DEVICE).expand(N, D))
        st.h.tracker_init((1 << 21) // case["ways"] if N > 4_000_000 else max(1, N // 4 // case["ways"]), case["ways"])
        st.batches = [ld.batch() for _ in range(n_batches)]
        torch.cuda.synchronize()
        for idx, off, _, _ in st.batches[: case["profile"]]:
            st.h.tracker_update(idx, off, B)
        st.h.main.synchronize()
    else:
        slots = 1 << 22
        st.geom = hl.make_geometry(rows, D, S)
        n = hl.hl_wide_workspace_bytes(st.geom, B, nnz, hot, nnz, slots)
        st.ws = torch.empty(n, dtype=torch.uint8, device=DEVICE)
        st.w = hl.hl_wide_create(st.geom, B, nnz, hot, nnz, slots, st.ws, n)
        weakref.finalize(st, hl.hl_wide_destroy, st.w)
        i32, i64 = (functools.partial(torch.zeros, dtype=t, device=DEVICE) for t in (torch.int32, torch.int64))
        st.hot_rows, st.n_hot = i64(hot), i64(1)
        st.perm, st.counts, st.pop_offsets, st.pop_ids = i32(B), i32(4), i32(bags + 1), i32(nnz)
        st.pop = hl.make_ubatch(st.pop_offsets, st.pop_ids, nnz)
        st.non_offsets, st.non_rows, st.non_slots, st.nnz = i32(bags + 1), i64(nnz), i32(nnz), nnz
        st.cold_rows, st.n_cold = i64(nnz), i64(1)
        s = torch.cuda.current_stream().cuda_stream
        for k in range(case["profile"]):
            idx, off, _, _ = ld.batch()
            hl.hl_wide_profile_hot(st.w, hl.make_batch(idx, off, B, idx.numel()), k == 0, False, hl.HL_HOT_TOPK_ROWS, hot,
                                   1, 4 * D, None, None, s)
        hl.hl_wide_profile_hot(st.w, None, False, True, hl.HL_HOT_TOPK_ROWS, hot, 1, 4 * D, st.hot_rows, st.n_hot, s)
        hl.hl_wide_build_remap(st.w, st.hot_rows, st.n_hot, s)
        st.batches = [ld.batch() for _ in range(n_batches)]
        torch.cuda.synchronize()
    return st


# ---- one pass -------------------------------------------------------------------------------------------------------
def _outputs(h, bufs):
    out = dict(perm=bufs.perm, counts=bufs.counts, pooled_pop=bufs.pooled_pop, pooled_non=bufs.pooled_non)
    if bufs.dense_out is not None:
        out["dense"] = bufs.dense_out
    return out


def run(st):
    kind, i = st.kind, st.i
    st.i = i + 1
    cur = torch.cuda.current_stream()
    if kind in ("pool", "wide"):
        s = cur.cuda_stream
        if kind == "pool":
            _, _, ub = st.bags[i % len(st.bags)]
            hl.hl_embbag_fwd(st.ctx, st.cache, ub, st.n, st.pooled, s)
            hl.hl_embbag_bwd_sgd(st.ctx, st.cache, ub, st.n, st.grad, LR, s)
            return dict(pooled=st.pooled, cache=st.cache)
        idx, off, B, _ = st.batches[i % len(st.batches)]
        hl.hl_wide_fragment(st.w, hl.make_batch(idx, off, B, idx.numel()), st.perm, st.counts, st.pop, st.non_offsets,
                            st.non_rows, st.nnz, s)
        hl.hl_wide_index_cold(st.w, st.non_offsets, st.non_rows, st.nnz, st.counts[1:], st.non_slots, st.cold_rows,
                              st.n_cold, s)
        return dict(perm=st.perm, counts=st.counts, pop_offsets=st.pop_offsets, pop_ids=st.pop_ids,
                    non_offsets=st.non_offsets, non_rows=st.non_rows, non_slots=st.non_slots, cold_rows=st.cold_rows,
                    n_cold=st.n_cold)
    # the surrounding program (dense layers, data loading) works on the current stream: the library's main stream takes
    # over from it and hands back to it
    h = st.h
    h.main.wait_stream(cur)
    if kind == "train":
        nxt = st.batches[(i + h.lookahead) % len(st.batches)]
        bufs = h.sets[h.step(st.grad_pop, st.grad_non, LR, next_batch=nxt, inputs_ready="resident")]
        out = dict(_outputs(h, bufs), popular_rows=h.cache[: h.hot_cap], table=h.host_table)
    elif kind == "step":
        idx, off, B, dense = st.batches[i % len(st.batches)]
        h.step(idx, off, B, st.grad_pop, st.grad_non, LR, dense=dense)
        out = dict(_outputs(h, h), popular_rows=h.cache[: h.hot_cap], table=h.host_table)
    elif kind == "infer":
        idx, off, B, dense = st.batches[i % len(st.batches)]
        h.fragment(idx, off, B, dense)
        h.gather_cold()
        h.fwd_pop()
        h.fwd_non()
        out = _outputs(h, h)
    elif kind == "learn":
        h.flush_hot()
        for k, (idx, off, B, _) in enumerate(st.windows[i % 2]):
            h.profile(idx, off, B, reset=(k == 0))
        h.profile(None, None, finalize=True, policy=hl.HL_HOT_TOPK_ROWS, p_num=h.hot_cap)
        h.build_remap()
        out = dict(hot_rows=h.hot_rows, n_hot=h.n_hot, popular_rows=h.cache[: h.hot_cap], table=h.host_table)
    else:
        idx, off, B, _ = st.batches[i % len(st.batches)]
        h.tracker_update(idx, off, B)
        out = dict(tags=h.trk_tags, rrpv=h.trk_rrpv, hits=h.trk_hits)
    cur.wait_stream(h.main)
    return out


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _distinct(alpha, rows, n):
    """Expected number of distinct rows among ``n`` draws from a table of ``rows`` rows."""
    if n == 0:
        return 0.0
    edges = np.unique(np.concatenate([np.arange(1, min(rows, 1000) + 1), np.geomspace(1, rows + 1, 2000)]))
    e = 1.0 - alpha
    mass = np.diff(edges ** e) / ((rows + 1.0) ** e - 1.0)
    width = np.diff(edges)
    return float(np.sum(width * -np.expm1(-n * mass / width)))


def work(case):
    kind, D, T, B = case["kind"], case["dim"], case["tables"], case["batch"]
    bags = _bags(case)
    L = int(bags * min(case["bag"], case["cap"]))
    rows = _table_rows(case)
    distinct = sum(_distinct(case["alpha"], r, L // T) for r in rows)
    index = 4 * L + 4 * (bags + 1)                         # a mini-batch's indices and offsets
    row = 4 * D
    if kind == "learn":
        n = case["profile"]
        hot = max(1, min(sum(rows), int(sum(rows) * case["hot"])))
        seen = min(hot, sum(_distinct(case["alpha"], r, n * L // T) for r in rows))
        return dict(bytes=n * index + 4 * row * seen + 4 * seen, flops=n * L)
    if kind == "track":
        return dict(bytes=index + 10 * distinct, flops=L)
    if kind == "wide":                                     # split, row ids, slots, distinct cold rows
        return dict(bytes=index + 4 * B + 12 * L + 4 * (bags + 1), flops=L)
    forward = index + row * (distinct + bags)
    backward = row * (bags + 2 * distinct)
    split = index + 4 * B + 4 * L + 8 * B * case["dense"]
    total = {"pool": forward + backward, "infer": forward + split}.get(kind, forward + backward + split)
    return dict(bytes=total, flops=(1 if kind == "infer" else 2) * L * D)


def tolerance(case):
    """Row ids, counts and copied rows are exact; sums of fp32 values are rounded once."""
    if case["kind"] in ("learn", "track", "wide"):
        return "exact"
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
