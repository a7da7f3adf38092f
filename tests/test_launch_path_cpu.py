"""How the library queues its kernels, without a GPU: its object files linked with a stand-in for the CUDA runtime
(fake_cudart.cpp) that writes down what is put on every stream and can make any call fail.

A pipeline slot launches kernel by kernel at first, later as graphs, and from then on with changed arguments: whichever way,
the same kernels with the same arguments have to reach the same streams in the same order, and when a graph cannot be had,
or a stream is being captured, the plain launches have to do."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2204_05436_b200", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import importlib.util
    spec = importlib.util.spec_from_file_location("hotline_build", os.path.join(CSRC, "build.py"))
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    build.build_library()
    d = tmp_path_factory.mktemp("fake")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))))
    fake, so = str(d / "fake_cudart.o"), str(d / "libhotline_fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-I", os.path.join(cuda, "include"), "-c",
                    os.path.join(ROOT, "tests", "fake_cudart.cpp"), "-o", fake], check=True)
    objs = [os.path.join(build.OBJ_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    # (-Bsymbolic: torch has brought the real runtime into the process)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so, fake] + objs + ["-lpthread"], check=True)
    from paper_2204_05436_b200 import binding as B
    with pytest.MonkeyPatch.context() as m:
        m.setattr(B, "_LIB_PATH", so)
        lib = B._load()
    lib.fake_line.restype = ctypes.c_char_p
    lib.fake_capture.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.fake_device_memory.argtypes = [ctypes.c_void_p]
    return lib


@pytest.fixture
def B(lib, monkeypatch):
    """The binding, on the stand-in."""
    from paper_2204_05436_b200 import binding
    monkeypatch.setattr(binding, "_lib", lib)
    lib.fake_reset()
    return binding


def _log(lib, since=0):
    return [lib.fake_line(i).decode() for i in range(since, lib.fake_lines())]


def _what(line):
    """A line of the log without how its kernel got there."""
    return line.split(" ", 1)[1] if line.split(" ")[0] in ("plain", "graph") else line


def _name(line):
    return line.split(" ")[2] if line.split(" ")[0] in ("plain", "graph") else line.split(" ")[0]


class _Memory:
    """Addresses that nothing is ever read from or written to."""

    def __init__(self):
        self.next = 0x7000_0000_0000

    def __call__(self, n=1 << 20):
        self.next += (n + 4095) // 4096 * 4096
        return self.next - (n + 4095) // 4096 * 4096


class _Context:
    workspace = np.zeros(1 << 26, dtype=np.uint8)            # (one, so that addresses in it are the same in every run)

    def __init__(self, B, tables=3, rows=1000, dim=16, batch=64, per_bag=1, hot=100, staging=400):
        self.B, self.T, self.batch, self.nnz = B, tables, batch, tables * batch * per_bag
        self.hot, self.staging, self.mem = hot, staging, _Memory()
        geom = B.make_geometry([rows] * tables, dim, 1)
        n = B.hl_workspace_bytes(geom, batch, self.nnz, hot, staging)
        assert n + 256 <= self.workspace.size
        self.ctx = B.hl_create(geom, batch, self.nnz, hot, staging, (self.workspace.ctypes.data + 255) // 256 * 256, n)
        self.cache, self.table = self.mem(), self.mem()

    def inputs(self, batch=None):
        batch = batch or self.batch
        return self.B.make_batch(self.mem(), self.mem(), batch, self.nnz * batch // self.batch)

    def one_set(self):
        B, m = self.B, self.mem
        return dict(perm=m(), counts=m(), pop=B.make_ubatch(m(), m(), self.nnz), non=B.make_ubatch(m(), m(), self.nnz),
                    cold_rows=m(), n_cold=m(), fwd_src=m(), pooled_pop=m(), pooled_non=m(), slots=m(), bags=m(), n=m())

    def close(self):
        self.B.hl_destroy(self.ctx)


def _pipe_run(B, lib, steps, n_sets=4, batch=64, order=0, same_inputs=3, traced_from=None):
    """A pipeline over ``steps`` mini-batches of two sizes (those from ``traced_from`` on traced); the log of what it queued."""
    c = _Context(B, batch=batch)
    sets = []
    for _ in range(n_sets):
        s = c.one_set()
        sets.append(B.hl_pipe_set(s["perm"], s["counts"], s["pop"], s["non"], s["cold_rows"], s["n_cold"], s["fwd_src"],
                                  s["pooled_pop"], s["pooled_non"], None, s["slots"], s["bags"], s["n"]))
    main = c.mem()
    p = B.hl_pipe_create(c.ctx, c.cache, c.table, c.staging // 2, sets, 0, main)
    B.hl_pipe_set_order(p, order)
    inputs = [c.inputs(batch if k % 2 else batch - 13) for k in range(same_inputs)]
    grads = [(c.mem(), c.mem()) for _ in range(3)]
    marks = []
    for j in range(n_sets - 2):
        B.hl_pipe_submit(p, inputs[j % same_inputs], None, "resident" if j % 2 else None)
    for j in range(steps):
        marks.append(lib.fake_lines())
        if j == traced_from:
            B.hl_pipe_trace_begin(p, 1000, B.HL_SPAN_ALL)
        gp, gn = grads[j % 3]
        B.hl_pipe_step(p, gp, gn, 0.1 + 0.01 * (j % 5), inputs[(j + n_sets - 2) % same_inputs], None, "resident")
    log = _log(lib)
    B.hl_pipe_destroy(p)
    c.close()
    return log, marks


@pytest.mark.parametrize("batch, order, n_sets", [(64, 0, 4), (64, 1, 3), (16384, 0, 4), (16384, 1, 5)])
def test_graphs_queue_what_plain_launches_queue(B, lib, batch, order, n_sets):
    """The same run with and without graphs, over the first, second and all later visits of every slot, with inputs,
    gradients, learning rates and mini-batch sizes that change from step to step (16 384: the sort on its own stream)."""
    steps = 3000
    lib.fake_reset()
    lib.fake_fail(b"cudaGraphInstantiate", -1)
    plain, _ = _pipe_run(B, lib, steps, n_sets, batch, order)
    assert not any(x.startswith("graph") for x in plain)
    lib.fake_reset()
    with_graphs, marks = _pipe_run(B, lib, steps, n_sets, batch, order)
    a, b = [_name(x) + " " + _what(x) for x in plain], [_name(x) + " " + _what(x) for x in with_graphs]
    assert len(a) == len(b)
    differ = [(x, y) for x, y in zip(a, b) if x != y]
    assert not differ, differ[:2]
    late = with_graphs[marks[-20]:]
    assert sum(x.startswith("graph") for x in late) > 100 and not any(x.startswith("plain") for x in late)


@pytest.mark.parametrize("tables, batch, lookups, sort", [
    (21, 4096, 21 * 4096, ["k_sort_segments"]), (3, 43008, 3 * 43008, ["k_sort_segments"]), (60, 16384, 60 * 16384, ["k_sort_segments"]),
    (21, 4096, 21 * 4096 - 1, ["k_sort_pass"] * 3), (21, 1000, 21 * 1000 - 1, ["k_sort_cluster"]),    # some bags empty, others long?
    (100, 82, 8200, ["k_sort_segments"]), (101, 81, 8181, ["k_sort_cluster"]), (1000, 8, 8000, ["k_sort_cluster"]),
    (120, 400, 48_000, ["k_sort_segments"]), (121, 400, 48_400, ["k_sort_pass"] * 3), (61, 8193, 61 * 8193, ["k_sort_pass"] * 3),
    (6, 16385, 6 * 16385, ["k_sort_segments"]), (7, 16385, 7 * 16385, ["k_sort_pass"] * 3),
    (3, 32769, 3 * 32769, ["k_sort_segments"]), (4, 32769, 4 * 32769, ["k_sort_pass"] * 3), (1, 65537, 65537, ["k_sort_pass"] * 3)])
def test_tables_are_sorted_by_themselves_where_their_clusters_fit_the_chip(B, lib, tables, batch, lookups, sort):
    """And where a mini-batch has as many lookups as bags: otherwise one table may have most of them."""
    c = _Context(B, tables=tables, batch=batch, rows=20, dim=4, hot=60_000, staging=60_000)
    s, side, st = c.mem(), c.mem(), c.one_set()
    step_buffers = B.make_step_buffers(st["perm"], st["counts"], st["pop"], st["non"], None, st["cold_rows"], st["n_cold"],
                                       st["pooled_pop"], st["pooled_non"])
    for n in (lookups, tables * batch - 1, lookups):         # (a mini-batch of the other kind in between)
        at = lib.fake_lines()
        B.hl_step(c.ctx, B.make_batch(c.mem(), c.mem(), batch, n), None, 0, step_buffers, c.cache, c.table, c.mem(), c.mem(),
                  0.1, False, s, side)
        if n == lookups:
            names = [_name(x).split("<")[0] for x in _log(lib, at)]
            assert [x for x in names if x.startswith("k_sort")] == sort
    c.close()


@pytest.mark.parametrize("dim, written, read", [(16, 32, 32), (64, 32, 296)])
def test_popular_rows_of_a_table_in_device_memory_move_with_the_whole_chip(B, lib, dim, written, read):
    """Few CTAs are for the host link: a table on the device, as one allocation or one per table, has none in its way."""
    c = _Context(B, dim=dim, hot=100_000, batch=16)
    s, hot_rows, n_hot = c.mem(), c.mem(), c.mem()

    def grids():
        at = lib.fake_lines()
        B.hl_flush_hot(c.ctx, c.cache, hot_rows, n_hot, c.table, s)
        B.hl_build_remap(c.ctx, hot_rows, n_hot, c.table, c.cache, None, s)
        return [int(x.split("grid=")[1].split(" ")[0]) for x in _log(lib, at) if _name(x).startswith("k_move_rows")]

    assert grids() == [written, read]
    lib.fake_device_memory(c.table)
    assert grids() == [296, 296]
    per_table = [c.mem() for _ in range(c.T)]
    for on_device in range(c.T + 1):             # (all of them have to be)
        B.hl_set_host_tables(c.ctx, per_table)
        assert grids() == ([296, 296] if on_device == c.T else [written, read])
        if on_device < c.T:
            lib.fake_device_memory(per_table[on_device])
    c.close()


def test_many_runs_of_kernels_with_many_argument_sets_all_become_graphs(B, lib):
    """A pipeline issued call by call: nine calls per mini-batch, four buffer sets, inputs that change.  No run of kernels
    may push out another's graph for ever: in the steady state nothing is built and nothing is launched plainly."""
    c = _Context(B, per_bag=3)
    sets, s = [c.one_set() for _ in range(4)], c.mem()
    inputs = [c.inputs() for _ in range(5)]
    gp, gn = c.mem(), c.mem()

    def mini_batch(j):
        st, prev = sets[j % 4], sets[(j - 1) % 4]
        w = c.staging // 2
        B.hl_fragment(c.ctx, inputs[j % 5], None, 0, st["perm"], st["counts"], st["pop"], st["non"], None, s)
        B.hl_index_cold(c.ctx, st["non"], st["counts"] + 4, w * (j % 2), w, st["cold_rows"], st["n_cold"], prev["cold_rows"],
                        prev["n_cold"], st["fwd_src"], s)
        B.hl_embbag_bwd_prepare2(c.ctx, st["pop"], st["counts"], st["non"], st["counts"] + 4, st["slots"], st["bags"],
                                 st["n"], s)
        B.hl_stage_cold(c.ctx, c.table, c.cache, w * (j % 2), w, st["cold_rows"], st["n_cold"], st["fwd_src"], s)
        B.hl_embbag_fwd(c.ctx, c.cache, st["pop"], st["counts"], st["pooled_pop"], s)
        B.hl_embbag_bwd_apply2(c.ctx, c.cache, st["slots"], st["bags"], st["n"], 0, gp, 0.1, s)
        B.hl_embbag_fwd(c.ctx, c.cache, st["non"], st["counts"] + 4, st["pooled_non"], s)
        B.hl_embbag_bwd_apply2(c.ctx, c.cache, st["slots"], st["bags"], st["n"], 1, gn, 0.1, s)
        B.hl_scatter_cold_at(c.ctx, c.cache, w * (j % 2), w, st["cold_rows"], st["n_cold"], c.table, s)

    for j in range(4000):
        mini_batch(j)
    at, built = lib.fake_lines(), lib.fake_calls(b"cudaGraphInstantiate")
    for j in range(4000, 4040):
        mini_batch(j)
    late = _log(lib, at)
    plain = sorted({_name(x) for x in late if x.startswith("plain")})
    assert plain == [] and sum(x.startswith("graph") for x in late) > 400
    assert lib.fake_calls(b"cudaGraphInstantiate") == built
    c.close()


def test_graphs_are_built_when_plain_launches_have_cost_as_much(B, lib):
    """A graph costs as much as some 30 plain launches: the first repeats of a call pay for none.  A pipeline builds those of
    all its slots before its first mini-batch, none later, and none that it never launches (the update of the popular rows
    by itself is the first mini-batch's alone)."""
    c = _Context(B)
    s, tags, rrpv, hits = c.mem(), c.mem(), c.mem(), c.mem()
    for k in range(5):
        B.hl_tracker_update(c.ctx, c.inputs(), tags, rrpv, 64, 16, hits, s)
    assert lib.fake_calls(b"cudaGraphInstantiate") == 0
    for k in range(100):
        B.hl_tracker_update(c.ctx, c.inputs(), tags, rrpv, 64, 16, hits, s)
    assert lib.fake_calls(b"cudaGraphInstantiate") >= 1
    c.close()
    for order, first in ((0, 1), (1, 0)):                # (the sort of 32 K lookups and more is a run of its own)
        for batch, more in ((64, 0), (16384, 1)):
            for n_sets, slots in ((4, 4), (3, 6)):
                lib.fake_reset()
                log, marks = _pipe_run(B, lib, 0, n_sets, batch, order)
                built = lib.fake_calls(b"cudaGraphInstantiate")
                assert built == slots * (5 + 2 * more) + first
                lib.fake_reset()
                log, marks = _pipe_run(B, lib, 60, n_sets, batch, order)
                # (the first two mini-batches have nothing to forward, and no sort before them to wait for)
                assert lib.fake_calls(b"cudaGraphInstantiate") == built
                assert len([x for x in log[marks[2]:] if x.startswith("plain")]) <= 2


def test_a_graph_that_cannot_be_changed_or_built_gives_way_to_plain_launches(B, lib):
    c = _Context(B)
    s, grads = c.mem(), [c.mem() for _ in range(40)]
    st = c.one_set()

    def update(k):
        at = lib.fake_lines()
        B.hl_embbag_bwd_sgd(c.ctx, c.cache, st["pop"], st["counts"], grads[k % 40], 0.1, s)
        return _log(lib, at)

    k = 0
    while not all(x.startswith("graph") for x in update(k)):
        k += 1
        assert k < 1000
    lib.fake_fail(b"cudaGraphExecKernelNodeSetParams", -1)
    for _ in range(200):
        k += 1
        lines = update(k)
        # whichever way: all kernels of the call, with this call's gradient
        assert [_name(x).split("<")[0] for x in lines if x[:5] in ("plain", "graph")][-2:] == ["k_bwd_chunks", "k_bwd_spans"]
        assert grads[k % 40].to_bytes(8, "little").hex() in [x for x in lines if "k_bwd_chunks" in x][0]
    lib.fake_fail(b"cudaGraphExecKernelNodeSetParams", 0)
    while not all(x.startswith("graph") for x in update(k)):
        k += 1
        assert k < 2000
    lib.fake_fail(b"cudaGraphLaunch", -1)
    with pytest.raises(B.HotlineError) as e:
        update(k)
    assert e.value.status == B.HL_ECUDA
    c.close()


def test_a_captured_stream_gets_plain_launches_only(B, lib):
    """Under stream capture the kernels go out one by one (they become nodes of the caller's graph), with no graph of the
    library's own launched or built, before and after the library has graphs of these kernels."""
    c = _Context(B)
    s, st, grad = c.mem(), c.one_set(), c.mem()

    def call():
        at = lib.fake_lines()
        B.hl_embbag_fwd(c.ctx, c.cache, st["pop"], st["counts"], st["pooled_pop"], s)
        B.hl_embbag_bwd_sgd(c.ctx, c.cache, st["pop"], st["counts"], grad, 0.1, s)
        return _log(lib, at)

    first = call()
    for warm in (0, 300):
        for _ in range(warm):
            call()
        built, launched = lib.fake_calls(b"cudaGraphInstantiate"), lib.fake_calls(b"cudaGraphLaunch")
        lib.fake_capture(s, 1)
        lines = [call() for _ in range(100)]
        lib.fake_capture(s, 0)
        assert all([_what(x) for x in ls] == [_what(x) for x in first] and all(x.startswith("plain") for x in ls)
                   for ls in lines)
        assert (lib.fake_calls(b"cudaGraphInstantiate"), lib.fake_calls(b"cudaGraphLaunch")) == (built, launched)
    assert launched > 100
    c.close()


def test_traced_mini_batches_launch_kernel_by_kernel(B, lib):
    """The spans of a trace bracket kernels: none of them holds the building of a graph."""
    lib.fake_reset()
    log, marks = _pipe_run(B, lib, 400, batch=16384, traced_from=100)
    untraced, traced = log[marks[90]:marks[100]], log[marks[100]:]
    assert any(x.startswith("graph") for x in untraced) and not any(x.startswith("graph") for x in traced)
    kernels = [_name(x) for x in untraced if x[:5] in ("plain", "graph")]
    assert sorted(kernels) == sorted(_name(x) for x in log[marks[300]:marks[310]] if x.startswith("plain"))


@pytest.mark.parametrize("which", ["hl_index_cold", "hl_gather_cold", "hl_index_cold_begin", "hl_step", "hl_pipe_submit"])
def test_marks_left_by_a_call_that_failed_are_cleared_before_the_next_ones(B, lib, which):
    """Cold rows are marked in the bitmap by one kernel and ranked (and the marks cleared) by another.  The launch of the
    second one fails: the call says so, and the next call on the context first clears the bitmap; the one after that
    does not."""
    lib.fake_fail(b"cudaGraphInstantiate", -1)               # (kernel by kernel)
    c = _Context(B)
    s, side, st, b = c.mem(), c.mem(), c.one_set(), c.inputs()
    pipe = None
    if which == "hl_pipe_submit":
        sets = [B.hl_pipe_set(x["perm"], x["counts"], x["pop"], x["non"], x["cold_rows"], x["n_cold"], x["fwd_src"],
                              x["pooled_pop"], x["pooled_non"], None, x["slots"], x["bags"], x["n"])
                for x in (c.one_set() for _ in range(6))]
        pipe = B.hl_pipe_create(c.ctx, c.cache, c.table, c.staging // 2, sets, 0, s)
    step_buffers = B.make_step_buffers(st["perm"], st["counts"], st["pop"], st["non"], None, st["cold_rows"], st["n_cold"],
                                       st["pooled_pop"], st["pooled_non"])

    def call():
        at = lib.fake_lines()
        if which == "hl_index_cold":
            B.hl_index_cold(c.ctx, st["non"], st["counts"] + 4, 0, c.staging, st["cold_rows"], st["n_cold"], None, None, None, s)
        elif which == "hl_gather_cold":
            B.hl_gather_cold(c.ctx, st["non"], st["counts"] + 4, c.table, c.cache, st["cold_rows"], st["n_cold"], s)
        elif which == "hl_index_cold_begin":
            B.hl_index_cold_begin(c.ctx, st["non"], st["counts"] + 4, 0, c.staging, st["cold_rows"], st["n_cold"], s)
        elif which == "hl_step":
            B.hl_step(c.ctx, b, None, 0, step_buffers, c.cache, c.table, c.mem(), c.mem(), 0.1, False, s, side)
        else:
            B.hl_pipe_submit(pipe, b, None, "resident")
        return _log(lib, at)

    def clears(lines):
        """Positions of clears of the bitmap and of the kernel that marks."""
        rank = [x for x in lines if _name(x).startswith("k_cold_rank")][0]
        bits, words = rank.split(" ")[7][:16], (3000 + 31) // 32
        cleared = [i for i, x in enumerate(lines) if _name(x) == "k_clear_words" and
                   x.split(" ")[7:9] == [bits, words.to_bytes(8, "little").hex()]]
        marked = [i for i, x in enumerate(lines) if _name(x).startswith(("k_cold_classify", "k_frag_place"))]
        return cleared, marked[0]

    assert clears(call())[0] == []
    lib.fake_fail_kernel(b"k_cold_rank")
    with pytest.raises(B.HotlineError) as e:
        call()
    assert e.value.status == B.HL_ECUDA
    lib.fake_fail_kernel(None)
    cleared, marked = clears(call())
    assert len(cleared) == 1 and cleared[0] < marked
    assert clears(call())[0] == []
    if pipe:
        B.hl_pipe_destroy(pipe)
    c.close()


@pytest.mark.parametrize("which", ["hl_embbag_bwd_sgd", "hl_embbag_bwd_apply", "hl_embbag_bwd_apply2", "hl_step", "hl_pipe_step"])
def test_runs_listed_by_a_call_that_failed_are_taken_off_the_list(B, lib, which):
    """The sum kernel lists the runs that the span kernel finishes.  The span kernel's launch fails: the call says so, and
    the next update on the context starts with an empty list; the one after that clears nothing."""
    lib.fake_fail(b"cudaGraphInstantiate", -1)               # (kernel by kernel)
    c = _Context(B)
    s, side, st, b, grad = c.mem(), c.mem(), c.one_set(), c.inputs(), c.mem()
    step_buffers = B.make_step_buffers(st["perm"], st["counts"], st["pop"], st["non"], None, st["cold_rows"], st["n_cold"],
                                       st["pooled_pop"], st["pooled_non"])
    sets = [B.hl_pipe_set(x["perm"], x["counts"], x["pop"], x["non"], x["cold_rows"], x["n_cold"], x["fwd_src"],
                          x["pooled_pop"], x["pooled_non"], None, x["slots"], x["bags"], x["n"])
            for x in (c.one_set() for _ in range(4))]
    pipe = B.hl_pipe_create(c.ctx, c.cache, c.table, c.staging // 2, sets, 0, s)
    if which == "hl_pipe_step":
        for _ in range(3):
            B.hl_pipe_submit(pipe, b, None, "resident")

    def call():
        at = lib.fake_lines()
        if which == "hl_embbag_bwd_sgd":
            B.hl_embbag_bwd_sgd(c.ctx, c.cache, st["pop"], st["counts"], grad, 0.1, s)
        elif which == "hl_embbag_bwd_apply":
            B.hl_embbag_bwd_apply(c.ctx, c.cache, st["slots"], st["bags"], st["n"], grad, 0.1, s)
        elif which == "hl_embbag_bwd_apply2":
            B.hl_embbag_bwd_apply2(c.ctx, c.cache, st["slots"], st["bags"], st["n"], 1, grad, 0.1, s)
        elif which == "hl_step":
            B.hl_step(c.ctx, b, None, 0, step_buffers, c.cache, c.table, grad, grad, 0.1, False, s, side)
        else:
            B.hl_pipe_step(pipe, grad, grad, 0.1, None, None)
        return _log(lib, at)

    def clears(lines):
        sums = [i for i, x in enumerate(lines) if _name(x).startswith("k_bwd_chunks")]
        count = lines[sums[0]].split(" ")[7 + 11]
        return [i for i, x in enumerate(lines) if _name(x) == "k_clear_words" and x.split(" ")[7] == count], sums[0]

    assert clears(call())[0] == []
    lib.fake_fail_kernel(b"k_bwd_spans")
    with pytest.raises(B.HotlineError) as e:
        call()
    assert e.value.status == B.HL_ECUDA
    lib.fake_fail_kernel(None)
    cleared, first = clears(call())
    assert len(cleared) == 1 and cleared[0] < first
    if which != "hl_pipe_step":
        assert clears(call())[0] == []
    B.hl_pipe_destroy(pipe)
    c.close()
