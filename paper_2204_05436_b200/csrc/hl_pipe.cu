// The software-pipelined schedule over mini-batches, issued from native code.
//
//   index stream  mini-batch j+L: fragment (X's lookups classified on the way), ranks of the cold rows, slots + match with
//                 the cold rows of j+L-1 + (slot, bag) pairs, sort (more than 32 K lookups: on the sort stream)
//   link stream   hl_stage_cold(j+1)           after the write-back of j-1 (host rows final, window free) and after
//                                              mini-batch j took the rows it shares with j-1 out of that window and
//                                              updated O (read_beside_update: or beside that)
//   main stream   forward O (+ those rows), update O, [rows of j staged] forward X, update X            mini-batch j
//   write-back    hl_scatter_cold_at(j)        after the update of X
//
// L = n_sets - 2 mini-batches of index-only work ahead; set j % n_sets holds mini-batch j; window j % 2 its cold rows.
//
// Small mini-batches are bound by the host: what counts is the number of launches and event operations per mini-batch.
// The index work is one stream (two), so that its steps need no events between them, and as few kernels as its data
// dependences allow (five where one kernel sorts, otherwise four and one per sort digit); the rows forwarded between
// windows ride on the popular forward.  13 to 15 kernels, no memset and 12 to 15 event operations, where separate calls on
// three streams made 22, 3 and 25 (8 K lookups: 88 us per mini-batch).  The kernels between two event operations go out as one
// graph (hl_graph.cu), five to eight of them: 17 us on the host instead of 41; 30 to 35 us per mini-batch instead of 54.
#include "hl_common.cuh"

#include <memory>
#include <new>
#include <vector>

struct hl_pipe {
    hl_ctx* ctx;
    float* cache;
    float* host_table;
    int64_t window_rows;
    int n_sets, n_dense;
    std::vector<hl_pipe_set> sets;
    cudaStream_t main, index, sort, link, wb;
    struct Events {
        cudaEvent_t inputs, pairs, index, gather, forward, x, scatter;
    };
    std::vector<Events> ev;
    // the graphs of mini-batch j's kernels: slot j % slots, so that set and window, and with them nearly all arguments, are
    // the same whenever a slot is used.  They are there before the first mini-batch is queued (build_graphs).
    std::vector<std::unique_ptr<hl::LaunchCache>> launches;
    // mini-batches whose index work is queued (indexed), whose host read is queued (submitted), whose main work is queued
    // (done)
    int64_t j_indexed, j_submitted, j_done;
    int order;                   // HL_PIPE_ORDER_*
    int wb_mode;                 // HL_PIPE_WB_*
    bool wb_pending;             // HL_PIPE_WB_AFTER_FORWARD: the write-back of mini-batch j_done - 1 is not queued yet
    // trace (hl_pipe_trace_begin / _end): one event pair per recorded span
    struct Span {
        cudaEvent_t b, e;
        int32_t mini_batch, what, stream;
        bool closed;
    };
    std::vector<Span> spans;
    size_t n_spans;              // spans opened so far
    uint32_t trace_mask;         // bit `what` set: spans of that kind are recorded; 0 = not tracing
    int64_t cur_mb;              // mini-batch the call being issued belongs to (for spans opened by the kernel timers)
    int cur_stream;
    int open_timer[HL_TIMER_COUNT];
};

using namespace hl;

namespace {

#define HL_PIPE_TRY(expr)                         \
    do {                                          \
        const int32_t st__ = (expr);              \
        if (st__ != HL_OK) return st__;           \
    } while (0)

int32_t wait(cudaStream_t s, cudaEvent_t e) { return cudaStreamWaitEvent(s, e, 0) == cudaSuccess ? HL_OK : HL_ECUDA; }
int32_t record(cudaEvent_t e, cudaStream_t s) { return cudaEventRecord(e, s) == cudaSuccess ? HL_OK : HL_ECUDA; }

// ---- trace ---------------------------------------------------------------------------------------------------
enum { kMain = 0, kIndex = 1, kSort = 2, kLink = 4, kWb = 5 };

cudaStream_t stream_of(hl_pipe* p, int id) {
    cudaStream_t all[6] = {p->main, p->index, p->sort, nullptr, p->link, p->wb};
    return all[id];
}

// Opens a span of kind `what` for mini-batch `mb` on stream `id`: its begin event is recorded now.  -1 = not recorded.
int span_open(hl_pipe* p, int what, int64_t mb, int id) {
    p->cur_mb = mb;
    p->cur_stream = id;
    if (!(p->trace_mask >> what & 1u) || p->n_spans >= p->spans.size()) return -1;
    hl_pipe::Span& sp = p->spans[p->n_spans];
    if (cudaEventRecord(sp.b, stream_of(p, id)) != cudaSuccess) return -1;
    sp.mini_batch = (int32_t)mb;
    sp.what = what;
    sp.stream = id;
    sp.closed = false;
    return (int)p->n_spans++;
}

void span_close(hl_pipe* p, int idx) {
    if (idx < 0) return;
    hl_pipe::Span& sp = p->spans[idx];
    sp.closed = cudaEventRecord(sp.e, stream_of(p, sp.stream)) == cudaSuccess;
}

// the library's kernel timers (the movers' kernels, the backward's sum kernel, the forward kernel) seen from here
void on_timer_mark(void* user, int which, int end, cudaStream_t) {
    hl_pipe* p = static_cast<hl_pipe*>(user);
    if (which < 0 || which >= HL_TIMER_COUNT) return;
    if (!end) p->open_timer[which] = span_open(p, HL_SPAN_KERNEL + which, p->cur_mb, p->cur_stream);
    else {
        span_close(p, p->open_timer[which]);
        p->open_timer[which] = -1;
    }
}

// RAII span around one library call
struct Scope {
    hl_pipe* p;
    int idx;
    Scope(hl_pipe* p_, int what, int64_t mb, int id) : p(p_), idx(span_open(p_, what, mb, id)) {}
    ~Scope() { span_close(p, idx); }
};

// where the launches made for mini-batch j are collected (traced spans bracket single calls: then nowhere)
hl::LaunchCache* launches_of(hl_pipe* p, int64_t j) {
    return p->trace_mask ? nullptr : p->launches[j % p->launches.size()].get();
}

// Whether the read of the next mini-batch's rows may start beside O's update (else behind it: queue_mini_batch): where the
// transfers of one mini-batch take hundreds of microseconds, so that the pipelines of a chip keep the link busy between them and
// every wait of a read is lost.  What a mini-batch will move is not known here; its largest number of lookups is.  Three
// pipelines in turn, behind / beside the update, us per mini-batch, bags of 20 lookups (64 at most), 8 tables, by lookups x row:
// 0.5 M x 512 bytes 410 / 414, 1 M 569 / 563, 1.6 M 774 / 762, 2.1 M 974 / 957, 4.2 M 1 663 / 1 637; 2.1 M x 256 bytes 573 / 574
// to 590, 4.2 M 931 / 922; 18 tables of bags of 2, 1.8 M x 336 bytes 382 / 385; all smaller ones 9 to 25 % faster behind it.
bool read_beside_update(const hl_ctx* ctx) { return ctx->max_nnz * ctx->D > int64_t(160) << 20; }

// Before the first mini-batch is queued: a graph of every run of kernels that a mini-batch like this one makes in slot j, so
// that no mini-batch has to launch them one by one or to wait while one is built (some 2 ms for the five to eight runs of four slots;
// built when a slot's mini-batch came, they made mini-batches three to eight 200 to 600 us each).  Nothing is launched.  The
// runs are those of queue_index and queue_mini_batch.
void build_graphs(hl_pipe* p, int64_t j, const hl_batch* b, const float* d_dense) {
    hl_ctx* ctx = p->ctx;
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (p->trace_mask || ctx->max_nnz == 0 || ctx->timing_on || ctx->mark_hook || ctx->marks_suspect ||
        ctx->spans_suspect)
        return;
    if (cudaStreamIsCapturing(p->main, &capturing) != cudaSuccess || capturing != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return;
    }
    const int n = p->n_sets;
    hl_pipe_set &st = p->sets[j % n], &prev = p->sets[(j + n - 1) % n];
    const int64_t rows = p->window_rows, w = (j % 2) * rows, w_other = rows - w;
    const bool merge = p->order == HL_PIPE_ORDER_EQ5;
    const bool by_table = backward_sorts_tables(ctx, b, merge);
    const int64_t n_clear = backward_sort_clear_words(ctx, merge, by_table);
    const SortAside aside{p->sort, p->ev[j % n].pairs, (int)(j % 2)};
    const SortAside* use = backward_sort_is_long(ctx) ? &aside : nullptr;
    const float* any = st.pooled_pop;                        // (some gradients)
    LaunchBatch batch(p->launches[j].get(), true);
    if (fragment_and_mark(ctx, b, d_dense, d_dense ? p->n_dense : 0, st.perm, st.counts, &st.pop, &st.non,
                          d_dense ? st.dense_out : nullptr, p->index) != HL_OK)
        return;                                              // (the call itself will say so)
    if (use) launch_flush();
    (void)cold_rank(ctx, rows, st.cold_rows, st.n_cold, p->index, ctx->r.bwd_hist[use ? j % 2 : 0], n_clear);
    (void)assign_and_prepare(ctx, &st.pop, st.counts, &st.non, st.counts + 1, w, rows, st.cold_rows, st.n_cold, prev.cold_rows,
                             prev.n_cold, st.fwd_src, st.sorted_slots, st.sorted_bags, st.sorted_n, merge, by_table, p->index, use);
    (void)hl_stage_cold(ctx, p->host_table, p->cache, w, rows, st.cold_rows, st.n_cold, st.fwd_src, p->link);
    launch_flush();
    const auto update = [&](int which) {
        (void)hl_embbag_bwd_apply2(ctx, p->cache, st.sorted_slots, st.sorted_bags, st.sorted_n, which, any, 0.f, p->main);
    };
    if (rows > 0)
        (void)fwd_and_forward_cold(ctx, p->cache, &st.pop, st.counts, st.pooled_pop, w_other, w, rows, st.fwd_src, st.n_cold,
                                   p->main);
    else
        (void)hl_embbag_fwd(ctx, p->cache, &st.pop, st.counts, st.pooled_pop, p->main);
    const bool apart = p->wb_mode == HL_PIPE_WB_AFTER_FORWARD || read_beside_update(ctx);
    if (apart) launch_flush();
    if (!merge) update(0);
    launch_flush();
    // the first mini-batch launches the update by itself, no later one of its slot or of another does
    if (!merge && !apart && j == 0) update(0);
    launch_flush();
    (void)hl_embbag_fwd(ctx, p->cache, &st.non, st.counts + 1, st.pooled_non, p->main);
    if (!merge) update(1);
    else (void)hl_embbag_bwd_apply(ctx, p->cache, st.sorted_slots, st.sorted_bags, st.sorted_n + 2, any, 0.f, p->main);
    (void)hl_scatter_cold_at(ctx, p->cache, w, rows, st.cold_rows, st.n_cold, p->host_table, p->wb);
}

// The index-only work of the next mini-batch (nothing here touches a row).
int32_t queue_index(hl_pipe* p, const hl_batch* b, const float* d_dense, void* inputs_ready) {
    const int64_t j = p->j_indexed;
    const int n = p->n_sets;
    hl_pipe_set& st = p->sets[j % n];
    hl_pipe::Events& e = p->ev[j % n];
    hl_pipe_set* prev = j >= 1 ? &p->sets[(j - 1) % n] : nullptr;
    const int64_t w = (j % 2) * p->window_rows;
    const bool merge = p->order == HL_PIPE_ORDER_EQ5;
    if (inputs_ready == nullptr) {                        // the inputs are complete in main-stream order
        HL_PIPE_TRY(record(e.inputs, p->main));
        HL_PIPE_TRY(wait(p->index, e.inputs));
    } else if (inputs_ready != HL_PIPE_INPUTS_RESIDENT) {
        HL_PIPE_TRY(wait(p->index, static_cast<cudaEvent_t>(inputs_ready)));
    }
    if (j >= n) HL_PIPE_TRY(wait(p->index, e.scatter));   // the buffers of this set were mini-batch j-n_sets's
    LaunchBatch batch(launches_of(p, j));
    {
        Scope sc(p, HL_SPAN_FRAGMENT, j, kIndex);
        HL_PIPE_TRY(fragment_and_mark(p->ctx, b, d_dense, d_dense ? p->n_dense : 0, st.perm, st.counts, &st.pop, &st.non,
                                      d_dense ? st.dense_out : nullptr, p->index));
    }
    if (p->ctx->max_nnz == 0) {
        HL_PIPE_TRY(hl_index_cold(p->ctx, &st.non, st.counts + 1, w, p->window_rows, st.cold_rows, st.n_cold, nullptr,
                                  nullptr, st.fwd_src, p->index));
    }
    // A sort of many pairs goes to a stream of its own, so that its passes overlap the next mini-batch's fragment; scratch
    // set j % 2 was the sort's of mini-batch j-2.
    const bool by_table = backward_sorts_tables(p->ctx, b, merge);
    const int64_t n_clear = backward_sort_clear_words(p->ctx, merge, by_table);
    const SortAside aside{p->sort, e.pairs, (int)(j % 2)};
    const SortAside* use = backward_sort_is_long(p->ctx) ? &aside : nullptr;
    if (use && j >= 2) {
        HL_PIPE_TRY(launch_flush() == cudaSuccess ? HL_OK : HL_ECUDA);
        HL_PIPE_TRY(wait(p->index, p->ev[(j - 2) % n].index));
    }
    if (p->ctx->max_nnz > 0) {
        Scope sc(p, HL_SPAN_INDEX_BEGIN, j, kIndex);
        HL_PIPE_TRY(cold_rank(p->ctx, p->window_rows, st.cold_rows, st.n_cold, p->index, p->ctx->r.bwd_hist[use ? j % 2 : 0],
                              n_clear));
    }
    {
        Scope sc(p, HL_SPAN_SORT, j, kIndex);
        HL_PIPE_TRY(assign_and_prepare(p->ctx, &st.pop, st.counts, &st.non, st.counts + 1, w, p->window_rows, st.cold_rows,
                                       st.n_cold, prev ? prev->cold_rows : nullptr, prev ? prev->n_cold : nullptr,
                                       st.fwd_src, st.sorted_slots, st.sorted_bags, st.sorted_n, merge, by_table, p->index,
                                       use));
    }
    HL_PIPE_TRY(batch.end());
    HL_PIPE_TRY(record(e.index, use ? p->sort : p->index));
    p->j_indexed += 1;
    return HL_OK;
}

int32_t submit_index(hl_pipe* p, const hl_batch* b, const float* d_dense, void* inputs_ready) {
    if (p->j_indexed == 0)
        for (size_t j = 0; j < p->launches.size(); ++j) build_graphs(p, (int64_t)j, b, d_dense);
    return scratch_kept(p->ctx, queue_index(p, b, d_dense, inputs_ready));
}

// the host read of the oldest indexed mini-batch whose rows are not staged yet
int32_t submit_link(hl_pipe* p) {
    const int64_t j = p->j_submitted;
    const int n = p->n_sets;
    hl_pipe_set& st = p->sets[j % n];
    const int64_t w = (j % 2) * p->window_rows;
    HL_PIPE_TRY(wait(p->link, p->ev[j % n].index));
    if (j >= 2) HL_PIPE_TRY(wait(p->link, p->ev[(j - 2) % n].scatter));   // host rows of j-2 final, its window free
    if (j >= 1) HL_PIPE_TRY(wait(p->link, p->ev[(j - 1) % n].forward));   // j-1 took what it needs out of the window
    {
        Scope sc(p, HL_SPAN_STAGE, j, kLink);
        LaunchBatch batch(launches_of(p, j));
        HL_PIPE_TRY(hl_stage_cold(p->ctx, p->host_table, p->cache, w, p->window_rows, st.cold_rows, st.n_cold,
                                  j >= 1 ? st.fwd_src : nullptr, p->link));
        HL_PIPE_TRY(batch.end());
    }
    HL_PIPE_TRY(record(p->ev[j % n].gather, p->link));
    p->j_submitted += 1;
    return HL_OK;
}

// the write-back of mini-batch j (whose main work is queued), behind its backward
int32_t queue_scatter(hl_pipe* p, int64_t j) {
    const int n = p->n_sets;
    hl_pipe_set& st = p->sets[j % n];
    hl_pipe::Events& e = p->ev[j % n];
    const int64_t w0 = (j % 2) * p->window_rows;
    HL_PIPE_TRY(wait(p->wb, e.x));
    {
        Scope sc(p, HL_SPAN_SCATTER, j, kWb);
        LaunchBatch batch(launches_of(p, j));
        HL_PIPE_TRY(hl_scatter_cold_at(p->ctx, p->cache, w0, p->window_rows, st.cold_rows, st.n_cold, p->host_table,
                                       p->wb));
        HL_PIPE_TRY(batch.end());
    }
    return record(e.scatter, p->wb);
}

// HL_PIPE_WB_AFTER_FORWARD: the write-back held over from the previous hl_pipe_step, if there is one
int32_t flush_scatter(hl_pipe* p) {
    if (!p->wb_pending) return HL_OK;
    p->wb_pending = false;
    return queue_scatter(p, p->j_done - 1);
}

}  // namespace

namespace {

// One mini-batch.  What bounds a small one is the chain of short kernels: fragment, ranks, pairs and sort (one for both
// updates, where a sort inside each update would cost its three passes twice), the host read beside the sort.  106 496
// lookups of 64-byte rows: 133 us with a call for each step, 104 us so.
int32_t queue_step(hl_ctx* ctx, const hl_batch* b, const float* d_dense, int32_t n_dense, const hl_step_buffers* s,
                   float* d_cache, float* host_table, const float* d_grad_pop, const float* d_grad_non, float lr,
                   int32_t flags, cudaStream_t main, cudaStream_t side) {
    if (!ctx || !b || !s || !d_cache || !host_table || !d_grad_pop || !d_grad_non || (flags & ~HL_STEP_DEFERRED))
        return HL_EINVAL;
    if (!s->cold_rows || !s->n_cold || !s->pooled_pop || !s->pooled_non || !s->pop.offsets || !s->non.offsets)
        return HL_EINVAL;
    const bool deferred = (flags & HL_STEP_DEFERRED) != 0;
    hl_ubatch pop = s->pop, non = s->non;
    // (2^30 cache slots and more: O's and X's slots do not fit one key space, and every update sorts its own)
    const bool one_sort = ctx->max_nnz > 0 && 2 * (ctx->hot_cap + ctx->staging_cap) + 2 < (int64_t(1) << 31);
    const int32_t* d_n_non = s->counts + 1;
    int32_t *slots = nullptr, *bags = nullptr;
    LaunchBatch batch(ctx->launches);
    const auto to_side = [&]() -> int32_t {                  // what comes next on `side` sees what `main` has so far
        if (side == main) return HL_OK;
        HL_PIPE_TRY(launch_flush() == cudaSuccess ? HL_OK : HL_ECUDA);
        HL_PIPE_TRY(record(ctx->step_ranked, main));
        return wait(side, ctx->step_ranked);
    };
    const auto side_done = [&]() -> int32_t {
        if (side == main) return HL_OK;
        HL_PIPE_TRY(launch_flush() == cudaSuccess ? HL_OK : HL_ECUDA);
        return record(ctx->step_staged, side);
    };
    if (one_sort) {
        const bool by_table = backward_sorts_tables(ctx, b, false);
        HL_PIPE_TRY(fragment_and_mark(ctx, b, d_dense, d_dense ? n_dense : 0, s->perm, s->counts, &pop, &non,
                                      d_dense ? s->dense_out : nullptr, main));
        HL_PIPE_TRY(cold_rank(ctx, ctx->staging_cap, s->cold_rows, s->n_cold, main, ctx->r.bwd_hist[0],
                              backward_sort_clear_words(ctx, false, by_table)));
        HL_PIPE_TRY(to_side());
        HL_PIPE_TRY(hl_stage_cold(ctx, host_table, d_cache, 0, ctx->staging_cap, s->cold_rows, s->n_cold, nullptr, side));
        HL_PIPE_TRY(side_done());
        HL_PIPE_TRY(hl_embbag_fwd(ctx, d_cache, &pop, s->counts, s->pooled_pop, main));
        HL_PIPE_TRY(assign_and_prepare(ctx, &pop, s->counts, &non, d_n_non, 0, ctx->staging_cap, s->cold_rows, s->n_cold,
                                       nullptr, nullptr, nullptr, nullptr, nullptr, ctx->r.bwd_n, false, by_table, main,
                                       nullptr, &slots, &bags));
    } else {
        HL_PIPE_TRY(hl_fragment(ctx, b, d_dense, d_dense ? n_dense : 0, s->perm, s->counts, &pop, &non,
                                d_dense ? s->dense_out : nullptr, main));
        HL_PIPE_TRY(to_side());
        HL_PIPE_TRY(hl_gather_cold(ctx, &non, d_n_non, host_table, d_cache, s->cold_rows, s->n_cold, side));
        HL_PIPE_TRY(side_done());
        HL_PIPE_TRY(hl_embbag_fwd(ctx, d_cache, &pop, s->counts, s->pooled_pop, main));
    }
    const auto update = [&](int which) -> int32_t {
        const float* grad = which ? d_grad_non : d_grad_pop;
        if (one_sort) return hl_embbag_bwd_apply2(ctx, d_cache, slots, bags, ctx->r.bwd_n, which, grad, lr, main);
        return hl_embbag_bwd_sgd(ctx, d_cache, which ? &non : &pop, which ? d_n_non : s->counts, grad, lr, main);
    };
    if (!deferred) HL_PIPE_TRY(update(0));
    if (side != main) {
        HL_PIPE_TRY(launch_flush() == cudaSuccess ? HL_OK : HL_ECUDA);
        HL_PIPE_TRY(wait(main, ctx->step_staged));
    }
    HL_PIPE_TRY(hl_embbag_fwd(ctx, d_cache, &non, d_n_non, s->pooled_non, main));
    if (deferred) HL_PIPE_TRY(update(0));
    HL_PIPE_TRY(update(1));
    HL_PIPE_TRY(hl_scatter_cold(ctx, d_cache, s->cold_rows, s->n_cold, host_table, main));
    return batch.end();
}

}  // namespace

extern "C" int32_t hl_step(hl_ctx* ctx, const hl_batch* b, const float* d_dense, int32_t n_dense,
                           const hl_step_buffers* s, float* d_cache, float* host_table, const float* d_grad_pop,
                           const float* d_grad_non, float lr, int32_t flags, void* main_stream, void* side_stream) {
    return scratch_kept(ctx, queue_step(ctx, b, d_dense, n_dense, s, d_cache, host_table, d_grad_pop, d_grad_non, lr, flags,
                                      static_cast<cudaStream_t>(main_stream), static_cast<cudaStream_t>(side_stream)));
}

extern "C" hl_pipe* hl_pipe_create_ex(hl_ctx* ctx, float* d_cache, float* host_table, int64_t window_rows,
                                      int32_t n_sets, const hl_pipe_set* sets, int32_t n_dense, void* main_stream,
                                      const hl_pipe_options* opt) {
    if (!ctx || !d_cache || !host_table || !sets || n_sets < 3 || n_sets > 16 || window_rows < 0 ||
        2 * window_rows > ctx->staging_cap || n_dense < 0)
        return nullptr;
    for (int i = 0; i < n_sets; ++i) {
        const hl_pipe_set& s = sets[i];
        if (!s.perm || !s.counts || !s.pop.offsets || !s.non.offsets || !s.cold_rows || !s.n_cold || !s.fwd_src ||
            !s.pooled_pop || !s.pooled_non || !s.sorted_n || (n_dense > 0 && !s.dense_out))
            return nullptr;
        if (ctx->max_nnz > 0 && (!s.pop.ids || !s.non.ids || !s.sorted_slots || !s.sorted_bags)) return nullptr;
    }
    if (opt && (opt->write_back < HL_PIPE_WB_OVERLAP || opt->write_back > HL_PIPE_WB_AFTER_FORWARD)) return nullptr;
    hl_pipe* p = new (std::nothrow) hl_pipe();
    if (!p) return nullptr;
    p->ctx = ctx;
    p->cache = d_cache;
    p->host_table = host_table;
    p->window_rows = window_rows;
    p->n_sets = n_sets;
    p->n_dense = n_dense;
    p->sets.assign(sets, sets + n_sets);
    p->main = static_cast<cudaStream_t>(main_stream);
    p->j_indexed = p->j_submitted = p->j_done = 0;
    p->order = HL_PIPE_ORDER_FIG8;
    p->wb_mode = opt ? opt->write_back : HL_PIPE_WB_OVERLAP;
    p->wb_pending = false;
    p->n_spans = 0;
    p->trace_mask = 0;
    p->cur_mb = 0;
    p->cur_stream = kMain;
    for (auto& t : p->open_timer) t = -1;
    int lo = 0, hi = 0;
    cudaDeviceGetStreamPriorityRange(&lo, &hi);          // hi = numerically lowest = highest priority
    auto clamp = [&](int prio) { return prio < hi ? hi : (prio > lo ? lo : prio); };
    const int index_prio = clamp(opt ? opt->index_priority : 0), link_prio = clamp(opt ? opt->link_priority : 0);
    cudaStream_t* side[4] = {&p->index, &p->sort, &p->link, &p->wb};
    bool ok = true;
    for (int i = 0; i < 4; ++i) {
        *side[i] = nullptr;
        ok = ok && cudaStreamCreateWithPriority(side[i], cudaStreamNonBlocking, i < 2 ? index_prio : link_prio) ==
                       cudaSuccess;
    }
    p->launches.resize(n_sets % 2 ? 2 * n_sets : n_sets);
    for (auto& l : p->launches) {
        l.reset(new (std::nothrow) LaunchCache(1));
        ok = ok && l;
    }
    p->ev.resize(n_sets);
    for (auto& e : p->ev) {
        cudaEvent_t* all[7] = {&e.inputs, &e.pairs, &e.index, &e.gather, &e.forward, &e.x, &e.scatter};
        for (auto x : all) {
            *x = nullptr;
            ok = ok && cudaEventCreateWithFlags(x, cudaEventDisableTiming) == cudaSuccess;
        }
    }
    if (!ok) {
        hl_pipe_destroy(p);
        return nullptr;
    }
    return p;
}

extern "C" hl_pipe* hl_pipe_create(hl_ctx* ctx, float* d_cache, float* host_table, int64_t window_rows,
                                   int32_t n_sets, const hl_pipe_set* sets, int32_t n_dense, void* main_stream) {
    return hl_pipe_create_ex(ctx, d_cache, host_table, window_rows, n_sets, sets, n_dense, main_stream, nullptr);
}

extern "C" void hl_pipe_destroy(hl_pipe* p) {
    if (!p) return;
    if (p->wb_pending && p->wb) (void)flush_scatter(p);      // a write-back held over is not lost
    cudaStream_t side[4] = {p->index, p->sort, p->link, p->wb};
    for (auto s : side)
        if (s) {
            cudaStreamSynchronize(s);
            cudaStreamDestroy(s);
        }
    for (auto& e : p->ev) {
        cudaEvent_t all[7] = {e.inputs, e.pairs, e.index, e.gather, e.forward, e.x, e.scatter};
        for (auto x : all)
            if (x) cudaEventDestroy(x);
    }
    if (p->ctx && p->ctx->mark_user == p) {
        p->ctx->mark_hook = nullptr;
        p->ctx->mark_user = nullptr;
    }
    for (auto& sp : p->spans) {
        if (sp.b) cudaEventDestroy(sp.b);
        if (sp.e) cudaEventDestroy(sp.e);
    }
    delete p;
}

extern "C" int32_t hl_pipe_submit(hl_pipe* p, const hl_batch* b, const float* d_dense, void* inputs_ready) {
    if (!p || !b) return HL_EINVAL;
    if (p->j_indexed - p->j_done >= p->n_sets - 1) return HL_ECAPACITY;    // every spare buffer set is in flight
    HL_PIPE_TRY(submit_index(p, b, d_dense, inputs_ready));
    if (p->j_submitted == p->j_done) HL_PIPE_TRY(submit_link(p));          // nothing staged ahead yet
    return HL_OK;
}

static int32_t queue_mini_batch(hl_pipe* p, const float* d_grad_pop, const float* d_grad_non, float lr, const hl_batch* next,
                                const float* d_next_dense, void* next_inputs_ready, int32_t* set_index) {
    if (!p || !d_grad_pop || (!d_grad_non && p->order != HL_PIPE_ORDER_EQ5)) return HL_EINVAL;
    const int64_t j = p->j_done;
    if (p->j_submitted < j + 1) return HL_EINVAL;          // hl_pipe_submit first
    const int n = p->n_sets;
    hl_pipe_set& st = p->sets[j % n];
    hl_pipe::Events& e = p->ev[j % n];
    const int64_t w0 = (j % 2) * p->window_rows, w1 = ((j + 1) % 2) * p->window_rows;
    if (next && p->j_indexed - j >= n - 1) return HL_ECAPACITY;
    HL_PIPE_TRY(wait(p->main, e.index));
    if (p->wb_mode == HL_PIPE_WB_EXCLUSIVE && j >= 1) HL_PIPE_TRY(wait(p->main, p->ev[(j - 1) % n].scatter));
    LaunchBatch popular(launches_of(p, j));
    {
        // with O's forward: the rows shared with mini-batch j-1, out of its staging window (its backward is done)
        Scope sc(p, HL_SPAN_FWD_POP, j, kMain);
        if (j >= 1 && p->window_rows > 0)
            HL_PIPE_TRY(fwd_and_forward_cold(p->ctx, p->cache, &st.pop, st.counts, st.pooled_pop, w1, w0, p->window_rows,
                                             st.fwd_src, st.n_cold, p->main));
        else
            HL_PIPE_TRY(hl_embbag_fwd(p->ctx, p->cache, &st.pop, st.counts, st.pooled_pop, p->main));
    }
    // The read of j+1's rows may start when those that j takes out of its window are gone.  It has to wait for the write-back of
    // j-1 in any case, which began when this forward did and takes about as long as forward and update, so the event comes
    // behind both, and they go out as one graph.  (In between it cost more than the 2 us from one graph to the next: the
    // update waited behind what the read put on the chip.  One pipeline / three in turn on one chip, us per mini-batch: Tiny
    // 36.3 -> 32.5 / 37.1 -> 32.7, click log 69.2 -> 68.3 / 77.4 -> 64.5, time series 58.3 -> 60.1 / 70.9 -> 57.4, DLRM-sized
    // 146 -> 137 / 150 -> 132.)  The first mini-batch has no write-back before it, one that is held over starts here, and the
    // longest transfers are better off beside the update (read_beside_update).
    const bool apart = j == 0 || p->wb_pending || read_beside_update(p->ctx);
    const auto read_next = [&]() -> int32_t {
        HL_PIPE_TRY(popular.end());
        HL_PIPE_TRY(record(e.forward, p->main));
        if (p->wb_pending) {
            // the write-back of j-1 starts when the popular forward of j is over: of all kernels of the main stream that
            // one loses most next to a write-back
            HL_PIPE_TRY(wait(p->wb, e.forward));
            HL_PIPE_TRY(flush_scatter(p));
        }
        if (p->j_submitted == j + 1 && p->j_submitted < p->j_indexed) return submit_link(p);   // mini-batch j+1
        return HL_OK;
    };
    if (apart) HL_PIPE_TRY(read_next());
    if (p->order == HL_PIPE_ORDER_FIG8) {
        Scope sc(p, HL_SPAN_BWD_POP, j, kMain);
        LaunchBatch update(launches_of(p, j));               // (part of `popular`, unless that has ended)
        HL_PIPE_TRY(hl_embbag_bwd_apply2(p->ctx, p->cache, st.sorted_slots, st.sorted_bags, st.sorted_n, 0, d_grad_pop,
                                         lr, p->main));
        HL_PIPE_TRY(update.end());
    }
    if (!apart) HL_PIPE_TRY(read_next());
    HL_PIPE_TRY(wait(p->main, e.gather));
    LaunchBatch batch(launches_of(p, j));
    {
        Scope sc(p, HL_SPAN_FWD_NON, j, kMain);
        HL_PIPE_TRY(hl_embbag_fwd(p->ctx, p->cache, &st.non, st.counts + 1, st.pooled_non, p->main));
    }
    {
        Scope sc(p, HL_SPAN_BWD_NON, j, kMain);
        if (p->order == HL_PIPE_ORDER_FIG8)
            HL_PIPE_TRY(hl_embbag_bwd_apply2(p->ctx, p->cache, st.sorted_slots, st.sorted_bags, st.sorted_n, 1, d_grad_non,
                                             lr, p->main));
        else   // one update of every touched row with the gradient of the whole mini-batch
            HL_PIPE_TRY(hl_embbag_bwd_apply(p->ctx, p->cache, st.sorted_slots, st.sorted_bags, st.sorted_n + 2, d_grad_pop,
                                            lr, p->main));
    }
    HL_PIPE_TRY(batch.end());
    HL_PIPE_TRY(record(e.x, p->main));
    p->j_done += 1;
    if (p->wb_mode == HL_PIPE_WB_AFTER_FORWARD && next)
        p->wb_pending = true;            // queued by the next hl_pipe_step (or by whatever call comes instead)
    else
        HL_PIPE_TRY(queue_scatter(p, j));
    if (next) {
        HL_PIPE_TRY(submit_index(p, next, d_next_dense, next_inputs_ready));
        if (p->j_submitted == j + 1) HL_PIPE_TRY(submit_link(p));           // j+1 was indexed only just now
    }
    if (set_index) *set_index = (int32_t)(j % n);
    return HL_OK;
}

extern "C" int32_t hl_pipe_step(hl_pipe* p, const float* d_grad_pop, const float* d_grad_non, float lr,
                                const hl_batch* next, const float* d_next_dense, void* next_inputs_ready,
                                int32_t* set_index) {
    return scratch_kept(p ? p->ctx : nullptr, queue_mini_batch(p, d_grad_pop, d_grad_non, lr, next, d_next_dense,
                                                               next_inputs_ready, set_index));
}

extern "C" int32_t hl_pipe_set_order(hl_pipe* p, int32_t order) {
    if (!p || (order != HL_PIPE_ORDER_FIG8 && order != HL_PIPE_ORDER_EQ5)) return HL_EINVAL;
    if (p->j_indexed != 0) return HL_EINVAL;       // the sorts queued so far were made for the other order
    p->order = order;
    return HL_OK;
}

extern "C" int32_t hl_pipe_trace_begin(hl_pipe* p, int32_t max_spans, uint32_t what_mask) {
    if (!p || max_spans < 1 || max_spans > (1 << 16) || what_mask == 0) return HL_EINVAL;
    if ((int)p->spans.size() < max_spans) {
        const size_t old = p->spans.size();
        p->spans.resize(max_spans);
        for (size_t i = old; i < p->spans.size(); ++i) p->spans[i].b = p->spans[i].e = nullptr;
        for (size_t i = old; i < p->spans.size(); ++i)
            if (cudaEventCreate(&p->spans[i].b) != cudaSuccess || cudaEventCreate(&p->spans[i].e) != cudaSuccess) {
                p->spans.resize(i);      // (an event of the failed pair, if any, is leaked with the pipeline's others)
                return HL_ECUDA;
            }
    }
    p->n_spans = 0;
    p->trace_mask = what_mask;
    for (auto& t : p->open_timer) t = -1;
    p->ctx->mark_hook = on_timer_mark;
    p->ctx->mark_user = p;
    return HL_OK;
}

extern "C" int32_t hl_pipe_trace_end(hl_pipe* p, hl_pipe_span* out, int32_t cap, int32_t* n_out) {
    if (!p || !n_out || cap < 0 || (cap > 0 && !out)) return HL_EINVAL;
    p->trace_mask = 0;
    if (p->ctx->mark_user == p) {
        p->ctx->mark_hook = nullptr;
        p->ctx->mark_user = nullptr;
    }
    HL_PIPE_TRY(hl_pipe_drain(p));
    // times are relative to the earliest begin among the recorded spans
    int first = -1;
    for (size_t i = 0; i < p->n_spans; ++i) {
        if (!p->spans[i].closed) continue;
        if (first < 0) {
            first = (int)i;
            continue;
        }
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, p->spans[first].b, p->spans[i].b) == cudaSuccess && ms < 0.f) first = (int)i;
    }
    int32_t n = 0;
    for (size_t i = 0; i < p->n_spans && n < cap; ++i) {
        const hl_pipe::Span& sp = p->spans[i];
        if (!sp.closed) continue;
        float b = 0.f, e = 0.f;
        if (cudaEventElapsedTime(&b, p->spans[first].b, sp.b) != cudaSuccess ||
            cudaEventElapsedTime(&e, p->spans[first].b, sp.e) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        out[n].mini_batch = sp.mini_batch;
        out[n].what = sp.what;
        out[n].stream = sp.stream;
        out[n].begin_ms = b;
        out[n].end_ms = e;
        ++n;
    }
    *n_out = n;
    p->n_spans = 0;
    return HL_OK;
}

extern "C" int32_t hl_pipe_wait_outputs(hl_pipe* p, void* stream) {
    // makes `stream` wait for the last write-back issued (the main stream's own work it sees in order)
    if (!p) return HL_EINVAL;
    if (p->j_done == 0) return HL_OK;
    HL_PIPE_TRY(flush_scatter(p));
    return wait(static_cast<cudaStream_t>(stream), p->ev[(p->j_done - 1) % p->n_sets].scatter);
}

extern "C" int32_t hl_pipe_wait_counts(hl_pipe* p, void* stream) {
    // perm and counts of the mini-batch last stepped are final once its index work has run
    if (!p) return HL_EINVAL;
    if (p->j_done == 0) return HL_OK;
    return wait(static_cast<cudaStream_t>(stream), p->ev[(p->j_done - 1) % p->n_sets].index);
}

extern "C" int32_t hl_pipe_drain(hl_pipe* p) {
    if (!p) return HL_EINVAL;
    HL_PIPE_TRY(flush_scatter(p));
    cudaStream_t all[5] = {p->main, p->index, p->sort, p->link, p->wb};
    for (auto s : all)
        if (cudaStreamSynchronize(s) != cudaSuccess) return HL_ECUDA;
    return HL_OK;
}
