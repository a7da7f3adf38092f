// Shared declarations of the Hotline sm_100a library: context layout, status word, remap probe.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include <mutex>
#include <tuple>
#include <type_traits>
#include <utility>
#include <vector>

#include "hotline.h"

namespace hl {

constexpr int kSMsFallback = 148;          // used only if the device's SM count cannot be queried (B200: 2 x 74)
constexpr int kRemapRowsPerBlock = 224;    // 7 bitmap words per 32-byte remap block
constexpr int kSortTile = 2048;            // keys per radix-sort tile (256 threads x 8)
constexpr int kSelTile = 8192;             // rows per hot-set selection tile (256 threads x 32)
constexpr int kBwdChunk = 32;              // sorted lookups per backward chunk
constexpr int kMoverCtasDefault = 16;      // working CTAs of a host-link mover inside a schedule: write-backs
constexpr int kReadCtasDefault = 24;       // ... and host reads (a wider read finishes sooner and costs the step nothing)
constexpr int kPacedCtas = 16;             // ... of either, when the transfer is short and therefore paced (hl_cold.cu)
// Per-mini-batch kernels are launched with one CTA per tile of work rather than as chip-filling persistent grids:
// they run next to the host-link movers of another micro-batch, which slow down the SMs they sit on, and the
// hardware block scheduler then simply hands those SMs fewer CTAs.
constexpr int kMaxGrid = 1 << 22;

// One 32-byte sector per 224 rows: w[0] = number of popular rows before this block, w[1..7] = hit bitmap.
struct __align__(32) RemapBlock {
    uint32_t w[8];
};

// State of the count-threshold selection (device memory).
struct SelectState {
    unsigned long long hist[256];
    unsigned long long k_remaining;    // rows still wanted among the current prefix class
    unsigned long long quota_eq;       // rows with count == threshold to keep (in ascending id)
    unsigned long long total;          // lookups counted so far
    unsigned int prefix;               // high digits of the threshold found so far
    unsigned int mask;                 // bits of `prefix` that are fixed
    unsigned int c_min;                // smallest admissible count (>= 1)
    unsigned int threshold;            // final: k-th largest admissible count
    unsigned int finished;             // CTAs done with the current digit
    int take_all;                      // fewer admissible rows than wanted: keep them all
};

struct Regions {
    // common
    int32_t* status;                   // [8]  status[0] = first device error
    int64_t* table_base;               // [T+1]
    unsigned char** table_ptrs;        // [T] host-memory base of every table (hl_set_host_tables), device copy
    RemapBlock* remap;                 // [n_remap_blocks]
    // profile
    uint32_t* counts;                  // [N]
    SelectState* sel;
    unsigned long long* sel_chain;     // [n_sel_tiles + 1]
    // fragment
    uint32_t* frag_words;              // [max_batch / 32 + 1] all-hit flags
    unsigned long long* frag_chain;    // [frag_chain_words]
    // backward
    int32_t* bwd_keys[2];              // [max_nnz]
    int32_t* bwd_vals[2];              // [max_nnz]
    uint32_t* bwd_hist[2];             // [256 * sort tiles]; the second one only for SortAside
    float* bwd_part;                   // [2 * n_chunks * D]
    int32_t* bwd_n;                    // [4] lookups in the micro-batch
    // cold
    uint32_t* cold_bits;               // [cold_bitmap_words] one bit per row; zero between calls
    uint32_t* cold_summary;            // [cold_summary_words] one bit per bitmap word; zero between calls
    uint2* cold_ranked;                // [cold_bitmap_words] bits of the word, rank of its first row
    unsigned long long* cold_chain;    // [cold_chain_words]
    int32_t* cold_n;                   // [4]; [1] = hl_index_cold_verdict, which stays 0
};

class LaunchCache;

}  // namespace hl

struct hl_ctx {
    int32_t T, D, S;
    int64_t N;
    int32_t max_batch;
    int64_t max_nnz, max_bags;
    int64_t hot_cap, staging_cap;
    int64_t n_remap_blocks, n_sel_tiles;
    int device;
    int sms;                           // multiprocessors of `device` (queried at hl_create)
    int mover_ctas, scatter_ctas;      // working CTAs of the host-link movers inside a schedule (hl_set_mover_ctas)
    int mover_width_set;               // 1: chosen by the caller
    int fwd_ctas, bwd_ctas;            // CTAs per multiprocessor of the forward / backward-sum kernel (0 = default)
    int test_poll_limit;               // > 0: poll limit of the bounded device waits (hl_test_bounded_waits)
    int64_t test_stall_tile;           // with it: the tile / mover stage that never delivers (-1: none)
    int64_t* h_table_base;             // host copy [T+1]
    int per_table;                     // 1: the host table is one allocation per table (r.table_ptrs is set)
    int tables_on_device;              // ... and all of them are device memory
    hl::Regions r;
    int timing_on;                     // optional kernel timers (hl_timing_enable)
    cudaEvent_t timer[HL_TIMER_COUNT][2];
    // optional observer of the kernel timers' marks (the pipeline's trace): called with (user, which, end, stream)
    void (*mark_hook)(void*, int, int, cudaStream_t);
    void* mark_user;
    // graphs of the calls that make several kernels, or one in a run of calls (nullptr: plain launches)
    hl::LaunchCache* launches;
    cudaEvent_t step_ranked, step_staged;      // of hl_step
    // a call has failed that may have left cold rows marked, or runs on the backward's list (scratch_kept)
    int marks_suspect, spans_suspect;
};

// Context of the wide-id index path (hl_wide_*): global row ids are 64-bit, every table still has fewer than 2^31
// rows.  Popularity is counted in a hashed counter and the popular rows are found through a hashed remap, so nothing
// here is sized by the number of rows.
struct hl_wide {
    int32_t T, S;
    int64_t N;
    int32_t max_batch;
    int64_t max_nnz, max_bags, hot_cap, staging_cap;
    int64_t counter_slots, remap_slots;     // powers of two
    int sms;
    int64_t* h_table_base;
    // device regions (carved from the caller's workspace)
    int32_t* status;
    int64_t* table_base;                     // [T+1]
    long long* c_keys;                       // [counter_slots] row id or -1
    uint32_t* c_cnt;                         // [counter_slots]
    hl::SelectState* sel;
    unsigned long long* sel_chain;           // [counter_slots / kSelTile + 1]
    int32_t* n_seen;                         // [4]
    int32_t *e_tab, *e_idx;                  // [counter_slots] table and table-local index of every counted row
    uint32_t *e_cnt, *s_cnt;                 // [counter_slots] its count; the counts in row order
    int32_t* s_ent;                          // [counter_slots] entry behind every position of the row order
    int32_t* sel_idx;                        // [hot_cap] selected positions
    long long* r_keys;                       // [remap_slots] popular row or -1
    int32_t* r_vals;                         // [remap_slots] its slot
    int32_t* sort_keys[2];                   // [max(counter_slots, max_nnz)]
    int32_t* sort_vals[2];
    uint32_t* sort_hist;
    uint32_t* frag_words;                    // [max_batch / 32 + 1]
    unsigned long long* frag_chain;
    uint32_t* cold_clear;                    // cold_n, cold_chain and sort_hist, one behind the other
    int32_t* cold_n;                         // cold lookups of X
    unsigned long long* cold_chain;          // [max_nnz / 1024 + 1]
    hl::LaunchCache* launches;
    int test_poll_limit;                     // as in hl_ctx
    int64_t test_stall_tile;
};

namespace hl {

#define HL_CUDA_TRY(...)                          \
    do {                                          \
        cudaError_t e__ = (__VA_ARGS__);          \
        if (e__ != cudaSuccess) return HL_ECUDA;  \
    } while (0)

#define HL_LAUNCH_CHECK()                                  \
    do {                                                   \
        if (cudaGetLastError() != cudaSuccess) return HL_ECUDA; \
    } while (0)

// ---- launches (hl_graph.cu) -----------------------------------------------------------------------------------
// Kernels are launched through `launch`.  Inside a LaunchBatch they are collected instead, per stream, and go out as one
// graph at its end, when the stream changes, or at launch_flush(), which has to come before anything else is put on the
// stream (an event, a memset).
class LaunchCache {
public:
    explicit LaunchCache(int variants);              // graphs of the same kernels, with different arguments, worth keeping
    ~LaunchCache();
    LaunchCache(const LaunchCache&) = delete;
    LaunchCache& operator=(const LaunchCache&) = delete;
    cudaError_t launch(const void* recording, cudaStream_t stream);
    void build(const void* recording);               // a graph of these kernels, if there is none; nothing is launched

private:
    // (A context's calls make some 40 different runs of kernels, over all sizes of mini-batches; a program that had more than
    // these in use would see the longest unused one's graphs built again.)
    static constexpr int kMaxLists = 64, kMaxVariants = 4;
    struct Entry;
    struct List;
    List* list_of(const void* recording);
    List* lists_ = nullptr;
    std::mutex mutex_;
    const int variants_;
    uint64_t tick_ = 0;
    int64_t lost_ns_ = 0;                            // what plain launches have cost, up to the price of a graph
};

class LaunchBatch {
public:
    // cache: nullptr, or inside another batch: nothing of its own.  build_only: the kernels get graphs and are not launched
    explicit LaunchBatch(LaunchCache* cache, bool build_only = false);
    ~LaunchBatch();
    int32_t end(int32_t st = HL_OK);                 // `st`, or HL_ECUDA if that is HL_OK and a launch failed

private:
    bool mine_;
};

cudaError_t launch_flush();
bool launches_build_only();
cudaError_t clear_words(uint32_t* p, int64_t n_words, cudaStream_t stream);      // p[0 .. n_words) = 0
cudaError_t launch_kernel(const void* func, dim3 grid, dim3 block, size_t smem, int cluster, void** args,
                          const uint32_t* sizes, int n_args, cudaStream_t stream);

template <typename... P, typename... A>
cudaError_t launch_cluster(void (*kernel)(P...), int64_t grid, int block, size_t smem, int cluster, cudaStream_t stream,
                           A&&... a) {
    static_assert(sizeof...(P) == sizeof...(A), "one argument per parameter");
    // (arguments are compared byte by byte: LaunchCache)
    static_assert(((std::has_unique_object_representations_v<P> || std::is_floating_point_v<P>) && ...), "no padding");
    std::tuple<P...> args(static_cast<P>(a)...);
    const uint32_t sizes[] = {(uint32_t)sizeof(P)...};
    return std::apply(
        [&](auto&... x) {
            void* ptrs[] = {const_cast<void*>(static_cast<const void*>(&x))...};
            return launch_kernel(reinterpret_cast<const void*>(kernel), dim3((unsigned)grid), dim3((unsigned)block), smem,
                                 cluster, ptrs, sizes, (int)sizeof...(P), stream);
        },
        args);
}
template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), int64_t grid, int block, cudaStream_t stream, A&&... a) {
    return launch_cluster(kernel, grid, block, 0, 0, stream, std::forward<A>(a)...);
}

// f() with its launches collected in `cache` (nullptr: not)
template <typename F>
int32_t as_graph(LaunchCache* cache, F f) {
    LaunchBatch batch(cache);
    return batch.end(f());
}

// Where a call of this context keeps its graphs.  (A call whose kernels are traced launches them one by one, as its spans
// show them, and does not pay for a graph inside a span.)
inline LaunchCache* kept_launches(const hl_ctx* ctx) { return ctx && !ctx->mark_hook ? ctx->launches : nullptr; }

// Records the start/end event of one of the optional kernel timers on `stream` (no-op unless enabled).
inline void timer_mark(hl_ctx* ctx, int which, int end, cudaStream_t stream) {
    if (!ctx->timing_on && !ctx->mark_hook) return;
    launch_flush();
    if (ctx->timing_on && ctx->timer[which][end]) cudaEventRecord(ctx->timer[which][end], stream);
    if (ctx->mark_hook) ctx->mark_hook(ctx->mark_user, which, end, stream);
}

inline int ctx_sms(const hl_ctx* ctx) { return ctx->sms > 0 ? ctx->sms : kSMsFallback; }
// CTAs per multiprocessor of the forward kernel (hl_set_kernel_width; defaults chosen by measurement)
// (rows of up to 128 fp32: the forward kernel is held to 64 registers, so four of its CTAs fit a multiprocessor)
inline int fwd_ctas_per_sm(const hl_ctx* ctx) { return ctx->fwd_ctas > 0 ? ctx->fwd_ctas : (ctx->D <= 128 ? 4 : 3); }

__device__ __forceinline__ void set_status(int32_t* status, int32_t code) {
    atomicCAS(status, 0, code);
}

// Popular rows are looked up in two halves, so that a thread with several lookups has all their loads on the way before it
// waits for the first: `request` (or `request_hit`, for the hit test only) issues them, the other half uses what came.
// Hit test: one 4-byte load.
__device__ __forceinline__ uint32_t remap_word(const RemapBlock* __restrict__ remap, int64_t g) {
    const uint32_t blk = (uint32_t)(g / kRemapRowsPerBlock);
    return __ldg(&remap[blk].w[1 + ((uint32_t)(g - (int64_t)blk * kRemapRowsPerBlock) >> 5)]);
}
__device__ __forceinline__ bool remap_hit(uint32_t word, int64_t g) {        // (a block's rows begin at a multiple of 32)
    return (word >> (g & 31)) & 1u;
}
static_assert(kRemapRowsPerBlock % 32 == 0, "whole words");

// Slot of global row g, or -1: one 32-byte sector.
struct RemapSector {
    uint4 lo, hi;
};
__device__ __forceinline__ RemapSector remap_sector(const RemapBlock* __restrict__ remap, int64_t g) {
    const uint32_t blk = (uint32_t)(g / kRemapRowsPerBlock);
    return {__ldg(reinterpret_cast<const uint4*>(&remap[blk].w[0])), __ldg(reinterpret_cast<const uint4*>(&remap[blk].w[4]))};
}
__device__ __forceinline__ int32_t remap_slot(const RemapSector& s, int64_t g) {
    const uint32_t r = (uint32_t)(g % kRemapRowsPerBlock);
    const uint32_t w[8] = {s.lo.x, s.lo.y, s.lo.z, s.lo.w, s.hi.x, s.hi.y, s.hi.z, s.hi.w};
    const uint32_t wi = 1 + (r >> 5), bit = r & 31;
    uint32_t slot = w[0];
    uint32_t word = 0;
#pragma unroll
    for (uint32_t i = 1; i < 8; ++i) {
        if (i < wi) slot += __popc(w[i]);
        if (i == wi) word = w[i];
    }
    if (!((word >> bit) & 1u)) return -1;
    slot += __popc(word & ((1u << bit) - 1u));
    return (int32_t)slot;
}

// Where the host-DRAM table's rows are: one allocation holding all tables back to back (ptrs == nullptr: row g at
// single + g * row_bytes), or one allocation per table (the address registers of the paper's Data Dispatcher,
// Section V-A): row g of table t at ptrs[t] + (g - base[t]) * row_bytes.
struct TableMap {
    unsigned char* single;
    unsigned char* const* ptrs;
    const int64_t* base;               // [T+1]
    int64_t T;
};

__device__ __forceinline__ unsigned char* row_address(const TableMap& m, int64_t g, int row_bytes) {
    if (m.ptrs == nullptr) return m.single + g * row_bytes;
    int lo = 0, hi = (int)m.T;         // base[lo] <= g < base[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(&m.base[mid]) <= g) lo = mid;
        else hi = mid;
    }
    return m.ptrs[lo] + (g - __ldg(&m.base[lo])) * row_bytes;
}

// ---- the hashed lookup structures of the wide-id path (global row ids beyond 2^31, hl_wide_*) ------------------
// Randomizer of Section V-C on a 64-bit row id: a 4-round Feistel network on its 32-bit halves (a bijection, so
// distinct rows never collide before the reduction to the table size), round function (x * 0x9E3779B1 + K_r)
// rotated by 15 bits.
__host__ __device__ __forceinline__ uint64_t randomize64(uint64_t g) {
    uint32_t l = (uint32_t)(g >> 32), r = (uint32_t)g;
    const uint32_t k[4] = {0x85EBCA6Bu, 0xC2B2AE35u, 0x27D4EB2Fu, 0x165667B1u};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t f = r * 0x9E3779B1u + k[i];
        f = (f << 15) | (f >> 17);
        const uint32_t nl = r;
        r = l ^ f;
        l = nl;
    }
    return ((uint64_t)l << 32) | r;
}

// Open-addressing table row id -> value (linear probing from randomize64(row) & mask; an empty entry holds -1).  A lookup asks
// for the aligned four entries around its first one at a time -- one sector of keys, and their values with them --, so that
// hardly any takes more than one trip to memory (one entry at a time: three or four, for the slowest lane of a warp).
struct HashProbe {
    const long long* keys;             // at least four entries
    const int32_t* vals;
    uint64_t mask;
    struct HitRequest {
        longlong2 k01, k23;
    };
    struct Request {
        HitRequest k;
        int4 v;
    };
    __device__ __forceinline__ uint64_t home(int64_t g) const { return randomize64((uint64_t)g) & mask; }
    __device__ __forceinline__ HitRequest keys_at(uint64_t four) const {
        const longlong2* p = reinterpret_cast<const longlong2*>(keys + four);
        return {__ldg(p), __ldg(p + 1)};
    }
    __device__ __forceinline__ HitRequest request_hit(int64_t g) const { return keys_at(home(g) & ~3ull); }
    __device__ __forceinline__ Request request(int64_t g) const {
        const uint64_t four = home(g) & ~3ull;
        return {keys_at(four), __ldg(reinterpret_cast<const int4*>(vals + four))};
    }
    // which of the four entries, from `from` on, is the first that holds g or nothing (4: none does); found: it holds g
    static __device__ __forceinline__ int stop(const HitRequest& r, int from, int64_t g, bool* found) {
        const long long k[4] = {r.k01.x, r.k01.y, r.k23.x, r.k23.y};
        int at = 4;
        *found = false;
#pragma unroll
        for (int i = 3; i >= 0; --i)
            if (i >= from && (k[i] == g || k[i] < 0)) {
                at = i;
                *found = k[i] == g;
            }
        return at;
    }
    // where g is beyond its first four entries, or -1
    __device__ __forceinline__ int64_t further(int64_t g) const {
        uint64_t four = home(g) & ~3ull;
        for (uint64_t seen = 0; seen <= mask; seen += 4) {           // (back at the first four: those in front of its home)
            four = (four + 4) & mask;
            bool found;
            const int at = stop(keys_at(four), 0, g, &found);
            if (at < 4) return found ? (int64_t)(four + at) : -1;
        }
        return -1;
    }
    __device__ __forceinline__ int32_t slot(const Request& r, int64_t g) const {
        bool found;
        const int at = stop(r.k, (int)(home(g) & 3), g, &found);
        if (at < 4) return !found ? -1 : at == 0 ? r.v.x : at == 1 ? r.v.y : at == 2 ? r.v.z : r.v.w;
        const int64_t h = further(g);
        return h < 0 ? -1 : __ldg(&vals[h]);
    }
    __device__ __forceinline__ bool hit(const HitRequest& r, int64_t g) const {
        bool found;
        const int at = stop(r, (int)(home(g) & 3), g, &found);
        return at < 4 ? found : further(g) >= 0;
    }
};

// The dense form used by the 32-bit path: one 32-byte block per 224 rows (see RemapBlock).
struct BitmapProbe {
    const RemapBlock* remap;
    using Request = RemapSector;
    using HitRequest = uint32_t;
    __device__ __forceinline__ Request request(int64_t g) const { return remap_sector(remap, g); }
    __device__ __forceinline__ HitRequest request_hit(int64_t g) const { return remap_word(remap, g); }
    __device__ __forceinline__ int32_t slot(const Request& r, int64_t g) const { return remap_slot(r, g); }
    __device__ __forceinline__ bool hit(HitRequest r, int64_t g) const { return remap_hit(r, g); }
};

// ---- the cold-row bitmap --------------------------------------------------------------------------------------
// Whether the bitmap is read directly or through a summary.  Reading all of it costs 8 us and 0.28 us per million rows,
// whatever it holds, and its words are dealt out evenly; behind a summary word the rows of small tables pile up on a few
// lanes, so that its time goes by the cold lookups.  k_cold_rank alone, directly / through the summary, 26 tables, us:
//   cold lookups     1.7 K        13 K         39 K         130 K        426 K
//    18 M rows    13.1 / 10.7  13.2 / 22.6  14.3 / 28.8  13.5 / 45.0  14.4 / 60.0
//    64 M         24.9 / 13.0  24.6 / 27.9  23.8 / 40.1  23.9 / 58.3  25.3 / 84.5
//   100 M         36.6 / 13.5  33.2 / 23.6  33.9 / 34.0  37.2 / 52.6  36.0 / 93.0
//   180 M         59.1 / 11.3  59.3 / 20.8  60.3 / 31.1  60.2 / 49.5  58.3 / 80.4
//   257 M         80.1 / 14.9  78.2 / 34.2  75.9 / 48.4  79.2 / 77.0  82.2 / 123.8
// What the host knows is how many lookups a mini-batch has at most.  (Of a learned model's 426 K some 22 K are cold.)
constexpr bool cold_direct(int64_t N, int64_t max_nnz) { return N <= int64_t(1) << (max_nnz > 4096 ? 26 : 24); }
constexpr int64_t cold_bitmap_words(int64_t N) { return (N + 31) / 32; }
constexpr int64_t cold_summary_words(int64_t N) { return (cold_bitmap_words(N) + 31) / 32; }
// one status word per tile of k_cold_rank (at least 256 words per tile)
constexpr int64_t cold_chain_words(int64_t N, int64_t max_nnz) {
    return 1 + (cold_direct(N, max_nnz) ? cold_bitmap_words(N) : cold_summary_words(N)) / 256;
}
// tally, ticket and one status word per tile of k_frag_place (at least 256 bags per tile)
constexpr int64_t frag_chain_words(int64_t max_bags) { return 3 + max_bags / 256 + 1; }

struct ColdMarks {
    uint32_t* bits;
    uint32_t* summary;                 // nullptr: no summary is kept
    uint2* ranked;
    unsigned long long* chain;         // state of k_cold_rank's chained tiles, cleared by the kernel that marks
    int64_t n_chain;
};
inline ColdMarks cold_marks(const hl_ctx* ctx) {
    return {ctx->r.cold_bits, cold_direct(ctx->N, ctx->max_nnz) ? nullptr : ctx->r.cold_summary, ctx->r.cold_ranked,
            ctx->r.cold_chain, cold_chain_words(ctx->N, ctx->max_nnz)};
}

// The chain of the ranking that follows, cleared by the kernel that marks the rows.  (Not by the last CTA of the ranking
// itself: nothing would order its clears behind what the other CTAs published.)
__device__ __forceinline__ void clear_cold_chain(const ColdMarks& marks) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < marks.n_chain; i += (int64_t)gridDim.x * blockDim.x)
        marks.chain[i] = 0ull;
}

// A lookup of X that addresses row g (inside the model) becomes its cache slot if the row is popular; otherwise the row is
// marked in the bitmap and the lookup becomes -2 - g.  (A row that is marked already, as popular cold rows are, costs a load:
// marks.bits[g >> 5], `word` below.)
__device__ __forceinline__ int32_t cold_id(int64_t g) { return (int32_t)(-2 - g); }
__device__ __forceinline__ void mark_cold(const ColdMarks& marks, int64_t g, uint32_t word) {
    const uint32_t bit = 1u << (g & 31);
    if (word & bit) return;
    const int64_t at = g >> 5;
    if (marks.summary == nullptr) {
        atomicOr(&marks.bits[at], bit);              // (nothing comes back, so nothing is waited for)
    } else if (atomicOr(&marks.bits[at], bit) == 0u) {
        atomicOr(&marks.summary[at >> 5], 1u << (at & 31));
    }
}

// Rows are marked and ranked in two kernels or two calls, and the marks must be gone when the next mini-batch's are set: a
// call that ends in between, because a launch or an event failed, would leave its rows to be staged as the next one's.  The
// same goes for the runs that the backward's sum kernel lists and the next kernel finishes and takes off the list.  So every
// call that marks rows or lists runs passes its result through scratch_kept, and the next one clears the bitmap
// (marks_fresh) or the list's counts (launch_bwd) first if one has failed.
inline int32_t scratch_kept(hl_ctx* ctx, int32_t st) {
    if (st != HL_OK && ctx) ctx->marks_suspect = ctx->spans_suspect = 1;
    return st;
}
int32_t marks_fresh(hl_ctx* ctx, cudaStream_t stream);

// The slot of such a lookup once the marked rows are ranked: slot0 + rank, or -1 if there is no room to stage the row
// (the lookup is dropped; k_cold_rank has set the status word).
__device__ __forceinline__ int32_t cold_slot(const uint2* __restrict__ ranked, int32_t id, int64_t slot0,
                                             int64_t staging_cap) {
    const int64_t g = -2 - (int64_t)id;
    const uint2 w = ranked[g >> 5];
    const int64_t rank = (int64_t)w.y + __popc(w.x & ((1u << (g & 31)) - 1u));
    return rank < staging_cap ? (int32_t)(slot0 + rank) : -1;
}

// Position of g in the ascending list rows[0 .. n), or -1.
__device__ __forceinline__ int32_t position_in(const int32_t* __restrict__ rows, int64_t n, int32_t g) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (rows[mid] < g) lo = mid + 1;
        else hi = mid;
    }
    return (lo < n && rows[lo] == g) ? (int32_t)lo : -1;
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// How long the bounded device-side waits poll before they give up (HL_ETIMEOUT), and -- for the tests of that
// path only -- which tile of a chained scan or sort pass publishes nothing, so that the tiles behind it wait in vain
// (-1: none).  Production value: about a second of polling, far beyond any wait that can occur.
struct WaitCfg {
    int max_polls = 1 << 20;
    int64_t stall_tile = -1;
};
template <typename Ctx>                // hl_ctx or hl_wide
inline WaitCfg wait_cfg(const Ctx* ctx) {
    WaitCfg w;
    if (ctx->test_poll_limit > 0) {
        w.max_polls = ctx->test_poll_limit;
        w.stall_tile = ctx->test_stall_tile;
    }
    return w;
}

// ---- chained tiles --------------------------------------------------------------------------------------------
// Sum over the tiles before `tile` of what each of them adds up to (62 bits), in one kernel: a tile publishes its own sum
// (AGGREGATE), all threads of its CTA then look at the tiles before it, one each, until somebody sees one that already
// knows its inclusive prefix (PREFIX), and the tile publishes its prefix.  One round of loads covers NT tiles, so a few
// hundred tiles cost one or two round trips to the L2, where one warp walks them 32 a step (placing 106 thousand bags:
// 11.7 us with a one-warp walk over 416 tiles, 8.2 us with this over 104).  A tile is the CTA's block index (CTAs are
// dispatched in that order, so the tiles before have started), and publishing never waits; every poll is bounded all the
// same, and one that runs out records HL_ETIMEOUT and carries on with what it has.  words[tile]: zero on entry.
// Both calls are made by all NT threads; chain_before's result is the same in all.
constexpr unsigned long long kChainAgg = 1ull << 62, kChainPrefix = 1ull << 63, kChainSum = kChainAgg - 1ull;

__device__ __forceinline__ unsigned long long ld_relaxed64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void chain_publish(unsigned long long* words, int tile, unsigned long long total) {
    if (threadIdx.x == 0) st_relaxed64(&words[tile], (tile == 0 ? kChainPrefix : kChainAgg) | total);
}

template <int NT>
__device__ __forceinline__ unsigned long long chain_before(unsigned long long* words, int tile, unsigned long long total,
                                                           bool publish, int max_polls, int32_t* status) {
    constexpr int NW = NT / 32;
    __shared__ unsigned long long s_sum[NW];
    __shared__ bool s_ends[NW];                      // a prefix among the warp's tiles
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long before = 0;
    for (int t0 = tile - 1; t0 >= 0; t0 -= NT) {
        const int t = t0 - (int)threadIdx.x;
        unsigned long long w = kChainPrefix;         // before tile 0: an empty prefix
        if (t >= 0) {
            int polls = 0;
            while (((w = ld_relaxed64(&words[t])) & (kChainAgg | kChainPrefix)) == 0) {
                if (++polls > max_polls) {
                    set_status(status, HL_ETIMEOUT);
                    w = kChainPrefix;
                    break;
                }
                __nanosleep(20);
            }
        }
        const unsigned with_prefix = __ballot_sync(0xffffffffu, (w & kChainPrefix) != 0);
        const int stop = with_prefix ? __ffs(with_prefix) - 1 : 31;
        unsigned long long val = lane <= stop ? w & kChainSum : 0;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) val += __shfl_xor_sync(0xffffffffu, val, d);
        if (lane == 0) {
            s_sum[warp] = val;
            s_ends[warp] = with_prefix != 0;
        }
        __syncthreads();
        bool ends = false;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            if (!ends) before += s_sum[k];
            ends = ends || s_ends[k];
        }
        __syncthreads();
        if (ends) break;
    }
    if (threadIdx.x == 0 && publish && tile > 0) st_relaxed64(&words[tile], kChainPrefix | ((before + total) & kChainSum));
    return before;
}

// ---- primitives implemented in hl_prims.cu -----------------------------------------------------------------
// Stable LSD radix sort of (key, value) pairs by the low key_bits bits of the keys (as unsigned numbers).
// n = *d_n (clamped to n_max).  Returns in *out_keys / *out_vals which of the two buffers holds the result.
int32_t radix_sort_pairs(int32_t* keys[2], int32_t* vals[2], const int32_t* d_n, int64_t n_max, int key_bits,
                         uint32_t* hist, int32_t* status, int32_t** out_keys, int32_t** out_vals,
                         cudaStream_t stream, WaitCfg w = WaitCfg(), bool counted = false);

// Words at the start of `hist` that must be zero before the sort's digits are counted; 0 if the sort that will be used
// counts none.  A caller that clears them and then counts the keys' digits itself (hist[pass * 256 + digit]) passes
// counted = true.
int64_t sort_clear_words(int64_t n_max, int key_bits, WaitCfg w);

// Whether that many pairs are too many for one cluster, so that their sort is a chain of kernels or fills the chip.
bool sort_is_long(int64_t n_max, WaitCfg w);

// The sort of pairs that lie table by table (O's tables, then X's, or, merged, every table's of O and X together), each
// table's by themselves: equal keys end up side by side, which is what the backward's sums need.
struct SortSide {
    const int32_t* offsets;
    const int32_t* d_n_samples;
    int32_t key_bias, unused;
};
struct SegmentArgs {
    int32_t *keys_in, *vals_in;        // (scratch, if a table does not fit)
    int32_t *keys_out, *vals_out;
    SortSide side[2];
    const int32_t* d_n_lookups;        // [0]: of the first side, [2]: of both
    int32_t tables, max_batch, bags_per_sample, merge, passes, unused;
    int64_t max_nnz;
};
bool sort_by_segments(int64_t n_max, int64_t n_bags, int tables, bool merge, WaitCfg w);
int32_t sort_segments(const SegmentArgs& a, cudaStream_t stream);

// 32-bit words of histogram scratch radix_sort_pairs needs for at most max_nnz pairs.
constexpr int64_t sort_hist_words(int64_t max_nnz) {
    const int64_t n_tiles = ((max_nnz > 0 ? max_nnz : 1) + kSortTile - 1) / kSortTile;
    return 4 * 256 + 4 * n_tiles * 256;   // digit counts, tile status words for up to 4 passes
}

// ints behind the backward's partial sums: count words + (chunk, key, last chunk of the run or -1, unused) per chunk
// of kBwdChunk sorted lookups.
constexpr int64_t bwd_span_list_words(int64_t max_nnz) {
    return 8 + 4 * (((max_nnz > 0 ? max_nnz : 1) + kBwdChunk - 1) / kBwdChunk);
}

// where those ints start
inline int32_t* span_count_of(const hl_ctx* ctx) {
    const int64_t max_chunks = ((ctx->max_nnz > 0 ? ctx->max_nnz : 1) + kBwdChunk - 1) / kBwdChunk;
    return reinterpret_cast<int32_t*>(ctx->r.bwd_part + 2 * max_chunks * ctx->D);
}

// Ranks the rows marked in the cold-row bitmap (hl_cold.cu): d_cold_rows, *d_n_cold, cold_ranked.  Also clears `clear`
// [n_clear words, a multiple of 4; 16-byte aligned], for the kernels that follow.
int32_t cold_rank(hl_ctx* ctx, int64_t stage_rows, int32_t* d_cold_rows, int64_t* d_n_cold, cudaStream_t stream,
                  uint32_t* clear = nullptr, int64_t n_clear = 0);

// hl_embbag_bwd_prepare2 / _merged on what fragment_and_mark and cold_rank left behind (hl_embbag.cu): X's cold lookups
// get their slots, the cold rows are matched against the previous ones, and the pairs are sorted (aside: may be null).  The
// sort's scratch, backward_sort_clear_words words of bwd_hist, is zero already.  d_sorted_slots / _bags may be null: the
// result then stays in the context's scratch, at *out_slots / *out_bags.  by_table: backward_sorts_tables, asked once for a
// mini-batch, since its ranks (which clear the scratch), pairs and sort have to go the same way.
bool backward_sorts_tables(const hl_ctx* ctx, const hl_batch* b, bool merge);
int64_t backward_sort_clear_words(const hl_ctx* ctx, bool merge, bool by_table);
bool backward_sort_is_long(const hl_ctx* ctx);

// The sort on a stream of its own, behind the pairs (event pairs_ready), with one of two sets of scratch (which): the
// pairs of the next mini-batch, written with the other set, need not wait for it.
struct SortAside {
    cudaStream_t stream;
    cudaEvent_t pairs_ready;
    int which;
};
int32_t assign_and_prepare(hl_ctx* ctx, const hl_ubatch* pop, const int32_t* d_n_pop, hl_ubatch* non,
                           const int32_t* d_n_non, int64_t stage_row0, int64_t stage_rows, const int32_t* d_cold_rows,
                           const int64_t* d_n_cold, const int32_t* d_prev_rows, const int64_t* d_n_prev,
                           int32_t* d_fwd_src, int32_t* d_sorted_slots, int32_t* d_sorted_bags, int32_t* d_n_lookups,
                           bool merge, bool by_table, cudaStream_t stream, const SortAside* aside,
                           int32_t** out_slots = nullptr, int32_t** out_bags = nullptr);

// Whether p is device memory (hl_cold.cu).
bool in_device_memory(const void* p);

// Asks for what the backward's sum kernel needs of shared memory for rows of D fp32, on the current device (hl_embbag.cu).
bool piece_memory_granted(int D);

// hl_embbag_fwd and hl_forward_cold in one launch (the bags read no staged row).
int32_t fwd_and_forward_cold(hl_ctx* ctx, float* d_cache, const hl_ubatch* ub, const int32_t* d_n_samples, float* d_out,
                             int64_t from_stage_row0, int64_t to_stage_row0, int64_t stage_rows, const int32_t* d_fwd_src,
                             const int64_t* d_n_cold, cudaStream_t stream);

// hl_fragment with X's lookups classified on the way (hl_fragment.cu): non->ids = cache slots, or -2 - g for a cold row.
int32_t fragment_and_mark(hl_ctx* ctx, const hl_batch* b, const float* d_dense, int32_t n_dense, int32_t* d_perm,
                          int32_t* d_counts, hl_ubatch* pop, hl_ubatch* non, float* d_dense_out, cudaStream_t stream);

// Selection of the rows with the k largest counts (implemented in hl_profile.cu; see there).
int32_t select_rows_by_count(const uint32_t* counts, int64_t n, SelectState* sel, unsigned long long* chain, long long k,
                             long long share_num, long long share_den, int64_t cap, int32_t* out_idx, int64_t* d_n_out,
                             int32_t* status, int sms, WaitCfg w, cudaStream_t stream);

// Process-wide count of kernels this library has launched (read by hl_launch_count).
void note_launches(int n);

inline int64_t div_up(int64_t a, int64_t b) { return (a + b - 1) / b; }
inline int grid_for(int64_t work_items, int per_block, int max_blocks) {
    int64_t b = div_up(work_items, per_block);
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (int)b;
}

}  // namespace hl
