// The approximate access logger of the learning phase (Section V-B "Efficient Embedding Tracking"): a set-associative
// table of row tags with a 2-bit re-reference prediction value per block, replaced by SRRIP with insertion one below
// the maximum, the set chosen by a Feistel randomizer of the (index, table) tuple (Section V-C).
//
// The ASIC serves one access after the other; the result depends on that order only within a set.  So the lookups of
// a mini-batch are keyed by their set and sorted stably (their order within a set stays the order of the layout),
// and a warp replays each set's run of the sorted list in turn, the ways of the set held one per lane.
#include "hl_common.cuh"

namespace hl {
namespace {

constexpr int kThreads = 256;
constexpr int kRrpvMax = 3;        // 2-bit counter; also the value of an empty way
constexpr int kRrpvInsert = 2;     // one below the maximum

// Four Feistel rounds on the 16-bit halves of the key; round function = upper half of (x * odd constant + round key).
__device__ __forceinline__ uint32_t randomizer(uint32_t g) {
    uint32_t left = g >> 16, right = g & 0xffffu;
    const uint32_t rk[4] = {0x85EBCA6Bu, 0xC2B2AE35u, 0x27D4EB2Fu, 0x165667B1u};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t f = (right * 0x9E3779B1u + rk[r]) >> 16;
        const uint32_t t = left ^ f;
        left = right;
        right = t;
    }
    return (left << 16) | right;
}

// (set, row) of every lookup, at the lookup's own position; lookups outside their table get the sentinel set n_sets.
// HIST: also the digit counts of the sort that follows (ghist [passes][256], zero on entry).
template <bool HIST>
__global__ void __launch_bounds__(kThreads) k_trk_keys(const int32_t* __restrict__ indices,
                                                       const int32_t* __restrict__ offsets, int64_t n_bags,
                                                       int64_t bags_per_table, const int64_t* __restrict__ table_base,
                                                       int64_t max_nnz, uint32_t n_sets, int32_t* __restrict__ keys,
                                                       int32_t* __restrict__ vals, int32_t* __restrict__ d_n,
                                                       uint32_t* ghist, int passes, int32_t* status) {
    __shared__ uint32_t h[HIST ? 4 : 1][256];
    if (HIST) {
        for (int i = threadIdx.x; i < 4 * 256; i += kThreads) (&h[0][0])[i] = 0;
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int64_t L = offsets[n_bags];
        if (L > max_nnz) {
            set_status(status, HL_ECAPACITY);
            L = max_nnz;
        }
        d_n[0] = (int32_t)(L < 0 ? 0 : L);
    }
    // the lookup at position j, of table t (first row `base`, so many rows)
    auto put = [&](int64_t j, int32_t idx, int64_t base, int64_t rows) {
        uint32_t key = n_sets;
        int32_t val = -1;
        if (idx < 0 || idx >= rows) {
            set_status(status, HL_EBOUNDS);
        } else {
            const uint32_t g = (uint32_t)(base + idx);
            key = randomizer(g) % n_sets;
            val = (int32_t)g;
        }
        keys[j] = (int32_t)key;
        vals[j] = val;
        if (HIST)
            for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(key >> (8 * p)) & 255u], 1u);
    };
    // a thread's bags, U at a time: their offsets and first lookups are asked for together
    constexpr int U = 4;
    const int64_t n_threads = (int64_t)gridDim.x * blockDim.x;
    for (int64_t bag0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; bag0 < n_bags; bag0 += U * n_threads) {
        int64_t lo[U], hi[U], base[U], rows[U];
        int32_t idx[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t bag = min(bag0 + u * n_threads, n_bags - 1);
            const uint32_t t = (uint32_t)bag / (uint32_t)bags_per_table;             // (fewer than 2^30 bags)
            base[u] = table_base[t];
            rows[u] = table_base[t + 1] - base[u];
            lo[u] = offsets[bag];
            hi[u] = bag0 + u * n_threads < n_bags ? min((int64_t)offsets[bag + 1], max_nnz) : lo[u];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) idx[u] = lo[u] < hi[u] ? indices[lo[u]] : 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (lo[u] < hi[u]) put(lo[u], idx[u], base[u], rows[u]);
            for (int64_t j = lo[u] + 1; j < hi[u]; ++j) put(j, indices[j], base[u], rows[u]);
        }
    }
    if (HIST) {
        __syncthreads();
        for (int i = threadIdx.x; i < passes * 256; i += kThreads) {
            const uint32_t c = (&h[0][0])[i];
            if (c) atomicAdd(&ghist[i], c);
        }
    }
}

// One warp per 32 positions of the sorted list: every position where a new set's run begins is a head, and the warp
// replays, head after head, the accesses of that set (the run of the last head may reach far beyond the warp's own 32 positions;
// the warps there find no head in it and leave it alone).  A set's ways are held one per lane; W lanes (the power of two that
// holds the ways) replay a set, so that 32 / W sets go on side by side.  The last head's run is then replayed by its W lanes
// alone, up to 32 lookups at a time.
//
// What bounds it is the chain of votes per access, and latency: of a set's blocks, which come from DRAM, and, in the set of a
// popular row (thousands of lookups of a mini-batch), of the lookups themselves.  So the blocks of the next rounds' sets are on
// their way while one round's are replayed, the 64 lookups behind the warp's first stay in registers, and beyond them four
// groups of 32 are read at once (eight: no faster).  426 K lookups, 131 072 sets of 16, the whole update: 72.9 us with a set per
// warp, 66.2 so (replay 30.1 -> 26.7, keys 8.3 -> 7.2); sets of 8 74.0 -> 64.7; 10 K lookups 26.4 -> 21.6.  A set that is replayed
// alone -- more than 16 ways, or the last head's run -- is asked for its oldest blocks only after a miss: with all five votes per
// access, as sets side by side have to, 10 K lookups, 20 ways 17.7 us instead of 14.1 (32 ways 14.5 / 11.2), 426 K of 6 250 sets of 16
// 49.3 / 43.5, of 65 536 sets of 32 42.3 / 38.4.  (16 ways with 48 registers instead of 40, five CTAs instead of six: 28.7 / 27.8.)
template <int W>
__global__ void __launch_bounds__(kThreads) k_trk_replay(const int32_t* __restrict__ keys,
                                                         const int32_t* __restrict__ vals,
                                                         const int32_t* __restrict__ d_n, int64_t n_max,
                                                         int32_t* __restrict__ tags, uint8_t* __restrict__ rrpv,
                                                         int64_t n_sets, int ways,
                                                         unsigned long long* __restrict__ d_hits) {
    constexpr unsigned kAll = 0xffffffffu, kMine = W == 32 ? kAll : (1u << (W & 31)) - 1u;
    constexpr int NG = 32 / W;                                   // sets side by side
    constexpr int kAhead = 4;                                    // groups of 32 lookups read at once
    int64_t n = d_n[0];
    n = n < 0 ? 0 : (n < n_max ? n : n_max);
    const int lane = threadIdx.x & 31, way = lane % W, group = lane / W, shift = group * W;
    const int64_t n_warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    unsigned hits = 0;                                           // of this lane's group
    struct Blocks {
        int64_t s;
        int tag, rr;
    };
    for (int64_t w0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; w0 < n; w0 += n_warps * 32) {
        auto key_at = [&](int64_t i) { return i < n ? keys[i] : -1; };
        auto val_at = [&](int64_t i) { return i < n ? vals[i] : -1; };
        const int64_t p = w0 + lane;
        const int32_t k0 = key_at(p), k1 = key_at(p + 32), g0 = val_at(p), g1 = val_at(p + 32);
        const int32_t before = w0 > 0 ? keys[w0 - 1] : -1;
        const int32_t up = __shfl_up_sync(kAll, k0, 1);
        // positions where a run begins, of a set or of lookups that are skipped; heads: of a set
        const unsigned begins = __ballot_sync(kAll, k0 != (lane ? up : before));
        unsigned heads = begins & __ballot_sync(kAll, k0 >= 0 && k0 < n_sets);
        if (!heads) continue;
        const int last_head = 31 - __clz((int)heads);
        // the next head of every group (32: none), and its blocks: -2 matches no row; RRPV -1 is never a victim and never aged
        auto take = [&]() {
            int mine = 32;
#pragma unroll
            for (int k = 0; k < NG; ++k) {
                const int h = heads ? __ffs((int)heads) - 1 : 32;
                heads &= heads - 1;
                if (k == group) mine = h;
            }
            return mine;
        };
        auto load = [&](int h) {
            Blocks b{-1, -2, -1};
            const int32_t s = __shfl_sync(kAll, k0, h & 31);
            if (h < 32) {
                b.s = s;
                if (way < ways) {
                    b.tag = tags[b.s * ways + way];
                    b.rr = (int)rrpv[b.s * ways + way];
                }
            }
            return b;
        };
        // One access of one set, whose lanes are on, row gg: asked for its oldest blocks only where the row is not among them (the
        // votes are what an access takes).
        auto access_one = [&](Blocks& b, int32_t gg, bool on) {
            const unsigned hit = __ballot_sync(kAll, on && b.tag == gg);
            if (hit) {
                if (lane == __ffs((int)hit) - 1) b.rr = 0;
                hits += on && way == 0;
                return;
            }
            unsigned oldest = __ballot_sync(kAll, on && b.rr == kRrpvMax);
            if (!oldest) {
                const int add = __any_sync(kAll, on && b.rr == 2) ? 1 : __any_sync(kAll, on && b.rr == 1) ? 2 : 3;
                if (on && b.rr >= 0) b.rr += add;
                oldest = __ballot_sync(kAll, on && b.rr == kRrpvMax);
            }
            if (lane == __ffs((int)oldest) - 1) {
                b.tag = gg;
                b.rr = kRrpvInsert;
            }
        };
        // one access of every group's set (active: it has one), row gg
        auto access = [&](Blocks& b, int32_t gg, bool active) {
            if constexpr (NG == 1) return access_one(b, gg, true);
            const unsigned hit = __ballot_sync(kAll, b.tag == gg) >> shift & kMine;
            const unsigned r3 = __ballot_sync(kAll, b.rr == kRrpvMax) >> shift & kMine;
            const unsigned r2 = __ballot_sync(kAll, b.rr == 2) >> shift & kMine;
            const unsigned r1 = __ballot_sync(kAll, b.rr == 1) >> shift & kMine;
            const unsigned r0 = __ballot_sync(kAll, b.rr == 0) >> shift & kMine;
            if (!active) return;
            if (hit) {
                if (way == __ffs((int)hit) - 1) b.rr = 0;
                hits += way == 0;
            } else {                      // (no block at the maximum: the whole set ages until its oldest one is)
                const int add = r3 ? 0 : r2 ? 1 : r1 ? 2 : 3;
                const unsigned oldest = r3 ? r3 : r2 ? r2 : r1 ? r1 : r0;
                if (b.rr >= 0) b.rr += add;
                if (way == __ffs((int)oldest) - 1) {
                    b.tag = gg;
                    b.rr = kRrpvInsert;
                }
            }
        };
        auto store = [&](const Blocks& b) {
            if (b.s >= 0 && way < ways) {
                tags[b.s * ways + way] = b.tag;
                rrpv[b.s * ways + way] = (uint8_t)b.rr;
            }
        };
        const auto any = [&](bool x) { return NG == 1 ? x : (bool)__any_sync(kAll, x); };      // (of one group: the same in all)
        int h = take(), h_next = take();
        Blocks next = load(h), after = load(h_next);
        while (any(h < 32)) {
            Blocks now = next;
            const int at = h;
            next = after;
            h = h_next;
            h_next = take();
            after = load(h_next);
            // its run: up to the next one's beginning, or, of the last head, what of it is among the 32
            const unsigned behind = at < 31 ? begins & (kAll << (at + 1)) : 0u;
            const int end = at < 32 ? (behind ? __ffs((int)behind) - 1 : 32) : 0;
            for (int t = at; any(t < end); ++t) access(now, __shfl_sync(kAll, g0, t & 31), t < end);
            // the last head's run may go on
            const bool on = at == last_head && end == 32;
            if (any(on)) {
                const int from = __ffs((int)__ballot_sync(kAll, on)) - 1;            // a lane of the group it is in
                const int32_t set = (int32_t)__shfl_sync(kAll, now.s, from);
                // the row of the previous access, and whether that left it at RRPV 0, so that repeating it changes nothing
                int32_t last = __shfl_sync(kAll, g0, 31);
                bool last_zero = __any_sync(kAll, on && now.tag == last && now.rr == 0);
                // replays one group of up to 32 lookups; false: the run ended in it
                auto replay = [&](int32_t k, int32_t g) {
                    const unsigned same = __ballot_sync(kAll, k == set);
                    const int c = same == kAll ? 32 : __ffs((int)~same) - 1;                       // leading lanes of the run
                    if (last_zero && __all_sync(kAll, lane >= c || g == last)) {
                        if (on && way == 0) hits += c;                                // a burst of one popular row
                        return c == 32;
                    }
                    for (int t = 0; t < c; ++t) {
                        const int32_t gg = __shfl_sync(kAll, g, t);
                        if (last_zero && gg == last) {
                            hits += on && way == 0;
                            continue;
                        }
                        access_one(now, gg, on);
                        last = gg;
                        last_zero = __any_sync(kAll, on && now.tag == gg && now.rr == 0);
                    }
                    return c == 32;
                };
                bool more = replay(k1, g1);
                for (int64_t i = w0 + 64; more; i += 32 * kAhead) {
                    int32_t k[kAhead], g[kAhead];
#pragma unroll
                    for (int u = 0; u < kAhead; ++u) {
                        k[u] = key_at(i + 32 * u + lane);
                        g[u] = val_at(i + 32 * u + lane);
                    }
#pragma unroll
                    for (int u = 0; u < kAhead; ++u)
                        if (more) more = replay(k[u], g[u]);
                }
            }
            store(now);
        }
    }
    unsigned long long all = hits;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) all += __shfl_down_sync(kAll, all, d);
    if (lane == 0 && d_hits && all) atomicAdd(d_hits, all);
}

// counts[row] = 4 - RRPV for every tracked row (the counters were cleared before).
__global__ void __launch_bounds__(kThreads) k_trk_export(const int32_t* __restrict__ tags,
                                                         const uint8_t* __restrict__ rrpv, int64_t n_blocks, int64_t N,
                                                         uint32_t* __restrict__ counts, SelectState* sel,
                                                         int32_t* status) {
    unsigned long long mine = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_blocks;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t g = tags[i];
        if (g < 0) continue;
        if (g >= N || rrpv[i] > kRrpvMax) {
            set_status(status, HL_EBOUNDS);
            continue;
        }
        const uint32_t c = (uint32_t)(kRrpvMax + 1 - rrpv[i]);
        counts[g] = c;
        mine += c;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, d);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&sel->total, mine);
}

int bits_for(int64_t max_value) {
    int b = 1;
    while ((int64_t(1) << b) <= max_value) ++b;
    return b;
}

bool tracker_shape_ok(int64_t n_sets, int32_t ways) {
    return n_sets >= 1 && n_sets < (int64_t(1) << 30) && ways >= 1 && ways <= 32;
}

}  // namespace
}  // namespace hl

using namespace hl;

extern "C" int32_t hl_tracker_reset(hl_ctx* ctx, int32_t* d_tags, uint8_t* d_rrpv, int64_t n_sets, int32_t ways,
                                    unsigned long long* d_hits, void* stream_) {
    if (!ctx || !d_tags || !d_rrpv || !tracker_shape_ok(n_sets, ways)) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    HL_CUDA_TRY(cudaMemsetAsync(d_tags, 0xff, sizeof(int32_t) * n_sets * ways, stream));
    HL_CUDA_TRY(cudaMemsetAsync(d_rrpv, kRrpvMax, (size_t)n_sets * ways, stream));
    if (d_hits) HL_CUDA_TRY(cudaMemsetAsync(d_hits, 0, sizeof(unsigned long long), stream));
    return HL_OK;
}

extern "C" int32_t hl_tracker_update(hl_ctx* ctx, const hl_batch* b, int32_t* d_tags, uint8_t* d_rrpv, int64_t n_sets,
                                     int32_t ways, unsigned long long* d_hits, void* stream_) {
    if (!ctx || !b || !d_tags || !d_rrpv || !tracker_shape_ok(n_sets, ways)) return HL_EINVAL;
    if (b->batch < 1 || b->batch > ctx->max_batch || b->nnz < 0 || b->nnz > ctx->max_nnz || !b->offsets ||
        (b->nnz > 0 && !b->indices))
        return HL_EINVAL;
    if (b->nnz == 0 || ctx->max_nnz == 0) return HL_OK;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    Regions& r = ctx->r;
    const int64_t bags_per_table = (int64_t)b->batch * ctx->S;
    const int64_t n_bags = bags_per_table * ctx->T;
    LaunchBatch batch(ctx->launches);
    const int key_bits = bits_for(n_sets);
    const int64_t n_clear = sort_clear_words(ctx->max_nnz, key_bits, WaitCfg());
    if (n_clear > 0) HL_CUDA_TRY(clear_words(r.bwd_hist[0], n_clear, stream));
    // (every CTA adds its digit counts to the same words in the end: 426 K lookups 8.4 us with 3 CTAs per SM, 9.3 with 4,
    // 18 with 16, 11.5 with 1)
    HL_CUDA_TRY(launch(n_clear > 0 ? k_trk_keys<true> : k_trk_keys<false>, grid_for(n_bags, kThreads, 3 * ctx_sms(ctx)),
                       kThreads, stream, b->indices, b->offsets, n_bags, bags_per_table, r.table_base, ctx->max_nnz,
                       (uint32_t)n_sets, r.bwd_keys[0], r.bwd_vals[0], r.bwd_n, r.bwd_hist[0], (key_bits + 7) / 8,
                       r.status));
    note_launches(1);
    HL_LAUNCH_CHECK();
    int32_t *keys, *vals;
    const int32_t st = radix_sort_pairs(r.bwd_keys, r.bwd_vals, r.bwd_n, ctx->max_nnz, key_bits, r.bwd_hist[0], r.status,
                                        &keys, &vals, stream, WaitCfg(), true);
    if (st != HL_OK) return st;
    const auto replay = ways <= 8 ? k_trk_replay<8> : ways <= 16 ? k_trk_replay<16> : k_trk_replay<32>;
    HL_CUDA_TRY(launch(replay, grid_for(ctx->max_nnz, kThreads, kMaxGrid), kThreads, stream, keys, vals, r.bwd_n,
                       ctx->max_nnz, d_tags, d_rrpv, n_sets, ways, d_hits));
    note_launches(1);
    HL_LAUNCH_CHECK();
    return batch.end();
}

extern "C" int32_t hl_tracker_export(hl_ctx* ctx, const int32_t* d_tags, const uint8_t* d_rrpv, int64_t n_sets,
                                     int32_t ways, void* stream_) {
    if (!ctx || !d_tags || !d_rrpv || !tracker_shape_ok(n_sets, ways)) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    Regions& r = ctx->r;
    HL_CUDA_TRY(cudaMemsetAsync(r.counts, 0, sizeof(uint32_t) * ctx->N, stream));
    HL_CUDA_TRY(cudaMemsetAsync(r.sel, 0, sizeof(SelectState), stream));
    const int64_t n_blocks = n_sets * ways;
    HL_CUDA_TRY(launch(k_trk_export, grid_for(n_blocks, kThreads, kMaxGrid), kThreads, stream, d_tags, d_rrpv, n_blocks,
                       ctx->N, r.counts, r.sel, r.status));
    note_launches(1);
    HL_LAUNCH_CHECK();
    return HL_OK;
}
