// Learning phase: exact access counting, selection of the popular rows, and the remap structure.
#include "hl_common.cuh"

namespace hl {
namespace {

constexpr int kThreads = 256;

// ---- counting -----------------------------------------------------------------------------------------------
// One thread per bag; a bag's table follows from its position (table-major layout).
__global__ void __launch_bounds__(kThreads) k_count(const int32_t* __restrict__ indices,
                                                    const int32_t* __restrict__ offsets, int64_t n_bags,
                                                    int64_t bags_per_table, const int64_t* __restrict__ table_base,
                                                    uint32_t* __restrict__ counts, SelectState* sel,
                                                    int32_t* status) {
    unsigned long long mine = 0;
    for (int64_t bag = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; bag < n_bags;
         bag += (int64_t)gridDim.x * blockDim.x) {
        const int t = (int)(bag / bags_per_table);
        const int64_t base = table_base[t], rows = table_base[t + 1] - base;
        const int32_t lo = offsets[bag], hi = offsets[bag + 1];
        for (int32_t j = lo; j < hi; ++j) {
            const int32_t idx = indices[j];
            if (idx < 0 || idx >= rows) {
                set_status(status, HL_EBOUNDS);
                continue;
            }
            atomicAdd(&counts[base + idx], 1u);
            ++mine;
        }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, d);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&sel->total, mine);
}

// ---- selection: k-th largest admissible count by 8-bit radix select, most significant digit first ----------
__global__ void k_select_begin(SelectState* sel, unsigned long long k, long long share_num, long long share_den) {
    for (int i = threadIdx.x; i < 256; i += blockDim.x) sel->hist[i] = 0;
    if (threadIdx.x == 0) {
        unsigned int c_min = 1;
        if (share_num > 0) {   // count * den >= total * num  <=>  count >= ceil(total * num / den)
            const unsigned __int128 prod = (unsigned __int128)sel->total * (unsigned __int128)share_num;
            const unsigned __int128 q = (prod + (unsigned __int128)(share_den - 1)) / (unsigned __int128)share_den;
            c_min = q > 0xffffffffull ? 0xffffffffu : (unsigned int)q;
            if (c_min < 1) c_min = 1;
        }
        sel->c_min = c_min;
        sel->k_remaining = k;
        sel->prefix = 0;
        sel->mask = 0;
        sel->take_all = 0;
        sel->threshold = c_min;
        sel->quota_eq = ~0ull;
        sel->finished = 0;
    }
}

// One digit: the histogram of the admissible counts that have the digits found so far, and, in the CTA that finishes last,
// the digit that holds the k-th largest of them (a kernel of one thread for that took 5.7 us a digit).  A digit that no
// count reaches (the lookups counted so far are fewer) is zero without looking.  chain / n_chain: the state of
// k_select_emit's chain, cleared here.
__global__ void __launch_bounds__(kThreads) k_select_digit(const uint32_t* __restrict__ counts, int64_t N, int shift,
                                                           SelectState* sel, unsigned long long* __restrict__ chain,
                                                           int64_t n_chain) {
    __shared__ unsigned int h[256];
    __shared__ unsigned long long s_warp[kThreads / 32];
    __shared__ bool s_last;
    const int64_t thread = (int64_t)blockIdx.x * kThreads + threadIdx.x, n_threads = (int64_t)gridDim.x * kThreads;
    for (int64_t i = thread; i < n_chain; i += n_threads) chain[i] = 0ull;
    if (shift > 0 && (sel->total >> shift) == 0) {           // (nobody changes what this reads)
        if (thread == 0) sel->mask |= 255u << shift;
        return;
    }
    if (sel->take_all) return;
    h[threadIdx.x] = 0;
    __syncthreads();
    const unsigned int c_min = sel->c_min, prefix = sel->prefix, mask = sel->mask;
    auto add = [&](unsigned int c) {
        if (c >= c_min && (c & mask) == prefix) atomicAdd(&h[(c >> shift) & 255u], 1u);
    };
    const uint4* counts4 = reinterpret_cast<const uint4*>(counts);
    for (int64_t g = thread; g < N / 4; g += n_threads) {
        const uint4 c = counts4[g];
        add(c.x);
        add(c.y);
        add(c.z);
        add(c.w);
    }
    if (thread < N % 4) add(counts[N - 1 - thread]);
    __syncthreads();
    if (h[threadIdx.x]) atomicAdd(&sel->hist[threadIdx.x], (unsigned long long)h[threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&sel->finished, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // thread t: digit 255 - t; rows with that digit or a larger one
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long mine = __ldcg(&sel->hist[255 - threadIdx.x]), k = sel->k_remaining;
    unsigned long long incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    for (int w = 0; w < warp; ++w) incl += s_warp[w];
    if (k == 0) {
        if (threadIdx.x == 0) {
            // nothing wanted: a threshold no count exceeds, and no row at the threshold either
            sel->take_all = 1;
            sel->threshold = 0xffffffffu;
            sel->quota_eq = 0ull;
        }
    } else if (incl >= k && incl - mine < k) {
        sel->k_remaining = k - (incl - mine);
        sel->prefix = prefix | (255u - threadIdx.x) << shift;
        sel->mask = mask | 255u << shift;
        if (shift == 0) {
            sel->threshold = sel->prefix;
            sel->quota_eq = sel->k_remaining;
        }
    } else if (threadIdx.x == kThreads - 1 && incl < k) {
        // fewer admissible rows than wanted: keep them all (threshold = c_min, no quota)
        sel->take_all = 1;
        sel->threshold = c_min;
        sel->quota_eq = ~0ull;
    }
    sel->hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) sel->finished = 0;
}

// Ordered compaction: a row is popular if its count beats the threshold, or equals it and fewer than quota_eq
// equal rows precede it.  Its position = popular rows with a smaller id.  A warp takes an eighth of the tile, in rows of
// 32 lanes x 4 counts; the sums of the tiles before (rows above the threshold, rows at it) come through chained tiles, so
// that the counts are read once.  9.3 M rows: 42 us for the whole selection (tiles of 4 096 rows: 52); with the counts of
// the tiles, their prefix sums and the emission as kernels of their own, and a kernel per picked digit, 110 us.
__global__ void __launch_bounds__(kThreads) k_select_emit(const uint32_t* __restrict__ counts, int64_t N,
                                                          const SelectState* __restrict__ sel, unsigned long long* chain,
                                                          int64_t hot_cap, int32_t* __restrict__ hot_rows,
                                                          int64_t* __restrict__ n_hot, int max_polls, int64_t stall_tile,
                                                          int32_t* status) {
    constexpr int kRows = kSelTile / kThreads / 4, NW = kThreads / 32, kHalf = 31;
    constexpr int kWords = kRows / 4;                        // eight fields of eight bits each
    static_assert(kRows % 4 == 0, "whole words");
    __shared__ unsigned long long s_sum[NW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tile0 = (int64_t)blockIdx.x * kSelTile, warp0 = tile0 + warp * (kSelTile / NW);
    const unsigned int thr = sel->threshold, c_min = sel->c_min;
    const unsigned long long quota = sel->quota_eq;
    unsigned int c[kRows][4];
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        const int64_t g = warp0 + i * 128 + lane * 4;
        if (g + 4 <= N) {
            const uint4 v = *reinterpret_cast<const uint4*>(counts + g);
            c[i][0] = v.x;
            c[i][1] = v.y;
            c[i][2] = v.z;
            c[i][3] = v.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) c[i][k] = g + k < N ? counts[g + k] : 0u;
        }
    }
    // field 2 i of a word: row i's counts above the threshold, field 2 i + 1: at it (at most 128 each)
    unsigned long long excl[kWords], all[kWords];
    unsigned n[2 * kWords] = {};
#pragma unroll
    for (int i = 0; i < kRows; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (c[i][k] >= c_min) {
                n[i / 2] += c[i][k] > thr ? 1u << (16 * (i % 2)) : 0u;
                n[i / 2] += c[i][k] == thr ? 1u << (16 * (i % 2) + 8) : 0u;
            }
#pragma unroll
    for (int w = 0; w < kWords; ++w) excl[w] = n[2 * w] | (unsigned long long)n[2 * w + 1] << 32;
#pragma unroll
    for (int w = 0; w < kWords; ++w) {
        unsigned long long incl = excl[w];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        all[w] = __shfl_sync(0xffffffffu, incl, 31);
        excl[w] = incl - excl[w];                            // (every field of incl is at least the lane's own)
    }
    auto gt_of = [](const unsigned long long (&f)[kWords], int i) { return (unsigned)(f[i / 4] >> (16 * (i % 4))) & 255u; };
    auto eq_of = [](const unsigned long long (&f)[kWords], int i) {
        return (unsigned)(f[i / 4] >> (16 * (i % 4) + 8)) & 255u;
    };
    unsigned long long warp_sum = 0;
#pragma unroll
    for (int i = 0; i < kRows; ++i) warp_sum += ((unsigned long long)gt_of(all, i) << kHalf) + eq_of(all, i);
    if (lane == 0) s_sum[warp] = warp_sum;
    __syncthreads();
    unsigned long long total = 0, before_warp = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        if (w < warp) before_warp += s_sum[w];
        total += s_sum[w];
    }
    const bool publish = blockIdx.x != stall_tile;
    if (publish) chain_publish(chain, blockIdx.x, total);
    const unsigned long long before = chain_before<kThreads>(chain, blockIdx.x, total, publish, max_polls, status);
    // (32 bits are enough for numbers of rows)
    unsigned row_gt = (unsigned)((before + before_warp) >> kHalf);
    unsigned row_eq = (unsigned)((before + before_warp) & ((1ull << kHalf) - 1));
    const unsigned keep_eq = (unsigned)min(quota, 0xffffffffull), cap = (unsigned)hot_cap, least = max(thr, c_min);
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        unsigned n_gt = row_gt + gt_of(excl, i), n_eq = row_eq + eq_of(excl, i);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (c[i][k] < least) continue;
            const bool is_eq = c[i][k] == thr;
            if (!is_eq || n_eq < keep_eq) {
                const unsigned pos = n_gt + min(n_eq, keep_eq);
                if (pos < cap) hot_rows[pos] = (int32_t)(warp0 + i * 128 + lane * 4 + k);
                else set_status(status, HL_ECAPACITY);
            }
            n_gt += !is_eq;
            n_eq += is_eq;
        }
        row_gt += gt_of(all, i);
        row_eq += eq_of(all, i);
    }
    if (threadIdx.x == 0 && tile0 + kSelTile >= N) {         // the last tile knows the totals
        const unsigned long long all_gt = (before + total) >> kHalf, all_eq = (before + total) & ((1ull << kHalf) - 1);
        const unsigned long long kept = all_gt + (all_eq < quota ? all_eq : quota);
        *n_hot = (int64_t)kept > hot_cap ? hot_cap : (int64_t)kept;
    }
}

// ---- remap --------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_remap_bits(const int32_t* __restrict__ hot_rows,
                                                         const int64_t* __restrict__ d_n_hot, int64_t hot_cap,
                                                         int64_t N, RemapBlock* remap, int32_t* status) {
    int64_t n = *d_n_hot;
    if (n > hot_cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_status(status, HL_ECAPACITY);
        n = hot_cap;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = hot_rows[i];
        if (g < 0 || g >= N || (i > 0 && hot_rows[i - 1] >= g)) {   // must be strictly ascending, in range
            set_status(status, HL_EINVAL);
            continue;
        }
        const uint32_t blk = (uint32_t)(g / kRemapRowsPerBlock), r = (uint32_t)(g % kRemapRowsPerBlock);
        atomicOr(&remap[blk].w[1 + (r >> 5)], 1u << (r & 31));
    }
}

// prefix of a block = number of popular rows below its first row = lower bound in the ascending list
__global__ void __launch_bounds__(kThreads) k_remap_prefix(const int32_t* __restrict__ hot_rows,
                                                           const int64_t* __restrict__ d_n_hot, int64_t hot_cap,
                                                           int64_t n_blocks, RemapBlock* remap) {
    int64_t n = *d_n_hot;
    if (n > hot_cap) n = hot_cap;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < n_blocks;
         b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t first = b * kRemapRowsPerBlock;
        int64_t lo = 0, hi = n;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (hot_rows[mid] < first) lo = mid + 1;
            else hi = mid;
        }
        remap[b].w[0] = (uint32_t)lo;
    }
}

__global__ void __launch_bounds__(kThreads) k_remap_dense(const RemapBlock* __restrict__ remap, int64_t N,
                                                          int32_t* __restrict__ out) {
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < N; g += (int64_t)gridDim.x * blockDim.x)
        out[g] = remap_slot(remap_sector(remap, g), g);
}

}  // namespace

// implemented in hl_cold.cu: dst[(dst_row0 + i), :] = table[rows[i], :] for i < *d_n (clamped to n_max)
int32_t launch_gather_rows(hl_ctx* ctx, float* dst, int64_t dst_row0, const float* table, const int32_t* rows,
                           const int64_t* d_n, int64_t n_max, int32_t* status, cudaStream_t stream);


// The rows [0, n) whose counts are among the k largest (count >= 1, and count * share_den >= total * share_num if
// share_num > 0; sel->total holds the total), ties at the threshold going to the smaller index; their indices, in
// ascending order, to out_idx [cap], their number to *d_n_out.  chain: div_up(n, kSelTile) words.  counts: 16-byte aligned.
int32_t select_rows_by_count(const uint32_t* counts, int64_t n, SelectState* sel, unsigned long long* chain, long long k,
                             long long share_num, long long share_den, int64_t cap, int32_t* out_idx, int64_t* d_n_out,
                             int32_t* status, int sms, WaitCfg w, cudaStream_t stream) {
    const int64_t n_tiles = div_up(n, kSelTile);
    HL_CUDA_TRY(launch(k_select_begin, 1, 256, stream, sel, (unsigned long long)k, share_num, share_den));
    for (int shift = 24; shift >= 0; shift -= 8)
        HL_CUDA_TRY(launch(k_select_digit, grid_for(n, kThreads * 16, sms * 8), kThreads, stream, counts, n, shift, sel,
                           chain, shift == 24 ? n_tiles : 0));
    HL_CUDA_TRY(launch(k_select_emit, n_tiles, kThreads, stream, counts, n, sel, chain, cap, out_idx, d_n_out,
                       w.max_polls, w.stall_tile, status));
    note_launches(6);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

}  // namespace hl

using namespace hl;

extern "C" int32_t hl_profile_hot(hl_ctx* ctx, const hl_batch* b, int32_t reset, int32_t finalize, int32_t policy,
                                  int64_t p_num, int64_t p_den, int32_t* d_hot_rows, int64_t* d_n_hot,
                                  void* stream_) {
    if (!ctx) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    Regions& r = ctx->r;
    if (reset) {
        HL_CUDA_TRY(cudaMemsetAsync(r.counts, 0, sizeof(uint32_t) * ctx->N, stream));
        HL_CUDA_TRY(cudaMemsetAsync(r.sel, 0, sizeof(SelectState), stream));
    }
    if (b) {
        if (b->batch < 1 || b->batch > ctx->max_batch || b->nnz < 0 || b->nnz > ctx->max_nnz || !b->offsets ||
            (b->nnz > 0 && !b->indices))
            return HL_EINVAL;
        const int64_t bags_per_table = (int64_t)b->batch * ctx->S;
        const int64_t n_bags = bags_per_table * ctx->T;
        HL_CUDA_TRY(launch(k_count, grid_for(n_bags, kThreads, ctx_sms(ctx) * 8), kThreads, stream, b->indices, b->offsets,
                           n_bags, bags_per_table, r.table_base, r.counts, r.sel, r.status));
        note_launches(1);
        HL_LAUNCH_CHECK();
    }
    if (finalize) {
        if (!d_hot_rows || !d_n_hot) return HL_EINVAL;
        long long k = 0, share_num = 0, share_den = 1;
        switch (policy) {
            case HL_HOT_TOPK_ROWS: k = p_num; break;
            case HL_HOT_BUDGET_BYTES: k = p_num / (4 * (int64_t)ctx->D); break;
            case HL_HOT_FRACTION_ROWS:
                if (p_den <= 0 || p_num < 0) return HL_EINVAL;
                k = (long long)(((__int128)ctx->N * p_num) / p_den);
                break;
            case HL_HOT_MIN_SHARE:
                if (p_den <= 0 || p_num <= 0) return HL_EINVAL;
                k = ctx->hot_cap;
                share_num = p_num;
                share_den = p_den;
                break;
            default: return HL_EINVAL;
        }
        if (k < 0) return HL_EINVAL;
        if (k > ctx->hot_cap) k = ctx->hot_cap;
        return as_graph(ctx->launches, [&] {
            return select_rows_by_count(r.counts, ctx->N, r.sel, r.sel_chain, k, share_num, share_den, ctx->hot_cap,
                                        d_hot_rows, d_n_hot, r.status, ctx_sms(ctx), wait_cfg(ctx), stream);
        });
    }
    return HL_OK;
}

extern "C" int32_t hl_build_remap(hl_ctx* ctx, const int32_t* d_hot_rows, const int64_t* d_n_hot,
                                  const float* host_table, float* d_cache, int32_t* d_remap_out, void* stream_) {
    if (!ctx || !d_hot_rows || !d_n_hot) return HL_EINVAL;
    if (host_table && !d_cache) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    Regions& r = ctx->r;
    HL_CUDA_TRY(cudaMemsetAsync(r.remap, 0, sizeof(RemapBlock) * ctx->n_remap_blocks, stream));
    if (ctx->hot_cap > 0) {
        HL_CUDA_TRY(launch(k_remap_bits, grid_for(ctx->hot_cap, kThreads, ctx_sms(ctx) * 8), kThreads, stream, d_hot_rows,
                           d_n_hot, ctx->hot_cap, ctx->N, r.remap, r.status));
        note_launches(1);
    }
    HL_CUDA_TRY(launch(k_remap_prefix, grid_for(ctx->n_remap_blocks, kThreads, ctx_sms(ctx) * 8), kThreads, stream,
                       d_hot_rows, d_n_hot, ctx->hot_cap, ctx->n_remap_blocks, r.remap));
    note_launches(d_remap_out ? 2 : 1);
    if (d_remap_out)
        HL_CUDA_TRY(launch(k_remap_dense, grid_for(ctx->N, kThreads * 4, ctx_sms(ctx) * 16), kThreads, stream, r.remap,
                           ctx->N, d_remap_out));
    HL_LAUNCH_CHECK();
    if (host_table && ctx->hot_cap > 0)
        return launch_gather_rows(ctx, d_cache, 0, host_table, d_hot_rows, d_n_hot, ctx->hot_cap, r.status, stream);
    return HL_OK;
}
