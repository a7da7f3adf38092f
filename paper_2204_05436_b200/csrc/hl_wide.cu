// The index-only calls of the path for models with 2^31 rows and more (the paper's SYN-M1/M2 sizes): global row ids
// are 64-bit, counted in a hashed counter and looked up in a hashed remap whose hash is the randomizer of Section
// V-C.  Every table still has fewer than 2^31 rows, so a row is the pair (table, table-local index), and the profile sorts
// its rows by those (by index, then, stable, by table).
#include <stdlib.h>

#include <new>

#include "hl_common.cuh"

namespace hl {
namespace {

constexpr int kThreads = 256;

struct Carver {
    char* base;
    size_t off = 0;
    template <typename T>
    T* take(int64_t count) {
        off = (off + 255) & ~size_t(255);
        T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
        off += (size_t)count * sizeof(T);
        return p;
    }
};

int64_t pow2_at_least(int64_t x) {
    int64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

int bits_for(int64_t max_value) {
    int b = 1;
    while ((int64_t(1) << b) <= max_value) ++b;
    return b;
}

size_t carve(char* base, hl_wide* w) {
    Carver c{base};
    const int64_t nnz = w->max_nnz > 0 ? w->max_nnz : 1;
    const int64_t E = w->counter_slots;
    const int64_t sort_n = E > nnz ? E : nnz;
    w->status = c.take<int32_t>(8);
    w->table_base = c.take<int64_t>(w->T + 1);
    w->c_keys = c.take<long long>(E);
    w->c_cnt = c.take<uint32_t>(E);
    w->sel = c.take<SelectState>(1);
    w->sel_chain = c.take<unsigned long long>(div_up(E, kSelTile) + 1);
    w->n_seen = c.take<int32_t>(4);
    w->e_tab = c.take<int32_t>(E);
    w->e_idx = c.take<int32_t>(E);
    w->e_cnt = c.take<uint32_t>(E);
    w->s_cnt = c.take<uint32_t>(E);
    w->s_ent = c.take<int32_t>(E);
    w->sel_idx = c.take<int32_t>(w->hot_cap > 0 ? w->hot_cap : 1);
    w->r_keys = c.take<long long>(w->remap_slots);
    w->r_vals = c.take<int32_t>(w->remap_slots);
    for (int i = 0; i < 2; ++i) {
        w->sort_keys[i] = c.take<int32_t>(sort_n);
        w->sort_vals[i] = c.take<int32_t>(sort_n);
    }
    // the cold-row search clears, in one go: its count, the chain words of its ranks, the scratch of its sort
    const int64_t chain_words = div_up(nnz, 1024) * 2;
    w->cold_clear = c.take<uint32_t>(8 + chain_words + sort_hist_words(sort_n));
    w->cold_n = reinterpret_cast<int32_t*>(w->cold_clear);
    w->cold_chain = reinterpret_cast<unsigned long long*>(w->cold_clear + 8);
    w->sort_hist = w->cold_clear + 8 + chain_words;
    w->frag_words = c.take<uint32_t>(w->max_batch / 32 + 1);
    w->frag_chain = c.take<unsigned long long>(frag_chain_words(w->max_bags));
    return (c.off + 255) & ~size_t(255);
}

bool fill(hl_wide* w, const hl_geometry* g, int32_t max_batch, int64_t max_nnz, int64_t hot_cap, int64_t staging_cap,
          int64_t counter_slots) {
    if (!g || g->num_tables < 1 || g->num_tables > 255 || g->bags_per_sample < 1 || !g->table_rows) return false;
    if (max_batch < 1 || max_nnz < 0 || hot_cap < 0 || staging_cap < 0 || counter_slots < 2) return false;
    int64_t n = 0;
    for (int t = 0; t < g->num_tables; ++t) {
        if (g->table_rows[t] < 1 || g->table_rows[t] >= (int64_t(1) << 31)) return false;   // table-local ids are int32
        n += g->table_rows[t];
        if (n >= (int64_t(1) << 56)) return false;
    }
    w->T = g->num_tables;
    w->S = g->bags_per_sample;
    w->N = n;
    w->max_batch = max_batch;
    w->max_nnz = max_nnz;
    w->max_bags = (int64_t)g->num_tables * max_batch * g->bags_per_sample;
    w->hot_cap = hot_cap;
    w->staging_cap = staging_cap;
    w->counter_slots = pow2_at_least(counter_slots);
    w->remap_slots = pow2_at_least(2 * (hot_cap > 2 ? hot_cap : 2));     // (HashProbe reads four entries at a time)
    if (w->max_bags >= (int64_t(1) << 30) || max_nnz >= (int64_t(1) << 30) || w->counter_slots >= (int64_t(1) << 30) ||
        hot_cap + staging_cap >= (int64_t(1) << 31) - 2)
        return false;
    return true;
}

// ---- hashed counter ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_wide_count(const int32_t* __restrict__ indices,
                                                         const int32_t* __restrict__ offsets, int64_t n_bags,
                                                         int64_t bags_per_table, const int64_t* __restrict__ table_base,
                                                         long long* keys, uint32_t* cnt, uint64_t mask,
                                                         SelectState* sel, int32_t* status) {
    unsigned long long mine = 0;
    for (int64_t bag = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; bag < n_bags;
         bag += (int64_t)gridDim.x * blockDim.x) {
        const int t = (int)(bag / bags_per_table);
        const int64_t base = table_base[t], rows = table_base[t + 1] - base;
        for (int32_t j = offsets[bag]; j < offsets[bag + 1]; ++j) {
            const int32_t idx = indices[j];
            if (idx < 0 || idx >= rows) {
                set_status(status, HL_EBOUNDS);
                continue;
            }
            const long long g = base + idx;
            uint64_t h = randomize64((uint64_t)g) & mask;
            bool placed = false;
            for (uint64_t tries = 0; tries <= mask; ++tries) {     // linear probing; the first free entry is claimed
                long long k = keys[h];
                if (k < 0) k = (long long)atomicCAS(reinterpret_cast<unsigned long long*>(&keys[h]),
                                                    (unsigned long long)-1LL, (unsigned long long)g);
                if (k < 0 || k == g) {
                    atomicAdd(&cnt[h], 1u);
                    placed = true;
                    break;
                }
                h = (h + 1) & mask;
            }
            if (!placed) set_status(status, HL_ECAPACITY);         // more distinct rows than the counter holds
            else ++mine;
        }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, d);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&sel->total, mine);
}

// every counted row as (table, index, count), in no particular order
__global__ void __launch_bounds__(kThreads) k_wide_entries(const long long* __restrict__ keys,
                                                           const uint32_t* __restrict__ cnt, int64_t slots,
                                                           const int64_t* __restrict__ table_base, int T,
                                                           int32_t* n_seen, int32_t* e_tab, int32_t* e_idx,
                                                           uint32_t* e_cnt, int32_t* sort_key, int32_t* sort_val) {
    for (int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; h < slots; h += (int64_t)gridDim.x * blockDim.x) {
        const long long g = keys[h];
        if (g < 0) continue;
        int lo = 0, hi = T;                      // table_base[lo] <= g < table_base[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (table_base[mid] <= g) lo = mid;
            else hi = mid;
        }
        const int32_t i = atomicAdd(n_seen, 1);
        e_tab[i] = lo;
        e_idx[i] = (int32_t)(g - table_base[lo]);
        e_cnt[i] = cnt[h];
        sort_key[i] = e_idx[i];
        sort_val[i] = i;
    }
}

// What a sort gives as the number of one of n entries.  (It is one, unless a wait of the sort ran out and left the place as it
// was: the status word says so, and the results are unspecified, but nothing outside the arrays may be read or written.)
__device__ __forceinline__ int32_t entry_in(int32_t e, int64_t n) { return (uint32_t)e < (uint64_t)n ? e : 0; }

// out_key[j] = table[val[j]]: the key of the second, stable sort
__global__ void __launch_bounds__(kThreads) k_wide_gather_key(const int32_t* __restrict__ val,
                                                              const int32_t* __restrict__ table, const int32_t* d_n,
                                                              int64_t n_max, int32_t* __restrict__ out_key) {
    int64_t n = *d_n;
    n = n < n_max ? n : n_max;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        out_key[j] = table[entry_in(val[j], n)];
}

// counts in row order (zero behind the last counted row), and the entry behind every position
__global__ void __launch_bounds__(kThreads) k_wide_row_order(const int32_t* __restrict__ val,
                                                             const uint32_t* __restrict__ e_cnt, const int32_t* d_n,
                                                             int64_t n_max, uint32_t* __restrict__ s_cnt,
                                                             int32_t* __restrict__ s_ent) {
    int64_t n = *d_n;
    n = n < n_max ? n : n_max;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n_max; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = j < n ? entry_in(val[j], n) : -1;
        s_cnt[j] = j < n ? e_cnt[e] : 0u;
        s_ent[j] = e;
    }
}

__global__ void __launch_bounds__(kThreads) k_wide_hot_rows(const int32_t* __restrict__ sel_idx,
                                                            const int64_t* __restrict__ d_n_hot, int64_t hot_cap,
                                                            const int32_t* __restrict__ s_ent, int64_t n_entries,
                                                            const int32_t* __restrict__ e_tab,
                                                            const int32_t* __restrict__ e_idx,
                                                            const int64_t* __restrict__ table_base,
                                                            long long* __restrict__ hot_rows) {
    int64_t n = *d_n_hot;
    n = n < hot_cap ? n : hot_cap;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = s_ent[entry_in(sel_idx[i], n_entries)];
        hot_rows[i] = e >= 0 ? table_base[e_tab[e]] + e_idx[e] : -1;
    }
}

// ---- hashed remap -----------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_wide_remap(const long long* __restrict__ hot_rows,
                                                         const int64_t* __restrict__ d_n_hot, int64_t hot_cap,
                                                         int64_t N, long long* keys, int32_t* vals, uint64_t mask,
                                                         int32_t* status) {
    int64_t n = *d_n_hot;
    if (n > hot_cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_status(status, HL_ECAPACITY);
        n = hot_cap;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const long long g = hot_rows[i];
        if (g < 0 || g >= N || (i > 0 && hot_rows[i - 1] >= g)) {   // must be strictly ascending, in range
            set_status(status, HL_EINVAL);
            continue;
        }
        uint64_t h = randomize64((uint64_t)g) & mask;
        for (uint64_t tries = 0; tries <= mask; ++tries) {
            const long long k = (long long)atomicCAS(reinterpret_cast<unsigned long long*>(&keys[h]),
                                                     (unsigned long long)-1LL, (unsigned long long)g);
            if (k < 0) {
                vals[h] = (int32_t)i;              // the slot of a popular row is its rank in the ascending list
                break;
            }
            h = (h + 1) & mask;
        }
    }
}

}  // namespace
}  // namespace hl

using namespace hl;

extern "C" size_t hl_wide_workspace_bytes(const hl_geometry* geom, int32_t max_batch, int64_t max_nnz,
                                          int64_t hot_cap_rows, int64_t staging_cap_rows, int64_t counter_slots) {
    hl_wide w{};
    if (!fill(&w, geom, max_batch, max_nnz, hot_cap_rows, staging_cap_rows, counter_slots)) return 0;
    return carve(nullptr, &w);
}

extern "C" int32_t hl_wide_create(hl_wide** out, const hl_geometry* geom, int32_t max_batch, int64_t max_nnz,
                                  int64_t hot_cap_rows, int64_t staging_cap_rows, int64_t counter_slots,
                                  void* d_workspace, size_t ws_bytes) {
    if (!out) return HL_EINVAL;
    *out = nullptr;
    if (!d_workspace || (reinterpret_cast<uintptr_t>(d_workspace) & 255)) return HL_EINVAL;
    hl_wide* w = static_cast<hl_wide*>(calloc(1, sizeof(hl_wide)));
    if (!w) return HL_EINVAL;
    if (!fill(w, geom, max_batch, max_nnz, hot_cap_rows, staging_cap_rows, counter_slots)) {
        free(w);
        return HL_EINVAL;
    }
    if (carve(static_cast<char*>(d_workspace), w) > ws_bytes) {
        free(w);
        return HL_ECAPACITY;
    }
    int dev = 0;
    w->h_table_base = static_cast<int64_t*>(malloc(sizeof(int64_t) * (w->T + 1)));
    if (!w->h_table_base || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&w->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        free(w->h_table_base);
        free(w);
        return HL_ECUDA;
    }
    w->h_table_base[0] = 0;
    for (int t = 0; t < w->T; ++t) w->h_table_base[t + 1] = w->h_table_base[t] + geom->table_rows[t];
    cudaError_t e = cudaMemcpy(w->table_base, w->h_table_base, sizeof(int64_t) * (w->T + 1), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(w->status, 0, 8 * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemset(w->c_keys, 0xff, sizeof(long long) * w->counter_slots);
    if (e == cudaSuccess) e = cudaMemset(w->c_cnt, 0, sizeof(uint32_t) * w->counter_slots);
    if (e == cudaSuccess) e = cudaMemset(w->r_keys, 0xff, sizeof(long long) * w->remap_slots);
    if (e == cudaSuccess) e = cudaMemset(w->sel, 0, sizeof(SelectState));
    if (e == cudaSuccess)
        e = cudaMemset(w->frag_chain, 0, sizeof(unsigned long long) * frag_chain_words(w->max_bags));
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        free(w->h_table_base);
        free(w);
        return HL_ECUDA;
    }
    w->launches = new (std::nothrow) LaunchCache(4);
    *out = w;
    return HL_OK;
}

extern "C" int32_t hl_wide_test_bounded_waits(hl_wide* w, int32_t poll_limit, int64_t stall_tile) {
    if (!w || poll_limit < 0) return HL_EINVAL;
    w->test_poll_limit = poll_limit;
    w->test_stall_tile = poll_limit > 0 ? stall_tile : -1;
    return HL_OK;
}

extern "C" int32_t hl_wide_destroy(hl_wide* w) {
    if (!w) return HL_EINVAL;
    delete w->launches;
    free(w->h_table_base);
    free(w);
    return HL_OK;
}

extern "C" int32_t hl_wide_status(hl_wide* w) {
    if (!w) return HL_EINVAL;
    HL_CUDA_TRY(cudaDeviceSynchronize());
    int32_t st = 0;
    HL_CUDA_TRY(cudaMemcpy(&st, w->status, sizeof(int32_t), cudaMemcpyDeviceToHost));
    if (st != 0) HL_CUDA_TRY(cudaMemset(w->status, 0, sizeof(int32_t)));
    return st;
}

namespace hl {
namespace {

// Sorts the pairs in sort_keys[0] / sort_vals[0] (n = *d_n of them; keys = table-local indices, values = entry numbers)
// by (table, index): a stable sort by index, then a stable sort by the tables gathered through the values.  Returns
// which buffer holds the result in *out_vals (the entry numbers in row order).
int32_t sort_by_row(hl_wide* w, const int32_t* table_of_entry, const int32_t* d_n, int64_t n_max, int32_t** out_vals,
                    cudaStream_t stream) {
    int32_t *k1, *v1;
    int32_t st = radix_sort_pairs(w->sort_keys, w->sort_vals, d_n, n_max, 31, w->sort_hist, w->status, &k1, &v1, stream,
                                  wait_cfg(w));
    if (st != HL_OK) return st;
    // the result sits in buffer `cur`; the second sort starts from buffer 0, so bring it there if needed
    const int cur = v1 == w->sort_vals[0] ? 0 : 1;
    if (cur == 1) {
        HL_CUDA_TRY(cudaMemcpyAsync(w->sort_vals[0], w->sort_vals[1], sizeof(int32_t) * n_max, cudaMemcpyDeviceToDevice,
                                    stream));
    }
    HL_CUDA_TRY(launch(k_wide_gather_key, grid_for(n_max, kThreads, 8 * w->sms), kThreads, stream, w->sort_vals[0],
                       table_of_entry, d_n, n_max, w->sort_keys[0]));
    note_launches(1);
    HL_LAUNCH_CHECK();
    int32_t* k2;
    return radix_sort_pairs(w->sort_keys, w->sort_vals, d_n, n_max, bits_for(w->T - 1), w->sort_hist, w->status, &k2,
                            out_vals, stream, wait_cfg(w));
}

// ---- cold rows of X -----------------------------------------------------------------------------------------------
// What bounds the search is the chain of sort passes and small kernels: a clear, this kernel, one pass per 8 bits of the
// rows, the ranks.  426 K lookups, 2.6 billion rows: fragment and search 105 us; with a sort by index, one by table, and
// heads, scan and assignment as kernels of their own, 149 us.
// X's lookups: a popular row gets its slot at once; a cold one goes on the list of pairs to sort (lower 32 bits of the
// row, position).  The list is in any order.  HIST: also the digit counts of the sort (ghist [4][256], zero on entry).
template <bool HIST>
__global__ void __launch_bounds__(kThreads) k_wide_classify(const long long* __restrict__ rows,
                                                            const int32_t* __restrict__ offsets,
                                                            const int32_t* __restrict__ d_n_non, int max_batch,
                                                            int bags_per_sample_all, int64_t cap, int64_t N,
                                                            HashProbe probe, int32_t* __restrict__ slots,
                                                            int32_t* __restrict__ sort_key, int32_t* __restrict__ sort_val,
                                                            int32_t* d_n_cold_lookups, int64_t max_nnz, uint32_t* ghist,
                                                            int passes, int32_t* status) {
    __shared__ uint32_t h[HIST ? 4 : 1][256];
    if (HIST) {
        for (int i = threadIdx.x; i < 4 * 256; i += kThreads) (&h[0][0])[i] = 0;
        __syncthreads();
    }
    int n_non = *d_n_non;
    n_non = n_non < 0 ? 0 : (n_non > max_batch ? max_batch : n_non);
    int64_t L = offsets[(int64_t)n_non * bags_per_sample_all];
    if (L > cap) L = cap;
    // A warp takes 32 * U lookups at a time, whose loads go out together, and one place in the list for all their cold ones: four a
    // lane where there are many, one where that leaves the chip idle.  One / four a lane, half of them cold and nearly all: 1 K lookups
    // 3.0 / 4.6, 3.1 / 5.0 us, 10 K 3.3 / 4.7, 3.8 / 6.6, 39 K 4.1 / 5.8, 4.9 / 7.8, 78 K 5.9 / 6.1, 7.0 / 7.8, 91 K 6.1 / 5.8, 7.6 / 7.8,
    // 112 K 7.1 / 6.1, 8.9 / 7.9, 426 K 14.8 / 10.5, 15.5 / 12.0.
    constexpr int64_t kFew = 81920;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, n_warps = (int64_t)gridDim.x * (kThreads / 32);
    const auto classify = [&](auto per_lane) {
        constexpr int U = decltype(per_lane)::value;
        for (int64_t j0 = warp * 32 * U + lane; j0 - lane < L; j0 += n_warps * 32 * U) {
            long long g[U];
            HashProbe::Request found[U];
            bool cold[U];
            unsigned m[U];
            int n_cold = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) g[u] = j0 + u * 32 < L ? rows[j0 + u * 32] : -1;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (g[u] >= N) {
                    set_status(status, HL_EBOUNDS);
                    g[u] = -1;
                }
                if (g[u] >= 0) found[u] = probe.request(g[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int32_t s = g[u] >= 0 ? probe.slot(found[u], g[u]) : -1;
                cold[u] = g[u] >= 0 && s < 0;
                if (j0 + u * 32 < L && !cold[u]) slots[j0 + u * 32] = s;
                m[u] = __ballot_sync(0xffffffffu, cold[u]);
                n_cold += __popc(m[u]);
            }
            int32_t first = 0;
            if (lane == 0 && n_cold) first = atomicAdd(d_n_cold_lookups, n_cold);
            int64_t i = __shfl_sync(0xffffffffu, first, 0);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t at = i + __popc(m[u] & ((1u << lane) - 1u));
                i += __popc(m[u]);
                if (cold[u] && at < max_nnz) {
                    const uint32_t key = (uint32_t)g[u];
                    sort_key[at] = (int32_t)key;
                    sort_val[at] = (int32_t)(j0 + u * 32);
                    if (HIST)
                        for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(key >> (8 * p)) & 255u], 1u);
                }
            }
        }
    };
    if (L > kFew) classify(std::integral_constant<int, 4>());
    else classify(std::integral_constant<int, 1>());
    if (HIST) {
        __syncthreads();
        for (int i = threadIdx.x; i < passes * 256; i += kThreads) {
            const uint32_t c = (&h[0][0])[i];
            if (c) atomicAdd(&ghist[i], c);
        }
    }
}

// the upper bits of the rows, in the order of their lower bits
__global__ void __launch_bounds__(kThreads) k_wide_upper_key(const int32_t* __restrict__ pos,
                                                             const long long* __restrict__ rows, int64_t n_rows,
                                                             const int32_t* d_n, int64_t n_max,
                                                             int32_t* __restrict__ key, int32_t* __restrict__ val) {
    int64_t n = *d_n;
    n = n < n_max ? n : n_max;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t p = entry_in(pos[j], n_rows);
        key[j] = (int32_t)(rows[p] >> 32);
        val[j] = p;
    }
}

// Ranks of the distinct rows among the sorted cold lookups, and the slot of every lookup: heads, their prefix sums
// (within the tile, then chained over the tiles) and the assignment in one kernel.  UPPER: the rows have more than 32
// bits, the sorted keys are not the rows.
constexpr int kRankItems = 4, kRankTile = kThreads * kRankItems;
template <bool UPPER>
__global__ void __launch_bounds__(kThreads) k_wide_ranks(const int32_t* __restrict__ keys, const int32_t* __restrict__ pos,
                                                         const long long* __restrict__ rows, const int32_t* d_n,
                                                         int64_t n_max, unsigned long long* chain, int64_t slot0,
                                                         int64_t staging_cap, int64_t cap_ids,
                                                         int32_t* __restrict__ slots, long long* __restrict__ cold_rows,
                                                         int64_t* __restrict__ d_n_cold, int max_polls, int64_t stall_tile,
                                                         int32_t* status) {
    __shared__ int s_warp[kThreads / 32];
    int64_t n = *d_n;
    n = n < n_max ? n : n_max;
    const int64_t tile0 = (int64_t)blockIdx.x * kRankTile;
    if (tile0 >= n) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *d_n_cold = 0;
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j0 = tile0 + threadIdx.x * kRankItems;
    auto row_at = [&](int64_t j) -> long long {
        return UPPER ? rows[entry_in(pos[j], cap_ids)] : (long long)(uint32_t)keys[j];
    };
    long long g[kRankItems];
    int32_t at[kRankItems];
    long long prev = j0 > 0 && j0 < n ? row_at(j0 - 1) : -1;
    int mine = 0;
    unsigned heads = 0;
#pragma unroll
    for (int k = 0; k < kRankItems; ++k) {
        const bool in = j0 + k < n;
        g[k] = in ? row_at(j0 + k) : -1;
        at[k] = in ? pos[j0 + k] : -1;
        if (in && g[k] != prev) {
            heads |= 1u << k;
            ++mine;
        }
        prev = g[k];
    }
    int incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        if (w < warp) before += s_warp[w];
        total += s_warp[w];
    }
    const bool publish = blockIdx.x != stall_tile;
    if (publish) chain_publish(chain, blockIdx.x, (unsigned long long)total);
    const int64_t base =
        (int64_t)chain_before<kThreads>(chain, blockIdx.x, (unsigned long long)total, publish, max_polls, status);
    int64_t rank = base + before + (incl - mine) - 1;
#pragma unroll
    for (int k = 0; k < kRankItems; ++k) {
        const bool head = heads >> k & 1u;
        rank += head;
        if (at[k] < 0 || at[k] >= cap_ids || rank < 0) continue;
        if (rank < staging_cap) {
            if (head) cold_rows[rank] = g[k];
            slots[at[k]] = (int32_t)(slot0 + rank);
        } else {
            slots[at[k]] = -1;      // no room to stage this row: the lookup is dropped, the status word says so
        }
    }
    if (threadIdx.x == 0 && tile0 + kRankTile >= n) {
        int64_t distinct = base + total;
        if (distinct > staging_cap) {
            set_status(status, HL_ECAPACITY);
            distinct = staging_cap;
        }
        *d_n_cold = distinct;
    }
}

}  // namespace
}  // namespace hl

extern "C" int32_t hl_wide_profile_hot(hl_wide* w, const hl_batch* b, int32_t reset, int32_t finalize, int32_t policy,
                                       int64_t p_num, int64_t p_den, int32_t row_bytes, int64_t* d_hot_rows,
                                       int64_t* d_n_hot, void* stream_) {
    if (!w) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const int64_t E = w->counter_slots;
    if (reset) {
        HL_CUDA_TRY(cudaMemsetAsync(w->c_keys, 0xff, sizeof(long long) * E, stream));
        HL_CUDA_TRY(cudaMemsetAsync(w->c_cnt, 0, sizeof(uint32_t) * E, stream));
        HL_CUDA_TRY(cudaMemsetAsync(w->sel, 0, sizeof(SelectState), stream));
    }
    if (b) {
        if (b->batch < 1 || b->batch > w->max_batch || b->nnz < 0 || b->nnz > w->max_nnz || !b->offsets ||
            (b->nnz > 0 && !b->indices))
            return HL_EINVAL;
        const int64_t bags_per_table = (int64_t)b->batch * w->S;
        const int64_t n_bags = bags_per_table * w->T;
        HL_CUDA_TRY(launch(k_wide_count, grid_for(n_bags, kThreads, w->sms * 8), kThreads, stream, b->indices, b->offsets,
                           n_bags, bags_per_table, w->table_base, w->c_keys, w->c_cnt, (uint64_t)(E - 1), w->sel,
                           w->status));
        note_launches(1);
        HL_LAUNCH_CHECK();
    }
    if (!finalize) return HL_OK;
    if (!d_hot_rows || !d_n_hot) return HL_EINVAL;
    long long k = 0, share_num = 0, share_den = 1;
    switch (policy) {
        case HL_HOT_TOPK_ROWS: k = p_num; break;
        case HL_HOT_BUDGET_BYTES:
            if (row_bytes < 1) return HL_EINVAL;
            k = p_num / row_bytes;
            break;
        case HL_HOT_FRACTION_ROWS:
            if (p_den <= 0 || p_num < 0) return HL_EINVAL;
            k = (long long)(((__int128)w->N * p_num) / p_den);
            break;
        case HL_HOT_MIN_SHARE:
            if (p_den <= 0 || p_num <= 0) return HL_EINVAL;
            k = w->hot_cap;
            share_num = p_num;
            share_den = p_den;
            break;
        default: return HL_EINVAL;
    }
    if (k < 0) return HL_EINVAL;
    if (k > w->hot_cap) k = w->hot_cap;
    // the counted rows in ascending order of their global id, with their counts: then the selection is the one of the
    // dense counter, over positions instead of rows (ties at the threshold go to the smaller position = smaller id)
    HL_CUDA_TRY(cudaMemsetAsync(w->n_seen, 0, 4 * sizeof(int32_t), stream));
    HL_CUDA_TRY(launch(k_wide_entries, grid_for(E, kThreads, w->sms * 8), kThreads, stream, w->c_keys, w->c_cnt, E,
                       w->table_base, w->T, w->n_seen, w->e_tab, w->e_idx, w->e_cnt, w->sort_keys[0], w->sort_vals[0]));
    note_launches(1);
    HL_LAUNCH_CHECK();
    int32_t* order;
    int32_t st = sort_by_row(w, w->e_tab, w->n_seen, E, &order, stream);
    if (st != HL_OK) return st;
    HL_CUDA_TRY(launch(k_wide_row_order, grid_for(E, kThreads, w->sms * 8), kThreads, stream, order, w->e_cnt, w->n_seen, E,
                       w->s_cnt, w->s_ent));
    note_launches(1);
    HL_LAUNCH_CHECK();
    st = select_rows_by_count(w->s_cnt, E, w->sel, w->sel_chain, k, share_num, share_den, w->hot_cap,
                              w->sel_idx, d_n_hot, w->status, w->sms, wait_cfg(w), stream);
    if (st != HL_OK) return st;
    HL_CUDA_TRY(launch(k_wide_hot_rows, grid_for(w->hot_cap, kThreads, w->sms * 8), kThreads, stream, w->sel_idx, d_n_hot,
                       w->hot_cap, w->s_ent, E, w->e_tab, w->e_idx, w->table_base,
                       reinterpret_cast<long long*>(d_hot_rows)));
    note_launches(1);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

extern "C" int32_t hl_wide_build_remap(hl_wide* w, const int64_t* d_hot_rows, const int64_t* d_n_hot, void* stream_) {
    if (!w || !d_hot_rows || !d_n_hot) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    HL_CUDA_TRY(cudaMemsetAsync(w->r_keys, 0xff, sizeof(long long) * w->remap_slots, stream));
    if (w->hot_cap > 0) {
        HL_CUDA_TRY(launch(k_wide_remap, grid_for(w->hot_cap, kThreads, w->sms * 8), kThreads, stream,
                           reinterpret_cast<const long long*>(d_hot_rows), d_n_hot, w->hot_cap, w->N, w->r_keys, w->r_vals,
                           (uint64_t)(w->remap_slots - 1), w->status));
        note_launches(1);
        HL_LAUNCH_CHECK();
    }
    return HL_OK;
}

extern "C" int32_t hl_wide_index_cold(hl_wide* w, const int32_t* d_non_offsets, const int64_t* d_non_rows,
                                      int64_t non_cap, const int32_t* d_n_non, int32_t* d_non_slots,
                                      int64_t* d_cold_rows, int64_t* d_n_cold, void* stream_) {
    if (!w || !d_non_offsets || !d_n_non || !d_cold_rows || !d_n_cold) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (w->max_nnz == 0) {
        HL_CUDA_TRY(cudaMemsetAsync(d_n_cold, 0, sizeof(int64_t), stream));
        return HL_OK;
    }
    if (!d_non_rows || !d_non_slots) return HL_EINVAL;
    LaunchBatch batch(w->launches);
    const HashProbe probe{w->r_keys, w->r_vals, (uint64_t)(w->remap_slots - 1)};
    // Rows of up to 32 bits are sorted as they are; others by their lower 32 bits, then (stable) by the rest.
    const int upper_bits = (w->N - 1) >> 32 ? bits_for((w->N - 1) >> 32) : 0;
    const int lower_bits = upper_bits ? 32 : bits_for(w->N - 1);
    const WaitCfg waits = wait_cfg(w);
    const int64_t sort_words = sort_clear_words(w->max_nnz, lower_bits, waits);
    HL_CUDA_TRY(clear_words(w->cold_clear, (int64_t)(w->sort_hist - w->cold_clear) + sort_words, stream));
    HL_CUDA_TRY(launch(sort_words ? k_wide_classify<true> : k_wide_classify<false>,
                       grid_for(w->max_nnz, kThreads, 3 * w->sms), kThreads, stream,
                       reinterpret_cast<const long long*>(d_non_rows), d_non_offsets, d_n_non, w->max_batch, w->T * w->S,
                       non_cap, w->N, probe, d_non_slots, w->sort_keys[0], w->sort_vals[0], w->cold_n, w->max_nnz,
                       w->sort_hist, (lower_bits + 7) / 8, w->status));
    note_launches(1);
    int32_t *keys, *pos;
    int32_t st = radix_sort_pairs(w->sort_keys, w->sort_vals, w->cold_n, w->max_nnz, lower_bits, w->sort_hist, w->status,
                                  &keys, &pos, stream, waits, true);
    if (st != HL_OK) return st;
    if (upper_bits) {
        const int other = pos == w->sort_vals[0] ? 1 : 0;
        int32_t* k2[2] = {w->sort_keys[other], w->sort_keys[other ^ 1]};
        int32_t* v2[2] = {w->sort_vals[other], w->sort_vals[other ^ 1]};
        HL_CUDA_TRY(launch(k_wide_upper_key, grid_for(w->max_nnz, kThreads, 8 * w->sms), kThreads, stream, pos,
                           reinterpret_cast<const long long*>(d_non_rows), non_cap, w->cold_n, w->max_nnz, k2[0], v2[0]));
        note_launches(1);
        st = radix_sort_pairs(k2, v2, w->cold_n, w->max_nnz, upper_bits, w->sort_hist, w->status, &keys, &pos, stream, waits);
        if (st != HL_OK) return st;
    }
    HL_CUDA_TRY(launch(upper_bits ? k_wide_ranks<true> : k_wide_ranks<false>, div_up(w->max_nnz, kRankTile), kThreads,
                       stream, keys, pos, reinterpret_cast<const long long*>(d_non_rows), w->cold_n, w->max_nnz,
                       w->cold_chain, w->hot_cap, w->staging_cap, non_cap, d_non_slots,
                       reinterpret_cast<long long*>(d_cold_rows), d_n_cold, waits.max_polls, waits.stall_tile, w->status));
    note_launches(1);
    return batch.end();
}
