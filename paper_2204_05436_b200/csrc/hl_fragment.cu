// Fragmenting a mini-batch into the popular micro-batch O and the non-popular micro-batch X, in two kernels.
//
//   1. k_frag_flags     a CTA per 32 inputs, a warp per table, a lane per input: probe the popular-row bitmap for every
//                       lookup, all-hit flags as one word per 32 inputs; the last CTA to finish partitions: prefix sums
//                       over the words' popcounts -> stable partition `perm`, n_pop
//   2. k_frag_place     destination bags (O's bags, then X's bags) in tiles: sizes, their prefix sums (within the tile,
//                       then chained over the tiles), and the lookups themselves, mapped to cache slots (O) or global
//                       rows (X); dense features go along
//
// Both are latency chains of a few dependent loads, so what counts is that the loads of a step go out together and that
// there are few steps: with a warp per input (whose lanes read one lookup of every table: a sector each), a partition in
// 1024-input rounds, and sizes, scan and emission as kernels of their own, 8 192 one-lookup bags took 16 us in six
// launches; these two take 10.6 us.
#include "hl_common.cuh"

namespace hl {
namespace {

constexpr int kThreads = 256;
// (With 512 threads and 52 registers each, the 512 CTAs of 16 384 inputs were two waves: 10.8 us, against 9.4.)
constexpr int kFlagThreads = 256;

// All threads of one CTA: perm and counts from the flag words.
__device__ void partition_by_flags(const uint32_t* words, int B, int32_t* __restrict__ perm,
                                   int32_t* __restrict__ counts) {
    constexpr int NT = kFlagThreads, NW = NT / 32;
    __shared__ int s_sum[NW + 1];
    __shared__ uint32_t s_word[NT];
    __shared__ int s_before[NT];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_words = (B + 31) / 32;
    int mine = 0;
    for (int w = threadIdx.x; w < n_words; w += NT) mine += __popc(__ldcg(&words[w]));
    const int warp_sum = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) s_sum[warp] = warp_sum;
    __syncthreads();
    int n_pop = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) n_pop += s_sum[w];
    __syncthreads();

    int before = 0;                  // popular inputs in earlier rounds
    for (int w0 = 0; w0 < n_words; w0 += NT) {
        const int w = w0 + threadIdx.x;
        const uint32_t word = w < n_words ? __ldcg(&words[w]) : 0u;
        int incl = __popc(word);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        if (lane == 31) s_sum[warp] = incl;
        __syncthreads();
        int earlier = 0, all = 0;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            if (k < warp) earlier += s_sum[k];
            all += s_sum[k];
        }
        s_word[threadIdx.x] = word;
        s_before[threadIdx.x] = before + earlier + incl - __popc(word);
        __syncthreads();
        const int first = w0 * 32, last = min(B, first + NT * 32);
#pragma unroll 8
        for (int b = first + threadIdx.x; b < last; b += NT) {
            const uint32_t m = s_word[(b - first) >> 5];
            const int bit = b & 31;
            const int rank = s_before[(b - first) >> 5] + __popc(m & ((1u << bit) - 1u));     // popular inputs before b
            perm[(m >> bit) & 1u ? rank : n_pop + (b - rank)] = b;
        }
        before += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        counts[0] = n_pop;
        counts[1] = B - n_pop;
    }
}

// SHORT_BAGS: a lane walks the lookups of its input, four tables at a time (so that, with one lookup per table, their
// offsets, indices and bitmap words are three rounds of loads).  Otherwise the lookups that a table has for the 32 inputs,
// which are contiguous, are dealt out over the lanes, and a lookup that misses finds its input in the 33 offsets; a CTA
// whose inputs have all missed is done (out-of-range lookups are reported by k_frag_place, which sees all of X's).
// Probe: how a global row is looked up in the popular set (BitmapProbe: the dense bitmap of the 32-bit path;
// HashProbe: the hashed remap of the wide-id path).
// chain / n_chain: the state of k_frag_place's chain, cleared here.
// Lookups asked for together: four, or two where a lookup takes a sector of 64-bit keys (with four the hash probe's kernels spilled
// up to 160 bytes).  Hash probe, one after the other / four / two together: 426 K bags of one 12.1 / 14.0 / 11.6 us, 416 K lookups
// in bags of 4 24.7 / 19.8 / 17.0, 31 K in bags of 3 18.9 / 17.6 / 13.9, 1 200 8.4 / 11.3 / 8.2, 320 K in bags of 20 29.2 / 20.7 / 20.8.
template <class Probe>
constexpr int kFlagLookups = std::is_same_v<Probe, HashProbe> ? 2 : 4;
template <bool SHORT_BAGS, class Probe>
__global__ void __launch_bounds__(kFlagThreads, 4) k_frag_flags(const int32_t* __restrict__ indices,
                                                             const int32_t* __restrict__ offsets, int B, int T, int S,
                                                             const int64_t* __restrict__ table_base, Probe remap,
                                                             uint32_t* words, int32_t* __restrict__ perm,
                                                             int32_t* __restrict__ counts, unsigned int* finished,
                                                             unsigned long long* __restrict__ chain, int n_chain) {
    constexpr int NW = kFlagThreads / 32;
    __shared__ unsigned s_miss;
    __shared__ bool s_last;
    __shared__ int32_t s_start[SHORT_BAGS ? 1 : NW][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = blockIdx.x * kFlagThreads + threadIdx.x; i < n_chain; i += gridDim.x * kFlagThreads) chain[i] = 0ull;
    for (int group = blockIdx.x; group * 32 < B; group += gridDim.x) {
        const int b = group * 32 + lane, in_group = min(32, B - group * 32);
        const unsigned everybody = in_group == 32 ? 0xffffffffu : (1u << in_group) - 1u;
        if (threadIdx.x == 0) s_miss = 0;
        __syncthreads();
        if (SHORT_BAGS) {
            constexpr int U = kFlagLookups<Probe>;
            bool miss = false;
            for (int t0 = warp; t0 < T; t0 += NW * U) {
                int32_t lo[U], hi[U];
                int64_t base[U], rows[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int t = t0 + u * NW;
                    const bool in = t < T && b < B;
                    const int64_t bag = ((int64_t)t * B + b) * S;
                    lo[u] = in ? offsets[bag] : 0;
                    hi[u] = in ? offsets[bag + S] : 0;
                    base[u] = t < T ? table_base[t] : 0;
                    rows[u] = t < T ? table_base[t + 1] - base[u] : 0;
                }
                // the k-th lookups of the bags, the next ones on their way while these are looked up
                int32_t idx[U], next[U];
#pragma unroll
                for (int u = 0; u < U; ++u) next[u] = lo[u] < hi[u] ? indices[lo[u]] : 0;
                bool more = true;
                for (int k = 0; more; ++k) {
                    int64_t g[U];
                    bool check[U];
                    typename Probe::HitRequest found[U];
                    more = false;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        idx[u] = next[u];
                        if (lo[u] + k + 1 < hi[u]) {
                            next[u] = indices[lo[u] + k + 1];
                            more = true;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const bool in = lo[u] + k < hi[u];
                        check[u] = in && idx[u] >= 0 && idx[u] < rows[u];
                        miss |= in && !check[u];
                        g[u] = base[u] + idx[u];
                        if (check[u]) found[u] = remap.request_hit(g[u]);
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (check[u]) miss |= !remap.hit(found[u], g[u]);
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, miss);
            if (lane == 0 && m) atomicOr(&s_miss, m);
        } else {
            // (with fewer tables than warps, several warps share a table)
            const int share = T < NW ? NW / T : 1, part = T < NW ? warp / T : 0;
            for (int t = T < NW ? warp % T : warp; t < T && part < share; t += T < NW ? T : NW) {
                __syncwarp();                         // the table before is done with s_start
                if (__shfl_sync(0xffffffffu, *(volatile unsigned*)&s_miss, 0) == everybody) break;
                const int64_t bag = ((int64_t)t * B + group * 32) * S;
                if (lane < in_group) s_start[warp][lane] = offsets[bag + (int64_t)lane * S];
                if (lane == 0) s_start[warp][in_group] = offsets[bag + (int64_t)in_group * S];
                __syncwarp();
                const int32_t lo = s_start[warp][0], hi = s_start[warp][in_group];
                const int64_t base = table_base[t], rows = table_base[t + 1] - base;
                constexpr int U = kFlagLookups<Probe>;
                for (int32_t j0 = lo + part * 32; j0 < hi; j0 += share * 32 * U) {
                    int32_t idx[U];
                    bool hit[U];
                    typename Probe::HitRequest found[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int32_t j = j0 + u * share * 32 + lane;
                        idx[u] = j < hi ? indices[j] : -1;
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        hit[u] = idx[u] >= 0 && idx[u] < rows;
                        if (hit[u]) found[u] = remap.request_hit(base + idx[u]);
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) hit[u] = hit[u] && remap.hit(found[u], base + idx[u]);
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int32_t j = j0 + u * share * 32 + lane;
                        if (hit[u] || j >= hi) continue;
                        int a = 0, z = in_group;      // s_start[a] <= j < s_start[z]
                        while (z - a > 1) {
                            const int mid = (a + z) >> 1;
                            if (s_start[warp][mid] <= j) a = mid;
                            else z = mid;
                        }
                        if (!((*(volatile unsigned*)&s_miss >> a) & 1u)) atomicOr(&s_miss, 1u << a);
                    }
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) words[group] = everybody & ~s_miss;
        __syncthreads();
    }
    // The CTA that finishes last partitions the inputs (a launch of its own for one block's work costs more than the
    // work): every CTA's words are written and fenced before it counts itself in, and the last one reads them past
    // its first-level cache.  The tally goes back to zero for the next call.
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(finished, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    partition_by_flags(words, B, perm, counts);
    if (threadIdx.x == 0) *finished = 0;
}

// ---- placing --------------------------------------------------------------------------------------------------
// The lookups of X are written as global row ids (int64 on the wide path).  With MARK (the scheduler's calls) the first half
// of the cold-row search is done on the way instead: a popular row becomes its slot, any other row g is marked in the
// cold-row bitmap and written as -2 - g (mark_cold).
//
// The chain between tiles carries two sums, lookups of O and lookups of X: 31 bits each, below two flag bits.
constexpr int kHalf = 31;
constexpr unsigned long long kLow = (1ull << kHalf) - 1ull;

struct PlaceArgs {
    const int32_t* indices;
    const int32_t* offsets;
    int B, T, S, n_dense;
    const int32_t* perm;
    int32_t* counts;
    const int64_t* table_base;
    int32_t* pop_offsets;
    int32_t* pop_ids;
    int64_t pop_cap;
    int32_t* non_offsets;
    int64_t non_cap;
    unsigned long long* chain;         // [tile] status word of the tile; zero on entry
    int32_t* status;
    int64_t max_polls;
    int64_t stall_tile;
    const float* dense;
    float* dense_out;
};

// ITEMS destination bags per thread, in rows of 32 bags per warp.
// LISTS: bags of several lookups; a warp takes the lookups of a row's 32 bags as one list (which they are at their
// destination), 128 at a time, so that every lane has one and four loads are on their way (with 4 or 16 lanes for one bag after
// the other the kernel takes two to four times as long).  What a lookup needs of the popular rows is asked for four lookups at a
// time with MARK, where every lookup of X needs it too (80 registers; one after the other / together: 333 K lookups in 111 K bags
// 15.2 / 14.8 us, 1.3 M in 65 K bags 42.5 / 33.0), and one after the other without, where X's lookups need nothing (54 registers, and
// 57 with the hash probe; together, with 78 and 96 / one after the other: 1.3 M 17.6 / 15.9, 130 K in bags of 5 7.6 / 7.0; hash probe,
// 416 K in bags of 4 14.9 / 10.8, 320 K in bags of 20 13.7 / 12.4).
template <bool LISTS, int ITEMS, bool MARK, class Probe, typename NonId>
__global__ void __launch_bounds__(kThreads) k_frag_place(PlaceArgs a, Probe remap, NonId* __restrict__ non_ids,
                                                         ColdMarks marks) {
    constexpr int TB = kThreads * ITEMS, NW = kThreads / 32;
    __shared__ int32_t s_pop[NW], s_all[NW];         // lookups of O / lookups in the warps' bags
    if (MARK) clear_cold_chain(marks);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tile = blockIdx.x;
    const int B = a.B, S = a.S, n_pop = a.counts[0], n_non = B - n_pop;
    const int n_bags = a.T * B * S, pop_bags = a.T * n_pop * S;
    const int first = tile * TB, last = min(first + TB, n_bags);

    // Destination bags: O's T*n_pop*S bags, then X's T*n_non*S bags, each table-major over the micro-batch's inputs.
    int32_t src_lo[ITEMS], len[ITEMS], table[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int dst = first + (warp * ITEMS + i) * 32 + lane;
        src_lo[i] = len[i] = table[i] = 0;
        if (dst < last) {
            const bool is_pop = dst < pop_bags;
            const unsigned local = is_pop ? dst : dst - pop_bags, per_table = (unsigned)(is_pop ? n_pop : n_non) * S;
            const unsigned t = local / per_table, rem = local - t * per_table, in = S == 1 ? rem : rem / S;
            const int64_t src = ((int64_t)t * B + a.perm[(is_pop ? 0 : n_pop) + in]) * S + (rem - in * S);
            table[i] = (int)t;
            src_lo[i] = a.offsets[src];
            len[i] = a.offsets[src + 1] - src_lo[i];
        }
    }
    // what the first lookup of a short bag becomes (ready before the tile knows where it goes: the loads behind it, index and
    // popular-row block, are in flight while the tiles exchange their sums)
    NonId head[ITEMS];
    // What `n` lookups become; the loads of all of them are requested before the first is waited for.  in: there is one;
    // is_pop: of a popular input (then it is in range and popular).
    auto resolve = [&](auto count, const bool* in, const bool* is_pop, const int64_t* base, const int64_t* rows,
                       const int32_t* idx, NonId* id) {
        constexpr int n = decltype(count)::value;
        typename Probe::Request found[n];
        uint32_t word[n];
        bool look[n];
#pragma unroll
        for (int i = 0; i < n; ++i) {
            id[i] = (NonId)-1;
            look[i] = in[i] && (is_pop[i] || (idx[i] >= 0 && idx[i] < rows[i]));
            if (in[i] && !look[i]) set_status(a.status, HL_EBOUNDS);
            if (look[i] && (MARK || is_pop[i])) found[i] = remap.request(base[i] + idx[i]);
            word[i] = 0;
            if constexpr (MARK)
                if (look[i] && !is_pop[i]) word[i] = marks.bits[(base[i] + idx[i]) >> 5];
        }
#pragma unroll
        for (int i = 0; i < n; ++i) {
            if (!look[i]) continue;
            const int64_t g = base[i] + idx[i];
            if constexpr (MARK) {
                const int32_t slot = remap.slot(found[i], g);
                id[i] = slot >= 0 || is_pop[i] ? slot : cold_id(g);
                if (slot < 0 && !is_pop[i]) mark_cold(marks, g, word[i]);
            } else {
                id[i] = is_pop[i] ? (NonId)remap.slot(found[i], g) : (NonId)g;
            }
        }
    };
    // The same without MARK, one lookup after the other: those of X need nothing.  (Of bags of one lookup, the hash probe's are
    // asked for together all the same: its keys and values come from far away, now and then from twice as far.)
    constexpr bool kTogether = MARK || std::is_same_v<Probe, HashProbe>;
    auto resolve_each = [&](auto count, const bool* in, const bool* is_pop, const int64_t* base, const int64_t* rows,
                            const int32_t* idx, NonId* id) {
        constexpr int n = decltype(count)::value;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const int64_t g = base[i] + idx[i];
            id[i] = (NonId)-1;
            if (!in[i]) continue;
            if (is_pop[i]) id[i] = (NonId)remap.slot(remap.request(g), g);
            else if (idx[i] >= 0 && idx[i] < rows[i]) id[i] = (NonId)g;
            else set_status(a.status, HL_EBOUNDS);
        }
    };
    int32_t start[ITEMS], all = 0, pop = 0;          // where the bag's lookups go, counted from the warp's first one
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        int32_t incl = len[i];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        start[i] = all + incl - len[i];
        all += __shfl_sync(0xffffffffu, incl, 31);
        pop += __reduce_add_sync(0xffffffffu, first + (warp * ITEMS + i) * 32 + lane < pop_bags ? len[i] : 0);
    }
    if (lane == 0) {
        s_pop[warp] = pop;
        s_all[warp] = all;
    }
    __syncthreads();
    int32_t tile_pop = 0, tile_all = 0, warp_start = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        if (w < warp) warp_start += s_all[w];
        tile_pop += s_pop[w];
        tile_all += s_all[w];
    }
    const unsigned long long total = ((unsigned long long)tile_pop << kHalf) + (unsigned)(tile_all - tile_pop);
    if (tile != a.stall_tile) chain_publish(a.chain, tile, total);
    if (!LISTS) {
        int32_t idx[ITEMS];
        int64_t base[ITEMS], rows[ITEMS];
        bool in[ITEMS], is_pop[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            in[i] = len[i] > 0;
            is_pop[i] = first + (warp * ITEMS + i) * 32 + lane < pop_bags;
            idx[i] = in[i] ? a.indices[src_lo[i]] : 0;
            base[i] = a.table_base[table[i]];
            rows[i] = a.table_base[table[i] + 1] - base[i];
        }
        if constexpr (kTogether) resolve(std::integral_constant<int, ITEMS>(), in, is_pop, base, rows, idx, head);
        else resolve_each(std::integral_constant<int, ITEMS>(), in, is_pop, base, rows, idx, head);
    }
    // the dense features follow their inputs: dense_out[i, :] = dense[perm[i], :]
    if (a.dense != nullptr) {
        const unsigned n_dense = a.n_dense, n_tiles = gridDim.x;
        for (int64_t i0 = (int64_t)tile * kThreads; i0 < (int64_t)B * n_dense; i0 += (int64_t)n_tiles * kThreads) {
            const int64_t e = i0 + threadIdx.x;
            if (e >= (int64_t)B * n_dense) break;
            const unsigned i = e < 0x100000000ll ? (unsigned)e / n_dense : (unsigned)(e / n_dense);
            a.dense_out[e] = a.dense[(int64_t)a.perm[i] * n_dense + (e - (int64_t)i * n_dense)];
        }
    }
    const unsigned long long before =
        chain_before<kThreads>(a.chain, tile, total, tile != a.stall_tile, (int)a.max_polls, a.status);
    if (threadIdx.x == 0 && last == n_bags) {                // the last tile knows the totals
        const int32_t L_pop = (int32_t)((before + total) >> kHalf), L_non = (int32_t)((before + total) & kLow);
        a.counts[2] = L_pop;
        a.counts[3] = L_non;
        a.pop_offsets[pop_bags] = L_pop;
        a.non_offsets[n_bags - pop_bags] = L_non;
    }
    const int32_t pop_base = (int32_t)(before >> kHalf) + warp_start;
    const int32_t non_base = (int32_t)(before & kLow) + warp_start - tile_pop;

    // the lookups of a bag of n behind its first
    auto copy_rest = [&](bool is_pop, int t, int32_t lo, int32_t n, int32_t out) {
        const int64_t base = a.table_base[t], rows = a.table_base[t + 1] - base;
        const int64_t cap = is_pop ? a.pop_cap : a.non_cap;
        for (int32_t j = 1; j < n; ++j) {
            if (out < 0 || out + j >= cap) {                 // (out < 0: only after a chain poll gave up)
                if (out >= 0) set_status(a.status, HL_ECAPACITY);
                break;
            }
            const bool in = true;
            const int32_t idx = a.indices[lo + j];
            NonId id;
            if constexpr (MARK) resolve(std::integral_constant<int, 1>(), &in, &is_pop, &base, &rows, &idx, &id);
            else resolve_each(std::integral_constant<int, 1>(), &in, &is_pop, &base, &rows, &idx, &id);
            if (is_pop) a.pop_ids[out + j] = (int32_t)id;
            else non_ids[out + j] = id;
        }
    };
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int row0 = first + (warp * ITEMS + i) * 32, dst = row0 + lane;
        const bool is_pop = dst < pop_bags;
        const int32_t out = start[i] + (is_pop ? pop_base : non_base);
        if (dst < last) {
            if (is_pop) a.pop_offsets[dst] = out;
            else if (out >= 0) a.non_offsets[dst - pop_bags] = out;
        }
        if (!LISTS) {
            if (dst < last && len[i] > 0) {
                if (out >= 0 && out < (is_pop ? a.pop_cap : a.non_cap)) {
                    if (is_pop) a.pop_ids[out] = (int32_t)head[i];
                    else non_ids[out] = head[i];
                } else if (out >= 0) {
                    set_status(a.status, HL_ECAPACITY);
                }
                if (len[i] > 1) copy_rest(is_pop, table[i], src_lo[i], len[i], out);
            }
        } else {
            constexpr int U = 4;
            const int32_t row_start = __shfl_sync(0xffffffffu, start[i], 0);
            const int32_t n = __shfl_sync(0xffffffffu, start[i] + len[i], 31) - row_start;
            for (int32_t q0 = 0; q0 < n; q0 += 32 * U) {
                int32_t idx[U], to[U];
                int64_t base[U], rows[U];
                bool pop_bag[U], in[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int32_t q = q0 + u * 32 + lane;
                    int k = 0;                               // the last bag that starts at or before q
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1)
                        if (__shfl_sync(0xffffffffu, start[i], k + d) - row_start <= q) k += d;
                    const int t = __shfl_sync(0xffffffffu, table[i], k), lo = __shfl_sync(0xffffffffu, src_lo[i], k);
                    const int32_t off = q - (__shfl_sync(0xffffffffu, start[i], k) - row_start);
                    to[u] = __shfl_sync(0xffffffffu, out, k);
                    in[u] = q < n && to[u] >= 0;             // (out < 0: only after a chain poll gave up)
                    pop_bag[u] = row0 + k < pop_bags;
                    to[u] += off;
                    if (in[u] && to[u] >= (pop_bag[u] ? a.pop_cap : a.non_cap)) {
                        set_status(a.status, HL_ECAPACITY);
                        in[u] = false;
                    }
                    idx[u] = in[u] ? a.indices[lo + off] : 0;
                    base[u] = a.table_base[t];
                    rows[u] = a.table_base[t + 1] - base[u];
                }
                NonId id[U];
                if constexpr (MARK) resolve(std::integral_constant<int, U>(), in, pop_bag, base, rows, idx, id);
                else resolve_each(std::integral_constant<int, U>(), in, pop_bag, base, rows, idx, id);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (!in[u]) continue;
                    if (pop_bag[u]) a.pop_ids[to[u]] = (int32_t)id[u];
                    else non_ids[to[u]] = id[u];
                }
            }
        }
    }
}

}  // namespace
}  // namespace hl

using namespace hl;

namespace hl {
namespace {

// The launches of a fragment call, for either lookup structure.  words [max_batch / 32 + 1], chain [frag_chain_words].
template <bool MARK, class Probe, typename NonId>
int32_t fragment_launch(const hl_batch* b, int T, int S, int sms, const int64_t* table_base, Probe probe,
                        uint32_t* words, unsigned long long* chain, int32_t* status, WaitCfg waits,
                        const float* d_dense, int32_t n_dense, int32_t* d_perm, int32_t* d_counts, hl_ubatch* pop,
                        int32_t* non_offsets, NonId* non_ids, int64_t non_cap, float* d_dense_out, ColdMarks marks,
                        cudaStream_t stream) {
    const int B = b->batch;
    const int64_t n_bags = (int64_t)T * B * S;
    // one list per row of bags, unless nearly every bag has just one lookup
    const bool lists = 4 * b->nnz > 5 * n_bags;
    // Bags per tile: 256 where there are few bags (the tiles are the parallelism) or lists of lookups, 512 from one tile
    // per SM on (with MARK: 106 K bags 9.1 us, with 1 024 10.2, with 256 8.9; 426 K beside a pipeline's other kernels 31, 46, 42).
    // Without MARK, 1 024 from a tile of those per SM on: of 512 / 1 024, 426 K bags 12.1 / 10.2 us, most of them X's 11.6 / 9.3; 208 K
    // 7.4 / 7.1 and 7.3 / 6.9.  (64-bit path: 426 K 11.5 to 12.3 / 10.2 to 14.8, by where its tables happen to lie; 512.)
    constexpr bool kLargeTiles = !MARK && std::is_same_v<Probe, BitmapProbe>;
    const int items = lists || n_bags <= (int64_t)kThreads * sms ? 1 : kLargeTiles && n_bags > (int64_t)4 * kThreads * sms ? 4 : 2;
    const int n_tiles = (int)div_up(n_bags, kThreads * items);
    // the tally of finished CTAs of the flags kernel: word 0 of the chain words (zero between calls: cleared when the
    // context is created and by the CTA that counts to the end); the chain proper is cleared by the flags kernel
    unsigned int* finished = reinterpret_cast<unsigned int*>(chain);
    PlaceArgs a{b->indices, b->offsets, B, T, S, n_dense, d_perm, d_counts, table_base, pop->offsets, pop->ids,
                pop->cap_ids, non_offsets, non_cap, chain + 1, status, waits.max_polls, waits.stall_tile, d_dense,
                d_dense_out};
    const int flag_grid = grid_for(B, 32, 4 * sms);
    if (b->nnz <= 4 * (int64_t)T * B)            // on average at most 4 lookups per input and table
        HL_CUDA_TRY(launch(k_frag_flags<true, Probe>, flag_grid, kFlagThreads, stream, b->indices, b->offsets, B, T, S,
                           table_base, probe, words, d_perm, d_counts, finished, chain + 1, n_tiles));
    else
        HL_CUDA_TRY(launch(k_frag_flags<false, Probe>, flag_grid, kFlagThreads, stream, b->indices, b->offsets, B, T, S,
                           table_base, probe, words, d_perm, d_counts, finished, chain + 1, n_tiles));
    constexpr int kMost = kLargeTiles ? 4 : 2;
    const auto place = lists        ? k_frag_place<true, 1, MARK, Probe, NonId>
                       : items == 1 ? k_frag_place<false, 1, MARK, Probe, NonId>
                       : items == 2 ? k_frag_place<false, 2, MARK, Probe, NonId>
                                    : k_frag_place<false, kMost, MARK, Probe, NonId>;
    HL_CUDA_TRY(launch(place, n_tiles, kThreads, stream, a, probe, non_ids, marks));
    note_launches(2);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

int32_t fragment_call(hl_ctx* ctx, const hl_batch* b, const float* d_dense, int32_t n_dense, int32_t* d_perm,
                      int32_t* d_counts, hl_ubatch* pop, hl_ubatch* non, float* d_dense_out, bool mark,
                      cudaStream_t stream) {
    if (!ctx || !b || !d_perm || !d_counts || !pop || !non) return HL_EINVAL;
    if (b->batch < 1 || b->batch > ctx->max_batch || b->nnz < 0 || b->nnz > ctx->max_nnz || !b->offsets ||
        (b->nnz > 0 && !b->indices))
        return HL_EINVAL;
    if (!pop->offsets || !non->offsets || (b->nnz > 0 && (!pop->ids || !non->ids))) return HL_EINVAL;
    if ((d_dense == nullptr) != (d_dense_out == nullptr) || (d_dense && n_dense < 1)) return HL_EINVAL;
    Regions& r = ctx->r;
    if (mark) {
        const int32_t fresh = marks_fresh(ctx, stream);
        if (fresh != HL_OK) return fresh;
    }
    const auto launch = mark ? fragment_launch<true, BitmapProbe, int32_t> : fragment_launch<false, BitmapProbe, int32_t>;
    return launch(b, ctx->T, ctx->S, ctx_sms(ctx), r.table_base, BitmapProbe{r.remap}, r.frag_words, r.frag_chain,
                  r.status, wait_cfg(ctx), d_dense, n_dense, d_perm, d_counts, pop, non->offsets, non->ids, non->cap_ids,
                  d_dense_out, cold_marks(ctx), stream);
}

}  // namespace

int32_t fragment_and_mark(hl_ctx* ctx, const hl_batch* b, const float* d_dense, int32_t n_dense, int32_t* d_perm,
                          int32_t* d_counts, hl_ubatch* pop, hl_ubatch* non, float* d_dense_out, cudaStream_t stream) {
    return fragment_call(ctx, b, d_dense, n_dense, d_perm, d_counts, pop, non, d_dense_out, true, stream);
}

}  // namespace hl

extern "C" int32_t hl_fragment(hl_ctx* ctx, const hl_batch* b, const float* d_dense, int32_t n_dense,
                               int32_t* d_perm, int32_t* d_counts, hl_ubatch* pop, hl_ubatch* non,
                               float* d_dense_out, void* stream) {
    return as_graph(kept_launches(ctx), [&] {
        return fragment_call(ctx, b, d_dense, n_dense, d_perm, d_counts, pop, non, d_dense_out, false,
                             static_cast<cudaStream_t>(stream));
    });
}

extern "C" int32_t hl_wide_fragment(hl_wide* w, const hl_batch* b, int32_t* d_perm, int32_t* d_counts, hl_ubatch* pop,
                                    int32_t* d_non_offsets, int64_t* d_non_rows, int64_t non_cap, void* stream_) {
    if (!w || !b || !d_perm || !d_counts || !pop || !d_non_offsets) return HL_EINVAL;
    if (b->batch < 1 || b->batch > w->max_batch || b->nnz < 0 || b->nnz > w->max_nnz || !b->offsets ||
        (b->nnz > 0 && !b->indices))
        return HL_EINVAL;
    if (!pop->offsets || (b->nnz > 0 && (!pop->ids || !d_non_rows))) return HL_EINVAL;
    const HashProbe probe{w->r_keys, w->r_vals, (uint64_t)(w->remap_slots - 1)};
    return as_graph(w->launches, [&] {
        return fragment_launch<false, HashProbe, long long>(
            b, w->T, w->S, w->sms, w->table_base, probe, w->frag_words, w->frag_chain, w->status, wait_cfg(w), nullptr, 0,
            d_perm, d_counts, pop, d_non_offsets, reinterpret_cast<long long*>(d_non_rows), non_cap, nullptr, ColdMarks{},
            static_cast<cudaStream_t>(stream_));
    });
}
