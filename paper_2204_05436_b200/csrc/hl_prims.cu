// Device-wide primitive used by several steps: stable LSD radix sort of pairs
// (few pairs: one kernel of one cluster; many: one kernel per digit, tiles chained through status words).
// It takes its element count from device memory, so that no step has to synchronise the host.
#include <cooperative_groups.h>

#include <atomic>

#include "hl_common.cuh"

namespace hl {

static std::atomic<unsigned long long> g_launches{0};
void note_launches(int n) {
    if (!launches_build_only()) g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed);
}
unsigned long long launches_so_far() { return g_launches.load(std::memory_order_relaxed); }

namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;
static_assert(kThreads * kItems == kSortTile, "tile shape");

__device__ __forceinline__ int warp_inclusive_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        int o = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += o;
    }
    return v;
}

// Exclusive scan of one value per thread over the block; `total` is the block sum (same in all threads).
// smem: at least blockDim.x / 32 + 1 ints.  Ends with a barrier, so smem can be reused right away.
__device__ __forceinline__ int block_exclusive_scan(int v, int* smem, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int incl = warp_inclusive_scan(v);
    if (lane == 31) smem[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = lane < n_warps ? smem[lane] : 0;
        int wi = warp_inclusive_scan(w);
        if (lane < n_warps) smem[lane] = wi - w;
        if (lane == 31) smem[32] = wi;
    }
    __syncthreads();
    const int res = smem[warp] + incl - v;
    total = smem[32];
    __syncthreads();
    return res;
}

__device__ __forceinline__ int64_t clamp_n(const int32_t* d_n, int64_t n_max) {
    if (d_n == nullptr) return n_max;
    int64_t n = *d_n;
    if (n < 0) n = 0;
    return n < n_max ? n : n_max;
}

// ---- single-pass chaining between tiles --------------------------------------------------------------------
// A tile is a CTA's block index, and CTAs are dispatched in that order, so a tile's predecessors are always held by blocks
// that have started.  A tile first publishes its own sum (AGGREGATE), then walks back over its predecessors adding their
// sums until it meets one that already knows its inclusive prefix (PREFIX), and finally publishes its own
// prefix.  Publishing never waits on anything, so the walk always terminates; every poll is bounded all the same,
// and a poll that runs out records HL_ETIMEOUT and carries on with what it has (positions are range-checked).
constexpr uint32_t kFlagAgg = 1u << 30, kFlagPrefix = 1u << 31, kValueMask = kFlagAgg - 1u;

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// ---- radix sort ---------------------------------------------------------------------------------------------
// Shared memory of the cluster sort: digit counters of every warp, then the pairs on their way to their new places.
template <int NT, int ITEMS>
struct SortSmem {
    uint32_t cnt[NT / 32][256];
    uint2 pair[NT * ITEMS];
};

// The valid lanes with the same 8-bit digit.  (Eight ballots: match.any does the same in one instruction but takes 60 cycles
// of the multiprocessor for random digits, the ballots 24; marking lanes in a shared-memory word per digit is no faster.)
__device__ __forceinline__ unsigned same_digit(uint32_t d, bool valid) {
    unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const unsigned bit = (d >> b) & 1u;
        peers &= __ballot_sync(0xffffffffu, bit) ^ (bit - 1u);       // those with the bit, or those without
    }
    return peers;
}

constexpr size_t sort_smem_bytes(int threads, int items) {
    return (size_t)threads / 32 * 256 * sizeof(uint32_t) + (size_t)threads * items * sizeof(uint2);
}
static_assert(sort_smem_bytes(512, 4) == sizeof(SortSmem<512, 4>), "the layout");

// Ranks a warp's items among the warp's items of the same digit (order: round, then lane) and counts them into cnt.
template <int ITEMS>
__device__ __forceinline__ void rank_in_warp(const uint32_t (&key)[ITEMS], int rounds, int n_mine, int shift,
                                             uint32_t* cnt, uint32_t (&rank)[ITEMS]) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        if (r >= rounds) break;
        const bool valid = r * 32 + lane < n_mine;
        const uint32_t d = (key[r] >> shift) & 255u;
        const unsigned peers = same_digit(d, valid);
        const uint32_t before = valid ? cnt[d] : 0u;
        __syncwarp();
        rank[r] = before + __popc(peers & lt);
        if (valid && (peers & lt) == 0) cnt[d] = before + __popc(peers);
        __syncwarp();
    }
}

// NT / 256 threads per digit (digit = thread / (NT / 256)): turns the warps' counts of a digit into prefix sums over the
// warps; returns the digit's total, the same in all threads of the digit.
template <int NT>
__device__ __forceinline__ uint32_t prefix_over_warps(uint32_t (*cnt)[256]) {
    constexpr int PD = NT / 256, PER = NT / 32 / PD;
    const int d = threadIdx.x / PD, q = threadIdx.x % PD;
    uint32_t c[PER], mine = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        c[k] = cnt[q * PER + k][d];
        mine += c[k];
    }
    uint32_t run = 0, total = 0;
#pragma unroll
    for (int k = 0; k < PD; ++k) {
        const uint32_t o = __shfl_sync(0xffffffffu, mine, k, PD);
        if (k < q) run += o;
        total += o;
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        cnt[q * PER + k][d] = run;
        run += c[k];
    }
    return total;
}

// Exclusive scan over the 256 digits of a value that the digit's PD threads share (only the first thread's counts, and
// only it gets the result).  smem: 33 ints.
template <int PD>
__device__ __forceinline__ uint32_t scan_digits(uint32_t v, int* smem) {
    int all;
    return (uint32_t)block_exclusive_scan(threadIdx.x % PD == 0 ? (int)v : 0, smem, all);
}

// Digit histograms of all passes in one sweep over the keys.
__global__ void __launch_bounds__(kThreads) k_sort_digit_hist(const int32_t* __restrict__ keys, const int32_t* d_n,
                                                              int64_t n_max, int passes,
                                                              uint32_t* __restrict__ ghist /* [passes][256] */) {
    __shared__ uint32_t h[4][256];
    for (int i = threadIdx.x; i < 4 * 256; i += kThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    const int64_t n = clamp_n(d_n, n_max);
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
        const uint32_t k = (uint32_t)keys[i];
        for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(k >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += kThreads) {
        const uint32_t c = (&h[0][0])[i];
        if (c) atomicAdd(&ghist[i], c);
    }
}

// One pass: stable scatter by one digit.  Order of the items of a tile: warp-major, then round, then lane.
// ghist: this pass's 256 digit counts; tstat[tile][256]: status words, zero on entry.  A tile is the CTA's block index: CTAs
// are dispatched in that order, so those of the tiles before have started.  With few tiles a pass is a chain of latencies:
// everything that does not depend on another load is requested first.  With many it is bound by the instructions that rank the
// items (so indices are 32 bits) and by the places that a warp writes to: ORDER checks no bounds in a full tile, puts the tile in
// order in shared memory first, while the tiles before publish their sums, and writes runs of one digit.  us a pass, before /
// without / with it: 42 K pairs 5.8 / 5.6 / 6.0, 106 K 6.8 / 6.6 / 6.9, 250 K 7.7 / 7.4 / 7.7, 426 K 10.2 / - / 9.3, 1.3 M 17.9 / - /
// 15.0, 2.6 M 31.5 / - / 26.  (Ordered tiles of 3 072 pairs, or of 4 096 in 512 threads: within 5 %.)
template <bool ORDER>
__global__ void __launch_bounds__(kThreads, ORDER ? 4 : 1) k_sort_pass(const int32_t* __restrict__ keys_in,
                                                           const int32_t* __restrict__ vals_in,
                                                           int32_t* __restrict__ keys_out, int32_t* __restrict__ vals_out,
                                                           const int32_t* d_n, int64_t n_max, int shift,
                                                           const uint32_t* __restrict__ ghist,
                                                           uint32_t* tstat, int32_t* status, int max_polls,
                                                           int64_t stall_tile) {
    constexpr int kWarps = kThreads / 32;
    __shared__ uint32_t cnt[kWarps][256];
    __shared__ uint2 ordered[ORDER ? kSortTile : 1];
    __shared__ uint32_t digit_base[256];
    __shared__ int scan_smem[40];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tile = blockIdx.x, first = tile * kSortTile;           // (fewer than 2^30 pairs)
    const int n = (int)clamp_n(d_n, n_max);
    if (first >= n) return;
    const int here = min(kSortTile, n - first);
    const bool full = here == kSortTile;
    const int mine = warp * (32 * kItems) + lane;                    // this lane's items: mine + 32 * r
    auto valid = [&](int r) { return (ORDER && full) || mine + r * 32 < here; };
    uint32_t key[kItems], val[kItems], rank[kItems];
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        key[r] = valid(r) ? (uint32_t)keys_in[first + mine + r * 32] : 0u;
        val[r] = valid(r) ? (uint32_t)vals_in[first + mine + r * 32] : 0u;
    }
    const int d = threadIdx.x;                                       // this thread's digit, between the barriers
    const int of_digit = (int)ghist[d];
    uint32_t* my_cnt = cnt[warp];
#pragma unroll
    for (int i = 0; i < 8; ++i) my_cnt[i * 32 + lane] = 0;
    __syncwarp();
    const unsigned lt = lanemask_lt();
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        const uint32_t dg = (key[r] >> shift) & 255u;
        const unsigned peers = same_digit(dg, valid(r));
        const uint32_t before = my_cnt[dg];
        __syncwarp();
        rank[r] = before + __popc(peers & lt);
        if (valid(r) && (peers & lt) == 0) my_cnt[dg] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // one thread per digit: where its items start in the tile, and in every warp's part of them
    uint32_t of_warp[kWarps], total = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        of_warp[w] = cnt[w][d];
        total += of_warp[w];
    }
    uint32_t* my = tstat + (int64_t)tile * 256 + d;
    if (tile > 0 && tile != stall_tile) st_relaxed(my, kFlagAgg | total);
    int all;
    const uint32_t start = ORDER ? (uint32_t)block_exclusive_scan((int)total, scan_smem, all) : 0u;
    uint32_t run = start;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        cnt[w][d] = run;
        run += of_warp[w];
    }
    const uint32_t gbase = (uint32_t)block_exclusive_scan(of_digit, scan_smem, all);   // keys with a smaller digit
    if (ORDER) {
#pragma unroll
        for (int r = 0; r < kItems; ++r)
            if (valid(r)) ordered[my_cnt[(key[r] >> shift) & 255u] + rank[r]] = make_uint2(key[r], val[r]);
    }
    uint32_t before = 0;                                             // items of the digit in earlier tiles
    if (tile > 0) {
        // walk back kLook tiles at a time (32 at a time was no faster and cost 16 registers): the kLook status
        // words are requested together, then consumed from the
        // nearest tile outwards until one of them already carries an inclusive prefix
        constexpr int kLook = 8;
        bool found = false, gave_up = false;
        for (int t0 = tile - 1; t0 >= 0 && !found && !gave_up; t0 -= kLook) {
            const uint32_t* p = tstat + (int64_t)t0 * 256 + d;
            uint32_t w[kLook];
#pragma unroll
            for (int k = 0; k < kLook; ++k) w[k] = t0 - k >= 0 ? ld_relaxed(p - k * 256) : kFlagPrefix;
#pragma unroll
            for (int k = 0; k < kLook; ++k) {
                if (found || gave_up) break;
                int polls = 0;
                while ((w[k] & (kFlagAgg | kFlagPrefix)) == 0) {
                    if (++polls > max_polls) {
                        set_status(status, HL_ETIMEOUT);
                        gave_up = true;
                        break;
                    }
                    __nanosleep(20);
                    w[k] = ld_relaxed(p - k * 256);
                }
                before += w[k] & kValueMask;
                found = (w[k] & kFlagPrefix) != 0;
            }
        }
    }
    if (tile != stall_tile) st_relaxed(my, kFlagPrefix | ((before + total) & kValueMask));
    digit_base[d] = gbase + before - start;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        const int i = r * kThreads + threadIdx.x;
        if (ORDER ? !(full || i < here) : !valid(r)) continue;
        const uint2 x = ORDER ? ordered[i] : make_uint2(key[r], val[r]);
        const uint32_t dg = (x.x >> shift) & 255u, pos = digit_base[dg] + (ORDER ? (uint32_t)i : my_cnt[dg] + rank[r]);
        if (pos < (uint32_t)n) {                 // always true unless a chain poll gave up
            keys_out[pos] = (int32_t)x.x;
            vals_out[pos] = (int32_t)x.y;
        }
    }
}

// The whole sort of at most CTAS * NT * ITEMS pairs in one kernel of one thread-block cluster.  The pairs stay in
// registers; every pass ranks them by one digit, adds up the digit counts of the CTAs through distributed shared memory, and
// sends each pair to the CTA that owns its new position (the last pass: to its place in the output).  CTA c owns
// positions [c * per, (c + 1) * per).  One launch instead of a memset, the digit counts and a kernel per pass, and nothing
// but the pairs themselves goes through the L2 (8 K pairs, three passes: 12.5 us, against 23 us in four kernels).
template <int CTAS, int NT, int ITEMS>
__global__ void __launch_bounds__(NT) k_sort_cluster(const int32_t* __restrict__ keys_in,
                                                               const int32_t* __restrict__ vals_in,
                                                               int32_t* __restrict__ keys_out,
                                                               int32_t* __restrict__ vals_out, const int32_t* d_n,
                                                               int64_t n_max, int passes) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int PD = NT / 256;                  // threads per digit
    extern __shared__ __align__(16) unsigned char sort_smem[];
    SortSmem<NT, ITEMS>& sm = *reinterpret_cast<SortSmem<NT, ITEMS>*>(sort_smem);
    __shared__ uint32_t cta_hist[256];            // this CTA's digit counts, read by the other CTAs
    __shared__ uint32_t digit_base[256];
    __shared__ int scan_smem[40];
    const int n = (int)clamp_n(d_n, n_max);
    if (n == 0) return;                           // the same in all CTAs
    const int cta = (int)cluster.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = max(2, (n + CTAS - 1) / CTAS);        // pairs per CTA (two at least: inv_per has 32 bits)
    const int rounds = (per + NT - 1) / NT;
    const uint32_t inv_per = (uint32_t)((0x100000000ull + per - 1) / per);       // pos / per = (pos * inv_per) >> 32
    const int here = max(0, min(n - cta * per, per));
    const int n_mine = max(0, min(here - warp * 32 * rounds, 32 * rounds));
    const int first = warp * 32 * rounds;         // of this warp, within the CTA
    uint32_t key[ITEMS], val[ITEMS], rank[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        key[r] = val[r] = 0u;
        if (r < rounds && r * 32 + lane < n_mine) {
            key[r] = (uint32_t)keys_in[cta * per + first + r * 32 + lane];
            val[r] = (uint32_t)vals_in[cta * per + first + r * 32 + lane];
        }
    }
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
#pragma unroll
        for (int i = 0; i < 8; ++i) sm.cnt[warp][i * 32 + lane] = 0;
        __syncwarp();
        rank_in_warp<ITEMS>(key, rounds, n_mine, shift, sm.cnt[warp], rank);
        __syncthreads();
        const uint32_t total = prefix_over_warps<NT>(sm.cnt);
        const int d = threadIdx.x / PD, q = threadIdx.x % PD;
        if (q == 0) cta_hist[d] = total;
        cluster.sync();     // all counts published; all CTAs have taken the previous pass's pairs out of shared memory
        uint32_t before = 0, all = 0;             // of this digit: in the CTAs before mine, in all CTAs
#pragma unroll
        for (int k = 0; k < CTAS / PD; ++k) {
            const int c = q * (CTAS / PD) + k;
            const uint32_t v = *cluster.map_shared_rank(&cta_hist[d], c);
            if (c < cta) before += v;
            all += v;
        }
#pragma unroll
        for (int o = 1; o < PD; o <<= 1) {
            before += __shfl_xor_sync(0xffffffffu, before, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        const uint32_t smaller = scan_digits<PD>(all, scan_smem);
        if (q == 0) digit_base[d] = smaller + before;
        __syncthreads();
        const bool last = p == passes - 1;
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if (r >= rounds) break;
            if (r * 32 + lane < n_mine) {
                const uint32_t dg = (key[r] >> shift) & 255u;
                const uint32_t pos = digit_base[dg] + sm.cnt[warp][dg] + rank[r];
                if (last) {
                    keys_out[pos] = (int32_t)key[r];
                    vals_out[pos] = (int32_t)val[r];
                } else {
                    const uint32_t owner = __umulhi(pos, inv_per);
                    *cluster.map_shared_rank(&sm.pair[pos - owner * per], owner) = make_uint2(key[r], val[r]);
                }
            }
        }
        cluster.sync();     // every pair has arrived (after the last pass: no CTA leaves while others read its counts)
        if (last) break;
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if (r >= rounds) break;
            if (r * 32 + lane < n_mine) {
                const uint2 x = sm.pair[first + r * 32 + lane];
                key[r] = x.x;
                val[r] = x.y;
            }
        }
    }
}

// ---- pairs that are grouped by table already ---------------------------------------------------------------------
// Where the pairs of a mini-batch are written table by table and no slot belongs to two tables, equal slots lie in one
// table's pairs, and all that the sums need is every table's pairs sorted by themselves: a cluster of CTAS CTAs per table (and
// side, if O's and X's pairs are kept apart) does all passes as k_sort_cluster does, in one kernel for all tables.  What bounds
// it is the chain count -> exchange -> scatter of a pass, with the larger tables' clusters on the chip together.  Alone, against
// three chained passes: 86 K pairs of 21 tables 8.5 / 19 us, 107 K of 26 8.6 / 19, 129 K of 3 15.5 / 21, 333 K of 37 15.7 / 24, 426 K
// of 26 18.5 / 28; 8 K of 8 tables 5.8, against 9.2 in one cluster.  (CTAs of 512 threads: 9.9, 9.9, 15.3, 21.5, 27.9, 7.6.)
// A table with more pairs than the cluster holds (the host knows the average only) is sorted by it through memory, every CTA
// taking a share of the pairs tile by tile: right, and slow (nearly all lookups in one of 20 to 26 tables, the sort alone, chained
// passes / this: 76 K pairs 21 / 100 us, 204 K 28 / 256, 1.7 M 71 / 474), so the mini-batches that come here are those that have
// as many lookups as bags (backward_sorts_tables).
template <int CTAS, int NT, int ITEMS>
__global__ void __launch_bounds__(NT)
    k_sort_segments(int32_t* keys_in, int32_t* vals_in, int32_t* keys_out, int32_t* vals_out, const int32_t* offsets_0,
                    const int32_t* d_n_samples_0, int32_t key_bias_0, const int32_t* offsets_1, const int32_t* d_n_samples_1,
                    int32_t key_bias_1, const int32_t* d_n_lookups, int32_t tables, int32_t max_batch, int32_t bags_per_sample,
                    int32_t merge, int32_t passes, int64_t max_nnz) {
    const SegmentArgs a{keys_in, vals_in, keys_out, vals_out,
                        {{offsets_0, d_n_samples_0, key_bias_0, 0}, {offsets_1, d_n_samples_1, key_bias_1, 0}},
                        d_n_lookups, tables, max_batch, bags_per_sample, merge, passes, 0, max_nnz};
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int PD = NT / 256;
    extern __shared__ __align__(16) unsigned char sort_smem[];
    SortSmem<NT, ITEMS>& sm = *reinterpret_cast<SortSmem<NT, ITEMS>*>(sort_smem);
    __shared__ uint32_t cta_hist[256];            // this CTA's digit counts, read by the other CTAs
    __shared__ uint32_t digit_base[256];
    __shared__ int scan_smem[40];
    // this cluster's pairs: [lo, lo + n)
    const int segment = blockIdx.x / CTAS, cta = (int)cluster.block_rank();
    const int which = a.merge ? 0 : segment / a.tables, table = a.merge ? segment : segment - which * a.tables;
    auto starts = [&](const int32_t* offsets, const int32_t* d_n_samples, int t) {       // table t's first lookup of a side
        const int samples = min(max(*d_n_samples, 0), a.max_batch);
        return offsets[(int64_t)t * samples * a.bags_per_sample];
    };
    const int most = (int)min((int64_t)max(a.d_n_lookups[2], 0), a.max_nnz);
    const int32_t* const offsets = which ? a.side[1].offsets : a.side[0].offsets;
    const int32_t* const d_n_samples = which ? a.side[1].d_n_samples : a.side[0].d_n_samples;
    int lo = starts(offsets, d_n_samples, table), hi = starts(offsets, d_n_samples, table + 1);
    if (a.merge) {
        lo += starts(a.side[1].offsets, a.side[1].d_n_samples, table);
        hi += starts(a.side[1].offsets, a.side[1].d_n_samples, table + 1);
    } else if (which) {
        lo += a.d_n_lookups[0];
        hi += a.d_n_lookups[0];
    }
    lo = min(max(lo, 0), most);
    const int n = max(min(hi, most) - lo, 0);
    const uint32_t bias = (uint32_t)(which ? a.side[1].key_bias : a.side[0].key_bias);
    if (n == 0) return;                           // the same in all CTAs of the cluster
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = threadIdx.x / PD, q = threadIdx.x % PD;
    // q's part of a digit's counts over the CTAs (published by a cluster.sync()) into: those of the CTAs before mine, all
    auto over_ctas = [&](uint32_t& before, uint32_t& all) {
        before = all = 0;
#pragma unroll
        for (int c = q; c < CTAS; c += PD) {
            const uint32_t v = *cluster.map_shared_rank(&cta_hist[d], c);
            if (c < cta) before += v;
            all += v;
        }
#pragma unroll
        for (int o = 1; o < PD; o <<= 1) {
            before += __shfl_xor_sync(0xffffffffu, before, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
    };
    uint32_t before, all;                         // of this thread's digit
    if (n > CTAS * NT * ITEMS) {
        int32_t *kin = a.keys_in + lo, *vin = a.vals_in + lo, *kout = a.keys_out + lo, *vout = a.vals_out + lo;
        constexpr int TILE = NT * ITEMS;
        const int share = (n + CTAS - 1) / CTAS, from = min(n, cta * share), to = min(n, from + share);     // of this CTA
        for (int p = 0; p < a.passes; ++p) {
            const int shift = 8 * p;
            if (threadIdx.x < 256) cta_hist[threadIdx.x] = 0;
            __syncthreads();
            for (int i = from + threadIdx.x; i < to; i += NT) atomicAdd(&cta_hist[((uint32_t)kin[i] - bias) >> shift & 255u], 1u);
            cluster.sync();                       // all counts published
            over_ctas(before, all);
            const uint32_t smaller = scan_digits<PD>(all, scan_smem);
            if (q == 0) digit_base[d] = smaller + before;
            for (int tile = from; tile < to; tile += TILE) {
                const int n_mine = max(0, min(to - tile - warp * 32 * ITEMS, 32 * ITEMS)), at = tile + warp * 32 * ITEMS + lane;
                uint32_t key[ITEMS], val[ITEMS], rank[ITEMS];
#pragma unroll
                for (int r = 0; r < ITEMS; ++r) {
                    key[r] = r * 32 + lane < n_mine ? (uint32_t)kin[at + r * 32] - bias : 0u;
                    val[r] = r * 32 + lane < n_mine ? (uint32_t)vin[at + r * 32] : 0u;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) sm.cnt[warp][i * 32 + lane] = 0;
                __syncwarp();
                rank_in_warp<ITEMS>(key, ITEMS, n_mine, shift, sm.cnt[warp], rank);
                __syncthreads();
                const uint32_t total = prefix_over_warps<NT>(sm.cnt);
                __syncthreads();
#pragma unroll
                for (int r = 0; r < ITEMS; ++r)
                    if (r * 32 + lane < n_mine) {
                        const uint32_t dg = (key[r] >> shift) & 255u, pos = digit_base[dg] + sm.cnt[warp][dg] + rank[r];
                        if (pos < (uint32_t)n) {     // always, unless a wait gave up when the pairs' places were worked out:
                            kout[pos] = (int32_t)(key[r] + bias);        // tables' shares may overlap then, and what is read
                            vout[pos] = (int32_t)val[r];                 // here not be what was counted
                        }
                    }
                __syncthreads();
                if (q == 0) digit_base[d] += total;
                __syncthreads();
            }
            cluster.sync();                       // all pairs written; no CTA clears its counts, or leaves, while others read them
            int32_t* const k = kin;
            int32_t* const v = vin;
            kin = kout;
            vin = vout;
            kout = k;
            vout = v;
        }
        if (a.passes % 2 == 0)                    // (the last pass wrote the input's place)
            for (int i = from + threadIdx.x; i < to; i += NT) {
                kout[i] = kin[i];
                vout[i] = vin[i];
            }
        return;
    }
    const int per = max(2, (n + CTAS - 1) / CTAS);        // pairs per CTA (two at least: inv_per has 32 bits)
    const int rounds = (per + NT - 1) / NT;
    const uint32_t inv_per = (uint32_t)((0x100000000ull + per - 1) / per);       // pos / per = (pos * inv_per) >> 32
    const int here = max(0, min(n - cta * per, per));
    const int first = warp * 32 * rounds;         // of this warp, within the CTA
    const int n_mine = max(0, min(here - first, 32 * rounds));
    uint32_t key[ITEMS], val[ITEMS], rank[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        key[r] = val[r] = 0u;
        if (r < rounds && r * 32 + lane < n_mine) {
            key[r] = (uint32_t)a.keys_in[lo + cta * per + first + r * 32 + lane] - bias;
            val[r] = (uint32_t)a.vals_in[lo + cta * per + first + r * 32 + lane];
        }
    }
    for (int p = 0; p < a.passes; ++p) {
        const int shift = 8 * p;
#pragma unroll
        for (int i = 0; i < 8; ++i) sm.cnt[warp][i * 32 + lane] = 0;
        __syncwarp();
        rank_in_warp<ITEMS>(key, rounds, n_mine, shift, sm.cnt[warp], rank);
        __syncthreads();
        const uint32_t total = prefix_over_warps<NT>(sm.cnt);
        if (q == 0) cta_hist[d] = total;
        cluster.sync();     // all counts published; all CTAs have taken the previous pass's pairs out of shared memory
        over_ctas(before, all);
        const uint32_t smaller = scan_digits<PD>(all, scan_smem);
        if (q == 0) digit_base[d] = smaller + before;
        __syncthreads();
        const bool last = p == a.passes - 1;
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if (r >= rounds) break;
            if (r * 32 + lane < n_mine) {
                const uint32_t dg = (key[r] >> shift) & 255u;
                const uint32_t pos = digit_base[dg] + sm.cnt[warp][dg] + rank[r];
                if (last) {
                    a.keys_out[lo + pos] = (int32_t)(key[r] + bias);
                    a.vals_out[lo + pos] = (int32_t)val[r];
                } else {
                    const uint32_t owner = __umulhi(pos, inv_per);
                    *cluster.map_shared_rank(&sm.pair[pos - owner * per], owner) = make_uint2(key[r], val[r]);
                }
            }
        }
        cluster.sync();     // every pair has arrived (after the last pass: no CTA leaves while others read its counts)
        if (last) break;
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if (r >= rounds) break;
            if (r * 32 + lane < n_mine) {
                const uint2 x = sm.pair[first + r * 32 + lane];
                key[r] = x.x;
                val[r] = x.y;
            }
        }
    }
}

constexpr int kClusterNT = 512, kClusterItems = 4;
constexpr int64_t kOrderTiles = 148;              // tiles of a pass from which on they are put in order first (k_sort_pass)

// CTAs of the widest cluster the current device can place: 16 (a non-portable size), 8, or 0; asked once per device.
int sort_cluster_ctas() {
    static std::atomic<int> known[64];            // 0 = not asked yet, else the answer + 1
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    const int k = known[dev].load(std::memory_order_acquire);
    if (k > 0) return k - 1;
    auto can = [](auto* kernel, int ctas, int threads, int items) {
        const size_t kBytes = sort_smem_bytes(threads, items);
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = ctas;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(ctas);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = kBytes;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
               cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBytes) == cudaSuccess &&
               cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters >= 1;
    };
    const int ctas = can(k_sort_cluster<16, kClusterNT, kClusterItems>, 16, kClusterNT, kClusterItems) &&
                             can(k_sort_segments<16, 256, 8>, 16, 256, 8) && can(k_sort_segments<16, 512, 8>, 16, 512, 8)
                         ? 16
                         : (can(k_sort_cluster<8, kClusterNT, kClusterItems>, 8, kClusterNT, kClusterItems) ? 8 : 0);
    (void)cudaGetLastError();
    known[dev].store(ctas + 1, std::memory_order_release);
    return ctas;
}

}  // namespace

// One cluster takes up to 2 048 pairs per CTA (32 768 with 16 CTAs).  Beyond that the exchange through distributed shared
// memory takes longer than the chip-wide passes: 106 K pairs in three passes 40 us, against 30 with the tiles.
// (With a tile made to stall -- the test of the bounded waits -- the chained passes are what is asked for.)
static bool sort_in_cluster(int64_t n_max, const WaitCfg& w) {
    return n_max <= (int64_t)sort_cluster_ctas() * kClusterNT * kClusterItems && w.stall_tile < 0;
}

bool sort_is_long(int64_t n_max, WaitCfg w) { return !sort_in_cluster(n_max, w); }

// For contexts of one lookup per bag at most, on average: the cluster of a table holds the pairs that an average table of the
// context can have.  (In contexts of several lookups per bag that is far more than a mini-batch's tables have: four times as many,
// 37 clusters of 16 CTAs of 512 threads for 9 K pairs each took 67 us beside a pipeline's other kernels, where the chained passes
// take 3 x 15.)
//
// There may be as many clusters as run side by side, more or less: the later ones wait for the first, and thousands of CTAs that
// find a few pairs each take longer to start than the list to sort.  Mini-batches one after the other (hl_step), us each, the sort
// alone in brackets, chained passes or one cluster / clusters per table.  Of 4 CTAs: 8 K pairs of 37 tables 62.5 (11) / 58.7 (8.4), of
// 100 65.5 (11) / 62 (10), of 128 61.0 (11) / 62.3 (15), of 300 77 (11) / 83 (25), of 1 000 108 (11) / 154 (76); 33 K of 100 76 (16) /
// 69 (11), of 200 81 (16) / 77 (18), of 300 90 (16) / 93 (25); 131 K of 200 108 (19) / 104 (22), of 300 117 (20) / 117 (29).  Of 8: 40
// tables of 16 384 184 (34) / 180 (41), 60 219 (43) / 213 (42), 80 of 8 193 180 (34) / 181 (41).  Of 16, which find few places: 6
// tables of 16 385 104 (19) / 91 (13), 12 125 (21) / 125 (27), 20 146 (27) / 153 (44), 40 184 (34) / 215 (81); pipelined, 9 of 30 000
// 64 / 71.  Of 16 with 512 threads, one to a multiprocessor: 3 of 32 769 114 (20) / 99 (14), 4 pipelined 82 / 81, 7 132 (22) / 134
// (37), 26 205 (38) / 262 (101).
static int64_t segment_pairs(int64_t n_max, int tables) { return div_up(n_max, tables); }
struct SegmentShape {
    int ctas, threads, most_ctas;      // of a cluster, of a CTA, of the launch
};
static SegmentShape segment_shape(int64_t pairs) {
    if (pairs <= 16384) return {pairs <= 8192 ? 4 : 8, 256, 960};
    return pairs <= 32768 ? SegmentShape{16, 256, 192} : SegmentShape{16, 512, 96};
}
bool sort_by_segments(int64_t n_max, int64_t n_bags, int tables, bool merge, WaitCfg w) {
    const int64_t pairs = segment_pairs(n_max, tables);
    if (n_max <= 0 || n_max > n_bags || w.stall_tile >= 0 || pairs > 65536) return false;
    const SegmentShape s = segment_shape(pairs);
    const int64_t launched = (int64_t)tables * (merge ? 1 : 2) * s.ctas;
    if (launched > s.most_ctas || (launched > 800 && sort_in_cluster(n_max, w))) return false;
    return s.ctas < 16 || sort_cluster_ctas() == 16;
}

int32_t sort_segments(const SegmentArgs& a, cudaStream_t stream) {
    const SegmentShape s = segment_shape(segment_pairs(a.max_nnz, a.tables));
    const auto kernel = s.threads == 512 ? k_sort_segments<16, 512, 8>
                        : s.ctas == 16   ? k_sort_segments<16, 256, 8>
                        : s.ctas == 8    ? k_sort_segments<8, 256, 8>
                                         : k_sort_segments<4, 256, 8>;
    HL_CUDA_TRY(launch_cluster(kernel, (int64_t)a.tables * (a.merge ? 1 : 2) * s.ctas, s.threads,
                               sort_smem_bytes(s.threads, 8), s.ctas, stream, a.keys_in, a.vals_in, a.keys_out, a.vals_out, a.side[0].offsets, a.side[0].d_n_samples,
                               a.side[0].key_bias, a.side[1].offsets, a.side[1].d_n_samples, a.side[1].key_bias, a.d_n_lookups,
                               a.tables, a.max_batch, a.bags_per_sample, a.merge, a.passes, a.max_nnz));
    note_launches(1);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

int64_t sort_clear_words(int64_t n_max, int key_bits, WaitCfg w) {
    if (n_max <= 0 || sort_in_cluster(n_max, w)) return 0;
    return 4 * 256 + (int64_t)((key_bits + 7) / 8) * div_up(n_max, kSortTile) * 256;
}

int32_t radix_sort_pairs(int32_t* keys[2], int32_t* vals[2], const int32_t* d_n, int64_t n_max, int key_bits,
                         uint32_t* hist, int32_t* status, int32_t** out_keys, int32_t** out_vals,
                         cudaStream_t stream, WaitCfg w, bool counted) {
    const int passes = n_max > 0 ? (key_bits + 7) / 8 : 0;
    if (passes > 4) return HL_EINVAL;
    const int out = passes & 1;
    *out_keys = keys[out];
    *out_vals = vals[out];
    if (n_max <= 0) return HL_OK;
    if (sort_in_cluster(n_max, w)) {
        const int ctas = sort_cluster_ctas();
        HL_CUDA_TRY(launch_cluster(ctas == 16 ? k_sort_cluster<16, kClusterNT, kClusterItems>
                                              : k_sort_cluster<8, kClusterNT, kClusterItems>,
                                   ctas, kClusterNT, sizeof(SortSmem<kClusterNT, kClusterItems>), ctas, stream, keys[0],
                                   vals[0], keys[out], vals[out], d_n, n_max, passes));
        note_launches(1);
        return HL_OK;
    }
    const int64_t n_tiles = div_up(n_max, kSortTile);
    // scratch: [4][256] digit counts, [passes][n_tiles][256] tile status words
    uint32_t* ghist = hist;
    uint32_t* tstat = hist + 4 * 256;
    if (!counted) {
        HL_CUDA_TRY(clear_words(hist, sort_clear_words(n_max, key_bits, w), stream));
        HL_CUDA_TRY(launch(k_sort_digit_hist, grid_for(n_max, kThreads * 8, 1024), kThreads, stream, keys[0], d_n, n_max,
                           passes, ghist));
        note_launches(1);
    }
    for (int p = 0; p < passes; ++p)
        HL_CUDA_TRY(launch(n_tiles > kOrderTiles ? k_sort_pass<true> : k_sort_pass<false>, (unsigned)n_tiles, kThreads,
                           stream, keys[p & 1], vals[p & 1], keys[(p & 1) ^ 1], vals[(p & 1) ^ 1], d_n, n_max, 8 * p,
                           ghist + 256 * p, tstat + (size_t)p * n_tiles * 256, status, w.max_polls, w.stall_tile));
    note_launches(passes);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

}  // namespace hl
