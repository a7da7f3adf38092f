// Embedding bag over the HBM cache: sum-pooling forward, and scatter-add + SGD backward with one update per
// distinct row.  Rows are fp32 [*, D]; a group of G lanes owns one row at a time, each lane NV float4 columns,
// so that a row is read with 128-bit loads that coalesce into whole sectors.
#include <mutex>
#include <type_traits>

#include "hl_common.cuh"

namespace hl {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float4 f4_zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }

// row[0..3] += v, done by the L2 (no value comes back, so nothing waits for the row)
__device__ __forceinline__ void red_add_f4(float4* p, float4 v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// acc = (restart ? 0 : acc) + r.  A restart clears the upper word only: what is left of acc is below 2^-1041, which an
// fp32 value absorbs when it is added (and if that value is a zero, rounds to zero with the sum), and it costs one
// select per column where clearing both words, which the compiler turns into predicated moves, costs two.
__device__ __forceinline__ double unless(bool restart, double acc) {
    return __hiloint2double(restart ? 0 : __double2hiint(acc), __double2loint(acc));
}
__device__ __forceinline__ void add_row(double (&acc)[4], float4 r, bool restart = false) {
    acc[0] = unless(restart, acc[0]) + (double)r.x;
    acc[1] = unless(restart, acc[1]) + (double)r.y;
    acc[2] = unless(restart, acc[2]) + (double)r.z;
    acc[3] = unless(restart, acc[3]) + (double)r.w;
}

__device__ __forceinline__ int clamp_samples(const int32_t* d_n_samples, int max_batch) {
    int n = *d_n_samples;
    if (n < 0) n = 0;
    return n < max_batch ? n : max_batch;
}

// ---- forward ------------------------------------------------------------------------------------------------
// FORWARD (both kernels): the launch also copies the staged rows that this mini-batch shares with the one before
// (ForwardRows), which no bag of this launch reads.
struct ForwardRows {
    float* cache;
    int64_t from_row0, to_row0;        // cache[to_row0 + i, :] = cache[from_row0 + src[i], :] where src[i] >= 0
    const int32_t* src;
    const int64_t* d_n;
    int64_t n_max;
};

__device__ __forceinline__ void forward_rows(const ForwardRows& fr, int D4) {
    int64_t n = *fr.d_n;
    n = n < 0 ? 0 : (n < fr.n_max ? n : fr.n_max);
    const int lane = threadIdx.x & 31;
    float4* c4 = reinterpret_cast<float4*>(fr.cache);
    for (int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - lane; i0 < n;
         i0 += (int64_t)gridDim.x * blockDim.x) {
        const int32_t mine = i0 + lane < n ? fr.src[i0 + lane] : -1;
        for (unsigned m = __ballot_sync(0xffffffffu, mine >= 0 && mine < fr.n_max); m; m &= m - 1) {
            const int k = __ffs((int)m) - 1;
            const int64_t from = fr.from_row0 + __shfl_sync(0xffffffffu, mine, k);
            for (int c = lane; c < D4; c += 32) c4[(fr.to_row0 + i0 + k) * D4 + c] = c4[from * D4 + c];
        }
    }
}

// ---- bags of one lookup, as a rule (contexts of at most 1.5 lookups per bag)
// A bag of several lookups, finished by one group of G lanes: rows are added in lookup order in fp64, four loads
// in flight, and the sum is rounded once (so cancellation between the rows of a bag costs no accuracy).
template <int G, int NV>
__device__ __forceinline__ void pool_long_bag(const float4* __restrict__ rows, const int32_t* __restrict__ ids,
                                           int32_t lo, int32_t len, int sub, int D4, int64_t n_slots,
                                           float4* __restrict__ dst, int32_t* status) {
    double acc[NV][4];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v][0] = acc[v][1] = acc[v][2] = acc[v][3] = 0.0;
    for (int32_t p = 0; p < len; p += 4) {
        int32_t id[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) id[k] = p + k < len ? __ldg(&ids[lo + p + k]) : -1;
        float4 r[4][NV];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool ok = id[k] >= 0 && id[k] < n_slots;
            if (id[k] >= n_slots) set_status(status, HL_EBOUNDS);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int c = sub + v * G;
                r[k][v] = (ok && c < D4) ? __ldg(&rows[(int64_t)id[k] * D4 + c]) : f4_zero();
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                acc[v][0] += (double)r[k][v].x;
                acc[v][1] += (double)r[k][v].y;
                acc[v][2] += (double)r[k][v].z;
                acc[v][3] += (double)r[k][v].w;
            }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const int c = sub + v * G;
        if (c < D4)
            __stcs(&dst[c], make_float4((float)acc[v][0], (float)acc[v][1], (float)acc[v][2], (float)acc[v][3]));
    }
}

// A group of G lanes takes UB consecutive bags per trip.  Bags of at most one lookup (the one-hot case) are plain
// row copies: the UB rows are loaded at once (UB independent 128-bit loads per lane), and the offsets and ids of
// the NEXT trip are requested before those rows are consumed, so that the offsets -> id -> row chain of one trip
// hides behind the rows of another.  Longer bags go through pool_long_bag one after the other.
template <int G, int NV, int UB, bool FORWARD>
__global__ void __launch_bounds__(kThreads, NV == 1 ? 4 : 1) k_embbag_fwd(const float* __restrict__ cache,
                                                         const int32_t* __restrict__ ids,
                                                         const int32_t* __restrict__ offsets,
                                                         const int32_t* __restrict__ d_n_samples, int max_batch,
                                                         int bags_per_sample_all /* T*S */, int D4, int64_t n_slots,
                                                         float* __restrict__ out, int32_t* status, ForwardRows fr) {
    if (FORWARD) forward_rows(fr, D4);
    const int64_t n_bags = (int64_t)clamp_samples(d_n_samples, max_batch) * bags_per_sample_all;
    const int sub = threadIdx.x % G;
    const float4* __restrict__ rows = reinterpret_cast<const float4*>(cache);
    float4* __restrict__ out4 = reinterpret_cast<float4*>(out);

    // lo/len of the UB bags of a trip, and the id of every bag that has exactly one lookup (-1 otherwise)
    auto load_index = [&](int64_t bag0, int32_t (&lo)[UB], int32_t (&len)[UB], int32_t (&id1)[UB]) {
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int64_t bag = bag0 + u;
            const bool valid = bag < n_bags;
            lo[u] = valid ? __ldg(&offsets[bag]) : 0;
            len[u] = valid ? __ldg(&offsets[bag + 1]) - lo[u] : -1;
        }
#pragma unroll
        for (int u = 0; u < UB; ++u) id1[u] = len[u] == 1 ? __ldg(&ids[lo[u]]) : -1;
    };

    // This CTA's share: the bags are dealt out in trips of (groups per CTA) x UB consecutive bags, every CTA gets a
    // contiguous run of trips, and the counts differ by at most one trip -- the grid is a fixed number of CTAs per
    // multiprocessor, whatever the number of bags.
    constexpr int kGroups = kThreads / G;
    int32_t lo[UB], len[UB], id1[UB];
    const int64_t trip_bags = (int64_t)kGroups * UB;
    const int64_t trips_all = (n_bags + trip_bags - 1) / trip_bags;
    const int64_t q = trips_all / gridDim.x, rem = trips_all % gridDim.x;
    const int64_t my_first = (int64_t)blockIdx.x * q + min((int64_t)blockIdx.x, rem);
    const int64_t my_trips = q + ((int64_t)blockIdx.x < rem ? 1 : 0);
    const int64_t tile0 = my_first * trip_bags;
    const int64_t tile_end = min(n_bags, tile0 + my_trips * trip_bags);
    int64_t bag0 = tile0 + (int64_t)(threadIdx.x / G) * UB;
    if (bag0 < tile_end) load_index(bag0, lo, len, id1);
    for (; bag0 < tile_end; bag0 += kGroups * UB) {
        float4 row[UB][NV];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const bool ok = id1[u] >= 0 && id1[u] < n_slots;
            if (id1[u] >= n_slots) set_status(status, HL_EBOUNDS);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int c = sub + v * G;
                row[u][v] = (ok && c < D4) ? __ldg(&rows[(int64_t)id1[u] * D4 + c]) : f4_zero();
            }
        }
        int32_t cur_len[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) cur_len[u] = len[u];
        const int64_t next0 = bag0 + kGroups * UB;
        if (next0 < tile_end) load_index(next0, lo, len, id1);   // in flight while this trip's rows arrive
        unsigned long_bags = 0;   // bit u: bag u of this trip has more than one lookup
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            if (cur_len[u] < 0) continue;   // past the last bag
            if (cur_len[u] > 1) {
                long_bags |= 1u << u;
                continue;
            }
            float4* dst = out4 + (bag0 + u) * D4;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int c = sub + v * G;
                if (c < D4) __stcs(&dst[c], row[u][v]);
            }
        }
        while (long_bags) {   // one copy of the pooling loop, whichever bag of the trip it serves
            const int u = __ffs(long_bags) - 1;
            long_bags &= long_bags - 1;
            const int64_t bag = bag0 + u;
            const int32_t b_lo = __ldg(&offsets[bag]), b_len = __ldg(&offsets[bag + 1]) - b_lo;
            pool_long_bag<G, NV>(rows, ids, b_lo, b_len, sub, D4, n_slots, out4 + bag * D4, status);
        }
    }
}

// ---- bags of several lookups
__device__ __forceinline__ void copy_16_async(uint32_t smem_to, const void* from, bool valid) {      // (else: zeros)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(smem_to), "l"(from), "r"(valid ? 16 : 0) : "memory");
}

// By columns per lane: lookups of a block, blocks of the ring, threads of a CTA, CTAs that fit a multiprocessor (registers).  Rows
// of 260 to 512 fp32: three CTAs of 80 registers spill 72 bytes; two, with a block more on its way instead, do not.  Rows of
// 2 KB, alone, L2 flushed, three CTAs / two / two and three blocks: 655 K lookups in bags of 20 268 / 147 / 137 us, 197 K in bags of
// 3 98 / 65 / 60, 82 K in bags of 20 47.8 / 30.0 / 27.4, 10 K 18.5 / 14.9 / 12.9; of 1 040 bytes 241 / 141 / 131, 84.5 / 57.8 / 54.5,
// 43.4 / 28.2 / 25.4, 18.2 / 15.3 / 12.8.  (CTAs of 128 threads, four or five of them: 3 to 20 % slower in the large calls.)
template <int NV>
struct FwdShape {
    static constexpr int U = NV >= 4 ? 1 : 4 / NV, kBlocks = NV == 4 ? 3 : 2;
    static constexpr int NT = NV >= 8 ? 128 : 256;
    static constexpr int CTAS = NV == 4 ? 2 : NV >= 8 ? 3 : 4;
    static constexpr size_t kSmem = sizeof(float4) * kBlocks * U * NV * NT;
    static_assert(kSmem <= 48 * 1024, "more than that has to be asked for");
};

// A group of G lanes pools a run of consecutive bags; the runs of all groups of the launch are equally long.  The lookups of
// a run are one list, which the group walks in blocks of U: while a block is summed, the rows of the next one are on their way
// into shared memory and the ids of the one after that into registers, whatever bags they belong to.  (A lane copies and reads
// the same 16 bytes of every row, so nothing but its own copies is waited for.)  Rows are added in lookup order in fp64 and the
// sum is rounded once, so that cancellation between the rows of a bag costs no accuracy; the row of a bag of one lookup is copied
// as it is where rows have up to 64 fp32 (the sign of a zero and the bits of a NaN with it), and added to zero in wider ones.  A
// lookup that is skipped (negative id) or outside the cache adds zeros.
//
// What bounds it is how many rows are on their way, and how often a bag makes them stop: with a loop over the lookups of one
// bag after the other (loads into registers, four at a time) 2.1 M lookups of 256-byte rows in bags of 5 took 114.7 us, 655 K of
// 64 bytes in bags of 10 28.7, 80 K of 128 bytes in bags of 4 17.5, 200 K of 144 bytes in bags of 3 23.4; so 84.8, 18.4, 10.5 and
// 18.5 (alone, L2 flushed, Zipf).  2.6 M lookups of 512 bytes in bags of 20: 149.5 -> 142.1 (9.4 TB/s).  Bags of one lookup, against
// a kernel made for them: 426 K of 256 bytes 36.9 -> 35.5, 106 K of 512 bytes 21.8 -> 22.4, 33 K of 1 KB 18.4 -> 15.7.  Blocks of 8 or
// 3 rows, and rings of three blocks: within 4 % or slower; five CTAs per multiprocessor: 2 % faster for bags of one lookup
// of 256 bytes, 10 % slower for 64-byte rows and 22 % for 1 KB.
template <int G, int NV, bool FORWARD>
__global__ void __launch_bounds__(FwdShape<NV>::NT, FwdShape<NV>::CTAS) k_embbag_pool(const float* __restrict__ cache,
                                                         const int32_t* __restrict__ ids,
                                                         const int32_t* __restrict__ offsets,
                                                         const int32_t* __restrict__ d_n_samples, int max_batch,
                                                         int bags_per_sample_all /* T*S */, int D4, int64_t n_slots,
                                                         float* __restrict__ out, int32_t* status, ForwardRows fr) {
    constexpr int U = FwdShape<NV>::U, NB = FwdShape<NV>::kBlocks, NT = FwdShape<NV>::NT;
    static_assert(U <= G, "a lane holds one id of a block");
    constexpr unsigned kAll = 0xffffffffu;
    extern __shared__ float4 ring[];                    // [NB][U][NV][NT]
    const int lane = threadIdx.x & 31, sub = lane % G;
    if (FORWARD) forward_rows(fr, D4);
    // this group's bags: [first, first + n_bags)  (numbers of bags and lookups are below 2^30)
    const int all_bags = clamp_samples(d_n_samples, max_batch) * bags_per_sample_all;
    const int groups = gridDim.x * (NT / G), me = (blockIdx.x * NT + threadIdx.x) / G;
    const int q = all_bags / groups, rem = all_bags - q * groups;
    const int first = me * q + min(me, rem), n_bags = q + (me < rem ? 1 : 0);
    const unsigned gmask = G == 32 ? kAll : ((1u << (G & 31)) - 1u) << (lane - sub);
    const uint32_t n_rows = (uint32_t)(n_slots < 0x7fffffff ? n_slots : 0x7fffffff), row_bytes = (uint32_t)D4 * 16u;
    const char* const column = reinterpret_cast<const char*>(cache) + sub * 16;
    const uint32_t ring0 = (uint32_t)__cvta_generic_to_shared(ring) + threadIdx.x * 16;

    const int32_t* __restrict__ ends = offsets + first + 1;              // where the group's bags end
    int32_t p = n_bags > 0 ? __ldg(ends - 1) : 0;
    const int32_t hi = n_bags > 0 ? __ldg(ends + n_bags - 1) : 0;
    auto ends_at = [&](int k) { return k + sub < n_bags ? __ldg(ends + k + sub) : 0x7fffffff; };
    auto ids_at = [&](int32_t at) { return sub < U && at + sub < hi ? __ldg(&ids[at + sub]) : -1; };
    auto request = [&](int b, int32_t mine) {           // the rows of a block, whose ids the first U lanes hold
        const bool ok = (uint32_t)mine < n_rows;
        if (!ok && mine >= 0) set_status(status, HL_EBOUNDS);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t id = __shfl_sync(kAll, ok ? (uint32_t)mine : 0xffffffffu, u, G);
            const bool valid = id != 0xffffffffu;
            const char* row = column + (uint64_t)(valid ? id : 0u) * row_bytes;
#pragma unroll
            for (int v = 0; v < NV; ++v)
                if (sub + v * G < D4)
                    copy_16_async(ring0 + ((b * U + u) * NV + v) * (NT * 16), row + v * G * 16, valid);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int32_t my_end = ends_at(0), next_ends = ends_at(G);
    int32_t next_ids = ids_at(p);
#pragma unroll
    for (int b = 0; b < NB - 1; ++b) {
        const int32_t mine = next_ids;
        next_ids = ids_at(p + (b + 1) * U);
        request(b, mine);
    }
    double acc[NV][4] = {};
    int k = 0;                                          // the bag being summed, and where it ends
    int32_t end = __shfl_sync(kAll, my_end, 0, G);
    bool copied = G < 32 && end - p == 1;               // its one row is copied, bit for bit, and not summed
    float4* to = reinterpret_cast<float4*>(out) + (int64_t)first * D4 + sub;
    auto next_bag = [&]() {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            if (sub + v * G < D4 && !copied)
                __stcs(to + v * G, make_float4((float)acc[v][0], (float)acc[v][1], (float)acc[v][2], (float)acc[v][3]));
            acc[v][0] = acc[v][1] = acc[v][2] = acc[v][3] = 0.0;
        }
        to += D4;
        ++k;
        if ((k & (G - 1)) == 0) {
            my_end = next_ends;
            next_ends = ends_at(k + G);
        }
        const int32_t begin = end;
        end = __shfl_sync(gmask, my_end, k & (G - 1), G);          // (behind the last bag: 2^31 - 1)
        copied = G < 32 && end - begin == 1;
    };
    for (int b = 0; __any_sync(kAll, p < hi); p += U, b = b == NB - 1 ? 0 : b + 1) {
        const int32_t mine = next_ids;
        next_ids = ids_at(p + NB * U);
        request(b == 0 ? NB - 1 : b - 1, mine);
        asm volatile("cp.async.wait_group %0;" ::"n"(NB - 1) : "memory");
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float4 r[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v)
                r[v] = sub + v * G < D4 ? ring[((b * U + u) * NV + v) * NT + threadIdx.x] : f4_zero();
            if (p + u < hi) {
                while (end <= p + u) next_bag();
                if (copied) {
                    if (sub < D4) __stcs(to, r[0]);
                } else {
#pragma unroll
                    for (int v = 0; v < NV; ++v) add_row(acc[v], r[v]);
                }
            }
        }
    }
    while (k < n_bags) next_bag();
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// ---- backward -----------------------------------------------------------------------------------------------
// One micro-batch's lookups as (slot, bag) pairs: keys are slot + key_bias, a skipped lookup (negative id) gets the
// sentinel slot n_slots, which sorts behind all others and is ignored.
struct PairSide {
    int32_t* ids;
    const int32_t* offsets;
    const int32_t* d_n_samples;
    int32_t key_bias, unused;          // (no padding in launch arguments)
};

struct PairArgs {
    PairSide side[2];                  // the second one's pairs follow the first one's
    int sides;
    int bags_follow;                   // the second side's bags are numbered behind the first one's
    int by_table;                      // the pairs lie table by table: of every table the first side's, then the second's
    int bags_per_sample;               // ... and table
    int max_batch, bags_per_sample_all;
    int64_t n_slots, max_nnz;
    int32_t* keys;
    int32_t* vals;
    int32_t* d_n_lookups;              // [0], [1]: lookups of the sides; [2]: their sum (two sides only)
    int32_t* status;
    // ASSIGN: the second side's ids of -2 - g are cold rows, ranked by now: they become slots here (and in its ids)
    const uint2* ranked;
    int64_t slot0, stage_rows;
    // ... and the cold rows are looked up in the previous mini-batch's (ascending; nullptr: there is none)
    const int32_t* cold_rows;
    const int64_t* d_n_cold;
    const int32_t* prev_rows;
    const int64_t* d_n_prev;
    int64_t n_prev_max;
    int32_t* fwd_src;
    // HIST: digit counts of the sort that follows, [passes][256], zero on entry
    uint32_t* ghist;
    int passes, unused;
};

template <int GROUP, bool ASSIGN, bool HIST>
__global__ void __launch_bounds__(kThreads) k_bwd_pairs(PairArgs a) {
    __shared__ uint32_t h[HIST ? 4 : 1][256];
    if (HIST) {
        for (int i = threadIdx.x; i < 4 * 256; i += kThreads) (&h[0][0])[i] = 0;
        __syncthreads();
    }
    const int64_t bags0 = (int64_t)clamp_samples(a.side[0].d_n_samples, a.max_batch) * a.bags_per_sample_all;
    const int64_t bags1 =
        a.sides > 1 ? (int64_t)clamp_samples(a.side[1].d_n_samples, a.max_batch) * a.bags_per_sample_all : 0;
    const int64_t L0 = a.side[0].offsets[bags0];
    const int64_t thread = (int64_t)blockIdx.x * kThreads + threadIdx.x, n_threads = (int64_t)gridDim.x * kThreads;
    if (thread == 0) {
        int64_t L1 = a.sides > 1 ? a.side[1].offsets[bags1] : 0, first = L0;
        if (L0 + L1 > a.max_nnz) {
            set_status(a.status, HL_ECAPACITY);
            if (first > a.max_nnz) first = a.max_nnz;
            if (L1 > a.max_nnz - first) L1 = a.max_nnz - first;
        }
        a.d_n_lookups[0] = (int32_t)first;
        if (a.sides > 1) {
            a.d_n_lookups[1] = (int32_t)L1;
            a.d_n_lookups[2] = (int32_t)(first + L1);
        }
    }
    for (int64_t all = thread / GROUP; all < bags0 + bags1; all += n_threads / GROUP) {
        const bool second = all >= bags0;
        const PairSide& s = a.side[second ? 1 : 0];
        const int64_t bag = second ? all - bags0 : all;
        int64_t pos0 = second ? L0 : 0;
        if (ASSIGN && a.by_table) {
            const int tables = a.bags_per_sample_all / a.bags_per_sample;
            const unsigned per_table = (unsigned)(second ? bags1 : bags0) / tables, t = (unsigned)bag / per_table;
            pos0 = second ? a.side[0].offsets[(int64_t)(t + 1) * (bags0 / tables)] : a.side[1].offsets[(int64_t)t * (bags1 / tables)];
        }
        const int32_t bag_value = (int32_t)(a.bags_follow ? all : bag);
        const int32_t lo = s.offsets[bag], hi = s.offsets[bag + 1];
        for (int32_t j = lo + (int)(thread % GROUP); j < hi; j += GROUP) {
            if (pos0 + j >= a.max_nnz) break;
            int32_t id = s.ids[j];
            if (ASSIGN && id <= -2 && second) {
                id = cold_slot(a.ranked, id, a.slot0, a.stage_rows);
                s.ids[j] = id;
            }
            if (id >= a.n_slots) set_status(a.status, HL_EBOUNDS);
            const int32_t key = ((id < 0 || id >= a.n_slots) ? (int32_t)a.n_slots : id) + s.key_bias;
            a.keys[pos0 + j] = key;
            a.vals[pos0 + j] = bag_value;
            if (HIST)
                for (int p = 0; p < a.passes; ++p) atomicAdd(&h[p][((uint32_t)key >> (8 * p)) & 255u], 1u);
        }
    }
    if (ASSIGN && a.prev_rows != nullptr) {
        int64_t n = *a.d_n_cold, np = *a.d_n_prev;
        n = n < 0 ? 0 : (n < a.stage_rows ? n : a.stage_rows);
        np = np < 0 ? 0 : (np < a.n_prev_max ? np : a.n_prev_max);
        for (int64_t i = thread; i < n; i += n_threads) a.fwd_src[i] = position_in(a.prev_rows, np, a.cold_rows[i]);
    }
    if (HIST) {
        __syncthreads();
        for (int i = threadIdx.x; i < a.passes * 256; i += kThreads) {
            const uint32_t c = (&h[0][0])[i];
            if (c) atomicAdd(&a.ghist[i], c);
        }
    }
}

// The sorted lookups are cut into chunks of 32, and these into windows of 8.  A CTA takes a window, a WARP a chunk: it sums, in
// order, the gradient rows of each run of equal slots inside its chunk.  A run that lies wholly inside the chunk is finished
// there (one reduction into its row).  Of a run that goes on over several chunks of the window, the later chunks' warps leave
// their sums in shared memory and the warp of the chunk it starts in adds them up.  A run that crosses a window's border
// leaves a partial sum: part[window][0] for the piece that continues a run from the previous window, part[window][1] for the
// piece that starts a run continuing into the next window.  k_bwd_spans adds those up.
//
// Every lane loads one (slot, bag) pair and the 32 / G groups of the warp take G consecutive lookups each, so that the
// gradient rows of a chunk are requested by all groups at once: a chunk of narrow rows (64 bytes: G = 4) is a chain of
// four dependent steps, not of 32, which is what bounds a call of few lookups (4-row groups: 7.6 K lookups 18.4 -> 4.6
// us, 86 K lookups 21.1 -> 6.3 us).  Where runs begin and end is settled by two ballots (a mask of run heads and one of
// run tails).  Runs that lie inside a group's lookups are finished by the group; a run over several groups is put
// together by a segmented scan of the groups' sums, in fixed order.  Everything that checks a pair (position inside
// the call, bag inside the gradient array) is done by the lane that loaded it, once.  Rows that fill the warp (G = 32)
// are bound by the float -> double conversions, the additions and the row updates in DRAM together (2.6 M lookups of
// 512 bytes: 183 -> 173 us; chunks of 64 / 128 / 256 lookups 177 / 190 / 197 us: the row updates of the warps at work
// then lie further apart).
//
// A run that starts in one window and ends in the next one's first chunk is finished by the warp of the chunk it starts in,
// which reads on into that chunk; the warp there leaves the run's lookups alone.  Both decide from the sorted slots alone and by
// the same test -- the run's head lies in the first of the two windows, and what lies behind the second one's first chunk does not
// begin with the run's slot -- so exactly one of them sums each lookup.  Only runs with more than 32 lookups in the next
// window go through partial sums and k_bwd_spans.
// (Without the windows, every run over three or more chunks went through them, a popular row's hundreds of pieces among them.
// Sums and spans, alone, L2 flushed, Zipf, by chunks / by windows: 426 K lookups of 256 bytes 53.2 / 47.1 us, 312 K 43.1 / 40.8, 333 K
// of 144 bytes 36.0 / 32.3, 129 K of 64 bytes 18.4 / 16.4, 2.6 M of 512 bytes 206.8 / 192.9, 262 K of 1 KB 70.1 / 59.3, 131 K of 2 KB
// 101.2 / 88.1; uniform slots the same.  Of the 2.6 M the sums take 173 instead of 166, the spans 14 instead of 32.)
constexpr int kWindowChunks = kThreads / 32, kBwdWindow = kWindowChunks * kBwdChunk;
constexpr int kSpanLookahead = 32;      // windows k_bwd_chunks looks ahead for the end of a run
static_assert(kBwdChunk == 32, "one lookup of a chunk per lane");

// Shared memory for the pieces of a window's runs, in fp64 whatever the width of a row, so that what a run adds up to inside a window
// is rounded nowhere: two sets, for windows in turn, where they fit (rows of up to 256 fp32), else one; rows of more than 512
// fp32 need more than the 48 KB that a kernel has without asking (piece_memory_granted).
template <int G, int NV>
struct PieceShape {
    static constexpr int kSets = NV <= 2 ? 2 : 1;
    static constexpr int kCount = kSets * kWindowChunks * NV * 2 * G;               // double2
    static constexpr bool kDynamic = NV >= 8;
    static constexpr size_t kDynamicBytes = kDynamic ? kCount * sizeof(double2) : 0;
};

//
// CTAS: CTAs that fit a multiprocessor.  Rows of 36 to 64 fp32 (G = 16): a warp waits for its pairs, then for gradient rows,
// and then puts two groups together, once per 32 lookups, so in a call of many chunks another warp should have something on
// its way meanwhile: four CTAs of 64 registers with four rows a lane in flight, instead of three of 80 (and a spill) with
// eight.  Rows of 256 bytes, alone, L2 flushed, three against four CTAs: Zipf over 26 tables 32 K lookups 11.5 / 13.0 us,
// 106 K 14.1 / 15.1, 150 K 19.1 / 16.6, 426 K 35.7 / 33.9; uniform 9.6 / 10.0, 13.8 / 13.6, 19.0 / 16.6, 48.4 / 46.5; bags of
// 20 lookups 8.4 / 8.8, 11.6 / 10.9, 15.7 / 12.8, 28.6 / 25.2.  So three as long as their warps have a chunk each at most.
// Rows of 68 to 128 fp32 (G = 32, one column per lane): four CTAs with four rows a lane in flight, instead of three with eight,
// where most gradient rows come out of the L2, that is where bags have many lookups.  Rows of 512 bytes, sums and spans, three
// against four CTAs: bags of 20 lookups, 2.6 M 193 / 184 us, 1.3 M 104.7 / 102.7; of 10, 1.6 M 125.6 / 119.6; of 5, 0.8 M 82.4 /
// 79.9; of 3, 0.6 M 69.6 / 75.8; of 2, 0.4 M 55.8 / 58.6; of 1, 0.3 M 57.4 / 64.5.  (The host knows how many a bag has at most.)

template <int G, int NV, int CTAS>
__global__ void __launch_bounds__(kThreads, CTAS) k_bwd_chunks(float* __restrict__ cache,
                                                         const int32_t* __restrict__ keys,
                                                         const int32_t* __restrict__ vals,
                                                         const int32_t* __restrict__ d_n_lookups,
                                                         const float* __restrict__ grad_out, int D4, int64_t n_slots,
                                                         float lr, float* __restrict__ part,
                                                         const int32_t* __restrict__ d_first, int32_t key_bias,
                                                         int32_t* __restrict__ span_count,
                                                         int32_t* __restrict__ span_list, int64_t n_grad_rows,
                                                         int64_t max_entries, int32_t* status) {
    // the lookups of this call are positions [first, first + *d_n_lookups) of the sorted arrays; their keys are
    // slot + key_bias.  A chunk in which a run starts that goes on into the next chunk is appended to span_list
    // (in any order): k_bwd_spans finishes those runs.
    static_assert(NV == 1 || G == 32, "several columns per lane only when a row fills the warp");
    constexpr int NG = 32 / G;                                              // groups per warp
    constexpr int U = NV >= 4 ? 2 : (NV >= 2 || G == 4 || CTAS > 3 ? 4 : 8);        // lookups in flight per lane
    static_assert(G % U == 0, "batch must divide the group");
    // (positions are below 2^30: 32-bit arithmetic)
    const int first = d_first ? d_first[0] : 0;
    const int count = d_n_lookups[0], n = first + count;
    const int n_chunks = (count + kBwdChunk - 1) / kBwdChunk;
    const int lane = threadIdx.x & 31, sub = lane % G, g0 = lane - sub;     // g0: first lane (= lookup) of my group
    constexpr unsigned gbits = G == 32 ? 0xffffffffu : ((1u << G) - 1u);
    const unsigned gmask = gbits << g0;
    const unsigned before_group = (1u << g0) - 1u;                          // lookups of the groups before mine
    const int wib = threadIdx.x >> 5;
    float4* __restrict__ part4 = reinterpret_cast<float4*>(part);
    // slots and bags are 32-bit numbers, so one unsigned comparison tells whether one lies inside its array
    const uint32_t n_rows_u = (uint32_t)(n_slots < 0x7fffffff ? n_slots : 0x7fffffff);
    const uint32_t n_grad_u = (uint32_t)(n_grad_rows < 0x7fffffff ? n_grad_rows : 0x7fffffff);
    // this lane's columns; a lane beyond the row's width reads column 0 and writes nothing
    // (row addresses: one wide multiply-add of the 32-bit row number and the row's bytes)
    bool on[NV];
    const char* gcol[NV];
    const uint32_t row_bytes = (uint32_t)D4 * 16u;
    __shared__ double2 s_first[G == 32 ? 1 : 2][G == 32 ? 1 : kThreads];      // sums of the groups' first runs
    // Of every chunk of the window that begins inside a run: what the run has there, and whether it ends there.
    using Shape = PieceShape<G, NV>;
    constexpr bool kTwo = Shape::kSets == 2;
    __shared__ double2 s_piece_static[Shape::kDynamic ? 1 : Shape::kCount];
    extern __shared__ double2 s_piece_dynamic[];
    double2* const s_piece = Shape::kDynamic ? s_piece_dynamic : s_piece_static;    // [set][chunk][NV][2][G]
    __shared__ int s_ends[Shape::kSets][kWindowChunks];
    const auto piece_at = [&](int set, int chunk, int v) {
        return s_piece + ((set * kWindowChunks + chunk) * NV + v) * 2 * G + sub;
    };
    const float minus_lr = -lr;               // -(lr * G) and (-lr) * G are the same number
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const int c = sub + v * G;
        on[v] = c < D4;
        gcol[v] = reinterpret_cast<const char*>(grad_out) + (on[v] ? c : 0) * 16;
    }
    char* cache_col = reinterpret_cast<char*>(cache) + sub * 16;
    auto grad_row = [&](int v, int32_t b) {
        return __ldg(reinterpret_cast<const float4*>(gcol[v] + (uint64_t)(uint32_t)b * row_bytes));
    };

    for (int window = blockIdx.x, turn = 0; window * kWindowChunks < n_chunks; window += gridDim.x, ++turn) {
        const int set = kTwo ? turn & 1 : 0;
        const int start = first + (window * kWindowChunks + wib) * kBwdChunk;          // (may lie behind the last lookup)
        const int window_end = first + (window + 1) * kBwdWindow;
        const int32_t key = start + lane < n ? keys[start + lane] : -1;       // -1: past the end; no slot has this key
        int32_t bag = start + lane < n ? vals[start + lane] : 0;
        const int32_t prev_key = start > first && start <= n ? keys[start - 1] : -3;      // -3: equal to no key
        const int32_t next_key = start + kBwdChunk < n ? keys[start + kBwdChunk] : -2;
        // the slot before the previous window, and the first slot behind the next window's first chunk
        const int32_t prev2_key = wib == 0 && window >= 2 ? keys[start - kBwdWindow - 1] : -3;
        const int32_t next2_key = window_end + kBwdChunk < n ? keys[window_end + kBwdChunk] : -2;
        // the next window's first pairs, for a run that ends there (narrow rows: asked for now, not when the sums are done)
        int32_t k2 = -1, b2 = 0;
        const auto load_next = [&]() {
            if (window_end + lane < n) {
                k2 = keys[window_end + lane];
                b2 = vals[window_end + lane];
            }
        };
        if (G < 32) load_next();
        // (a bag id outside the gradient array can only be what a given-up chain poll of the sort left behind; such a
        // call has its error status set, and reads bag 0 instead)
        bag = (uint32_t)bag < n_grad_u ? bag : 0;

        // a segment's sum is kept in fp64: a popular row can collect tens of thousands of gradient rows, and the
        // rounding of many fp32 partial sums would show in the updated row.
        double acc[NV][4];            // of the group's run that is not over yet
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v][0] = acc[v][1] = acc[v][2] = acc[v][3] = 0.0;

        // a run is complete in acc: one reduction into its row
        auto apply = [&](uint32_t row, const double (&acc)[NV][4]) {
            float4* to = reinterpret_cast<float4*>(cache_col + (uint64_t)row * row_bytes);
#pragma unroll
            for (int v = 0; v < NV; ++v)
                if (on[v])
                    red_add_f4(to + v * G,
                               make_float4(minus_lr * (float)acc[v][0], minus_lr * (float)acc[v][1],
                                           minus_lr * (float)acc[v][2], minus_lr * (float)acc[v][3]));
        };
        // a piece of a run that crosses the window's border (which: 0 = it comes in from the left, 1 = it starts here)
        auto store_piece = [&](int which, const double (&acc)[NV][4]) {
#pragma unroll
            for (int v = 0; v < NV; ++v)
                if (on[v])
                    part4[(int64_t)(window * 2 + which) * D4 + sub + v * G] =
                        make_float4((float)acc[v][0], (float)acc[v][1], (float)acc[v][2], (float)acc[v][3]);
        };
        // the same for a run that this chunk began inside: kept for the warp of the chunk it starts in
        auto put_piece = [&](const double (&acc)[NV][4]) {
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                double2* to = piece_at(set, wib, v);
                to[0] = make_double2(acc[v][0], acc[v][1]);
                to[G] = make_double2(acc[v][2], acc[v][3]);
            }
        };
        // adds the pieces of a run in the chunks from `chunk` on; true: it ends in this window
        auto add_pieces = [&](double (&sum)[NV][4], int chunk) {
            for (; chunk < kWindowChunks; ++chunk) {
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const double2* from = piece_at(set, chunk, v);
                    const double2 p = from[0], q = from[G];
                    sum[v][0] += p.x;
                    sum[v][1] += p.y;
                    sum[v][2] += q.x;
                    sum[v][3] += q.y;
                }
                if (s_ends[set][chunk]) return true;
            }
            return false;
        };

        int32_t l = __shfl_up_sync(0xffffffffu, key, 1), r = __shfl_down_sync(0xffffffffu, key, 1);
        if (lane == 0) l = prev_key;
        if (lane == 31) r = next_key;
        // bit q of `heads`: lookup q of the chunk begins a run; of `tails`: it ends one
        const unsigned heads = __ballot_sync(0xffffffffu, key != l), tails = __ballot_sync(0xffffffffu, key != r);
        // A run that comes in from the previous window, began there and ends in this one's first chunk was finished there:
        // its lookups count for nothing here, and a row that is loaded anyway stands in for theirs.
        const bool skip = wib == 0 && window >= 1 && !(heads & 1u) && tails != 0u && prev2_key != prev_key;
        if (skip) {
            const int32_t other = __shfl_sync(0xffffffffu, bag, 31);
            if (key == prev_key) bag = other;
        }
        // Tails that end a run of a row inside the cache, begun in this chunk: one reduction each.  (A row outside is a
        // skipped lookup's sentinel, or past the end.)  The first tail of a chunk that begins inside a run leaves a
        // piece instead, or nothing if the window before has seen to it.
        const uint32_t row = (uint32_t)(key - key_bias);
        const unsigned valid = __ballot_sync(0xffffffffu, row < n_rows_u);
        unsigned piece = (heads & 1u) ? 0u : tails & (0u - tails);
        const unsigned done = tails & valid & ~piece;
        piece = skip ? 0u : piece & valid;

        if constexpr (G == 32) {
            unsigned hs = heads, ds = done, es = done | piece;
            // (kept rolled: with all 32 lookups unrolled the kernel is tens of KB of straight-line code that every
            // warp runs through about once, and it waits for instructions)
#pragma unroll 1
            for (int j = 0; j < 32; j += U) {
                float4 x[U][NV];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int32_t b = __shfl_sync(0xffffffffu, bag, j + u);
#pragma unroll
                    for (int v = 0; v < NV; ++v) x[u][v] = grad_row(v, b);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) add_row(acc[v], x[u][v], hs & (1u << u));
                    if (es & (1u << u)) {
                        if (ds & (1u << u)) apply(__shfl_sync(0xffffffffu, row, j + u), acc);
                        else put_piece(acc);
                    }
                }
                hs >>= U;
                ds >>= U;
                es >>= U;
            }
        } else {
            const unsigned h = (heads >> g0) & gbits, t = (tails >> g0) & gbits;
            // my first tail, if it ends a run that began further left: finished below
            const unsigned late = (h & 1u) ? 0u : t & (0u - t);
            const unsigned d = (done >> g0) & gbits & ~late;
            const unsigned ends = d | late;
#pragma unroll
            for (int j = 0; j < G; j += U) {
                float4 x[U];
#pragma unroll
                for (int u = 0; u < U; ++u) x[u] = grad_row(0, __shfl_sync(0xffffffffu, bag, j + u, G));
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    add_row(acc[0], x[u], h & (1u << (j + u)));
                    if (ends & (1u << (j + u))) {
                        if (late & (1u << (j + u))) {      // (kept in shared memory: registers would cost eight moves a step)
                            s_first[0][threadIdx.x] = make_double2(acc[0][0], acc[0][1]);
                            s_first[1][threadIdx.x] = make_double2(acc[0][2], acc[0][3]);
                        } else {
                            apply(__shfl_sync(gmask, row, j + u, G), acc);
                        }
                    }
                }
            }
            // What the run open at the right edge of every group has collected: an inclusive scan of the groups'
            // trailing sums that restarts at groups with a head.
            const unsigned upto = heads & (before_group | gmask);
            const int from = upto ? (31 - __clz((int)upto)) / G : 0, gi = g0 / G;
            double in[1][4];          // what the run has collected in the groups before mine
#pragma unroll
            for (int s = 1; s < NG; s <<= 1) {
                const bool add = gi - s >= from;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    in[0][e] = __shfl_up_sync(0xffffffffu, acc[0][e], s * G);
                    if (add) acc[0][e] += in[0][e];
                }
            }
            if (NG > 2) {             // (of two groups, the scan's one step brought the first one's sum)
#pragma unroll
                for (int e = 0; e < 4; ++e) in[0][e] = __shfl_up_sync(0xffffffffu, acc[0][e], G);
            }
            const uint32_t row0 = __shfl_sync(0xffffffffu, row, 0, G);
            if (late) {
                const double2 p = s_first[0][threadIdx.x], q = s_first[1][threadIdx.x];
                const bool from_left = gi > 0;
                in[0][0] = p.x + (from_left ? in[0][0] : 0.0);
                in[0][1] = p.y + (from_left ? in[0][1] : 0.0);
                in[0][2] = q.x + (from_left ? in[0][2] : 0.0);
                in[0][3] = q.y + (from_left ? in[0][3] : 0.0);
                if (late & (done >> g0)) apply(row0, in);
                else if (late & (piece >> g0)) put_piece(in);
            }
        }
        // The chunk's last lookup does not end its run: the run goes on in the next chunk (only a full chunk has a next
        // one), and the last group's acc holds what it has collected here.
        const bool last_group = lane >= 32 - G;
        const int32_t last_key = __shfl_sync(0xffffffffu, key, 31);
        const bool goes_on = !(tails >> 31) && (uint32_t)(last_key - key_bias) < n_rows_u;
        if (goes_on && !heads && last_group) put_piece(acc);
        if (lane == 0) s_ends[set][wib] = tails != 0u;
        __syncthreads();
        if (wib == 0 && !(heads & 1u) && !skip && (valid & 1u)) {       // what this window has of a run begun in one before
            double sum[NV][4] = {};
            add_pieces(sum, 0);
            if (lane < G) store_piece(0, sum);
        }
        if (goes_on && heads) {
            // The run began in this chunk: the next ones' pieces, if it ends among them, complete it.
            if (add_pieces(acc, wib + 1)) {
                if (last_group) apply((uint32_t)(last_key - key_bias), acc);
            } else if (next2_key != last_key) {
                // it ends in the next window's first chunk: its lookups there are summed here as well (they are a prefix of
                // that chunk: m of them), and the row gets its one update
                double more[NV][4] = {};
                if (G == 32) load_next();
                b2 = (uint32_t)b2 < n_grad_u ? b2 : 0;
                const int m = __popc(__ballot_sync(0xffffffffu, k2 == last_key));
                const int mine = m - g0;             // lookups of my group that belong to the run
#pragma unroll 1
                for (int j = 0; j < (G == 32 ? m : G); j += U) {
                    float4 x[U][NV];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int32_t b = __shfl_sync(0xffffffffu, b2, j + u, G);
#pragma unroll
                        for (int v = 0; v < NV; ++v) x[u][v] = j + u < mine ? grad_row(v, b) : f4_zero();
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
#pragma unroll
                        for (int v = 0; v < NV; ++v) add_row(more[v], x[u][v]);
                }
#pragma unroll
                for (int v = 0; v < NV; ++v)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
#pragma unroll
                        for (int off = G; off < 32; off <<= 1)
                            more[v][e] += __shfl_xor_sync(0xffffffffu, more[v][e], off);
                        more[v][e] += acc[v][e];
                    }
                if (last_group) apply((uint32_t)(last_key - key_bias), more);
            } else {
                if (last_group) store_piece(1, acc);
                // List it, with its last window if that is among the next 32 (window w > window holds a piece of the run iff
                // its first slot is the run's; equal slots lie together: those windows form a prefix).  Nearly every run ends
                // there, and k_bwd_spans then has nothing to search; the longer ones go to the list's other end.
                const int64_t at = window_end + (int64_t)lane * kBwdWindow;
                const bool there = at < n && keys[at] == last_key;
                const int cnt = __popc(__ballot_sync(0xffffffffu, there));
                if (lane == 0) {
                    const bool is_long = cnt == kSpanLookahead;
                    const int32_t i = atomicAdd(&span_count[is_long ? 1 : 0], 1);
                    // (one entry per window at most, and the counts are zero when a call starts: the list cannot overflow
                    // unless an earlier call was cut short between its two kernels)
                    if (i >= 0 && i < max_entries)
                        reinterpret_cast<int4*>(span_list)[is_long ? max_entries - 1 - i : i] =
                            make_int4(window, last_key, is_long ? -1 : window + cnt, 0);
                    else
                        set_status(status, HL_ECAPACITY);
                }
            }
        }
        if (!kTwo) __syncthreads();                 // (the one set of pieces is free for the next window's)
    }
}

// Finishes the listed runs: those that start in a window and have more than 32 lookups in the next.  Two lists share one array.
//
// From its front: runs whose last window is known (up to kSpanLookahead windows on).  One WARP per run: the 32/G groups add
// the run's continuation pieces in an interleaved, fixed order in fp64, the group sums are combined by shuffles in a
// fixed order, and group 0 applies the single SGD update of the row.
// From its back: longer runs (a popular row can own hundreds of windows).  One CTA per run: its warps close in on the end with a
// 32-way search over the sorted keys, every group takes every (8 * 32/G)-th piece, and one group combines the group sums in
// a fixed order.
//
// A run is a chain of round trips to the L2 (entry, pieces, reduction), so what helps is to have the pieces of the next trip on
// their way: two CTAs per multiprocessor (the grid is no more than that) leave the compiler 120 registers for it.
template <int G, int NV>
__global__ void __launch_bounds__(kThreads, 2) k_bwd_spans(float* __restrict__ cache, const int32_t* __restrict__ keys,
                                                        const int32_t* __restrict__ d_n_lookups, int D4,
                                                        int64_t n_slots, float lr, const float* __restrict__ part,
                                                        const int32_t* __restrict__ d_first, int32_t key_bias,
                                                        int32_t* span_count,
                                                        const int32_t* __restrict__ span_list, int64_t max_entries) {
    constexpr int GW = 32 / G;   // groups per warp
    constexpr int kWarps = kThreads / 32;
    constexpr int U = NV >= 4 ? 2 : (NV >= 2 ? 4 : 8);   // pieces in flight per lane
    __shared__ double s_sum[kThreads][4];
    const int64_t first = d_first ? d_first[0] : 0;
    const int64_t n = first + d_n_lookups[0];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int sub = lane % G, gi = lane / G;
    const float4* __restrict__ part4 = reinterpret_cast<const float4*>(part);
    const int4* __restrict__ list = reinterpret_cast<const int4*>(span_list);
    float4* cache4 = reinterpret_cast<float4*>(cache);
    const int64_t n_windows = (n - first + kBwdWindow - 1) / kBwdWindow;
    const int64_t most = n_windows < max_entries ? n_windows : max_entries;
    auto clamped = [&](int32_t c) { return c < 0 ? (int64_t)0 : ((int64_t)c < most ? (int64_t)c : most); };
    const int64_t n_short = clamped(span_count[0]), n_long = clamped(span_count[1]);

    // sum over pieces from + step * {first, first + groups, ...} <= last of this lane's columns
    auto add_pieces = [&](double (&acc)[NV][4], int64_t from, int64_t last, int64_t groups) {
        for (int64_t c2 = from; c2 <= last; c2 += groups * U) {
            float4 t[U][NV];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const int c = sub + v * G;
                    const int64_t cc = c2 + u * groups;
                    t[u][v] = (cc <= last && c < D4) ? part4[(cc * 2) * D4 + c] : f4_zero();
                }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int v = 0; v < NV; ++v) add_row(acc[v], t[u][v]);
        }
    };
    auto apply = [&](int64_t row, int v, double x, double y, double z, double w) {
        const int c = sub + v * G;
        if (c < D4)
            red_add_f4(&cache4[row * D4 + c],
                       make_float4(-(lr * (float)x), -(lr * (float)y), -(lr * (float)z), -(lr * (float)w)));
    };

    for (int64_t i = blockIdx.x; i < n_long; i += gridDim.x) {
        const int4 e = list[max_entries - 1 - i];            // (window, slot key of the run, -, -)
        const int64_t window = e.x, row = (int64_t)e.y - key_bias;
        if (window < 0 || window + 1 >= n_windows || row < 0 || row >= n_slots) continue;     // the same for all threads
        // last window that holds a piece of the run: window w > window holds one iff its first slot is the run's; window lo
        // does, window hi (if any) does not
        int64_t lo = window + 1, hi = n_windows;
        while (hi - lo > 1) {
            const int64_t step = (hi - lo + 31) / 32;
            const int64_t cc = lo + (lane + 1) * step;
            const bool t = cc < hi && keys[first + cc * kBwdWindow] == e.y;
            const int cnt = __popc(__ballot_sync(0xffffffffu, t));     // sorted keys: a prefix of the lanes
            const int64_t new_hi = min(hi, lo + (cnt + 1) * step);
            lo += cnt * step;
            hi = new_hi;
        }
        double acc[NV][4];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v][0] = acc[v][1] = acc[v][2] = acc[v][3] = 0.0;
        add_pieces(acc, window + 1 + wib * GW + gi, lo, (int64_t)kWarps * GW);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
#pragma unroll
            for (int k = 0; k < 4; ++k) s_sum[threadIdx.x][k] = acc[v][k];
            __syncthreads();
            const int c = sub + v * G;
            if (threadIdx.x < G && c < D4) {       // group 0 of warp 0: lane sub owns column c
                const float4 p = part4[(window * 2 + 1) * D4 + c];      // the piece in the run's first window
                double a[4] = {p.x, p.y, p.z, p.w};
#pragma unroll 8
                for (int g2 = 0; g2 < kWarps * GW; ++g2)
#pragma unroll
                    for (int k = 0; k < 4; ++k) a[k] += s_sum[g2 * G + sub][k];
                apply(row, v, a[0], a[1], a[2], a[3]);
            }
            __syncthreads();
        }
    }

    for (int64_t i = (int64_t)blockIdx.x * kWarps + wib; i < n_short; i += (int64_t)gridDim.x * kWarps) {
        const int4 e = list[i];                              // (window, slot key of the run, its last window, -)
        const int64_t window = e.x, last = e.z, row = (int64_t)e.y - key_bias;
        if (window < 0 || last <= window || last >= n_windows || row < 0 || row >= n_slots) continue;
        double acc[NV][4];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int c = sub + v * G;
            const float4 p = gi == 0 && c < D4 ? part4[(window * 2 + 1) * D4 + c] : f4_zero();
            acc[v][0] = p.x;
            acc[v][1] = p.y;
            acc[v][2] = p.z;
            acc[v][3] = p.w;
        }
        add_pieces(acc, window + 1 + gi, last, GW);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int off = G; off < 32; off <<= 1) acc[v][k] += __shfl_xor_sync(0xffffffffu, acc[v][k], off);
            if (gi == 0) apply(row, v, acc[v][0], acc[v][1], acc[v][2], acc[v][3]);
        }
    }

    // The lists are empty again for the next call: the last CTA to get here clears the counts (words 0 and 1) and the
    // tally of finished CTAs (word 2).  Every CTA read the counts when it started, and the next call's kernels start
    // after this grid has ended.
    __syncthreads();
    if (threadIdx.x == 0) {
        const int32_t finished = atomicAdd(&span_count[2], 1);
        if (finished == (int32_t)gridDim.x - 1) {
            span_count[0] = 0;
            span_count[1] = 0;
            span_count[2] = 0;
        }
    }
}

template <int G, int NV>
int32_t launch_fwd(hl_ctx* ctx, const float* cache, const hl_ubatch* ub, const int32_t* d_n, float* out,
                   const ForwardRows* fr, cudaStream_t stream) {
    constexpr int UB = NV >= 4 ? 1 : (NV >= 2 ? 2 : 4);
    timer_mark(ctx, HL_TIMER_FWD, 0, stream);
    // More than 1.5 lookups per bag at most: the loop for bags of one is not worth trying first.  (For those it is the better
    // one beside other kernels: click log 75 us per mini-batch, 77 with the other.)
    const bool many = 2 * ctx->max_nnz > 3 * (int64_t)ctx->max_bags;
    // a fixed number of CTAs per multiprocessor; in small calls of bags of several lookups a group has a bag or two
    using Shape = FwdShape<NV>;
    int per_sm = fwd_ctas_per_sm(ctx);
    if (many && ctx->fwd_ctas <= 0 && per_sm > Shape::CTAS) per_sm = Shape::CTAS;
    const int grid = grid_for(ctx->max_bags, many ? Shape::NT / G : kThreads / G * UB, per_sm * ctx_sms(ctx));
    const auto kernel = many ? (fr ? k_embbag_pool<G, NV, true> : k_embbag_pool<G, NV, false>)
                             : (fr ? k_embbag_fwd<G, NV, UB, true> : k_embbag_fwd<G, NV, UB, false>);
    HL_CUDA_TRY(launch_cluster(kernel, grid, many ? Shape::NT : kThreads, many ? Shape::kSmem : 0, 0, stream, cache, ub->ids,
                               ub->offsets, d_n, ctx->max_batch, ctx->T * ctx->S, ctx->D / 4,
                               ctx->hot_cap + ctx->staging_cap, out, ctx->r.status, fr ? *fr : ForwardRows{}));
    timer_mark(ctx, HL_TIMER_FWD, 1, stream);
    note_launches(1);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

template <int G, int NV>
int32_t launch_bwd(hl_ctx* ctx, float* cache, const int32_t* keys, const int32_t* vals, const int32_t* d_n_lookups,
                   const float* grad, float lr, cudaStream_t stream, const int32_t* d_first = nullptr,
                   int32_t key_bias = 0) {
    const int64_t max_chunks = div_up(ctx->max_nnz, kBwdChunk);
    // a fixed number of CTAs per multiprocessor (the warps stride over the chunks), so that kernels of other streams find
    // room beside this one: two rounds of those that fit
    constexpr bool kFour = G >= 16 && NV == 1;
    const bool four = kFour && max_chunks > 3 * (kThreads / 32) * ctx_sms(ctx) &&
                      (G == 16 || ctx->max_nnz > 16 * ctx->max_bags);
    const auto sums = four ? k_bwd_chunks<G, NV, kFour ? 4 : NV == 1 ? 3 : 1> : k_bwd_chunks<G, NV, NV == 1 ? 3 : 1>;
    const int per_sm = ctx->bwd_ctas > 0 ? ctx->bwd_ctas : four ? 8 : 6;
    const int grid = grid_for(max_chunks * 32, kThreads, per_sm * ctx_sms(ctx));
    const int64_t n_slots = ctx->hot_cap + ctx->staging_cap;
    timer_mark(ctx, HL_TIMER_BWD_REDUCE, 0, stream);
    // the list of runs that cross a chunk border sits behind the partial sums: [count words (8 ints)] [entries].
    // The count is zero between calls: hl_create clears it and k_bwd_spans clears it again when it is done (a call that
    // failed may have left it otherwise: scratch_kept).
    int32_t* span_count = span_count_of(ctx);
    int32_t* span_list = span_count + 8;
    if (ctx->spans_suspect) {
        HL_CUDA_TRY(clear_words(reinterpret_cast<uint32_t*>(span_count), 8, stream));
        ctx->spans_suspect = 0;
    }
    HL_CUDA_TRY(launch_cluster(sums, grid, kThreads, PieceShape<G, NV>::kDynamicBytes, 0, stream, cache, keys, vals, d_n_lookups,
                               grad, ctx->D / 4, n_slots, lr, ctx->r.bwd_part, d_first, key_bias, span_count, span_list,
                               ctx->max_bags, max_chunks, ctx->r.status));
    timer_mark(ctx, HL_TIMER_BWD_REDUCE, 1, stream);
    const int span_grid = grid_for(max_chunks * 32, kThreads, 2 * ctx_sms(ctx));   // the warps stride over the listed runs
    HL_CUDA_TRY(launch(k_bwd_spans<G, NV>, span_grid, kThreads, stream, cache, keys, d_n_lookups, ctx->D / 4, n_slots, lr,
                       ctx->r.bwd_part, d_first, key_bias, span_count, (const int32_t*)span_list, max_chunks));
    note_launches(2);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

int bits_for(int64_t max_value) {
    int b = 1;
    while ((int64_t(1) << b) <= max_value) ++b;
    return b;
}

}  // namespace
}  // namespace hl

using namespace hl;

#define HL_DISPATCH_ROW_SHAPE(D4, CALL)                  \
    do {                                                 \
        if ((D4) <= 4) return CALL(4, 1);                \
        if ((D4) <= 8) return CALL(8, 1);                \
        if ((D4) <= 16) return CALL(16, 1);              \
        if ((D4) <= 32) return CALL(32, 1);              \
        if ((D4) <= 64) return CALL(32, 2);              \
        if ((D4) <= 128) return CALL(32, 4);             \
        if ((D4) <= 256) return CALL(32, 8);             \
        return HL_EINVAL;                                \
    } while (0)

namespace hl {
namespace {

int32_t fwd_call(hl_ctx* ctx, const float* d_cache, const hl_ubatch* ub, const int32_t* d_n_samples, float* d_out,
                 const ForwardRows* fr, cudaStream_t stream) {
    if (!ctx || !d_cache || !ub || !ub->offsets || !d_n_samples || !d_out) return HL_EINVAL;
    if (ctx->max_nnz > 0 && !ub->ids) return HL_EINVAL;
#define HL_FWD(G, NV) launch_fwd<G, NV>(ctx, d_cache, ub, d_n_samples, d_out, fr, stream)
    HL_DISPATCH_ROW_SHAPE(ctx->D / 4, HL_FWD);
#undef HL_FWD
}

}  // namespace

bool piece_memory_granted(int D) {
    using Shape = PieceShape<32, 8>;
    if (D / 4 <= 128) return true;
    return cudaFuncSetAttribute(k_bwd_chunks<32, 8, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Shape::kDynamicBytes) == cudaSuccess;
}

int32_t fwd_and_forward_cold(hl_ctx* ctx, float* d_cache, const hl_ubatch* ub, const int32_t* d_n_samples, float* d_out,
                             int64_t from_stage_row0, int64_t to_stage_row0, int64_t stage_rows, const int32_t* d_fwd_src,
                             const int64_t* d_n_cold, cudaStream_t stream) {
    const ForwardRows fr{d_cache, ctx->hot_cap + from_stage_row0, ctx->hot_cap + to_stage_row0, d_fwd_src, d_n_cold,
                         stage_rows};
    return fwd_call(ctx, d_cache, ub, d_n_samples, d_out, &fr, stream);
}

}  // namespace hl

extern "C" int32_t hl_embbag_fwd(hl_ctx* ctx, const float* d_cache, const hl_ubatch* ub, const int32_t* d_n_samples,
                                 float* d_out, void* stream) {
    return as_graph(kept_launches(ctx), [&] {
        return fwd_call(ctx, d_cache, ub, d_n_samples, d_out, nullptr, static_cast<cudaStream_t>(stream));
    });
}

namespace hl {
namespace {

// The pairs described by `a` (its buffers and scratch are filled in here), sorted by key (stable).  The result lands in
// out_keys / out_vals: either the caller's arrays (which then serve as one half of the sort's ping-pong buffers) or, if
// they are null, whichever scratch buffer the last pass wrote.  cleared: the sort's scratch (sort_clear_words words of
// bwd_hist) is zero already.  aside: see SortAside.
// by_table: every table's pairs by themselves (the schedules' pairs: fragment laid them out by table, and no row belongs to two).
int32_t pairs_and_sort(hl_ctx* ctx, PairArgs a, int64_t max_key, bool assign, bool by_table, bool cleared, int32_t* caller_keys,
                       int32_t* caller_vals, int32_t* d_n_lookups, int32_t** out_keys, int32_t** out_vals,
                       cudaStream_t stream, const SortAside* aside = nullptr) {
    Regions& r = ctx->r;
    const int key_bits = bits_for(max_key), passes = by_table ? 1 : (key_bits + 7) / 8;
    const int which = aside ? aside->which : 0;          // (with caller arrays, one of the two scratch buffers is free)
    uint32_t* sort_scratch = r.bwd_hist[which];
    int32_t* keys[2] = {r.bwd_keys[which], r.bwd_keys[which ^ 1]};
    int32_t* vals[2] = {r.bwd_vals[which], r.bwd_vals[which ^ 1]};
    if (caller_keys) {   // make the buffer the last pass writes the caller's
        if ((passes & 1) == 0) {
            keys[1] = keys[0];
            vals[1] = vals[0];
        }
        keys[passes & 1] = caller_keys;
        vals[passes & 1] = caller_vals;
    }
    a.max_batch = ctx->max_batch;
    a.bags_per_sample_all = ctx->T * ctx->S;
    a.bags_per_sample = ctx->S;
    a.by_table = by_table && a.bags_follow;
    a.n_slots = ctx->hot_cap + ctx->staging_cap;
    a.max_nnz = ctx->max_nnz;
    a.keys = keys[0];
    a.vals = vals[0];
    a.d_n_lookups = d_n_lookups;
    a.status = r.status;
    a.ghist = sort_scratch;
    a.passes = passes;
    // the tile sort wants its digit counts, which cost less here than in a sweep of their own
    const int64_t clear_words = by_table ? 0 : sort_clear_words(ctx->max_nnz, key_bits, wait_cfg(ctx));
    const bool hist = clear_words > 0;
    if (hist && !cleared) HL_CUDA_TRY(hl::clear_words(sort_scratch, clear_words, stream));
    // lanes per bag: by the most lookups a bag has on average (bags of 20 out of at most 64: 20.8 us with 8 lanes, 22.2 with
    // 16, 25.5 with 32, which a bag does not fill; what is left is mostly the digit counts' shared-memory atomics)
    const int lanes = ctx->max_nnz <= 4 * ctx->max_bags ? 1 : (ctx->max_nnz <= 64 * ctx->max_bags ? 8 : 32);
    const int grid = grid_for(ctx->max_bags, kThreads / lanes, (lanes == 1 ? 4 : 8) * ctx_sms(ctx));
    const auto pick = [](bool as, bool hi, auto g) {
        constexpr int G = decltype(g)::value;
        return as ? (hi ? k_bwd_pairs<G, true, true> : k_bwd_pairs<G, true, false>)
                  : (hi ? k_bwd_pairs<G, false, true> : k_bwd_pairs<G, false, false>);
    };
    const auto kernel = lanes == 1   ? pick(assign, hist, std::integral_constant<int, 1>())
                        : lanes == 8 ? pick(assign, hist, std::integral_constant<int, 8>())
                                     : pick(assign, hist, std::integral_constant<int, 32>());
    HL_CUDA_TRY(launch(kernel, grid, kThreads, stream, a));
    note_launches(1);
    HL_LAUNCH_CHECK();
    if (aside) {
        HL_CUDA_TRY(launch_flush());
        HL_CUDA_TRY(cudaEventRecord(aside->pairs_ready, stream));
        HL_CUDA_TRY(cudaStreamWaitEvent(aside->stream, aside->pairs_ready, 0));
        stream = aside->stream;
    }
    if (by_table) {
        SegmentArgs g{};
        g.keys_in = keys[0];
        g.vals_in = vals[0];
        g.keys_out = *out_keys = keys[1];
        g.vals_out = *out_vals = vals[1];
        for (int i = 0; i < 2; ++i) g.side[i] = {a.side[i].offsets, a.side[i].d_n_samples, a.side[i].key_bias, 0};
        g.d_n_lookups = d_n_lookups;
        g.tables = ctx->T;
        g.max_batch = ctx->max_batch;
        g.bags_per_sample = ctx->S;
        g.merge = a.bags_follow;
        g.passes = (bits_for(a.n_slots) + 7) / 8;
        g.max_nnz = ctx->max_nnz;
        return sort_segments(g, stream);
    }
    return radix_sort_pairs(keys, vals, d_n_lookups + (a.sides > 1 ? 2 : 0), ctx->max_nnz, key_bits, sort_scratch, r.status,
                            out_keys, out_vals, stream, wait_cfg(ctx), hist);
}

int32_t sort_lookups(hl_ctx* ctx, const hl_ubatch* ub, const int32_t* d_n_samples, int32_t* caller_keys,
                     int32_t* caller_vals, int32_t* d_n_lookups, int32_t** out_keys, int32_t** out_vals,
                     cudaStream_t stream) {
    PairArgs a{};
    a.sides = 1;
    a.side[0] = {ub->ids, ub->offsets, d_n_samples, 0};
    return pairs_and_sort(ctx, a, ctx->hot_cap + ctx->staging_cap, false, false, false, caller_keys, caller_vals, d_n_lookups,
                          out_keys, out_vals, stream);
}

}  // namespace
}  // namespace hl

extern "C" int32_t hl_embbag_bwd_sgd(hl_ctx* ctx, float* d_cache, const hl_ubatch* ub, const int32_t* d_n_samples,
                                     const float* d_grad_out, float lr, void* stream_) {
    if (!ctx || !d_cache || !ub || !ub->offsets || !d_n_samples || !d_grad_out) return HL_EINVAL;
    if (ctx->max_nnz == 0) return HL_OK;
    if (!ub->ids) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    return scratch_kept(ctx, as_graph(kept_launches(ctx), [&]() -> int32_t {
        int32_t *keys, *vals;
        const int32_t st = sort_lookups(ctx, ub, d_n_samples, nullptr, nullptr, ctx->r.bwd_n, &keys, &vals, stream);
        if (st != HL_OK) return st;
#define HL_BWD(G, NV) launch_bwd<G, NV>(ctx, d_cache, keys, vals, ctx->r.bwd_n, d_grad_out, lr, stream)
        HL_DISPATCH_ROW_SHAPE(ctx->D / 4, HL_BWD);
#undef HL_BWD
    }));
}

extern "C" int32_t hl_embbag_bwd_prepare(hl_ctx* ctx, const hl_ubatch* ub, const int32_t* d_n_samples,
                                         int32_t* d_sorted_slots, int32_t* d_sorted_bags, int32_t* d_n_lookups,
                                         void* stream_) {
    if (!ctx || !ub || !ub->offsets || !d_n_samples || !d_n_lookups) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (ctx->max_nnz == 0) {
        HL_CUDA_TRY(cudaMemsetAsync(d_n_lookups, 0, sizeof(int32_t), stream));
        return HL_OK;
    }
    if (!ub->ids || !d_sorted_slots || !d_sorted_bags) return HL_EINVAL;
    return as_graph(kept_launches(ctx), [&] {
        int32_t *keys, *vals;
        return sort_lookups(ctx, ub, d_n_samples, d_sorted_slots, d_sorted_bags, d_n_lookups, &keys, &vals, stream);
    });
}

namespace hl {
namespace {

// merge = false: X's keys are offset by the number of slots + 1, so that the sorted list is O's pairs, then X's;
// merge = true: one key space, and X's bags are numbered behind O's: the lookups of a row from both micro-batches form one
// run, over one gradient array [bags of O; bags of X].
// Skipped lookups have the key n_slots (of X, merge = false: 2 * n_slots + 1): they are last among O's, or X's, pairs, or, where
// every table's pairs are sorted by themselves, last among each table's.
int32_t prepare_both(hl_ctx* ctx, const hl_ubatch* pop, const int32_t* d_n_pop, const hl_ubatch* non,
                     const int32_t* d_n_non, int32_t* d_sorted_slots, int32_t* d_sorted_bags, int32_t* d_n_lookups,
                     bool merge, PairArgs a, bool assign, bool by_table, bool cleared, cudaStream_t stream,
                     const SortAside* aside = nullptr, int32_t** out_slots = nullptr, int32_t** out_bags = nullptr) {
    if (!ctx || !pop || !non || !pop->offsets || !non->offsets || !d_n_pop || !d_n_non || !d_n_lookups)
        return HL_EINVAL;
    if (ctx->max_nnz == 0) {
        HL_CUDA_TRY(cudaMemsetAsync(d_n_lookups, 0, 4 * sizeof(int32_t), stream));
        return HL_OK;
    }
    if (!pop->ids || !non->ids || (!out_slots && (!d_sorted_slots || !d_sorted_bags))) return HL_EINVAL;
    const int64_t n_slots = ctx->hot_cap + ctx->staging_cap;
    if (2 * n_slots + 2 >= (int64_t(1) << 31)) return HL_EINVAL;
    a.sides = 2;
    a.bags_follow = merge;
    a.side[0] = {pop->ids, pop->offsets, d_n_pop, 0};
    a.side[1] = {non->ids, non->offsets, d_n_non, merge ? 0 : (int32_t)(n_slots + 1)};
    return as_graph(kept_launches(ctx), [&] {
        int32_t *ok, *ov;
        return pairs_and_sort(ctx, a, merge ? n_slots : 2 * n_slots + 1, assign, by_table, cleared, d_sorted_slots, d_sorted_bags,
                              d_n_lookups, out_slots ? out_slots : &ok, out_bags ? out_bags : &ov, stream, aside);
    });
}

}  // namespace

bool backward_sort_is_long(const hl_ctx* ctx) { return sort_is_long(ctx->max_nnz, wait_cfg(ctx)); }

// As many lookups as bags: one in every bag, in all likelihood, so that the tables have equally many.  (Otherwise some bags are
// empty and others long, and one table may have most of the lookups: k_sort_segments.)
bool backward_sorts_tables(const hl_ctx* ctx, const hl_batch* b, bool merge) {
    return b->nnz == (int64_t)ctx->T * b->batch * ctx->S &&
           sort_by_segments(ctx->max_nnz, ctx->max_bags, ctx->T, merge, wait_cfg(ctx));
}

int64_t backward_sort_clear_words(const hl_ctx* ctx, bool merge, bool by_table) {
    if (by_table) return 0;
    const int64_t n_slots = ctx->hot_cap + ctx->staging_cap;
    return sort_clear_words(ctx->max_nnz, bits_for(merge ? n_slots : 2 * n_slots + 1), wait_cfg(ctx));
}

int32_t assign_and_prepare(hl_ctx* ctx, const hl_ubatch* pop, const int32_t* d_n_pop, hl_ubatch* non,
                           const int32_t* d_n_non, int64_t stage_row0, int64_t stage_rows, const int32_t* d_cold_rows,
                           const int64_t* d_n_cold, const int32_t* d_prev_rows, const int64_t* d_n_prev,
                           int32_t* d_fwd_src, int32_t* d_sorted_slots, int32_t* d_sorted_bags, int32_t* d_n_lookups,
                           bool merge, bool by_table, cudaStream_t stream, const SortAside* aside, int32_t** out_slots,
                           int32_t** out_bags) {
    PairArgs a{};
    a.ranked = ctx->r.cold_ranked;
    a.slot0 = ctx->hot_cap + stage_row0;
    a.stage_rows = stage_rows;
    a.cold_rows = d_cold_rows;
    a.d_n_cold = d_n_cold;
    a.prev_rows = d_prev_rows;
    a.d_n_prev = d_n_prev;
    a.n_prev_max = ctx->staging_cap;
    a.fwd_src = d_fwd_src;
    return prepare_both(ctx, pop, d_n_pop, non, d_n_non, d_sorted_slots, d_sorted_bags, d_n_lookups, merge, a, true,
                        by_table, true, stream, aside, out_slots, out_bags);
}

}  // namespace hl

extern "C" int32_t hl_embbag_bwd_prepare2(hl_ctx* ctx, const hl_ubatch* pop, const int32_t* d_n_pop,
                                          const hl_ubatch* non, const int32_t* d_n_non, int32_t* d_sorted_slots,
                                          int32_t* d_sorted_bags, int32_t* d_n_lookups, void* stream) {
    return prepare_both(ctx, pop, d_n_pop, non, d_n_non, d_sorted_slots, d_sorted_bags, d_n_lookups, false, PairArgs{}, false,
                        false, false, static_cast<cudaStream_t>(stream));
}

extern "C" int32_t hl_embbag_bwd_prepare_merged(hl_ctx* ctx, const hl_ubatch* pop, const int32_t* d_n_pop,
                                                const hl_ubatch* non, const int32_t* d_n_non, int32_t* d_sorted_slots,
                                                int32_t* d_sorted_bags, int32_t* d_n_lookups, void* stream) {
    return prepare_both(ctx, pop, d_n_pop, non, d_n_non, d_sorted_slots, d_sorted_bags, d_n_lookups, true, PairArgs{}, false,
                        false, false, static_cast<cudaStream_t>(stream));
}

extern "C" int32_t hl_embbag_bwd_apply2(hl_ctx* ctx, float* d_cache, const int32_t* d_sorted_slots,
                                        const int32_t* d_sorted_bags, const int32_t* d_n_lookups, int32_t which,
                                        const float* d_grad_out, float lr, void* stream_) {
    if (!ctx || !d_cache || !d_n_lookups || !d_grad_out || (which != 0 && which != 1)) return HL_EINVAL;
    if (ctx->max_nnz == 0) return HL_OK;
    if (!d_sorted_slots || !d_sorted_bags) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const int32_t* d_first = which == 0 ? nullptr : d_n_lookups;             // X's block starts behind O's
    const int32_t bias = which == 0 ? 0 : (int32_t)(ctx->hot_cap + ctx->staging_cap + 1);
    return scratch_kept(ctx, as_graph(kept_launches(ctx), [&]() -> int32_t {
#define HL_BWD(G, NV) \
    launch_bwd<G, NV>(ctx, d_cache, d_sorted_slots, d_sorted_bags, d_n_lookups + which, d_grad_out, lr, stream, d_first, bias)
        HL_DISPATCH_ROW_SHAPE(ctx->D / 4, HL_BWD);
#undef HL_BWD
    }));
}

extern "C" int32_t hl_embbag_bwd_apply(hl_ctx* ctx, float* d_cache, const int32_t* d_sorted_slots,
                                       const int32_t* d_sorted_bags, const int32_t* d_n_lookups,
                                       const float* d_grad_out, float lr, void* stream_) {
    if (!ctx || !d_cache || !d_n_lookups || !d_grad_out) return HL_EINVAL;
    if (ctx->max_nnz == 0) return HL_OK;
    if (!d_sorted_slots || !d_sorted_bags) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    return scratch_kept(ctx, as_graph(kept_launches(ctx), [&]() -> int32_t {
#define HL_BWD(G, NV) launch_bwd<G, NV>(ctx, d_cache, d_sorted_slots, d_sorted_bags, d_n_lookups, d_grad_out, lr, stream)
        HL_DISPATCH_ROW_SHAPE(ctx->D / 4, HL_BWD);
#undef HL_BWD
    }));
}

// ---------------------------------------------------------------------------------------------------------------
// Backward without a context or a workspace: the scratch is a fixed array inside the library image.
// ---------------------------------------------------------------------------------------------------------------
namespace hl {
namespace {

constexpr int64_t kStaticMaxNnz = HL_STATIC_MAX_NNZ;
constexpr int64_t kStaticMaxDim = HL_STATIC_MAX_DIM;

constexpr size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
// layout of the static scratch: [header: status (8 ints), bag count word + lookup count (8 ints)] [keys x2]
// [vals x2] [histogram] [partial sums]
constexpr size_t kStaticHeaderBytes = 256;
constexpr size_t kStaticPairBytes = align256(size_t(kStaticMaxNnz) * sizeof(int32_t));
constexpr int64_t kStaticHistWords = sort_hist_words(kStaticMaxNnz);
constexpr size_t kStaticHistBytes = align256(size_t(kStaticHistWords) * sizeof(uint32_t));
constexpr size_t kStaticPartBytes =
    align256(size_t(2) * ((kStaticMaxNnz + kBwdChunk - 1) / kBwdChunk) * kStaticMaxDim * sizeof(float) +
             bwd_span_list_words(kStaticMaxNnz) * sizeof(int32_t));
constexpr size_t kStaticScratchBytes = kStaticHeaderBytes + 4 * kStaticPairBytes + kStaticHistBytes + kStaticPartBytes;

// Lives in every device's copy of the library image from load to exit (about 3 MB).  The name below is only a
// host-side handle for cudaGetSymbolAddress; kernels get the real device address as an argument.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

std::mutex g_static_mutex;
unsigned char* g_static_ptr[64] = {};   // device address of g_static_scratch, per device ordinal

__global__ void k_static_begin(int32_t* header, int32_t n_bags, int32_t* span_count) {
    header[0] = 0;        // status word: every call starts clean
    header[8] = n_bags;   // the backward kernels read their bag count from device memory
    // the count words of the backward's run list: their place in the array depends on the call's sizes, so an earlier
    // call may have left partial sums there
    for (int i = 0; i < 8; ++i) span_count[i] = 0;
}

__global__ void k_static_end(const int32_t* header, int32_t* d_status) { *d_status = header[0]; }

}  // namespace
}  // namespace hl

extern "C" int32_t hl_embbag_bwd_sgd_static(float* d_cache, int64_t cache_rows, int32_t dim,
                                            const int32_t* d_offsets, const int32_t* d_ids, int32_t n_bags,
                                            int64_t nnz, const float* d_grad_out, float lr, int32_t* d_status,
                                            void* stream_) {
    if (!d_cache || !d_offsets || !d_grad_out || cache_rows < 1 || cache_rows >= (int64_t(1) << 31) - 2)
        return HL_EINVAL;
    if (dim < 4 || (dim & 3) || n_bags < 0 || nnz < 0 || (nnz > 0 && !d_ids)) return HL_EINVAL;
    if (nnz > kStaticMaxNnz || n_bags > kStaticMaxNnz || dim > kStaticMaxDim) return HL_ECAPACITY;
    if (sort_hist_words(nnz) > kStaticHistWords) return HL_ECAPACITY;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);

    // set-up, once per device: ask the runtime where this device keeps the array
    int dev = 0;
    HL_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return HL_EINVAL;
    unsigned char* base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_ptr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) return HL_ECUDA;
            g_static_ptr[dev] = static_cast<unsigned char*>(p);
        }
        base = g_static_ptr[dev];
    }
    if (nnz == 0 || n_bags == 0) {
        if (d_status) HL_CUDA_TRY(cudaMemsetAsync(d_status, 0, sizeof(int32_t), stream));
        return HL_OK;
    }

    // a context on the stack whose backward region points into the static array; nothing else is used
    hl_ctx tmp{};
    tmp.T = 1;
    tmp.S = 1;
    tmp.D = dim;
    tmp.N = cache_rows;
    tmp.max_batch = n_bags;
    tmp.max_bags = n_bags;
    tmp.max_nnz = nnz;
    tmp.hot_cap = cache_rows;
    tmp.staging_cap = 0;
    int32_t* header = reinterpret_cast<int32_t*>(base);
    unsigned char* p = base + kStaticHeaderBytes;
    tmp.r.status = header;
    tmp.r.bwd_n = header + 12;
    for (int i = 0; i < 2; ++i) {
        tmp.r.bwd_keys[i] = reinterpret_cast<int32_t*>(p);
        p += kStaticPairBytes;
        tmp.r.bwd_vals[i] = reinterpret_cast<int32_t*>(p);
        p += kStaticPairBytes;
    }
    tmp.r.bwd_hist[0] = reinterpret_cast<uint32_t*>(p);
    p += kStaticHistBytes;
    tmp.r.bwd_part = reinterpret_cast<float*>(p);

    HL_CUDA_TRY(launch(k_static_begin, 1, 1, stream, header, n_bags, span_count_of(&tmp)));
    note_launches(1);
    HL_LAUNCH_CHECK();
    hl_ubatch ub{const_cast<int32_t*>(d_offsets), const_cast<int32_t*>(d_ids), nnz};
    const int32_t st = hl_embbag_bwd_sgd(&tmp, d_cache, &ub, header + 8, d_grad_out, lr, stream_);
    if (st != HL_OK) return st;
    if (d_status) {
        HL_CUDA_TRY(launch(k_static_end, 1, 1, stream, header, d_status));
        note_launches(1);
        HL_LAUNCH_CHECK();
    }
    return HL_OK;
}
