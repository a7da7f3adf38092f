// The non-popular micro-batch's working set: classify its lookups, find the distinct cold rows, stage them from the
// host-DRAM table (bulk copies over the host link, row by row) behind the hot cache, and write them back.
#include "hl_common.cuh"

namespace hl {
namespace {

constexpr int kThreads = 256;

// ---- the distinct cold rows, in ascending order --------------------------------------------------------------
// One bit per row of the model: classifying X's lookups sets the bits of its cold rows (mark_cold), k_cold_rank
// reads the bitmap in row order -- which is ascending order without a sort -- and hands out the ranks, and k_cold_assign
// turns every cold lookup into the slot of its row's rank.  The work depends on the lookups and (a 32nd or a 1024th of
// a word per row) on the size of the model, not on how many cold lookups there are, so there is one path for all
// mini-batches: three kernels where a sort of the cold lookups took a cluster of 16 CTAs 21-43 us (up to 40 960 lookups)
// or ten device-launched kernels and 0.3-0.7 ms (above).
__global__ void __launch_bounds__(kThreads) k_cold_classify(int32_t* __restrict__ ids,
                                                            const int32_t* __restrict__ offsets,
                                                            const int32_t* __restrict__ d_n_non, int max_batch,
                                                            int bags_per_sample_all, int64_t cap_ids, int64_t N,
                                                            BitmapProbe remap, ColdMarks marks, int32_t* status) {
    clear_cold_chain(marks);
    int n_non = *d_n_non;
    n_non = n_non < 0 ? 0 : (n_non > max_batch ? max_batch : n_non);
    int64_t L = offsets[(int64_t)n_non * bags_per_sample_all];
    if (L > cap_ids) L = cap_ids;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < L; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t g = ids[j];
        if (g >= N) {
            set_status(status, HL_EBOUNDS);
            ids[j] = -1;
        } else if (g >= 0) {
            const uint32_t word = marks.bits[g >> 5];
            const int32_t slot = remap.slot(remap.request(g), g);
            ids[j] = slot >= 0 ? slot : cold_id(g);
            if (slot < 0) mark_cold(marks, g, word);
        }
    }
}

// Tiles of kThreads * ITEMS words, chained (chain_before; marks.chain is zero on entry).
// SUMMARY: the words are those of the summary, which has a bit for every bitmap word that is not zero (large models, whose
// bitmap would be megabytes of zeros to read: cold_direct); otherwise the bitmap's own.  Bitmap and summary
// are left cleared; marks.ranked[word] keeps what k_cold_assign needs: the word's bits and the rank of its first one.
template <bool SUMMARY, int ITEMS>
__global__ void __launch_bounds__(kThreads) k_cold_rank(ColdMarks marks, int n_words, int64_t staging_cap,
                                                        int32_t* __restrict__ cold_rows, int64_t* __restrict__ d_n_cold,
                                                        int32_t* status, int max_polls, int64_t stall_tile,
                                                        uint32_t* __restrict__ clear, int64_t n_clear) {
    constexpr int NW = kThreads / 32;
    __shared__ int s_sum[NW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n_clear / 4; i += (int64_t)gridDim.x * kThreads)
        reinterpret_cast<uint4*>(clear)[i] = make_uint4(0u, 0u, 0u, 0u);
    const int tile = blockIdx.x;
    const int first = tile * kThreads * ITEMS;
    uint32_t word[ITEMS];
    int start[ITEMS], all = 0;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int w = first + (warp * ITEMS + i) * 32 + lane;
        word[i] = w < n_words ? (SUMMARY ? marks.summary[w] : marks.bits[w]) : 0u;
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int w = first + (warp * ITEMS + i) * 32 + lane;
        int n = 0;
        if (SUMMARY) {
            for (uint32_t m = word[i]; m; m &= m - 1) n += __popc(marks.bits[(int64_t)w * 32 + __ffs((int)m) - 1]);
        } else {
            n = __popc(word[i]);
        }
        int incl = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        start[i] = all + incl - n;
        all += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) s_sum[warp] = all;
    __syncthreads();
    int tile_sum = 0, warp_start = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        if (k < warp) warp_start += s_sum[k];
        tile_sum += s_sum[k];
    }
    if (tile != stall_tile) chain_publish(marks.chain, tile, (unsigned long long)tile_sum);
    const int before = (int)chain_before<kThreads>(marks.chain, tile, (unsigned long long)tile_sum, tile != stall_tile,
                                                   max_polls, status);
    if (threadIdx.x == 0 && first + kThreads * ITEMS >= n_words) {       // the last tile knows the total
        int64_t distinct = (int64_t)before + tile_sum;
        if (distinct > staging_cap) {
            set_status(status, HL_ECAPACITY);
            distinct = staging_cap;
        }
        *d_n_cold = distinct;
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int w = first + (warp * ITEMS + i) * 32 + lane;
        int rank = before + warp_start + start[i];
        auto take = [&](int64_t at, uint32_t bits) {         // bitmap word `at`
            marks.bits[at] = 0u;
            marks.ranked[at] = make_uint2(bits, (unsigned)rank);
            for (uint32_t m = bits; m; m &= m - 1, ++rank)
                if (rank < staging_cap) cold_rows[rank] = (int32_t)(at * 32 + __ffs((int)m) - 1);
        };
        if (word[i] == 0u) continue;
        if (SUMMARY) {
            marks.summary[w] = 0u;
            for (uint32_t m = word[i]; m; m &= m - 1) {
                const int64_t at = (int64_t)w * 32 + __ffs((int)m) - 1;
                take(at, marks.bits[at]);
            }
        } else {
            take(w, word[i]);
        }
    }
}

// Every cold lookup of X (an id of -2 - g) gets the staging slot of its row: slot0 + rank (slot0 = start of the window).
__global__ void __launch_bounds__(kThreads) k_cold_assign(int32_t* __restrict__ ids, const int32_t* __restrict__ offsets,
                                                          const int32_t* __restrict__ d_n_non, int max_batch,
                                                          int bags_per_sample_all, int64_t cap_ids,
                                                          const uint2* __restrict__ ranked, int64_t slot0,
                                                          int64_t staging_cap) {
    int n_non = *d_n_non;
    n_non = n_non < 0 ? 0 : (n_non > max_batch ? max_batch : n_non);
    int64_t L = offsets[(int64_t)n_non * bags_per_sample_all];
    if (L > cap_ids) L = cap_ids;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < L; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t id = ids[j];
        if (id <= -2) ids[j] = cold_slot(ranked, id, slot0, staging_cap);
    }
}

// dst[(dst_row0 + i), :] = table[rows[i], :] (or the other way round); G lanes per row, UR rows in flight per
// group.  Rows i with skip[i] >= 0 are left alone.
template <int G, bool TO_TABLE>
__global__ void __launch_bounds__(kThreads) k_move_rows(float* __restrict__ dense_side, int64_t dense_row0,
                                                        TableMap table, const int32_t* __restrict__ rows,
                                                        const int64_t* __restrict__ d_n, int64_t n_max,
                                                        int64_t table_rows, int D4,
                                                        const int32_t* __restrict__ skip, int32_t* status) {
    constexpr int UR = 16;
    int64_t n = *d_n;
    n = n < 0 ? 0 : (n < n_max ? n : n_max);
    const int sub = threadIdx.x % G;
    const int64_t group = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / G;
    const int64_t n_groups = (int64_t)gridDim.x * kThreads / G;
    float4* dense4 = reinterpret_cast<float4*>(dense_side) + dense_row0 * D4;
    for (int64_t i0 = group * UR; i0 < n; i0 += n_groups * UR) {
        float4* trow[UR];              // the row in the host table, nullptr = nothing to move
#pragma unroll
        for (int u = 0; u < UR; ++u) {
            int64_t g = i0 + u < n ? (int64_t)rows[i0 + u] : -1;
            if (skip != nullptr && g >= 0 && skip[i0 + u] >= 0) g = -1;   // row comes from elsewhere
            if (g >= table_rows) {
                set_status(status, HL_EBOUNDS);
                g = -1;
            }
            trow[u] = g >= 0 ? reinterpret_cast<float4*>(row_address(table, g, D4 * 16)) : nullptr;
        }
        for (int c = sub; c < D4; c += G) {
            float4 v[UR];
#pragma unroll
            for (int u = 0; u < UR; ++u)
                if (trow[u]) v[u] = TO_TABLE ? dense4[(i0 + u) * D4 + c] : trow[u][c];
#pragma unroll
            for (int u = 0; u < UR; ++u)
                if (trow[u]) {
                    if (TO_TABLE) trow[u][c] = v[u];
                    else dense4[(i0 + u) * D4 + c] = v[u];
                }
        }
    }
}

// src[i] = position of rows[i] in the ascending list prev[0 .. *d_n_prev), or -1.
__global__ void __launch_bounds__(kThreads) k_cold_match(const int32_t* __restrict__ rows,
                                                         const int64_t* __restrict__ d_n, int64_t n_max,
                                                         const int32_t* __restrict__ prev,
                                                         const int64_t* __restrict__ d_n_prev, int64_t n_prev_max,
                                                         int32_t* __restrict__ src) {
    int64_t n = *d_n, np = *d_n_prev;
    n = n < 0 ? 0 : (n < n_max ? n : n_max);
    np = np < 0 ? 0 : (np < n_prev_max ? np : n_prev_max);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        src[i] = position_in(prev, np, rows[i]);
    }
}

// cache[to_row0 + i, :] = cache[from_row0 + src[i], :] for every i < *d_n with src[i] >= 0.
template <int G>
__global__ void __launch_bounds__(kThreads) k_forward_rows(float* cache, int64_t from_row0, int64_t to_row0,
                                                           const int32_t* __restrict__ src,
                                                           const int64_t* __restrict__ d_n, int64_t n_max, int D4) {
    int64_t n = *d_n;
    n = n < 0 ? 0 : (n < n_max ? n : n_max);
    const int sub = threadIdx.x % G;
    const int64_t group = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / G;
    const int64_t n_groups = (int64_t)gridDim.x * kThreads / G;
    float4* c4 = reinterpret_cast<float4*>(cache);
    for (int64_t i = group; i < n; i += n_groups) {
        const int32_t j = src[i];
        if (j < 0 || j >= n_max) continue;
        for (int c = sub; c < D4; c += G) c4[(to_row0 + i) * D4 + c] = c4[(from_row0 + j) * D4 + c];
    }
}

// ---- row mover on the bulk-copy (TMA) engine ----------------------------------------------------------------
// The same copy as k_move_rows, issued as asynchronous bulk copies: every row is one cp.async.bulk from its
// source into shared memory (completion counted in bytes on an mbarrier) and one cp.async.bulk from shared memory
// to its destination.  The rows in flight are then requests of the copy engine of the SM, not pending loads of
// its load-store unit, so that embedding-bag CTAs of another micro-batch that share the SM keep their own
// loads moving while hundreds of host rows, each waiting microseconds for its address translation, are pending.
// Source, destination and row size are multiples of 16 bytes (dim % 4 == 0, 16-byte aligned bases).
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bulk_load(void* smem_dst, const void* gmem_src, uint32_t bytes, uint64_t* mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(smem_dst)),
                 "l"(gmem_src), "r"(bytes), "r"(smem_u32(mbar))
                 : "memory");
}
__device__ __forceinline__ void bulk_store(void* gmem_dst, const void* smem_src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gmem_dst),
                 "r"(smem_u32(smem_src)), "r"(bytes)
                 : "memory");
}

constexpr int kBulkThreads = 128;
constexpr int kBulkStages = 3;
constexpr int kBulkStageBytes = 12288;
constexpr int kBulkMaxPolls = 1 << 22;
constexpr int kBulkStagesPerCta = 200;    // stages of rows per working CTA before another CTA joins in
// How many rows are on the link at a time decides what the transfer costs everything else on the chip.  The link takes
// some 300 M requests a second of a mini-batch's rows (a request: a row's 128-byte line, or what there is of it; rows that lie
// close to one another, as a popular set's do, up to 580 M a second) and answers in about 1.5 us, so
// 400 to 500 outstanding requests fill it; any more queue up in front of it, and the memory system behind the queue comes
// to a near standstill.  Measured beside write-backs of random rows of 64 bytes (256 bytes): 16 CTAs that put up to 32 KB
// each on the way move 288 M (302 M) requests a second, a streaming read of 256 MB takes 217 us (104) instead of 62, and a
// kernel that does next to nothing takes 24 us (12) instead of 4; 8 CTAs with 48 requests each move 210 M (193 M), and
// the read takes 65 us (66), the small kernel 6.8 us (6.4).  Reads of host rows are milder: 8 CTAs with 16 KB each reach
// 226 M (259 M) requests a second, and the streaming read takes 67 us (68).  So inside a schedule a transfer that is short
// all the same is paced: writes with kPacedRequests requests per CTA and every store completed before the next ones start,
// reads with two stages of kPacedReadBytes on the way.  16 CTAs of these move the 7.4 thousand rows of 64 bytes of a
// click-log mini-batch in 34 us (in) and 29 us (out), the 8.7 thousand rows of 256 bytes of a DLRM-sized one in 75 us and
// 70 us: what the full-rate mover takes while nothing else runs, and one pass of the schedule went from 174 to 157 us
// (DLRM-sized) and from 86 to 76 us (click log).  Above kPacedMost requests the link is what the mini-batch waits for, and
// the mover takes it all.
constexpr int kPacedRequests = 40;
constexpr int kPacedReadBytes = 8192;
constexpr int64_t kPacedMost = 1 << 16;
// How many CTAs a paced read gets goes by its rows.  Up to some 10 thousand the rows are there in time with 16 CTAs, and more
// of them only disturb the kernels beside them; beyond that the read is what the mini-batch waits for.  One pipeline, 16
// against 24 CTAs, us per mini-batch (26 tables; rows read): rows of 256 bytes out of 2 GiB 5.0 K 83 / 84, 7.3 K 114 / 114,
// 10.9 K 167 / 161; out of 24 GiB 4.7 K 82 / 85, 7.7 K 115 / 115, 12.5 K 183 / 170, 19.9 K 294 / 264; out of 6, 36, 48, 61 GiB
// 15.5 K 236 / 210, 19.3 K 281 / 260, 18.5 K 281 / 251, 16.1 K 246 / 225.  Rows of 64 bytes: 3.7 K 56 / 56, 8.8 K 89 / 86, 13.3 K
// 127 / 121 (2 GiB); 5.1 K 67 / 67, 8.6 K 91 / 90, 13.6 K 139 / 128, 22.3 K 221 / 200 (24 GiB).  Rows of 512 bytes: 3.7 K 110 /
// 115, 5.3 K 150 / 153, 7.4 K 218 / 224 (2 GiB); 6.3 K 157 / 167, 9.5 K 237 / 236, 14.5 K 362 / 353 (24 GiB).  The size of the
// table plays no part.  (32 CTAs: within 2 % of 24 for wide rows, 5 % faster for 20 K rows of 64 bytes.  Three pipelines in
// turn on one chip, which no program runs, lose 1 to 4 % with 24: 12.4 K rows of 256 bytes 175 / 181.)
constexpr int64_t kPacedFewRows = 10240;

// A transfer with nothing else on the chip (the popular rows, out and in) has 32 CTAs, which put 3 to 8 thousand requests on
// the way; rows from 256 bytes on are read with two CTAs per multiprocessor.  More requests than that do not make the link
// faster, and rows that are asked for far apart from one another miss more of what translates and holds their neighbours
// (the rows of a transfer are in ascending order).  330 K rows, 2 GiB table, two CTAs per multiprocessor / 32 CTAs, us: rows of
// 64 bytes read 732 / 610, written 759 / 624; 144 bytes (300 K) 1 822 / 1 685, 1 944 / 1 445; 192 bytes (250 K) 1 053 / 1 027,
// 1 103 / 1 040; 256 bytes (200 K) 1 016 / 1 013, 1 065 / 1 062.  40 GiB table: 64 bytes 1 233 / 1 076, 1 224 / 1 125; 256 bytes
// 1 664 / 1 814, 1 906 / 1 870; 512 bytes (200 K) 2 008 / 2 240, 2 116 / 2 098.
// (A table in device memory has no link in between: two CTAs per multiprocessor, 1 M of 2 M rows of 64 bytes written 86 us, read 106,
// with 32 CTAs 645 and 645; of 256 bytes 201 and 222, written with 32 CTAs 1 697.)
constexpr int kAloneCtas = 32;
constexpr int kAloneWideRow = 256;

// What a launch of the mover needs to know about its context.
struct MoveCfg {
    int sms;            // multiprocessors of the device: the launch has at most 2 CTAs per SM
    bool link_alone;    // nothing else on the chip, and the table is behind the link
    int min_ctas;       // CTAs that work however few rows there are (at full rate)
    int paced_ctas;     // CTAs of a paced transfer of up to kPacedFewRows rows; 0: never paced
    int paced_more;     // ... of more rows
    int max_polls;      // poll limit of the wait for a stage to fill
    int stall;          // tests only: CTA 0 issues no loads for its first stage, whose wait then runs out
};

// One row per thread and stage.  While the rows of one stage travel, the next stage's are requested (and the row ids of
// the one after that are read): the loop waits for one thing at a time.
template <bool TO_TABLE>
__global__ void __launch_bounds__(kBulkThreads) k_move_rows_bulk(float* dense_side, int64_t dense_row0, TableMap table,
                                                                 const int32_t* __restrict__ rows,
                                                                 const int64_t* __restrict__ d_n, int64_t n_max,
                                                                 int64_t table_rows, int row_bytes,
                                                                 int rows_per_stage,
                                                                 const int32_t* __restrict__ skip, int32_t* status,
                                                                 int min_ctas, int paced_ctas, int paced_more,
                                                                 int64_t paced_most,
                                                                 int paced_rows, int max_polls, int stall) {
    __shared__ __align__(128) unsigned char stage[kBulkStages][kBulkStageBytes];
    __shared__ __align__(8) uint64_t mbar[kBulkStages];
    __shared__ int s_gave_up;
    int64_t n = *d_n;
    n = n < 0 ? 0 : (n < n_max ? n : n_max);
    const int tid = threadIdx.x;
    if (tid == 0) {
        for (int s = 0; s < kBulkStages; ++s)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&mbar[s])), "r"(1) : "memory");
        s_gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    unsigned char* dense = reinterpret_cast<unsigned char*>(dense_side) + dense_row0 * row_bytes;
    const bool paced = paced_ctas > 0 && n <= paced_most;
    if (paced) rows_per_stage = paced_rows;
    const int64_t n_batches = (n + rows_per_stage - 1) / rows_per_stage;
    // The launch has as many CTAs as the largest transfer could use; how many of them work is decided here, from the
    // number of rows there really are: few for a mini-batch's worth of a DLRM-sized model (more would only slow
    // the kernels that run beside the mover), up to all of them when a mini-batch moves hundreds of thousands of rows
    // (the link is then all that matters): one more CTA for every kBulkStagesPerCta stages of rows.
    int64_t active = n_batches / kBulkStagesPerCta;
    active = active < min_ctas ? min_ctas : active;
    if (paced) active = n > kPacedFewRows ? paced_more : paced_ctas;
    active = active < (int64_t)gridDim.x ? active : (int64_t)gridDim.x;
    if ((int64_t)blockIdx.x >= active) return;

    // this thread's row of a batch, -1 if it has none or the row does not move
    auto row_of = [&](int64_t batch) -> int64_t {
        const int64_t i = batch * rows_per_stage + tid;
        if (tid >= rows_per_stage || i >= n) return -1;
        const int64_t g = rows[i];
        if (g >= table_rows) {
            set_status(status, HL_EBOUNDS);
            return -1;
        }
        return skip != nullptr && skip[i] >= 0 ? -1 : g;
    };
    auto dense_row = [&](int64_t batch) { return dense + (batch * rows_per_stage + tid) * row_bytes; };
    // all threads: requests the rows of a batch into stage s
    auto request = [&](int s, int64_t batch, int64_t g, bool withhold) {
        const int moving = __syncthreads_count(g >= 0);
        if (tid == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&mbar[s])),
                         "r"((unsigned)moving * (unsigned)row_bytes)
                         : "memory");
        if (g >= 0 && !withhold)
            bulk_load(&stage[s][tid * row_bytes], TO_TABLE ? dense_row(batch) : row_address(table, g, row_bytes),
                      (uint32_t)row_bytes, &mbar[s]);
    };

    int64_t batch = blockIdx.x;
    if (batch >= n_batches) return;
    int64_t g = row_of(batch), g1 = batch + active < n_batches ? row_of(batch + active) : -1;
    request(0, batch, g, stall && blockIdx.x == 0);          // (stall: tests; the expected bytes never arrive)
    for (int it = 0; batch < n_batches; batch += active, ++it) {
        const int s = it % kBulkStages;
        const uint32_t parity = (uint32_t)(it / kBulkStages) & 1u;
        if (batch + active < n_batches) {
            // the stores that last left from the next stage's place have finished reading shared memory
            asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kBulkStages - 2) : "memory");
            request((it + 1) % kBulkStages, batch + active, g1, false);
        }
        const int64_t g2 = batch + 2 * active < n_batches ? row_of(batch + 2 * active) : -1;
        // wait for the stage to fill (bounded)
        uint32_t done = 0;
        for (int polls = 0; !done; ++polls) {
            asm volatile(
                "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                : "=r"(done)
                : "r"(smem_u32(&mbar[s])), "r"(parity)
                : "memory");
            if (!done && polls > max_polls) {
                set_status(status, HL_ETIMEOUT);
                s_gave_up = 1;
                break;
            }
        }
        // A wait that ran out ends this CTA's work: the stage is not written, no further stage is started (its
        // barrier phases would be out of step), and the CTA leaves once its earlier stores have completed.  The rows
        // it was responsible for stay unmoved; the status word says so.
        __syncthreads();
        if (s_gave_up) break;
        // (paced: this thread's earlier store has arrived)
        if (TO_TABLE && paced) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        if (g >= 0)
            bulk_store(TO_TABLE ? row_address(table, g, row_bytes) : dense_row(batch), &stage[s][tid * row_bytes],
                       (uint32_t)row_bytes);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        g = g1;
        g1 = g2;
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (s_gave_up) {
        // loads of the abandoned stages that are still on their way get a bounded grace period to land before the
        // shared memory goes back to the SM
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
}

template <bool TO_TABLE>
int32_t launch_move_rows(float* dense_side, int64_t dense_row0, TableMap table, const int32_t* rows,
                         const int64_t* d_n, int64_t n_max, int64_t table_rows, int D, const int32_t* skip,
                         MoveCfg cfg, int32_t* status, cudaStream_t stream) {
    if (n_max <= 0) return HL_OK;
    const int D4 = D / 4;
    const int row_bytes = D * 4;
    if (row_bytes <= kBulkStageBytes) {
        const int rows_per_stage = kBulkStageBytes / row_bytes < kBulkThreads ? kBulkStageBytes / row_bytes : kBulkThreads;
        const bool few = cfg.link_alone && (TO_TABLE || row_bytes < kAloneWideRow);
        const int grid = grid_for(n_max, rows_per_stage, few ? kAloneCtas : 2 * cfg.sms);
        const int requests = (row_bytes + 127) / 128;        // of one row
        const int paced_fit = TO_TABLE ? kPacedRequests / requests : kPacedReadBytes / row_bytes;
        const int paced_rows = paced_fit > 1 ? paced_fit : 1;
        HL_CUDA_TRY(launch(k_move_rows_bulk<TO_TABLE>, grid, kBulkThreads, stream, dense_side, dense_row0, table, rows, d_n,
                           n_max, table_rows, row_bytes, rows_per_stage, skip, status,
                           cfg.min_ctas < grid ? cfg.min_ctas : grid, cfg.paced_ctas, cfg.paced_more,
                           kPacedMost / requests,
                           paced_rows < rows_per_stage ? paced_rows : rows_per_stage, cfg.max_polls, cfg.stall));
        note_launches(1);
        HL_LAUNCH_CHECK();
        return HL_OK;
    }
    // Rows wider than a stage of the bulk mover (12 KB): plain 128-bit loads and stores, 48 CTAs x 16 groups x 16 rows
    // in flight on a third of the SMs, so that the kernels of the other streams keep CTA slots.
    const int grid = 48;
    if (D4 <= 4)
        HL_CUDA_TRY(launch(k_move_rows<4, TO_TABLE>, grid, kThreads, stream, dense_side, dense_row0, table, rows, d_n,
                           n_max, table_rows, D4, skip, status));
    else if (D4 <= 8)
        HL_CUDA_TRY(launch(k_move_rows<8, TO_TABLE>, grid, kThreads, stream, dense_side, dense_row0, table, rows, d_n,
                           n_max, table_rows, D4, skip, status));
    else if (D4 <= 16)
        HL_CUDA_TRY(launch(k_move_rows<16, TO_TABLE>, grid, kThreads, stream, dense_side, dense_row0, table, rows, d_n,
                           n_max, table_rows, D4, skip, status));
    else
        HL_CUDA_TRY(launch(k_move_rows<32, TO_TABLE>, grid, kThreads, stream, dense_side, dense_row0, table, rows, d_n,
                           n_max, table_rows, D4, skip, status));
    note_launches(1);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

}  // namespace

int32_t marks_fresh(hl_ctx* ctx, cudaStream_t stream) {
    if (!ctx->marks_suspect) return HL_OK;
    const ColdMarks marks = cold_marks(ctx);
    HL_CUDA_TRY(clear_words(marks.bits, cold_bitmap_words(ctx->N), stream));
    if (marks.summary) HL_CUDA_TRY(clear_words(marks.summary, cold_summary_words(ctx->N), stream));
    ctx->marks_suspect = 0;
    return HL_OK;
}

int32_t cold_rank(hl_ctx* ctx, int64_t stage_rows, int32_t* d_cold_rows, int64_t* d_n_cold, cudaStream_t stream,
                  uint32_t* clear, int64_t n_clear) {
    const Regions& r = ctx->r;
    const ColdMarks marks = cold_marks(ctx);
    const bool summary = marks.summary != nullptr;
    const int64_t words = summary ? cold_summary_words(ctx->N) : cold_bitmap_words(ctx->N);
    // words per thread: as in hl_fragment, one until there is a tile per multiprocessor
    const bool many = words > (int64_t)kThreads * ctx_sms(ctx);
    // and eight for large bitmaps, where a tile is mostly its wait for the one before it.  Four / eight, alone, us: 16.8 M rows
    // with 10 K lookups 10.4 / 8.9, 26 K 11.0 / 9.0, 106 K 12.1 / 13.1, 426 K 14.8 / 15.8; 25 M 16.1 / 12.1, 14.1 / 12.0, 14.7 / 14.3,
    // 13.6 / 14.8; 30 M 14.9 / 12.1, 16.4 / 11.7, 14.6 / 13.2, 14.9 / 16.1; 40 M 15.9 / 11.9, 16.2 / 11.4, 18.1 / 13.0, 20.7 / 14.8;
    // 64 M 22.2 / 14.9, 21.4 / 14.0, 23.1 / 15.2, 21.0 / 15.9.  (7.7 M with 26 K 11.9 / 10.1, with 426 K 11.8 / 14.8.)
    const bool most = !summary && ctx->N > int64_t(1) << (ctx->max_nnz > 65536 ? 25 : 24);
    const unsigned grid = (unsigned)div_up(words, kThreads * (most ? 8 : many ? 4 : 1));
    const auto kernel = summary ? (many ? k_cold_rank<true, 4> : k_cold_rank<true, 1>)
                                : (most ? k_cold_rank<false, 8> : many ? k_cold_rank<false, 4> : k_cold_rank<false, 1>);
    const WaitCfg w = wait_cfg(ctx);
    HL_CUDA_TRY(launch(kernel, grid, kThreads, stream, marks, (int)words, stage_rows, d_cold_rows, d_n_cold, r.status,
                       w.max_polls, w.stall_tile, clear, n_clear));
    note_launches(1);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

// the host table as the movers see it: `host_table` itself, or the per-table allocations installed by
// hl_set_host_tables (then `host_table` only says that there is a table)
static TableMap table_map(const hl_ctx* ctx, const float* host_table) {
    TableMap m;
    m.single = reinterpret_cast<unsigned char*>(const_cast<float*>(host_table));
    m.ptrs = ctx->per_table ? ctx->r.table_ptrs : nullptr;
    m.base = ctx->r.table_base;
    m.T = ctx->T;
    return m;
}

bool in_device_memory(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) == cudaSuccess) return at.type == cudaMemoryTypeDevice;
    (void)cudaGetLastError();
    return false;
}

// how the movers of this context are launched: beside the kernels of other mini-batches (`width` = the context's setting),
// or alone on the chip (`alone`, for the table they move to or from)
static MoveCfg move_cfg(const hl_ctx* ctx, int width, bool in_schedule = false, bool reads = false,
                        const float* alone = nullptr) {
    MoveCfg c;
    c.sms = ctx_sms(ctx);
    c.link_alone = alone && !(ctx->per_table ? ctx->tables_on_device != 0 : in_device_memory(alone));
    c.min_ctas = width > 0 ? width : 2 * c.sms;
    c.paced_ctas = in_schedule ? (ctx->mover_width_set ? width : kPacedCtas) : 0;
    c.paced_more = in_schedule && reads && !ctx->mover_width_set ? kReadCtasDefault : c.paced_ctas;
    c.max_polls = ctx->test_poll_limit > 0 ? ctx->test_poll_limit : kBulkMaxPolls;
    c.stall = ctx->test_poll_limit > 0 && ctx->test_stall_tile >= 0;
    return c;
}

int32_t launch_gather_rows(hl_ctx* ctx, float* dst, int64_t dst_row0, const float* table, const int32_t* rows,
                           const int64_t* d_n, int64_t n_max, int32_t* status, cudaStream_t stream) {
    // loading the hot cache happens with nothing else on the chip
    return launch_move_rows<false>(dst, dst_row0, table_map(ctx, table), rows, d_n, n_max, ctx->N, ctx->D, nullptr,
                                   move_cfg(ctx, 0, false, true, table), status, stream);
}

}  // namespace hl

using namespace hl;

namespace hl {
namespace {

// Shared body of hl_gather_cold and hl_gather_cold_ahead.  Staging window: cache slots
// [hot_cap + stage_row0, hot_cap + stage_row0 + stage_rows).
// First half of the cold-row search: classify X's lookups, rank the rows they mark, assign the slots.
int32_t index_begin(hl_ctx* ctx, hl_ubatch* non, const int32_t* d_n_non, int64_t stage_row0, int64_t stage_rows,
                    int32_t* d_cold_rows, int64_t* d_n_cold, cudaStream_t stream) {
    Regions& r = ctx->r;
    if (ctx->max_nnz == 0) {
        HL_CUDA_TRY(clear_words(reinterpret_cast<uint32_t*>(d_n_cold), 2, stream));
        return HL_OK;
    }
    if (!non->ids) return HL_EINVAL;
    const int32_t fresh = marks_fresh(ctx, stream);
    if (fresh != HL_OK) return fresh;
    const int grid = grid_for(ctx->max_nnz, kThreads, 4 * ctx_sms(ctx));
    HL_CUDA_TRY(launch(k_cold_classify, grid, kThreads, stream, non->ids, non->offsets, d_n_non, ctx->max_batch,
                       ctx->T * ctx->S, non->cap_ids, ctx->N, BitmapProbe{r.remap}, cold_marks(ctx), r.status));
    const int32_t st = cold_rank(ctx, stage_rows, d_cold_rows, d_n_cold, stream);
    if (st != HL_OK) return st;
    HL_CUDA_TRY(launch(k_cold_assign, grid, kThreads, stream, non->ids, non->offsets, d_n_non, ctx->max_batch,
                       ctx->T * ctx->S, non->cap_ids, r.cold_ranked, ctx->hot_cap + stage_row0, stage_rows));
    note_launches(2);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

// Second half: the match against the previous mini-batch's cold rows.
int32_t index_end(hl_ctx* ctx, int64_t stage_rows, int32_t* d_cold_rows, int64_t* d_n_cold,
                  const int32_t* d_prev_rows, const int64_t* d_n_prev, int32_t* d_fwd_src, cudaStream_t stream) {
    if (ctx->max_nnz == 0) return HL_OK;
    if (d_prev_rows) {
        HL_CUDA_TRY(launch(k_cold_match, grid_for(stage_rows, kThreads, 2 * ctx_sms(ctx)), kThreads, stream, d_cold_rows,
                           d_n_cold, stage_rows, d_prev_rows, d_n_prev, ctx->staging_cap, d_fwd_src));
        note_launches(1);
        HL_LAUNCH_CHECK();
    }
    return HL_OK;
}

int32_t gather_impl(hl_ctx* ctx, hl_ubatch* non, const int32_t* d_n_non, const float* host_table, float* d_cache,
                    int64_t stage_row0, int64_t stage_rows, int32_t* d_cold_rows, int64_t* d_n_cold,
                    const int32_t* d_prev_rows, const int64_t* d_n_prev, int32_t* d_fwd_src,
                    cudaEvent_t record_after_index, cudaEvent_t wait_a, cudaEvent_t wait_b, bool do_index,
                    bool do_move, cudaStream_t stream) {
    Regions& r = ctx->r;
    LaunchBatch batch(kept_launches(ctx));
    if (!do_index) {
        if (ctx->max_nnz == 0) return HL_OK;
        timer_mark(ctx, HL_TIMER_GATHER_MOVE, 0, stream);
        const int32_t st = launch_move_rows<false>(d_cache, ctx->hot_cap + stage_row0,
                                                   table_map(ctx, host_table), d_cold_rows, d_n_cold, stage_rows,
                                                   ctx->N, ctx->D, d_fwd_src, move_cfg(ctx, ctx->mover_ctas, true, true),
                                                   r.status, stream);
        timer_mark(ctx, HL_TIMER_GATHER_MOVE, 1, stream);
        return batch.end(st);
    }
    int32_t st = index_begin(ctx, non, d_n_non, stage_row0, stage_rows, d_cold_rows, d_n_cold, stream);
    if (st != HL_OK) return st;
    st = index_end(ctx, stage_rows, d_cold_rows, d_n_cold, d_prev_rows, d_n_prev, d_fwd_src, stream);
    if (st != HL_OK) return st;
    if (record_after_index || wait_a || wait_b) HL_CUDA_TRY(launch_flush());
    if (record_after_index) HL_CUDA_TRY(cudaEventRecord(record_after_index, stream));
    if (!do_move) return batch.end();
    if (wait_a) HL_CUDA_TRY(cudaStreamWaitEvent(stream, wait_a, 0));
    if (wait_b) HL_CUDA_TRY(cudaStreamWaitEvent(stream, wait_b, 0));
    timer_mark(ctx, HL_TIMER_GATHER_MOVE, 0, stream);
    st = launch_move_rows<false>(d_cache, ctx->hot_cap + stage_row0, table_map(ctx, host_table), d_cold_rows,
                                 d_n_cold, stage_rows, ctx->N, ctx->D, d_prev_rows ? d_fwd_src : nullptr,
                                 move_cfg(ctx, ctx->mover_ctas), r.status, stream);
    timer_mark(ctx, HL_TIMER_GATHER_MOVE, 1, stream);
    return batch.end(st);
}

bool window_ok(const hl_ctx* ctx, int64_t row0, int64_t rows) {
    return row0 >= 0 && rows >= 0 && row0 + rows <= ctx->staging_cap;
}

}  // namespace
}  // namespace hl

extern "C" int32_t hl_gather_cold(hl_ctx* ctx, hl_ubatch* non, const int32_t* d_n_non, const float* host_table,
                                  float* d_cache, int32_t* d_cold_rows, int64_t* d_n_cold, void* stream_) {
    if (!ctx || !non || !non->offsets || !d_n_non || !host_table || !d_cache || !d_cold_rows || !d_n_cold)
        return HL_EINVAL;
    return scratch_kept(ctx, gather_impl(ctx, non, d_n_non, host_table, d_cache, 0, ctx->staging_cap, d_cold_rows, d_n_cold,
                                       nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, true, true,
                                       static_cast<cudaStream_t>(stream_)));
}

extern "C" int32_t hl_gather_cold_ahead(hl_ctx* ctx, hl_ubatch* non, const int32_t* d_n_non, const float* host_table,
                                        float* d_cache, int64_t stage_row0, int64_t stage_rows, int32_t* d_cold_rows,
                                        int64_t* d_n_cold, const int32_t* d_prev_cold_rows, const int64_t* d_n_prev,
                                        int32_t* d_fwd_src, void* record_after_index, void* wait_before_move_a,
                                        void* wait_before_move_b, void* stream_) {
    if (!ctx || !non || !non->offsets || !d_n_non || !host_table || !d_cache || !d_cold_rows || !d_n_cold)
        return HL_EINVAL;
    if (!window_ok(ctx, stage_row0, stage_rows)) return HL_EINVAL;
    if ((d_prev_cold_rows != nullptr) != (d_n_prev != nullptr) || (d_prev_cold_rows && !d_fwd_src)) return HL_EINVAL;
    return scratch_kept(ctx, gather_impl(ctx, non, d_n_non, host_table, d_cache, stage_row0, stage_rows, d_cold_rows, d_n_cold,
                                       d_prev_cold_rows, d_n_prev, d_fwd_src,
                                       static_cast<cudaEvent_t>(record_after_index),
                                       static_cast<cudaEvent_t>(wait_before_move_a),
                                       static_cast<cudaEvent_t>(wait_before_move_b), true, true,
                                       static_cast<cudaStream_t>(stream_)));
}

extern "C" int32_t hl_index_cold(hl_ctx* ctx, hl_ubatch* non, const int32_t* d_n_non, int64_t stage_row0,
                                 int64_t stage_rows, int32_t* d_cold_rows, int64_t* d_n_cold,
                                 const int32_t* d_prev_cold_rows, const int64_t* d_n_prev, int32_t* d_fwd_src,
                                 void* stream_) {
    if (!ctx || !non || !non->offsets || !d_n_non || !d_cold_rows || !d_n_cold) return HL_EINVAL;
    if (!window_ok(ctx, stage_row0, stage_rows)) return HL_EINVAL;
    if ((d_prev_cold_rows != nullptr) != (d_n_prev != nullptr) || (d_prev_cold_rows && !d_fwd_src)) return HL_EINVAL;
    return scratch_kept(ctx, gather_impl(ctx, non, d_n_non, nullptr, nullptr, stage_row0, stage_rows, d_cold_rows, d_n_cold,
                                       d_prev_cold_rows, d_n_prev, d_fwd_src, nullptr, nullptr, nullptr, true, false,
                                       static_cast<cudaStream_t>(stream_)));
}

extern "C" int32_t hl_index_cold_begin(hl_ctx* ctx, hl_ubatch* non, const int32_t* d_n_non, int64_t stage_row0,
                                       int64_t stage_rows, int32_t* d_cold_rows, int64_t* d_n_cold, void* stream_) {
    if (!ctx || !non || !non->offsets || !d_n_non || !d_cold_rows || !d_n_cold) return HL_EINVAL;
    if (!window_ok(ctx, stage_row0, stage_rows)) return HL_EINVAL;
    LaunchBatch batch(kept_launches(ctx));
    return scratch_kept(ctx, batch.end(index_begin(ctx, non, d_n_non, stage_row0, stage_rows, d_cold_rows, d_n_cold,
                                                 static_cast<cudaStream_t>(stream_))));
}

extern "C" const int32_t* hl_index_cold_verdict(hl_ctx* ctx) { return ctx ? ctx->r.cold_n + 1 : nullptr; }

extern "C" int32_t hl_index_cold_end(hl_ctx* ctx, hl_ubatch* non, int64_t stage_row0, int64_t stage_rows,
                                     int32_t* d_cold_rows, int64_t* d_n_cold, const int32_t* d_prev_cold_rows,
                                     const int64_t* d_n_prev, int32_t* d_fwd_src, int32_t general_not_needed,
                                     void* stream_) {
    if (!ctx || !non || !d_cold_rows || !d_n_cold) return HL_EINVAL;
    if (!window_ok(ctx, stage_row0, stage_rows)) return HL_EINVAL;
    if ((d_prev_cold_rows != nullptr) != (d_n_prev != nullptr) || (d_prev_cold_rows && !d_fwd_src)) return HL_EINVAL;
    (void)general_not_needed;
    return index_end(ctx, stage_rows, d_cold_rows, d_n_cold, d_prev_cold_rows, d_n_prev, d_fwd_src,
                     static_cast<cudaStream_t>(stream_));
}

extern "C" int32_t hl_stage_cold(hl_ctx* ctx, const float* host_table, float* d_cache, int64_t stage_row0,
                                 int64_t stage_rows, const int32_t* d_cold_rows, const int64_t* d_n_cold,
                                 const int32_t* d_fwd_src, void* stream_) {
    if (!ctx || !host_table || !d_cache || !d_cold_rows || !d_n_cold) return HL_EINVAL;
    if (!window_ok(ctx, stage_row0, stage_rows)) return HL_EINVAL;
    return gather_impl(ctx, nullptr, nullptr, host_table, d_cache, stage_row0, stage_rows,
                       const_cast<int32_t*>(d_cold_rows), const_cast<int64_t*>(d_n_cold), nullptr, nullptr,
                       const_cast<int32_t*>(d_fwd_src), nullptr, nullptr, nullptr, false, true,
                       static_cast<cudaStream_t>(stream_));
}

extern "C" int32_t hl_forward_cold(hl_ctx* ctx, float* d_cache, int64_t from_stage_row0, int64_t to_stage_row0,
                                   int64_t stage_rows, const int32_t* d_fwd_src, const int64_t* d_n_cold,
                                   void* stream_) {
    if (!ctx || !d_cache || !d_fwd_src || !d_n_cold) return HL_EINVAL;
    if (!window_ok(ctx, from_stage_row0, stage_rows) || !window_ok(ctx, to_stage_row0, stage_rows)) return HL_EINVAL;
    if (stage_rows == 0) return HL_OK;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const int D4 = ctx->D / 4;
    const int grid = 2 * ctx_sms(ctx);
    const int64_t from = ctx->hot_cap + from_stage_row0, to = ctx->hot_cap + to_stage_row0;
    if (D4 <= 4) HL_CUDA_TRY(launch(k_forward_rows<4>, grid, kThreads, stream, d_cache, from, to, d_fwd_src, d_n_cold,
                                    stage_rows, D4));
    else if (D4 <= 8) HL_CUDA_TRY(launch(k_forward_rows<8>, grid, kThreads, stream, d_cache, from, to, d_fwd_src, d_n_cold,
                                         stage_rows, D4));
    else if (D4 <= 16) HL_CUDA_TRY(launch(k_forward_rows<16>, grid, kThreads, stream, d_cache, from, to, d_fwd_src,
                                          d_n_cold, stage_rows, D4));
    else HL_CUDA_TRY(launch(k_forward_rows<32>, grid, kThreads, stream, d_cache, from, to, d_fwd_src, d_n_cold, stage_rows,
                            D4));
    note_launches(1);
    HL_LAUNCH_CHECK();
    return HL_OK;
}

static int32_t scatter_call(hl_ctx* ctx, const float* d_cache, int64_t stage_row0, int64_t stage_rows,
                            const int32_t* d_cold_rows, const int64_t* d_n_cold, float* host_table, bool in_schedule,
                            void* stream_) {
    if (!ctx || !d_cache || !d_cold_rows || !d_n_cold || !host_table) return HL_EINVAL;
    if (!window_ok(ctx, stage_row0, stage_rows)) return HL_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    LaunchBatch batch(kept_launches(ctx));
    timer_mark(ctx, HL_TIMER_SCATTER_MOVE, 0, stream);
    const int32_t st = launch_move_rows<true>(const_cast<float*>(d_cache), ctx->hot_cap + stage_row0,
                                              table_map(ctx, host_table),
                                              d_cold_rows, d_n_cold, stage_rows, ctx->N, ctx->D, nullptr,
                                              move_cfg(ctx, ctx->scatter_ctas, in_schedule), ctx->r.status, stream);
    timer_mark(ctx, HL_TIMER_SCATTER_MOVE, 1, stream);
    return batch.end(st);
}

extern "C" int32_t hl_scatter_cold_at(hl_ctx* ctx, const float* d_cache, int64_t stage_row0, int64_t stage_rows,
                                      const int32_t* d_cold_rows, const int64_t* d_n_cold, float* host_table,
                                      void* stream) {
    return scatter_call(ctx, d_cache, stage_row0, stage_rows, d_cold_rows, d_n_cold, host_table, true, stream);
}

extern "C" int32_t hl_scatter_cold(hl_ctx* ctx, const float* d_cache, const int32_t* d_cold_rows,
                                   const int64_t* d_n_cold, float* host_table, void* stream_) {
    if (!ctx) return HL_EINVAL;
    // (one mini-batch after the other: nothing runs beside this)
    return scatter_call(ctx, d_cache, 0, ctx->staging_cap, d_cold_rows, d_n_cold, host_table, false, stream_);
}

extern "C" int32_t hl_flush_hot(hl_ctx* ctx, const float* d_cache, const int32_t* d_hot_rows, const int64_t* d_n_hot,
                                float* host_table, void* stream_) {
    if (!ctx || !d_cache || !d_hot_rows || !d_n_hot || !host_table) return HL_EINVAL;
    // runs between learning phases, with nothing else on the chip
    return launch_move_rows<true>(const_cast<float*>(d_cache), 0, table_map(ctx, host_table), d_hot_rows, d_n_hot,
                                  ctx->hot_cap, ctx->N,
                                  ctx->D, nullptr, move_cfg(ctx, 0, false, false, host_table), ctx->r.status,
                                  static_cast<cudaStream_t>(stream_));
}
