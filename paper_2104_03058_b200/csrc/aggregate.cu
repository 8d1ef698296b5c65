// Chunked gather-aggregate for GCN and GraphSAGE (Algorithm 1: Message + Aggregate per decomposition
// layer, Concat by writing each chunk into its own output columns) and the second-level reduction
// of hub rows.
//
// Work decomposition.  One launch sweeps the chunks one after the other (the block index is
// chunk-major), so at any time the blocks in flight gather from one chunk's n x chunk_width slice of
// x, which is what keeps the gathered working set small enough for L2.  Inside a sweep the rows come
// grouped by degree class.  A row is owned by S = LPR * EP lanes: LPR lanes cover the chunk's columns
// with one to three 16-byte vectors each, and EP groups of LPR lanes walk interleaved entries of the
// row, each keeping 8 loads in flight (6 with three vectors); column indices and edge weights are staged per warp in shared
// memory.  The EP partial sums are combined by a fixed shuffle tree, the parts of a long row that several warps share by shared
// memory, first warp to last, hub rows (degree > GNNFD_HUB_DEGREE) by per-segment partial sums that a second kernel adds in
// ascending segment order: no atomics, bit-identical from run to run.
#include "schedule.cuh"
#include "vec.cuh"

namespace gnnfd {

struct GatherArgs {
    const int32_t* row_ptr;
    const int32_t* col_idx;
    const float* edge_w;
    const float* rdeg;
    const int32_t* row_order;
    const int32_t* seg_row;
    const int32_t* seg_begin;
    const int32_t* seg_end;
    const int32_t* seg_slot;
    const void* x;
    void* out;
    float* partial;
    int64_t ldx, ldo;
    int32_t f, chunk_width, n_ctiles, blocks_per_tile, fpad, out_bf16, out_vec_ok, wide_ok;
    int32_t part_filled;     // some lanes' vectors lie past the end of the chunk
    int32_t chunk_base;      // first chunk of this launch (a launch covers at most 65,535 chunks)
    int32_t n_ranges;
    Range range[kMaxRanges];
};

#ifndef GNNFD_GATHER_LOADS
#define GNNFD_GATHER_LOADS 8
#endif
constexpr int kLoads = GNNFD_GATHER_LOADS;      // 16-byte feature loads kept in flight per lane

// index registers per lane and batch, and the column indices (and weights) a warp stages per batch
constexpr int index_regs(int lpr, int vpl) { return kLoads / vpl > lpr ? kLoads / vpl / lpr : 1; }
constexpr int stage_slots(int lpr, int vpl, bool roomy) { return roomy ? 256 : 32 * index_regs(lpr, vpl); }

// fp32 chunks of 9 - 16 vectors on graphs that fill the chip take rows from the shortest of a class up and, oddly, gain from a
// smaller L1 beside 40 instead of 12 KB of shared memory per block.  132,534 rows of 300 entries, 64 columns: longest first
// 583 us, shortest first 567, with both 564; 304 columns in chunks of 64 3.15 / 3.03 / 3.04 ms; 60,000 of 200, 128 in chunks of 64 378 / 373 / 366 us.
// All other widths are the same or up to 5 % faster longest first, bf16 ones too.
constexpr bool shortest_first(int elem_bytes, int vecn, int lpr, int vpl, bool shared)
{
    return elem_bytes == 4 && vecn == 4 && lpr == 8 && vpl == 2 && !shared;
}

// Blocks per SM that the registers are shared out for.  Four where the loop fits 64 registers without giving up loads in flight: rows are
// bound by waiting for the loads of their own chain, and more of them wait side by side.  Three / four blocks: SAGE fp32, 100,000 rows of
// 20 entries, 128 columns in chunks of 64 96 -> 86 us, 200,000 of 16, 64 columns 90 -> 76, 32 39 -> 32, RMAT 2^19, 64 columns 368 -> 315; GCN fp32
// without split rows, 41 columns on 132,534 rows of 300 542 -> 515, 304 in chunks of 64 371 -> 348, 32 on 233,000 of 86 211 -> 190.  But wider
// rows lose: GCN of 144 / 256 columns 214 -> 228 / 240 -> 277, SAGE of 256 on 20,000 rows of 50 59 -> 65; so do split rows of GCN (64 columns 28 -> 31)
// and bf16 (SAGE of 64 / 256 columns 35 -> 41 / 130 -> 151, GCN of 64 on RMAT 2^21 1487 -> 1832).  Chunks of 65 - 96 fp32 columns, three vectors
// per lane, too: 72 / 96 columns SAGE on 200,000 rows of 16 105 -> 91 / 113 -> 98, on 132,534 of 300 728 -> 692 / 768 -> 726, GCN there 770 -> 760 / 788 -> 785.
// Spilled at 64 registers, outside the loop over entries: 4 - 32 bytes of <4, 8, 3> and <4, 2, 2> SAGE, 24 - 56 of <4, 8, 2>, <4, 2, 2> and <4, 8, 3> GCN.
constexpr int min_blocks(int elem_bytes, bool weighted, bool shared, int lpr)
{
    return elem_bytes == 4 && lpr <= 8 && !(weighted && shared) ? 4 : 3;
}

// One row (or hub segment) per S = LPR * EP lanes.  The S lanes fetch the row's indices and weights
// S at a time with one coalesced streaming load each (R rounds per batch) and stage them in the
// warp's shared-memory buffer (double-buffered; the next batch is already in registers, on its way
// from HBM, while this one is consumed).  In step s of a batch, group g works on entry
// r*S + t*EP + g (r = s / LPR, t = s % LPR), read back as a broadcast.  A lane covers VPL vectors of the
// chunk (columns c + q*LPR, q < VPL, in vector units) so that the index traffic, the address
// arithmetic and the shuffles are paid once per VPL * 16 gathered bytes.
// The thread's second-level sums live in shared memory as tot_s[k][thread]; with a multiple of four sums
// they are moved four at a time (tot_s is then indexed as float4 rows of the same array).
template <int NV, bool ZERO_ACC>
__device__ __forceinline__ void second_level(float (*tot_s)[kBlock], int tid, float* acc, int mode /*0 clear, 1 add acc, 2 fetch, 3 set to acc*/)
{
    if constexpr (NV % 4 == 0) {
        float4* t4 = reinterpret_cast<float4*>(&tot_s[0][0]) + tid;          // element k4 of the thread: t4[k4 * kBlock]
#pragma unroll
        for (int k4 = 0; k4 < NV / 4; ++k4) {
            float4& slot = t4[k4 * kBlock];
            if (mode == 0) {
                slot = make_float4(0.f, 0.f, 0.f, 0.f);
            } else if (mode == 3) {
                slot = make_float4(acc[4 * k4], acc[4 * k4 + 1], acc[4 * k4 + 2], acc[4 * k4 + 3]);
            } else if (mode == 1) {
                float4 v = slot;
                v.x += acc[4 * k4]; v.y += acc[4 * k4 + 1]; v.z += acc[4 * k4 + 2]; v.w += acc[4 * k4 + 3];
                slot = v;
                if (ZERO_ACC) acc[4 * k4] = acc[4 * k4 + 1] = acc[4 * k4 + 2] = acc[4 * k4 + 3] = 0.f;
            } else {
                const float4 v = slot;
                acc[4 * k4] += v.x; acc[4 * k4 + 1] += v.y; acc[4 * k4 + 2] += v.z; acc[4 * k4 + 3] += v.w;
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            if (mode == 0) tot_s[k][tid] = 0.f;
            else if (mode == 3) tot_s[k][tid] = acc[k];
            else if (mode == 1) { tot_s[k][tid] += acc[k]; if (ZERO_ACC) acc[k] = 0.f; }
            else acc[k] += tot_s[k][tid];
        }
    }
}

template <typename T, int VECN, int LPR, int VPL, bool WEIGHTED, bool SHARED, bool WIDE, int EP, int SLOTS>
__device__ __forceinline__ void gather_rows(const GatherArgs& a, const Range& rg, int block_in_range, int col0,
                                            int chunk_end, int32_t (*stage_col)[kBlock / 32][SLOTS], float (*stage_w)[kBlock / 32][SLOTS],
                                            float (*tot_s)[kBlock])
{
    constexpr int S = LPR * EP;
    constexpr int ROWS = kBlock / S;
    constexpr int UB = kLoads / VPL;                      // steps whose loads are issued together
    constexpr int R = index_regs(LPR, VPL);
    constexpr int SPB = R * LPR;                          // steps per batch
    constexpr int EPB = R * S;                            // entries per batch
    constexpr unsigned kFull = 0xffffffffu;
    const int tid = threadIdx.x;
    const int group = tid / S;
    const int sl = tid % S;
    const int g = sl / LPR;
    const int c = sl % LPR;
    const int warp = tid >> 5, lane = tid & 31;
    const int seg = lane - sl;                   // first lane of this row's segment inside the warp

    int jq[VPL];
    bool okq[VPL];
    const T* xq[VPL];
    // A vector past the end of the chunk re-reads the chunk's last vector (or pair of them), which a neighbour reads in the same
    // instruction.  The L1's lookups bound rows that end inside a line (88 % busy): with the chunk's first column in its place, 41 columns (11 of
    // 16 vectors) on 132,534 rows of 300 entries looked up two lines where one was needed, 622 -> 542 us; 48 on 60,000 rows 295 -> 260.
    const int last = col0 + (chunk_end - 1 - col0) / (WIDE ? VPL * VECN : VECN) * (WIDE ? VPL * VECN : VECN);
#pragma unroll
    for (int q = 0; q < VPL; ++q) {
        // with 32-byte loads a lane's two vectors are neighbours, otherwise they lie LPR vectors apart
        jq[q] = col0 + (WIDE ? c * VPL + q : c + q * LPR) * VECN;
        okq[q] = jq[q] < chunk_end;
        xq[q] = static_cast<const T*>(a.x) + (okq[q] ? jq[q] : last);
    }
    // Pair loads are for all lanes or none: a lane whose second vector, or both, lie past the chunk's end loads a pair all the
    // same (padding of its own row, or the chunk's last pair) and drops it.  With a branch per lane, rows of 5 and 7 vectors took
    // both sides of it: 116 M entries of 20 / 25 fp32 columns 1.58 / 1.59 -> 0.90 / 0.93 ms, of 48 bf16 columns 1.56 -> 1.19.
    // For weighted bf16 sums the test stays in the code (full chunks: no lane fails it): without it the loads are scheduled differently
    // and 64 columns on 2 M RMAT rows take 1.61 instead of 1.50 ms.  Unweighted ones are faster without it: 32 / 48 / 64 columns
    // there 1003 / 1471 / 1452 -> 883 / 1419 / 1396 us.
    const bool pairs = sizeof(T) == 4 || !WEIGHTED || okq[VPL - 1] || a.part_filled;
    const uint32_t ld = (uint32_t)a.ldx;

    // a long row may be shared by several warps of the block, which take consecutive parts of it
    const int warps_log2 = SHARED && S == 32 ? rg.warps_log2 : 0, sharer = group & ((1 << warps_log2) - 1);
    const int slot = block_in_range * (ROWS >> warps_log2) + (group >> warps_log2);
    const bool active = slot < rg.item_count;
    int32_t row = 0, b = 0, e = 0, part = 0;      // part: where a hub segment's partial sums go
    if (active) {
        if (rg.hub) {
            row = a.seg_row[slot];
            b = a.seg_begin[slot];
            e = a.seg_end[slot];
            part = a.seg_slot[slot];
        } else {
            row = a.row_order[rg.item_first + rg.item_step * slot];
            b = a.row_ptr[row];
            e = a.row_ptr[row + 1];
        }
    }
    if (SHARED && S == 32 && warps_log2 > 0) {
        const int32_t share = ((e - b) >> warps_log2) + 1;
        b = min(b + sharer * share, e);
        e = min(b + share, e);
    }
    int32_t ucur[R];
    float wcur[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int32_t kk = b + r * S + sl;
        const bool ok = kk < e;
        ucur[r] = ok ? __ldcs(a.col_idx + kk) : -1;
        wcur[r] = (WEIGHTED && ok) ? __ldcs(a.edge_w + kk) : 0.f;
    }

    // Two levels of accumulation: `acc` takes at most kChain products in a row, then moves into the
    // thread's second-level sums (kept in shared memory, they cost no registers), so that no fp32 chain
    // of a lane is longer than kChain + (entries of the lane) / kChain terms.  Long runs of equal-sign
    // terms (a hub row fed by one source many times) otherwise drift by half an ulp per term.
    constexpr int kChain = 64;
    constexpr int FLUSH = SPB >= kChain ? 1 : kChain / SPB;      // batches between two moves
    float acc[VPL][VECN];
#pragma unroll
    for (int q = 0; q < VPL; ++q)
#pragma unroll
        for (int i = 0; i < VECN; ++i) acc[q][i] = 0.f;

    const int n_batches = __reduce_max_sync(kFull, (e - b + EPB - 1) / EPB);     // the warp loops together
    const bool two_level = n_batches > FLUSH;                                    // short rows never leave the first level
    if (two_level) second_level<VPL * VECN, true>(tot_s, tid, &acc[0][0], 0);

    for (int ib = 0; ib < n_batches; ++ib) {
        const int32_t kb = b + ib * EPB;
        // the next batch's indices are requested before this batch's gathers are consumed
        int32_t unext[R];
        float wnext[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int32_t kk = kb + EPB + r * S + sl;
            const bool ok = kk < e;
            unext[r] = ok ? __ldcs(a.col_idx + kk) : -1;
            wnext[r] = (WEIGHTED && ok) ? __ldcs(a.edge_w + kk) : 0.f;
        }
        const bool full = __all_sync(kFull, kb + EPB <= e);
        const int buf = ib & 1;
        if (LPR > 1) {      // with one lane per row every lane consumes exactly the entries it fetched
#pragma unroll
            for (int r = 0; r < R; ++r) {
                stage_col[buf][warp][r * 32 + lane] = ucur[r];
                if (WEIGHTED) stage_w[buf][warp][r * 32 + lane] = wcur[r];
            }
            __syncwarp();
        }
        auto consume = [&](const Vec<T, VECN> (&v)[UB][VPL], const float (&wv)[UB]) {
#pragma unroll
            for (int i = 0; i < UB; ++i)
#pragma unroll
                for (int q = 0; q < VPL; ++q)
#pragma unroll
                    for (int k = 0; k < VECN; ++k) {
                        if constexpr (!WEIGHTED && sizeof(T) == 2 && VECN > 1) {
                            if (k % 2 == 0) add_widened(acc[q][k], acc[q][k + 1], v[i][q].word(k / 2));
                        } else if (WEIGHTED) acc[q][k] = fmaf(wv[i], v[i][q].get(k), acc[q][k]);
                        else acc[q][k] += v[i][q].get(k);
                    }
        };
        if (full) {
            // every lane has all of the batch's entries: straight-line code, no tests
#pragma unroll
            for (int s0 = 0; s0 < SPB; s0 += UB) {
                Vec<T, VECN> v[UB][VPL];
                float wv[UB];
#pragma unroll
                for (int i = 0; i < UB; ++i) {
                    const int r = (s0 + i) / LPR, tt = (s0 + i) % LPR;
                    const int32_t u = LPR > 1 ? stage_col[buf][warp][r * 32 + seg + tt * EP + g] : ucur[r];
                    if (WEIGHTED) wv[i] = LPR > 1 ? stage_w[buf][warp][r * 32 + seg + tt * EP + g] : wcur[r];
                    const size_t off = (size_t)(uint32_t)u * ld;
                    if (WIDE && pairs) {
                        load_pair(v[i][0], v[i][VPL - 1], xq[0] + off);
                    } else {
#pragma unroll
                        for (int q = 0; q < VPL; ++q) v[i][q].load(xq[q] + off);
                    }
                }
                consume(v, wv);
            }
        } else {
            // A ragged batch.  Step s works on entries s * EP .. of a row's batch, so the steps past the longest
            // remainder in the warp have nothing to do for any lane (a row of 3 entries in a class whose batch
            // holds 16 would otherwise pay for 16).
            const int rem = __reduce_max_sync(kFull, e - kb);
#pragma unroll
            for (int s0 = 0; s0 < SPB; s0 += UB) {
                if (s0 > 0 && s0 * EP >= rem) break;
                Vec<T, VECN> v[UB][VPL];
                float wv[UB];
#pragma unroll
                for (int i = 0; i < UB; ++i) {
                    const int r = (s0 + i) / LPR, tt = (s0 + i) % LPR;
                    const int32_t u = LPR > 1 ? stage_col[buf][warp][r * 32 + seg + tt * EP + g] : ucur[r];
                    if (WEIGHTED) wv[i] = LPR > 1 ? stage_w[buf][warp][r * 32 + seg + tt * EP + g] : wcur[r];
                    const size_t off = (size_t)(uint32_t)max(u, 0) * ld;
                    if (WIDE && pairs) {
                        if (u >= 0) load_pair(v[i][0], v[i][VPL - 1], xq[0] + off);
                        else { v[i][0].zero(); v[i][VPL - 1].zero(); }
                    } else {
#pragma unroll
                        for (int q = 0; q < VPL; ++q) {
                            if (u >= 0) v[i][q].load(xq[q] + off);
                            else v[i][q].zero();
                        }
                    }
                }
                consume(v, wv);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) { ucur[r] = unext[r]; wcur[r] = wnext[r]; }
        if (two_level && (ib + 1) % FLUSH == 0) second_level<VPL * VECN, true>(tot_s, tid, &acc[0][0], 1);
    }
    if (two_level) second_level<VPL * VECN, true>(tot_s, tid, &acc[0][0], 2);

    // fixed-order combination of the EP partial sums of the row
#pragma unroll
    for (int o = S / 2; o >= LPR; o >>= 1)
#pragma unroll
        for (int q = 0; q < VPL; ++q)
#pragma unroll
            for (int i = 0; i < VECN; ++i) acc[q][i] += __shfl_down_sync(kFull, acc[q][i], o, S);

    if (SHARED && S == 32 && warps_log2 > 0) {                 // the sharers' sums, first to last; the whole block is on this side
        if (sharer > 0) second_level<VPL * VECN, false>(tot_s, tid, &acc[0][0], 3);
        __syncthreads();
        if (sharer > 0) return;
        for (int w = 1; w < 1 << warps_log2; ++w) second_level<VPL * VECN, false>(tot_s, tid + 32 * w, &acc[0][0], 2);
    }

    if (active && g == 0) {
        const float scale = (WEIGHTED || rg.hub) ? 1.f : a.rdeg[row];
#pragma unroll
        for (int q = 0; q < VPL; ++q) {
            if (!okq[q]) continue;
            const int j = jq[q];
            if (rg.hub) {
                float* p = a.partial + (int64_t)part * a.fpad + j;
#pragma unroll
                for (int i = 0; i < VECN; ++i)
                    if (j + i < chunk_end) p[i] = acc[q][i];
                continue;
            }
            const int64_t o = (int64_t)row * a.ldo + j;
            if (VECN % 4 == 0 && a.out_vec_ok && j + VECN <= chunk_end) {
#pragma unroll
                for (int i = 0; i < VECN; i += 4)
                    __stcs(reinterpret_cast<float4*>(static_cast<float*>(a.out) + o + i),
                           make_float4(acc[q][i] * scale, acc[q][i + 1] * scale, acc[q][i + 2] * scale, acc[q][i + 3] * scale));
            } else {
#pragma unroll
                for (int i = 0; i < VECN; ++i)
                    if (j + i < chunk_end) store_elem(a.out, a.out_bf16, o + i, acc[q][i] * scale);
            }
        }
    }
}

template <typename T, int VECN, int LPR, int VPL, bool WEIGHTED, bool SHARED, bool WIDE = false>
__global__ void __launch_bounds__(kBlock, min_blocks(sizeof(T), WEIGHTED, SHARED, LPR)) gather_aggregate(const __grid_constant__ GatherArgs a)
{
    grid_dependency<true>();
    constexpr int SLOTS = stage_slots(LPR, VPL, shortest_first(sizeof(T), VECN, LPR, VPL, SHARED));
    __shared__ int32_t stage_col[2][kBlock / 32][SLOTS];
    __shared__ float stage_w[2][kBlock / 32][SLOTS];
    __shared__ __align__(16) float tot_s[VPL * VECN][kBlock];   // second-level sums of every thread
    // grid: x = (block of the sweep, column tile), y = chunk; blocks are issued x first, so the sweeps follow each
    // other chunk by chunk.  (Dividing the chunk out of a linear 64-bit block number would take two 64-bit
    // divisions per thread, more instructions than a short row's whole walk.)
    const int chunk = a.chunk_base + (int)blockIdx.y;
    const unsigned n_ct = (unsigned)a.n_ctiles;
    const int rb = n_ct == 1 ? (int)blockIdx.x : (int)(blockIdx.x / n_ct);
    const int ctile = n_ct == 1 ? 0 : (int)(blockIdx.x % n_ct);
    const int chunk_begin = chunk * a.chunk_width;
    const int chunk_end = min(a.f, chunk_begin + a.chunk_width);
    const int col0 = chunk_begin + ctile * (LPR * VPL * VECN);
    if (col0 >= chunk_end) return;
    int r = 0;
#pragma unroll
    for (int i = 1; i < (SHARED ? kMaxRanges : kNumBins); ++i)      // unsplit, the fourth class is one range
        if (i < a.n_ranges && rb >= a.range[i].first_block) r = i;
    const Range rg = a.range[r];
    const int bir = rb - rg.first_block;
    switch (rg.ep_log2) {
        case 0: gather_rows<T, VECN, LPR, VPL, WEIGHTED, SHARED, WIDE, 1, SLOTS>(a, rg, bir, col0, chunk_end, stage_col, stage_w, tot_s); break;
        case 1: if constexpr (LPR * 2 <= 32) gather_rows<T, VECN, LPR, VPL, WEIGHTED, SHARED, WIDE, 2, SLOTS>(a, rg, bir, col0, chunk_end, stage_col, stage_w, tot_s); break;
        case 2: if constexpr (LPR * 4 <= 32) gather_rows<T, VECN, LPR, VPL, WEIGHTED, SHARED, WIDE, 4, SLOTS>(a, rg, bir, col0, chunk_end, stage_col, stage_w, tot_s); break;
        case 3: if constexpr (LPR * 8 <= 32) gather_rows<T, VECN, LPR, VPL, WEIGHTED, SHARED, WIDE, 8, SLOTS>(a, rg, bir, col0, chunk_end, stage_col, stage_w, tot_s); break;
        case 4: if constexpr (LPR * 16 <= 32) gather_rows<T, VECN, LPR, VPL, WEIGHTED, SHARED, WIDE, 16, SLOTS>(a, rg, bir, col0, chunk_end, stage_col, stage_w, tot_s); break;
        default: if constexpr (LPR == 1) gather_rows<T, VECN, LPR, VPL, WEIGHTED, SHARED, WIDE, 32, SLOTS>(a, rg, bir, col0, chunk_end, stage_col, stage_w, tot_s); break;
    }
}

// out[row, j] = scale * sum over the row's segments, ascending, of partial[segment, j]
__global__ void __launch_bounds__(kBlock)
hub_reduce(const int32_t* row_order, const int32_t* hub_seg_ptr, const float* rdeg,
           const float* partial, int64_t hub_begin, int32_t n_hub, int32_t f, int32_t fpad, int use_rdeg,
           void* __restrict__ out, int64_t ldo, int out_bf16)
{
    grid_dependency<true>();
    const int i = blockIdx.x;
    const int j = blockIdx.y * kBlock + threadIdx.x;
    if (i >= n_hub || j >= f) return;
    const int32_t row = row_order[hub_begin + i];
    const int32_t s0 = hub_seg_ptr[i], s1 = hub_seg_ptr[i + 1];
    // segment sums in ascending order, in runs of 32 so that a row of very many segments keeps short chains
    float acc = 0.f, run = 0.f;
    for (int32_t s = s0; s < s1; ++s) {
        run += partial[(int64_t)s * fpad + j];
        if (((s - s0) & 31) == 31) { acc += run; run = 0.f; }
    }
    acc += run;
    if (use_rdeg) acc *= rdeg[row];
    store_elem(out, out_bf16, (int64_t)row * ldo + j, acc);
}

// ------------------------------------------------------------------ host side

typedef void (*GatherKernel)(const GatherArgs);

template <typename T, int VECN, bool WEIGHTED, bool SHARED>
static GatherKernel pick_lpr(int lpr, int vpl, bool wide)
{
    if (vpl == 1) return gather_aggregate<T, VECN, 1, 1, WEIGHTED, SHARED>;
    if constexpr (VECN * sizeof(T) == 16) {
        if (wide) {          // narrow chunks whose vector pairs start on 32-byte boundaries
            switch (lpr) {
                case 1: return gather_aggregate<T, VECN, 1, 2, WEIGHTED, SHARED, true>;
                case 2: return gather_aggregate<T, VECN, 2, 2, WEIGHTED, SHARED, true>;
                default: return gather_aggregate<T, VECN, 4, 2, WEIGHTED, SHARED, true>;
            }
        }
    }
    if constexpr (VECN > 1) {
        if (vpl == 3) return lpr == 8 ? gather_aggregate<T, VECN, 8, 3, WEIGHTED, SHARED> : gather_aggregate<T, VECN, 16, 3, WEIGHTED, SHARED>;
    }
    switch (lpr) {
        case 1: return gather_aggregate<T, VECN, 1, 2, WEIGHTED, SHARED>;
        case 2: return gather_aggregate<T, VECN, 2, 2, WEIGHTED, SHARED>;
        case 4: return gather_aggregate<T, VECN, 4, 2, WEIGHTED, SHARED>;
        case 8: return gather_aggregate<T, VECN, 8, 2, WEIGHTED, SHARED>;
        case 16: return gather_aggregate<T, VECN, 16, 2, WEIGHTED, SHARED>;
        default: return gather_aggregate<T, VECN, 32, 2, WEIGHTED, SHARED>;
    }
}

template <bool WEIGHTED, bool SHARED>
static GatherKernel pick_kernel(gnnfd_dtype_t xdt, bool vec, int lpr, int vpl, bool wide)
{
    if (xdt == GNNFD_F32)
        return vec ? pick_lpr<float, 4, WEIGHTED, SHARED>(lpr, vpl, wide) : pick_lpr<float, 1, WEIGHTED, SHARED>(lpr, vpl, false);
    return vec ? pick_lpr<__nv_bfloat16, 8, WEIGHTED, SHARED>(lpr, vpl, wide) : pick_lpr<__nv_bfloat16, 1, WEIGHTED, SHARED>(lpr, vpl, false);
}

// ---- aligned copy of features whose rows or chunks do not start on 16-byte boundaries

// One 16-byte vector of the copy per thread: chunks of cw columns placed `pitch` columns apart, rows ld apart, zeros between.
template <typename T>
__global__ void __launch_bounds__(kBlock)
align_features(const T* x, int64_t ldx, int64_t n, int32_t f, int32_t cw, int32_t pitch, uint32_t ld, uint4* __restrict__ out)
{
    grid_dependency<true>();
    constexpr int VECN = 16 / sizeof(T);
    const uint32_t vectors = ld / VECN;
    const int64_t idx = (int64_t)blockIdx.x * kBlock + threadIdx.x;
    const int64_t row = idx <= 0xffffffffll ? (int64_t)((uint32_t)idx / vectors) : idx / vectors;
    if (row >= n) return;
    const int32_t at = (int32_t)(idx - row * vectors) * VECN;
    const int32_t chunk = at / pitch, in_chunk = at - chunk * pitch, j = chunk * cw + in_chunk;
    const int32_t count = min(f - j, cw - in_chunk);       // none in the padding
    const T* p = x + row * ldx + j;
    union { T e[VECN]; uint4 v; } u;
    u.v = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int i = 0; i < VECN; ++i)
        if (i < count) u.e[i] = p[i];
    out[idx] = u.v;
}

// Each row has to be gathered a few times, and the launch has to be won back within one chunk.  `per_entry` is what an entry of
// the chunk costs without the copy.
bool copy_pays(const gnnfd_csr_t* csr, int64_t per_entry, int64_t least)
{
    return csr->nnz >= 4 * csr->n && csr->nnz * per_entry >= least;
}

AlignedCopy layout_copy(int64_t n, gnnfd_dtype_t xdt, int32_t f, int32_t cw, int32_t unit_bytes, int32_t row_bytes)
{
    const int xsize = xdt == GNNFD_F32 ? 4 : 2, unit = unit_bytes / xsize, row_unit = row_bytes / xsize;
    const int64_t pitch = ((int64_t)cw + unit - 1) / unit * unit;
    const int64_t ld = ((f - 1) / cw * pitch + ((f - 1) % cw + unit) / unit * unit + row_unit - 1) / row_unit * row_unit;
    if (ld > 0x7fffffffll || n * ld > 0x7fffffffll * kBlock) return AlignedCopy{cw, f, 0};
    return AlignedCopy{(int32_t)pitch, ld, align_up((size_t)n * ld * xsize, 256)};
}

void launch_copy(const void* d_x, int64_t ldx, gnnfd_dtype_t xdt, int64_t n, int32_t f, int32_t cw, const AlignedCopy& copy,
                 void* d_aligned, cudaStream_t s)
{
    const int vecn = xdt == GNNFD_F32 ? 4 : 8;
    const unsigned grid = (unsigned)((n * (copy.ld / vecn) + kBlock - 1) / kBlock);
    if (xdt == GNNFD_F32)
        GNNFD_LAUNCH("align_features", s, align_features<float>, grid, kBlock, 0, static_cast<const float*>(d_x), ldx, n, f, cw,
                     copy.pitch, (uint32_t)copy.ld, static_cast<uint4*>(d_aligned));
    else
        GNNFD_LAUNCH("align_features", s, align_features<__nv_bfloat16>, grid, kBlock, 0, static_cast<const __nv_bfloat16*>(d_x),
                     ldx, n, f, cw, copy.pitch, (uint32_t)copy.ld, static_cast<uint4*>(d_aligned));
}

static bool aligned_for_vectors(const void* d_x, int64_t ldx, gnnfd_dtype_t xdt, int32_t f, int32_t cw)
{
    const int xsize = xdt == GNNFD_F32 ? 4 : 2;
    return ((uintptr_t)d_x % 16 == 0) && ((ldx * xsize) % 16 == 0) && (f <= cw || (cw * xsize) % 16 == 0);
}

// Where the copy is faster than element-wise loads: fp32 from where those need a whole warp for 64 columns (33 up), bf16 from 3
// columns, below which the padding to 16 bytes outweighs the loads.  132,534 rows of 300 entries, loads -> copy: bf16 1 / 2 / 3 / 5 / 9 /
// 41 columns 113 / 170 / 221 / 281 / 387 / 866 -> 182 / 182 / 183 / 184 / 240 / 443 us, 301 in chunks of 4 17.7 -> 15.7 ms, fp32
// 33 / 41 / 301 columns 803 / 806 / 5410 -> 636 / 644 / 3704 us; 200,000 rows of 150, 25 fp32 columns 0.45 -> 0.49 ms.
static AlignedCopy plan_copy(const gnnfd_csr_t* csr, const void* d_x, int64_t ldx, gnnfd_dtype_t xdt, int32_t f, int32_t cw)
{
    const int xsize = xdt == GNNFD_F32 ? 4 : 2;
    if (aligned_for_vectors(d_x, ldx, xdt, f, cw) || cw <= (xsize == 4 ? 32 : 2)) return AlignedCopy{cw, ldx, 0};
    // In lanes that the element-wise kernel puts on an entry (two columns each).  Loads -> copy: 50,000 rows of 9 entries, 41 bf16
    // columns (14 M) 41 -> 29 us; 200,000 of 17, 7 columns (14 M) 41 -> 38, 4 columns (7 M) 33 -> 35; 5,000 of 51, 41 fp32 columns (8 M)
    // 15 -> 18.
    int64_t lanes = 1;
    while (lanes < 32 && 2 * lanes < cw) lanes <<= 1;
    if (!copy_pays(csr, lanes * ((cw + 63) / 64), 10000000)) return AlignedCopy{cw, ldx, 0};
    // Chunks of one vector start on 16 bytes, wider ones on 32-byte sectors, so the copy is at most 2.7 times the features.  Rows
    // of more than a line start on one where they are gathered often enough to make up for the larger copy (41 fp32 columns
    // on 116 M entries: pitch 48 1.78 ms, 64 1.69; on 200,000 rows of 16 entries 93 and 97 us).
    const int unit = cw * xsize <= 16 ? 16 : 32;
    const bool lines = csr->nnz >= 64 * csr->n && (int64_t)f * xsize > 128;
    return layout_copy(csr->n, xdt, f, cw, unit, lines ? 128 : unit);
}

static size_t partial_bytes(const gnnfd_csr_t* csr, int32_t f)
{
    const size_t fpad = align_up((size_t)f, 4);
    return align_up((size_t)csr->n_segments * fpad * sizeof(float), 256);
}

static int aggregate(bool weighted, const gnnfd_csr_t* csr, const void* d_x, int64_t ldx, gnnfd_dtype_t xdt, void* d_out,
                     int64_t ldo, gnnfd_dtype_t odt, int32_t f, int32_t chunk_width, void* d_scratch,
                     size_t scratch_bytes, cudaStream_t s)
{
    if (!csr || !d_x || !d_out || f <= 0 || chunk_width <= 0 || ldx < f || ldo < f || ldx > 0x7fffffffll)
        return GNNFD_INVALID_ARG;
    if ((xdt != GNNFD_F32 && xdt != GNNFD_BF16) || (odt != GNNFD_F32 && odt != GNNFD_BF16)) return GNNFD_UNSUPPORTED;
    const size_t need = partial_bytes(csr, f);
    if (need > 0 && (!d_scratch || scratch_bytes < need)) return GNNFD_WORKSPACE_TOO_SMALL;
    if (need > 0 && ((uintptr_t)d_scratch & 15u)) return GNNFD_INVALID_ARG;

    const int cw = chunk_width < f ? chunk_width : f;
    const int n_chunks = (f + cw - 1) / cw;
    const int xsize = xdt == GNNFD_F32 ? 4 : 2;
    const int vecn = 16 / xsize;
    // 128-bit loads need 16-byte aligned row starts and chunk starts: those of the features, or of a copy where the scratch
    // buffer has room for one
    const AlignedCopy copy = plan_copy(csr, d_x, ldx, xdt, f, cw);
    const bool copied = copy.bytes > 0 && d_scratch && ((uintptr_t)d_scratch & 15u) == 0 && scratch_bytes >= need + copy.bytes;
    int32_t x_gap = 0;
    if (copied) {
        void* aligned = static_cast<char*>(d_scratch) + need;
        launch_copy(d_x, ldx, xdt, csr->n, f, cw, copy, aligned, s);
        d_x = aligned;
        ldx = copy.ld;
        x_gap = copy.pitch - cw;
    }
    const bool vec = copied || aligned_for_vectors(d_x, ldx, xdt, f, cw);
    const int elems = vec ? vecn : 1;
    // a lane covers two vectors of the chunk unless the chunk is a single vector wide
    const int vectors = (cw + elems - 1) / elems;
    int vpl = vectors > 1 ? 2 : 1;
    int lpr = 1;
    while (lpr * vpl < vectors && lpr < 32) lpr <<= 1;
    // 17 - 24 and 33 - 48 vectors fit three per lane on half the lanes instead of leaving up to half of them idle: 192 fp32 columns on
    // 200,000 rows of 16 entries 300 -> 230 us, 96 columns on 116 M entries 3.02 -> 2.64 ms.  Not 9 - 12: four lanes' vectors make
    // 64-byte pieces, which split more cache lines than the idle lanes cost (44 columns there 1.88 -> 2.01 ms).
    if (vec && lpr >= 16 && vectors <= lpr / 2 * 3) {
        vpl = 3;
        lpr /= 2;
    }
    // Wider chunks go out in tiles of 64 vectors, or of 32 where the last tile of 64 would be mostly empty: 76 vectors (304
    // fp32 columns) on 200,000 rows of 16 entries 0.60 -> 0.52 ms; with full tiles the narrower one is 0 - 8 % slower.
    if (vec && vectors > 64 && (vectors + 31) / 32 * 32 * 1.04 < (vectors + 63) / 64 * 64) lpr = 16;

    GatherArgs a;
    a.row_ptr = csr->row_ptr; a.col_idx = csr->col_idx; a.edge_w = csr->edge_w; a.rdeg = csr->rdeg;
    a.row_order = csr->row_order; a.seg_row = csr->seg_row; a.seg_begin = csr->seg_begin;
    a.seg_end = csr->seg_end; a.seg_slot = csr->seg_slot;
    a.x = d_x; a.out = d_out; a.partial = static_cast<float*>(d_scratch);
    a.ldx = ldx; a.ldo = ldo; a.f = f; a.chunk_width = cw;
    a.n_ctiles = (cw + lpr * vpl * elems - 1) / (lpr * vpl * elems);
    a.part_filled = vectors != lpr * vpl;
    a.fpad = (int32_t)align_up((size_t)f, 4);
    a.out_bf16 = odt == GNNFD_BF16;
    // 32-byte loads of a lane's vector pair: every pair must start on a 32-byte boundary, and the chunk must
    // be narrow (up to 128 bytes, four lanes per row).  There the pair load halves the cache lines an
    // instruction touches (hidden width 8 / 16 / 32 on the config-4 graph: 0.84 / 1.04 / 1.28 -> 0.61 / 0.77 /
    // 0.99 ms); with eight or more lanes per row the strided single vectors already cover whole lines and
    // the pair form is slower (config 4 at 64 columns 16.2 -> 18.4 ms).
    a.wide_ok = vec && vpl == 2 && lpr <= 4 && ((uintptr_t)d_x % 32 == 0) && ((ldx * xsize) % 32 == 0) &&
                (n_chunks == 1 || ((cw + x_gap) * xsize) % 32 == 0);
    a.out_vec_ok = odt == GNNFD_F32 && ((uintptr_t)d_out % 16 == 0) && (ldo % 4 == 0) && (n_chunks == 1 || cw % 4 == 0);

    const int per_step = kLoads / vpl * (32 / lpr);
    bool shared = false;
    int64_t blocks = 0;
    auto plan = [&](int blocks_per_sm) {
        blocks = plan_ranges(csr, gather_groups(), lpr, per_step, walk_limit(csr, per_step, a.n_ctiles, 16, blocks_per_sm), a.range, &a.n_ranges);
        for (int i = 0; i < a.n_ranges; ++i) shared = shared || a.range[i].warps_log2 > 0;
    };
    const int unsplit = min_blocks(xsize, weighted, false, lpr), split = min_blocks(xsize, weighted, true, lpr);
    // GCN's kernel for unsplit rows has four blocks per SM, that for split ones three.  From where four would call for splitting to where three do
    // (3.6 to 4.8 M entries), the longest rows decide and three are faster unsplit: 100,000 rows of 40, 16 / 64 / 96 columns 44 / 99 / 125 us
    // with four, 36 / 79 / 104 with three; above, 200,000 of 30, 50 / 113 / 165 with four, 52 / 121 / 170 with three.
    plan(unsplit);
    if (shared && split != unsplit) plan(split);
    a.blocks_per_tile = (int32_t)blocks;
    const int64_t grid_x = blocks * a.n_ctiles;
    if (grid_x > 0x7fffffffll) return GNNFD_TOO_LARGE;

    if (grid_x > 0) {
        if (shortest_first(xsize, elems, lpr, vpl, shared))
            for (int i = 0; i < a.n_ranges; ++i) {
                a.range[i].item_first -= a.range[i].item_count - 1;
                a.range[i].item_step = 1;
            }
        const bool wide = a.wide_ok != 0;
        GatherKernel kernel = weighted ? (shared ? pick_kernel<true, true>(xdt, vec, lpr, vpl, wide) : pick_kernel<true, false>(xdt, vec, lpr, vpl, wide))
                                       : (shared ? pick_kernel<false, true>(xdt, vec, lpr, vpl, wide) : pick_kernel<false, false>(xdt, vec, lpr, vpl, wide));
        // A copy with columns between its chunks is gathered chunk by chunk: with the offset computed in the kernel every other call pays
        // for it too (GCN, 48 fp32 columns on 60,000 rows of 200 entries 209 -> 214 us).
        const int per_launch = x_gap > 0 ? 1 : kMaxGridY;
        for (int c0 = 0; c0 < n_chunks; c0 += per_launch) {
            a.chunk_base = c0;
            a.x = static_cast<const char*>(d_x) + (int64_t)c0 * x_gap * xsize;
            const dim3 grid((unsigned)grid_x, (unsigned)(n_chunks - c0 < per_launch ? n_chunks - c0 : per_launch));
            GNNFD_LAUNCH(weighted ? "gather_aggregate_gcn" : "gather_aggregate_sage", s, kernel, grid, kBlock, 0, a);
        }
    }
    const int64_t n_hub = csr->bin_count[4];
    if (n_hub > 0) {
        dim3 g((unsigned)n_hub, (unsigned)((f + kBlock - 1) / kBlock));
        GNNFD_LAUNCH("hub_reduce", s, hub_reduce, g, kBlock, 0, csr->row_order, csr->hub_seg_ptr, csr->rdeg, a.partial,
                     csr->bin_start[4], (int32_t)n_hub, f, a.fpad, weighted ? 0 : 1, d_out, ldo, a.out_bf16);
    }
    GNNFD_CUDA_CHECK(cudaGetLastError());
    return GNNFD_OK;
}

}  // namespace gnnfd

extern "C" {

int gnnfd_aggregate_workspace_bytes(const gnnfd_csr_t* csr, int32_t f, size_t* scratch_bytes)
{
    if (!csr || f <= 0 || !scratch_bytes) return GNNFD_INVALID_ARG;
    *scratch_bytes = gnnfd::partial_bytes(csr, f);
    return GNNFD_OK;
}

int gnnfd_aggregate_best_workspace_bytes(const gnnfd_csr_t* csr, const void* d_x, int64_t ldx, gnnfd_dtype_t xdt, int32_t f,
                                         int32_t chunk_width, size_t* scratch_bytes)
{
    if (!csr || f <= 0 || chunk_width <= 0 || ldx < f || ldx > 0x7fffffffll || !scratch_bytes) return GNNFD_INVALID_ARG;
    if (xdt != GNNFD_F32 && xdt != GNNFD_BF16) return GNNFD_UNSUPPORTED;
    *scratch_bytes = gnnfd::partial_bytes(csr, f) +
                     gnnfd::plan_copy(csr, d_x, ldx, xdt, f, chunk_width < f ? chunk_width : f).bytes;
    return GNNFD_OK;
}

int gnnfd_aggregate_gcn(const gnnfd_csr_t* csr, const void* d_x, int64_t ldx, gnnfd_dtype_t xdt, void* d_out, int64_t ldo,
                        gnnfd_dtype_t odt, int32_t f, int32_t chunk_width, void* d_scratch, size_t scratch_bytes,
                        void* stream)
{
    return gnnfd::aggregate(true, csr, d_x, ldx, xdt, d_out, ldo, odt, f, chunk_width, d_scratch, scratch_bytes,
                            static_cast<cudaStream_t>(stream));
}

int gnnfd_aggregate_sage(const gnnfd_csr_t* csr, const void* d_x, int64_t ldx, gnnfd_dtype_t xdt, void* d_out, int64_t ldo,
                         gnnfd_dtype_t odt, int32_t f, int32_t chunk_width, void* d_scratch, size_t scratch_bytes,
                         void* stream)
{
    return gnnfd::aggregate(false, csr, d_x, ldx, xdt, d_out, ldo, odt, f, chunk_width, d_scratch, scratch_bytes,
                            static_cast<cudaStream_t>(stream));
}

}  // extern "C"
