// GAT: attention scores and the fused logit + online-softmax + weighted-sum aggregation.
//
// The attention logits always use the full head width (scores are computed once from all of z);
// feature decomposition only cuts the weighted sum into column chunks, so the chunked result equals
// the undecomposed one.  The fused kernel walks a row once, keeping a running maximum m, a running
// denominator l and the un-normalised weighted sum per lane; edge-parallel groups and hub segments
// are merged by the usual log-sum-exp rule in a fixed order.
#include <math_constants.h>

#include <type_traits>

#include "schedule.cuh"
#include "vec.cuh"

namespace gnnfd {

struct GatArgs {
    const int32_t* row_ptr;
    const int32_t* col_idx;
    const int32_t* row_order;
    const int32_t* seg_row;
    const int32_t* seg_begin;
    const int32_t* seg_end;
    const int32_t* seg_slot;
    const float* s_src;
    const float* s_dst;
    const void* z;
    void* out;
    float* partial;      // [n_segments, fpad] un-normalised sums of hub segments
    float* partial_ml;   // [n_segments, heads, 2] running max and denominator of hub segments
    int64_t ldz, ldo;
    float slope;
    int32_t f, heads, dim, chunk_width, n_ctiles, blocks_per_tile, fpad, out_bf16, out_vec_ok, wide_ok;   // columns as z holds them
    int32_t out_dim;         // columns of a head in the output (dim, or less where z is a copy with padded heads)
    int32_t chunk_base;      // first chunk of this launch (a launch covers at most 65,535 chunks)
    int32_t n_ranges;
    Range range[kMaxRanges];
};

constexpr float kLog2e = 1.4426950408889634f;

// 2^x by the hardware approximation (2 ulp; results below 2^-126 become 0, 2^-inf = 0)
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// weight of a partial result with running maximum m (a base-2 logit) when merged under the maximum m_new
__device__ __forceinline__ float merge_scale(float m, float m_new)
{
    return m == -CUDART_INF_F ? 0.f : exp2f(m - m_new);
}

// ------------------------------------------------------------------ scores

// One thread per vertex and head, elements in ascending order.  With VECN > 1 the head's elements come in 16-byte vectors
// (a head is a whole number of them and starts on a 16-byte boundary): the element-wise form left half of every sector
// it touched to a later instruction (25 us for [200,000, 8 x 8] fp32, 51 MB).
template <typename T, int VECN>
__global__ void __launch_bounds__(kBlock)
gat_scores(const T* z, int64_t ldz, const float* a_src, const float* a_dst,
           int64_t n, int heads, int dim, float* __restrict__ s_src, float* __restrict__ s_dst)
{
    grid_dependency<true>();
    const int64_t idx = (int64_t)blockIdx.x * kBlock + threadIdx.x;
    if (idx >= n * heads) return;
    const int64_t v = idx <= 0x7fffffffll ? (int64_t)((uint32_t)idx / (uint32_t)heads) : idx / heads;
    const int h = (int)(idx - v * heads);
    const T* zr = z + v * ldz + (int64_t)h * dim;
    const float *as = a_src + h * dim, *ad = a_dst + h * dim;
    float ss = 0.f, sd = 0.f;
    for (int d = 0; d < dim; d += VECN) {
        Vec<T, VECN> zv;
        zv.load(zr + d);
#pragma unroll
        for (int i = 0; i < VECN; ++i) {
            ss = fmaf(load4(as + d + i), zv.get(i), ss);
            sd = fmaf(load4(ad + d + i), zv.get(i), sd);
        }
    }
    s_src[idx] = ss;
    s_dst[idx] = sd;
}

// ------------------------------------------------------------------ fused aggregation

constexpr int kLoads = 8;      // 16-byte feature loads kept in flight per lane

// index registers per lane and batch, and the column indices a warp stages per batch
constexpr int index_regs(int lpr, int vpl) { return kLoads / vpl > lpr ? kLoads / vpl / lpr : 1; }
constexpr int stage_slots(int lpr, int vpl) { return 32 * index_regs(lpr, vpl); }

// On graphs that fill the chip an entry costs a logit, an exponential and the unpacking of its features on top of the
// gather, so products and rescalings go two to an instruction: on 200,000 rows of
// 150 entries 8 heads of 16 bf16 columns 0.96 -> 0.89 ms, 8 x 8 bf16 0.54 -> 0.48, fp32 unchanged.  On smaller graphs the
// longest row decided; shared by warps (see schedule.cuh) 4,000 rows of 10 entries, 8 x 16 fp32, take 23 us
// instead of 71, 20,000 of 50 64 instead of 155, 100,000 of 20 146 instead of 221.
//
// One row (or hub segment) per S = LPR * EP lanes, same batching as the GCN / SAGE gather: the S lanes
// fetch S column indices per round with one coalesced load and stage them in shared memory.  A lane
// covers VPL adjacent vectors, all inside one head, so it needs one logit per entry.
template <typename T, int VECN, int LPR, int VPL, bool SHARED, int EP>
__device__ __forceinline__ void gat_rows(const GatArgs& a, const Range& rg, int block_in_range, int col0, int chunk_end,
                                         int32_t (*stage_col)[kBlock / 32][stage_slots(LPR, VPL)], float (*tot_s)[kBlock])
{
    constexpr int S = LPR * EP;
    constexpr int ROWS = kBlock / S;
    constexpr int UB = kLoads / VPL;
    constexpr int R = index_regs(LPR, VPL);
    constexpr int SPB = R * LPR;
    constexpr int EPB = R * S;
    constexpr unsigned kFull = 0xffffffffu;
    const int tid = threadIdx.x;
    // a long row may be shared by several warps of the block, which take consecutive parts of it
    const int warps_log2 = SHARED && S == 32 ? rg.warps_log2 : 0, sharer = tid / S & ((1 << warps_log2) - 1);
    const int slot = block_in_range * (ROWS >> warps_log2) + (tid / S >> warps_log2);
    const int sl = tid % S;
    const int g = sl / LPR;
    const int c = sl % LPR;
    const int j0 = col0 + c * (VPL * VECN);
    const int warp = tid >> 5, lane = tid & 31;
    const int seg = lane - sl;                   // first lane of this row's segment inside the warp
    const bool active = slot < rg.item_count;
    const bool lane_ok = j0 < chunk_end;
    // lanes past the end of the chunk read what the last lane inside it reads, in the same instruction
    const int jl = lane_ok ? j0 : col0 + (chunk_end - 1 - col0) / (VPL * VECN) * (VPL * VECN);
    const int h = jl / a.dim;

    bool okq[VPL];
    const T* zq[VPL];
#pragma unroll
    for (int q = 0; q < VPL; ++q) {
        okq[q] = j0 + q * VECN < chunk_end;
        zq[q] = static_cast<const T*>(a.z) + (jl + q * VECN < chunk_end ? jl + q * VECN : jl);
    }

    int32_t row = 0, b = 0, e = 0;
    if (active) {
        if (rg.hub) {
            row = a.seg_row[slot];
            b = a.seg_begin[slot];
            e = a.seg_end[slot];
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
    // one 32-byte load per entry where every row start allows it (a lane past the chunk's end loads the chunk's last pair)
    const bool wide = a.wide_ok;
    const float sd = active ? a.s_dst[(int64_t)row * a.heads + h] : 0.f;
    const float* ssrc = a.s_src + h;
    // logits are kept in base 2: LeakyReLU(x) * log2 e = c1 * x + c2 * |x|
    const float c1 = 0.5f * kLog2e * (1.f + a.slope), c2 = 0.5f * kLog2e * (1.f - a.slope);
    auto leaky2 = [c1, c2](float x) { return fmaf(fabsf(x), c2, x * c1); };
    const uint32_t ld = (uint32_t)a.ldz;
    const uint32_t heads = (uint32_t)a.heads;

    // Two levels of accumulation (as in the GCN / SAGE gather): `acc` and `l` take at most kChain terms in a
    // row, then move into the thread's second-level sums in shared memory (slot VPL * VECN holds the
    // denominator).  The second level is expressed under its own maximum m_tot and is brought to the
    // current one only when something is added to it.
    constexpr int kChain = 64;
    constexpr int FLUSH = SPB >= kChain ? 1 : kChain / SPB;
    float m = -CUDART_INF_F, l = 0.f, m_tot = -CUDART_INF_F;
    float acc[VPL][VECN];
#pragma unroll
    for (int q = 0; q < VPL; ++q)
#pragma unroll
        for (int i = 0; i < VECN; ++i) acc[q][i] = 0.f;
    auto move_to_second_level = [&]() {
        const float sc = m_tot == -CUDART_INF_F ? 0.f : ex2(m_tot - m);     // m >= m_tot; both -inf before any entry
        m_tot = m;
        tot_s[VPL * VECN][tid] = fmaf(tot_s[VPL * VECN][tid], sc, l);
        l = 0.f;
#pragma unroll
        for (int q = 0; q < VPL; ++q)
#pragma unroll
            for (int i = 0; i < VECN; ++i) {
                tot_s[q * VECN + i][tid] = fmaf(tot_s[q * VECN + i][tid], sc, acc[q][i]);
                acc[q][i] = 0.f;
            }
    };

    const int n_batches = __reduce_max_sync(kFull, (e - b + EPB - 1) / EPB);
    const bool two_level = n_batches > FLUSH;          // short rows never leave the first level
    if (two_level) {
#pragma unroll
        for (int k = 0; k <= VPL * VECN; ++k) tot_s[k][tid] = 0.f;
    }
    int32_t ucur[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int32_t kk = b + r * S + sl;
        ucur[r] = kk < e ? __ldcs(a.col_idx + kk) : -1;
    }

    for (int ib = 0; ib < n_batches; ++ib) {
        const int32_t kb = b + ib * EPB;
        int32_t unext[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int32_t kk = kb + EPB + r * S + sl;
            unext[r] = kk < e ? __ldcs(a.col_idx + kk) : -1;
        }
        const int buf = ib & 1;
#pragma unroll
        for (int r = 0; r < R; ++r) stage_col[buf][warp][r * 32 + lane] = ucur[r];
        __syncwarp();
        // one group of UB entries: gathers issued together, then one update of the running softmax
        auto steps = [&](auto full_tag) {
            constexpr bool FULL = decltype(full_tag)::value;
            // in a ragged batch step s works on entries s * EP .. of a row's batch: the steps past the longest
            // remainder in the warp have nothing to do for any lane
            const int rem = FULL ? EPB : __reduce_max_sync(kFull, e - kb);
#pragma unroll
            for (int s0 = 0; s0 < SPB; s0 += UB) {
                if (!FULL && s0 > 0 && s0 * EP >= rem) break;
                Vec<T, VECN> v[UB][VPL];
                float lg[UB];
                bool valid[UB];
#pragma unroll
                for (int i = 0; i < UB; ++i) {
                    const int r = (s0 + i) / LPR, t = (s0 + i) % LPR;
                    const int32_t u = stage_col[buf][warp][r * 32 + seg + t * EP + g];
                    valid[i] = FULL || u >= 0;
                    const uint32_t uu = FULL ? (uint32_t)u : (uint32_t)max(u, 0);
                    lg[i] = valid[i] ? load4(ssrc + (size_t)uu * heads) : 0.f;
                    const size_t off = (size_t)uu * ld;
                    if (VPL == 2 && VECN * sizeof(T) == 16 && wide) {
                        if (valid[i]) load_pair(v[i][0], v[i][VPL - 1], zq[0] + off);     // the lane's two vectors are adjacent
                        else { v[i][0].zero(); v[i][VPL - 1].zero(); }
                    } else {
#pragma unroll
                        for (int q = 0; q < VPL; ++q) {
                            if (valid[i]) v[i][q].load(zq[q] + off);
                            else v[i][q].zero();
                        }
                    }
                }
                float mx = m;
#pragma unroll
                for (int i = 0; i < UB; ++i) {
                    lg[i] = leaky2(lg[i] + sd);
                    if (valid[i]) mx = fmaxf(mx, lg[i]);
                }
                if (FULL || mx != -CUDART_INF_F) {      // a group with no entry at all leaves the state alone
                    const float rescale = ex2(m - mx);  // 2^-inf = 0 on the first group
                    m = mx;
                    l *= rescale;
#pragma unroll
                    for (int q = 0; q < VPL; ++q)
#pragma unroll
                        for (int i = 0; i < VECN; i += VECN > 1 ? 2 : 1) {
                            if constexpr (VECN > 1) mul_pair(acc[q][i], acc[q][i + 1], rescale, rescale);
                            else acc[q][i] *= rescale;
                        }
                }
#pragma unroll
                for (int i = 0; i < UB; ++i) {
                    // hardware 2^x: the argument is <= 0 and its error (about 2 ulp + |x| * 2^-23 relative) stays
                    // two orders below the 1e-5 bound on the weighted sum
                    const float p = valid[i] ? ex2(lg[i] - m) : 0.f;
                    l += p;
#pragma unroll
                    for (int q = 0; q < VPL; ++q)
#pragma unroll
                        for (int k = 0; k < VECN; k += VECN > 1 ? 2 : 1) {
                            if constexpr (VECN > 1) fma_pair(acc[q][k], acc[q][k + 1], p, v[i][q].get(k), v[i][q].get(k + 1));
                            else acc[q][k] = fmaf(p, v[i][q].get(k), acc[q][k]);
                        }
                }
            }
        };
        if (__all_sync(kFull, kb + EPB <= e)) steps(std::true_type{});
        else steps(std::false_type{});
#pragma unroll
        for (int r = 0; r < R; ++r) ucur[r] = unext[r];
        if (two_level && (ib + 1) % FLUSH == 0) move_to_second_level();
    }
    if (two_level) {
        move_to_second_level();
        l = tot_s[VPL * VECN][tid];
#pragma unroll
        for (int q = 0; q < VPL; ++q)
#pragma unroll
            for (int i = 0; i < VECN; ++i) acc[q][i] = tot_s[q * VECN + i][tid];
    }

    // merge the EP groups of the row, fixed tree
#pragma unroll
    for (int o = S / 2; o >= LPR; o >>= 1) {
        const float m2 = __shfl_down_sync(kFull, m, o, S);
        const float l2 = __shfl_down_sync(kFull, l, o, S);
        const float mn = fmaxf(m, m2);
        const float sa = merge_scale(m, mn), sb = merge_scale(m2, mn);
        l = l * sa + l2 * sb;
#pragma unroll
        for (int q = 0; q < VPL; ++q)
#pragma unroll
            for (int i = 0; i < VECN; ++i) {
                const float a2 = __shfl_down_sync(kFull, acc[q][i], o, S);
                acc[q][i] = acc[q][i] * sa + a2 * sb;
            }
        m = mn;
    }

    if (SHARED && S == 32 && warps_log2 > 0) {      // the sharers' results, first to last; the whole block is on this side
        constexpr int L = VPL * VECN, M = L + 1;
        if (sharer > 0) {
#pragma unroll
            for (int k = 0; k < L; ++k) tot_s[k][tid] = acc[k / VECN][k % VECN];
            tot_s[L][tid] = l;
            tot_s[M][tid] = m;
        }
        __syncthreads();
        if (sharer > 0) return;
        for (int w = 1; w < 1 << warps_log2; ++w) {
            const int other = tid + 32 * w;
            const float m2 = tot_s[M][other], mn = fmaxf(m, m2);
            const float sa = merge_scale(m, mn), sb = merge_scale(m2, mn);
            l = l * sa + tot_s[L][other] * sb;
#pragma unroll
            for (int k = 0; k < L; ++k) acc[k / VECN][k % VECN] = acc[k / VECN][k % VECN] * sa + tot_s[k][other] * sb;
            m = mn;
        }
    }

    if (!active || g != 0 || !lane_ok) return;
    // where a hub segment's partial results go (read here, at the end, so that it occupies no register during the walk)
    const int32_t part = rg.hub ? a.seg_slot[slot] : 0;
    if (rg.hub) {
        // every lane of a head holds the same (m, l); the first lane of each head inside this column tile stores
        // it (sweeps that share a head store identical values)
        if (j0 % a.dim == 0 || c == 0) {
            float* ml = a.partial_ml + ((int64_t)part * a.heads + h) * 2;
            ml[0] = m;
            ml[1] = l;
        }
    }
    const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
    for (int q = 0; q < VPL; ++q) {
        if (!okq[q]) continue;
        const int j = j0 + q * VECN;
        if (rg.hub) {
            float* p = a.partial + (int64_t)part * a.fpad + j;
#pragma unroll
            for (int i = 0; i < VECN; ++i)
                if (j + i < chunk_end) p[i] = acc[q][i];
        } else {
            const int d = j - h * a.dim;                                     // column inside the head
            const int64_t o = (int64_t)row * a.ldo + h * a.out_dim + d;
            if (VECN % 4 == 0 && a.out_vec_ok) {
#pragma unroll
                for (int i = 0; i < VECN; i += 4)
                    if (d + i < a.out_dim)
                        __stcs(reinterpret_cast<float4*>(static_cast<float*>(a.out) + o + i),
                               make_float4(acc[q][i] * inv, acc[q][i + 1] * inv, acc[q][i + 2] * inv, acc[q][i + 3] * inv));
            } else {
#pragma unroll
                for (int i = 0; i < VECN; ++i)
                    if (j + i < chunk_end && d + i < a.out_dim) store_elem(a.out, a.out_bf16, o + i, acc[q][i] * inv);
            }
        }
    }
}

template <typename T, int VECN, int LPR, int VPL, bool SHARED>
// Register budget: left to itself the compiler gives the wide instantiations anything between 80 and 126
// registers from one build to the next (two blocks per SM instead of three, 20 % slower); three blocks per SM for
// the vector-pair forms and four for the others is what the measured-good builds had.
__global__ void __launch_bounds__(kBlock, (VPL == 2 && VECN > 1) ? 3 : 4) gat_aggregate(const __grid_constant__ GatArgs a)
{
    grid_dependency<false>();
    __shared__ int32_t stage_col[2][kBlock / 32][stage_slots(LPR, VPL)];
    // second-level sums and denominator (and a sharer's maximum), one column per thread
    __shared__ float tot_s[VPL * VECN + 1 + SHARED][kBlock];
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
        case 0: gat_rows<T, VECN, LPR, VPL, SHARED, 1>(a, rg, bir, col0, chunk_end, stage_col, tot_s); break;
        case 1: if constexpr (LPR * 2 <= 32) gat_rows<T, VECN, LPR, VPL, SHARED, 2>(a, rg, bir, col0, chunk_end, stage_col, tot_s); break;
        case 2: if constexpr (LPR * 4 <= 32) gat_rows<T, VECN, LPR, VPL, SHARED, 4>(a, rg, bir, col0, chunk_end, stage_col, tot_s); break;
        case 3: if constexpr (LPR * 8 <= 32) gat_rows<T, VECN, LPR, VPL, SHARED, 8>(a, rg, bir, col0, chunk_end, stage_col, tot_s); break;
        case 4: if constexpr (LPR * 16 <= 32) gat_rows<T, VECN, LPR, VPL, SHARED, 16>(a, rg, bir, col0, chunk_end, stage_col, tot_s); break;
        default: if constexpr (LPR == 1) gat_rows<T, VECN, LPR, VPL, SHARED, 32>(a, rg, bir, col0, chunk_end, stage_col, tot_s); break;
    }
}

// out[row, j] = sum_s partial[s, j] e^(m_s - M) / sum_s l_s e^(m_s - M) over the segments s of a hub row.
// A block covers kReduceCols columns of one row; kReduceWays threads per column walk interleaved
// segments and their results are combined in a fixed order through shared memory.
constexpr int kReduceCols = 64;
constexpr int kReduceWays = kBlock / kReduceCols;

__global__ void __launch_bounds__(kBlock)
gat_hub_reduce(const int32_t* row_order, const int32_t* hub_seg_ptr,
               const float* partial, const float* partial_ml, int64_t hub_begin, int32_t n_hub,
               int32_t f, int32_t fpad, int32_t heads, int32_t dim, int32_t out_dim, void* __restrict__ out, int64_t ldo, int out_bf16)
{
    grid_dependency<true>();
    __shared__ float s_max[kReduceWays][kReduceCols], s_num[kReduceWays][kReduceCols], s_den[kReduceWays][kReduceCols];
    const int i = blockIdx.x;
    const int c = threadIdx.x % kReduceCols, q = threadIdx.x / kReduceCols;
    const int j = blockIdx.y * kReduceCols + c;
    const bool ok = j < f;
    const int h = ok ? j / dim : 0;
    const int32_t row = row_order[hub_begin + i];
    const int32_t s0 = hub_seg_ptr[i], s1 = hub_seg_ptr[i + 1];
    float mx = -CUDART_INF_F;
    if (ok)
        for (int32_t s = s0 + q; s < s1; s += kReduceWays) mx = fmaxf(mx, partial_ml[((int64_t)s * heads + h) * 2]);
    s_max[q][c] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kReduceWays; ++w) mx = fmaxf(mx, s_max[w][c]);
    float num = 0.f, den = 0.f;
    if (ok) {
        float num_run = 0.f, den_run = 0.f;
        int in_run = 0;
        for (int32_t s = s0 + q; s < s1; s += kReduceWays) {
            const float* ml = partial_ml + ((int64_t)s * heads + h) * 2;
            const float w = merge_scale(ml[0], mx);
            den_run = fmaf(ml[1], w, den_run);
            num_run = fmaf(partial[(int64_t)s * fpad + j], w, num_run);
            if (++in_run == 32) { num += num_run; den += den_run; num_run = den_run = 0.f; in_run = 0; }   // short chains
        }
        num += num_run;
        den += den_run;
    }
    s_num[q][c] = num;
    s_den[q][c] = den;
    __syncthreads();
    if (q != 0 || !ok) return;
    num = 0.f;
    den = 0.f;
#pragma unroll
    for (int w = 0; w < kReduceWays; ++w) { num += s_num[w][c]; den += s_den[w][c]; }
    const int d = j - h * dim;
    if (d < out_dim) store_elem(out, out_bf16, (int64_t)row * ldo + h * out_dim + d, den > 0.f ? num / den : 0.f);
}

// ------------------------------------------------------------------ host side

typedef void (*GatKernel)(const GatArgs);

template <typename T, int VECN, int VPL, bool SHARED>
static GatKernel pick_lpr(int lpr)
{
    switch (lpr) {
        case 1: return gat_aggregate<T, VECN, 1, VPL, SHARED>;
        case 2: return gat_aggregate<T, VECN, 2, VPL, SHARED>;
        case 4: return gat_aggregate<T, VECN, 4, VPL, SHARED>;
        case 8: return gat_aggregate<T, VECN, 8, VPL, SHARED>;
        case 16: return gat_aggregate<T, VECN, 16, VPL, SHARED>;
        default: return gat_aggregate<T, VECN, 32, VPL, SHARED>;
    }
}

template <typename T, int VECN>
static GatKernel pick_vpl(int lpr, int vpl, bool shared)
{
    if (shared) return vpl == 2 ? pick_lpr<T, VECN, 2, true>(lpr) : pick_lpr<T, VECN, 1, true>(lpr);
    return vpl == 2 ? pick_lpr<T, VECN, 2, false>(lpr) : pick_lpr<T, VECN, 1, false>(lpr);
}

struct GatScratch {
    float *s_src, *s_dst, *partial, *partial_ml;
};

static void carve_gat(Carver& c, const gnnfd_csr_t* csr, int32_t heads, int32_t dim, GatScratch* g)
{
    const size_t fpad = align_up((size_t)heads * dim, 4);
    g->s_src = c.take<float>((size_t)csr->n * heads);
    g->s_dst = c.take<float>((size_t)csr->n * heads);
    g->partial = c.take<float>((size_t)csr->n_segments * fpad);
    g->partial_ml = c.take<float>((size_t)csr->n_segments * heads * 2);
}

static int launch_scores(int64_t n, const void* d_z, int64_t ldz, gnnfd_dtype_t zdt, const float* d_a_src,
                         const float* d_a_dst, int32_t heads, int32_t dim, float* d_s_src, float* d_s_dst, cudaStream_t s)
{
    const int64_t total = n * heads;
    const unsigned grid = (unsigned)((total + kBlock - 1) / kBlock);
    const int zsize = zdt == GNNFD_F32 ? 4 : 2;
    const bool vec = (uintptr_t)d_z % 16 == 0 && ldz * zsize % 16 == 0 && dim * zsize % 16 == 0;
    if (zdt == GNNFD_F32) {
        const float* z = static_cast<const float*>(d_z);
        GNNFD_LAUNCH("gat_scores", s, (vec ? gat_scores<float, 4> : gat_scores<float, 1>), grid, kBlock, 0, z, ldz, d_a_src, d_a_dst,
                     n, heads, dim, d_s_src, d_s_dst);
    } else {
        const __nv_bfloat16* z = static_cast<const __nv_bfloat16*>(d_z);
        GNNFD_LAUNCH("gat_scores", s, (vec ? gat_scores<__nv_bfloat16, 8> : gat_scores<__nv_bfloat16, 1>), grid, kBlock, 0, z, ldz,
                     d_a_src, d_a_dst, n, heads, dim, d_s_src, d_s_dst);
    }
    GNNFD_CUDA_CHECK(cudaGetLastError());
    return GNNFD_OK;
}

// A copy of z whose heads are padded to whole 16-byte vectors, for heads that are not (7 fp32 or 4 bf16 columns): the vector
// kernels need a vector to stay inside one head.  Heads are the copy's chunks, so the sweeps have to hold whole heads.  132,534
// rows of 300 entries, 8 x 3 / 5 / 7 fp32 1.03 / 2.02 / 2.02 -> 0.43 / 0.71 / 0.72 ms, bf16 1.06 / 2.09 / 2.09 -> 0.54 / 0.55 / 0.55;
// 100,000 rows of 4, 4 x 7 fp32 118 -> 38 us.  Not for heads of one or two columns (8 x 1 fp32 367 -> 428 us, 8 x 2 bf16 474 -> 542;
// on 200,000 rows of 17 8 x 2 fp32 81 -> 90, 32 x 2 286 -> 344), so z grows by 8/3 at most, nor for chunks of up to four
// columns (1 x 3 fp32 273 -> 281; 1 x 5 363 -> 307).
static AlignedCopy plan_head_copy(const gnnfd_csr_t* csr, const void* d_z, int64_t ldz, gnnfd_dtype_t zdt, int32_t heads, int32_t dim,
                                  int32_t cw)
{
    const int zsize = zdt == GNNFD_F32 ? 4 : 2;
    const int32_t f = heads * dim;
    cw = cw < f ? cw : f;
    const int32_t vecn = 16 / zsize;
    const bool aligned = (uintptr_t)d_z % 16 == 0 && ldz * zsize % 16 == 0 && dim * zsize % 16 == 0;
    // In elements, each of which costs a load, a logit and an exponential.  Loads -> copy: 50,000 rows of 9 entries, 4 x 5 fp32 (9 M)
    // 49 -> 29 us; 200,000 of 6, 1 x 7 bf16 (8 M) 49 -> 39; 20,000 of 51, 1 x 7 bf16 (7 M) 25 -> 29.
    if (aligned || (cw < f && cw % dim != 0) || cw <= 4 || dim <= 2 || !copy_pays(csr, cw, 8000000)) return AlignedCopy{dim, ldz, 0};
    return layout_copy(csr->n, zdt, f, dim, 16, f <= vecn ? 16 : 32);
}

size_t gat_copy_bytes(const gnnfd_csr_t* csr, const void* d_z, int64_t ldz, gnnfd_dtype_t zdt, int32_t heads, int32_t dim,
                      int32_t chunk_width)
{
    const AlignedCopy copy = plan_head_copy(csr, d_z, ldz, zdt, heads, dim, chunk_width);
    if (copy.bytes == 0) return 0;
    Carver plain(nullptr, ~size_t(0)), padded(nullptr, ~size_t(0));        // the partial sums have the copy's columns
    GatScratch g;
    carve_gat(plain, csr, heads, dim, &g);
    carve_gat(padded, csr, heads, copy.pitch, &g);
    return padded.off - plain.off + copy.bytes;
}

// scores_ready: the two score arrays at the head of the scratch buffer (see gat_scratch_scores) already hold the
// scores of d_z (the dense transform's epilogue wrote them), so the scores pass is left out.
int gat_aggregate_impl(const gnnfd_csr_t* csr, const void* d_z, int64_t ldz, gnnfd_dtype_t zdt, const float* d_a_src,
                       const float* d_a_dst, int32_t heads, int32_t dim, float negative_slope, void* d_out, int64_t ldo,
                       gnnfd_dtype_t odt, int32_t chunk_width, void* d_scratch, size_t scratch_bytes, bool scores_ready,
                       cudaStream_t s)
{
    if (!csr || !d_z || !d_out || heads <= 0 || dim <= 0 || chunk_width <= 0) return GNNFD_INVALID_ARG;
    if (!scores_ready && (!d_a_src || !d_a_dst)) return GNNFD_INVALID_ARG;
    const int64_t f64 = (int64_t)heads * dim;
    if (f64 > 0x7fffffffll || ldz < f64 || ldo < f64 || ldz > 0x7fffffffll) return GNNFD_INVALID_ARG;
    if ((zdt != GNNFD_F32 && zdt != GNNFD_BF16) || (odt != GNNFD_F32 && odt != GNNFD_BF16)) return GNNFD_UNSUPPORTED;
    if (!d_scratch || ((uintptr_t)d_scratch & 255u)) return GNNFD_INVALID_ARG;
    const int32_t out_dim = dim;
    int32_t f = (int32_t)f64;
    int cw = chunk_width < f ? chunk_width : f;
    Carver c(d_scratch, scratch_bytes);
    GatScratch g;
    carve_gat(c, csr, heads, dim, &g);
    if (!c.ok) return GNNFD_WORKSPACE_TOO_SMALL;
    if (!scores_ready) {
        int rc = launch_scores(csr->n, d_z, ldz, zdt, d_a_src, d_a_dst, heads, dim, g.s_src, g.s_dst, s);
        if (rc) return rc;
    }
    const AlignedCopy copy = plan_head_copy(csr, d_z, ldz, zdt, heads, dim, cw);
    if (copy.bytes > 0) {
        Carver with_copy(d_scratch, scratch_bytes);          // the scores keep their place at the head of the buffer
        GatScratch wider;
        carve_gat(with_copy, csr, heads, copy.pitch, &wider);
        void* aligned = with_copy.take<char>(copy.bytes);
        if (with_copy.ok) {
            launch_copy(d_z, ldz, zdt, csr->n, f, dim, copy, aligned, s);
            g = wider;
            cw = cw / dim * copy.pitch;
            dim = copy.pitch;
            f = heads * dim;
            d_z = aligned;
            ldz = copy.ld;
        }
    }

    const int n_chunks = (f + cw - 1) / cw;
    const int zsize = zdt == GNNFD_F32 ? 4 : 2;
    const int vecn = 16 / zsize;
    // a lane's vector must start 16-byte aligned and stay inside one head
    const bool vec = ((uintptr_t)d_z % 16 == 0) && ((ldz * zsize) % 16 == 0) && (n_chunks == 1 || cw % vecn == 0) &&
                     (dim % vecn == 0);
    const int elems = vec ? vecn : 1;
    // a lane covers two adjacent vectors when both stay inside one head and chunks start on such pairs
    const int vectors = (cw + elems - 1) / elems;
    const int vpl = (vectors > 1 && dim % (2 * elems) == 0 && (n_chunks == 1 || cw % (2 * elems) == 0)) ? 2 : 1;
    int lpr = 1;
    while (lpr * vpl < vectors && lpr < 32) lpr <<= 1;

    GatArgs a;
    a.row_ptr = csr->row_ptr; a.col_idx = csr->col_idx; a.row_order = csr->row_order;
    a.seg_row = csr->seg_row; a.seg_begin = csr->seg_begin; a.seg_end = csr->seg_end; a.seg_slot = csr->seg_slot;
    a.s_src = g.s_src; a.s_dst = g.s_dst; a.z = d_z; a.out = d_out;
    a.partial = g.partial; a.partial_ml = g.partial_ml;
    a.ldz = ldz; a.ldo = ldo; a.slope = negative_slope;
    a.f = f; a.heads = heads; a.dim = dim; a.out_dim = out_dim; a.chunk_width = cw;
    a.n_ctiles = (cw + lpr * vpl * elems - 1) / (lpr * vpl * elems);
    a.fpad = (int32_t)align_up((size_t)f, 4);
    a.out_bf16 = odt == GNNFD_BF16;
    // Four columns leave as one 16-byte store where rows and heads start on such boundaries (then every vector of z, which is inside one
    // head, is stored whole or, in fours, not at all).  Stored one by one they touched every sector eight times: [200,000, 8 x 8] fp32,
    // 3.2 M entries, 140 -> 118 us; [100,000, 6 x 8], 2.1 M entries, 83 -> 69; [60,000, 8 x 16] bf16, 6 M entries, 187 -> 173.
    a.out_vec_ok = odt == GNNFD_F32 && (uintptr_t)d_out % 16 == 0 && ldo % 4 == 0 && out_dim % 4 == 0;
    // 32-byte loads of a lane's vector pair need every pair to start on a 32-byte boundary
    a.wide_ok = vec && vpl == 2 && ((uintptr_t)d_z % 32 == 0) && ((ldz * zsize) % 32 == 0) &&
                (n_chunks == 1 || (cw * zsize) % 32 == 0);

    const int per_step = kLoads / vpl * (32 / lpr);
    const int64_t limit = walk_limit(csr, per_step, a.n_ctiles);
    const int64_t blocks = plan_ranges(csr, gather_groups(), lpr, per_step, limit, a.range, &a.n_ranges);
    a.blocks_per_tile = (int32_t)blocks;
    const int64_t grid_x = blocks * a.n_ctiles;
    if (grid_x > 0x7fffffffll) return GNNFD_TOO_LARGE;
    if (grid_x > 0) {
        bool shared = false;
        for (int i = 0; i < a.n_ranges; ++i) shared = shared || a.range[i].warps_log2 > 0;
        GatKernel kernel;
        if (zdt == GNNFD_F32) kernel = vec ? pick_vpl<float, 4>(lpr, vpl, shared) : pick_vpl<float, 1>(lpr, vpl, shared);
        else kernel = vec ? pick_vpl<__nv_bfloat16, 8>(lpr, vpl, shared) : pick_vpl<__nv_bfloat16, 1>(lpr, vpl, shared);
        for (int c0 = 0; c0 < n_chunks; c0 += kMaxGridY) {
            a.chunk_base = c0;
            const dim3 grid((unsigned)grid_x, (unsigned)(n_chunks - c0 < kMaxGridY ? n_chunks - c0 : kMaxGridY));
            GNNFD_LAUNCH("gat_aggregate", s, kernel, grid, kBlock, 0, a);
        }
    }
    const int64_t n_hub = csr->bin_count[4];
    if (n_hub > 0) {
        dim3 gr((unsigned)n_hub, (unsigned)((f + kReduceCols - 1) / kReduceCols));
        GNNFD_LAUNCH("gat_hub_reduce", s, gat_hub_reduce, gr, kBlock, 0, csr->row_order, csr->hub_seg_ptr, g.partial,
                     g.partial_ml, csr->bin_start[4], (int32_t)n_hub, f, a.fpad, heads, dim, out_dim, d_out, ldo, a.out_bf16);
    }
    GNNFD_CUDA_CHECK(cudaGetLastError());
    return GNNFD_OK;
}

// where gnnfd_aggregate_gat keeps the two [n, heads] score arrays inside its scratch buffer
int gat_scratch_scores(const gnnfd_csr_t* csr, int32_t heads, int32_t dim, void* d_scratch, size_t scratch_bytes,
                       float** s_src, float** s_dst)
{
    if (!csr || heads <= 0 || dim <= 0 || !d_scratch || ((uintptr_t)d_scratch & 255u)) return GNNFD_INVALID_ARG;
    Carver c(d_scratch, scratch_bytes);
    GatScratch g;
    carve_gat(c, csr, heads, dim, &g);
    if (!c.ok) return GNNFD_WORKSPACE_TOO_SMALL;
    *s_src = g.s_src;
    *s_dst = g.s_dst;
    return GNNFD_OK;
}

}  // namespace gnnfd

extern "C" {

int gnnfd_gat_scores(int64_t n, const void* d_z, int64_t ldz, gnnfd_dtype_t zdt, const float* d_a_src, const float* d_a_dst,
                     int32_t heads, int32_t dim, float* d_s_src, float* d_s_dst, void* stream)
{
    if (n <= 0 || !d_z || !d_a_src || !d_a_dst || !d_s_src || !d_s_dst || heads <= 0 || dim <= 0 ||
        ldz < (int64_t)heads * dim)
        return GNNFD_INVALID_ARG;
    if (zdt != GNNFD_F32 && zdt != GNNFD_BF16) return GNNFD_UNSUPPORTED;
    if (n * heads > 0x7fffffffll * gnnfd::kBlock) return GNNFD_TOO_LARGE;
    return gnnfd::launch_scores(n, d_z, ldz, zdt, d_a_src, d_a_dst, heads, dim, d_s_src, d_s_dst,
                                static_cast<cudaStream_t>(stream));
}

int gnnfd_gat_workspace_bytes(const gnnfd_csr_t* csr, int32_t heads, int32_t dim, size_t* scratch_bytes)
{
    if (!csr || heads <= 0 || dim <= 0 || !scratch_bytes) return GNNFD_INVALID_ARG;
    gnnfd::Carver c(nullptr, ~size_t(0));
    gnnfd::GatScratch g;
    gnnfd::carve_gat(c, csr, heads, dim, &g);
    *scratch_bytes = c.off;
    return GNNFD_OK;
}

int gnnfd_gat_best_workspace_bytes(const gnnfd_csr_t* csr, const void* d_z, int64_t ldz, gnnfd_dtype_t zdt, int32_t heads,
                                   int32_t dim, int32_t chunk_width, size_t* scratch_bytes)
{
    int rc = gnnfd_gat_workspace_bytes(csr, heads, dim, scratch_bytes);
    if (rc) return rc;
    if (chunk_width <= 0 || (int64_t)heads * dim > 0x7fffffffll || ldz < (int64_t)heads * dim) return GNNFD_INVALID_ARG;
    if (zdt != GNNFD_F32 && zdt != GNNFD_BF16) return GNNFD_UNSUPPORTED;
    *scratch_bytes += gnnfd::gat_copy_bytes(csr, d_z, ldz, zdt, heads, dim, chunk_width);
    return GNNFD_OK;
}

int gnnfd_aggregate_gat(const gnnfd_csr_t* csr, const void* d_z, int64_t ldz, gnnfd_dtype_t zdt, const float* d_a_src,
                        const float* d_a_dst, int32_t heads, int32_t dim, float negative_slope, void* d_out, int64_t ldo,
                        gnnfd_dtype_t odt, int32_t chunk_width, void* d_scratch, size_t scratch_bytes, void* stream)
{
    return gnnfd::gat_aggregate_impl(csr, d_z, ldz, zdt, d_a_src, d_a_dst, heads, dim, negative_slope, d_out, ldo, odt,
                                     chunk_width, d_scratch, scratch_bytes, false, static_cast<cudaStream_t>(stream));
}

}  // extern "C"
