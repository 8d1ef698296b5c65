// Device CSR-by-destination builder: digit histograms of the (dst, src) keys, stable LSD radix sort with one
// sweep per digit, duplicate removal, row pointers, degree normalisers, GCN edge weights and the launch
// schedule (degree bins, hub segments).  Integer work throughout; the only host synchronisation is the
// final read of the counters.
#include <cstddef>
#include <cstring>
#include <new>
#include <type_traits>

#include "common.cuh"

namespace gnnfd {

using u64 = unsigned long long;

constexpr int kThreads = 256;
constexpr int kMaxDigitBits = 9;
constexpr int kRadix = 1 << kMaxDigitBits;           // histogram bins (a pass may use fewer)
constexpr int kSmCount = 148;

static inline unsigned blocks_for(size_t count, int per_block)
{
    size_t b = (count + per_block - 1) / per_block;
    return (unsigned)(b ? b : 1);
}

// ------------------------------------------------------------------ keys

// Candidate i < e: input edge i.  e <= i < 2e (symmetrise): reverse of edge i - e.  Then one
// self-loop per vertex (value -1).  key = (dst << src_bits) | src; dropped candidates get the
// destination n, above every valid key, so the sort moves them behind the kept ones.  When key and
// value fit one 64-bit word together (val_bits > 0) the word is key << val_bits | (value + 1) and
// every later kernel reads the key as word >> val_bits.  Candidates are never written out as such: the
// histogram kernel and the first sweep both form them from the edge list.
struct Candidates {
    const void* src;
    const void* dst;
    int64_t n, e, m;
    uint32_t flags;
    int src_bits;
};

template <typename IdT>
__device__ __forceinline__ u64 edge_key(const Candidates& c, IdT s, IdT d, bool reverse, bool* kept, bool* bad)
{
    using U = typename std::make_unsigned<IdT>::type;              // negative ids are above n too
    *bad = (U)s >= (U)c.n || (U)d >= (U)c.n;
    *kept = !*bad && !((reverse || (c.flags & GNNFD_CSR_ADD_SELF_LOOPS)) && s == d);
    return *kept ? ((u64)d << c.src_bits) | (u64)s : (u64)c.n << c.src_bits;
}

// `count` candidates from `first` on that are reverses of input edges alone: their loads are issued together, like those of the edges.  One at a
// time through candidate_key, builds of RMAT 2^21 / 2^19 took 6.69 / 3.38 ms instead of 6.38 / 3.24.
__device__ __forceinline__ bool inside_reverses(const Candidates& c, int64_t first, int64_t count)
{
    return (c.flags & GNNFD_CSR_SYMMETRIZE) && first >= c.e && first + count <= 2 * c.e;
}

// key and value of candidate i < m
template <typename IdT>
__device__ __forceinline__ u64 candidate_key(const Candidates& c, int64_t i, int32_t* val, bool* kept, bool* bad)
{
    const IdT* src = static_cast<const IdT*>(c.src);
    const IdT* dst = static_cast<const IdT*>(c.dst);
    *val = (int32_t)i;
    if (i < c.e) return edge_key<IdT>(c, __ldcs(src + i), __ldcs(dst + i), false, kept, bad);
    const int64_t n_rev = (c.flags & GNNFD_CSR_SYMMETRIZE) ? c.e : 0;
    if (i < c.e + n_rev) {
        const u64 key = edge_key<IdT>(c, __ldcs(dst + i - c.e), __ldcs(src + i - c.e), true, kept, bad);
        *bad = false;                                  // counted once, by the edge itself
        return key;
    }
    const u64 v = (u64)(i - c.e - n_rev);
    *val = -1;
    *kept = true;
    *bad = false;
    return (v << c.src_bits) | v;
}

// Digit counts of every pass, the number of kept candidates and of bad ids, in one read of the edge list.  The
// grid is a few blocks per SM that walk the list, so that the counters are flushed with few global atomics.
constexpr int kHistItems = 8;                        // candidates per thread and step
constexpr int kHistTile = kThreads * kHistItems;

template <typename IdT, int PASSES>
__global__ void __launch_bounds__(kThreads)
edge_histograms(const __grid_constant__ Candidates c, int first_bit, int digit_bits, int n_passes, int32_t* __restrict__ hist,
                BuildCounts* __restrict__ counts)
{
    const int passes = PASSES > 0 ? PASSES : n_passes;
    grid_dependency<true>();
    extern __shared__ int32_t hist_smem[];           // [passes][kRadix]
    for (int i = threadIdx.x; i < passes * kRadix; i += kThreads) hist_smem[i] = 0;
    __syncthreads();
    const unsigned mask = (1u << digit_bits) - 1u;
    int n_kept = 0, n_bad = 0;
    auto count = [&](u64 key) {
        key >>= first_bit;
#pragma unroll
        for (int p = 0; p < passes; ++p, key >>= digit_bits) atomicAdd(&hist_smem[p * kRadix + ((unsigned)key & mask)], 1);
    };
    const IdT* src = static_cast<const IdT*>(c.src);
    const IdT* dst = static_cast<const IdT*>(c.dst);
    for (int64_t base = (int64_t)blockIdx.x * kHistTile; base < c.m; base += (int64_t)gridDim.x * kHistTile) {
        const bool reverse = inside_reverses(c, base, kHistTile);
        if (reverse || base + kHistTile <= c.e) {
            // edges or reverses alone: all loads are issued before the first shared-memory atomic
            IdT sv[kHistItems], dv[kHistItems];
            const int64_t at = base + threadIdx.x - (reverse ? c.e : 0);
            const IdT* const s0 = (reverse ? dst : src) + at;
            const IdT* const d0 = (reverse ? src : dst) + at;
#pragma unroll
            for (int j = 0; j < kHistItems; ++j) {
                sv[j] = __ldcs(s0 + j * kThreads);
                dv[j] = __ldcs(d0 + j * kThreads);
            }
#pragma unroll
            for (int j = 0; j < kHistItems; ++j) {
                bool kept, bad;
                const u64 key = edge_key<IdT>(c, sv[j], dv[j], reverse, &kept, &bad);
                n_kept += kept;
                n_bad += bad && !reverse;              // counted once, by the edge itself
                count(key);
            }
        } else {
#pragma unroll 2
            for (int j = 0; j < kHistItems; ++j) {
                const int64_t i = base + j * kThreads + threadIdx.x;
                if (i >= c.m) break;
                int32_t val;
                bool kept, bad;
                const u64 key = candidate_key<IdT>(c, i, &val, &kept, &bad);
                n_kept += kept;
                n_bad += bad;
                count(key);
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * kRadix; i += kThreads)
        if (hist_smem[i]) atomicAdd(hist + i, hist_smem[i]);
    n_kept = __reduce_add_sync(0xffffffffu, n_kept);
    n_bad = __reduce_add_sync(0xffffffffu, n_bad);
    if ((threadIdx.x & 31) == 0) {
        if (n_kept) atomicAdd(&counts->n_valid, n_kept);
        if (n_bad) atomicAdd(&counts->bad_index, n_bad);
    }
}

// ------------------------------------------------------------------ radix sort (one digit of up to 9 bits per sweep)
//
// A sweep reads every key once and writes it once to its place in the order of the digit.  A block takes a tile
// of keys, ranks them, publishes how many keys of each digit value it holds, and finds out how many the tiles
// before it hold by walking back over their published counts until it meets one that already knows its own sum
// (a chained scan with look-back, after Merrill and Garland's single-pass scan).  A histogram, a scan and a scatter per digit
// would read the keys once more and take four more launches.
//
// The walk waits for other blocks, but only for tiles with a smaller number, and tile numbers are drawn from a
// counter by blocks that are already running: tile 0 never waits, and every tile publishes its own counts before it
// waits, so some waiting block can always go on.  The wait is limited all the same: a block that polls one
// word kMaxPolls times marks the build as failed and leaves, the others follow, and the host returns
// GNNFD_CUDA_ERROR.  The launches after it are queued already and would take partly unwritten keys, so every kernel that
// works on the sort's results looks at the mark first and does nothing.

// A published word: 0 nothing yet; count + 1: the tile's own count; kSumBit | sum: keys of this digit value in all tiles
// up to and including this one, plus the keys of smaller digit values (so the sum is a position).
constexpr uint32_t kSumBit = 0x80000000u;
constexpr int kMaxPolls = 1 << 20;                   // at up to 1 us a poll

__device__ __forceinline__ uint32_t load_published(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void publish(uint32_t* p, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

// position of the tile's first key of one digit value: `column` points at the digit's word of tile 0, the chain starts at first_tile, words of
// consecutive tiles are kRadix apart; kWalk of them are read together.  false: gave up.
template <int kWalk>
__device__ __forceinline__ bool look_back(const uint32_t* column, int64_t tile, int64_t first_tile, int max_polls, const int32_t* failed, uint32_t* before)
{
    uint32_t sum = 0;
    int polls = 0;
    for (int64_t t = tile - 1; t >= first_tile;) {
        uint32_t w[kWalk];
#pragma unroll
        for (int i = 0; i < kWalk; ++i) w[i] = t - i >= first_tile ? load_published(column + (t - i) * kRadix) : 0u;
        int used = 0;
#pragma unroll
        for (int i = 0; i < kWalk; ++i) {
            if (used == i && w[i] != 0u) {
                if (w[i] & kSumBit) { *before = sum + (w[i] & ~kSumBit); return true; }
                sum += w[i] - 1u;
                ++used;
            }
        }
        t -= used;
        if (used == 0 && (++polls & 255) == 0 && (polls >= max_polls || load_published(reinterpret_cast<const uint32_t*>(failed)) != 0u))
            return false;
    }
    *before = sum;
    return true;
}

// exclusive scan of one value per thread over a block of up to 1024 threads; *total receives the block sum.
// smem[32] must not be in use by a scan that another thread may still be reading.
__device__ __forceinline__ int32_t block_scan(int32_t v, int32_t* total, int32_t* smem)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) smem[warp] = inc;
    __syncthreads();
    const int32_t sums = lane < (int)(blockDim.x >> 5) ? smem[lane] : 0;       // every warp adds up the warps before it
    *total = __reduce_add_sync(0xffffffffu, sums);
    return __reduce_add_sync(0xffffffffu, lane < warp ? sums : 0) + inc - v;
}

enum Source { kWords, kEdges32, kEdges64, kRows, kBucketWords };    // where a sweep takes its keys from
enum Output { kToWords, kToEntries, kToBuckets, kToKeys };          // what it writes: words (and values apart), entries, see below

// Keys and values that do not share a 64-bit word: the sort of a large input starts with the HIGHEST digit of the destination
// (kToBuckets).  It is the same for all words of the bucket they land in and need not be stored, and what is left fits one word with its value.  The
// other digits follow from the lowest up, each bucket by itself (kBucketWords): a tile lies in one bucket, its walk ends at the
// bucket's first tile, and every bucket has digit counts of its own, taken after the first sweep (bucket_histograms).  The last sweep puts
// the highest digit back and writes keys and values apart (kToKeys).  Sweeps of 8 + 4 bytes a key instead: RMAT 2^21, 122 M candidates 5.55 ms
// against 4.62 and 0.26 for the histograms.
constexpr int kBuckets = kRadix;
struct BucketTables {              // filled by bucket_tables
    int32_t first[kBuckets + 1];   // position of each bucket's first word, and their number
    int32_t tile[kBuckets + 1];    // number of its first tile, and of all tiles
};

// The degrees of a sorted list's rows: lanes hold consecutive entries, the first of each run of one destination adds the run's length.
// All lanes take part; `ok`: the lane holds an entry.
__device__ __forceinline__ void count_runs(uint32_t dst, bool ok, int32_t* __restrict__ degree)
{
    const int lane = threadIdx.x & 31;
    const uint32_t before = __shfl_up_sync(0xffffffffu, dst, 1);
    const unsigned present = __ballot_sync(0xffffffffu, ok);                     // the first so many lanes
    const bool first = ok && (lane == 0 || dst != before);
    const unsigned later = __ballot_sync(0xffffffffu, first) & ~((2u << lane) - 1u);
    const int end = later ? __ffs(later) - 1 : __popc(present);
    if (first) atomicAdd(degree + dst, end - lane);
}

struct SweepArgs {
    Candidates cand;               // kEdges*: the edge list (first sweep)
    const u64* keys_in;            // kWords
    const int32_t* vals_in;        // kWords, values apart from the keys
    const int32_t* row_ptr;        // kRows: the keys are the rows' degree classes
    u64* keys_out;
    int32_t* vals_out;             // values apart from the keys; kRows: the row ids
    int out_val_bits;              // kToBuckets: values of this many bits join the keys' low_bits lowest ones
    int low_bits;
    const BucketTables* buckets;   // kBucketWords; a bucket's digit counts are bucket_pitch from the next one's
    int bucket_pitch;
    int32_t* col_out;              // kToEntries: the finished entries and the rows' degrees (zeroed)
    int32_t* degree;
    int64_t m;
    int n_tiles;
    int shift, mask, val_bits;
    const int32_t* digit_count;    // [kRadix] keys per digit value
    int32_t* ticket;               // next tile number
    uint32_t* published;           // [tiles][kRadix], all 0
    uint32_t* published_next;      // set to 0 for the next sweep (may be null)
    BuildCounts* counts;
    int max_polls;                 // of one word, before a block gives up
};

// Degree class of a row: exact degree up to 8, then quarter octaves of (deg - 1) up to the hub
// threshold, then one class for hub rows.  Classes are monotone in the degree, so each of the five
// launch bins (<= 8, <= 32, <= 128, <= hub threshold, hub) is a contiguous range of classes.
constexpr int kHubClass = 41;
constexpr int kClassMask = 63;                       // digit values of the row sweep
__device__ __forceinline__ int degree_class(int32_t deg)
{
    if (deg <= kBinDeg0) return deg;
    if (deg > kBinDeg3) return kHubClass;
    const int t = deg - 1;
    const int o = 31 - __clz(t);                       // 3 .. 10
    return 9 + (o - 3) * 4 + ((t >> (o - 2)) & 3);
}
__device__ __forceinline__ int degree_bin(int32_t deg)
{
    return deg <= kBinDeg0 ? 0 : deg <= kBinDeg1 ? 1 : deg <= kBinDeg2 ? 2 : deg <= kBinDeg3 ? 3 : 4;
}

// Block shapes of a sweep.  Large inputs: 512 threads x 16 keys, two blocks per SM.  Inputs of fewer than 4 such tiles
// per SM: 256 threads x 8 keys, so that more SMs take part.
struct LargeTile { static constexpr int kThreads = 512, kItems = 16, kMinBlocks = 2; };
struct SmallTile { static constexpr int kThreads = 256, kItems = 8, kMinBlocks = 4; };
// Where all tiles run at once none knows its sum yet, and the walks go back over most of them: more words are read together.  220,000
// candidates, 8 / 16 / 32 words: 143 / 145 / 150 us a build.
constexpr int kWalk = 4, kLongWalk = 8;
template <typename Shape> constexpr int tile_keys() { return Shape::kThreads * Shape::kItems; }
constexpr int64_t kSmallInput = (int64_t)4 * kSmCount * tile_keys<LargeTile>();
static bool use_large_tile(int64_t m) { return m >= kSmallInput; }
static int64_t sweep_tiles(int64_t m)
{
    const int keys = use_large_tile(m) ? tile_keys<LargeTile>() : tile_keys<SmallTile>();
    return m > 0 ? (m + keys - 1) / keys : 1;
}
// Tiles to reserve words for: at least those of the largest input in small tiles, where this one is in large tiles, so that
// buffers sized for an input hold every smaller one.
static int64_t reserved_tiles(int64_t m)
{
    constexpr int64_t kMostSmall = (int64_t)4 * kSmCount * tile_keys<LargeTile>() / tile_keys<SmallTile>();
    const int64_t tiles = sweep_tiles(m);
    return use_large_tile(m) && tiles < kMostSmall ? kMostSmall : tiles;
}

template <typename Shape>
struct SweepSmem {
    u64 keys[tile_keys<Shape>()];
    union {
        int32_t warp_count[Shape::kThreads / 32][kRadix];      // keys of a warp per digit value, then their first slot
        int32_t vals[tile_keys<Shape>()];                      // while writing out
    };
    int32_t to_global[kRadix];      // global position of tile slot i holding digit value d: to_global[d] + i
    int32_t scan[32];
    int32_t tile[2];
    int32_t long_run;               // kToEntries: a quarter of the tile's keys have one digit value
};

// The tile a block is at: its keys, the first tile of the chain it belongs to, its bucket (kBucketWords).
struct TilePlace { int64_t base; int count, first_tile, bucket; };

// Ranking: a warp owns 32 * kItems consecutive keys and walks them 32 at a time, with a running count per digit value.
// Rounds are ranked in one of two ways, which load different pipes.  (1) The match instruction gives the lanes
// with the same digit, and the first of them adds their number to the count; the instruction holds its pipe
// for about 56 cycles.  (2) Every lane reads its digit's count and then adds one to it atomically.  A lane whose
// addition found the count as it was read comes first; any other shares its digit with a lane of this round, and
// the order in which the hardware served them says nothing, so those digits (about one per round for random
// keys) are ranked by lane, one ballot each.  Across rounds the running count ranks, across warps a prefix over the
// per-warp counts.  The tile is then laid out sorted by digit in shared memory and written out run by run, so
// that consecutive threads store to consecutive addresses.
//
// Blocks stay and draw one tile after the other; the next tile's keys are requested as soon as this tile's have
// moved to shared memory, so that they arrive while the block walks back and writes out.
//
// Not bound by HBM: 116 M words of 8 bytes on 233 k vertices take 0.74 ms per sweep (2.5 TB/s).  Measured per four sweeps: of every four
// rounds 0 / 1 / 2 / 3 / 4 with the match instruction 3.02 / 3.03 / 3.28 / 3.70 / 4.18 ms (with values of their own,
// 122 M keys, five sweeps: 6.63 / 6.24 / 6.36 / 6.65 / 7.60); 2 / 4 / 8 / 16 earlier tiles read together in the walk 3.11 /
// 2.97 / 3.03 / 3.49 ms; 512 x 8 keys with three blocks per SM 3.69, 256 x 16 with four 3.79 ms.
constexpr int kRankRounds = 4;      // rounds whose counts are in flight together
constexpr int kMatchRounds = 1;     // how many of them use the match instruction

template <typename Shape, int SOURCE, bool HAS_VALS, int OUT>
__global__ void __launch_bounds__(Shape::kThreads, Shape::kMinBlocks) radix_sweep(const __grid_constant__ SweepArgs a)
{
    grid_dependency<(Shape::kMinBlocks > 2)>();
    constexpr int kBlock = Shape::kThreads, kItems = Shape::kItems, kWarps = kBlock / 32, kTile = kBlock * kItems;
    constexpr int kOwn = kRadix / kBlock;            // digit values a thread looks after
    static_assert(kRadix % kBlock == 0 && kTile <= kWarps * kRadix, "digit values per thread; values fit the counts' place");
    static_assert(kItems % kRankRounds == 0 && kTile <= 1 << 16, "rounds; 16-bit slots");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SweepSmem<Shape>& sm = *reinterpret_cast<SweepSmem<Shape>*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int in_tile = warp * (32 * kItems) + lane;       // key r of this thread: in_tile + r * 32 within its tile
    constexpr bool BUCKETS = SOURCE == kBucketWords;
    static_assert(!(BUCKETS || OUT == kToBuckets) || HAS_VALS == (OUT == kToBuckets), "values inside the words of the buckets");
    BucketTables& tables = *reinterpret_cast<BucketTables*>(&sm + 1);        // BUCKETS only
    u64 key[kItems];

    auto load_keys = [&](int64_t base, int count) {
        const int64_t first = base + in_tile;
        if constexpr (SOURCE == kWords || BUCKETS) {
            if (count == kTile) {
#pragma unroll
                for (int r = 0; r < kItems; ++r) key[r] = __ldcs(a.keys_in + first + r * 32);
            } else {
#pragma unroll
                for (int r = 0; r < kItems; ++r) key[r] = in_tile + r * 32 < count ? __ldcs(a.keys_in + first + r * 32) : 0ull;
            }
        } else if constexpr (SOURCE == kRows) {
#pragma unroll
            for (int r = 0; r < kItems; ++r) {
                const int64_t v = first + r * 32;
                key[r] = v < a.m ? ((u64)degree_class(a.row_ptr[v + 1] - a.row_ptr[v]) << 32) | (u64)v : 0ull;
            }
        } else {
            using IdT = typename std::conditional<SOURCE == kEdges32, int32_t, long long>::type;
            auto word = [&](u64 k, int32_t val) { return HAS_VALS || a.val_bits == 0 ? k : (k << a.val_bits) | (u64)(uint32_t)(val + 1); };
            bool kept, bad;
            const bool reverse = inside_reverses(a.cand, base, kTile);
            if (reverse || base + kTile <= a.cand.e) {        // edges or reverses alone: straight-line loads
                const IdT* const src = static_cast<const IdT*>(reverse ? a.cand.dst : a.cand.src) + (reverse ? first - a.cand.e : first);
                const IdT* const dst = static_cast<const IdT*>(reverse ? a.cand.src : a.cand.dst) + (reverse ? first - a.cand.e : first);
#pragma unroll
                for (int r = 0; r < kItems; ++r)
                    key[r] = word(edge_key<IdT>(a.cand, __ldcs(src + r * 32), __ldcs(dst + r * 32), reverse, &kept, &bad), (int32_t)(first + r * 32));
            } else {
#pragma unroll
                for (int r = 0; r < kItems; ++r) {
                    int32_t val;
                    key[r] = 0ull;
                    if (first + r * 32 < a.m) {
                        const u64 k = candidate_key<IdT>(a.cand, first + r * 32, &val, &kept, &bad);
                        key[r] = word(k, val);
                    }
                }
            }
        }
    };
    auto clear_counts = [&]() {
        for (int i = tid; i < kWarps * kRadix / 4; i += kBlock) reinterpret_cast<int4*>(&sm.warp_count[0][0])[i] = make_int4(0, 0, 0, 0);
    };

    int n_tiles = a.n_tiles;
    if constexpr (BUCKETS) {
        for (int i = tid; i <= kBuckets; i += kBlock) {
            tables.first[i] = a.buckets->first[i];
            tables.tile[i] = a.buckets->tile[i];
        }
        __syncthreads();
        n_tiles = tables.tile[kBuckets];
    }
    auto place_of = [&](int t) {
        if constexpr (!BUCKETS) return TilePlace{(int64_t)t * kTile, (int)min((int64_t)kTile, a.m - (int64_t)t * kTile), 0, 0};
        int lo = 0, hi = kBuckets;                   // the last bucket whose first tile is not after t
        while (hi - lo > 1) {
            const int mid = (lo + hi) / 2;
            if (tables.tile[mid] <= t) lo = mid; else hi = mid;
        }
        const int64_t base = (int64_t)tables.first[lo] + (int64_t)(t - tables.tile[lo]) * kTile;
        return TilePlace{base, (int)min((int64_t)kTile, tables.first[lo + 1] - base), tables.tile[lo], lo};
    };
    if (tid == 0) {
        const int first = atomicAdd(a.ticket, 1);
        sm.tile[0] = load_published(reinterpret_cast<const uint32_t*>(&a.counts->sort_failed)) ? n_tiles : first;
    }
    clear_counts();
    __syncthreads();
    int tile = sm.tile[0];
    if (tile >= n_tiles) return;
    TilePlace place = place_of(tile);
    load_keys(place.base, place.count);

    for (int turn = 1;; turn ^= 1) {
        if (tid == 0) {
            sm.tile[turn] = atomicAdd(a.ticket, 1);
            sm.long_run = 0;
        }
        const int64_t tile_base = place.base;
        const int count = place.count, first_tile = place.first_tile, bucket = place.bucket;
        uint32_t* const published = a.published + (int64_t)tile * kRadix;
        if (a.published_next)
            for (int i = tid; i < kRadix / 4; i += kBlock)
                reinterpret_cast<uint4*>(a.published_next + (int64_t)tile * kRadix)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (OUT == kToBuckets && tile < kBuckets)    // every bucket may end in a tile that is not full: as many more words
            for (int i = tid; i < kRadix / 4; i += kBlock)
                reinterpret_cast<uint4*>(a.published_next + (int64_t)(n_tiles + tile) * kRadix)[i] = make_uint4(0u, 0u, 0u, 0u);

        uint32_t rank[kItems / 2];                   // two 16-bit numbers per register
        int32_t* const warp_count = sm.warp_count[warp];
#pragma unroll
        for (int r0 = 0; r0 < kItems; r0 += kRankRounds) {
            int digit[kRankRounds];
            int32_t before[kRankRounds], mine[kRankRounds];
#pragma unroll
            for (int g = 0; g < kRankRounds; ++g) {
                const bool valid = in_tile + (r0 + g) * 32 < count;
                digit[g] = valid ? (int)(key[r0 + g] >> a.shift) & a.mask : -1;
                if (g < kMatchRounds) {
                    const unsigned same = __match_any_sync(0xffffffffu, digit[g]);
                    mine[g] = 0;
                    if (valid && lane == __ffs(same) - 1) mine[g] = atomicAdd(warp_count + digit[g], __popc(same));
                    before[g] = (int32_t)same;
                } else {
                    before[g] = valid ? *(volatile int32_t*)(warp_count + digit[g]) : 0;
                    __syncwarp();
                    mine[g] = valid ? atomicAdd(warp_count + digit[g], 1) : 0;
                }
                __syncwarp();
            }
#pragma unroll
            for (int g = 0; g < kRankRounds; ++g) {
                const unsigned lower = (1u << lane) - 1u;
                if (g < kMatchRounds) {
                    const unsigned same = (unsigned)before[g];
                    mine[g] = __shfl_sync(0xffffffffu, mine[g], __ffs(same) - 1) + __popc(same & lower);
                } else {
                    unsigned shared = __ballot_sync(0xffffffffu, mine[g] != before[g]);
                    while (shared) {
                        const int d = __shfl_sync(0xffffffffu, digit[g], __ffs(shared) - 1);
                        const unsigned same = __ballot_sync(0xffffffffu, digit[g] == d);
                        if (digit[g] == d) mine[g] = before[g] + __popc(same & lower);
                        shared &= ~same;
                    }
                }
                const int r = r0 + g;
                rank[r / 2] = r & 1 ? rank[r / 2] | ((uint32_t)mine[g] << 16) : (uint32_t)mine[g];
            }
        }
        __syncthreads();
        const int next = sm.tile[turn];
        // the tile's totals are published at once; the walk back over the earlier tiles comes after the keys
        // have moved to their slots
        int32_t total[kOwn], base[kOwn], carry = 0;
#pragma unroll
        for (int q = 0; q < kOwn; ++q) {
            total[q] = 0;
            if (q * kBlock > a.mask) continue;       // no such digit in this sweep
#pragma unroll
            for (int w = 0; w < kWarps; ++w) total[q] += sm.warp_count[w][tid + q * kBlock];
            if (tile > first_tile) publish(published + tid + q * kBlock, (uint32_t)total[q] + 1u);
            if (OUT == kToEntries && total[q] >= kTile / 4) sm.long_run = 1;
        }
#pragma unroll
        for (int q = 0; q < kOwn; ++q) {
            int32_t sum;
            if (q * kBlock > a.mask) continue;
            if (q) __syncthreads();
            base[q] = block_scan(total[q], &sum, sm.scan) + carry;
            carry += sum;
            int32_t run = base[q];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const int32_t c = sm.warp_count[w][tid + q * kBlock];
                sm.warp_count[w][tid + q * kBlock] = run;
                run += c;
            }
        }
        if (tile == first_tile) {                    // the only tile that starts from the digit counts of the whole input or bucket
            int32_t smaller = BUCKETS ? tables.first[bucket] : 0;
            const int32_t* const digit_count = a.digit_count + (BUCKETS ? bucket * a.bucket_pitch : 0);
#pragma unroll
            for (int q = 0; q < kOwn; ++q) {
                int32_t sum;
                if (q * kBlock > a.mask) continue;
                __syncthreads();
                const int32_t start = block_scan(digit_count[tid + q * kBlock], &sum, sm.scan) + smaller;
                smaller += sum;
                publish(published + tid + q * kBlock, kSumBit | (uint32_t)(start + total[q]));
                sm.to_global[tid + q * kBlock] = start - base[q];
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kItems; ++r) {
            if (in_tile + r * 32 < count) {
                const uint32_t ahead = (uint32_t)warp_count[(int)(key[r] >> a.shift) & a.mask];
                rank[r / 2] += r & 1 ? ahead << 16 : ahead;              // now the key's slot
                u64 word = key[r];
                if constexpr (OUT == kToBuckets) {
                    const int64_t i = tile_base + in_tile + r * 32, edges = a.cand.e + ((a.cand.flags & GNNFD_CSR_SYMMETRIZE) ? a.cand.e : 0);
                    word = (word & ((1ull << a.low_bits) - 1ull)) << a.out_val_bits | (u64)(i < edges ? i + 1 : 0);
                }
                sm.keys[rank[r / 2] >> (r & 1 ? 16 : 0) & 0xffffu] = word;
            }
        }
        int32_t val[HAS_VALS ? kItems : 1];
        if constexpr (HAS_VALS) {
#pragma unroll
            for (int r = 0; r < kItems; ++r) {
                const int64_t i = tile_base + in_tile + r * 32;
                if constexpr (OUT == kToBuckets) {
                    val[r] = (int)(key[r] >> a.shift) & a.mask;             // the digit, which the word has lost
                } else if constexpr (SOURCE == kWords) {
                    val[r] = in_tile + r * 32 < count ? __ldcs(a.vals_in + i) : 0;
                } else {
                    const int64_t edges = a.cand.e + ((a.cand.flags & GNNFD_CSR_SYMMETRIZE) ? a.cand.e : 0);
                    val[r] = i < edges ? (int32_t)i : -1;
                }
            }
        }
        if (next < n_tiles) place = place_of(next);
        if (!HAS_VALS && next < n_tiles) load_keys(place.base, place.count);
        bool ok = true;
        if (tile > first_tile) {
#pragma unroll
            for (int q = 0; q < kOwn; ++q) {
                const int d = tid + q * kBlock;
                if (d > a.mask) continue;
                uint32_t before = 0;
                const bool together = Shape::kMinBlocks > 2 && n_tiles <= Shape::kMinBlocks * kSmCount;
                if (together ? look_back<kLongWalk>(a.published + d, tile, first_tile, a.max_polls, &a.counts->sort_failed, &before)
                             : look_back<kWalk>(a.published + d, tile, first_tile, a.max_polls, &a.counts->sort_failed, &before))
                    publish(published + d, kSumBit | (before + (uint32_t)total[q]));
                else
                    ok = false;
                sm.to_global[d] = (int32_t)before - base[q];
            }
        }
        if (__syncthreads_or(!ok)) {
            if (tid == 0) atomicExch(&a.counts->sort_failed, 1);
            return;
        }
        if constexpr (HAS_VALS) {                    // the values take the place of the counts, which nobody reads any more
#pragma unroll
            for (int r = 0; r < kItems; ++r)
                if (in_tile + r * 32 < count) sm.vals[rank[r / 2] >> (r & 1 ? 16 : 0) & 0xffffu] = val[r];
            if (next < n_tiles) load_keys(place.base, place.count);
            __syncthreads();
        }
        if constexpr (OUT == kToEntries) {                     // the words are keys alone, and these are their final places
            // the order inside a digit's run is the final one, so the tile's destinations ascend
            const uint32_t src_mask = (uint32_t)((1ull << a.cand.src_bits) - 1ull);
            auto dst_at = [&](int i) { return i < count ? (uint32_t)(sm.keys[i] >> a.cand.src_bits) : 0xffffffffu; };
            auto write = [&](int i, u64 k) {
                const int64_t pos = (int64_t)sm.to_global[(int)(k >> a.shift) & a.mask] + i;
                __stcs(a.col_out + pos, (int32_t)((uint32_t)k & src_mask));
            };
            const uint32_t n = (uint32_t)a.cand.n;                               // dropped candidates have it for a destination and come last
            // An atomic for every 32 entries of a row, all on a few words, made the two sweeps of 40 M entries of 1 / 10 / 1000 rows
            // 1225 / 1310 / 775 us instead of 584 / 665 / 539.  So in a tile with many keys of one digit value, kBlock entries of one row are added
            // together (asked of every tile, 132,534 rows would take 1.5 % longer).
            if (!sm.long_run) {
#pragma unroll 4
                for (int i0 = tid - lane; i0 < count; i0 += kBlock) {
                    const int i = i0 + lane;
                    const u64 k = i < count ? sm.keys[i] : ~0ull;
                    const uint32_t d = (uint32_t)(k >> a.cand.src_bits);
                    const bool ok = i < count && d < n;
                    if (ok) write(i, k);
                    count_runs(d, ok, a.degree);
                }
            } else {
                static_assert(kTile / kBlock <= 32, "a lane for kBlock entries");
                const unsigned whole = __ballot_sync(0xffffffffu, lane < kTile / kBlock && (lane + 1) * kBlock <= count &&
                                                                  dst_at(lane * kBlock) == dst_at((lane + 1) * kBlock - 1));
#pragma unroll 1
                for (int i = tid; i < count; i += kBlock) {
                    const u64 k = sm.keys[i];
                    if ((uint32_t)(k >> a.cand.src_bits) < n) write(i, k);
                }
                if (tid < kTile / kBlock && (whole >> tid & 1u) && dst_at(tid * kBlock) < n) atomicAdd(a.degree + dst_at(tid * kBlock), kBlock);
                for (unsigned rest = ~whole & ((1u << (count + kBlock - 1) / kBlock) - 1u); rest; rest &= rest - 1u) {
                    const uint32_t d = dst_at((__ffs(rest) - 1) * kBlock + tid);
                    count_runs(d, d < n, a.degree);
                }
            }
        } else
#pragma unroll 4
        for (int i = tid; i < count; i += kBlock) {
            const u64 k = sm.keys[i];
            const int64_t pos = (int64_t)sm.to_global[OUT == kToBuckets ? sm.vals[i] : (int)(k >> a.shift) & a.mask] + i;
            if constexpr (SOURCE == kRows) {
                a.vals_out[pos] = (int32_t)(uint32_t)k;
            } else if constexpr (OUT == kToKeys) {
                a.keys_out[pos] = (u64)bucket << a.low_bits | k >> a.val_bits;
                a.vals_out[pos] = (int32_t)(k & ((1ull << a.val_bits) - 1ull)) - 1;
            } else {
                a.keys_out[pos] = k;
                if constexpr (HAS_VALS && OUT != kToBuckets) a.vals_out[pos] = sm.vals[i];
            }
        }
        if (next >= n_tiles) return;
        if constexpr (HAS_VALS) __syncthreads();
        clear_counts();
        tile = next;
        __syncthreads();
    }
}

// The buckets' first words and tiles from the counts of the highest digit; one block.
__global__ void __launch_bounds__(kBuckets)
bucket_tables(const int32_t* count, int tile_keys, BucketTables* __restrict__ tables)
{
    grid_dependency<true>();
    __shared__ int32_t smem[32];
    const int mine = count[threadIdx.x], tiles = (int)(((int64_t)mine + tile_keys - 1) / tile_keys);
    int32_t total;
    tables->first[threadIdx.x] = block_scan(mine, &total, smem);
    if (threadIdx.x == 0) tables->first[kBuckets] = total;
    __syncthreads();
    tables->tile[threadIdx.x] = block_scan(tiles, &total, smem);
    if (threadIdx.x == 0) tables->tile[kBuckets] = total;
}

// Digit counts of every further pass, for every bucket: blocks take runs of consecutive tiles and add to the global counts when they
// come to another bucket.
__global__ void __launch_bounds__(kThreads)
bucket_histograms(const u64* keys, const BucketTables* tables, const BuildCounts* counts, int tile_keys,
                  int first_bit, int digit_bits, int passes, int32_t* __restrict__ hist)
{
    grid_dependency<true>();
    extern __shared__ int32_t hist_smem[];           // [passes][kRadix]
    if (counts->sort_failed) return;
    const int n_tiles = tables->tile[kBuckets], per_block = (n_tiles + gridDim.x - 1) / gridDim.x;
    const int t0 = blockIdx.x * per_block, t1 = min(t0 + per_block, n_tiles);
    if (t0 >= t1) return;
    int bucket = 0;
    for (int step = kBuckets / 2; step > 0; step /= 2)                       // the last bucket whose first tile is not after t0
        if (tables->tile[bucket + step] <= t0) bucket += step;
    const unsigned mask = (1u << digit_bits) - 1u;
    for (int i = threadIdx.x; i < passes * kRadix; i += kThreads) hist_smem[i] = 0;
    __syncthreads();
    for (int t = t0; t < t1;) {
        while (tables->tile[bucket + 1] <= t) ++bucket;                      // empty buckets have no tile
        const int last = min(t1, tables->tile[bucket + 1]);
        const int64_t begin = tables->first[bucket] + (int64_t)(t - tables->tile[bucket]) * tile_keys;
        const int64_t end = min((int64_t)tables->first[bucket + 1], begin + (int64_t)(last - t) * tile_keys);
        for (int64_t at = begin + threadIdx.x; at < end; at += kThreads * kHistItems) {
            u64 word[kHistItems];
#pragma unroll
            for (int j = 0; j < kHistItems; ++j) word[j] = at + j * kThreads < end ? keys[at + j * kThreads] : 0ull;
#pragma unroll
            for (int j = 0; j < kHistItems; ++j) {
                u64 k = word[j] >> first_bit;
                if (at + j * kThreads < end)
                    for (int p = 0; p < passes; ++p, k >>= digit_bits) atomicAdd(&hist_smem[p * kRadix + ((unsigned)k & mask)], 1);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < passes * kRadix; i += kThreads) {
            if (hist_smem[i]) atomicAdd(hist + (int64_t)bucket * passes * kRadix + i, hist_smem[i]);
            hist_smem[i] = 0;
        }
        __syncthreads();
        t = last;
    }
}

// ------------------------------------------------------------------ after the sort

// Duplicate removal after the sort, in two sweeps with a scan of one count per tile between them: a
// sorted candidate is kept when it is valid and its key differs from its predecessor's.  A thread
// looks after kUniqueItems consecutive candidates, a block after kUniqueTile.  (One sweep that chains the tiles' sums, like
// rows_from_degrees, is slower: 122 M candidates in 1.10 ms against 0.77.)
constexpr int kUniqueItems = 8;
constexpr int kUniqueTile = kThreads * kUniqueItems;

__device__ __forceinline__ int64_t sorted_candidates(const BuildCounts* counts) { return counts->sort_failed ? 0 : counts->n_valid; }

// bit j of the result: candidate first + j is the first of a run of equal keys among the n_valid kept ones
__device__ __forceinline__ uint32_t first_of_run_mask(const u64* keys, int64_t first, int64_t n_valid, int val_bits,
                                                      u64 (&word)[kUniqueItems])
{
    u64 prev = first > 0 && first <= n_valid ? (keys[first - 1] >> val_bits) : 0ull;
    if (first + kUniqueItems <= n_valid) {            // whole group present: 16-byte loads (first is a multiple of 8)
        const ulonglong2* k2 = reinterpret_cast<const ulonglong2*>(keys + first);
#pragma unroll
        for (int j = 0; j < kUniqueItems; j += 2) {
            const ulonglong2 v = __ldcs(k2 + j / 2);
            word[j] = v.x;
            word[j + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int j = 0; j < kUniqueItems; ++j) word[j] = first + j < n_valid ? __ldcs(keys + first + j) : 0ull;
    }
    uint32_t mask = 0;
#pragma unroll
    for (int j = 0; j < kUniqueItems; ++j) {
        const int64_t i = first + j;
        const u64 key = word[j] >> val_bits;
        if (i < n_valid && (i == 0 || key != prev)) mask |= 1u << j;
        prev = key;
    }
    return mask;
}

// sum of one value per thread over the block, and the exclusive prefix of this thread's value
__device__ __forceinline__ int32_t block_prefix_256(int32_t v, int32_t* total, int32_t* smem /*[8]*/)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) smem[warp] = inc;
    __syncthreads();
    int32_t off = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        const int32_t t = smem[w];
        if (w < warp) off += t;
        all += t;
    }
    *total = all;
    return off + inc - v;
}

__global__ void __launch_bounds__(kThreads)
unique_tile_counts(const u64* keys, int val_bits, const BuildCounts* counts,
                   int32_t* __restrict__ tile_count)
{
    grid_dependency<true>();
    __shared__ int32_t smem[kThreads / 32];
    u64 word[kUniqueItems];
    const int64_t first = (int64_t)blockIdx.x * kUniqueTile + (int64_t)threadIdx.x * kUniqueItems;
    const int32_t mine = __popc(first_of_run_mask(keys, first, sorted_candidates(counts), val_bits, word));
    int32_t total;
    block_prefix_256(mine, &total, smem);
    if (threadIdx.x == 0) tile_count[blockIdx.x] = total;
}

// tile_first[t] = kept candidates in earlier tiles; the kept ones move to keys_out / perm in order
__global__ void __launch_bounds__(kThreads)
compact_unique(const u64* keys, const int32_t* vals, const int32_t* tile_first,
               int64_t m, int val_bits, u64* __restrict__ keys_out, int32_t* __restrict__ perm,
               BuildCounts* __restrict__ counts)
{
    grid_dependency<false>();
    __shared__ int32_t smem[kThreads / 32];
    __shared__ u64 kept_key[kUniqueTile];
    __shared__ int32_t kept_val[kUniqueTile];
    u64 word[kUniqueItems];
    const int64_t first = (int64_t)blockIdx.x * kUniqueTile + (int64_t)threadIdx.x * kUniqueItems;
    const uint32_t mask = first_of_run_mask(keys, first, sorted_candidates(counts), val_bits, word);
    int32_t total;
    int32_t pos = block_prefix_256(__popc(mask), &total, smem);
    // the kept candidates of the tile are gathered in shared memory so that they leave as one contiguous piece
#pragma unroll
    for (int j = 0; j < kUniqueItems; ++j) {
        if (mask >> j & 1u) {
            kept_key[pos] = word[j];
            kept_val[pos] = vals ? vals[first + j] : (int32_t)(word[j] & ((1ull << val_bits) - 1ull)) - 1;
            ++pos;
        }
    }
    __syncthreads();
    const int32_t out0 = tile_first[blockIdx.x];
    for (int i = threadIdx.x; i < total; i += kThreads) {
        keys_out[out0 + i] = kept_key[i];
        perm[out0 + i] = kept_val[i];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) counts->nnz = tile_first[blockIdx.x] + total;
}

// row_ptr[v] = number of kept keys with dst < v (searched in the sorted keys), then the degree normalisers
// (rounded once from fp64), the bin sizes and the counts of the degree classes.  A block looks after kThreads - 1
// rows, whose pointers and the one behind them its threads search.  Without duplicate removal every kept candidate
// is an entry, which thread 0 records.
constexpr int kRowsPerBlock = kThreads - 1;
constexpr unsigned kSpanBlocks = 4 * 8 * kSmCount;      // several rounds of blocks on every SM
constexpr int kClasses = kHubClass + 1;
static_assert(kClasses <= kClassMask + 1 && kClassMask < kRadix, "digit of the row sweep");

__global__ void __launch_bounds__(kThreads)
rows_and_degrees(const u64* keys, BuildCounts* __restrict__ counts, int64_t n, int src_bits, int val_bits,
                 int dedup, int32_t* __restrict__ row_ptr, float* __restrict__ dinv, float* __restrict__ rdeg,
                 int32_t* __restrict__ class_count)
{
    grid_dependency<true>();
    __shared__ int32_t ptr[kThreads], span[2], class_smem[kClasses], bin_smem[kNumBins], octave_smem[kOctaves], max_smem;
    if (counts->sort_failed) return;
    if (threadIdx.x < kClasses) class_smem[threadIdx.x] = 0;
    if (threadIdx.x < kNumBins) bin_smem[threadIdx.x] = 0;
    if (threadIdx.x < kOctaves) octave_smem[threadIdx.x] = 0;
    if (threadIdx.x == 0) max_smem = 0;
    const int64_t v = (int64_t)blockIdx.x * kRowsPerBlock + threadIdx.x;
    const int32_t nnz = dedup ? counts->nnz : counts->n_valid;
    if (v == 0 && !dedup) counts->nnz = nnz;
    // Many blocks search between the first and the last of their rows, which a warp each finds first, 31 words a step: with all keys to search,
    // threads of vertices without entries all read the same words.  All / between, 33 M vertices, 6.5 M entries into 1000 of
    // them 750 / 349 us, anywhere 777 / 588; 2 M vertices, 8 M entries 52 / 29 and 60 / 58.  With few blocks the extra steps count: 4096 vertices,
    // 40,000 entries 9.6 / 10.7.
    const bool between = gridDim.x > kSpanBlocks;
    if (between && threadIdx.x < 64) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int64_t row = min((int64_t)blockIdx.x * kRowsPerBlock + (warp ? kRowsPerBlock : 0), n);
        const u64 first_key = (u64)row << src_bits;
        int32_t begin = 0, end = nnz;
        while (begin < end) {
            const int32_t step = (end - begin - 1) / 32 + 1;
            const int64_t at = begin + (int64_t)lane * step;
            const int below = __popc(__ballot_sync(0xffffffffu, at < end && (keys[at] >> val_bits) < first_key));    // the first so many lanes
            const int64_t stop = begin + (int64_t)below * step;
            if (stop < end) end = (int32_t)stop;
            begin = below ? begin + (below - 1) * step + 1 : end;
        }
        if (lane == 0) span[warp] = begin;
    }
    if (between) __syncthreads();
    int32_t lo = between && v <= n ? span[0] : 0, hi = v > n ? 0 : between ? span[1] : nnz;
    const u64 target = (u64)v << src_bits;
    // three words a step while there are as many: half as many steps, each of which waits for memory
    while (hi - lo >= 4) {
        const int32_t q = (hi - lo) >> 2;
        bool below[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) below[j] = (keys[lo + (j + 1) * q] >> val_bits) < target;
        const int32_t lo0 = lo;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (below[j]) lo = lo0 + (j + 1) * q + 1;
            else hi = min(hi, lo0 + (j + 1) * q);
        }
    }
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if ((keys[mid] >> val_bits) < target) lo = mid + 1; else hi = mid;
    }
    ptr[threadIdx.x] = lo;
    __syncthreads();
    if (threadIdx.x < kRowsPerBlock && v <= n) row_ptr[v] = lo;      // v == n belongs to the block after the last full one
    if (threadIdx.x < kRowsPerBlock && v < n) {
        const int32_t deg = ptr[threadIdx.x + 1] - lo;
        dinv[v] = deg > 0 ? (float)(1.0 / sqrt((double)deg)) : 0.f;
        rdeg[v] = deg > 0 ? (float)(1.0 / (double)deg) : 0.f;
        atomicAdd(&class_smem[degree_class(deg)], 1);
        atomicAdd(&bin_smem[degree_bin(deg)], 1);
        if (degree_bin(deg) == 3) atomicAdd(&octave_smem[31 - __clz((deg - 1) / kBinDeg2)], 1);
        atomicMax(&max_smem, deg);
    }
    __syncthreads();
    // few global atomics: all blocks add to the same words
    if (threadIdx.x < kClasses && class_smem[threadIdx.x]) atomicAdd(class_count + threadIdx.x, class_smem[threadIdx.x]);
    if (threadIdx.x < kNumBins && bin_smem[threadIdx.x]) atomicAdd(&counts->bin_count[threadIdx.x], bin_smem[threadIdx.x]);
    if (threadIdx.x < kOctaves && octave_smem[threadIdx.x]) atomicAdd(&counts->octave_count[threadIdx.x], octave_smem[threadIdx.x]);
    if (threadIdx.x == 0 && max_smem) atomicMax(&counts->max_degree, max_smem);
}

constexpr int kKeyItems = 4;                          // entries per thread of finalize_entries

// col_idx, the GCN weight and (unless the duplicate removal already wrote it) perm of every slot
__global__ void __launch_bounds__(kThreads)
finalize_entries(const u64* keys, const int32_t* vals, int write_perm,
                 const BuildCounts* counts, int src_bits, int val_bits, const float* dinv,
                 int32_t* __restrict__ col_idx, float* __restrict__ edge_w, int32_t* __restrict__ perm, int64_t m)
{
    grid_dependency<true>();
    const int64_t base = (int64_t)blockIdx.x * (kThreads * kKeyItems) + threadIdx.x;
    const int64_t nnz = counts->sort_failed ? 0 : counts->nnz;
    u64 word[kKeyItems];
#pragma unroll
    for (int j = 0; j < kKeyItems; ++j) {
        const int64_t k = base + j * kThreads;
        word[j] = (k < m && k < nnz) ? __ldcs(keys + k) : 0ull;
    }
    float ws[kKeyItems], wd[kKeyItems];
#pragma unroll
    for (int j = 0; j < kKeyItems; ++j) {
        const u64 key = word[j] >> val_bits;
        ws[j] = dinv[(int32_t)(key & ((1ull << src_bits) - 1ull))];       // 0 for the padding words: in range
        wd[j] = dinv[(int32_t)(key >> src_bits)];
    }
#pragma unroll
    for (int j = 0; j < kKeyItems; ++j) {
        const int64_t k = base + j * kThreads;
        if (k >= m || k >= nnz) continue;
        const u64 key = word[j] >> val_bits;
        __stcs(col_idx + k, (int32_t)(key & ((1ull << src_bits) - 1ull)));
        __stcs(edge_w + k, ws[j] * wd[j]);
        if (write_perm) __stcs(perm + k, vals ? __ldcs(vals + k) : (int32_t)(word[j] & ((1ull << val_bits) - 1ull)) - 1);
    }
}

// ---- entries written by the last sweep itself (ENTRIES), where no words are left to search.  39.6 M edges without ids: the last sweep 310
// instead of 277 us, and 14 us for the rows instead of 28 and 200 for finalize_entries.

// A chain of sums over tiles that are drawn in order (like look_back, one value per tile, 64-bit words): 0 nothing yet, kOwn64 |
// count: the tile's own count, kSum64 | sum: of all tiles up to and including this one.
constexpr u64 kOwn64 = 1ull << 61, kSum64 = 1ull << 62;

// By one whole warp: the sum of all tiles before `tile`, which holds `total` itself; publishes both.  Every lane gets the result,
// or -1: gave up (and the build is marked as failed).
__device__ __forceinline__ int64_t chain_sums(u64* __restrict__ words, int64_t tile, int32_t total, int max_polls, int32_t* failed)
{
    const int lane = threadIdx.x & 31;
    auto store = [&](u64 v) { asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" :: "l"(words + tile), "l"(v) : "memory"); };
    if (lane == 0) store((tile == 0 ? kSum64 : kOwn64) | (u64)(uint32_t)total);
    int64_t before = 0;
    for (int64_t t = tile - 1; t >= 0; t -= 32) {
        u64 w = kSum64;                                // before the first tile: a sum of nothing
        unsigned sums;
        for (int polls = 0;; ++polls) {
            if (t - lane >= 0) asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(words + t - lane) : "memory");
            const unsigned missing = __ballot_sync(0xffffffffu, w == 0ull);
            sums = __ballot_sync(0xffffffffu, (w & kSum64) != 0ull);
            // everything up to the nearest sum is there
            if (missing == 0u || (sums != 0u && (missing & ((sums & (0u - sums)) - 1u)) == 0u)) break;
            if ((polls & 255) == 255 && (polls >= max_polls - 1 || load_published(reinterpret_cast<const uint32_t*>(failed)) != 0u)) {
                if (lane == 0) atomicExch(failed, 1);
                return -1;
            }
        }
        const int nearest = sums ? __ffs(sums) - 1 : 31;
        int64_t part = lane <= nearest ? (int64_t)(w & (kOwn64 - 1ull)) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        before += part;
        if (sums) break;
    }
    if (lane == 0 && tile > 0) store(kSum64 | (u64)(before + total));
    return before;
}

// What rows_and_degrees does, from the degrees: row_ptr is their sums, chained over tiles of rows.  Also (slot_tile_row, unless null), for
// every piece of kSlotTile entries, the row that its first one belongs to, and behind the last piece the row of the last entry.
constexpr int kRowItems = 8;
constexpr int kRowTile = kThreads * kRowItems;
constexpr int kSlotItems = 8;                        // entries per thread of slot_weights
constexpr int kSlotTile = kThreads * kSlotItems;

__global__ void __launch_bounds__(kThreads)
rows_from_degrees(const int32_t* degree, BuildCounts* __restrict__ counts, int64_t n, int32_t* __restrict__ ticket,
                  u64* __restrict__ words, int32_t* __restrict__ row_ptr, float* __restrict__ dinv, float* __restrict__ rdeg,
                  int32_t* __restrict__ class_count, int32_t* __restrict__ slot_tile_row, int max_polls)
{
    grid_dependency<true>();
    __shared__ int32_t smem[kThreads / 32], class_smem[kClasses], bin_smem[kNumBins], octave_smem[kOctaves], max_smem, drawn;
    __shared__ int64_t before;
    if (threadIdx.x == 0) {
        drawn = counts->sort_failed ? -1 : atomicAdd(ticket, 1);
        max_smem = 0;
    }
    if (threadIdx.x < kClasses) class_smem[threadIdx.x] = 0;
    if (threadIdx.x < kNumBins) bin_smem[threadIdx.x] = 0;
    if (threadIdx.x < kOctaves) octave_smem[threadIdx.x] = 0;
    __syncthreads();
    const int tile = drawn;
    if (tile < 0 || (int64_t)tile * kRowTile >= n) return;             // (a drawn number is past the last tile only where the drill left out the first)
    if (tile == 0 && threadIdx.x == 0) counts->nnz = counts->n_valid;
    const int64_t first = (int64_t)tile * kRowTile + threadIdx.x * kRowItems;
    int32_t deg[kRowItems], sum = 0, total;
#pragma unroll
    for (int j = 0; j < kRowItems; ++j) {
        deg[j] = first + j < n ? degree[first + j] : 0;
        sum += deg[j];
    }
    const int32_t in_tile = block_prefix_256(sum, &total, smem);
    if (threadIdx.x < 32) {
        const int64_t start = chain_sums(words, tile, total, max_polls, &counts->sort_failed);
        if (threadIdx.x == 0) before = start;
    }
    int32_t most = 0;
#pragma unroll
    for (int j = 0; j < kRowItems; ++j) {
        const int64_t v = first + j;
        if (v >= n) break;
        dinv[v] = deg[j] > 0 ? (float)(1.0 / sqrt((double)deg[j])) : 0.f;
        rdeg[v] = deg[j] > 0 ? (float)(1.0 / (double)deg[j]) : 0.f;
        atomicAdd(&class_smem[degree_class(deg[j])], 1);
        atomicAdd(&bin_smem[degree_bin(deg[j])], 1);
        if (degree_bin(deg[j]) == 3) atomicAdd(&octave_smem[31 - __clz((deg[j] - 1) / kBinDeg2)], 1);
        most = max(most, deg[j]);
    }
    if (most) atomicMax(&max_smem, most);
    __syncthreads();
    if (before < 0) return;
    const int32_t n_entries = counts->n_valid;
    int32_t ptr = (int32_t)before + in_tile;
#pragma unroll
    for (int j = 0; j < kRowItems; ++j) {
        const int64_t v = first + j;
        if (v < n) row_ptr[v] = ptr;
        if (slot_tile_row) {
            int32_t t = (int32_t)(((int64_t)ptr + kSlotTile - 1) / kSlotTile);
            const int32_t t_end = (int32_t)(((int64_t)ptr + deg[j] + kSlotTile - 1) / kSlotTile);      // t where the row starts no piece
            // many pieces of one row are written by the whole warp: by one thread, those of a row of 40 M entries took 90 us (but 20 pieces each
            // of 1000 neighbouring rows by whole warps 56 instead of 21)
            unsigned many = __ballot_sync(0xffffffffu, t_end - t > 64);
            if (t_end - t <= 64)
                for (; t < t_end; ++t) slot_tile_row[t] = (int32_t)v;
            for (; many; many &= many - 1u) {
                const int from = __ffs(many) - 1;
                const int32_t row = __shfl_sync(0xffffffffu, (int32_t)v, from), end = __shfl_sync(0xffffffffu, t_end, from);
                for (int32_t i = __shfl_sync(0xffffffffu, t, from) + (int)(threadIdx.x & 31); i < end; i += 32) slot_tile_row[i] = row;
            }
            if (deg[j] > 0 && ptr + deg[j] == n_entries) slot_tile_row[t_end] = (int32_t)v;
        }
        ptr += deg[j];
        if (v == n - 1) row_ptr[n] = ptr;
    }
    // few global atomics: all blocks add to the same words
    if (threadIdx.x < kClasses && class_smem[threadIdx.x]) atomicAdd(class_count + threadIdx.x, class_smem[threadIdx.x]);
    if (threadIdx.x < kNumBins && bin_smem[threadIdx.x]) atomicAdd(&counts->bin_count[threadIdx.x], bin_smem[threadIdx.x]);
    if (threadIdx.x < kOctaves && octave_smem[threadIdx.x]) atomicAdd(&counts->octave_count[threadIdx.x], octave_smem[threadIdx.x]);
    if (threadIdx.x == 0 && max_smem) atomicMax(&counts->max_degree, max_smem);
}

// The GCN weight of every entry.  A block takes a piece of kSlotTile consecutive entries: the row starts that fall into it are marked in
// shared memory, and a running maximum gives every entry its row.  Bound by the L1's lookups (one line
// per gathered dinv[source]), like finalize_entries.  Where a piece spans more than kMarkedRows rows, most of them without entries, each
// entry's row is searched instead: marking takes the block 0.3 us per 256 rows while the chip is idle.  2 M vertices, marked / searched:
// 4,000 entries 1150 / 23 us, 200,000 35 / 17, 500,000 20.7 / 18.7, 1 M 18.6 / 20.8, 4 M 31 / 39.
constexpr int kMarkedRows = 3 * kSlotTile;

__global__ void __launch_bounds__(kThreads)
slot_weights(const int32_t* row_ptr, const int32_t* col_idx, const int32_t* slot_tile_row,
             const float* dinv, const BuildCounts* counts, float* __restrict__ edge_w)
{
    grid_dependency<true>();
    __shared__ __align__(16) int32_t row_of[kSlotTile];
    __shared__ int32_t warp_last[kThreads / 32];
    const int64_t nnz = counts->sort_failed ? 0 : counts->nnz, base = (int64_t)blockIdx.x * kSlotTile;
    if (base >= nnz) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t first = base + tid * kSlotItems;
    int32_t u[kSlotItems];
    const bool whole = first + kSlotItems <= nnz;
    if (whole) {
#pragma unroll
        for (int j = 0; j < kSlotItems; j += 4) {
            const int4 v = __ldcs(reinterpret_cast<const int4*>(col_idx + first + j));
            u[j] = v.x; u[j + 1] = v.y; u[j + 2] = v.z; u[j + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < kSlotItems; ++j) u[j] = first + j < nnz ? __ldcs(col_idx + first + j) : 0;
    }
    const int32_t row0 = slot_tile_row[blockIdx.x], row1 = slot_tile_row[blockIdx.x + 1];
    float ws[kSlotItems];
    int32_t row[kSlotItems], earlier = 0;                // counted from row0
    if (row1 - row0 <= kMarkedRows) {
#pragma unroll
        for (int j = 0; j < kSlotItems; j += 4) reinterpret_cast<int4*>(row_of)[tid + j / 4 * kThreads] = make_int4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < kSlotItems; ++j) ws[j] = dinv[u[j]];
        __syncthreads();
        for (int32_t r = row0 + 1 + tid; r <= row1; r += kThreads) {     // empty rows share their start with a later one, which counts
            const int64_t at = row_ptr[r] - base;
            if (at < kSlotTile) atomicMax(&row_of[at], r - row0);
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSlotItems; j += 4) {
            const int4 v = reinterpret_cast<const int4*>(row_of)[(tid * kSlotItems + j) / 4];
            row[j] = v.x; row[j + 1] = v.y; row[j + 2] = v.z; row[j + 3] = v.w;
        }
#pragma unroll
        for (int j = 1; j < kSlotItems; ++j) row[j] = max(row[j], row[j - 1]);
        int32_t upto = row[kSlotItems - 1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) upto = max(upto, __shfl_up_sync(0xffffffffu, upto, o));
        if (lane == 31) warp_last[warp] = upto;
        earlier = __shfl_up_sync(0xffffffffu, upto, 1);
        if (lane == 0) earlier = 0;
        __syncthreads();
        for (int w = 0; w < warp; ++w) earlier = max(earlier, warp_last[w]);
    } else {
#pragma unroll
        for (int j = 0; j < kSlotItems; ++j) {
            ws[j] = dinv[u[j]];
            row[j] = 0;
        }
        // the last row that starts at the entry or before it: the searches of a thread's entries take the same steps side by side
        for (int32_t left = row1 - row0 + 1; left > 1;) {
            const int32_t half = left / 2;
#pragma unroll
            for (int j = 0; j < kSlotItems; ++j)
                if (row_ptr[row0 + row[j] + half] <= first + j) row[j] += half;
            left -= half;
        }
    }
    float w[kSlotItems];
#pragma unroll
    for (int j = 0; j < kSlotItems; ++j) w[j] = ws[j] * dinv[row0 + max(row[j], earlier)];
    if (whole) {
#pragma unroll
        for (int j = 0; j < kSlotItems; j += 4)
            __stcs(reinterpret_cast<float4*>(edge_w + first + j), make_float4(w[j], w[j + 1], w[j + 2], w[j + 3]));
    } else {
#pragma unroll
        for (int j = 0; j < kSlotItems; ++j)
            if (first + j < nnz) __stcs(edge_w + first + j, w[j]);
    }
}

// Hub rows are cut twice: at the boundaries of source ranges of `range_rows` vertex ids (a row's sources are
// ascending, so a range is a contiguous piece of the row) and then into segments of at most GNNFD_HUB_SEGMENT
// entries.  Segments are scheduled range by range (all hub rows' pieces of source range 0, then range 1, ...),
// so the hub rows that are gathered at the same time read the same narrow band of x: a source that several
// hub rows share is fetched from HBM once per sweep instead of once per row.  A segment keeps a second number,
// its slot: slots count a row's segments in ascending source order, row after row, and index the partial
// results, so that the per-row reductions run over a contiguous, ordered slot range.

__device__ __forceinline__ int32_t lower_bound_col(const int32_t* col, int32_t lo, int32_t hi, int64_t bound)
{
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if ((int64_t)col[mid] < bound) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// segments of hub row v per source range (stored `pitch` apart) and altogether
__device__ __forceinline__ int32_t count_row_segments(const int32_t* row_ptr, const int32_t* col_idx,
                                                      int32_t v, int32_t* range_count, int64_t pitch, int32_t n_ranges,
                                                      int64_t range_rows)
{
    int32_t pos = row_ptr[v], total = 0;
    const int32_t e = row_ptr[v + 1];
    for (int32_t r = 0; r < n_ranges; ++r) {
        const int32_t nxt = r == n_ranges - 1 ? e : lower_bound_col(col_idx, pos, e, (int64_t)(r + 1) * range_rows);
        const int32_t c = (nxt - pos + kHubSegment - 1) / kHubSegment;
        range_count[r * pitch] = c;
        total += c;
        pos = nxt;
    }
    return total;
}

// the segments themselves: `slot` is the row's first slot, range_first (`pitch` apart) its first schedule position per range
__device__ __forceinline__ void fill_row_segments(const int32_t* row_ptr, const int32_t* col_idx,
                                                  int32_t v, int32_t slot, const int32_t* range_first, int64_t pitch,
                                                  int32_t n_ranges, int64_t range_rows, int32_t* __restrict__ seg_row,
                                                  int32_t* __restrict__ seg_begin, int32_t* __restrict__ seg_end,
                                                  int32_t* __restrict__ seg_slot)
{
    int32_t pos = row_ptr[v];
    const int32_t e = row_ptr[v + 1];
    for (int32_t r = 0; r < n_ranges; ++r) {
        const int32_t nxt = r == n_ranges - 1 ? e : lower_bound_col(col_idx, pos, e, (int64_t)(r + 1) * range_rows);
        int32_t p = range_first[r * pitch];
        for (int32_t x0 = pos; x0 < nxt; x0 += kHubSegment, ++p, ++slot) {
            seg_row[p] = v;
            seg_begin[p] = x0;
            seg_end[p] = min(x0 + kHubSegment, nxt);
            seg_slot[p] = slot;
        }
        pos = nxt;
    }
}

// per hub row and source range: the number of segments (range-major: count[r * hub_cap + i]) and per hub row
// the total; entries past the last hub row are 0 so that the scans yield the totals
__global__ void __launch_bounds__(kThreads)
hub_segment_counts(const int32_t* row_ptr, const int32_t* col_idx,
                   const int32_t* row_order, int64_t n, const BuildCounts* counts, int64_t hub_cap,
                   int32_t n_ranges, int64_t range_rows, int32_t* __restrict__ range_count, int32_t* __restrict__ seg_count)
{
    grid_dependency<true>();
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i > hub_cap) return;
    const int32_t n_hub = counts->sort_failed ? 0 : counts->bin_count[4];
    int32_t total = 0;
    if (i < n_hub) {
        total = count_row_segments(row_ptr, col_idx, row_order[n - n_hub + i], range_count + i, hub_cap, n_ranges, range_rows);
    } else if (i < hub_cap) {
        for (int32_t r = 0; r < n_ranges; ++r) range_count[(int64_t)r * hub_cap + i] = 0;
    }
    seg_count[i] = total;
    if (i == 0) range_count[(int64_t)n_ranges * hub_cap] = 0;
}

// range_first: exclusive scan of range_count (the schedule position of a row's first segment in a range);
// hub_seg_ptr: exclusive scan of seg_count (the row's first slot)
__global__ void __launch_bounds__(kThreads)
fill_segments(const int32_t* row_ptr, const int32_t* col_idx, const int32_t* row_order,
              int64_t n, BuildCounts* __restrict__ counts, const int32_t* hub_seg_ptr,
              const int32_t* range_first, int64_t hub_cap, int32_t n_ranges, int64_t range_rows,
              int32_t* __restrict__ seg_row, int32_t* __restrict__ seg_begin, int32_t* __restrict__ seg_end,
              int32_t* __restrict__ seg_slot)
{
    grid_dependency<true>();
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int32_t n_hub = counts->sort_failed ? 0 : counts->bin_count[4];
    if (i == 0) counts->n_segments = hub_seg_ptr[n_hub];
    if (i >= hub_cap || i >= n_hub) return;
    fill_row_segments(row_ptr, col_idx, row_order[n - n_hub + i], hub_seg_ptr[i], range_first + i, hub_cap, n_ranges, range_rows,
                      seg_row, seg_begin, seg_end, seg_slot);
}

// The three steps above in one block, for graphs that can have few hub rows (hub_cap * n_ranges up to kFewHubPieces):
// counts, both scans and the fill without a launch in between.
constexpr int kFewHubPieces = 8192;
constexpr int kHubThreads = 1024;

__global__ void __launch_bounds__(kHubThreads)
hub_segments_few(const int32_t* row_ptr, const int32_t* col_idx, const int32_t* row_order,
                 int64_t n, BuildCounts* __restrict__ counts, int32_t n_ranges, int64_t range_rows, int32_t* range_count,
                 int32_t* hub_seg_ptr, int32_t* __restrict__ seg_row, int32_t* __restrict__ seg_begin,
                 int32_t* __restrict__ seg_end, int32_t* __restrict__ seg_slot)
{
    grid_dependency<true>();
    __shared__ int32_t smem[32];
    const int32_t n_hub = counts->sort_failed ? 0 : counts->bin_count[4];
    for (int32_t i = threadIdx.x; i < n_hub; i += kHubThreads)
        hub_seg_ptr[i] = count_row_segments(row_ptr, col_idx, row_order[n - n_hub + i], range_count + i, n_hub, n_ranges, range_rows);
    __syncthreads();
    auto scan_in_place = [&](int32_t* p, int32_t count) {
        int32_t carry = 0;
        for (int32_t base = 0; base < count; base += kHubThreads) {
            const int32_t i = base + threadIdx.x;
            const int32_t mine = i < count ? p[i] : 0;
            int32_t sum;
            const int32_t before = block_scan(mine, &sum, smem) + carry;
            if (i < count) p[i] = before;
            carry += sum;
            __syncthreads();
        }
        return carry;
    };
    const int32_t total = scan_in_place(hub_seg_ptr, n_hub);
    scan_in_place(range_count, n_hub * n_ranges);
    if (threadIdx.x == 0) {
        hub_seg_ptr[n_hub] = total;
        counts->n_segments = total;
    }
    for (int32_t i = threadIdx.x; i < n_hub; i += kHubThreads)
        fill_row_segments(row_ptr, col_idx, row_order[n - n_hub + i], hub_seg_ptr[i], range_count + i, n_hub, n_ranges, range_rows,
                          seg_row, seg_begin, seg_end, seg_slot);
}

// ------------------------------------------------------------------ host side

struct BuildLayout {
    int64_t m;             // candidate edges
    int64_t n_tiles;       // tiles of an edge sweep
    int64_t row_tiles;     // tiles of the row (degree class) sweep
    int64_t tile_cap, row_tile_cap;      // tiles that words are reserved for
    int64_t hub_cap;       // upper bound on hub rows
    int64_t seg_cap;       // upper bound on hub segments
    int range_cap;         // source ranges that words are reserved for
    int src_bits, key_bits, passes, digit_bits;     // passes: sweeps over the edges but the one that makes buckets
    int first_bit;         // lowest key bit the sort looks at (0; src_bits when rows keep their input order)
    int n_ranges;          // source ranges the hub rows are cut at (1: no cut)
    int64_t range_rows;    // vertex ids per source range
    int val_bits;          // > 0: keys and values share one 64-bit word (key << val_bits | value + 1)
    int64_t row_words;     // tiles of rows_from_degrees
    bool with_vals;        // edge ids travel through the sort
    int top_bits;          // > 0: the first sweep takes this many highest bits of the destination and makes buckets of them
    int sweeps() const { return passes + (top_bits > 0); }
};

static void reserve_ranges(BuildLayout* L, int ranges)
{
    L->range_cap = ranges;
    L->seg_cap = L->m / kHubSegment + L->hub_cap * ranges + 1;
}

static int make_layout(int64_t n, int64_t e, uint32_t flags, BuildLayout* L, bool with_vals = true)
{
    if (n <= 0 || e < 0) return GNNFD_INVALID_ARG;
    if (flags & ~(uint32_t)(GNNFD_CSR_ADD_SELF_LOOPS | GNNFD_CSR_DEDUP | GNNFD_CSR_SYMMETRIZE | GNNFD_CSR_INPUT_ORDER))
        return GNNFD_INVALID_ARG;
    // duplicates are found as neighbours of the (dst, src) order, which the input-order build does not establish
    if ((flags & GNNFD_CSR_INPUT_ORDER) && (flags & GNNFD_CSR_DEDUP)) return GNNFD_INVALID_ARG;
    const int64_t limit = (int64_t(1) << 31) - 1;
    if (n > limit || e > limit) return GNNFD_TOO_LARGE;
    int64_t m = e;
    if (flags & GNNFD_CSR_SYMMETRIZE) m += e;
    if (flags & GNNFD_CSR_ADD_SELF_LOOPS) m += n;
    if (m > limit) return GNNFD_TOO_LARGE;
    L->m = m;
    L->n_tiles = sweep_tiles(m);
    L->row_tiles = sweep_tiles(n);
    L->row_tile_cap = reserved_tiles(n);
    L->row_words = (n + kRowTile - 1) / kRowTile;
    L->hub_cap = m / (GNNFD_HUB_DEGREE + 1) + 1;
    // source ranges of GNNFD_HUB_RANGE_ROWS vertices, at most 64 of them (narrower ranges would keep a band of x
    // resident in L2, but on the RMAT workload the extra, shorter segments cost more than the saved traffic: 32
    // ranges cut the gather's DRAM bytes by 27 % and made it 13 % slower, 4 ranges are 3 % faster than none); a row
    // whose sources are not ascending (input-order build) cannot be cut by range
    L->range_rows = GNNFD_HUB_RANGE_ROWS;
    while ((n + L->range_rows - 1) / L->range_rows > 64) L->range_rows <<= 1;
    L->n_ranges = (flags & GNNFD_CSR_INPUT_ORDER) ? 1 : (int)((n + L->range_rows - 1) / L->range_rows);
    // (beyond 2^25 vertices wider ranges are fewer: as many are reserved for as smaller graphs have)
    const int64_t narrow = (n + GNNFD_HUB_RANGE_ROWS - 1) / GNNFD_HUB_RANGE_ROWS;
    reserve_ranges(L, (flags & GNNFD_CSR_INPUT_ORDER) ? 1 : narrow < 64 ? (int)narrow : 64);
    int bits = 1;
    while ((int64_t(1) << bits) < n) ++bits;
    int dst_bits = 1;
    while ((int64_t(1) << dst_bits) < n + 1) ++dst_bits;      // destination n marks dropped candidates
    L->src_bits = bits;
    L->key_bits = bits + dst_bits;
    // Rows in input order: the stable sort looks at the destination bits only, so entries of a row stay in the
    // order of their candidate numbers (input edges, then reverses, then the added loop).
    L->first_bit = (flags & GNNFD_CSR_INPUT_ORDER) ? bits : 0;
    int vb = 1;
    while ((int64_t(1) << vb) < m + 2) ++vb;                  // values -1 .. m-1 stored as 0 .. m
    L->val_bits = L->key_bits + vb <= 64 ? vb : 0;
    // Buckets from where large tiles are used: below, the two launches that they add cost more than the narrower records save.
    const int top = dst_bits < kMaxDigitBits ? dst_bits : kMaxDigitBits;
    const bool buckets = with_vals && L->val_bits == 0 && use_large_tile(m) && L->key_bits - top + vb <= 64 && L->key_bits - top > L->first_bit;
    L->top_bits = buckets ? top : 0;
    if (buckets) L->val_bits = vb;
    const int sort_bits = L->key_bits - L->first_bit - L->top_bits;
    L->passes = (sort_bits + kMaxDigitBits - 1) / kMaxDigitBits;
    L->digit_bits = (sort_bits + L->passes - 1) / L->passes;
    L->tile_cap = reserved_tiles(m) + (buckets ? kBuckets : 0);
    L->with_vals = with_vals;
    return GNNFD_OK;
}

struct PersistentPtrs {
    int32_t *row_ptr, *col_idx, *perm, *row_order, *seg_row, *seg_begin, *seg_end, *seg_slot, *hub_seg_ptr;
    float *edge_w, *dinv, *rdeg;
    BuildCounts* counts;
};

static void carve_persistent(Carver& c, int64_t n, const BuildLayout& L, PersistentPtrs* p)
{
    const size_t cap = (size_t)(L.m > 0 ? L.m : 1);
    p->row_ptr = c.take<int32_t>((size_t)n + 1);
    p->col_idx = c.take<int32_t>(cap);
    p->perm = c.take<int32_t>(cap);
    p->edge_w = c.take<float>(cap);
    p->dinv = c.take<float>((size_t)n);
    p->rdeg = c.take<float>((size_t)n);
    p->row_order = c.take<int32_t>((size_t)n);            // may hold the degrees until the rows are sorted by them
    p->counts = c.take<BuildCounts>(1);
    p->seg_row = c.take<int32_t>((size_t)L.seg_cap);
    p->seg_begin = c.take<int32_t>((size_t)L.seg_cap);
    p->seg_end = c.take<int32_t>((size_t)L.seg_cap);
    p->seg_slot = c.take<int32_t>((size_t)L.seg_cap);
    p->hub_seg_ptr = c.take<int32_t>((size_t)L.hub_cap + 1);
}

struct ScratchPtrs {
    u64 *keys_a, *keys_b;
    int32_t *vals_a, *vals_b, *flags, *scan_temp;
    // zeroed together before the first kernel: digit counts (a row per edge sweep, then the degree classes), tile
    // counters (likewise, then of rows_from_degrees), the words that the tiles of the latter, of the row sweep and of the first edge sweep publish
    int32_t *digit_count, *bucket_count, *ticket;
    u64* row_words;
    BucketTables* buckets;         // not zeroed
    uint32_t *row_published, *published, *published_alt;
    size_t zero_bytes;
};

static size_t flag_ints(const BuildLayout& L)
{
    // one count per tile of the duplicate removal, or a row per piece of the entries; hub segment counts (per source range and hub row, then per hub row)
    static_assert(kUniqueTile == kSlotTile, "one count or one row for as many candidates");
    size_t a = (size_t)L.m / kUniqueTile + 2, c = (size_t)L.hub_cap * (L.range_cap + 1) + 4;
    return (a > c ? a : c) + 1;
}

static void carve_scratch(Carver& c, const BuildLayout& L, ScratchPtrs* p)
{
    const size_t cap = (size_t)(L.m > 0 ? L.m : 1);
    p->keys_a = c.take<u64>(cap);
    p->keys_b = c.take<u64>(cap);
    // No value buffers when the values travel inside the key words.  With buckets one is enough, but the other is as large as the largest
    // input without buckets needs that has fewer candidates.
    const size_t val_cap = !L.with_vals || (L.val_bits > 0 && L.top_bits == 0) ? 1 : cap;
    p->vals_a = c.take<int32_t>(val_cap);
    p->vals_b = c.take<int32_t>(L.top_bits > 0 && (size_t)kSmallInput < val_cap ? (size_t)kSmallInput : val_cap);
    const size_t zero_begin = c.off;
    p->digit_count = c.take<int32_t>((size_t)(L.sweeps() + 1) * kRadix);
    p->bucket_count = c.take<int32_t>(L.top_bits ? (size_t)kBuckets * L.passes * kRadix : 0);
    p->ticket = c.take<int32_t>((size_t)L.sweeps() + 2);
    p->row_words = c.take<u64>((size_t)L.row_words);
    p->row_published = c.take<uint32_t>((size_t)kRadix * L.row_tile_cap);
    p->zero_bytes = c.off - zero_begin + (size_t)kRadix * L.n_tiles * sizeof(uint32_t);
    p->published = c.take<uint32_t>((size_t)kRadix * L.tile_cap);
    p->published_alt = c.take<uint32_t>((size_t)kRadix * L.tile_cap);
    p->buckets = c.take<BucketTables>(L.top_bits ? 1 : 0);
    const size_t fl = flag_ints(L);
    p->flags = c.take<int32_t>(fl);
    p->scan_temp = c.take<int32_t>(scan_temp_ints(fl));
}

// The usual numbers of passes are compiled in: 80 M edges, four digits 199 -> 160 us.
typedef void (*HistogramKernel)(const Candidates, int, int, int, int32_t*, BuildCounts*);
template <typename IdT>
static HistogramKernel histogram_kernel(int passes)
{
    switch (passes) {
        case 1: return edge_histograms<IdT, 1>;
        case 2: return edge_histograms<IdT, 2>;
        case 3: return edge_histograms<IdT, 3>;
        case 4: return edge_histograms<IdT, 4>;
        default: return edge_histograms<IdT, 0>;
    }
}

template <typename Shape, int SOURCE, bool HAS_VALS, int OUT>
static int launch_sweep_shape(const char* name, const SweepArgs& a, cudaStream_t s)
{
    const auto kernel = radix_sweep<Shape, SOURCE, HAS_VALS, OUT>;
    const int blocks = SOURCE != kBucketWords && a.n_tiles < Shape::kMinBlocks * kSmCount ? a.n_tiles : Shape::kMinBlocks * kSmCount;
    const int smem = (int)(sizeof(SweepSmem<Shape>) + (SOURCE == kBucketWords ? sizeof(BucketTables) : 0));
    GNNFD_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    GNNFD_LAUNCH(name, s, kernel, (unsigned)blocks, Shape::kThreads, smem, a);
    return GNNFD_OK;
}

template <int SOURCE, bool HAS_VALS, int OUT>
static int launch_sweep(const char* name, SweepArgs& a, cudaStream_t s)
{
    a.n_tiles = (int)sweep_tiles(a.m);
    return use_large_tile(a.m) ? launch_sweep_shape<LargeTile, SOURCE, HAS_VALS, OUT>(name, a, s)
                               : launch_sweep_shape<SmallTile, SOURCE, HAS_VALS, OUT>(name, a, s);
}

template <int SOURCE>
static int launch_edge_sweep(bool has_vals, bool entries, SweepArgs& a, cudaStream_t s)
{
    if (has_vals) return launch_sweep<SOURCE, true, kToWords>("radix_sweep", a, s);
    return entries ? launch_sweep<SOURCE, false, kToEntries>("radix_sweep", a, s) : launch_sweep<SOURCE, false, kToWords>("radix_sweep", a, s);
}

// One-shot settings of the drill (see gnnfd_debug_build_fault): consumed by the next build on this thread.
struct BuildDrill { int max_polls, sweep; };
static thread_local BuildDrill t_drill = {kMaxPolls, -1};

// need_perm, need_weights: whether the caller looks at perm and edge_w (their places are left as they are where not).  Edge ids that nobody
// needs do not travel through the sort, unless duplicates are removed, where the order among them decides.
int build_csr_impl(int64_t n, int64_t e, const void* d_src, const void* d_dst, gnnfd_itype_t itype, uint32_t flags, bool need_perm,
                   bool need_weights, void* d_persistent, size_t persistent_bytes, void* d_scratch, size_t scratch_bytes, cudaStream_t s,
                   gnnfd_csr_t** out)
{
    const BuildDrill drill = t_drill;
    t_drill = BuildDrill{kMaxPolls, -1};
    if (!out) return GNNFD_INVALID_ARG;
    *out = nullptr;
    BuildLayout L;
    int rc = make_layout(n, e, flags, &L, need_perm || (flags & GNNFD_CSR_DEDUP));
    if (rc) return rc;
    if (itype != GNNFD_I32 && itype != GNNFD_I64) return GNNFD_UNSUPPORTED;
    if ((e > 0 && (!d_src || !d_dst)) || !d_persistent || !d_scratch) return GNNFD_INVALID_ARG;
    if (((uintptr_t)d_persistent | (uintptr_t)d_scratch) & 255u) return GNNFD_INVALID_ARG;

    L.tile_cap = L.n_tiles + (L.top_bits ? kBuckets : 0);      // the query reserves more; what this input needs is enough
    L.row_tile_cap = L.row_tiles;
    reserve_ranges(&L, L.n_ranges);
    Carver pc(d_persistent, persistent_bytes), sc(d_scratch, scratch_bytes);
    PersistentPtrs P;
    ScratchPtrs S;
    carve_persistent(pc, n, L, &P);
    carve_scratch(sc, L, &S);
    if (!pc.ok || !sc.ok) return GNNFD_WORKSPACE_TOO_SMALL;

    // the drill leaves out a sweep's first tile: another one has to be there to miss it, of the same bucket where there are buckets
    if (drill.sweep > 0 && drill.sweep < L.sweeps() && L.top_bits > 0) return GNNFD_INVALID_ARG;
    if (drill.sweep >= 0) {
        const int64_t tiles = drill.sweep < L.sweeps() ? L.n_tiles : drill.sweep == L.sweeps() ? L.row_tiles :
                              drill.sweep == L.sweeps() + 1 && !L.with_vals ? L.row_words : 0;
        if (tiles < 2) return GNNFD_INVALID_ARG;
    }

    const int64_t m = L.m;
    // Without ids the last sweep writes the entries and counts the degrees.  With them it is better to write words once more: 80 M
    // entries 2.86 ms with words, 2.92 without.
    const bool entries = !L.with_vals;
    char* const zero_from = entries ? reinterpret_cast<char*>(P.row_order) : reinterpret_cast<char*>(P.counts);      // the degrees lie before the counts
    GNNFD_CUDA_CHECK(cudaMemsetAsync(zero_from, 0, (size_t)(reinterpret_cast<char*>(P.counts + 1) - zero_from), s));

    BuildCounts host_counts;
    std::memset(&host_counts, 0, sizeof(host_counts));
    u64* keys = S.keys_a;
    u64* keys_alt = S.keys_b;
    int32_t* vals = S.vals_a;
    int32_t* vals_alt = S.vals_b;

    const bool dedup = (flags & GNNFD_CSR_DEDUP) != 0;
    int vb = L.with_vals ? L.val_bits : 0;
    const bool buckets = L.top_bits > 0;
    bool apart = L.with_vals && vb == 0;            // values in arrays of their own, else in the low bits of the keys
    int32_t* const degree = P.row_order;
    GNNFD_CUDA_CHECK(cudaMemsetAsync(S.digit_count, 0, S.zero_bytes, s));
    if (drill.sweep >= 0) GNNFD_CUDA_CHECK(cudaMemsetAsync(S.ticket + drill.sweep, 1, 1, s));      // tile 0 is never drawn
    SweepArgs sw{};
    sw.cand = Candidates{d_src, d_dst, n, e, m, flags, L.src_bits};
    sw.m = m;
    sw.val_bits = vb;
    sw.counts = P.counts;
    sw.col_out = P.col_idx;
    sw.degree = degree;
    sw.max_polls = drill.max_polls;
    sw.n_tiles = (int)L.n_tiles;
    sw.out_val_bits = vb;
    sw.low_bits = L.key_bits - L.top_bits;
    sw.buckets = S.buckets;
    sw.bucket_pitch = L.passes * kRadix;
    if (m > 0) {
        const unsigned walkers = blocks_for(m, kHistTile) < 6u * kSmCount ? blocks_for(m, kHistTile) : 6u * kSmCount;
        // the counts of all digits, or those of the buckets' digit
        const int hist_first = buckets ? L.key_bits - L.top_bits : L.first_bit, hist_bits = buckets ? L.top_bits : L.digit_bits;
        const int hist_passes = buckets ? 1 : L.passes;
        const size_t hist_bytes = (size_t)hist_passes * kRadix * sizeof(int32_t);
        GNNFD_LAUNCH("edge_histograms", s, itype == GNNFD_I32 ? histogram_kernel<int32_t>(hist_passes) : histogram_kernel<long long>(hist_passes),
                     walkers, kThreads, hist_bytes, sw.cand, hist_first, hist_bits, hist_passes, S.digit_count, P.counts);
        uint32_t* published = S.published;
        uint32_t* published_alt = S.published_alt;
        for (int sweep = 0; sweep < L.sweeps(); ++sweep) {
            const bool last = sweep + 1 == L.sweeps();
            const int pass = buckets ? sweep - 1 : sweep;
            sw.shift = L.first_bit + pass * L.digit_bits + vb;
            sw.mask = (1 << L.digit_bits) - 1;
            sw.digit_count = buckets ? S.bucket_count + (size_t)pass * kRadix : S.digit_count + (size_t)pass * kRadix;
            sw.ticket = S.ticket + sweep;
            sw.published = published;
            sw.published_next = last ? nullptr : published_alt;
            sw.keys_in = keys; sw.keys_out = keys_alt;
            sw.vals_in = vals; sw.vals_out = vals_alt;
            if (buckets && sweep == 0) {
                sw.shift = L.key_bits - L.top_bits;
                sw.mask = (1 << L.top_bits) - 1;
                sw.digit_count = S.digit_count;
                rc = itype == GNNFD_I32 ? launch_sweep_shape<LargeTile, kEdges32, true, kToBuckets>("radix_sweep", sw, s)
                                        : launch_sweep_shape<LargeTile, kEdges64, true, kToBuckets>("radix_sweep", sw, s);
                if (rc) return rc;
                GNNFD_LAUNCH("bucket_tables", s, bucket_tables, 1, kBuckets, 0, S.digit_count, tile_keys<LargeTile>(), S.buckets);
                GNNFD_LAUNCH("bucket_histograms", s, bucket_histograms, 6u * kSmCount, kThreads, L.passes * kRadix * sizeof(int32_t), keys_alt,
                             S.buckets, P.counts, tile_keys<LargeTile>(), L.first_bit + vb, L.digit_bits, L.passes, S.bucket_count);
            } else if (buckets) {
                sw.vals_out = S.vals_a;
                rc = last ? launch_sweep_shape<LargeTile, kBucketWords, false, kToKeys>("radix_sweep", sw, s)
                          : launch_sweep_shape<LargeTile, kBucketWords, false, kToWords>("radix_sweep", sw, s);
            } else if (sweep > 0) rc = launch_edge_sweep<kWords>(apart, entries && last, sw, s);
            else if (itype == GNNFD_I32) rc = launch_edge_sweep<kEdges32>(apart, entries && last, sw, s);
            else rc = launch_edge_sweep<kEdges64>(apart, entries && last, sw, s);
            if (rc) return rc;
            u64* tk = keys; keys = keys_alt; keys_alt = tk;
            int32_t* tv = vals; vals = vals_alt; vals_alt = tv;
            uint32_t* tp = published; published = published_alt; published_alt = tp;
        }
        if (buckets) {                                  // from here on as after a sort of keys and values apart
            vals = S.vals_a;
            apart = true;
            vb = 0;
        }
        if (dedup) {
            const unsigned unique_tiles = blocks_for(m, kUniqueTile);
            int32_t* tile_first = S.flags;
            GNNFD_LAUNCH("unique_tile_counts", s, unique_tile_counts, unique_tiles, kThreads, 0, keys, vb, P.counts, tile_first);
            rc = exclusive_scan_i32(tile_first, tile_first, (size_t)unique_tiles, S.scan_temp, s);
            if (rc) return rc;
            GNNFD_LAUNCH("compact_unique", s, compact_unique, unique_tiles, kThreads, 0, keys,
                         apart ? (const int32_t*)vals : (const int32_t*)nullptr, (const int32_t*)tile_first, m, vb, keys_alt,
                         P.perm, P.counts);
            u64* tk = keys; keys = keys_alt; keys_alt = tk;
        }
    }
    int32_t* class_count = S.digit_count + (size_t)L.sweeps() * kRadix;
    if (entries) {
        int32_t* slot_tile_row = need_weights ? S.flags : nullptr;
        GNNFD_LAUNCH("rows_from_degrees", s, rows_from_degrees, (unsigned)L.row_words, kThreads, 0, degree, P.counts, n,
                     S.ticket + L.sweeps() + 1, S.row_words, P.row_ptr, P.dinv, P.rdeg, class_count, slot_tile_row,
                     drill.max_polls);
        if (m > 0 && need_weights)
            GNNFD_LAUNCH("slot_weights", s, slot_weights, blocks_for(m, kSlotTile), kThreads, 0, P.row_ptr, P.col_idx, slot_tile_row,
                         P.dinv, P.counts, P.edge_w);
    } else {
        GNNFD_LAUNCH("rows_and_degrees", s, rows_and_degrees, blocks_for((size_t)n + 1, kRowsPerBlock), kThreads, 0, keys, P.counts, n,
                     L.src_bits, vb, dedup ? 1 : 0, P.row_ptr, P.dinv, P.rdeg, class_count);
        if (m > 0)
            GNNFD_LAUNCH("finalize_entries", s, finalize_entries, blocks_for(m, kThreads * kKeyItems), kThreads, 0, keys,
                         apart ? (const int32_t*)vals : (const int32_t*)nullptr, dedup ? 0 : 1, P.counts, L.src_bits, vb,
                         P.dinv, P.col_idx, P.edge_w, P.perm, m);
    }
    // row_order = rows sorted by degree class, ascending row id inside a class: one sweep over the rows
    sw.row_ptr = P.row_ptr;
    sw.vals_out = P.row_order;
    sw.m = n;
    sw.shift = 32;
    sw.mask = kClassMask;
    sw.digit_count = class_count;
    sw.ticket = S.ticket + L.sweeps();
    sw.published = S.row_published;
    sw.published_next = nullptr;
    rc = launch_sweep<kRows, false, kToWords>("radix_sweep_rows", sw, s);
    if (rc) return rc;
    // segment counts per (source range, hub row), then per hub row
    int32_t* range_count = S.flags;
    if (L.hub_cap * L.n_ranges <= kFewHubPieces) {
        GNNFD_LAUNCH("hub_segments_few", s, hub_segments_few, 1, kHubThreads, 0, P.row_ptr, P.col_idx, P.row_order, n, P.counts,
                     L.n_ranges, L.range_rows, range_count, P.hub_seg_ptr, P.seg_row, P.seg_begin, P.seg_end, P.seg_slot);
    } else {
        int32_t* seg_count = S.flags + (size_t)L.hub_cap * L.n_ranges + 1;
        GNNFD_LAUNCH("hub_segment_counts", s, hub_segment_counts, blocks_for((size_t)L.hub_cap + 1, kThreads), kThreads, 0,
                     P.row_ptr, P.col_idx, P.row_order, n, P.counts, L.hub_cap, L.n_ranges, L.range_rows, range_count, seg_count);
        rc = exclusive_scan_i32(seg_count, P.hub_seg_ptr, (size_t)L.hub_cap + 1, S.scan_temp, s);
        if (rc) return rc;
        rc = exclusive_scan_i32(range_count, range_count, (size_t)L.hub_cap * L.n_ranges + 1, S.scan_temp, s);
        if (rc) return rc;
        GNNFD_LAUNCH("fill_segments", s, fill_segments, blocks_for((size_t)L.hub_cap, kThreads), kThreads, 0, P.row_ptr, P.col_idx,
                     P.row_order, n, P.counts, P.hub_seg_ptr, range_count, L.hub_cap, L.n_ranges, L.range_rows, P.seg_row,
                     P.seg_begin, P.seg_end, P.seg_slot);
    }
    GNNFD_CUDA_CHECK(cudaGetLastError());
    GNNFD_CUDA_CHECK(cudaMemcpyAsync(&host_counts, P.counts, sizeof(BuildCounts), cudaMemcpyDeviceToHost, s));
    GNNFD_CUDA_CHECK(cudaStreamSynchronize(s));

    if (host_counts.bad_index > 0) return GNNFD_BAD_INDEX;
    if (host_counts.sort_failed) {
        set_cuda_error(cudaErrorLaunchTimeout);
        return GNNFD_CUDA_ERROR;
    }

    gnnfd_csr_t* h = new (std::nothrow) gnnfd_csr_t;
    if (!h) return GNNFD_INVALID_ARG;
    h->n = n;
    h->nnz = host_counts.nnz;
    h->max_degree = host_counts.max_degree;
    int64_t start = 0;
    for (int b = 0; b < kNumBins; ++b) {
        h->bin_count[b] = host_counts.bin_count[b];
        h->bin_start[b] = start;
        start += host_counts.bin_count[b];
    }
    for (int o = 0; o < kOctaves; ++o) h->octave_count[o] = host_counts.octave_count[o];
    h->n_segments = host_counts.n_segments;
    h->row_ptr = P.row_ptr;
    h->col_idx = P.col_idx;
    h->perm = P.perm;
    h->dinv = P.dinv;
    h->rdeg = P.rdeg;
    h->edge_w = P.edge_w;
    h->row_order = P.row_order;
    h->seg_row = P.seg_row;
    h->seg_begin = P.seg_begin;
    h->seg_end = P.seg_end;
    h->seg_slot = P.seg_slot;
    h->hub_seg_ptr = P.hub_seg_ptr;
    *out = h;
    return GNNFD_OK;
}

static size_t scratch_size(const BuildLayout& L)
{
    Carver c(nullptr, ~size_t(0));
    ScratchPtrs s;
    carve_scratch(c, L, &s);
    return c.off;
}

// Sizes of a build's buffers and the most hub segments of such a graph (each may be null).  for_smaller: buffers that hold every graph with
// fewer vertices or edges too, which is what the queries return.  Larger inputs need more in nearly every place.  Where one more vertex ends the buckets
// (their keys no longer share a word with the values), the buckets' words are kept: 33,554,432 vertices with 4.9 M edges
// need 136 MB, one vertex less 144.
int csr_sizes(int64_t n, int64_t e, uint32_t flags, bool for_smaller, size_t* persistent_bytes, size_t* scratch_bytes, int64_t* segments)
{
    BuildLayout L;
    const int rc = make_layout(n, e, flags, &L);
    if (rc) return rc;
    if (!for_smaller) reserve_ranges(&L, L.n_ranges);
    if (persistent_bytes) {
        Carver c(nullptr, ~size_t(0));
        PersistentPtrs p;
        carve_persistent(c, n, L, &p);
        *persistent_bytes = c.off;
    }
    if (segments) *segments = L.seg_cap;
    if (!scratch_bytes) return GNNFD_OK;
    *scratch_bytes = scratch_size(L);
    if (!for_smaller || L.top_bits > 0 || !use_large_tile(L.m)) return GNNFD_OK;
    for (int bits = 31; bits > 0; --bits)                   // the largest graph with buckets: key bits grow at 2^bits and behind it
        for (int64_t less = int64_t(1) << bits; less >= (int64_t(1) << bits) - 1; --less) {
            BuildLayout with;
            if (less >= n || make_layout(less, e, flags, &with) || with.top_bits == 0) continue;
            const size_t bytes = scratch_size(with);
            if (bytes > *scratch_bytes) *scratch_bytes = bytes;
            return GNNFD_OK;
        }
    return GNNFD_OK;
}

}  // namespace gnnfd

extern "C" {

int gnnfd_csr_workspace_bytes(int64_t n, int64_t e, uint32_t flags, size_t* persistent_bytes, size_t* scratch_bytes)
{
    return gnnfd::csr_sizes(n, e, flags, true, persistent_bytes, scratch_bytes, nullptr);
}

int gnnfd_build_csr(int64_t n, int64_t e, const void* d_src, const void* d_dst, gnnfd_itype_t itype, uint32_t flags,
                    void* d_persistent, size_t persistent_bytes, void* d_scratch, size_t scratch_bytes, void* stream,
                    gnnfd_csr_t** out)
{
    return gnnfd::build_csr_impl(n, e, d_src, d_dst, itype, flags, true, true, d_persistent, persistent_bytes, d_scratch, scratch_bytes,
                                 static_cast<cudaStream_t>(stream), out);
}

int gnnfd_debug_build_fault(int32_t max_polls, int32_t sweep)
{
    using namespace gnnfd;
    if (max_polls < 0 || max_polls > kMaxPolls || sweep < 0) return GNNFD_INVALID_ARG;
    t_drill = BuildDrill{max_polls ? max_polls : kMaxPolls, sweep};
    return GNNFD_OK;
}

}  // extern "C"
