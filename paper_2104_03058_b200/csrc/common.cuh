// Shared host-side plumbing of the gnnfd library: handle layout, launch bookkeeping, error capture.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <utility>

#include "gnnfd.h"

namespace gnnfd {

constexpr int kNumBins = 5;                 // four degree classes + hub rows
constexpr int kBinDeg0 = 8, kBinDeg1 = 32, kBinDeg2 = 128, kBinDeg3 = GNNFD_HUB_DEGREE;   // upper degree of each class
constexpr int kOctaves = 4;                 // octaves of the degree in the fourth class
constexpr int kHubSegment = GNNFD_HUB_SEGMENT;

// Device-side counters filled during the build and copied to the host once.
struct BuildCounts {
    int32_t bad_index;       // ids outside [0, n)
    int32_t n_valid;         // candidate edges that survive the self-loop / reverse-edge rules
    int32_t nnz;             // entries after dedup
    int32_t max_degree;
    int32_t n_segments;      // hub segments
    int32_t bin_count[kNumBins];
    int32_t sort_failed;     // a sweep of the sort gave up waiting: nothing after it is meaningful
    int32_t octave_count[kOctaves]; // rows of the fourth bin by octave of the degree: 129..256, ..512, ..1024, ..2048
    int32_t pad[1];
};

}  // namespace gnnfd

struct gnnfd_csr {
    int64_t n, nnz;
    int32_t max_degree;
    int64_t bin_count[gnnfd::kNumBins];
    int64_t bin_start[gnnfd::kNumBins];
    int64_t octave_count[gnnfd::kOctaves];       // the fourth bin (129 .. 2048 entries) by octave of the degree, ascending
    int64_t n_segments;
    const int32_t* row_ptr;
    const int32_t* col_idx;
    const int32_t* perm;
    const float* dinv;
    const float* rdeg;
    const float* edge_w;
    const int32_t* row_order;
    const int32_t* seg_row;
    const int32_t* seg_begin;
    const int32_t* seg_end;
    const int32_t* seg_slot;
    const int32_t* hub_seg_ptr;
};

namespace gnnfd {

void set_cuda_error(cudaError_t e);

// Records the launch (count, optional event bracket).  Use through GNNFD_LAUNCH.
struct LaunchScope {
    LaunchScope(const char* name, cudaStream_t s);
    ~LaunchScope();
    const char* name;
    cudaStream_t stream;
    void* rec;
};

// A call is a chain of launches, on small graphs of a few microseconds each.  Every kernel of the library is launched with
// programmatic stream serialisation: where the kernel before it lets it (grid_dependency<true>), its blocks take their places as soon as all
// blocks of that one have started.  They wait there (grid_dependency, the first statement of every kernel) until that launch has
// ended and its writes can be seen.  Every kernel waits before it reads or writes memory, and reads what launches before it may have written
// by plain loads: the non-coherent path is for memory that nobody writes while the kernel exists, and it exists already while the one before it
// writes (plain loads cost nothing: GAT 8 x 16 bf16 on 39.6 M entries 906 -> 889 us, all else the same).
// Build and aggregation of 20,000 vertices and 89,000 edges 134 -> 118 us, GAT 8 x 8 on 200,000 rows 121 -> 115.
// A kernel lets the next one start when it has waited itself, not before: with several launches lined up, the longest rows of one, which come
// first, took the places that the last blocks of another left, a few SMs for most of them.  20,000 rows of 50 entries, GCN, 256 bf16
// columns one at a time 46, lined up 53, now 44 us; GAT 1 x 64 40, 42, 35; 5000 rows of 100, GAT 4 x 32 fp32 37, 45, 34.  The
// GAT aggregation, whose scores come in between, does not let it start at all (20,000 rows of 50, 4 x 32 64 -> 56 us).
// Nor do kernels that leave an SM with little L1 (tensor tiles, large sort tiles, compaction): the next one would keep
// that share for as long as it runs (GCN layer 602 -> 64 on 116 M entries 1.78 -> 2.28 ms, build of 80 M edges 2.85 -> 3.14); nor the edge
// softmax kernels (20,000 rows of 50 entries 37 -> 41 us).
template <typename... Params, typename... Args>
inline void launch_early(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args&&... args)
{
    cudaLaunchAttribute attribute;
    attribute.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attribute.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t config{};
    config.gridDim = grid;
    config.blockDim = block;
    config.dynamicSmemBytes = smem;
    config.stream = stream;
    config.attrs = &attribute;
    config.numAttrs = 1;
    cudaLaunchKernelEx(&config, kernel, std::forward<Args>(args)...);      // errors are picked up by cudaGetLastError
}

template <bool LET_NEXT_START>
__device__ __forceinline__ void grid_dependency()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (LET_NEXT_START) asm volatile("griddepcontrol.launch_dependents;");
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Bump allocator over a caller-provided device buffer.
struct Carver {
    char* base;
    size_t off, cap;
    bool ok;
    Carver(void* p, size_t bytes) : base(static_cast<char*>(p)), off(0), cap(bytes), ok(true) {}
    template <typename T>
    T* take(size_t count)
    {
        size_t bytes = align_up(count * sizeof(T), 256);
        if (off + bytes > cap) { ok = false; off += bytes; return nullptr; }
        T* r = reinterpret_cast<T*>(base + off);
        off += bytes;
        return r;
    }
};

// Exclusive prefix sum of `count` int32 values (in -> out, may alias), temp from scan_temp_ints().
size_t scan_temp_ints(size_t count);
int exclusive_scan_i32(const int32_t* d_in, int32_t* d_out, size_t count, int32_t* d_temp, cudaStream_t s);

// ---- aligned copies of features (aggregate.cu): chunks of cw columns placed `pitch` columns apart, rows ld apart

struct AlignedCopy {
    int32_t pitch;       // columns from one chunk's start to the next one's
    int64_t ld;          // row pitch
    size_t bytes;        // 0: no copy
};
bool copy_pays(const gnnfd_csr_t* csr, int64_t per_entry, int64_t least);
AlignedCopy layout_copy(int64_t n, gnnfd_dtype_t xdt, int32_t f, int32_t cw, int32_t unit_bytes, int32_t row_bytes);
void launch_copy(const void* d_x, int64_t ldx, gnnfd_dtype_t xdt, int64_t n, int32_t f, int32_t cw, const AlignedCopy& copy,
                 void* d_aligned, cudaStream_t s);

// ---- pieces of one translation unit that the layer entry points (layer.cu) put together

int csr_sizes(int64_t n, int64_t e, uint32_t flags, bool for_smaller, size_t* persistent_bytes, size_t* scratch_bytes,
              int64_t* segments);                                     // csr_build.cu
int build_csr_impl(int64_t n, int64_t e, const void* d_src, const void* d_dst, gnnfd_itype_t itype, uint32_t flags, bool need_perm,
                   bool need_weights, void* d_persistent, size_t persistent_bytes, void* d_scratch, size_t scratch_bytes, cudaStream_t s,
                   gnnfd_csr_t** out);                                // csr_build.cu
int combine_impl(int64_t n, const void* d_x, int64_t ldx, gnnfd_dtype_t xdt, int32_t f_in, const void* d_w_t, int64_t ldw,
                 int32_t f_out, void* d_z, int64_t ldz, gnnfd_dtype_t zdt, int mode, const float* d_a_src,
                 const float* d_a_dst, int32_t heads, int32_t dim, float* d_s_src, float* d_s_dst, int32_t* d_status,
                 cudaStream_t s);
int gat_aggregate_impl(const gnnfd_csr_t* csr, const void* d_z, int64_t ldz, gnnfd_dtype_t zdt, const float* d_a_src,
                       const float* d_a_dst, int32_t heads, int32_t dim, float negative_slope, void* d_out, int64_t ldo,
                       gnnfd_dtype_t odt, int32_t chunk_width, void* d_scratch, size_t scratch_bytes, bool scores_ready,
                       cudaStream_t s);
size_t gat_copy_bytes(const gnnfd_csr_t* csr, const void* d_z, int64_t ldz, gnnfd_dtype_t zdt, int32_t heads, int32_t dim,
                      int32_t chunk_width);
int gat_scratch_scores(const gnnfd_csr_t* csr, int32_t heads, int32_t dim, void* d_scratch, size_t scratch_bytes,
                       float** s_src, float** s_dst);

}  // namespace gnnfd

#define GNNFD_LAUNCH(name, stream, kernel, grid, block, smem, ...)                   \
    do {                                                                             \
        ::gnnfd::LaunchScope scope_(name, stream);                                   \
        ::gnnfd::launch_early(kernel, grid, block, smem, stream, __VA_ARGS__);       \
    } while (0)

#define GNNFD_CUDA_CHECK(expr)                                                       \
    do {                                                                             \
        cudaError_t err_ = (expr);                                                   \
        if (err_ != cudaSuccess) { ::gnnfd::set_cuda_error(err_); return GNNFD_CUDA_ERROR; } \
    } while (0)
