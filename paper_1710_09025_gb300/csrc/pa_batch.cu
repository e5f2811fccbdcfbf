// pa_batch.cu -- the batched sweep: persistent launches over the replica tiles of
// many instances (mixed L, +-J and real couplings): one for the packed tiles (and
// the real couplings without threshold tables), one beside it for the tables.
//
// Blocks take work items (instance, tile) from a queue in global memory (one
// atomic counter per temperature) and run the same tile functions as the
// single-instance kernels, so every instance gets exactly the results of its
// own context.  Items are ordered by decreasing cost so that the expensive
// tiles start first and the tail is made of cheap ones.
#include "pa_real_table.cuh"
#include "pa_sweep_tiles.cuh"

#include <algorithm>

namespace pa {

constexpr int kBatchThreads = 256;

// 3D lattices the batched sweep dispatches to: packed +-J (two groups-per-
// block choices) and int8 real couplings.
#define PA_BATCH_PACKED(X) X(0, 4) X(1, 6) X(2, 8) X(3, 10) X(4, 12) X(5, 16)
#define PA_BATCH_REAL(X) X(3, 10) X(4, 12)
// 3D lattices of the threshold-table launch (index, L, with a field)
#define PA_BATCH_TABLE(X) \
    X(0, 4, false) X(1, 6, false) X(2, 8, false) X(3, 10, false) X(4, 4, true) X(5, 6, true) X(6, 8, true)

__global__ void __launch_bounds__(kBatchThreads, 3) sweep_batch_kernel(PackedStep ps, RealStep rs,
                                                                    const BatchSweepInst* insts,
                                                                    const int2* items, int n_items,
                                                                    int mult, int* counter)
{
    extern __shared__ __align__(16) unsigned char smem_b[];
    __shared__ int s_item;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= n_items) return;
        const int2 w = items[it];
        const BatchSweepInst& bi = insts[w.x];
        const int cls = bi.cls < kBatchRealBase ? bi.cls + (mult - 1) : bi.cls;
        switch (cls) {
#define XP(idx, l)                                                                                  \
    case 2 * idx: {                                                                                 \
        constexpr int g = default_shape<3, l>().gpb;                                                \
        sweep_packed_tile<3, l, g, kBatchThreads, false, false>(                                     \
            ps, bi.pk, w.y * g, min(w.y * g + g, packed_groups(bi.pk)), smem_b);                    \
    } break;                                                                                        \
    case 2 * idx + 1: {                                                                             \
        constexpr int g = 2 * default_shape<3, l>().gpb;                                            \
        sweep_packed_tile<3, l, g, kBatchThreads, false, false>(                                     \
            ps, bi.pk, w.y * g, min(w.y * g + g, packed_groups(bi.pk)), smem_b);                    \
    } break;
            PA_BATCH_PACKED(XP)
#undef XP
#define XR(idx, l)                                                                                  \
    case kBatchRealBase + idx:                                                                      \
        real_stage<3, l, kBatchThreads / 32>(bi.re, smem_b, false);                                 \
        sweep_real_tile<3, l, kBatchThreads / 32>(rs, bi.re, w.y, smem_b, false);                   \
        break;
            PA_BATCH_REAL(XR)
#undef XR
            default:
                break;
        }
    }
}

// Real couplings on threshold tables: blocks take (instance, chunk of at most
// `chunk` replica groups) items.  A chunk of 256 replicas amortises the
// instance's table (at most 64 rule evaluations per site against 2560 attempts
// per site); small batches take smaller chunks so that every SM has one.
__global__ void __launch_bounds__(kTabThreads) sweep_batch_table_kernel(RealStep rs, const BatchSweepInst* insts,
                                                                        const int2* items, int n_items, int chunk,
                                                                        int* counter)
{
    extern __shared__ __align__(128) unsigned char smem_bt[];
    __shared__ int s_item;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= n_items) return;
        const int2 w = items[it];
        const BatchSweepInst& bi = insts[w.x];
        const int R = bi.re.R, G4 = (R + 3) / 4, n = (G4 + chunk - 1) / chunk;
        const int g0 = (int)((long long)G4 * w.y / n), g1 = (int)((long long)G4 * (w.y + 1) / n);
        switch (bi.cls) {
#define XT(idx, l, f)                                                            \
    case kBatchTableBase + idx:                                                  \
        static_assert(8 * TabShape<3, l, f>::W >= kBatchTableGroups, "a chunk fits"); \
        tab_stage_offsets<3, l, f>(smem_bt);                                     \
        sweep_real_table<3, l, f>(rs, bi.re, R, g0, g1, smem_bt, false);         \
        break;
            PA_BATCH_TABLE(XT)
#undef XT
            default:
                break;
        }
    }
}

// class id, tiles and shared memory of an instance in the batched sweep
bool batch_class(int D, int L, int kind, bool field, int mult, int chunk, int G, int R, int* cls, int* tiles,
                 size_t* smem)
{
    if (D != 3) return false;
    if (kind == 0) {
#define XP(idx, l)                                                                            \
    if (L == l) {                                                                             \
        constexpr int g = default_shape<3, l>().gpb;                                          \
        *cls = 2 * idx;                                                                       \
        *tiles = (G + g * mult - 1) / (g * mult);                                             \
        *smem = mult == 1 ? PackedShape<3, l, g, kBatchThreads, false>::SMEM                  \
                          : PackedShape<3, l, 2 * g, kBatchThreads, false>::SMEM;             \
        return true;                                                                          \
    }
        PA_BATCH_PACKED(XP)
#undef XP
        return false;
    }
#define XT(idx, l, f)                                                                         \
    if (L == l && field == f) {                                                               \
        static_assert(TabShape<3, l, f>::FITS, "table fits");                                 \
        *cls = kBatchTableBase + idx;                                                         \
        *tiles = ((R + 3) / 4 + chunk - 1) / chunk;                                           \
        *smem = TabShape<3, l, f>::SMEM;                                                      \
        return true;                                                                          \
    }
    PA_BATCH_TABLE(XT)
#undef XT
#define XR(idx, l)                                                                            \
    if (L == l) {                                                                             \
        *cls = kBatchRealBase + idx;                                                          \
        *tiles = (R + 31) / 32;                                                               \
        *smem = RealShape<3, l, kBatchThreads / 32>::SMEM;                                    \
        return true;                                                                          \
    }
    PA_BATCH_REAL(XR)
#undef XR
    return false;
}

// Shared memory of the largest item of each launch.  The limit belongs to the
// kernel on a device, not to a batch: it is raised to this once and never set to
// what one batch needs, which would refuse the launches of another batch with
// larger items.
#define XP(idx, l)                                                          \
    PackedShape<3, l, default_shape<3, l>().gpb, kBatchThreads, false>::SMEM, \
        PackedShape<3, l, 2 * default_shape<3, l>().gpb, kBatchThreads, false>::SMEM,
#define XR(idx, l) RealShape<3, l, kBatchThreads / 32>::SMEM,
#define XT(idx, l, f) TabShape<3, l, f>::SMEM,
constexpr size_t kBatchSmem = std::max({PA_BATCH_PACKED(XP) PA_BATCH_REAL(XR) size_t(0)});
constexpr size_t kBatchTableSmem = std::max({PA_BATCH_TABLE(XT) size_t(0)});
#undef XP
#undef XR
#undef XT

cudaError_t batch_sweep_occupancy(size_t smem, int* blocks_per_sm)
{
    static std::atomic<unsigned long long> done{0};
    const cudaError_t e = allow_smem(sweep_batch_kernel, (int)kBatchSmem, done);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, sweep_batch_kernel,
                                                         kBatchThreads, smem);
}

cudaError_t launch_sweep_batched(const PackedStep& ps, const RealStep& rs, const BatchSweepInst* insts,
                                 const int2* items, int n_items, int mult, int* counter, int blocks,
                                 size_t smem, cudaStream_t st)
{
    sweep_batch_kernel<<<blocks, kBatchThreads, smem, st>>>(ps, rs, insts, items, n_items, mult, counter);
    return cudaGetLastError();
}

cudaError_t batch_table_occupancy(size_t smem, int* blocks_per_sm)
{
    static std::atomic<unsigned long long> done{0};
    const cudaError_t e = allow_smem(sweep_batch_table_kernel, (int)kBatchTableSmem, done);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, sweep_batch_table_kernel, kTabThreads, smem);
}

cudaError_t launch_sweep_batched_table(const RealStep& rs, const BatchSweepInst* insts, const int2* items,
                                       int n_items, int chunk, int* counter, int blocks, size_t smem, cudaStream_t st)
{
    sweep_batch_table_kernel<<<blocks, kTabThreads, smem, st>>>(rs, insts, items, n_items, chunk, counter);
    return cudaGetLastError();
}

}  // namespace pa
