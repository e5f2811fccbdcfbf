// pa_packed_sweep.cuh -- the packed (+-J) sweep kernel and its launch
// templates.  Each lattice size instantiates four kernels (two groups-per-
// block choices, packed or int8 storage); the sizes are spread over the
// translation units pa_packed_part0..3.cu so that they compile in parallel.
#pragma once
#include "pa_launch.h"
#include "pa_sweep_tiles.cuh"

namespace pa {

// Block b takes GPB groups; with spread > 0 the groups are spread evenly instead:
// every SM gets an even share (blocks b, b + spread, ... run on one SM), and that
// is split over its blocks (at most GPB a block).
template <int D, int L, int GPB, int THREADS, bool I8, bool SHARD = false>
__global__ void __launch_bounds__(THREADS, 4) sweep_packed_kernel(PackedSweepArgs a, int spread)
{
    extern __shared__ __align__(16) unsigned char smem_packed[];
    const int G = packed_groups(a.i);
    int g0 = blockIdx.x * GPB, gend = min(g0 + GPB, G);
    if (GPB > 1 && spread) {
        const int sm = blockIdx.x % spread, slot = blockIdx.x / spread, slots = (gridDim.x - sm + spread - 1) / spread;
        const int a0 = (int)((long long)G * sm / spread), a1 = (int)((long long)G * (sm + 1) / spread);
        g0 = a0 + (a1 - a0) * slot / slots;
        gend = a0 + (a1 - a0) * (slot + 1) / slots;
    }
    sweep_packed_tile<D, L, GPB, THREADS, I8, true, SHARD>(a.s, a.i, g0, gend, smem_packed);
}

// threads per word of the team variant: at most eight, at most 512 threads a
// block; 1 where the lattice has more than 256 words per sublattice
template <int D, int L> __host__ __device__ constexpr int team_of()
{
    constexpr int NH = Lat<D, L>::NH;
    int t = 8;
    while (t > 1 && t * NH > 512) t /= 2;
    return t;
}
template <int D, int L> __host__ __device__ constexpr int team_threads()
{
    int n = 32;
    while (n < team_of<D, L>() * Lat<D, L>::NH) n *= 2;
    return n;
}
template <int D, int L, bool I8>
__global__ void __launch_bounds__(team_threads<D, L>()) sweep_packed_team_kernel(PackedSweepArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_packed[];
    const int G = packed_groups(a.i), g0 = blockIdx.x;
    sweep_packed_tile<D, L, 1, team_threads<D, L>(), I8, true, false, team_of<D, L>()>(a.s, a.i, g0, min(g0 + 1, G), smem_packed);
}
template <int D, int L, bool I8>
static cudaError_t launch_team(const PackedSweepArgs& a, cudaStream_t st)
{
    constexpr size_t smem = PackedShape<D, L, 1, team_threads<D, L>(), false>::SMEM;
    static_assert(smem <= 48 * 1024, "no opt-in needed");
    sweep_packed_team_kernel<D, L, I8><<<a.i.G, team_threads<D, L>(), smem, st>>>(a);
    return cudaGetLastError();
}

// ---------------- shapes and dispatch ----------------

template <int D, int L, int GPB, int THREADS, bool I8, bool SHARD = false>
static cudaError_t launch_one(const PackedSweepArgs& a, int grid, int spread, cudaStream_t st)
{
    const size_t smem = PackedShape<D, L, GPB, THREADS>::SMEM;
    auto kern = sweep_packed_kernel<D, L, GPB, THREADS, I8, SHARD>;
    static std::atomic<unsigned long long> done{0};
    const cudaError_t e = allow_smem(kern, (int)smem, done);
    if (e != cudaSuccess) return e;
    kern<<<grid, THREADS, smem, st>>>(a, spread);
    return cudaGetLastError();
}

template <int D, int L>
static cudaError_t launch_dl(const PackedSweepArgs& a, int gpb, int threads, cudaStream_t st)
{
    constexpr Shape s = default_shape<D, L>();
    const bool i8 = a.i.S8_out != nullptr;
    int grid = (a.i.G + gpb - 1) / gpb;
    if (a.i.goff != 0) {  // a shard (packed words, default shape)
        if (i8 || gpb != s.gpb || threads != s.threads) return cudaErrorInvalidConfiguration;
        return launch_one<D, L, s.gpb, s.threads, false, true>(a, grid, 0, st);
    }
    // the one tuned alternative: twice the groups per block, same thread count
    if (gpb == 2 * s.gpb && threads == s.threads)
        return i8 ? launch_one<D, L, 2 * s.gpb, s.threads, true>(a, grid, 0, st)
                  : launch_one<D, L, 2 * s.gpb, s.threads, false>(a, grid, 0, st);
    if (gpb != s.gpb || threads != s.threads) return cudaErrorInvalidConfiguration;
    // few threads to an SM even with a team per word: the team variant (us a
    // launch before -> with it: L=4, R=1000 36 -> 18; L=4, R=30000 44 -> 38; L=6,
    // R=5000 39 -> 29; L=8, R=5000 52 -> 36; above the line it does more work than
    // it hides: L=6, R=30000 66 -> 86)
    if constexpr (team_of<D, L>() > 1) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int per_sm = team_threads<D, L>() <= 256 ? 1024 : 512;
        if ((long long)a.i.G * team_threads<D, L>() <= (long long)sms * per_sm)
            return i8 ? launch_team<D, L, true>(a, st) : launch_team<D, L, false>(a, st);
    }
    // less than a wave of full blocks (four to an SM): an SM with one block more
    // than another sets the time, so the groups are spread evenly over as many
    // blocks to an SM as full ones would need, at least two (us a launch, full
    // blocks -> spread: L=6, R=40001 111 -> 74; L=6, R=2x10^5 213 -> 188; L=8,
    // R=5x10^4 149 -> 126; L=8, R=1.2x10^5 260 -> 232; 2D L=16, R=6x10^4 116 -> 88).
    // Tiles with late compaction lose more to their partly filled queue rounds
    // than the balance gives when the blocks would be four fifths full (L=8,
    // R=10^5: 205 -> 209; R=1.5x10^5: 268 -> 272)
    int spread = 0;
    if constexpr (s.gpb > 1) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int k = grid <= 2 * sms ? 2 : (grid + sms - 1) / sms;
        const long long room = (long long)k * sms * s.gpb;
        if (grid < 4 * sms && (!PackedShape<D, L, s.gpb, s.threads>::kLate || 10ll * a.i.G < 8 * room)) {
            grid = a.i.G < k * sms ? a.i.G : k * sms;
            spread = grid < sms ? grid : sms;
        }
    }
    return i8 ? launch_one<D, L, s.gpb, s.threads, true>(a, grid, spread, st)
              : launch_one<D, L, s.gpb, s.threads, false>(a, grid, spread, st);
}

// launch for the lattice sizes of one part: *handled is false when (D, L)
// belongs to another part
cudaError_t launch_sweep_packed_part0(int D, int L, const PackedSweepArgs& a, int gpb, int threads,
                                      cudaStream_t st, bool* handled);
cudaError_t launch_sweep_packed_part1(int D, int L, const PackedSweepArgs& a, int gpb, int threads,
                                      cudaStream_t st, bool* handled);
cudaError_t launch_sweep_packed_part2(int D, int L, const PackedSweepArgs& a, int gpb, int threads,
                                      cudaStream_t st, bool* handled);
cudaError_t launch_sweep_packed_part3(int D, int L, const PackedSweepArgs& a, int gpb, int threads,
                                      cudaStream_t st, bool* handled);

}  // namespace pa
