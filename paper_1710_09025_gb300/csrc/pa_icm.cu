// pa_icm.cu -- isoenergetic cluster moves (Sec. II.C) between random pairs.
//
// Round t of step k pairs replicas pi_t(2i) and pi_t(2i+1), i < floor(R/2);
// pi_t is a 4-round Feistel permutation of [0, 2^m) (m even, the smallest
// with 2^m >= R, at least 2) walked in cycles back into [0, R): halves of m/2
// bits, (Lh, Rh) -> (Rh, Lh ^ F_j(Rh)), F_j(v) = out0 of Philox at counter
// (v, k, 4t + j) of the ICM stream.  For a pair, the overlap q_i = S^a_i S^b_i
// splits the lattice into islands; the sector (q = -1 or +1) with fewer
// sites is used (ties: -1), its idx-th site in site order is drawn with
// idx = floor(r32 n_sector / 2^32), r32 = out0 at counter (i, k, 16 + t), and
// the spins of that site's island are flipped in both replicas.  With a zero
// field E_a + E_b is unchanged, so the move is always accepted.
//
// Five launches with packed words (three with int8 rows, which need no turning):
// both rounds' pairings, one thread per replica; the words turned into one bit row
// per replica; two rounds of moves, one warp per pair; the rows turned back.  A
// pair then reads N / 8 bytes per replica instead
// of a 64-bit word per site, and its island grows by whole x-rows: the sector and
// the island are L-bit rows in shared memory, a row takes the bits next to the
// rows around it and fills the sector's runs that touch them with one addition
// (a carry runs through a run of ones) upwards and, bit-reversed, downwards.  The
// island grows every pass until it is complete, so at most N passes run; the
// bound sets an error flag.  Bound by the passes' integer work and their
// shared-memory round trips.  One block per pair with a union-find over sites
// took 304 us a round at 2D L=32, R=20000; now 34 us, and the pairings and the
// two turns 28 us a step.
#include "pa_device.cuh"
#include "pa_internal.h"
#include "pa_sweep_tiles.cuh"

#include <algorithm>

namespace pa {

constexpr int kIcmWarps = 4;
constexpr int kIcmMaxN = 4096;

__device__ __forceinline__ uint32_t icm_feistel(uint32_t x, int h, int k, int t, uint32_t k0, uint32_t k1,
                                                uint32_t c3)
{
    const uint32_t mask = (1u << h) - 1u;  // h <= 16
    uint32_t Lh = (x >> h) & mask, Rh = x & mask;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const u32x4 o = philox(Rh, (uint32_t)k, (uint32_t)(4 * t + j), c3, k0, k1);
        const uint32_t nr = Lh ^ (o.x & mask);
        Lh = Rh;
        Rh = nr;
    }
    return (Lh << h) | Rh;
}

__device__ uint32_t icm_perm(uint32_t i, uint32_t n, int k, int t, uint32_t k0, uint32_t k1, uint32_t c3)
{
    int m = 2;
    while (m < 32 && (1ull << m) < (unsigned long long)n) m += 2;
    uint32_t y = icm_feistel(i, m / 2, k, t, k0, k1, c3);
    // cycle walking: the permutation of [0, 2^m) restricted to [0, n); each
    // step leaves [0, n) with probability below 3/4, and n <= 2^26 bounds the walk
    for (int guard = 0; y >= n && guard < (1 << 26); ++guard) y = icm_feistel(y, m / 2, k, t, k0, k1, c3);
    return y;
}

// both rounds' pairings
__global__ void __launch_bounds__(256) icm_pairs_kernel(IcmArgs a)
{
    const int R = a.Rdev ? *a.Rdev : a.R;
    const int i = blockIdx.x * 256 + threadIdx.x, t = blockIdx.y;
    if (i < (R & ~1)) a.perm[(size_t)t * a.R + i] = (int)icm_perm((uint32_t)i, (uint32_t)R, a.k, t, a.key0, a.key1, a.c3);
}

// packed words -> bit rows of NW words per replica (back = 0), or the rows of the
// population back into the words (back = 1; padding lanes keep their bits); one
// warp per group and 32-site chunk
__global__ void __launch_bounds__(256) icm_rows_kernel(IcmArgs a, int back)
{
    const int lane = threadIdx.x & 31, N = a.N, NW = (N + 31) / 32;
    const int R = a.Rdev ? *a.Rdev : a.R, G = (R + 63) >> 6;
    const int tup = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (tup >= G * NW) return;  // warp-uniform
    const int g = tup / NW, c = tup - g * NW, i = 32 * c + lane;
    const int ra = 64 * g + lane, rb = ra + 32;
    uint64_t* w = a.S + (size_t)g * N + i;
    if (!back) {
        const uint64_t x = i < N ? *w : 0ull;
        const uint32_t lo = transpose32((uint32_t)x, lane), hi = transpose32((uint32_t)(x >> 32), lane);
        if (ra < R) a.rows[(size_t)ra * NW + c] = lo;
        if (rb < R) a.rows[(size_t)rb * NW + c] = hi;
    } else {
        const uint32_t lo = transpose32(ra < R ? a.rows[(size_t)ra * NW + c] : 0u, lane);
        const uint32_t hi = transpose32(rb < R ? a.rows[(size_t)rb * NW + c] : 0u, lane);
        const int left = R - 64 * g;
        const uint64_t valid = left >= 64 ? ~0ull : (1ull << left) - 1ull;
        if (i < N) *w = (*w & ~valid) | (((uint64_t)hi << 32 | lo) & valid);
    }
}

// sign bits of 32 int8 spins (sites 32 w ...) of a row of NP bytes
__device__ __forceinline__ uint32_t icm_signs(const int8_t* row, int w, int NP)
{
    uint32_t bits = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (32 * w + 16 * h >= NP) break;
        const uint4 v = *reinterpret_cast<const uint4*>(row + 32 * w + 16 * h);
        const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)  // bit 7 of the four bytes, gathered by a multiply
            bits |= ((((x[j] >> 7) & 0x01010101u) * 0x01020408u) >> 24) << (16 * h + 4 * j);
    }
    return bits;
}
// flip (change the sign of) the spins whose bits are set
__device__ __forceinline__ void icm_flip(int8_t* row, int w, int NP, uint32_t bits)
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t b = (bits >> (16 * h)) & 0xFFFFu;
        if (!b || 32 * w + 16 * h >= NP) continue;
        uint4* p = reinterpret_cast<uint4*>(row + 32 * w + 16 * h);
        uint4 v = *p;
        auto bytes = [&](int j) { return ((((b >> (4 * j)) & 15u) * 0x00204081u) & 0x01010101u) * 0xFEu; };
        v.x ^= bytes(0); v.y ^= bytes(1); v.z ^= bytes(2); v.w ^= bytes(3);  // 1 <-> -1
        *p = v;
    }
}

__device__ __forceinline__ uint32_t brev(uint32_t x) { return __brev(x); }
__device__ __forceinline__ uint64_t brev(uint64_t x) { return __brevll(x); }
__device__ __forceinline__ int popc(uint32_t x) { return __popc(x); }
__device__ __forceinline__ int popc(uint64_t x) { return __popcll(x); }

// ROW: the type of an x-row (32 bits up to L = 32, 64 for L = 64)
template <class ROW>
__global__ void __launch_bounds__(32 * kIcmWarps) icm_kernel(IcmArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_icm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int N = a.N, L = a.L, NW = (N + 31) / 32, M = N / L;  // M rows
    const int R = a.Rdev ? *a.Rdev : a.R, npairs = R / 2;
    ROW* s = reinterpret_cast<ROW*>(smem_icm) + (size_t)warp * 2 * M;  // sector rows
    ROW* f = s + M;                                                    // island rows
    uint32_t* bits = reinterpret_cast<uint32_t*>(smem_icm + sizeof(ROW) * 2 * M * kIcmWarps) + warp * (NW + 2);
    const ROW full = L == (int)(8 * sizeof(ROW)) ? ~(ROW)0 : ((ROW)1 << (L & 63)) - 1;
    const int rpl = (M + 31) / 32, m0 = min(M, lane * rpl), m1 = min(M, m0 + rpl);  // rows in site order
    bool bad = false;
    for (int i = blockIdx.x * kIcmWarps + warp; i < npairs; i += gridDim.x * kIcmWarps) {
        const int ra = a.perm[(size_t)a.t * a.R + 2 * i], rb = a.perm[(size_t)a.t * a.R + 2 * i + 1];
        const uint32_t r32 = philox((uint32_t)i, (uint32_t)a.k, (uint32_t)(16 + a.t), a.c3, a.key0, a.key1).x;
        int nneg = 0;
        for (int w = lane; w < NW; w += 32) {
            uint32_t q;
            if (a.S8) q = icm_signs(a.S8 + (size_t)ra * a.NP, w, a.NP) ^ icm_signs(a.S8 + (size_t)rb * a.NP, w, a.NP);
            else q = a.rows[(size_t)ra * NW + w] ^ a.rows[(size_t)rb * NW + w];
            if (32 * w + 32 > N) q &= (1u << (N & 31)) - 1u;
            bits[w] = q;
            nneg += __popc(q);
        }
        nneg = __reduce_add_sync(0xffffffffu, nneg);
        const bool want = nneg <= N - nneg;  // the sector with fewer sites (ties: q = -1)
        const int nsec = want ? nneg : N - nneg;
        if (lane == 0) bits[NW] = bits[NW + 1] = 0u;
        __syncwarp();
        if (nsec == 0) continue;  // warp-uniform
        int cnt = 0;
        for (int r = m0; r < m1; ++r) {
            const int at = r * L, w = at >> 5, sh = at & 31;
            ROW row = (ROW)__funnelshift_r(bits[w], bits[w + 1], sh);
            if (sizeof(ROW) == 8) row |= (ROW)((uint64_t)__funnelshift_r(bits[w + 1], bits[w + 2], sh) << 32);
            row &= full;
            if (!want) row ^= full;
            s[r] = row;
            f[r] = 0;
            cnt += popc(row);
        }
        // the idx-th sector site in site order
        const int idx = (int)(((uint64_t)r32 * (uint64_t)nsec) >> 32);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        int rest = idx - (incl - cnt);
        if (rest >= 0 && rest < cnt) {
            int r = m0;
            while (rest >= popc(s[r])) rest -= popc(s[r++]);
            ROW x = s[r];
            for (; rest > 0; --rest) x &= x - 1;
            f[r] = x & (~x + 1);
        }
        __syncwarp();
        // grow the island until a pass changes nothing; passes only add bits, so
        // rows read while another lane writes them are taken up by a later pass
        int guard = 0;
        for (;;) {
            bool changed = false;
            for (int r = m0; r < m1; ++r) {
                const ROW s0 = s[r], f0 = f[r];
                if (s0 == f0) continue;
                const int y = r % L, zr = r - y;
                ROW nb = f[zr + (y == L - 1 ? 0 : y + 1)] | f[zr + (y == 0 ? L - 1 : y - 1)];
                if (a.D == 3) nb |= f[r + L < M ? r + L : r + L - M] | f[r >= L ? r - L : r - L + M];
                nb |= (f0 << 1) | (f0 >> (L - 1)) | (f0 >> 1) | (f0 << (L - 1));  // x, periodic
                ROW x = f0 | (nb & s0);
                if (x == 0) continue;
                // runs of the sector that touch x, upwards, then downwards
                x |= s0 & ~(s0 + x);
                const ROW sr = brev(s0), xr = brev(x);
                x |= brev((ROW)(sr & ~(sr + xr)));
                if (x != f0) {
                    f[r] = x;
                    changed = true;
                }
            }
            __syncwarp();
            if (!__any_sync(0xffffffffu, changed)) break;
            if (++guard > N) { bad = true; break; }
        }
        // the island as site bits, then into both replicas
        for (int w = lane; w < NW; w += 32) bits[w] = 0u;
        __syncwarp();
        for (int r = m0; r < m1; ++r) {
            const ROW x = f[r];
            if (!x) continue;
            const int at = r * L, w = at >> 5, sh = at & 31;
            const uint64_t v = (uint64_t)x << sh;  // L = 64 has sh = 0
            if ((uint32_t)v) atomicOr(&bits[w], (uint32_t)v);
            if (v >> 32) atomicOr(&bits[w + 1], (uint32_t)(v >> 32));
        }
        __syncwarp();
        for (int w = lane; w < NW; w += 32) {
            const uint32_t x = bits[w];
            if (!x) continue;
            if (a.S8) {
                icm_flip(a.S8 + (size_t)ra * a.NP, w, a.NP, x);
                icm_flip(a.S8 + (size_t)rb * a.NP, w, a.NP, x);
            } else {
                a.rows[(size_t)ra * NW + w] ^= x;
                a.rows[(size_t)rb * NW + w] ^= x;
            }
        }
        __syncwarp();  // the arrays are reused by the next pair
    }
    if (bad && lane == 0) atomicExch(a.err, 1);
}

template <class ROW>
static void launch_pairs(const IcmArgs& a, int sms, cudaStream_t st)
{
    const int NW = (a.N + 31) / 32, M = a.N / a.L, npairs = a.R / 2;
    const size_t smem = sizeof(ROW) * 2 * M * kIcmWarps + sizeof(uint32_t) * (NW + 2) * kIcmWarps;
    const int grid = std::min((npairs + kIcmWarps - 1) / kIcmWarps, sms * 16);
    for (int t = 0; t < 2; ++t) {
        IcmArgs r = a;
        r.t = t;
        icm_kernel<ROW><<<grid, 32 * kIcmWarps, smem, st>>>(r);
    }
}

// both rounds of step k; *launches: kernels enqueued
cudaError_t launch_icm(const IcmArgs& a, int* launches, cudaStream_t st)
{
    *launches = 0;
    if (a.N > kIcmMaxN) return cudaErrorInvalidValue;
    if (a.R / 2 == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    icm_pairs_kernel<<<dim3((a.R + 255) / 256, 2), 256, 0, st>>>(a);
    const long long tiles = (long long)((a.R + 63) / 64) * ((a.N + 31) / 32);
    const unsigned rgrid = (unsigned)((tiles + 7) / 8);
    if (!a.S8) icm_rows_kernel<<<rgrid, 256, 0, st>>>(a, 0);
    if (a.L <= 32) launch_pairs<uint32_t>(a, sms, st);
    else launch_pairs<uint64_t>(a, sms, st);
    if (!a.S8) icm_rows_kernel<<<rgrid, 256, 0, st>>>(a, 1);
    *launches = a.S8 ? 3 : 5;
    return cudaGetLastError();
}

}  // namespace pa
