// pa_real_table.cuh -- the Metropolis sweep with FP32 couplings, decided by
// threshold tables (Sec. II.B, checkerboard order of Sec. III.A).
//
// The specified rule (f = (((t_-x + t_+x) + t_-y) + ...) + h in FP32 with
// t = J S_nb, dE = 2 S f, x = f32(beta) dE, accept iff x <= 0 or
// r < floor(spec_expf(-x) 2^32)) depends on a site only through the signs of
// its 2D neighbours and of its own spin.  A block therefore evaluates the rule
// once for every sign pattern of every site and keeps the thresholds in shared
// memory; an attempted flip is then a pattern lookup and a compare.  Lattices
// whose table would be too large keep the upper 16 bits of the thresholds: the
// compare decides whenever the upper halves of r and of the threshold differ,
// and the other attempts (one in 65536) evaluate the rule itself.  With whole
// thresholds the only attempts left open are uniforms of all ones (the entry of
// an always accepted pattern is 0xFFFFFFFF, every other one at most
// 0xFFFFFF00).  So every decision is the specified one.  Without a field only
// the products with the last neighbour's sign matter (IEEE sums of negated
// terms are the negated sums), which halves the patterns.
//
// What bounds it: integer instructions, of which the ALU takes more than the
// multiplier; no unit is full (ncu at 3D L = 10: ALU pipe 64 % of its cycles,
// multiplier 53 %, issue slots 59 %; 384 to 1024 threads a block within 5 %), but
// the time has followed their number.  A Philox call serves four attempts (the WORD
// stream: the four sites of a quad, one replica) with 34 of them; four replicas
// of a quad take about 285, 18 per attempt.  Field, exponential and guard band
// per attempt took 86.  Gaussian couplings, N_S = 10, sweep time per
// temperature before -> now: 3D L = 10, R = 20000 760 -> 231 us; 3D L = 6,
// R = 50000 with gradient counts 388 -> 148 us; 2D L = 4 with a field,
// R = 50000 43 -> 25 us.
//
// Spins are bits: plane w holds 32 replicas in one word per site; replica
// 4 j + b of the plane is bit 8 b + j, so that four replicas of one group j sit
// in the four bytes and (word >> j) & 0x01010101 spreads them.  A thread owns a
// quad (four consecutive sublattice sites, one Philox block) and goes through
// replica groups; a slot is the set of threads that together own all quads, and
// slots work on disjoint replicas, so that only a slot's threads synchronise.
// Table columns are lanes: lookups are free of bank conflicts whatever the
// patterns.
#pragma once
#include "pa_device.cuh"
#include "pa_internal.h"
#include "pa_launch.h"
#include "pa_sweep_tiles.cuh"

namespace pa {

// 16 warps of 128 registers: 384 and 768 threads measured 263 and 261 us against
// 251 at 3D L = 10, R = 20000 (the integer pipes are the limit, not latency)
constexpr int kTabThreads = 512;
// shared memory that a threshold table may take: what leaves room for the
// energies (an int128 per pattern of the +e_d bonds takes the same at 3D
// L = 10), the planes and the gradient sums
constexpr size_t kTabMax = 131072;
// whole thresholds wherever they fit: 3D L = 6 156 us against 168 with halves
constexpr size_t kTabWide = kTabMax;

template <int D, int L, bool FIELD>
struct TabShape {
    static constexpr int N = Lat<D, L>::N, NH = Lat<D, L>::NH;
    static constexpr int NQ = (NH + 3) / 4;  // quads per sublattice
    static constexpr int pow2_at_least(int v) { int p = 1; while (p < v) p *= 2; return p; }
    // quads padded to whole warps, or to a divisor of a warp
    static constexpr int NQP = NQ >= 32 ? (NQ + 31) / 32 * 32 : pow2_at_least(NQ);
    static constexpr int NBLK = NQP >= 32 ? NQP / 32 : 1;  // warps of a slot
    static constexpr int SEG = NQP < 32 ? NQP : 32;        // a slot's lanes within a warp
    static constexpr int SLOTS = kTabThreads / NQP;
    // pattern bits: the neighbours (relative to the last one without a field),
    // then the own spin
    static constexpr int KI = FIELD ? 2 * D : 2 * D - 1;
    static constexpr int ROWS = 2 << KI;
    // WIDE: whole thresholds, two rows of 256 bytes per pattern and 32 quads
    // (sites t = 0, 1 of lane l in words l and 32 + l, sites 2, 3 in the same
    // words of a second block of rows).  Else the upper halves, one row per
    // pattern: sites 0, 1 in the halves of word l, sites 2, 3 of word 32 + l.
    static constexpr bool WIDE = (size_t)2 * NBLK * 2 * ROWS * 256 <= kTabWide;
    static constexpr size_t BLOCK = (size_t)(WIDE ? 2 : 1) * ROWS * 256;  // bytes of 32 quads
    static constexpr size_t TABLE = (size_t)2 * NBLK * BLOCK;
    __host__ __device__ static constexpr int tpart(int t) { return WIDE ? (t >> 1) * ROWS * 256 + (t & 1) * 128 : (t >> 1) * 128 + (t & 1) * 2; }
    static constexpr bool FITS = TABLE <= kTabMax && SLOTS >= 1 && SLOTS * NQP == kTabThreads;
    // energies: one int128 per site and pattern of its +e_d bonds (and own spin)
    static constexpr int EROWS = FIELD ? (2 << D) : (1 << D);
    static constexpr size_t ETABLE = (size_t)2 * 4 * NBLK * EROWS * 512;
    static constexpr int PLANE = 2 * 4 * NQP;  // words of 32 replicas
    // planes per chunk: about 16 to 32 KB of spins, at most 16 planes (512 replicas)
    static constexpr int W = PLANE * 4 >= 4096 ? 8 : 16;
    static constexpr int COLS = 2 * 4 * NQP;   // sites, with the quads' padding
    static constexpr size_t OFFS = (size_t)COLS * 16;
    static constexpr size_t POS = ((size_t)N * 2 + 15) / 16 * 16;  // byte offset of a site in a plane
    static constexpr size_t SPIN = (size_t)W * PLANE * 4;
    static constexpr size_t SRC = (size_t)W * 32 * 4;  // the replicas' parents
    // the warps' energy sums of a slot
    static constexpr size_t EPART = NBLK > 1 ? (size_t)8 * W * NBLK * 64 : 0;
    static constexpr size_t GRAD = (size_t)(D + 1) * N * 4;
    static constexpr size_t O_OFFS = TABLE > ETABLE ? TABLE : ETABLE;
    static constexpr size_t O_POS = O_OFFS + OFFS, O_SPIN = O_POS + POS, O_SRC = O_SPIN + SPIN, O_EPART = O_SRC + SRC,
                            O_GRAD = O_EPART + EPART;
    static constexpr size_t SMEM = O_GRAD, SMEM_GRAD = O_GRAD + GRAD;
    static_assert(PLANE * 4 < 65536 && N % 4 == 0, "16-bit offsets within a plane, four sites at a time");
};

__device__ __forceinline__ uint32_t rotl32(uint32_t x, int n) { return __funnelshift_l(x, x, n); }
__device__ __forceinline__ uint32_t rotr32(uint32_t x, int n) { return __funnelshift_r(x, x, n); }

// address bits of a table column (quad block, lane) with byte 1 taken from
// byte B of the patterns: one permute per lookup
template <int B>
__device__ __forceinline__ uint32_t tab_addr(uint32_t idx4, uint32_t col)
{
    uint32_t a;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(a) : "r"(idx4), "r"(col), "n"(0x7604 | (B << 4)));
    return a;
}

// where site i sits in a plane, in bytes
template <int D, int L, bool FIELD>
__device__ __forceinline__ int tab_pos(int i)
{
    using SH = TabShape<D, L, FIELD>;
    const int q = i >> 1;
    return 4 * ((site_parity<D, L>(i) * 4 + (q & 3)) * SH::NQP + (q >> 2));
}

// neighbour offsets and positions of every site, once per instance
template <int D, int L, bool FIELD>
__device__ __forceinline__ void tab_stage_offsets(unsigned char* smem)
{
    using SH = TabShape<D, L, FIELD>;
    using LT = Lat<D, L>;
    uint4* offs = reinterpret_cast<uint4*>(smem + SH::O_OFFS);
    for (int u = threadIdx.x; u < SH::COLS; u += kTabThreads) {
        const int p = u / (4 * SH::NQP), v = u - p * 4 * SH::NQP, t = v / SH::NQP, q = 4 * (v - t * SH::NQP) + t;
        uint32_t o[6] = {0, 0, 0, 0, 0, 0};
        if (q < SH::NH) {
            const auto nb = LT::neighbours(p, q);
#pragma unroll
            for (int k = 0; k < 2 * D; ++k) o[k] = 4u * (uint32_t)((nb.q[k] & 3) * SH::NQP + (nb.q[k] >> 2));
        }
        offs[u] = make_uint4(o[0] | (o[1] << 16), o[2] | (o[3] << 16), o[4] | (o[5] << 16), 0u);
    }
    uint16_t* pos = reinterpret_cast<uint16_t*>(smem + SH::O_POS);
    for (int i = threadIdx.x; i < SH::N; i += kTabThreads) pos[i] = (uint16_t)tab_pos<D, L, FIELD>(i);
}

// couplings (in field order) and field of site (p, q)
template <int D, int L, bool FIELD>
__device__ __forceinline__ void tab_couplings(const RealInst& in, int p, int q, float (&J)[2 * D], float& h)
{
    using LT = Lat<D, L>;
    const auto nb = LT::neighbours(p, q);
#pragma unroll
    for (int k = 0; k < 2 * D; ++k) J[k] = __ldg(in.J + (k >> 1) * LT::N + ((k & 1) ? nb.site : nb.site_m[k >> 1]));
    h = FIELD ? __ldg(in.h + nb.site) : 0.0f;
}
// J with the sign of pattern bit k
__device__ __forceinline__ float tab_term(float J, uint32_t m, int k)
{
    return __uint_as_float(__float_as_uint(J) ^ (((m >> k) & 1u) << 31));
}
// f summed over the first K neighbours of pattern m (bit k: neighbour k is -1)
template <int K, int NB>
__device__ __forceinline__ float tab_sum(const float (&J)[NB], uint32_t m)
{
    float f = tab_term(J[0], m, 0);
#pragma unroll
    for (int k = 1; k < K; ++k) f = add32(f, tab_term(J[k], m, k));
    return f;
}

// thresholds of every site and pattern at this temperature.  The sums over the
// first three neighbours are kept for the patterns that share them.
template <int D, int L, bool FIELD>
__device__ __forceinline__ void tab_stage_thresholds(const RealInst& in, float beta, unsigned char* smem)
{
    using SH = TabShape<D, L, FIELD>;
    constexpr int NPAT = 1 << SH::KI;                    // neighbour patterns
    constexpr int NCOL = 2 * 4 * SH::NBLK * 32;          // table columns (sites)
    // threads per column: with eight, each takes one pattern of the first three neighbours
    constexpr int SPLIT = NCOL >= kTabThreads ? 1 : 8;
    constexpr int LOW = 8 / SPLIT;
    for (int it = threadIdx.x; it < NCOL * SPLIT; it += kTabThreads) {
        const int lane = it & 31, c = (it >> 5) % (NCOL / 32), part = it / NCOL;
        const int blk = c % SH::NBLK, t = (c / SH::NBLK) & 3, p = c / (4 * SH::NBLK);
        const int q = 4 * (blk * 32 + lane % SH::SEG) + t;
        unsigned char* col = smem + (size_t)(p * SH::NBLK + blk) * SH::BLOCK + SH::tpart(t) + lane * 4;
        const bool valid = q < SH::NH;
        float J[2 * D], h = 0.0f;
#pragma unroll
        for (int k = 0; k < 2 * D; ++k) J[k] = 0.0f;
        if (valid) tab_couplings<D, L, FIELD>(in, p, q, J, h);
        float s3[LOW];
#pragma unroll
        for (int i = 0; i < LOW; ++i) s3[i] = tab_sum<3>(J, (uint32_t)(SPLIT == 1 ? i : part));
#pragma unroll 1
        for (uint32_t hi = 0; hi < NPAT / 8; ++hi) {
            // without a field bit 2D - 1 of m is 0: the last neighbour is +1
            float t3[2 * D];
#pragma unroll
            for (int k = 3; k < 2 * D; ++k) t3[k] = tab_term(J[k], hi << 3, k);
#pragma unroll
            for (int i = 0; i < LOW; ++i) {
                const uint32_t m = (hi << 3) | (uint32_t)(SPLIT == 1 ? i : part);
                float f = s3[i];
#pragma unroll
                for (int k = 3; k < 2 * D; ++k) f = add32(f, t3[k]);
                // uphill for the spin +1 if x > 0, else for the spin -1 (or free)
                const float x = mul32(beta, mul32(add32(f, h), 2.0f));
                const bool pos = x > 0.0f;
                const float e = spec_expf(fminf(-fabsf(x), 0.0f));
                uint32_t up = e == 1.0f ? 0xFFFFFFFFu : __float2uint_rz(mul32(e, 4294967296.0f)), down = 0xFFFFFFFFu;
                if (!valid) up = down = 0u;  // the padding's spins never flip
                if constexpr (SH::WIDE) {
                    *reinterpret_cast<uint32_t*>(col + m * 256) = pos ? up : down;
                    *reinterpret_cast<uint32_t*>(col + (m + NPAT) * 256) = pos ? down : up;
                } else {
                    *reinterpret_cast<uint16_t*>(col + m * 256) = (uint16_t)((pos ? up : down) >> 16);
                    *reinterpret_cast<uint16_t*>(col + (m + NPAT) * 256) = (uint16_t)((pos ? down : up) >> 16);
                }
            }
        }
    }
}

// the specified decision for an attempt that the 16-bit compare leaves open
template <int D, int L, bool FIELD>
__device__ __noinline__ bool tab_exact(const RealInst& in, float beta, int p, int q, uint32_t pat, uint32_t r)
{
    using SH = TabShape<D, L, FIELD>;
    if (q >= SH::NH) return false;
    float J[2 * D], h;
    tab_couplings<D, L, FIELD>(in, p, q, J, h);
    const float f = add32(tab_sum<2 * D>(J, pat & ((1u << SH::KI) - 1u)), h);
    const float x = mul32(beta, mul32(f, 2.0f));
    return accept_real_exact(((pat >> SH::KI) & 1u) ? -x : x, r);
}

// energies of every site and pattern of its +e_d bonds (and own spin), rows of 32
// columns of type A (64 bits, in units of 2^(shift - 96), or 128)
template <int D, int L, bool FIELD, class A>
__device__ __forceinline__ void tab_stage_energies(const RealInst& in, unsigned char* smem)
{
    using SH = TabShape<D, L, FIELD>;
    using LT = Lat<D, L>;
    constexpr int N = SH::N, NCOL = 2 * 4 * SH::NBLK * 32;
    auto value = [&](const longlong2* p) -> A {
        const longlong2 v = __ldg(p);
        const __int128 x = ((__int128)v.y << 64) | (unsigned long long)v.x;
        return sizeof(A) == 8 ? (A)(x >> in.eshift) : (A)x;
    };
    for (int it = threadIdx.x; it < NCOL; it += kTabThreads) {
        const int lane = it & 31, c = it >> 5;
        const int blk = c % SH::NBLK, t = (c / SH::NBLK) & 3, p = c / (4 * SH::NBLK);
        const int q = 4 * (blk * 32 + lane % SH::SEG) + t;
        const bool valid = q < SH::NH;
        A J[D], h = 0;
#pragma unroll
        for (int d = 0; d < D; ++d) J[d] = 0;
        if (valid) {
            const auto nb = LT::neighbours(p, q);
#pragma unroll
            for (int d = 0; d < D; ++d) J[d] = value(&in.Jfix[d * N + nb.site]);
            if (FIELD) h = value(&in.hfix[nb.site]);
        }
        for (int m = 0; m < SH::EROWS; ++m) {
            A e = 0;
#pragma unroll
            for (int d = 0; d < D; ++d) e += ((m >> d) & 1) ? J[d] : -J[d];
            if (FIELD) e += ((m >> D) & 1) ? h : -h;
            *reinterpret_cast<A*>(smem + (((size_t)((p * 4 + t) * SH::NBLK + blk) * SH::EROWS + m) * 32 + lane) * sizeof(A)) = e;
        }
    }
}

// Energies of the block's replicas: exact sums of J 2^96 as int128, accumulated
// as 64-bit integers where every coupling and field is a multiple of 2^shift and
// the largest possible sum fits (in.eshift >= 0: half the additions, shuffles and
// table bytes).
template <int D, int L, bool FIELD, class A>
__device__ __forceinline__ void tab_energies(const RealInst& in, int R, int r0, int ng, int ga, int gb, int gstep,
                                             unsigned char* smem)
{
    using SH = TabShape<D, L, FIELD>;
    constexpr int NQP = SH::NQP, PLANE = SH::PLANE, ROT = sizeof(A) == 16 ? 1 : 0;
    constexpr int ROWB = 32 * (int)sizeof(A);  // bytes of a row: 256 or 512
    const int tid = threadIdx.x, lane = tid & 31;
    const int slot = tid / NQP, quad = tid - slot * NQP;
    const bool owner = quad < SH::NQ;
    const uint32_t* spin = reinterpret_cast<const uint32_t*>(smem + SH::O_SPIN);
    const unsigned char* planes = smem + SH::O_SPIN;
    const uint4* offs = reinterpret_cast<const uint4*>(smem + SH::O_OFFS);
    tab_stage_energies<D, L, FIELD, A>(in, smem);
    __syncthreads();
    auto store = [&](int r, A v) {
        const __int128 x = sizeof(A) == 8 ? (__int128)v << in.eshift : (__int128)v;
        longlong2 o;
        o.x = (long long)(unsigned long long)x;
        o.y = (long long)(x >> 64);
        in.E[r] = o;
    };
    auto shfl = [](const A& v, int off) -> A {
        if constexpr (sizeof(A) == 8) return __shfl_xor_sync(0xffffffffu, v, off);
        else {
            const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)v, off);
            const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(v >> 64), off);
            return (A)(((unsigned __int128)hi << 64) | lo);
        }
    };
    A* part = reinterpret_cast<A*>(smem + SH::O_EPART);
    const int wsl = quad >> 5;  // this warp's index within its slot
    const int gn = NQP < 32 ? (ng + SH::SLOTS - 1) / SH::SLOTS : gb - ga;  // warp-uniform trip count
    const uint32_t ecol = (uint32_t)((quad >> 5) * SH::EROWS * ROWB + lane * (int)sizeof(A));
    const uint32_t ehi = ((ecol >> 8) & 0xFFu) * 0x01010101u;
    int wheld = -1;
    uint32_t u[8][D + FIELD];  // pattern bits of the thread's eight sites, bit d rotated left by d + ROT
    for (int n = 0; n < gn; ++n) {
        const int g = ga + n * gstep;
        const bool act = g < gb;
        A e[4] = {0, 0, 0, 0};
        if (act && owner) {
            const int w = g >> 3, j = g & 7;
            if (w != wheld) {
                wheld = w;
#pragma unroll
                for (int pt = 0; pt < 8; ++pt) {
                    const uint4 o = offs[pt * NQP + quad];
                    const uint32_t op[3] = {o.x >> 16, o.y >> 16, o.z >> 16};
                    const uint32_t own = spin[w * PLANE + pt * NQP + quad];
                    const unsigned char* oth = planes + (w * PLANE + ((pt >> 2) ^ 1) * 4 * NQP) * 4;
#pragma unroll
                    for (int dd = 0; dd < D; ++dd)
                        u[pt][dd] = rotl32(own ^ *reinterpret_cast<const uint32_t*>(oth + op[dd]), dd + ROT);
                    if (FIELD) u[pt][D] = rotl32(own, D + ROT);
                }
            }
            const uint32_t bit = rotl32(0x01010101u, j + ROT);
#pragma unroll
            for (int pt = 0; pt < 8; ++pt) {
                // the pattern (twice the pattern for rows of 512 bytes) in each byte
                uint32_t x = 0;
#pragma unroll
                for (int dd = 0; dd < D + FIELD; ++dd) x |= u[pt][dd] & rotl32(bit, dd);
                x = rotr32(x, j) | ehi;
                const unsigned char* et = smem + (size_t)pt * SH::NBLK * SH::EROWS * ROWB;
                e[0] += *reinterpret_cast<const A*>(et + tab_addr<0>(x, ecol));
                e[1] += *reinterpret_cast<const A*>(et + tab_addr<1>(x, ecol));
                e[2] += *reinterpret_cast<const A*>(et + tab_addr<2>(x, ecol));
                e[3] += *reinterpret_cast<const A*>(et + tab_addr<3>(x, ecol));
            }
        }
        // sum over the quads; the first two steps also halve the replicas a
        // lane holds (lane bits 0 and 1 of the slot: replica)
        auto put = [&](int b, const A& v) {
            if constexpr (SH::NBLK > 1) part[(g * SH::NBLK + wsl) * 4 + b] = v;
            else if (r0 + 4 * g + b < R) store(r0 + 4 * g + b, v);
        };
        if constexpr (SH::SEG >= 4) {
            const bool h0 = lane & 1, h1 = lane & 2;
            A k0 = (h0 ? e[1] : e[0]) + shfl(h0 ? e[0] : e[1], 1);
            A k1 = (h0 ? e[3] : e[2]) + shfl(h0 ? e[2] : e[3], 1);
            A k = (h1 ? k1 : k0) + shfl(h1 ? k0 : k1, 2);
#pragma unroll
            for (int off = 4; off < SH::SEG; off <<= 1) k += shfl(k, off);
            if (act && (lane & (SH::SEG - 1)) < 4) put(lane & 3, k);
        } else {
#pragma unroll
            for (int off = 1; off < SH::SEG; off <<= 1) {
#pragma unroll
                for (int b = 0; b < 4; ++b) e[b] += shfl(e[b], off);
            }
            if (act && (lane & (SH::SEG - 1)) == 0) {
#pragma unroll
                for (int b = 0; b < 4; ++b) put(b, e[b]);
            }
        }
    }
    __syncthreads();  // the table, the planes and the parts are reused by the next chunk
    if constexpr (SH::NBLK > 1) {
        for (int t = tid; t < 4 * ng; t += kTabThreads) {
            A e = 0;
            for (int k = 0; k < SH::NBLK; ++k) e += part[((t >> 2) * SH::NBLK + k) * 4 + (t & 3)];
            if (r0 + t < R) store(r0 + t, e);
        }
        __syncthreads();
    }
}

// a slot's threads only share replicas among themselves
template <int NQP>
__device__ __forceinline__ void slot_sync(int slot)
{
    if constexpr (NQP <= 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(slot + 1), "n"(NQP) : "memory");
}

// Replica groups [gr0, gr1) (four replicas each, at most 8 W groups) of one
// instance: rows in, N_S sweeps, energies (and gradient counts into shared
// memory), rows out.  tab_stage_offsets must have run.
template <int D, int L, bool FIELD>
__device__ __forceinline__ void sweep_real_table(const RealStep& s, const RealInst& in, int R, int gr0, int gr1,
                                                 unsigned char* smem, bool grad)
{
    using SH = TabShape<D, L, FIELD>;
    constexpr int N = SH::N, NH = SH::NH, NQP = SH::NQP, KI = SH::KI, PLANE = SH::PLANE;
    constexpr int NWARP = kTabThreads / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ng = gr1 - gr0, nw = (ng + 7) >> 3, r0 = 4 * gr0;
    uint32_t* spin = reinterpret_cast<uint32_t*>(smem + SH::O_SPIN);
    const uint4* offs = reinterpret_cast<const uint4*>(smem + SH::O_OFFS);
    unsigned char* planes = smem + SH::O_SPIN;
    const uint16_t* pos = reinterpret_cast<const uint16_t*>(smem + SH::O_POS);
    constexpr int NC = (N + 31) / 32;
    const int lr = 4 * (lane & 7) + (lane >> 3);  // the replica of this lane's bit within its plane

    // ---- rows (gathered through parent) -> planes, 32 sites at a time: a lane
    // packs the sign bits of its replica, a transpose across the warp gives it a
    // site's word.  The parents go to shared memory first, and a warp has four
    // row pieces in flight (one at a time, two dependent loads each, took a
    // quarter of the kernel at 3D L = 10 with 132 replicas a block)
    int* psrc = reinterpret_cast<int*>(smem + SH::O_SRC);
    for (int t = tid; t < 32 * nw; t += kTabThreads) {
        const int r = r0 + t;
        psrc[t] = r < R && t < 4 * ng ? (in.parent ? in.parent[r] : r) : -1;
    }
    __syncthreads();  // offsets, positions, parents are staged
    constexpr int kBatch = 4;
    for (int tup0 = warp; tup0 < nw * NC; tup0 += NWARP * kBatch) {
        uint4 v[kBatch][2];
#pragma unroll
        for (int x = 0; x < kBatch; ++x) {
            const int tup = tup0 + x * NWARP, w = tup / NC, c = tup - w * NC;
            v[x][0] = v[x][1] = make_uint4(0u, 0u, 0u, 0u);
            const int src = tup < nw * NC ? psrc[32 * w + lr] : -1;
            if (src >= 0) {
                const uint4* row = reinterpret_cast<const uint4*>(in.Sin + (size_t)src * in.NP + 32 * c);
                v[x][0] = row[0];
                if (32 * c + 16 < in.NP) v[x][1] = row[1];
            }
        }
#pragma unroll
        for (int x = 0; x < kBatch; ++x) {
            const int tup = tup0 + x * NWARP, w = tup / NC, c = tup - w * NC;
            if (tup >= nw * NC) break;  // warp-uniform
            const uint32_t wv[8] = {v[x][0].x, v[x][0].y, v[x][0].z, v[x][0].w, v[x][1].x, v[x][1].y, v[x][1].z, v[x][1].w};
            uint32_t bits = 0;
#pragma unroll
            for (int t = 0; t < 8; ++t)  // bit 7 of the four bytes, gathered by a multiply
                bits |= ((((wv[t] >> 7) & 0x01010101u) * 0x01020408u) >> 24) << (4 * t);
            const uint32_t mine = transpose32(bits, lane);
            const int i = 32 * c + lane;
            if (i < N) *reinterpret_cast<uint32_t*>(planes + w * PLANE * 4 + pos[i]) = mine;
        }
    }
    if constexpr (NH % 4 != 0) {  // the last quad's missing sites
        for (int t = tid; t < nw * 8; t += kTabThreads) {
            const int w = t >> 3, p = (t >> 2) & 1, k = t & 3;
            if (4 * (NH >> 2) + k >= NH) spin[w * PLANE + (p * 4 + k) * NQP + (NH >> 2)] = 0u;
        }
    }
    tab_stage_thresholds<D, L, FIELD>(in, s.beta, smem);
    __syncthreads();

    // ---- N_S sweeps
    const int slot = tid / NQP, quad = tid - slot * NQP;
    const bool owner = quad < SH::NQ;
    const uint32_t c3 = in.c3;
    // whole slots in a warp take groups in turn (neighbouring slots then share
    // words), larger slots take runs of groups (one word's loads serve eight)
    int ga, gb, gstep;
    if constexpr (NQP < 32) {
        ga = slot; gb = ng; gstep = SH::SLOTS;
    } else {
        ga = ng * slot / SH::SLOTS; gb = ng * (slot + 1) / SH::SLOTS; gstep = 1;
    }
    for (int sw = 0; sw < s.n_sweeps; ++sw) {
#pragma unroll 1
        for (int p = 0; p < 2; ++p) {
            const uint32_t hs = s.hs0 + 2u * (uint32_t)sw + (uint32_t)p;
            // this thread's table column, and the bits of byte 1 that lie above the pattern
            const uint32_t col = (uint32_t)((p * SH::NBLK + (quad >> 5)) * SH::BLOCK + lane * 4);
            const uint32_t colhi = ((col >> 8) & 0xFFu) * 0x01010101u;
            if (owner) {
#pragma unroll 1
                for (int g = ga; g < gb;) {
                    const int w = g >> 3;
                    const int gend = NQP < 32 ? g + 1 : min(gb, 8 * w + 8);
                    uint32_t* cur = spin + w * PLANE + p * 4 * NQP + quad;
                    const unsigned char* oth = reinterpret_cast<const unsigned char*>(spin + w * PLANE + (p ^ 1) * 4 * NQP);
                    // pattern bits of the four sites, bit k rotated left by k so
                    // that those of one replica group do not overlap
                    uint32_t v[4][KI + 1];
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        uint32_t n[2 * D];
                        const uint4 o = offs[(p * 4 + t) * NQP + quad];
                        const uint32_t ow[3] = {o.x, o.y, o.z};
#pragma unroll
                        for (int k = 0; k < 2 * D; ++k)
                            n[k] = *reinterpret_cast<const uint32_t*>(oth + ((k & 1) ? ow[k >> 1] >> 16 : ow[k >> 1] & 0xFFFFu));
                        const uint32_t own = cur[t * NQP];
                        const uint32_t ref = FIELD ? 0u : n[2 * D - 1];
#pragma unroll
                        for (int k = 0; k < KI; ++k) v[t][k] = rotl32(n[k] ^ ref, k);
                        v[t][KI] = rotl32(own ^ ref, KI);
                    }
#pragma unroll 1
                    for (; g < gend; ++g) {
                        const int j = g & 7;
                        uint32_t flip[4], idx[4];
                        uint32_t bit = rotl32(0x01010101u, j);
                        const uint32_t hi = rotl32(colhi, j);
#pragma unroll
                        for (int t = 0; t < 4; ++t) { idx[t] = hi; flip[t] = 0; }
#pragma unroll
                        for (int k = 0; k <= KI; ++k) {
#pragma unroll
                            for (int t = 0; t < 4; ++t) idx[t] |= v[t][k] & bit;
                            bit = rotl32(bit, 1);
                        }
#pragma unroll
                        for (int t = 0; t < 4; ++t) idx[t] = rotr32(idx[t], j);
                        const uint32_t rep = (uint32_t)(r0 + 4 * g);
                        // attempts left open: a uniform of all ones (WIDE), or
                        // equal upper halves (a value below 0x10000)
                        uint32_t open = SH::WIDE ? 0u : 0xFFFFFFFFu;
                        auto replica = [&](auto BB) {
                            constexpr int b = decltype(BB)::value;
                            const u32x4 o = philox_rk((uint32_t)quad, hs, rep + b, c3, s.rk);
                            const uint32_t rs[4] = {o.x, o.y, o.z, o.w};
                            uint32_t th[4];
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                const unsigned char* e = smem + tab_addr<b>(idx[t], col);
                                if (SH::WIDE) th[t] = *reinterpret_cast<const uint32_t*>(e + SH::tpart(t));
                                // upper halves: sites 1 and 3 compare as they are
                                else if (t & 1) th[t] = *reinterpret_cast<const uint32_t*>(e + SH::tpart(t) - 2);
                                else th[t] = (uint32_t)*reinterpret_cast<const uint16_t*>(e + SH::tpart(t)) * 65536u;
                                if (rs[t] < th[t]) flip[t] |= 1u << (8 * b);
                            }
                            if (SH::WIDE) {
                                open = __vimax3_u32(open, rs[0], rs[1]);
                                open = __vimax3_u32(open, rs[2], rs[3]);
                            } else {
                                open = __vimin3_u32(open, rs[0] ^ th[0], rs[1] ^ th[1]);
                                open = __vimin3_u32(open, rs[2] ^ th[2], rs[3] ^ th[3]);
                            }
                        };
                        replica(std::integral_constant<int, 0>{});
                        replica(std::integral_constant<int, 1>{});
                        replica(std::integral_constant<int, 2>{});
                        replica(std::integral_constant<int, 3>{});
                        if (SH::WIDE ? open == 0xFFFFFFFFu : open < 0x10000u) {
#pragma unroll 1
                            for (int b = 0; b < 4; ++b) {
                                const u32x4 o = philox_rk((uint32_t)quad, hs, rep + b, c3, s.rk);
                                const uint32_t rs[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                                for (int t = 0; t < 4; ++t) {
                                    const uint32_t pat = (idx[t] >> (8 * b)) & (uint32_t)(SH::ROWS - 1);
                                    const unsigned char* e =
                                        smem + (col & ~0xFF00u) + (((idx[t] >> (8 * b)) & 0xFFu) << 8) + SH::tpart(t);
                                    if (SH::WIDE ? rs[t] != 0xFFFFFFFFu : (rs[t] >> 16) != *reinterpret_cast<const uint16_t*>(e)) continue;
                                    const bool acc = tab_exact<D, L, FIELD>(in, s.beta, p, 4 * quad + t, pat, rs[t]);
                                    flip[t] = (flip[t] & ~(1u << (8 * b))) | ((uint32_t)acc << (8 * b));
                                }
                            }
                        }
#pragma unroll
                        for (int t = 0; t < 4; ++t) atomicXor(cur + t * NQP, flip[t] << j);
                    }
                    if constexpr (NQP < 32) g += gstep - 1;
                }
            }
            slot_sync<NQP>(slot);
        }
    }
    __syncthreads();

    // ---- gradient counts: n - 2 popc of the differing replicas
    if (grad) {
        int* gJ = reinterpret_cast<int*>(smem + SH::O_GRAD);
        int* gh = gJ + D * N;
        const int nrep = min(4 * ng, R - r0);
        for (int u = tid; u < SH::COLS; u += kTabThreads) {
            const int p = u / (4 * NQP), vv = u - p * 4 * NQP, t = vv / NQP, q = 4 * (vv - t * NQP) + t;
            if (q >= NH) continue;
            const int i = Lat<D, L>::neighbours(p, q).site;
            const uint4 o = offs[u];
            const uint32_t op[3] = {o.x >> 16, o.y >> 16, o.z >> 16};
            int neg = 0, diff[3] = {0, 0, 0};
            for (int w = 0; w < nw; ++w) {
                // replicas 4 j + b < nrep - 32 w of the plane: bits 8 b + j
                const int left = nrep - 32 * w;
                uint32_t valid = 0xFFFFFFFFu;
                if (left < 32) {
                    valid = 0;
                    for (int b = 0; b < 4; ++b) {
                        const int cnt = left > b ? (left - b + 3) >> 2 : 0;  // groups that hold this byte's replica
                        valid |= ((1u << cnt) - 1u) << (8 * b);
                    }
                }
                const uint32_t own = spin[w * PLANE + u];
                const unsigned char* oth = reinterpret_cast<const unsigned char*>(spin + w * PLANE + (p ^ 1) * 4 * NQP);
                neg += __popc(own & valid);
#pragma unroll
                for (int dd = 0; dd < D; ++dd)
                    diff[dd] += __popc((own ^ *reinterpret_cast<const uint32_t*>(oth + op[dd])) & valid);
            }
            gh[i] += nrep - 2 * neg;
#pragma unroll
            for (int dd = 0; dd < D; ++dd) gJ[dd * N + i] += nrep - 2 * diff[dd];
        }
    }
    // ---- rows out: the transpose back, then a byte per bit
    for (int tup = warp; tup < nw * NC; tup += NWARP) {
        const int w = tup / NC, c = tup - w * NC, i = 32 * c + lane;
        const uint32_t bits =
            transpose32(i < N ? *reinterpret_cast<const uint32_t*>(planes + w * PLANE * 4 + pos[i]) : 0u, lane);
        uint32_t wv[8];
#pragma unroll
        for (int t = 0; t < 8; ++t)  // 1 -> -1 (0xFF), 0 -> +1
            wv[t] = (((((bits >> (4 * t)) & 15u) * 0x00204081u) & 0x01010101u) * 0xFEu) ^ 0x01010101u;
        const int r = r0 + 32 * w + lr;
        if (r < R && 32 * w + lr < 4 * ng) {
            uint4* row = reinterpret_cast<uint4*>(in.Sout + (size_t)r * in.NP + 32 * c);
            row[0] = make_uint4(wv[0], wv[1], wv[2], wv[3]);
            if (32 * c + 16 < in.NP) row[1] = make_uint4(wv[4], wv[5], wv[6], wv[7]);
        }
    }
    // ---- energies: the table gives way to the sites' energies
    if (in.eshift >= 0) tab_energies<D, L, FIELD, long long>(in, R, r0, ng, ga, gb, gstep, smem);
    else tab_energies<D, L, FIELD, __int128>(in, R, r0, ng, ga, gb, gstep, smem);
}

// zero the block's gradient sums; add them to the step's counters at the end
template <int D, int L, bool FIELD>
__device__ __forceinline__ void tab_zero_grad(unsigned char* smem)
{
    using SH = TabShape<D, L, FIELD>;
    int* gJ = reinterpret_cast<int*>(smem + SH::O_GRAD);
    for (int t = threadIdx.x; t < (D + 1) * SH::N; t += kTabThreads) gJ[t] = 0;
}
template <int D, int L, bool FIELD>
__device__ __forceinline__ void tab_flush_grad(const RealInst& in, unsigned char* smem)
{
    using SH = TabShape<D, L, FIELD>;
    constexpr int N = SH::N;
    const int* gJ = reinterpret_cast<const int*>(smem + SH::O_GRAD);
    const int* gh = gJ + D * N;
    for (int t = threadIdx.x; t < D * N; t += kTabThreads)
        if (gJ[t]) atomicAdd(&in.cJ[t], (unsigned long long)(long long)gJ[t]);
    for (int t = threadIdx.x; t < N; t += kTabThreads)
        if (gh[t]) atomicAdd(&in.ch[t], (unsigned long long)(long long)gh[t]);
}

// an instance's replica groups spread evenly over the grid; a block goes through
// its share in chunks of at most 8 W groups
template <int D, int L, bool FIELD>
__global__ void __launch_bounds__(kTabThreads) sweep_real_table_kernel(RealSweepArgs a)
{
    using SH = TabShape<D, L, FIELD>;
    extern __shared__ __align__(128) unsigned char smem_tab[];
    const int R = a.i.Rdev ? __ldg(a.i.Rdev) : a.i.R;
    const long long G4 = (R + 3) / 4;
    const int g0 = (int)(G4 * blockIdx.x / gridDim.x), g1 = (int)(G4 * (blockIdx.x + 1) / gridDim.x);
    if (g0 >= g1) return;  // block-uniform
    const bool grad = a.i.cJ != nullptr;
    tab_stage_offsets<D, L, FIELD>(smem_tab);
    if (grad) tab_zero_grad<D, L, FIELD>(smem_tab);
    const int nc = (g1 - g0 + 8 * SH::W - 1) / (8 * SH::W);
    for (int c = 0; c < nc; ++c) {
        const int a0 = g0 + (int)((long long)(g1 - g0) * c / nc), a1 = g0 + (int)((long long)(g1 - g0) * (c + 1) / nc);
        sweep_real_table<D, L, FIELD>(a.s, a.i, R, a0, a1, smem_tab, grad);
    }
    if (grad) tab_flush_grad<D, L, FIELD>(a.i, smem_tab);
}

template <int D, int L, bool FIELD>
static cudaError_t launch_real_table(const RealSweepArgs& a, cudaStream_t st)
{
    using SH = TabShape<D, L, FIELD>;
    auto kern = sweep_real_table_kernel<D, L, FIELD>;
    static std::atomic<unsigned long long> done{0};
    const cudaError_t e = allow_smem(kern, (int)SH::SMEM_GRAD, done);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per = 0;
    const size_t smem = a.i.cJ ? SH::SMEM_GRAD : SH::SMEM;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kTabThreads, smem);
    const int G4 = (a.i.R + 3) / 4, least = 32 / SH::SEG;  // at least a full warp of groups
    const int most = (G4 + least - 1) / least;
    const int grid = sms * (per > 0 ? per : 1);
    kern<<<grid < most ? grid : most, kTabThreads, smem, st>>>(a);
    return cudaGetLastError();
}

// launch for the lattices of one translation unit (with or without a field);
// *handled is false where the table does not fit
cudaError_t launch_sweep_real_table_plain(int D, int L, const RealSweepArgs& a, cudaStream_t st, bool* handled);
cudaError_t launch_sweep_real_table_field(int D, int L, const RealSweepArgs& a, cudaStream_t st, bool* handled);

}  // namespace pa
