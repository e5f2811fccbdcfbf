// pa_resample.cu -- resampling, observables and the gradient backward pass.
//
// Resampling (Sec. II.B): when beta rises to beta', replica i gets on average
// R w_i / S copies, w_i = exp[-(beta'-beta)(E_i - E_min)], S = sum_i w_i
// (multinomial: R independent draws).  Free-energy perturbation: ln Q =
// -(beta'-beta) E_min + ln S - ln R and beta F_k = -N ln 2 - sum_{l<=k} ln Q_l.
//
// Fixed order, so that the draws do not depend on the launch geometry:
// runs of 32 weights are summed left to right; the run totals are summed the
// same way, recursively, until one run is left; entry j of run c is
// Q_{c-1} + l_j (l_j its sum inside the run, Q the inclusive prefix of the
// run totals; run 0: l_j alone).  P_i is the running maximum of those sums
// (exact; it only repairs the one-unit steps that two summation orders can
// leave at a run boundary) and S = P_{R-1}.  Draw q (RES stream) picks the
// smallest i with u_q S < P_i (if u_q S == S after rounding: the smallest i
// with P_i >= u_q S).  Copy numbers are exact integer counts; their exclusive
// scan places the copies of replica i in slots [C_i, C_i + n_i), so families
// stay contiguous (Sec. V.A).
#include "pa_device.cuh"
#include "pa_internal.h"
#include "pa_launch.h"

namespace pa {

__device__ __forceinline__ __int128 ll2_to_i128(longlong2 v)
{
    return ((__int128)v.y << 64) | (unsigned long long)v.x;
}

__device__ __forceinline__ double e_minus_min_to_double(const ResampleArgs& a, int i)
{
    if (a.kind == 0) return (double)(a.E32[i] - (int)a.prev->emin_lo);  // exact integer
    __int128 emin = ((__int128)a.prev->emin_hi << 64) | (unsigned long long)a.prev->emin_lo;
    return __dmul_rn(i128_to_double(ll2_to_i128(a.E128[i]) - emin), 0x1p-96);
}

// true in the block that finishes last (each of n_blocks calls it once); the
// counter is reset for the next launch.  Writes before the call are visible
// to the last block: one acquire-release addition after the block's barrier
// (a fence on each side of a relaxed one took about 1 us more).
__device__ __forceinline__ bool last_block(int* counter, int n_blocks)
{
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        int done;
        asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(done) : "l"(counter) : "memory");
        s_last = done == n_blocks - 1;
        if (s_last) *counter = 0;
    }
    __syncthreads();
    return s_last;
}

constexpr int kWThreads = 256;

// source population: in device memory for the nearest-integer scheme
__device__ __forceinline__ int rs_src(const ResampleArgs& a) { return a.Rsrc ? *a.Rsrc : a.R; }

// Weights and the two lowest levels of the prefix, one block of T threads per
// kWBlock weights.  GB300 has little FP64 throughput (two operations a clock
// and SM), so every operation of the specified order is executed once: thread c
// of the first warp sums run c (32 weights, staged in shared memory) left to
// right, then one thread sums the block's run totals left to right.  +-J
// energies of a block span a few dozen to a few hundred levels, so the block
// evaluates each level's weight once (spec_exp64 of the same argument) and looks
// the weights up.
//
// Two shapes (and the cluster below).  Populations of at most kFuseR: the last
// block to finish sums levels 1 and up and completes the run search table and S
// (rs_fused): a second and third launch cost more than one SM's work.  Blocks of
// 1024 weights with +-J, where a block evaluates few exponentials and more warps
// serve the last block; of 256 with real couplings, so that the exponentials (one
// per replica) spread over the SMs.  Larger ones: 1024 weights and 256 threads, so
// that several blocks' dependent FP64 chains overlap on an SM, and the run table
// is its own launch (rs_runs_kernel).  By ncu: +-J R = 10^5 level table + weights +
// finalize 24 us -> 14.3 (blocks of 256: 16.9), most of it 62-cycle FP64 additions
// in a chain; real couplings R = 5 x 10^4 20.2 us in blocks of 1024, 16.8 of 256.
constexpr int kFuseR = 128 * kWBlock;
// weights of replicas i0 + tid + j T, j < PER (those below i0 + n), into w; tab:
// PER T doubles of shared memory; also to a.w for the nearest-integer scheme
template <int T, int PER>
__device__ __forceinline__ void rs_block_weights(const ResampleArgs& a, int i0, int n, int emin, double (&w)[PER],
                                                 double* tab)
{
    __shared__ int s_lo[T / 32], s_hi[T / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (a.kind == 0) {
        int lv[PER], lo = 0x7fffffff, hi = -1;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int t = tid + j * T;
            lv[j] = t < n ? a.E32[i0 + t] - emin : -1;
            if (t < n) {
                lo = min(lo, lv[j]);
                hi = max(hi, (lv[j] & 3) ? 0x7ffffffe : lv[j]);  // not a level: no table
            }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) { s_lo[warp] = lo; s_hi[warp] = hi; }
        __syncthreads();
        lo = __reduce_min_sync(0xffffffffu, lane < T / 32 ? s_lo[lane] : 0x7fffffff);
        hi = __reduce_max_sync(0xffffffffu, lane < T / 32 ? s_hi[lane] : -1);
        // levels lo/4 .. hi/4 evaluated once each
        const int nlev = hi < 0x7ffffff0 && lo >= 0 ? (hi >> 2) - (lo >> 2) + 1 : PER * T;
        if (nlev <= PER * T / 2) {
            for (int t = tid; t < nlev; t += T)
                tab[t] = spec_exp64(-__dmul_rn(a.dbeta, (double)(4 * ((lo >> 2) + t))));
            __syncthreads();
#pragma unroll
            for (int j = 0; j < PER; ++j) w[j] = lv[j] >= 0 ? tab[(lv[j] >> 2) - (lo >> 2)] : 0.0;
        } else {
#pragma unroll
            for (int j = 0; j < PER; ++j)
                w[j] = tid + j * T < n ? spec_exp64(-__dmul_rn(a.dbeta, (double)lv[j])) : 0.0;
        }
    } else {
#pragma unroll
        for (int j = 0; j < PER; ++j)
            w[j] = tid + j * T < n ? spec_exp64(-__dmul_rn(a.dbeta, e_minus_min_to_double(a, i0 + tid + j * T))) : 0.0;
    }
    if (a.scheme == 1) {
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (tid + j * T < n) a.w[i0 + tid + j * T] = w[j];
    }
}
// Sum of a run of cnt <= kFan weights at x, left to right, the sums left in place
// (starting from +0 and adding +0 past the end changes nothing: no sum is
// negative).  By whole warps.  The barriers keep the loads and stores out of the
// chain of additions: stored one by one between them they hold up the next
// addition (32 additions by one warp 3500 cycles, with the barriers 2260).
__device__ __forceinline__ double rs_run_sums(double* x, int cnt)
{
    double tot = 0.0;
#pragma unroll
    for (int j0 = 0; j0 < kFan; j0 += 8) {
        if (j0 > 0 && !__any_sync(0xffffffffu, j0 < cnt)) break;
        double v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = j0 + j < cnt ? x[j0 + j] : 0.0;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = tot = __dadd_rn(tot, v[j]);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j0 + j < cnt) x[j0 + j] = v[j];
    }
    return tot;
}
// the sums of the warp's values, left to right: lane l gets that of lanes 0 .. l
template <int N>
__device__ __forceinline__ double rs_lane_sums(double mine)
{
    const int lane = threadIdx.x & 31;
    double acc = 0.0, res = 0.0;
#pragma unroll
    for (int c0 = 0; c0 < N; c0 += 8) {
        double v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = __shfl_sync(0xffffffffu, mine, c0 + c);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = acc = __dadd_rn(acc, v[c]);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (lane == c0 + c) res = v[c];
    }
    return res;
}
// a weights block of kWBlock weights by T threads: levels 0 and 1
template <int T>
__device__ __forceinline__ void rs_levels_body(const ResampleArgs& a, int b, int R, int emin)
{
    constexpr int PER = kWBlock / T;
    __shared__ double s_w[kFan * (kFan + 1)];  // run c at [c (kFan + 1)], padded against bank conflicts
    const int i0 = b * kWBlock;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = min(kWBlock, R - i0);
    if (tid == 0 && a.bcount && b < rs_scan_blocks(R)) a.bcount[b] = 0;
    double w[PER];
    rs_block_weights<T, PER>(a, i0, n, emin, w, s_w);
    __syncthreads();  // the level table in s_w has been read
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int t = tid + j * T;
        if (t < n) s_w[(t / kFan) * (kFan + 1) + t % kFan] = w[j];
    }
    __syncthreads();
    const int nruns = (n + kFan - 1) / kFan;
    if (warp == 0) {
        const double tot = rs_run_sums(s_w + lane * (kFan + 1), min(kFan, n - lane * kFan));
        const double l1 = rs_lane_sums<kFan>(tot);  // the block's run totals (0 past the last)
        if (lane == 31) a.upper[b] = l1;
        if (lane < nruns) {
            a.lev1[b * kFan + lane] = l1;
            if (a.runP) a.runP[b * kFan + lane] = tot;
        }
    }
    __syncthreads();
    for (int t = tid; t < n; t += T) a.P[i0 + t] = s_w[(t / kFan) * (kFan + 1) + t % kFan];
}

// one weights block's run table, by one warp (lane = run c): q_c, the sum of
// everything before the run (Q1_{c-1}), and the largest cumulative weight up to
// the run's end inside the block; returns the block's largest.  Inside a run
// q_c + l_i does not decrease, so the smallest i with P_i > x lies in the first
// run whose entry here exceeds x: the cumulative weights themselves are never
// written out.
__device__ __forceinline__ long long dbits(double x);
__device__ __forceinline__ long long rs_run_table(const ResampleArgs& a, int b, int R, const double* upper)
{
    const int lane = threadIdx.x & 31, c = b * kFan + lane;
    double q = 0.0;
    long long m = 0;  // bits of +0.0: weights are >= 0
    const bool live = (long long)c * kFan < R;
    if (live) {
        const double tot = __ldcg(a.runP + c);
        if (c > 0) {
            const double l1 = __ldcg(a.lev1 + c - 1);
            const int cb = (c - 1) / kFan;  // block of run c - 1
            q = cb == 0 ? l1 : __dadd_rn(upper[cb - 1], l1);
        }
        m = dbits(c == 0 ? tot : __dadd_rn(q, tot));
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, m, o);
        if (lane >= o) m = max(m, u);
    }
    if (live) {
        a.runq[c] = q;
        a.runP[c] = __longlong_as_double(m);
    }
    return __shfl_sync(0xffffffffu, m, 31);
}

__device__ __forceinline__ void rs_top_levels(double* up, int nb);
// the last sub-block of a population of at most kFuseR: levels 1 and up of the
// prefix, run table, running maximum over the weights blocks, S
constexpr int kFuseBlocks = kFuseR / kWBlock;
template <int T>
__device__ __forceinline__ void rs_fused(const ResampleArgs& a, int R)
{
    // run totals, then the level-1 sums, of weights block b at [b (kFan + 1)]
    __shared__ double s_l1[kFuseBlocks * (kFan + 1)];
    __shared__ double s_up[rs_upper_size(kFuseR)];
    __shared__ long long s_bm[kFuseBlocks];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = rs_wblocks(R), leaves = rs_leaves(R);
    for (int t = tid; t < nb * kFan; t += T)
        s_l1[(t / kFan) * (kFan + 1) + t % kFan] = t < leaves ? __ldcg(a.runP + t) : 0.0;
    if (tid < kFuseBlocks) s_bm[tid] = 0;
    __syncthreads();
    if (warp < (nb + 31) / 32) {
        const double tot = rs_run_sums(s_l1 + tid * (kFan + 1), tid < nb ? kFan : 0);
        if (tid < nb) s_up[tid] = tot;
    }
    __syncthreads();
    rs_top_levels(s_up, nb);
    double next = warp * kFan + lane < leaves ? __ldcg(a.runP + warp * kFan + lane) : 0.0;
    for (int b = warp; b < nb; b += T / 32) {
        const int c = b * kFan + lane;
        const double tot = next;
        next = c + T < leaves ? __ldcg(a.runP + c + T) : 0.0;
        const int pb = lane > 0 ? b : b - 1;  // block of run c - 1
        double q = 0.0;
        if (c > 0) {
            const double l1 = s_l1[pb * (kFan + 1) + (lane > 0 ? lane - 1 : kFan - 1)];
            q = pb == 0 ? l1 : __dadd_rn(s_up[pb - 1], l1);
        }
        long long m = c < leaves ? dbits(c == 0 ? tot : __dadd_rn(q, tot)) : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, m, o);
            if (lane >= o) m = max(m, u);
        }
        if (c < leaves) {
            a.runq[c] = q;
            a.runP[c] = __longlong_as_double(m);
        }
        if (lane == 31) s_bm[b] = m;
    }
    __syncthreads();
    if (warp == 0) {
        constexpr int PER = kFuseBlocks / 32;
        long long v[PER], m = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) { m = max(m, s_bm[lane * PER + j]); v[j] = m; }
        long long inc = m;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc = max(inc, u);
        }
        long long before = __shfl_up_sync(0xffffffffu, inc, 1);
        if (lane == 0) before = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int b = lane * PER + j;
            if (b < nb) a.bmax[nb + b] = __longlong_as_double(j == 0 ? before : max(before, v[j - 1]));
        }
        if (lane == 31) a.cur->S = __longlong_as_double(inc);
    }
}
// a sub-block: its weights and the sums inside its eight runs
template <int T>
__global__ void __launch_bounds__(T) rs_weights_fused_kernel(ResampleArgs a)
{
    constexpr int kRuns = T / kFan;
    __shared__ double s_w[kRuns * (kFan + 1)];
    const int R = rs_src(a), live = max(1, (R + T - 1) / T);
    const int b = blockIdx.x, i0 = b * T, tid = threadIdx.x;
    if (b >= live) return;  // block-uniform: past the source population
    const int n = min(T, R - i0);
    if (tid == 0 && i0 % rs_scan_size(R) == 0 && i0 / rs_scan_size(R) < rs_scan_blocks(R)) a.bcount[i0 / rs_scan_size(R)] = 0;
    double w[1];
    rs_block_weights<T, 1>(a, i0, n, (int)a.prev->emin_lo, w, s_w);
    __syncthreads();  // the level table in s_w has been read
    s_w[(tid / kFan) * (kFan + 1) + tid % kFan] = w[0];  // 0 past the population
    __syncthreads();
    if (tid < 32) {
        const double tot = rs_run_sums(s_w + min(tid, kRuns - 1) * (kFan + 1), tid < kRuns ? kFan : 0);
        if (tid < kRuns && tid * kFan < n) a.runP[b * kRuns + tid] = tot;
    }
    __syncthreads();
    if (tid < n) a.P[i0 + tid] = s_w[(tid / kFan) * (kFan + 1) + tid % kFan];
    if (last_block(a.sync, live)) rs_fused<T>(a, R);
}

__device__ __forceinline__ void rs_top_body(const ResampleArgs& a);
// blocks of an instance that take part (block 0 always: it resets the copy
// totals and S even of a population that died out)
__device__ __forceinline__ int rs_live_blocks(int R) { return max(1, rs_wblocks(R)); }
template <int T>
__device__ __forceinline__ void rs_weights_launch(const ResampleArgs& a, int b)
{
    const int R = rs_src(a), live = rs_live_blocks(R);
    if (b >= live) return;  // block-uniform: past the source population
    rs_levels_body<T>(a, b, R, (int)a.prev->emin_lo);
    if (!last_block(a.sync, live)) return;
    rs_top_body(a);  // levels >= 2 of the prefix
}
__global__ void __launch_bounds__(kWThreads) rs_weights_kernel(ResampleArgs a) { rs_weights_launch<kWThreads>(a, blockIdx.x); }
__global__ void __launch_bounds__(kWThreads) rs_weights_batched(const ResampleArgs* tab)
{
    rs_weights_launch<kWThreads>(tab[blockIdx.y], blockIdx.x);
}
// a shard: the levels >= 2 need every shard's block totals
__global__ void __launch_bounds__(kWThreads) rs_weights_shard_kernel(ResampleArgs a)
{
    rs_levels_body<kWThreads>(a, blockIdx.x, a.R, (int)a.prev->emin_lo);
}

// Levels >= 2 of the prefix, by one block: bottom-up sums inside runs of the nb
// block totals at up, then
// top-down Q_{c-1} + l_j; up[0 .. nb) ends as the inclusive prefix.
__device__ __forceinline__ void rs_top_levels(double* up, int nb)
{
    constexpr int kMaxLev = 8;  // kFan^(kMaxLev+1) > 2^31 weights
    const int tid = threadIdx.x, nt = blockDim.x;
    int base[kMaxLev], len[kMaxLev], nl = 0;
    int n = nb, off = 0;
    for (;;) {
        base[nl] = off; len[nl] = n; ++nl;
        const int nc = n <= kFan ? 1 : (n + kFan - 1) / kFan;
        for (int c = tid; c - (tid & 31) < nc; c += nt) {  // by whole warps
            const int cnt = c < nc ? min(kFan, n - c * kFan) : 0;
            const double acc = rs_run_sums(up + off + (cnt ? c * kFan : 0), cnt);
            if (c < nc && n > kFan) up[off + n + c] = acc;
        }
        __syncthreads();
        if (n <= kFan) break;  // one run left: its sums are the prefix of this level
        off += n;
        n = nc;
    }
    for (int v = nl - 2; v >= 0; --v) {
        double* x = up + base[v];
        const double* q = up + base[v + 1];
        for (int j = kFan + tid; j < len[v]; j += nt) x[j] = __dadd_rn(q[j / kFan - 1], x[j]);
        __syncthreads();
    }
}
__device__ __forceinline__ void rs_top_body(const ResampleArgs& a)
{
    rs_top_levels(a.upper, rs_wblocks(a.gR ? a.gR : rs_src(a)));  // a shard sums the global block totals
}
__global__ void __launch_bounds__(kWBlock) rs_top_kernel(ResampleArgs a) { rs_top_body(a); }

// Non-negative doubles compare as their bit patterns do (as signed 64-bit
// integers): maxima and the draw search use the integer compare, which is
// exact and leaves GB300's scarce FP64 units to the specified additions.
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }

// (shards) Level 0 and the running maximum inside one weights block: weight i of run
// c gets Q1_{c-1} + l_i (Q1_{c-1} = Q2_{b'-1} + l1_{c-1} with b' the block of
// run c - 1, the level-1 sums alone in block 0), then P_i = the largest of
// these up to i within the block; bmax[b] = the block's largest.
__device__ __forceinline__ void rs_finalize_body(const ResampleArgs& a, int b)
{
    constexpr int PER = kWBlock / kWThreads;  // consecutive weights per thread
    __shared__ double s_q[kFan];
    __shared__ long long s_m[kWThreads / 32];
    const int R = rs_src(a);
    const int i0 = b * kWBlock;
    if (i0 >= R) return;  // block-uniform
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cg0 = a.gb0 * kFan;  // global index of local run 0 (0 unless a shard)
    if (tid < kFan) {  // Q1 of the run before run c = b kFan + tid (one addition per run)
        const int c = b * kFan + tid;
        double q = 0.0;
        if (cg0 + c > 0 && c * kFan < R) {
            const int cb = (cg0 + c - 1) / kFan;  // global block of run c - 1
            // l1 of run c - 1; before a shard's first run it is the last run of
            // the previous (remote) block, whose l1 is that block's total
            const double l1 = c > 0 ? a.lev1[c - 1] : a.t2g[cb];
            q = cb == 0 ? l1 : __dadd_rn(a.upper[cb - 1], l1);
        }
        s_q[tid] = q;
    }
    __syncthreads();
    long long v[PER];
    long long m = 0;  // bits of +0.0: weights are >= 0
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = i0 + tid * PER + j;
        long long x = 0;
        if (i < R) {
            const double l = a.P[i];
            x = dbits(cg0 == 0 && i < kFan ? l : __dadd_rn(s_q[(tid * PER + j) / kFan], l));
        }
        m = max(m, x);
        v[j] = m;  // inclusive maximum within this thread's weights
    }
    long long incl = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl = max(incl, u);
    }
    if (lane == 31) s_m[warp] = incl;
    const long long up = __shfl_up_sync(0xffffffffu, incl, 1);
    __syncthreads();
    long long before = lane > 0 ? up : 0;
    for (int w = 0; w < warp; ++w) before = max(before, s_m[w]);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = i0 + tid * PER + j;
        if (i < R) a.P[i] = __longlong_as_double(max(before, v[j]));
    }
    if (tid == 0) {
        long long bm = 0;
        for (int w = 0; w < kWThreads / 32; ++w) bm = max(bm, s_m[w]);
        a.bmax[b] = __longlong_as_double(bm);
    }
}
// running maximum over the weights blocks (bmax[nb + b] = the largest
// cumulative weight before block b) and S, the largest cumulative weight; one
// block, as many block maxima per pass as it has threads (integer maxima of the
// bit patterns)
__device__ __forceinline__ void rs_blockmax_body(const ResampleArgs& a)
{
    __shared__ long long s_w[32];
    __shared__ long long s_carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R = a.gR ? a.gR : rs_src(a);  // a shard: the global block maxima
    const int nb = rs_wblocks(R);
    if (tid == 0) s_carry = 0;
    __syncthreads();
    const int nt = blockDim.x;
    for (int b0 = 0; b0 < nb; b0 += nt) {
        const int b = b0 + tid;
        long long m = b < nb ? dbits(a.bmax[b]) : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, m, o);
            if (lane >= o) m = max(m, u);
        }
        if (lane == 31) s_w[warp] = m;
        const long long carry = s_carry;
        __syncthreads();
        long long before = carry;
        for (int w = 0; w < warp; ++w) before = max(before, s_w[w]);
        const long long up = __shfl_up_sync(0xffffffffu, m, 1);
        const long long excl = lane > 0 ? max(before, up) : before;
        if (b < nb) a.bmax[nb + b] = __longlong_as_double(excl);
        if (tid == nt - 1) s_carry = max(before, m);
        __syncthreads();
    }
    if (tid == 0) a.cur->S = __longlong_as_double(s_carry);
}
// ln Q and the running free energy, by one thread, once S is there
__device__ __forceinline__ void rs_lnq(const ResampleArgs& a)
{
    const double S = a.cur->S;
    double emin_d;
    if (a.kind == 0) {
        emin_d = (double)(int)a.prev->emin_lo;
    } else {
        __int128 emin = ((__int128)a.prev->emin_hi << 64) | (unsigned long long)a.prev->emin_lo;
        emin_d = __dmul_rn(i128_to_double(emin), 0x1p-96);
    }
    const double log_R = a.Rsrc ? log((double)rs_src(a)) : a.log_R;
    const double lnQ = __dsub_rn(__dadd_rn(-__dmul_rn(a.dbeta, emin_d), log(S)), log_R);
    const double sum = __dadd_rn(a.prev->sum_lnQ, lnQ);
    a.cur->lnQ = lnQ;
    a.cur->sum_lnQ = sum;
    a.cur->betaF = __dsub_rn(a.betaF0, sum);
    if (a.lnQ_out) *a.lnQ_out = lnQ;
}
__global__ void __launch_bounds__(kWThreads) rs_finalize_shard_kernel(ResampleArgs a) { rs_finalize_body(a, blockIdx.x); }
__global__ void __launch_bounds__(kWBlock) rs_blockmax_shard_kernel(ResampleArgs a)
{
    rs_blockmax_body(a);
    __syncthreads();
    if (threadIdx.x == 0) rs_lnq(a);
}

// the run table of a population above kFuseR: one warp per weights block, the
// last block takes the running maximum over the weights blocks and S
constexpr int kRunWarps = 8;
__device__ __forceinline__ void rs_runs_launch(const ResampleArgs& a, int blk)
{
    const int R = rs_src(a), nb = rs_wblocks(R), live = max(1, (nb + kRunWarps - 1) / kRunWarps);
    if (blk >= live) return;
    const int b = blk * kRunWarps + (threadIdx.x >> 5);
    if (b < nb) {
        const long long m = rs_run_table(a, b, R, a.upper);
        if ((threadIdx.x & 31) == 0) a.bmax[b] = __longlong_as_double(m);
    }
    if (last_block(a.sync + 3, live)) rs_blockmax_body(a);
}
__global__ void __launch_bounds__(32 * kRunWarps) rs_runs_kernel(ResampleArgs a) { rs_runs_launch(a, blockIdx.x); }
__global__ void __launch_bounds__(32 * kRunWarps) rs_runs_batched(const ResampleArgs* tab)
{
    rs_runs_launch(tab[blockIdx.y], blockIdx.x);
}

// Multinomial draws: the smallest i with x < P_i.  Each block stages the ends of
// the segments of P (whole weights blocks) in shared memory and finds a draw's
// segment there; the block's run table gives the run, four ways at a time (three
// independent loads a round, three rounds, instead of five dependent loads), and
// rs_first_near the index.  Copies are counted per replica and, through shared
// memory, per scan block, so that the placement needs no pass over the counts
// first.
constexpr int kDrawThreads = 512;
constexpr int kMaxSeg = 2048;
constexpr int kMaxHist = 1024;   // scan blocks counted in shared memory
__device__ __forceinline__ int rs_seg_blocks(int nb)
{
    int s = 1;
    while ((nb + s - 1) / s > kMaxSeg) s *= 2;
    return s;
}
// the first index of 32 where pred holds (it holds somewhere, and from there on)
template <class Pred>
__device__ __forceinline__ int first_of_32(Pred pred)
{
    const bool p7 = pred(7), p15 = pred(15), p23 = pred(23);
    int lo = p7 ? 0 : p15 ? 8 : p23 ? 16 : 24;
    const bool q1 = pred(lo + 1), q3 = pred(lo + 3), q5 = pred(lo + 5);
    lo += q1 ? 0 : q3 ? 2 : q5 ? 4 : 6;
    return pred(lo) ? lo : lo + 1;
}
// v 2^-53 for v < 2^53, exactly, as the double's bits: integer work instead of
// an FP64 conversion and product
__device__ __forceinline__ double uniform53_int(uint32_t hi, uint32_t lo)
{
    const unsigned long long v = (unsigned long long)(hi >> 5) << 26 | (lo >> 6);
    if (v == 0) return 0.0;
    const int lz = __clzll((long long)v);
    return __longlong_as_double((long long)(((unsigned long long)(1032 - lz) << 52) + (v << (lz - 11))));
}
// The first i of run c (sums l_0 .. l_{n-1}, q before the run) with q + l_i past x.
// q + l_i does not decrease with i and x - q, rounded, is within a unit of the
// sum that reaches x, so the search compares l_i with it (integer compares of the
// bit patterns) and the specified sums settle the last step or two: two or three
// FP64 additions a draw instead of seven (GB300 has few FP64 units).
template <class Past, class Load>
__device__ __forceinline__ int rs_first_in_run(double q, long long x, int n, Past past, Load load)
{
    const long long t = dbits(__dsub_rn(__longlong_as_double(x), q));  // negative: below every sum
    int i = first_of_32([&](int j) { return j >= n || dbits(load(j)) >= t; });
    auto reached = [&](int j) { return past(dbits(__dadd_rn(q, load(j)))); };
    i = min(i, n - 1);
    while (i > 0 && reached(i - 1)) --i;
    while (i < n - 1 && !reached(i)) ++i;
    return i;
}
// about the double's value, by integer work (only ever a guess)
__device__ __forceinline__ float about(long long bits)
{
    return __int_as_float((int)max((bits >> 29) - (896ll << 23), 0ll));
}
// The same search for sums in global memory (l 32-byte aligned; readable up to
// the next multiple of 32 bytes), four sums a load from where x would lie among
// equal weights (next: the sum before the following run).  The lookups per lane
// are what the search costs: two to four here, a dozen by three at a time.
template <class Past>
__device__ __forceinline__ int rs_first_near(const double* l, double q, double next, long long x, int n, Past past)
{
    const long long t = dbits(__dsub_rn(__longlong_as_double(x), q));
    const float fq = about(dbits(q)), frac = (about(x) - fq) / (about(dbits(next)) - fq);
    const int smax = (n - 1) >> 2;
    int s = min(max((int)(frac * (kFan / 4)), 0), smax), i;
    long long v0, v1, v2, v3;
    bool left = false, right = false;
    for (;;) {
        asm("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(v0), "=l"(v1), "=l"(v2), "=l"(v3) : "l"(l + 4 * s));
        if (s < smax && v3 < t) {  // past this quad
            i = 4 * ++s;
            if (left) break;
            right = true;
        } else if (s > 0 && !right && v0 >= t) {
            --s;
            left = true;
        } else {
            const int m = n - 4 * s;
            i = 4 * s + (v0 < t) + (m > 1 && v1 < t) + (m > 2 && v2 < t) + (m > 3 && v3 < t);
            break;
        }
    }
    i = min(i, n - 1);
    auto reached = [&](int j) { return past(dbits(__dadd_rn(q, l[j]))); };
    while (i > 0 && reached(i - 1)) --i;
    while (i < n - 1 && !reached(i)) ++i;
    return i;
}
__device__ __forceinline__ void rs_draws_body(const ResampleArgs& a, int q0, int per)
{
    __shared__ long long s_end[kMaxSeg];
    __shared__ int s_hist[kMaxHist];
    const int R = a.R, tid = threadIdx.x, nt = blockDim.x;
    const int nb = rs_wblocks(R), leaves = rs_leaves(R);
    const int sb = rs_seg_blocks(nb), nseg = (nb + sb - 1) / sb;
    const int ns = rs_scan_blocks(R), sbits = rs_scan_size(R);
    const bool hist = ns <= kMaxHist;
    const double S = a.cur->S;
    // largest P up to the end of block b: the largest before block b + 1, or S
    auto block_end = [&](int b) { return b + 1 < nb ? dbits(a.bmax[nb + b + 1]) : dbits(S); };
    for (int k = tid; k < nseg; k += nt) s_end[k] = block_end(min(nb - 1, k * sb + sb - 1));
    if (hist)
        for (int k = tid; k < ns; k += nt) s_hist[k] = 0;
    __syncthreads();
    for (int d = 0; d < per; ++d) {
        const int q = q0 + d * nt + tid;
        if (q >= a.Rn) break;
        const u32x4 o = philox((uint32_t)q, (uint32_t)a.k, 0u, a.c3, a.key0, a.key1);
        const long long x = dbits(__dmul_rn(uniform53_int(o.x, o.y), S));  // x >= 0
        int lo = 0, hi = nseg;  // first segment whose end exceeds x
        while (lo < hi) {
            const int mid = lo + ((hi - lo) >> 1);
            if (x < s_end[mid]) hi = mid; else lo = mid + 1;
        }
        const bool strict = lo < nseg;  // some P exceeds x; else x == S after rounding: the first P >= x
        int b0 = strict ? lo * sb : 0, b1 = strict ? min(nb - 1, lo * sb + sb - 1) : nb - 1;
        while (b0 < b1) {
            const int mid = b0 + ((b1 - b0) >> 1);
            const long long e = block_end(mid);
            if (strict ? x < e : e >= x) b1 = mid; else b0 = mid + 1;
        }
        // the largest P before the block does not pass the test, so neither it
        // nor the runs before the first that does matter
        const int c = b0 * kFan + first_of_32([&](int t) {
            if (b0 * kFan + t >= leaves) return true;
            const long long p = dbits(a.runP[b0 * kFan + t]);
            return strict ? x < p : p >= x;
        });
        const int cc = min(c, leaves - 1), i0 = cc * kFan;
        const int w = i0 + rs_first_near(a.P + i0, a.runq[cc], cc + 1 < leaves ? a.runq[cc + 1] : S, x, min(kFan, R - i0),
                                         [&](long long p) { return strict ? x < p : p >= x; });
        atomicAdd(&a.counts[w], 1);
        if (hist) atomicAdd(&s_hist[w / sbits], 1);
        else atomicAdd(&a.bcount[w / sbits], 1);
    }
    if (!hist) return;  // block-uniform
    __syncthreads();
    for (int k = tid; k < ns; k += nt)
        if (s_hist[k]) atomicAdd(&a.bcount[k], s_hist[k]);
}
// A shard's draws: all gR global draws are evaluated, a draw's weights block
// is found from the global block ends, and only draws that land on a local
// block are resolved (bisection in the local P) and counted.
__device__ __forceinline__ void rs_draws_shard_body(const ResampleArgs& a, int q)
{
    __shared__ long long s_end[kMaxSeg];
    const int nb = rs_wblocks(a.gR), nloc = rs_wblocks(a.R);
    const int sb = rs_seg_blocks(nb), nseg = (nb + sb - 1) / sb;
    const double S = a.cur->S;
    // largest P up to the end of block b: the largest before block b + 1, or S
    auto block_end = [&](int b) { return b + 1 < nb ? dbits(a.bmax[nb + b + 1]) : dbits(S); };
    for (int k = threadIdx.x; k < nseg; k += blockDim.x) s_end[k] = block_end(min(nb - 1, k * sb + sb - 1));
    __syncthreads();
    if (q >= a.Rn) return;
    const u32x4 o = philox((uint32_t)q, (uint32_t)a.k, 0u, a.c3, a.key0, a.key1);
    const long long x = dbits(__dmul_rn(uniform53(o.x, o.y), S));  // x >= 0
    int lo = 0, hi = nseg;
    while (lo < hi) {
        const int mid = lo + ((hi - lo) >> 1);
        if (x < s_end[mid]) hi = mid; else lo = mid + 1;
    }
    const bool strict = lo < nseg;  // some P exceeds x; else x == S: the first P >= x
    int b0 = strict ? lo * sb : 0, b1 = strict ? min(nb - 1, lo * sb + sb - 1) : nb - 1;
    while (b0 < b1) {  // the first block whose end exceeds x (or reaches x)
        const int mid = b0 + ((b1 - b0) >> 1);
        const long long e = block_end(mid);
        if (strict ? x < e : e >= x) b1 = mid; else b0 = mid + 1;
    }
    const int bl = b0 - a.gb0;
    if (bl < 0 || bl >= nloc) return;  // another shard's draw
    const long long before = dbits(a.bmax[nb + b0]);
    int i = bl * kWBlock, j = min(a.R, i + kWBlock) - 1;
    while (i < j) {
        const int mid = i + ((j - i) >> 1);
        const long long p = max(before, dbits(a.P[mid]));
        if (strict ? x < p : p >= x) j = mid; else i = mid + 1;
    }
    atomicAdd(&a.counts[i], 1);
}
__global__ void __launch_bounds__(kDrawThreads) rs_draws_shard_kernel(ResampleArgs a)
{
    rs_draws_shard_body(a, blockIdx.x * blockDim.x + threadIdx.x);
}
// Draws of a population of at most kFuseR: the whole run table in shared memory
// (at most 64 KB), one block per SM, so that a draw makes only the gathers inside
// its run.  Random gathers are what a draw costs: one L1 lookup per lane and load
// (twenty a draw through global tables took half of the launch).  By ncu +-J
// R = 10^5 10.3 -> 7.9 us, R = 5 x 10^4 8.3 -> 6.4 us.
__global__ void __launch_bounds__(1024) rs_draws_fused_kernel(ResampleArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_draws[];
    static_assert(kFuseR <= kSmallScanR, "scan blocks of 1024");
    __shared__ int s_hist[kFuseR / 1024];
    const int R = a.R, tid = threadIdx.x, nt = blockDim.x;
    const int nb = rs_wblocks(R), leaves = rs_leaves(R), ns = rs_scan_blocks(R);
    long long* s_end = reinterpret_cast<long long*>(smem_draws);      // largest cumulative weight up to each run's end
    double* s_q = reinterpret_cast<double*>(smem_draws) + leaves;     // sum before each run
    for (int c = tid; c < leaves; c += nt) {
        s_end[c] = max(dbits(a.bmax[nb + c / kFan]), dbits(a.runP[c]));
        s_q[c] = a.runq[c];
    }
    if (tid < ns) s_hist[tid] = 0;
    const double S = a.cur->S;
    __syncthreads();
    const int q = blockIdx.x * nt + tid;
    if (q < a.Rn) {
        const u32x4 o = philox((uint32_t)q, (uint32_t)a.k, 0u, a.c3, a.key0, a.key1);
        const long long x = dbits(__dmul_rn(uniform53_int(o.x, o.y), S));  // x >= 0
        const bool strict = x < s_end[leaves - 1];  // else x == S after rounding: the first P >= x
        auto past = [&](long long p) { return strict ? x < p : p >= x; };
        int lo = 0, hi = leaves - 1;  // the first run whose end is past x (the last one is)
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (past(s_end[mid])) hi = mid; else lo = mid + 1;
        }
        const int i0 = lo * kFan;
        const int w = i0 + rs_first_near(a.P + i0, s_q[lo], lo + 1 < leaves ? s_q[lo + 1] : S, x, min(kFan, R - i0), past);
        atomicAdd(&a.counts[w], 1);
        atomicAdd(&s_hist[w / 1024], 1);
    }
    __syncthreads();
    if (tid < ns && s_hist[tid]) atomicAdd(&a.bcount[tid], s_hist[tid]);
}
static cudaError_t launch_draws_fused(const ResampleArgs& a, cudaStream_t st)
{
    static std::atomic<unsigned long long> done{0};
    const cudaError_t e = allow_smem(rs_draws_fused_kernel, 16 * rs_leaves(kFuseR), done);
    if (e != cudaSuccess) return e;
    // one block per SM where that gives it 128 to 1024 draws
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int t = ((a.Rn + sms - 1) / sms + 31) / 32 * 32;
    t = t < 128 ? 128 : t > 1024 ? 1024 : t;
    rs_draws_fused_kernel<<<(a.Rn + t - 1) / t, t, 16 * rs_leaves(a.R), st>>>(a);
    return cudaGetLastError();
}

// two draws a thread in large populations: half the flushes of the copy totals
constexpr int kDrawPer = 2;
__global__ void __launch_bounds__(kDrawThreads) rs_draws_kernel(ResampleArgs a, int per)
{
    rs_draws_body(a, blockIdx.x * blockDim.x * per, per);
}
__global__ void __launch_bounds__(kDrawThreads) rs_draws_batched(const ResampleArgs* tab)
{
    const ResampleArgs& a = tab[blockIdx.y];
    if ((int)(blockIdx.x * blockDim.x) >= a.Rn) return;  // block-uniform: no draw of this instance
    rs_draws_body(a, blockIdx.x * blockDim.x, 1);
}

// nearest-integer copy numbers (Sec. II.B, population in expectation):
// tau_i = target w_i / S, n_i = floor(tau_i) + [u_i < tau_i - floor(tau_i)],
// u_i from the RESAMPLE stream at counter (i, k, 1)
__device__ __forceinline__ int rs_nearest_copies(const ResampleArgs& a, int i, double S)
{
    const u32x4 o = philox((uint32_t)i, (uint32_t)a.k, 1u, a.c3, a.key0, a.key1);
    const double u = uniform53_int(o.x, o.y);
    const double tau = __ddiv_rn(__dmul_rn(a.target, a.w[i]), S);
    const double fl = floor(tau);
    return (int32_t)fl + (u < __dsub_rn(tau, fl) ? 1 : 0);
}
__global__ void __launch_bounds__(256) rs_nearest_kernel(ResampleArgs a)
{
    __shared__ int s_n[8];
    const int R = rs_src(a), i = blockIdx.x * 256 + threadIdx.x;
    if ((int)blockIdx.x * 256 >= R) return;  // block-uniform
    int n = 0;
    if (i < R) {
        n = rs_nearest_copies(a, i, a.cur->S);
        a.counts[i] = n;
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0) s_n[threadIdx.x >> 5] = n;
    __syncthreads();
    if (threadIdx.x < 32) {
        n = __reduce_add_sync(0xffffffffu, threadIdx.x < 8 ? s_n[threadIdx.x] : 0);
        // 256 replicas lie in one scan block
        if (threadIdx.x == 0) atomicAdd(&a.bcount[(blockIdx.x * 256) / rs_scan_size(R)], n);
    }
}

// ---- copy-number scan and placement of a shard ----
__device__ __forceinline__ void rs_blocksum_body(const int32_t* counts, int R, int32_t* blocksum, int b)
{
    __shared__ int ws[32];
    const int tid = threadIdx.x;
    int s = 0;
    for (int t = 0; t < kScanBlock / 1024; ++t) {
        const int i = b * kScanBlock + t * 1024 + tid;
        if (i < R) s += counts[i];
    }
    s = __reduce_add_sync(0xffffffffu, s);
    if ((tid & 31) == 0) ws[tid >> 5] = s;
    __syncthreads();
    if (tid < 32) {
        int v = __reduce_add_sync(0xffffffffu, ws[tid]);
        if (tid == 0) blocksum[b] = v;
    }
}
__global__ void __launch_bounds__(1024) rs_blocksum_shard_kernel(ResampleArgs a)
{
    rs_blocksum_body(a.counts, a.R, a.blocksum, blockIdx.x);
}

__device__ __forceinline__ int rs_scan_blocks_body(int32_t* blocksum, int nb)
{
    int acc = 0;
    for (int b = 0; b < nb; ++b) {
        const int v = blocksum[b];
        blocksum[b] = acc;
        acc += v;
    }
    return acc;
}
__global__ void rs_scan_shard_kernel(ResampleArgs a)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int nbs = (a.R + kScanBlock - 1) / kScanBlock;
    a.blocksum[nbs] = rs_scan_blocks_body(a.blocksum, nbs);  // the copies placed
}

// exclusive scan inside the block + block offset; write parents and families
__device__ __forceinline__ void rs_fill_body(const ResampleArgs& a, int b)
{
    __shared__ int ws[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int PER = kScanBlock / 1024;
    const int i0 = b * kScanBlock + tid * PER;
    int c[PER];
    int s = 0;
    const int R = rs_src(a);
    const int cap = a.Rdst ? a.cap : 0x7fffffff;
#pragma unroll
    for (int t = 0; t < PER; ++t) {
        c[t] = (i0 + t < R) ? a.counts[i0 + t] : 0;
        s += c[t];
    }
    int incl = s;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int v = ws[lane];
        int inc = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += u;
        }
        ws[lane] = inc - v;  // exclusive warp offsets
    }
    __syncthreads();
    int off = a.blocksum[b] + ws[warp] + (incl - s);
    const int pbase = a.gb0 * kWBlock;  // a shard writes global replica indices
#pragma unroll
    for (int t = 0; t < PER; ++t) {
        const int i = i0 + t;
        if (i < R) {
            const int f = a.fam_in[i];
            const int n = min(c[t], max(cap - off, 0));  // slots past the capacity are dropped
            for (int u = 0; u < n; ++u) {
                a.parent[off + u] = pbase + i;
                a.fam_out[off + u] = f;
            }
            off += c[t];
            a.counts[i] = 0;
        }
    }
}
__global__ void __launch_bounds__(1024) rs_fill_shard_kernel(ResampleArgs a) { rs_fill_body(a, blockIdx.x); }

// Placement: a block takes one scan block of SB replicas.  Its first slot is the
// sum of the copy totals before it; the inclusive scan of its copy numbers stays
// in shared memory and every thread takes slots, finding the slot's replica there
// by bisection, so that a replica with many copies is written by the whole block
// (one thread per replica took 6.8 ms when one replica filled 10^6 slots).
// Block 0 also takes the logarithm of S, beside the placement.
template <int SB>
__device__ __forceinline__ void rs_place_body(const ResampleArgs& a, int b, int R)
{
    constexpr int PER = SB / 1024;
    __shared__ int s_cum[SB], s_fam[SB];
    __shared__ int s_w[32], s_off;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i0 = b * SB, ns = rs_scan_blocks(R);
    int c[PER], s = 0, pre = 0, all = 0;
#pragma unroll
    for (int t = 0; t < PER; ++t) {
        const int i = i0 + tid * PER + t;
        c[t] = i < R ? __ldcg(a.counts + i) : 0;
        s_fam[tid * PER + t] = i < R && a.fam_in ? a.fam_in[i] : 0;
        s += c[t];
        c[t] = s;
    }
    for (int t = tid; t < ((a.Rdst && b == 0) ? ns : b); t += 1024) {
        const int v = __ldcg(a.bcount + t);
        all += v;
        if (t < b) pre += v;
    }
    // inclusive scan of the copy numbers over the block
    int incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    pre = __reduce_add_sync(0xffffffffu, b == 0 ? all : pre);
    if (lane == 31) s_w[warp] = incl;
    if (tid == 0) s_off = 0;
    __syncthreads();
    if (lane == 0 && pre) atomicAdd(&s_off, pre);
    int before = lane < warp ? s_w[lane] : 0;
    before = __reduce_add_sync(0xffffffffu, before);
#pragma unroll
    for (int t = 0; t < PER; ++t) {
        const int i = i0 + tid * PER + t;
        s_cum[tid * PER + t] = before + incl - s + c[t];
        if (i < R) a.counts[i] = 0;
    }
    __syncthreads();
    const int total = s_cum[SB - 1], cap = a.Rdst ? a.cap : 0x7fffffff;
    const int off = b == 0 ? 0 : s_off;
    if (b == 0 && tid == 0 && a.Rdst) {  // the drawn population, copies beyond the capacity dropped
        const int Rn = min(s_off, cap);
        *a.Rdst = Rn;
        *a.Rdst_d = (double)Rn;
    }
    for (int t = tid; t < total && off + t < cap; t += 1024) {
        int lo = 0, hi = SB - 1;  // the first replica whose inclusive sum exceeds t
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (t < s_cum[mid]) hi = mid; else lo = mid + 1;
        }
        a.parent[off + t] = i0 + lo;
        if (a.fam_out) a.fam_out[off + t] = s_fam[lo];
    }
}

// A population of at most kClusterR replicas: the whole resampling in one launch
// of one cluster, a CTA per weights block.  The steps between which the larger
// populations change launches are cluster barriers here (every CTA of a cluster
// is resident, and the barrier's release and acquire order the global writes),
// and every CTA completes the few values above its block by itself.  Always eight
// CTAs: the draws, FP64 operations of which an SM completes one warp's in 19
// cycles, are shared out among them even if one block has all the weights.  By
// ncu: R = 1000 18.6 us with one CTA, 14.5 us with eight (the launches of the larger
// populations: 25 us); R = 4096 20.5 -> 18.4 us by the caller's clock.
constexpr int kClusterCtas = 8;  // the portable cluster size
constexpr int kClusterR = kClusterCtas * kWBlock;
// staged, so that the draws' gathers stay off the L1 lookups: the sums inside the runs
constexpr int cluster_smem(int R) { return (int)sizeof(double) * R; }
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__global__ void __launch_bounds__(kWBlock) rs_cluster_kernel(ResampleArgs a)
{
    constexpr int kRuns = kClusterCtas * kFan;
    __shared__ double s_up[kClusterCtas], s_rp[kRuns], s_rq[kRuns];
    __shared__ long long s_end[kClusterCtas];
    __shared__ int s_hist[kClusterCtas], s_min[32];
    extern __shared__ __align__(16) unsigned char smem_cluster[];
    double* s_P = reinterpret_cast<double*>(smem_cluster);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x, R = rs_src(a), nb = rs_wblocks(R), leaves = rs_leaves(R);
    int emin = 0;
    if (a.self) {
        // no earlier launch: E_min, and the copy numbers' initial zeros
        int m = 0x7fffffff;
        for (int t = tid; t < R; t += kWBlock) m = min(m, a.E32[t]);
        m = __reduce_min_sync(0xffffffffu, m);
        if (lane == 0) s_min[warp] = m;
        __syncthreads();
        emin = __reduce_min_sync(0xffffffffu, s_min[lane]);
        if (b * kWBlock + tid < R) a.counts[b * kWBlock + tid] = 0;
        if (b == 0 && tid == 0) {
            StepAcc* prev = const_cast<StepAcc*>(a.prev);
            prev->emin_lo = emin;
            prev->emin_hi = emin < 0 ? -1 : 0;
            prev->sum_lnQ = 0.0;
        }
    } else if (a.kind == 0) {
        emin = (int)a.prev->emin_lo;
    }
    if (b < rs_live_blocks(R)) rs_levels_body<kWBlock>(a, b, R, emin);
    cluster_sync();
    if (warp == 0) {  // at most kFan block totals: one run of the next level
        const double up = rs_lane_sums<kClusterCtas>(lane < nb ? __ldcg(a.upper + lane) : 0.0);
        if (lane < nb) s_up[lane] = up;
    }
    if (tid < kClusterCtas) s_hist[tid] = 0;
    __syncthreads();
    if (warp == 0 && b < nb) {
        const long long m = rs_run_table(a, b, R, s_up);
        if (lane == 0) a.bmax[b] = __longlong_as_double(m);
    }
    cluster_sync();
    for (int t = tid; t < leaves; t += kWBlock) {
        s_rp[t] = __ldcg(a.runP + t);
        s_rq[t] = __ldcg(a.runq + t);
    }
    if (a.scheme == 0)
        for (int t = tid; t < R; t += kWBlock) s_P[t] = __ldcg(a.P + t);
    if (warp == 0) {
        long long m = lane < nb ? dbits(__ldcg(a.bmax + lane)) : 0;
#pragma unroll
        for (int o = 1; o < kClusterCtas; o <<= 1) m = max(m, __shfl_up_sync(0xffffffffu, m, o));
        if (lane < nb) s_end[lane] = m;
        if (b == kClusterCtas - 1 && lane == kClusterCtas - 1) a.cur->S = __longlong_as_double(m);
    }
    __syncthreads();
    const double S = nb > 0 ? __longlong_as_double(s_end[nb - 1]) : 0.0;
    if (b == kClusterCtas - 1 && tid == kWBlock - 1) rs_lnq(a);  // rarely a warp with draws
    if (a.scheme == 1) {
        const int i = b * kWBlock + tid;
        int n = 0;
        if (i < R) {
            n = rs_nearest_copies(a, i, S);
            a.counts[i] = n;
        }
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0 && n) atomicAdd(&s_hist[b], n);
    } else {
        const int share = ((a.Rn + kClusterCtas - 1) / kClusterCtas + 31) / 32 * 32, end = min(a.Rn, (b + 1) * share);
        for (int q = b * share + tid; q < end; q += kWBlock) {
            const u32x4 o = philox((uint32_t)q, (uint32_t)a.k, 0u, a.c3, a.key0, a.key1);
            const long long x = dbits(__dmul_rn(uniform53_int(o.x, o.y), S));  // x >= 0
            const bool strict = x < s_end[nb - 1];  // else x == S after rounding: the first P >= x
            auto past = [&](long long p) { return strict ? x < p : p >= x; };
            int bl = 0;
            while (bl < nb - 1 && !past(s_end[bl])) ++bl;
            const int c = min(leaves - 1, bl * kFan + first_of_32([&](int t) {
                return bl * kFan + t >= leaves || past(dbits(s_rp[bl * kFan + t]));
            }));
            const int i = c * kFan + rs_first_in_run(s_rq[c], x, min(kFan, R - c * kFan), past,
                                                     [&](int t) { return s_P[c * kFan + t]; });
            atomicAdd(&a.counts[i], 1);
            atomicAdd(&s_hist[i / kWBlock], 1);
        }
    }
    __syncthreads();
    if (tid < nb && s_hist[tid]) atomicAdd(&a.bcount[tid], s_hist[tid]);
    cluster_sync();
    if (b < max(1, rs_scan_blocks(R))) rs_place_body<kWBlock>(a, b, R);
}

__device__ __forceinline__ void rs_place_launch(const ResampleArgs& a, int b)
{
    if (b == (int)gridDim.x - 1) {  // one more block than the placement needs: two FP64 logarithms
        if (threadIdx.x == 0) rs_lnq(a);
        return;
    }
    const int R = rs_src(a);
    if (b >= max(1, rs_scan_blocks(R))) return;  // block-uniform
    if (rs_scan_size(R) == 1024) rs_place_body<1024>(a, b, R);
    else rs_place_body<4096>(a, b, R);
}
__global__ void __launch_bounds__(1024) rs_place_kernel(ResampleArgs a) { rs_place_launch(a, blockIdx.x); }
__global__ void __launch_bounds__(1024) rs_place_batched(const ResampleArgs* tab) { rs_place_launch(tab[blockIdx.y], blockIdx.x); }

// blocks that cover the scan blocks of every population up to R: a smaller one
// (drawn on the device) may have smaller scan blocks
static int place_grid(int R) { return rs_bcount_size(R); }

cudaError_t launch_resample(const ResampleArgs& a, cudaStream_t st)
{
    // a.R sizes the grids (the capacity when the population is in device memory)
    if (a.R <= kClusterR) {
        static std::atomic<unsigned long long> done{0};
        const cudaError_t e = allow_smem(rs_cluster_kernel, cluster_smem(kClusterR), done);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = kClusterCtas;
        cfg.blockDim = kWBlock;
        cfg.dynamicSmemBytes = cluster_smem(a.R);
        cfg.stream = st;
        cudaLaunchAttribute at = {};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kClusterCtas;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, rs_cluster_kernel, a);
    }
    const bool fused = a.R <= kFuseR;
    if (fused) {
        if (a.kind == 0) rs_weights_fused_kernel<1024><<<(a.R + 1023) / 1024, 1024, 0, st>>>(a);
        else rs_weights_fused_kernel<256><<<(a.R + 255) / 256, 256, 0, st>>>(a);
    } else {
        rs_weights_kernel<<<rs_wblocks(a.R), kWThreads, 0, st>>>(a);
        rs_runs_kernel<<<(rs_wblocks(a.R) + kRunWarps - 1) / kRunWarps, 32 * kRunWarps, 0, st>>>(a);
    }
    if (a.scheme == 1)
        rs_nearest_kernel<<<(a.R + 255) / 256, 256, 0, st>>>(a);
    else if (fused) {
        const cudaError_t e = launch_draws_fused(a, st);
        if (e != cudaSuccess) return e;
    } else
        rs_draws_kernel<<<(a.Rn + kDrawPer * kDrawThreads - 1) / (kDrawPer * kDrawThreads), kDrawThreads, 0, st>>>(a, kDrawPer);
    rs_place_kernel<<<place_grid(a.R) + 1, 1024, 0, st>>>(a);
    return cudaGetLastError();
}
int resample_launches(const ResampleArgs& a) { return a.R <= kClusterR ? 1 : a.R <= kFuseR ? 3 : 4; }
bool resample_one_launch(int R) { return R <= kClusterR; }

// the phases of a shard's resampling (the host exchanges the block totals,
// the block maxima and the copy totals between them)
cudaError_t launch_resample_shard(const ResampleArgs& a, int phase, cudaStream_t st)
{
    const int nb = (a.R + kScanBlock - 1) / kScanBlock;
    switch (phase) {
    case 0:  // weights, levels 0 and 1 of the local blocks -> local block totals in upper
        rs_weights_shard_kernel<<<rs_wblocks(a.R), kWThreads, 0, st>>>(a);
        break;
    case 1:  // global levels >= 2 (upper holds every shard's block totals), local P, block maxima
        rs_top_kernel<<<1, kWBlock, 0, st>>>(a);
        rs_finalize_shard_kernel<<<rs_wblocks(a.R), kWThreads, 0, st>>>(a);
        break;
    case 2:  // running maximum over every shard's blocks, S, ln Q; draws; copy totals
        rs_blockmax_shard_kernel<<<1, kWBlock, 0, st>>>(a);
        rs_draws_shard_kernel<<<(a.Rn + kDrawThreads - 1) / kDrawThreads, kDrawThreads, 0, st>>>(a);
        rs_blocksum_shard_kernel<<<nb, 1024, 0, st>>>(a);
        rs_scan_shard_kernel<<<1, 32, 0, st>>>(a);
        break;
    default:  // placement: global parent indices and families of the local copies
        rs_fill_shard_kernel<<<nb, 1024, 0, st>>>(a);
        break;
    }
    return cudaGetLastError();
}

cudaError_t launch_resample_batched(const ResampleArgs* tab, int n_inst, int maxR, cudaStream_t st)
{
    const unsigned ni = (unsigned)n_inst;
    rs_weights_batched<<<dim3(rs_wblocks(maxR), ni), kWThreads, 0, st>>>(tab);
    rs_runs_batched<<<dim3((rs_wblocks(maxR) + kRunWarps - 1) / kRunWarps, ni), 32 * kRunWarps, 0, st>>>(tab);
    rs_draws_batched<<<dim3((maxR + kDrawThreads - 1) / kDrawThreads, ni), kDrawThreads, 0, st>>>(tab);
    rs_place_batched<<<dim3(place_grid(maxR) + 1, ni), 1024, 0, st>>>(tab);
    return cudaGetLastError();
}

// c ln c for c < kLogC (entries 0 and 1 are never read: a run of one adds 0)
__global__ void logc_table_kernel(double* t)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < kLogC) t[c] = c > 0 ? __dmul_rn((double)c, log((double)c)) : 0.0;
}
cudaError_t launch_logc_table(double* t, cudaStream_t st)
{
    logc_table_kernel<<<(kLogC + 255) / 256, 256, 0, st>>>(t);
    return cudaGetLastError();
}

// ---------------- observables (Sec. V.A, Eq. 9; Sec. II.B, Eq. 2) ----------------
// At most kObsBlocks blocks each reduce a contiguous slice of the population; the
// last block to finish combines the partials.  Sums of +-J energies and the
// family entropy's sum of c ln c are integers (a term is a double of at least 1,
// so a multiple of 2^-52: two 64-bit sums hold every one exactly), the same in
// any order and off the FP64 units; real-coupling energies are FP64 in a fixed
// order.  The partition depends only on R, so the result does not depend on the
// GPU.  The launch is latency: one round of loads, then short chains.  A run of
// equal family ids ends at the next start, found from the warp's ballot, the
// other warps' first starts, and only for the last run of a window by a search
// beyond it (the whole warp, 32 probes a round).  R = 10^5: 15.6 -> 10.1 us, 5 x 10^4
// with real couplings 17.2 -> 11.2 us (small blocks: the FP64 sums spread over the
// SMs).
constexpr int kObsThreads = 256;
constexpr int kObsWarps = kObsThreads / 32;
__device__ __forceinline__ void observe_partial_body(const ObsArgs& a)
{
    __shared__ long long s_ll[4][kObsWarps];
    __shared__ double s_d[2][kObsWarps];
    __shared__ __int128 s_min[kObsWarps];
    __shared__ int s_first[kObsWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R = a.Rdev ? *a.Rdev : a.R;
    const int nb = obs_blocks(R);
    if ((int)blockIdx.x >= nb) return;  // block-uniform
    const int per = (R + nb - 1) / nb;
    const int j0 = blockIdx.x * per, j1 = min(R, j0 + per);
    long long se = 0, se2 = 0, chi = 0, clo = 0;
    double sed = 0.0, se2d = 0.0;
    int mn32 = 0x7fffffff;
    __int128 mn = (__int128)(((unsigned __int128)1 << 127) - 1);
    for (int jb = j0; jb < j1; jb += kObsThreads) {
        const int j = jb + tid, jend = min(j1, jb + kObsThreads);
        int f = 0, fprev = 0;
        if (j < j1) {
            f = a.family[j];
            fprev = j > 0 ? a.family[j - 1] : f;
            if (a.kind == 0) {
                const int e = a.E32[j];
                se += e;
                se2 += (long long)e * e;
                mn32 = min(mn32, e);
            } else {
                const longlong2 v = a.E128[j];
                const __int128 e = ((__int128)v.y << 64) | (unsigned long long)v.x;
                const double ed = __dmul_rn(i128_to_double(e), 0x1p-96);
                sed = __dadd_rn(sed, ed);
                se2d = __fma_rn(ed, ed, se2d);
                if (e < mn) mn = e;
            }
        }
        const bool start = j < j1 && (j == 0 || fprev != f);
        const unsigned bal = __ballot_sync(0xffffffffu, start);
        if (lane == 0) s_first[warp] = bal ? jb + warp * 32 + __ffs(bal) - 1 : 0x7fffffff;
        __syncthreads();
        if (bal) {  // warp-uniform
            // first start in a later warp, or beyond the window for the last run
            int nxt = __reduce_min_sync(0xffffffffu, lane > warp && lane < kObsWarps ? s_first[lane] : 0x7fffffff);
            if (nxt == 0x7fffffff) {
                const int fl = __shfl_sync(0xffffffffu, f, 31 - __clz(bal));
                int lo = jend, hi = R;  // the first index in [lo, hi) of another family, else hi
                while (lo < hi) {
                    const int step = (hi - lo + 31) / 32, at = lo + lane * step;
                    const unsigned ne = __ballot_sync(0xffffffffu, at < hi && a.family[at] != fl);
                    // the end lies after the last equal probe, at or before the first other one
                    const int k = ne ? __ffs(ne) - 1 : __popc(__ballot_sync(0xffffffffu, at < hi));
                    const int nlo = k == 0 ? lo : lo + (k - 1) * step + 1;
                    hi = ne ? lo + k * step : hi;
                    lo = min(nlo, hi);
                }
                nxt = lo;
            }
            if (start) {
                const unsigned later = bal & ~((2u << lane) - 1u);
                const int e = later ? jb + warp * 32 + __ffs(later) - 1 : nxt;
                // c ln c of the run (a run of one adds 0; short runs read it from
                // the context's table)
                const int cn = e - j;
                if (cn > 1) {
                    const double c = (double)cn, v = cn < kLogC ? a.logc[cn] : __dmul_rn(c, log(c));
                    // v = m 2^(x - 52), 0 <= x < 31: high part in units of 2^-20, low 32 bits below
                    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
                    const int x = (int)(bits >> 52) - 1023;
                    const unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
                    chi += (long long)(m >> (32 - x));
                    clo += (long long)((m << x) & 0xFFFFFFFFull);
                }
            }
        }
        __syncthreads();  // s_first is rewritten by the next window
    }
    // fixed shuffle trees
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        chi += __shfl_down_sync(0xffffffffu, chi, off);
        clo += __shfl_down_sync(0xffffffffu, clo, off);
    }
    if (a.kind == 0) {
        mn = __reduce_min_sync(0xffffffffu, mn32);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            se += __shfl_down_sync(0xffffffffu, se, off);
            se2 += __shfl_down_sync(0xffffffffu, se2, off);
        }
    } else {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            sed = __dadd_rn(sed, __shfl_down_sync(0xffffffffu, sed, off));
            se2d = __dadd_rn(se2d, __shfl_down_sync(0xffffffffu, se2d, off));
            const long long lo = __shfl_down_sync(0xffffffffu, (long long)(unsigned long long)mn, off);
            const long long hi = __shfl_down_sync(0xffffffffu, (long long)(mn >> 64), off);
            const __int128 o = ((__int128)hi << 64) | (unsigned long long)lo;
            if (o < mn) mn = o;
        }
    }
    if (lane == 0) {
        s_ll[0][warp] = se; s_ll[1][warp] = se2; s_ll[2][warp] = chi; s_ll[3][warp] = clo;
        s_d[0][warp] = sed; s_d[1][warp] = se2d;
        s_min[warp] = mn;
    }
    __syncthreads();
    ObsPartial& p = a.part[blockIdx.x];
    if (tid < 4) {
        long long v = 0;
#pragma unroll
        for (int w = 0; w < kObsWarps; ++w) v += s_ll[tid][w];
        if (tid == 0) p.sumE = v;
        else if (tid == 1) p.sumE2 = v;
        else if (tid == 2) p.chi = v;
        else p.clo = v;
    } else if (tid >= 32 && tid < 34) {  // the warps' FP64 sums in warp order
        double v = s_d[tid - 32][0];
        if (a.kind != 0)
#pragma unroll
            for (int w = 1; w < kObsWarps; ++w) v = __dadd_rn(v, s_d[tid - 32][w]);
        if (tid == 32) p.sumEd = v;
        else p.sumE2d = v;
    } else if (tid == 64) {
        __int128 M = s_min[0];
#pragma unroll
        for (int w = 1; w < kObsWarps; ++w)
            if (s_min[w] < M) M = s_min[w];
        p.min_lo = (long long)(unsigned long long)M;
        p.min_hi = (long long)(M >> 64);
    }
}
// partials combined by one warp: lane l adds blocks l, l + 32, ... in order,
// then the 32 lane sums are added by a fixed shuffle tree (the same order on
// every GPU)
__device__ __forceinline__ void observe_final_body(const ObsArgs& a)
{
    const int lane = threadIdx.x & 31;
    long long A = 0, B = 0, H = 0, Lw = 0;
    double C = 0.0, Dd = 0.0;
    __int128 M = (__int128)(((unsigned __int128)1 << 127) - 1);
    const int nb = obs_blocks(a.Rdev ? *a.Rdev : a.R);
    for (int b = lane; b < nb; b += 32) {
        const ObsPartial* p = a.part + b;
        A += __ldcg(&p->sumE); B += __ldcg(&p->sumE2);
        H += __ldcg(&p->chi); Lw += __ldcg(&p->clo);
        if (a.kind != 0) {
            C = __dadd_rn(C, __ldcg(&p->sumEd));
            Dd = __dadd_rn(Dd, __ldcg(&p->sumE2d));
        }
        const __int128 m = ((__int128)__ldcg(&p->min_hi) << 64) | (unsigned long long)__ldcg(&p->min_lo);
        if (m < M) M = m;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        A += __shfl_down_sync(0xffffffffu, A, off);
        B += __shfl_down_sync(0xffffffffu, B, off);
        H += __shfl_down_sync(0xffffffffu, H, off);
        Lw += __shfl_down_sync(0xffffffffu, Lw, off);
        const long long lo = __shfl_down_sync(0xffffffffu, (long long)(unsigned long long)M, off);
        const long long hi = __shfl_down_sync(0xffffffffu, (long long)(M >> 64), off);
        const __int128 o = ((__int128)hi << 64) | (unsigned long long)lo;
        if (o < M) M = o;
    }
    if (a.kind != 0) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            C = __dadd_rn(C, __shfl_down_sync(0xffffffffu, C, off));
            Dd = __dadd_rn(Dd, __shfl_down_sync(0xffffffffu, Dd, off));
        }
    }
    if (lane != 0) return;
    a.cur->sumE = A; a.cur->sumE2 = B;
    a.cur->sumEd = C; a.cur->sumE2d = Dd;
    a.cur->sum_clnc = __dmul_rn(i128_to_double(((__int128)H << 32) + Lw), 0x1p-52);
    a.cur->emin_lo = (long long)(unsigned long long)M;
    a.cur->emin_hi = (long long)(M >> 64);
}
__device__ __forceinline__ void observe_launch(const ObsArgs& a)
{
    observe_partial_body(a);
    const int nb = obs_blocks(a.Rdev ? *a.Rdev : a.R);
    if ((int)blockIdx.x < nb && last_block(a.sync, nb) && threadIdx.x < 32) observe_final_body(a);
}
__global__ void __launch_bounds__(kObsThreads) observe_kernel(ObsArgs a) { observe_launch(a); }
__global__ void __launch_bounds__(kObsThreads) observe_batched(const ObsArgs* tab) { observe_launch(tab[blockIdx.y]); }

cudaError_t launch_observe(const ObsArgs& a, cudaStream_t st)
{
    observe_kernel<<<obs_blocks(a.R), kObsThreads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_observe_batched(const ObsArgs* tab, int n_inst, int maxR, cudaStream_t st)
{
    observe_batched<<<dim3(obs_blocks(maxR), (unsigned)n_inst), kObsThreads, 0, st>>>(tab);
    return cudaGetLastError();
}

// ---------------- backward pass of sum_k gbar_k beta_k F_k ----------------
// d(beta F)/dJ_b = -beta <S_i S_j>, d(beta F)/dh_i = -beta <S_i> (from Eq. 1),
// estimated with the exact population sums after the sweeps at beta_k.
__global__ void grad_backward_kernel(const unsigned long long* cJ, const unsigned long long* ch,
                                     const double* gbar, const double* betas, const double* Rk,
                                     int n_temps, int nJ, int N, double* dJ, double* dh)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nJ + N) return;
    const bool isJ = b < nJ;
    const int idx = isJ ? b : b - nJ;
    const int stride = isJ ? nJ : N;
    const unsigned long long* c = isJ ? cJ : ch;
    double acc = 0.0;
    for (int k = 0; k < n_temps; ++k) {
        const double m = __ddiv_rn((double)(long long)c[(size_t)k * stride + idx], Rk[k]);
        acc = __dadd_rn(acc, __dmul_rn(gbar[k], -__dmul_rn(betas[k], m)));
    }
    if (isJ) dJ[idx] = acc; else dh[idx] = acc;
}

cudaError_t launch_grad_backward(const unsigned long long* cJ, const unsigned long long* ch,
                                 const double* gbar, const double* betas, const double* Rk,
                                 int n_temps, int nJ, int N, double* dJ, double* dh, cudaStream_t st)
{
    const int n = nJ + N;
    grad_backward_kernel<<<(n + 255) / 256, 256, 0, st>>>(cJ, ch, gbar, betas, Rk, n_temps, nJ, N, dJ, dh);
    return cudaGetLastError();
}

}  // namespace pa
