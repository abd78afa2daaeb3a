// kern.cuh -- launch and reduction helpers shared by the cycle kernels of
// one right-hand side (cycle.cu) and of interleaved blocks of right-hand
// sides (block.cu).
#pragma once

#include <algorithm>
#include <utility>

#include "gw_internal.cuh"

namespace gw {

constexpr int BS = 256;  // threads per block of every cycle and CG kernel

// Blocks a grid-stride loop over `threads` work items asks for.
static inline int blocks_for(long long threads)
{
    const long long b = (threads + BS - 1) / BS;
    return (int)std::max(1LL, std::min<long long>(b, 1LL << 30));
}

#ifndef GW_GRID_BALANCE
#define GW_GRID_BALANCE 0
#endif

// The grid actually launched for `blocks`: at most one wave of the kernel
// (its resident blocks per SM times the SMs, from the occupancy calculator),
// and within that as few blocks as give every thread the same number of
// grid-stride iterations.
static inline int wave_grid(const void *fn, int blocks)
{
    const int cap = kernel_wave(fn, BS);
    if (blocks <= cap) return std::max(1, blocks);
    if (!GW_GRID_BALANCE) return cap;
    const int iters = (blocks + cap - 1) / cap;
    return (blocks + iters - 1) / iters;
}

#define ROWS(i, n) for (int i = blockIdx.x * BS + threadIdx.x; i < (n); i += gridDim.x * BS)

// The block index and block count a kernel body works with: the launch's own
// grid, or, in a batched launch that runs one pass for several solves, the
// virtual grid of one solve (each solve keeps its own row partition and
// reduction order, so its results do not depend on what else runs).
struct VB {
    int bid, nb;
};
__device__ __forceinline__ VB vb_grid() { return VB{(int)blockIdx.x, (int)gridDim.x}; }

// Programmatic dependent launch: every kernel of the cycle and of CG is
// launched so that the next kernel in the stream may be scheduled while this
// one runs; each kernel waits for its predecessors to complete (and their
// writes to be visible) before it touches global memory, then lets its own
// dependents launch.  Inside captured graphs this hides the launch gap
// between the 20-30 dependent kernels of a CG iteration.
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... KArgs, class... Args>
static void launch_pdl(void (*kernel)(KArgs...), int grid, cudaStream_t st, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)wave_grid((const void *)kernel, grid));
    cfg.blockDim = dim3(BS);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    GW_CUDA(cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...));
}


// ------------------------------------------------------------- reductions --
// A thread's share of an FP32 dot product without FP32 rounding of the sum:
// each product is split exactly into p + e (e by a fused multiply-add) and
// the products are added in two FP32 words by the error-free TwoSum, which
// keeps about 46 bits; the pair becomes an FP64 value at the reduction.  FP32
// operations only (FP64 throughput is scarce on this GPU); explicitly rounded
// intrinsics keep the compiler from contracting the transformations.
struct Sum2 {
    float hi = 0.f, lo = 0.f;
};
__device__ __forceinline__ void sum2_prod(Sum2 &s, float x, float y)
{
    const float p = __fmul_rn(x, y);
    const float e = __fmaf_rn(x, y, -p);
    const float t = __fadd_rn(s.hi, p);
    const float bp = __fsub_rn(t, s.hi);
    const float err = __fadd_rn(__fsub_rn(s.hi, __fsub_rn(t, bp)), __fsub_rn(p, bp));
    s.hi = t;
    s.lo = __fadd_rn(s.lo, __fadd_rn(err, e));
}
__device__ __forceinline__ double sum2_value(const Sum2 &s) { return (double)s.hi + (double)s.lo; }

// A thread's running share of a dot product over all its rows: for FP32
// operands the error-free pair above, carried from row block to row block;
// for FP64 operands a plain FP64 sum.
struct DAcc {
    Sum2 s;
    double d = 0.0;
};

// adds the dot product of R consecutive entries
template <int R, class T, class U>
__device__ __forceinline__ void dot_add(DAcc &acc, const T (&a)[R], const U (&b)[R])
{
    if constexpr (sizeof(T) == 4 && sizeof(U) == 4) {
#pragma unroll
        for (int k = 0; k < R; ++k) sum2_prod(acc.s, (float)a[k], (float)b[k]);
    } else {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < R; ++k) s += (double)a[k] * (double)b[k];
        acc.d += s;
    }
}
__device__ __forceinline__ double warp_sum(double v)
{
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// block sum in a fixed order (shuffle tree, then warp 0 adds the 8 warp sums)
__device__ __forceinline__ double block_sum(double v, double *sh)
{
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
    if (w == 0) {
        t = lane < BS / 32 ? sh[lane] : 0.0;
        t = warp_sum(t);
    }
    return t;  // valid in thread 0
}

// Writes this block's partial sums; returns true in the last block to arrive,
// which then holds the grand totals (summed over blocks in index order) in tot[].
template <int K>
__device__ __forceinline__ bool reduce_last(VB vb, const double (&loc)[K], double *part, unsigned *cnt,
                                            double (&tot)[K])
{
    constexpr int W = BS / 32;
    __shared__ double sh[K][W];
    __shared__ unsigned ticket;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // warps (shuffle tree), then one thread per value adds the warps in order
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const double v = warp_sum(loc[k]);
        if (lane == 0) sh[k][w] = v;
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < W; ++q) s += sh[threadIdx.x][q];
        part[(size_t)threadIdx.x * vb.nb + vb.bid] = s;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) ticket = atomicAdd(cnt, 1u);
    __syncthreads();
    if (ticket != (unsigned)vb.nb - 1) return false;
    __threadfence();
    // last block: every thread adds the partials b = t, t + BS, ... (their
    // loads issued together), then the warps' shuffle trees and the warps in
    // order, a fixed order for a given block count
    __shared__ double fin[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        double s = 0.0;
#pragma unroll 8
        for (int b = threadIdx.x; b < vb.nb; b += BS) s += __ldcg(part + (size_t)k * vb.nb + b);
        s = warp_sum(s);
        if (lane == 0) sh[k][w] = s;
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < W; ++q) s += sh[threadIdx.x][q];
        fin[threadIdx.x] = s;
    }
    if (threadIdx.x == 0) *cnt = 0u;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) tot[k] = fin[k];
    return true;
}

template <int K>
__device__ __forceinline__ bool reduce_last(const double (&loc)[K], double *part, unsigned *cnt, double (&tot)[K])
{
    return reduce_last<K>(vb_grid(), loc, part, cnt, tot);
}

// Reduction of FP32 pairs over warps, blocks and the grid in FP32 only.  FP64
// issue is about 2 operations a cycle an SM here: a shuffle tree in FP64 over
// a thread's converted sums held a warp for ~130 cycles a sum, 2-4 us at the
// end of every reducing pass of a full grid.  In FP32 the level-0
// post-smoothing pass with its two dots went from 21.8 to 19.8 us at 128^3 and
// from 6.9 to 5.6 us on 128 x 128 x 1, the CG product at 128^3 from 19.3 to 17.8,
// the update from 14.1 to 12.9; on eight columns the post-smoothing pass from
// 121 to 104 us (times not overlapped by the kernels before; one solve
// 1.02-1.14x by size).  The pair gains a
// third word that takes the rounding errors of the second, so every addition
// is error-free but for the last bits of the third word (TwoSum cascades as in
// Ogita, Rump & Oishi 2005): about 70 bits, more than the FP64 tree kept.
// Sums whose high word reaches 2^100 in some thread (or is not finite) take the
// same steps in FP64, so the range stays that of FP64 above a thread.
struct Sum3 {
    float h, m, l;
};
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ Sum3 red_add(const Sum3 &a, const Sum3 &b)
{
    Sum3 r;
    float e1, e2, e3, m;
    two_sum(a.h, b.h, r.h, e1);
    two_sum(a.m, b.m, m, e2);
    two_sum(m, e1, r.m, e3);
    r.l = __fadd_rn(__fadd_rn(a.l, b.l), __fadd_rn(e2, e3));
    return r;
}
__device__ __forceinline__ double red_add(double a, double b) { return a + b; }
__device__ __forceinline__ Sum3 red_shfl(const Sum3 &a, int o)
{
    return Sum3{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.m, o),
                __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ double red_shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }

// A partial sum in shared or global memory: three FP32 words, or (dbl set) an
// FP64 value in the first two.
struct alignas(16) Part {
    float h, m, l;
    unsigned dbl;
};
__device__ __forceinline__ Part to_part(const Sum3 &a) { return Part{a.h, a.m, a.l, 0u}; }
__device__ __forceinline__ Part to_part(double v)
{
    return Part{__int_as_float(__double2hiint(v)), __int_as_float(__double2loint(v)), 0.f, 1u};
}
__device__ __forceinline__ double part_value(const Part &p)
{
    if (p.dbl) return __hiloint2double(__float_as_int(p.h), __float_as_int(p.m));
    return ((double)p.h + (double)p.m) + (double)p.l;
}
__device__ __forceinline__ bool pair_big(const Sum2 &a) { return !(fabsf(a.hi) < 1.2676506e30f); }  // 2^100

// N sums a thread over a warp, lanes that agree below TPR added: each step
// halves the sums a lane keeps and hands the other half over, then the
// remaining steps add the one left.  The lane ends with sum red_index<N>(lane).
template <int N, int TPR, class T>
__device__ __forceinline__ void red_warp(T (&v)[N], int lane)
{
    int o = 16;
#pragma unroll
    for (int n = N; n > 1; n >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < n / 2; ++k) {
            const T keep = up ? v[k + n / 2] : v[k], give = up ? v[k] : v[k + n / 2];
            v[k] = red_add(keep, red_shfl(give, o));
        }
    }
#pragma unroll
    for (; o >= TPR; o >>= 1) v[0] = red_add(v[0], red_shfl(v[0], o));
}
template <int N>
__device__ __forceinline__ int red_index(int lane)
{
    int k = 0;
#pragma unroll
    for (int n = N, o = 16; n > 1; n >>= 1, o >>= 1) k += (lane & o) ? n / 2 : 0;
    return k;
}
// the warp's sums of pairs (every lane calls it); valid as red_warp says
template <int N, int TPR>
__device__ __forceinline__ Part red_pairs(const Sum2 (&a)[N], int lane)
{
    bool big = false;
#pragma unroll
    for (int k = 0; k < N; ++k) big |= pair_big(a[k]);
    if (!__any_sync(0xffffffffu, big)) {
        Sum3 v[N];
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] = Sum3{a[k].hi, a[k].lo, 0.f};
        red_warp<N, TPR>(v, lane);
        return to_part(v[0]);
    }
    double v[N];
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = sum2_value(a[k]);
    red_warp<N, TPR>(v, lane);
    return to_part(v[0]);
}
// sum of the eight partials held by aligned groups of eight lanes (every lane
// of the warp calls it); valid in all eight
__device__ __forceinline__ Part red_eight(const Part &p)
{
    if (!__any_sync(0xffffffffu, p.dbl)) {
        Sum3 v{p.h, p.m, p.l};
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v = red_add(v, red_shfl(v, o));
        return to_part(v);
    }
    double v = part_value(p);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return to_part(v);
}
// a thread's sum of the partials b = b0, b0 + step, ... < nb of one value,
// loaded together; then over the warp
__device__ __forceinline__ Part red_partials(const Part *part, int nb, int b0, int step)
{
    Sum3 v{0.f, 0.f, 0.f};
    unsigned dbl = 0u;
#pragma unroll 4
    for (int b = b0; b < nb; b += step) {
        const float4 t = __ldcg(reinterpret_cast<const float4 *>(part + b));
        dbl |= __float_as_uint(t.w);
        v = red_add(v, Sum3{t.x, t.y, t.z});
    }
    if (!__any_sync(0xffffffffu, dbl)) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = red_add(v, red_shfl(v, o));
        return to_part(v);
    }
    double s = 0.0;
    for (int b = b0; b < nb; b += step) {
        const float4 t = __ldcg(reinterpret_cast<const float4 *>(part + b));
        s += part_value(Part{t.x, t.y, t.z, __float_as_uint(t.w)});
    }
    return to_part(warp_sum(s));
}
// Counts a block in: the writes that its other threads made before the last
// barrier become visible with the count, and those of the blocks counted
// before are visible after it (and after the block's next barrier).
__device__ __forceinline__ unsigned arrive_gpu(unsigned *cnt)
{
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    const unsigned t = atomicAdd(cnt, 1u);
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    return t;
}

// As reduce_last, for K = 1 or 2 sums of FP32 pairs: true in thread 0 of the last
// block to arrive, which then holds the totals.  part: K records a block.
template <int K>
__device__ __forceinline__ bool reduce_pairs_last(VB vb, const Sum2 (&loc)[K], double *part_, unsigned *cnt,
                                                  double (&tot)[K])
{
    constexpr int W = BS / 32;
    static_assert(W == 8 && (K == 1 || K == 2), "eight warps a block, one or two sums");
    __shared__ Part sh[K * W];
    __shared__ unsigned ticket;
    Part *part = reinterpret_cast<Part *>(part_);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {
        const Part p = red_pairs<K, 1>(loc, lane);
        if ((lane & (K == 1 ? 31 : 15)) == 0) sh[red_index<K>(lane) * W + w] = p;
    }
    __syncthreads();
    const Part zero{0.f, 0.f, 0.f, 0u};
    if (w == 0) {
        const Part p = red_eight(lane < K * W ? sh[lane] : zero);
        if (lane < K * W && (lane & 7) == 0) part[(size_t)(lane >> 3) * vb.nb + vb.bid] = p;
        __syncwarp();
        if (lane == 0) ticket = arrive_gpu(cnt);
    }
    __syncthreads();
    if (ticket != (unsigned)vb.nb - 1) return false;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const Part p = red_partials(part + (size_t)k * vb.nb, vb.nb, threadIdx.x, BS);
        if (lane == 0) sh[k * W + w] = p;
    }
    if (threadIdx.x == 0) *cnt = 0u;
    __syncthreads();
    if (w == 0) {
        const double t = part_value(red_eight(lane < K * W ? sh[lane] : zero));
        tot[0] = t;
        if constexpr (K == 2) tot[1] = __shfl_sync(0xffffffffu, t, 8);
    }
    __syncthreads();  // sh may be written again by the block's next pass
    return threadIdx.x == 0;
}

// totals of a pass's dot products, in thread 0 of the last block (true there)
template <class T, int K>
__device__ __forceinline__ bool reduce_dots(VB vb, const DAcc (&acc)[K], double *part, unsigned *cnt, double (&tot)[K])
{
    if constexpr (sizeof(T) == 4) {
        Sum2 loc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) loc[k] = acc[k].s;
        return reduce_pairs_last<K>(vb, loc, part, cnt, tot);
    } else {
        double loc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) loc[k] = acc[k].d;
        return reduce_last<K>(vb, loc, part, cnt, tot) && threadIdx.x == 0;
    }
}

__device__ __forceinline__ bool finished(const Ctl *c) { return c && *(volatile const int *)&c->done; }

// Ends the solve with the given status.  Under a graph while node the loop
// itself is ended by the kernel that checks the true residual (k_rel_res, or
// k_cg_true in the FP64 form): it stops the loop when it finds the solve done
// on entry, or when it finds it converged, so that the heavy kernels make no
// device graph call (profilers skip kernels that make one).
__device__ __forceinline__ void ctl_stop(Ctl *c, int status)
{
    c->status = status;
    c->done = 1;
}

// ends the while loop of the solve's graph (one thread: the condition is
// never set concurrently)
__device__ __forceinline__ void ctl_end_loop(const Ctl *c)
{
    if (c->cond) cudaGraphSetConditional((cudaGraphConditionalHandle)c->cond, 0u);
}

}  // namespace gw
