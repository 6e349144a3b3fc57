// Sums over the neighbours of every node, balanced for power-law degrees.
//
// One thread per row leaves the kernel waiting for its longest row (a hub's
// tens of thousands of entries, one dependent pair of loads after the other).
// Here a thread takes a row of at most kRowThread entries, a warp one of at most
// LAP_HUB_DEGREE, and a CTA of its own each longer row (the graph's hubs, listed
// once when the graph is created).  Every sum has a fixed order (per-lane strides,
// then a fixed tree), so results do not change from run to run.
//
// Against one thread per row (GB300): solve of 300,000 nodes 8.5 -> 3.6 ms; root and
// breadth-first search 1.33 -> 0.42 ms (10^6 nodes, 10^7 arcs, largest degree 4183)
// and 11.4 -> 0.72 ms (R-MAT, 3.1 10^7 arcs, 64668); its features 69 -> 3.3 ms.
// The solve with hubs from 256 / 512 / 2048 neighbours: 3.6 / 4.1 / 6.9 ms.  Where a
// thread's rows end matters little: up to 16 / 48 / 128 entries 4.1 / 4.1 / 4.3 ms (hubs
// from 512).
#pragma once

#include "lap_internal.h"

namespace lap_rows {

constexpr int kBlock = 256;
constexpr int kRowThread = 48;

// A functor F has
//   using T           the accumulator (with +=),
//   bool skip()       whether the launch has nothing to do,
//   bool begin(u)     whether node u's row is wanted,
//   T zero(), T edge(w)   the value of neighbour w,
//   void end(u, r, t) the row record and the sum.
template <class T>
__device__ __forceinline__ T shfl_xor(T x, int o) { return __shfl_xor_sync(0xFFFFFFFFu, x, o); }
struct Pair {
    double a, b;
    __device__ __forceinline__ Pair &operator+=(const Pair &o)
    {
        a = __dadd_rn(a, o.a);
        b = __dadd_rn(b, o.b);
        return *this;
    }
};
template <>
__device__ __forceinline__ Pair shfl_xor(Pair x, int o)
{
    return {__shfl_xor_sync(0xFFFFFFFFu, x.a, o), __shfl_xor_sync(0xFFFFFFFFu, x.b, o)};
}
template <class T>
__device__ __forceinline__ T warp_sum(T x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += shfl_xor(x, o);
    return x;
}

// Entries first, first + step, ... of the row: four loads in flight, added in order.
template <class F>
__device__ __forceinline__ typename F::T strided(F &f, const int32_t *__restrict__ col, int2 r, int32_t first, int32_t step)
{
    typename F::T t = f.zero();
    int32_t e = first;
    for (; e + 3 * step < r.y; e += 4 * step) {
        int32_t w[4];
#pragma unroll
        for (int y = 0; y < 4; ++y) w[y] = col[(int64_t)r.x + e + y * step];
        typename F::T v[4];
#pragma unroll
        for (int y = 0; y < 4; ++y) v[y] = f.edge(w[y]);
#pragma unroll
        for (int y = 0; y < 4; ++y) t += v[y];
    }
    for (; e < r.y; e += step) t += f.edge(col[(int64_t)r.x + e]);
    return t;
}

// Rows of nodes [lo, hi) by the block's warps (base: first node of the warp,
// step: nodes between the warp's turns), hubs left out.
template <class F>
__device__ void node_rows(F &f, const int2 *__restrict__ rowinfo, const int32_t *__restrict__ col, int64_t base,
                          int64_t step, int64_t hi)
{
    const int lane = threadIdx.x & 31;
    for (; base < hi; base += step) {
        const int64_t u = base + lane;
        int2 r = make_int2(0, 0);
        bool on = u < hi && f.begin((int32_t)u);
        if (on) r = rowinfo[u];
        on = on && r.y <= LAP_HUB_DEGREE;
        typename F::T t = f.zero();
        if (on && r.y <= kRowThread) t = strided(f, col, r, 0, 1);
        for (unsigned big = __ballot_sync(0xFFFFFFFFu, on && r.y > kRowThread); big; big &= big - 1u) {
            const int o = __ffs(big) - 1;
            const int2 q = make_int2(__shfl_sync(0xFFFFFFFFu, r.x, o), __shfl_sync(0xFFFFFFFFu, r.y, o));
            const typename F::T s = warp_sum(strided(f, col, q, lane, 32));
            if (lane == o) t = s;
        }
        if (on) f.end((int32_t)u, r, t);
    }
}

// Block-wide sum (kBlock threads) in thread 0.
template <class T>
__device__ T block_total(T x, T zero)
{
    __shared__ T sh[kBlock / 32];
    x = warp_sum(x);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    T t = zero;
    if (threadIdx.x == 0)
        for (int w = 0; w < kBlock / 32; ++w) t += sh[w];
    __syncthreads();
    return t;
}

template <class F>
__device__ void hub_row(F &f, const int2 *__restrict__ rowinfo, const int32_t *__restrict__ col, int32_t u)
{
    if (!f.begin(u)) return;                        // the same in all threads
    const int2 r = rowinfo[u];
    const typename F::T t = block_total(strided(f, col, r, (int32_t)threadIdx.x, kBlock), f.zero());
    if (threadIdx.x == 0) f.end(u, r, t);
}

// One launch over all rows: the first `hubs.count` blocks take a hub each.
template <class F>
__global__ void __launch_bounds__(kBlock) rows_kernel(F f, const int2 *__restrict__ rowinfo, const int32_t *__restrict__ col, int32_t n,
                                                     LapHubs hubs)
{
    if (f.skip()) return;
    if ((int32_t)blockIdx.x < hubs.count) {
        hub_row(f, rowinfo, col, hubs.ids[blockIdx.x]);
        return;
    }
    const int64_t warps = (int64_t)(gridDim.x - hubs.count) * (kBlock / 32);
    const int64_t w = (int64_t)(blockIdx.x - hubs.count) * (kBlock / 32) + (threadIdx.x >> 5);
    node_rows(f, rowinfo, col, w * 32, warps * 32, n);
}

inline int node_blocks(int32_t n)
{
    const int64_t g = ((int64_t)n + kBlock - 1) / kBlock;
    return (int)(g > 152 * 8 ? 152 * 8 : g);
}

template <class F>
cudaError_t launch_rows(const F &f, const int2 *rowinfo, const int32_t *col, int32_t n, LapHubs hubs, cudaStream_t st)
{
    rows_kernel<F><<<(unsigned)(node_blocks(n) + hubs.count), kBlock, 0, st>>>(f, rowinfo, col, n, hubs);
    return cudaGetLastError();
}

}  // namespace lap_rows
