// FP64 solves with L_v (the Laplacian without row and column v, Section 3.1)
// on the GPU: conjugate gradients (Hestenes and Stiefel, 1952) with the
// Jacobi preconditioner D^{-1}.  L_v is symmetric positive definite for a
// connected graph.  The quantities the samplers estimate that are linear in
// L_v^{-1} applied to a known vector come out exactly (to the tolerance):
// L_v^{-1} 1 gives y2 (Alg. 2) and the row-sum terms of (L^+)_uu (Section
// 3.1, element-wise Theorem 1); L_v^{-1} d gives the hitting times h(., v)
// and E[Y2] (Section 3.2, Alg. 4).
//
// An iteration is three launches: the product with L_v and p.q; the update of
// x, r, z with r.r and r.z; the new direction.  The last block of a launch adds
// the launch's partial sums and keeps the scalars, so the host reads one state
// record per kBatch iterations; iterations queued beyond the last one return
// at once.  At 300,000 nodes and 3 million arcs an iteration was 8 launches
// and a host read, with one thread on each hub's row: 290 us.
//
// All reductions have a fixed order (per-thread strides, a fixed tree per
// block, one thread order over the blocks), so the iterates are the same run to
// run.
#include "lap_internal.h"
#include "rows.cuh"

namespace {

using lap_rows::kBlock;
constexpr int kBatch = 8;

// Scalars of the iteration, on the device.
struct State {
    double rz, pq, rr, bb, rz_new;
    int32_t it, done;                 // iterations taken; converged, or nothing to solve
    unsigned int turn[3];             // blocks finished, per kernel
    unsigned int pad;
};

#define NODE_LOOP(u, n) for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < (n); u += (int64_t)gridDim.x * blockDim.x)

// Whether this block is the launch's last to get here; its threads then see
// the others' partial sums.
__device__ bool last_block(unsigned int *turn)
{
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int t = atomicAdd(turn, 1u);
        last = t + 1u == gridDim.x;
        if (last) *turn = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}
// Sum of part[0 .. count) in thread 0 (fixed order).
__device__ double total(const double *part, int count)
{
    double t = 0.0;
    for (int k = threadIdx.x; k < count; k += kBlock) t = __dadd_rn(t, part[k]);
    return lap_rows::block_total(t, 0.0);
}

// q = L_v p (p[v] read as 0, q[v] = 0): q_u = d_u p_u - sum_{w in N(u), w != v} p_w;
// `acc` collects p_u q_u of this thread's nodes.
struct Product {
    using T = double;
    const double *p;
    double *q;
    int32_t v;
    double acc;
    __device__ bool begin(int32_t) const { return true; }
    __device__ T zero() const { return 0.0; }
    __device__ T edge(int32_t w) const { return w == v ? 0.0 : p[w]; }
    __device__ void end(int32_t u, int2 r, T t)
    {
        const double pu = p[u], qu = u == v ? 0.0 : __dsub_rn(__dmul_rn((double)r.y, pu), t);
        q[u] = qu;
        acc = __dadd_rn(acc, __dmul_rn(pu, qu));
    }
};

__global__ void __launch_bounds__(kBlock) product_kernel(const int2 *__restrict__ rowinfo, const int32_t *__restrict__ col, int32_t n,
                                                        LapHubs hubs, int32_t v, const double *__restrict__ p,
                                                        double *__restrict__ q, double *part, State *s)
{
    if (s->done) return;
    Product f{p, q, v, 0.0};
    if ((int32_t)blockIdx.x < hubs.count) {
        lap_rows::hub_row(f, rowinfo, col, hubs.ids[blockIdx.x]);
    } else {
        const int64_t warps = (int64_t)(gridDim.x - hubs.count) * (kBlock / 32);
        const int64_t w = (int64_t)(blockIdx.x - hubs.count) * (kBlock / 32) + (threadIdx.x >> 5);
        lap_rows::node_rows(f, rowinfo, col, w * 32, warps * 32, n);
    }
    const double t = lap_rows::block_total(f.acc, 0.0);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
    if (last_block(&s->turn[0])) {
        const double pq = total(part, (int)gridDim.x);
        if (threadIdx.x == 0) s->pq = pq;
    }
}

// r = b (b[v] = 0), z = r / d, p = z, x = 0; r.z and b.b.
__global__ void __launch_bounds__(kBlock) init_kernel(const int2 *__restrict__ rowinfo, int32_t n, int32_t v, const double *__restrict__ b,
                                                     double *x, double *r, double *z, double *p, double *part, State *s)
{
    double rz = 0.0, bb = 0.0;
    NODE_LOOP(u, n)
    {
        const double bu = (u == v) ? 0.0 : b[u];
        x[u] = 0.0;
        r[u] = bu;
        const double zu = __ddiv_rn(bu, (double)rowinfo[u].y);
        z[u] = zu;
        p[u] = zu;
        rz = __dadd_rn(rz, __dmul_rn(bu, zu));
        bb = __dadd_rn(bb, __dmul_rn(bu, bu));
    }
    rz = lap_rows::block_total(rz, 0.0);
    bb = lap_rows::block_total(bb, 0.0);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = rz;
        part[gridDim.x + blockIdx.x] = bb;
    }
    if (last_block(&s->turn[1])) {
        const double a = total(part, (int)gridDim.x), c = total(part + gridDim.x, (int)gridDim.x);
        if (threadIdx.x == 0) {
            s->rz = a;
            s->bb = c;
            s->rr = c;
            s->done = c == 0.0;
        }
    }
}

// x += alpha p, r -= alpha q, z = r / d (alpha = rz / pq); r.r and r.z.
__global__ void __launch_bounds__(kBlock) update_kernel(const int2 *__restrict__ rowinfo, int32_t n, const double *__restrict__ p,
                                                       const double *__restrict__ q, double *x, double *r, double *z,
                                                       double rtol, double *part, State *s)
{
    if (s->done) return;
    const double alpha = __ddiv_rn(s->rz, s->pq);
    double rr = 0.0, rz = 0.0;
    NODE_LOOP(u, n)
    {
        x[u] = __fma_rn(alpha, p[u], x[u]);
        const double ru = __fma_rn(-alpha, q[u], r[u]);
        r[u] = ru;
        const double zu = __ddiv_rn(ru, (double)rowinfo[u].y);
        z[u] = zu;
        rr = __dadd_rn(rr, __dmul_rn(ru, ru));
        rz = __dadd_rn(rz, __dmul_rn(ru, zu));
    }
    rr = lap_rows::block_total(rr, 0.0);
    rz = lap_rows::block_total(rz, 0.0);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = rr;
        part[gridDim.x + blockIdx.x] = rz;
    }
    if (last_block(&s->turn[1])) {
        const double a = total(part, (int)gridDim.x), c = total(part + gridDim.x, (int)gridDim.x);
        if (threadIdx.x == 0) {
            s->rr = a;
            s->rz_new = c;
            ++s->it;
            // Read by the direction kernel and by the next iteration's launches.
            if (__dsqrt_rn(a) / __dsqrt_rn(s->bb) <= rtol) s->done = 1;
        }
    }
}

// p = z + beta p (beta = rz_new / rz).
__global__ void __launch_bounds__(kBlock) direction_kernel(int32_t n, const double *__restrict__ z, double *p, State *s)
{
    if (s->done) return;
    const double beta = __ddiv_rn(s->rz_new, s->rz);
    NODE_LOOP(u, n) p[u] = __fma_rn(beta, p[u], z[u]);
    if (last_block(&s->turn[2]) && threadIdx.x == 0) s->rz = s->rz_new;
}

int partial_count(int32_t n, LapHubs hubs)
{
    const int rows = lap_rows::node_blocks(n);
    return rows + hubs.count > 2 * rows ? rows + hubs.count : 2 * rows;
}

}  // namespace

uint64_t lap_lv_solve_scratch(int32_t n, LapHubs hubs)
{
    return 4ull * (uint64_t)n + (uint64_t)partial_count(n, hubs) + sizeof(State) / sizeof(double);
}

// Solves L_v x = b on the device; scratch: lap_lv_solve_scratch doubles.
cudaError_t lap_run_lv_solve(const int2 *rowinfo, const int32_t *col, int32_t n, LapHubs hubs, int32_t v,
                             const double *b, double *x, double *scratch, double rtol, int32_t maxiter,
                             int32_t *iterations, double *residual, cudaStream_t st)
{
    double *r = scratch, *z = r + n, *p = z + n, *q = p + n, *part = q + n;
    State *s = reinterpret_cast<State *>(part + partial_count(n, hubs));
    const int rows = lap_rows::node_blocks(n);
    *iterations = 0;
    *residual = 0.0;
    cudaError_t e = cudaMemsetAsync(s, 0, sizeof(State), st);
    if (e != cudaSuccess) return e;
    init_kernel<<<rows, kBlock, 0, st>>>(rowinfo, n, v, b, x, r, z, p, part, s);
    State h;
    for (int32_t queued = 0;;) {
        for (int t = 0; t < kBatch && queued < maxiter; ++t, ++queued) {
            product_kernel<<<rows + hubs.count, kBlock, 0, st>>>(rowinfo, col, n, hubs, v, p, q, part, s);
            update_kernel<<<rows, kBlock, 0, st>>>(rowinfo, n, p, q, x, r, z, rtol, part, s);
            direction_kernel<<<rows, kBlock, 0, st>>>(n, z, p, s);
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(&h, s, sizeof(h), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
        if (h.done || queued >= maxiter) break;
    }
    *iterations = h.it;
    // (Not a number where b holds one: no tolerance is met by it.)
    if (h.bb != 0.0) *residual = sqrt(h.rr) / sqrt(h.bb);
    return cudaSuccess;
}
