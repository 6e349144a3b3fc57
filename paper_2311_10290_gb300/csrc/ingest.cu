// Graph ingest on the GPU (hot-path row a1; cold, once per graph):
// CSR validation against the graph model of Section 2 (undirected, simple),
// per-node row records, the landmark choice of Section 6 (highest degree,
// smallest id on ties) and a breadth-first search from the landmark that
// checks connectivity (Section 2 assumes G connected; Wilson's algorithm does
// not terminate otherwise) and records hop distances.
#include "lap_internal.h"
#include "rows.cuh"

namespace {

constexpr int kBlock = 256;

int grid_for(int64_t work, int block)
{
    int64_t g = (work + block - 1) / block;
    if (g < 1) g = 1;
    if (g > 152 * 32) g = 152 * 32;
    return (int)g;
}

__device__ __forceinline__ bool row_contains(const int32_t *col, int32_t a, int32_t b, int32_t x)
{
    // Rows are checked to be strictly ascending, so binary search applies.
    while (a < b) {
        int32_t mid = a + ((b - a) >> 1);
        int32_t y = col[mid];
        if (y == x) return true;
        if (y < x) a = mid + 1; else b = mid;
    }
    return false;
}

__global__ void validate_kernel(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                int32_t n, int64_t arcs, unsigned int *status)
{
    unsigned int bad = 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        int32_t a = row_ptr[u], b = row_ptr[u + 1];
        if (a < 0 || b < a || (int64_t)b > arcs) { bad |= LAP_DEV_BAD_CSR; continue; }
        for (int32_t e = a; e < b; ++e) {
            int32_t w = col[e];
            if (w < 0 || w >= n) { bad |= LAP_DEV_BAD_CSR; continue; }
            if (w == (int32_t)u) bad |= LAP_DEV_SELF_LOOP;
            if (e > a && col[e - 1] >= w) bad |= LAP_DEV_BAD_CSR;
        }
    }
    if (bad) atomicOr(status, bad);
}

// Symmetry needs sorted rows, so it runs after validate_kernel succeeded.
__global__ void symmetry_kernel(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                int32_t n, unsigned int *status)
{
    unsigned int bad = 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        int32_t a = row_ptr[u], b = row_ptr[u + 1];
        for (int32_t e = a; e < b; ++e) {
            int32_t w = col[e];
            if (!row_contains(col, row_ptr[w], row_ptr[w + 1], (int32_t)u)) { bad |= LAP_DEV_NOT_SYMMETRIC; break; }
        }
    }
    if (bad) atomicOr(status, bad);
}

__global__ void rowinfo_kernel(const int32_t *__restrict__ row_ptr, int32_t n, int2 *__restrict__ rowinfo)
{
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        int32_t a = row_ptr[u];
        rowinfo[u] = make_int2(a, row_ptr[u + 1] - a);
    }
}

// Packs (degree, ~id) so that the maximum is the highest degree with the
// smallest id among ties.
__global__ void argmax_degree_kernel(const int2 *__restrict__ rowinfo, int32_t n, unsigned long long *best)
{
    unsigned long long m = 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long key = ((unsigned long long)(uint32_t)rowinfo[u].y << 32) | (0xFFFFFFFFu - (uint32_t)u);
        m = key > m ? key : m;
    }
    for (int off = 16; off > 0; off >>= 1) {
        unsigned long long o = __shfl_down_sync(0xFFFFFFFFu, m, off);
        m = o > m ? o : m;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(best, m);
}

__global__ void find_hubs_kernel(const int2 *__restrict__ rowinfo, int32_t n, int32_t *__restrict__ ids, unsigned int *count)
{
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x)
        if (rowinfo[u].y > LAP_HUB_DEGREE) ids[atomicAdd(count, 1u)] = (int32_t)u;
}

__global__ void bfs_start_kernel(int32_t *hops, int32_t n, int32_t root, unsigned int *flags)
{
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x)
        hops[u] = (u == root) ? 0 : -1;
    if (blockIdx.x == 0 && threadIdx.x == 0) flags[0] = 1u;
}

// One level: flag[0] says whether any node has it, flag[1] is set when a node
// is found.  A neighbour that has its hops already (most) is only read.
struct BfsLevel {
    using T = unsigned int;
    int32_t *hops;
    unsigned int *flag;
    int32_t level;
    __device__ bool skip() const { return *flag == 0u; }
    __device__ bool begin(int32_t u) const { return hops[u] == level; }
    __device__ T zero() const { return 0u; }
    __device__ T edge(int32_t w) const { return hops[w] == -1 && atomicCAS(&hops[w], -1, level + 1) == -1 ? 1u : 0u; }
    __device__ void end(int32_t, int2, T found) const
    {
        if (found) flag[1] = 1u;
    }
};

__global__ void count_reached_kernel(const int32_t *__restrict__ hops, int32_t n, unsigned int *count)
{
    unsigned int got = 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x)
        got += hops[u] >= 0;
    got = __reduce_add_sync(0xFFFFFFFFu, got);
    if ((threadIdx.x & 31) == 0 && got) atomicAdd(count, got);
}

// Batches of graphs: one thread per row, all graphs' levels queued together.
__global__ void bfs_init_kernel(int32_t *hops, int32_t n, int32_t root)
{
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x)
        hops[u] = (u == root) ? 0 : -1;
}

__global__ void bfs_level_kernel(const int2 *__restrict__ rowinfo, const int32_t *__restrict__ col,
                                 int32_t *hops, int32_t n, int32_t level, unsigned int *found)
{
    unsigned int got = 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        if (hops[u] != level) continue;
        int2 r = rowinfo[u];
        for (int32_t e = 0; e < r.y; ++e) {
            int32_t w = col[r.x + e];
            if (atomicCAS(&hops[w], -1, level + 1) == -1) ++got;
        }
    }
    if (got) atomicAdd(found, got);
}

}  // namespace

cudaError_t lap_launch_validate(const int32_t *row_ptr, const int32_t *col, int32_t n, int64_t arcs,
                                unsigned int *status, cudaStream_t st)
{
    validate_kernel<<<grid_for(n, kBlock), kBlock, 0, st>>>(row_ptr, col, n, arcs, status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    unsigned int h = 0;
    if ((e = cudaMemcpyAsync(&h, status, sizeof(h), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    if (h & LAP_DEV_BAD_CSR) return cudaSuccess;     // symmetry search needs a well-formed CSR
    symmetry_kernel<<<grid_for(n, kBlock), kBlock, 0, st>>>(row_ptr, col, n, status);
    return cudaGetLastError();
}

cudaError_t lap_launch_rowinfo(const int32_t *row_ptr, int32_t n, int2 *rowinfo, cudaStream_t st)
{
    rowinfo_kernel<<<grid_for(n, kBlock), kBlock, 0, st>>>(row_ptr, n, rowinfo);
    return cudaGetLastError();
}

cudaError_t lap_launch_argmax_degree(const int2 *rowinfo, int32_t n, unsigned long long *best, cudaStream_t st)
{
    argmax_degree_kernel<<<grid_for(n, kBlock), kBlock, 0, st>>>(rowinfo, n, best);
    return cudaGetLastError();
}

cudaError_t lap_launch_find_hubs(const int2 *rowinfo, int32_t n, int32_t *ids, unsigned int *count, cudaStream_t st)
{
    find_hubs_kernel<<<grid_for(n, kBlock), kBlock, 0, st>>>(rowinfo, n, ids, count);
    return cudaGetLastError();
}

cudaError_t lap_run_bfs(const int2 *rowinfo, const int32_t *col, int32_t n, LapHubs hubs, int32_t root, int32_t *hops,
                        unsigned int *flags, int64_t *reached, cudaStream_t st)
{
    // Levels are queued kLevels at a time and the host looks once per batch; a
    // level that no node has returns at once.
    constexpr int kLevels = 8;
    cudaError_t e = cudaMemsetAsync(flags, 0, sizeof(unsigned int) * (kLevels + 2), st);
    if (e != cudaSuccess) return e;
    bfs_start_kernel<<<grid_for(n, kBlock), kBlock, 0, st>>>(hops, n, root, flags);
    for (int32_t base = 0;; base += kLevels) {
        for (int32_t l = 0; l < kLevels; ++l) {
            e = lap_rows::launch_rows(BfsLevel{hops, flags + l, base + l}, rowinfo, col, n, hubs, st);
            if (e != cudaSuccess) return e;
        }
        count_reached_kernel<<<grid_for(n, kBlock), kBlock, 0, st>>>(hops, n, flags + kLevels + 1);
        unsigned int h[2] = {0, 0};
        if ((e = cudaMemcpyAsync(h, flags + kLevels, sizeof(h), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
        *reached = h[1];
        if (h[0] == 0) return cudaGetLastError();
        if ((e = cudaMemsetAsync(flags + 1, 0, sizeof(unsigned int) * (kLevels + 1), st)) != cudaSuccess) return e;   // flags[0] stays 1
    }
}

cudaError_t lap_launch_bfs_init(int32_t *hops, int32_t n, int32_t root, cudaStream_t st)
{
    bfs_init_kernel<<<grid_for(n, kBlock), kBlock, 0, st>>>(hops, n, root);
    return cudaGetLastError();
}

cudaError_t lap_launch_bfs_level(const int2 *rowinfo, const int32_t *col, int32_t *hops, int32_t n,
                                 int32_t level, unsigned int *found, cudaStream_t st)
{
    bfs_level_kernel<<<grid_for(n, kBlock), kBlock, 0, st>>>(rowinfo, col, hops, n, level, found);
    return cudaGetLastError();
}
