// Choice between the small-graph kernel (sampler_small.cu) and the block kernel
// (sampler_block.cu), the layout of their workspace, and the absorbed walks that
// run beside them.
#include "walk_tasks.cuh"

namespace {

using namespace lap_walks;

// The absorbed walks, in CTAs of one warp: a walk is a chain of dependent loads,
// so these warps take little issue time from the Wilson runs on the same SM, and
// the longest walks of a call keep no Wilson CTA's shared memory.  They start
// with the early phase of the block kernel.  Against a last warp of each Wilson CTA:
// Barabasi-Albert, 10^6 nodes 217 -> 204 ms, 2 * 10^5 nodes with control variate and
// paths 31 -> 27 ms.
template <bool CV, bool PACK>
__global__ void __launch_bounds__(32) walks_kernel(LapSampleLaunch p, LapBlockLaunch b)
{
    const Graph<PACK> g{p.g.rowinfo, p.g.col, b.arcs, b.bw, b.bo, policy_evict_last()};
    walk_tasks<CV, PACK>(p, b, g);
}

// The small-graph kernel is the faster one where the first walk passes much of the
// graph before it meets the root (2m / d_v steps), so that more walkers would
// follow each other.  Small against block kernel, 1000 samples: Erdos-Renyi, average
// degree 20, 1000 nodes 2.7 / 4.6 ms, 4000 nodes 15 / 19 ms; Barabasi-Albert rooted
// at a leaf, 1000 nodes 11 / 42 ms; rooted at its hub 1.3 / 0.6 ms.
constexpr int32_t kSmallNodes = 4096;

}  // namespace

bool lap_cta_plan(int32_t n, int64_t arcs, int32_t root_degree, int32_t max_degree, uint64_t count, uint64_t slots_opt, uint64_t ws_bytes, int num_sms, bool paths,
                  bool cv, bool pack, LapCtaPlan *out)
{
    LapCtaPlan pl;
    const uint64_t first = (uint64_t)arcs / (uint64_t)(root_degree > 0 ? root_degree : 1);
    pl.small = pack && n <= kSmallNodes && 8ull * first >= (uint64_t)n &&
               lap_small_plan(n, arcs, count, slots_opt, ws_bytes, num_sms, paths, &pl.lane);
    if (!pl.small && !lap_block_plan(n, arcs, root_degree, max_degree, count, slots_opt, ws_bytes, num_sms, paths, cv, pack, &pl.block)) return false;
    *out = pl;
    return true;
}

void lap_cta_bind(LapSampleLaunch &p, LapCtaPlan &pl, void *ws_ptr, const unsigned long long *arcs, uint32_t tag_base)
{
    uint8_t *ws = reinterpret_cast<uint8_t *>(ws_ptr);
    LapBlockLaunch &b = pl.small ? pl.lane.b : pl.block.b;
    p.slots = pl.small ? pl.lane.slots : pl.block.slots;
    b.arcs = arcs;
    if (arcs) lap_pack_bits(p.g.n, p.g.arcs, &b.bw, &b.bo);
    b.tag_base = tag_base;
    if (pl.small) {
        b.path_words = reinterpret_cast<unsigned long long *>(ws);
        b.stacks = reinterpret_cast<uint2 *>(ws + pl.lane.stack_offset);
        b.sweep = reinterpret_cast<uint32_t *>(ws + pl.lane.many_offset);
        return;
    }
    b.words = reinterpret_cast<unsigned long long *>(ws);
    b.path_words = reinterpret_cast<unsigned long long *>(ws + pl.block.path_offset);
    b.stacks = reinterpret_cast<uint2 *>(ws + pl.block.stack_offset);
    b.sweep = reinterpret_cast<uint32_t *>(ws + pl.block.sweep_offset);
    b.early = reinterpret_cast<uint32_t *>(ws + pl.block.early_offset);
    b.early_stacks = b.early + (uint64_t)b.early_entries * b.early_count;
    b.early_pops = b.early_stacks + (uint64_t)b.early_cap * b.early_count;
}

cudaError_t lap_launch_cta_wilson(const LapSampleLaunch &p, const LapCtaPlan &pl, cudaStream_t st)
{
    return pl.small ? lap_launch_sample_small(p, pl.lane, st) : lap_launch_sample_block(p, pl.block, st);
}

cudaError_t lap_launch_cta_walks(const LapSampleLaunch &p, const LapCtaPlan &pl, cudaStream_t st)
{
    if (p.count == 0) return cudaSuccess;
    const LapBlockLaunch &b = pl.small ? pl.lane.b : pl.block.b;
    const bool cv = p.cv_h1 || p.cv_h2, pack = b.arcs != nullptr;
    uint64_t ctas = pl.small ? pl.lane.walk_ctas : pl.block.walk_ctas;
    const uint64_t need = (2ull * p.count + 31ull) / 32ull;
    if (ctas > need) ctas = need;
    if (cv) {
        if (pack) walks_kernel<true, true><<<(unsigned)ctas, 32, 0, st>>>(p, b);
        else walks_kernel<true, false><<<(unsigned)ctas, 32, 0, st>>>(p, b);
    } else {
        if (pack) walks_kernel<false, true><<<(unsigned)ctas, 32, 0, st>>>(p, b);
        else walks_kernel<false, false><<<(unsigned)ctas, 32, 0, st>>>(p, b);
    }
    return cudaGetLastError();
}
