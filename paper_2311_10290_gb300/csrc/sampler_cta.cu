// Choice between the small-graph kernel (sampler_small.cu) and the block kernel
// (sampler_block.cu), the layout of their workspace, and the absorbed walks that
// run beside them.
#include <cmath>

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

// A lane per sample costs the time of one run for every round of `lanes` samples,
// little more per sample until the lanes fill the memory system; a CTA per sample ends a
// run ten to thirty times sooner, but a few hundred run at a time.  So few samples go to
// the CTAs, and many samples of small graphs, of graphs with long first walks (f = 2m / d_v
// steps) or in a workspace that holds few CTAs' state to the lanes.  Fitted to 462
// measured pairs: n from 300 to 100,000, f from 17 to 37,000, 64 to 10^6 samples,
// workspaces from 1 MB to 17 GB; in 449 of them the choice by these estimates is within 1.1
// of the faster side, in the others within 1.5.  Both sides (lane / CTA kernel):
// Barabasi-Albert, 1000 nodes, 10^4 samples 4.2 / 2.4 ms, 10^5 samples 7.9 / 22 ms;
// 8000 nodes, 10^5 samples 60 / 59 ms; Erdos-Renyi, 10^4 nodes, 10^4 samples 107 / 54 ms,
// 4 10^4 samples 128 / 129 ms, 10^5 samples 185 / 289 ms.
double lap_lanes_estimate(int32_t n, int64_t arcs, int32_t root_degree, uint64_t count, uint64_t lanes, bool wide,
                          bool paths, bool cv)
{
    const double f = (double)arcs / (double)(root_degree > 0 ? root_degree : 1), c = (double)count;
    const double walk = 15.0 * (paths ? (cv ? 2.2 : 1.6) : cv ? 1.3 : 1.0);
    const double rounds = lanes < count ? c / (double)(lanes > 0 ? lanes : 1) : 1.0;
    const double each = wide ? 0.25e-3 * n + 0.25e-3 * f : 0.056e-3 * n + 0.1e-3 * f;
    return rounds * (3.2 * n + walk * f) + c * each;
}

// Eight lanes shorten the Wilson run, not the first walk; later rounds overlap the longest
// runs of earlier ones.  Erdos-Renyi, 18,000 nodes, 17,300 samples in 267 MB 1508 ms (estimate
// 1700), 57,000 nodes, 5500 samples in 552 MB 1359 (1380), 10^5 nodes, 512 samples 1258 (1060).
double lap_group_estimate(int32_t n, int64_t arcs, int32_t root_degree, uint64_t count, uint64_t groups)
{
    const double f = (double)arcs / (double)(root_degree > 0 ? root_degree : 1), c = (double)count;
    const double rounds = groups < count ? c / (double)(groups > 0 ? groups : 1) : 1.0;
    return (0.5 + 0.5 * rounds) * (1.1 * n + 25.0 * f) + c * (0.084e-3 * n + 0.15e-3 * f);
}

double lap_cta_estimate(int32_t n, int64_t arcs, int32_t root_degree, uint64_t count, const LapCtaPlan &pl)
{
    const double f = (double)arcs / (double)(root_degree > 0 ? root_degree : 1), c = (double)count;
    if (pl.small) {
        // 0.9 us per step of a sample, or the issue rate.
        const double steps = 1.4 * n + 3.0 * f, lat = 0.9 / (double)pl.lane.slots;
        return 1.5 * (n + 2.0 * f) + c * steps * (lat > 0.08e-3 ? lat : 0.08e-3);
    }
    // Every part of the call waits for the longest of its samples' first walks (an early
    // table each), whose lengths scatter like exponential ones; a first walk without a table
    // costs the CTAs more; fewer CTAs than the SMs hold leave each of them faster.
    const LapBlockPlan &b = pl.block;
    const bool in_parts = b.b.part < count;
    const double part = in_parts ? (double)b.b.part : c, parts = ceil(c / part);
    const double early = in_parts || b.b.early_count >= count ? 1.0 : (double)b.b.early_count / c;
    const double rounds = c > (double)b.slots ? c / (double)b.slots : 1.0, starved = 0.8 * (double)b.walk_ctas * rounds;
    return 0.75 * f * log(part + 1.0) * parts + c * early * f * 0.5e-3 * (1.0 + 0.5e-5 * n) +
           (c > starved ? c : starved) * (0.17 + 0.045e-3 * n + (1.0 - early) * 2.2e-3 * f);
}

double lap_cta_work(int32_t n, int64_t arcs, int32_t root_degree, uint64_t count, const LapCtaPlan &pl, int num_sms)
{
    const double f = (double)arcs / (double)(root_degree > 0 ? root_degree : 1), c = (double)count;
    if (pl.small) {
        // A CTA has an SM's shared memory to itself.
        const double steps = 1.4 * n + 3.0 * f, waves = ceil(c / (double)pl.lane.slots);
        const double share = (double)pl.lane.blocks / (double)num_sms, issue = c * steps * 0.08e-3;
        return share * waves * steps * 0.9 > issue ? share * waves * steps * 0.9 : issue;
    }
    return c * (0.17 + 0.045e-3 * n + f * 0.5e-3 * (1.0 + 0.5e-5 * n));
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
