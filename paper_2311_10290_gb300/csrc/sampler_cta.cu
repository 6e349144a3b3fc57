// Choice between the small-graph kernel (sampler_small.cu) and the block kernel
// (sampler_block.cu), and the layout of their workspace.
#include "lap_internal.h"

namespace {

// Graphs up to this size take the small-graph kernel where a warp's samples fit
// in shared memory.
constexpr int32_t kSmallNodes = 4096;

}  // namespace

bool lap_cta_plan(int32_t n, int64_t arcs, uint64_t count, uint64_t slots_opt, uint64_t ws_bytes, int num_sms, bool paths,
                  bool cv, bool pack, LapCtaPlan *out)
{
    LapCtaPlan pl;
    pl.small = n <= kSmallNodes && pack && lap_small_plan(n, arcs, count, slots_opt, ws_bytes, num_sms, paths, &pl.lane);
    if (!pl.small && !lap_block_plan(n, count, slots_opt, ws_bytes, num_sms, paths, cv, pack, &pl.block)) return false;
    *out = pl;
    return true;
}

cudaError_t lap_launch_cta(LapSampleLaunch &p, LapCtaPlan &pl, void *ws_ptr, const unsigned long long *arcs, uint32_t tag_base,
                           cudaStream_t st)
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
        return lap_launch_sample_small(p, pl.lane, st);
    }
    b.words = reinterpret_cast<unsigned long long *>(ws);
    b.path_words = reinterpret_cast<unsigned long long *>(ws + pl.block.path_offset);
    b.stacks = reinterpret_cast<uint2 *>(ws + pl.block.stack_offset);
    b.sweep = reinterpret_cast<uint32_t *>(ws + pl.block.sweep_offset);
    b.early = reinterpret_cast<uint32_t *>(ws + pl.block.early_offset);
    b.early_stacks = b.early + (uint64_t)b.early_entries * b.early_count;
    b.early_pops = b.early_stacks + (uint64_t)b.early_cap * b.early_count;
    return lap_launch_sample_block(p, pl.block, st);
}
