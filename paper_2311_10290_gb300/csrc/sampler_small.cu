// LEWalk sampler for small graphs: the whole state of a sample, and the graph,
// in shared memory.
//
// One lane runs one sample's Wilson LE_v run as Alg. 2 and Alg. 4 state it
// (draw k at node u is the Philox draw (u, k, i, 0)).  A run on a graph of a thousand
// nodes is a chain of a few thousand dependent steps that more walkers do not
// shorten (its walks hit the root late and meet each other before), so what
// counts is the time of one step: about 300 cycles here, where the 1-byte
// kernel waits for three L2 or DRAM accesses per step.
//
// State per sample: one tree bit, one path bit and one byte of draws per node,
// laid out word by word across the warp's samples (word w of lane l at w * lanes +
// l).  The current loop-erased path is a stack of 16-bit node ids in the workspace,
// its two topmost entries in registers (most loops have two nodes).  From its 255th
// draw on a node is counted in a 32-bit word of the workspace.
//
// Lanes of a warp in different phases of a step wait for each other, so a warp has
// few samples: 10000 samples of an Erdos-Renyi graph of 1000 nodes take 5.1 / 4.3 /
// 4.3 / 4.3 ms with 22 / 8 / 4 / 2 per warp (the 1-byte kernel: 9.4 ms).
#include "walk_tasks.cuh"

namespace {

using namespace lap_walks;

constexpr uint32_t kMany = 255u;
enum : uint32_t { S_CLAIM = 0, S_SCAN, S_STEP, S_ADD };

// LOCAL: packed arcs and row records are in shared memory.
template <bool CV, bool LOCAL>
__global__ void __launch_bounds__(512) lewalk_small_kernel(LapSampleLaunch p, LapBlockLaunch b, uint32_t lanes)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const uint32_t n = (uint32_t)p.g.n, v = (uint32_t)p.root;
    const Graph<true> g{p.g.rowinfo, p.g.col, b.arcs, b.bw, b.bo, policy_evict_last()};
    unsigned long long *const arcs = reinterpret_cast<unsigned long long *>(smem);
    uint2 *const rows = reinterpret_cast<uint2 *>(arcs + p.g.arcs);
    uint32_t *const state0 = LOCAL ? reinterpret_cast<uint32_t *>(rows + n) : reinterpret_cast<uint32_t *>(smem);
    if (LOCAL) {
        for (int64_t x = threadIdx.x; x < p.g.arcs; x += blockDim.x) arcs[x] = b.arcs[x];
        for (uint32_t x = threadIdx.x; x < n; x += blockDim.x)
            rows[x] = make_uint2((uint32_t)p.g.rowinfo[x].x, (uint32_t)p.g.rowinfo[x].y);
        __syncthreads();
    }
    const uint32_t nw = (n + 31u) >> 5, nk = (n + 3u) >> 2;
    uint32_t *const tree = state0 + warp * (2u * nw + nk) * lanes + lane, *const path = tree + nw * lanes;
    uint8_t *const draws = reinterpret_cast<uint8_t *>(path + nw * lanes);
    const uint64_t slot = (blockIdx.x * (uint64_t)warps + warp) * lanes + lane;
    uint16_t *const stk = reinterpret_cast<uint16_t *>(b.stacks) + slot * b.stack_entries;
    uint32_t *const many = b.sweep + slot * n;
    const uint32_t key0 = (uint32_t)p.seed, key1 = (uint32_t)(p.seed >> 32);
    auto draws_at = [&](uint32_t u) -> uint8_t & { return draws[(u >> 2) * (4u * lanes) + (u & 3u)]; };
    auto row = [&](uint32_t u, uint32_t &off, uint32_t &deg) {
        if (LOCAL) {
            const uint2 r = rows[u];
            off = r.x;
            deg = r.y;
        } else {
            g.row(u, off, deg);
        }
    };

    uint32_t phase = lane < lanes && slot < p.slots ? (uint32_t)S_CLAIM : 0xFFu;
    uint32_t i = 0, q = 0, s = 0, u = 0, off = 0, deg = 1, sp = 0, top = 0, below = 0;
    uint32_t add = 0;                            // S_ADD: path entries still to be added to the tree
    unsigned long long y1 = 0, acc1 = 0;
    unsigned int bad = 0;

    while (phase != 0xFFu) {
        if (phase == S_STEP) {
            // u has just been reached.
            const uint32_t m = 1u << (u & 31u), x = (u >> 5) * lanes;
            if (tree[x] & m) {
                add = sp;
                phase = S_ADD;
            } else {
                const uint32_t on = path[x];
                if (on & m) {
                    // A loop closed at u: its nodes leave the path.
                    if (below == u && sp > 1u) {
                        path[(top >> 5) * lanes] &= ~(1u << (top & 31u));
                        path[x] &= ~m;
                        sp -= 2u;
                    } else {
                        for (;;) {
                            const uint32_t w = stk[--sp];
                            path[(w >> 5) * lanes] &= ~(1u << (w & 31u));
                            if (w == u) break;
                        }
                    }
                    top = sp > 0u ? stk[sp - 1u] : 0u;
                }
                // The draw index; a node's byte stays at kMany once it has been drawn
                // that often, and the workspace counts on.
                uint32_t k = draws_at(u);
                if (k < kMany) {
                    draws_at(u) = (uint8_t)(k + 1u);
                    if (k + 1u == kMany) many[u] = kMany;
                } else {
                    k = many[u];
                    many[u] = k + 1u;
                }
                const uint32_t e = off + below32(lap::philox_r64(u, k, i, 0u, key0, key1), deg);
                const uint64_t a = LOCAL ? arcs[e] : g.arc(e);
                const uint32_t w = g.target(a);
                path[x] |= m;
                stk[sp++] = (uint16_t)u;
                below = top;
                top = u;
                if (k) atomicAdd(&p.rep1[u], 1ull);
                if (CV && p.cv_h1) atomicAdd(&p.cv_a1[u], (unsigned long long)ld_pot(p.cv_h1 + w));
                if (++y1 > p.step_limit) {
                    bad = LAP_DEV_STEP_LIMIT;
                    phase = 0xFFu;
                }
                u = w;
                const uint32_t d = (uint32_t)(a >> (b.bw + b.bo));
                off = (uint32_t)(a >> b.bw) & (uint32_t)((1ull << b.bo) - 1ull);
                deg = d;
                if (d == (uint32_t)((1ull << (64u - b.bw - b.bo)) - 1ull)) row(w, off, deg);
            }
        }
        if (phase == S_ADD) {
            // The path joins the tree: a few nodes at a time, or all its bits.
            if (add > 24u) {
                for (uint32_t x = 0; x < nw * lanes; x += lanes) {
                    tree[x] |= path[x];
                    path[x] = 0u;
                }
                add = 0;
            } else {
                uint32_t w = top;
                for (int t = 0; t < 4 && add > 0u; ++t) {
                    if (add != sp) w = stk[add - 1u];
                    --add;
                    tree[(w >> 5) * lanes] |= 1u << (w & 31u);
                    path[(w >> 5) * lanes] &= ~(1u << (w & 31u));
                }
            }
            if (add == 0u) phase = S_SCAN;
        }
        if (phase == S_SCAN) {
            // The next start: the first node not in the tree.
            sp = 0;
            uint32_t t = ~tree[s * lanes];
            if (t == 0u && ++s < nw) t = ~tree[s * lanes];
            if (t) {
                u = s * 32u + (uint32_t)__ffs(t) - 1u;
                row(u, off, deg);
                phase = S_STEP;
            } else if (s >= nw) {
                acc1 += y1;
                if (p.y1_out) p.y1_out[q] = y1;
                phase = S_CLAIM;
            }
        }
        if (phase == S_CLAIM) {
            q = atomicAdd(&p.acc->claim, 1u);
            if (q >= p.count) break;
            i = p.first + q;
            for (uint32_t x = 0; x < (2u * nw + nk) * lanes; x += lanes) tree[x] = 0u;
            if (n & 31u) tree[(nw - 1u) * lanes] = ~((1u << (n & 31u)) - 1u);
            tree[(v >> 5) * lanes] |= 1u << (v & 31u);
            s = 0;
            sp = 0;
            top = 0;
            y1 = 0;
            phase = S_SCAN;
        }
    }
    if (acc1) atomicAdd(&p.acc->sum_y1, acc1);
    if (bad) atomicOr(&p.acc->status, bad);
}

constexpr uint64_t kSmem = 227ull << 10;
constexpr uint64_t kLanes = 4;         // samples per warp, where 16 warps hold the call's

}  // namespace

bool lap_small_plan(int32_t n, int64_t arcs, uint64_t count, uint64_t slots_opt, uint64_t ws_bytes, int num_sms, bool paths,
                    LapSmallPlan *out)
{
    LapSmallPlan pl;
    const uint64_t nn = (uint64_t)n, per_lane = 4ull * (2ull * ((nn + 31ull) / 32ull) + (nn + 3ull) / 4ull);
    const uint64_t graph = 8ull * (uint64_t)arcs + 8ull * nn;
    if (num_sms < 1) num_sms = 1;
    if (per_lane > kSmem || nn > 65535ull) return false;
    uint64_t want = count;
    if (slots_opt && slots_opt < want) want = slots_opt;
    if (want == 0) want = 1;
    // What the workspace holds: a sample's stack and words of nodes drawn often, with
    // loop-included paths 3/8 of a walk's words (a sample's two walks take at most that share
    // of its run's time) and one walk's at least.
    const uint64_t entries = (nn + 7ull) & ~7ull, slot_bytes = 2ull * entries + 4ull * nn;
    const uint64_t path_bytes = paths ? 8ull * nn : 0ull, least = 512ull + path_bytes;
    const uint64_t hold = ws_bytes > least ? (ws_bytes - least) / (slot_bytes + 3ull * path_bytes / 8ull) : 0ull;
    if (hold == 0) return false;
    if (want > hold) want = hold;
    uint64_t per_sm = (want + num_sms - 1) / num_sms;
    if (per_sm > 16ull * 32ull) per_sm = 16ull * 32ull;
    // The graph's copy stays if it leaves room for the samples the call can use,
    // or for 96.
    pl.local = graph < kSmem && (kSmem - graph) / per_lane >= (per_sm < 96ull ? per_sm : 96ull);
    const uint64_t fit = (kSmem - (pl.local ? graph : 0ull)) / per_lane;
    if (per_sm > fit) per_sm = fit;
    // Few samples per warp: lanes in different phases of a step wait for each other.
    uint64_t warps = (per_sm + kLanes - 1ull) / kLanes;
    if (warps > 16) warps = 16;
    const uint64_t lanes = (per_sm + warps - 1) / warps;
    if (warps * lanes > fit) warps = fit / lanes;
    const uint64_t blocks = (want + warps * lanes - 1) / (warps * lanes);
    pl.warps = (int)warps;
    pl.walk_ctas = 4ull * num_sms;
    pl.lanes = (uint32_t)lanes;
    pl.blocks = blocks < (uint64_t)num_sms ? blocks : (uint64_t)num_sms;
    pl.smem = (pl.local ? graph : 0ull) + warps * lanes * per_lane;
    // Workspace: path words of the loop-included paths, the stacks, the words of
    // nodes drawn often.
    pl.slots = pl.blocks * warps * lanes;
    if (pl.slots > hold) pl.slots = hold;
    if (slots_opt && slots_opt < pl.slots) pl.slots = slots_opt;
    const uint64_t stacks = slot_bytes * pl.slots + 512ull;
    pl.b.path_lanes = 0;
    if (paths) {
        pl.b.path_lanes = (ws_bytes - stacks) / path_bytes;
        if (pl.b.path_lanes > pl.walk_ctas * 32ull) pl.b.path_lanes = pl.walk_ctas * 32ull;
    }
    pl.words_bytes = pl.b.path_lanes * path_bytes;
    pl.stack_offset = (pl.words_bytes + 255ull) & ~255ull;
    pl.many_offset = pl.stack_offset + 2ull * entries * pl.slots;
    pl.bytes = pl.words_bytes + stacks;
    pl.b.stack_entries = entries;
    *out = pl;
    return true;
}

cudaError_t lap_launch_sample_small(const LapSampleLaunch &p, const LapSmallPlan &pl, cudaStream_t st)
{
    if (p.count == 0 || pl.blocks == 0) return cudaSuccess;
    const bool cv = p.cv_h1 || p.cv_h2;
    const void *kernel = cv ? (pl.local ? (const void *)lewalk_small_kernel<true, true> : (const void *)lewalk_small_kernel<true, false>)
                            : (pl.local ? (const void *)lewalk_small_kernel<false, true> : (const void *)lewalk_small_kernel<false, false>);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    uint32_t lanes = pl.lanes;
    void *args[3] = {const_cast<LapSampleLaunch *>(&p), const_cast<LapBlockLaunch *>(&pl.b), &lanes};
    e = cudaLaunchKernel(kernel, dim3((unsigned)pl.blocks), dim3((unsigned)(32 * pl.warps)), args, (size_t)pl.smem, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}
