// Cycle-popping LEWalk sampler with the tree in shared memory: one CTA runs one
// sample's Wilson LE_v run.  Counts are those of the sequential run, bit for bit.
// (The absorbed walks of Alg. 2 and Alg. 4 run beside it, sampler_cta.cu.)
//
// Why it is exact.  In the stack representation of Section 3.4 (Fig. 1) node
// u's j-th draw is the Philox draw (u, j, i, 0); Wilson's run pops cycles of
// stack tops, and the set of popped cycles does not depend on the order in
// which they are found.  So visits(u) = 1 + (popped cycles through u), and a
// first visit needs no counting at all.  Walkers own nothing: a walker follows
// the current arrows a(u, k(u)) from a start node, remembers the nodes it
// passed with the k it saw, and
//   - at a node whose arrow leads into the tree, checks that k(u) is still the
//     k it saw (then the current arrow of u leads into the tree for good) and
//     sets u's tree bit, then does the same for the node below on its path;
//   - at a node whose arrow closes a cycle of its path, excludes other pops of
//     its nodes and checks that every k is the one it saw.  Then the arrows are
//     a cycle of current stack tops: it is popped (k + 1 and one repeat visit
//     for each node).  If a k has changed, another walker has popped one of the
//     nodes: the walk goes on from the closing node.
// Two-node cycles (nearly all of them) take the lock bits of their two nodes,
// lowest lock first; longer ones take the sample's exclusive flag, which keeps
// two-node pops out, and are checked and popped by all lanes of the warp.
// A stale path entry can only fail such a check, never count; nodes walked by
// two walkers cost time and no counts.  Locks are held across straight-line
// code only; a walker that finds one taken goes on and comes back (the
// exclusive flag's holder alone waits, bounded, for pops that have begun).
//
// Four phases, by the share f of the nodes in the tree:
//   early     lewalk_early_kernel, a lane per sample, all samples of the launch
//             side by side, until f is about 5.7 / sqrt(n): the first walks are
//             long chains that more walkers do not shorten, so the latency is
//             hidden by samples instead.
//   walkers   until f = 0.35.  A walk takes about 1/f steps and meets the
//             paths of the others, so about n f^2 walkers are useful: the active
//             lanes grow as `grow` n f^2 from a minimum.
//   sweeps    every node outside the tree has its arrow computed once, and passes
//             over the list of these nodes add those whose arrow leads into the
//             tree; where a pass gains little, the next one pops the two-node
//             cycles.  No paths, no locks on the way, full warps.
//   walkers   on the list's rest (n / 200 nodes, at least 64).
// The sweep's line: 0.2 / 0.28 / 0.35 / 0.4 of the nodes take 43.3 / 40.9 / 40.6 / 40.8 ms
// on the 100,000-node Barabasi-Albert graph (8192 samples), 29.3 / 30.3 / 30.9 / 31.3 ms on
// an R-MAT graph of 31 million arcs (1520 samples), whose columns are read from HBM.
//
// Memory.  Per sample in flight, in shared memory: one tree bit per node; lock
// bits (of the nodes' low id bits); a filter bit per 2^fshift nodes, set before
// the first pop of one of them.  k of popped nodes is an 8-byte word
// {tag 32 | k 32} in the workspace (the tag names the sample, so the words are
// not cleared between samples).  All walkers of a sample are on one SM, so CTA
// scope orders their accesses.  A step needs one column load, whose row record is
// packed into the column entry when the packed arcs stay in L2.
//
// What bounds it: the walkers' dependent chain (Philox, one L2 load, shared
// memory) while few lanes have work, and instruction issue (about 130 per
// step) when all have; the profile of 2 * 10^5 nodes has 55 % of the issue rate.  At 64
// registers per thread (two CTAs of 480 threads on an SM) the kernel spills 104 to 120 bytes
// in all instances.  Against a lane per sample with byte counts in HBM
// (sampler_compact.cu), sampling only: Barabasi-Albert, 10^5 nodes, 16384
// samples 173 -> 75 ms; 10^6 nodes, 4096 samples 750 -> 203 ms; R-MAT of 31
// million arcs, 2048 samples 312 -> 39 ms; 2 * 10^5 nodes with control variate and
// paths, 2048 samples 196 -> 27 ms; Erdos-Renyi, 10^5 nodes, 512 samples
// 1288 -> 169 ms.
#include <cmath>

#include "walk_tasks.cuh"

namespace {

using namespace lap_walks;

constexpr unsigned long long kStallNs = 4000000000ull;    // 4 s without progress: withdraw the sample
constexpr unsigned kStLimit = 1u, kStWithdraw = 2u, kStOverflow = 4u;
constexpr uint32_t kLongPath = 8u, kLongRun = 2u;         // paths this long are added by the whole warp after a run
                                                          // of entries that were
constexpr uint32_t kKMax = 0x3FFFFFFFu;                   // as in the 8-byte kernel
enum : uint32_t { B_OFF = 0, B_SCAN, B_STEP, B_PAIR, B_COMMIT };

// A group's control block: byte offsets in its shared memory.
constexpr uint32_t cPops = 0;         // u64: popped nodes of the sample, Y1 = (n - 1) + pops
constexpr uint32_t cDone = 8;         // nodes in the tree, the root included
constexpr uint32_t cCursor = 12;      // 32-node words handed out for starts (wraps around: sweeps)
constexpr uint32_t cStatus = 16;
constexpr uint32_t cClaim = 20;       // the sample's offset in the launch
constexpr uint32_t cExcl = 24;        // a cycle of more than two nodes is being popped
constexpr uint32_t cInflight = 28;    // two-node pops under way
constexpr uint32_t cIn = 32;          // sweeps: entries of the list read ...
constexpr uint32_t cTake = 36;        // ... taken so far ...
constexpr uint32_t cOut = 40;         // ... and written
constexpr uint32_t kCtlBytes = 48;
constexpr uint32_t kQueue = 64;        // nodes a warp collects for a batch of 32 arrows
constexpr uint32_t kNoArrow = 0xFFFFFFFFu;
constexpr uint32_t kArrowK = 11, kArrowKBits = (1u << kArrowK) - 1u, kArrowKMax = kArrowKBits - 1u;   // {node : 21 | k : 11}

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Shared memory by 32-bit address.
__device__ __forceinline__ uint32_t lds(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long lds64(uint32_t a)
{
    unsigned long long v;
    asm volatile("ld.volatile.shared.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts(uint32_t a, uint32_t v)
{
    asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t atoms_or(uint32_t a, uint32_t v)
{
    uint32_t o;
    asm volatile("atom.shared.or.b32 %0, [%1], %2;" : "=r"(o) : "r"(a), "r"(v) : "memory");
    return o;
}
__device__ __forceinline__ void reds_or(uint32_t a, uint32_t v)
{
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void reds_and(uint32_t a, uint32_t v)
{
    asm volatile("red.shared.and.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t atoms_add(uint32_t a, uint32_t v)
{
    uint32_t o;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(o) : "r"(a), "r"(v) : "memory");
    return o;
}
__device__ __forceinline__ unsigned long long atoms_add64(uint32_t a, unsigned long long v)
{
    unsigned long long o;
    asm volatile("atom.shared.add.u64 %0, [%1], %2;" : "=l"(o) : "r"(a), "l"(v) : "memory");
    return o;
}
__device__ __forceinline__ uint32_t atoms_cas(uint32_t a, uint32_t x, uint32_t v)
{
    uint32_t o;
    asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;" : "=r"(o) : "r"(a), "r"(x), "r"(v) : "memory");
    return o;
}
// Bit u of a bit array.
__device__ __forceinline__ uint32_t word_of(uint32_t a, uint32_t u) { return a + ((u >> 5) << 2); }
__device__ __forceinline__ bool test_bit(uint32_t a, uint32_t u) { return (lds(word_of(a, u)) >> (u & 31u)) & 1u; }

// k (draws popped so far) and lock bit of the nodes of one sample.
struct Draws {
    uint32_t locks;                    // shared: lock bits; lock of node u: bit u & lmask
    uint32_t side;                     // shared: filter bits
    uint32_t lmask, fshift;
    unsigned long long *words;         // in the workspace
    unsigned long long tag;            // sample tag, in the high half

    __device__ __forceinline__ uint32_t k(uint32_t u) const
    {
        if (!test_bit(side, u >> fshift)) return 0u;
        const unsigned long long x = ld_word(words + u);
        return (x ^ tag) >> 32 ? 0u : (uint32_t)x;       // another sample's word: never popped in this one
    }
    // The same in two parts: the load (0: none), and its reading.
    __device__ __forceinline__ unsigned long long k_load(uint32_t u, bool on) const
    {
        return ld_word_if(words + u, on && test_bit(side, u >> fshift));
    }
    __device__ __forceinline__ uint32_t k_of(unsigned long long x) const { return (x ^ tag) >> 32 ? 0u : (uint32_t)x; }
    __device__ __forceinline__ void set_k(uint32_t u, uint32_t x) const
    {
        const uint32_t f = u >> fshift;
        reds_or(word_of(side, f), 1u << (f & 31u));
        st_word(words + u, tag | x);
    }
    __device__ __forceinline__ bool locked(uint32_t u) const { return test_bit(locks, u & lmask); }
    __device__ __forceinline__ bool try_lock(uint32_t u) const
    {
        const uint32_t l = u & lmask, bit = 1u << (l & 31u);
        return !(atoms_or(word_of(locks, l), bit) & bit);
    }
    __device__ __forceinline__ void unlock(uint32_t u) const
    {
        const uint32_t l = u & lmask;
        reds_and(word_of(locks, l), ~(1u << (l & 31u)));
    }
};

// Books one popped node: its k, its repeat visit and, with the control
// variate, the potential of the popped arrow's target t.
template <bool CV>
__device__ __forceinline__ unsigned pop_node(const Draws &d, uint32_t u, uint32_t k, uint32_t t,
                                             const LapSampleLaunch &p)
{
    d.set_k(u, k + 1u);
    atomicAdd(&p.rep1[u], 1ull);
    if (CV && p.cv_h1) atomicAdd(&p.cv_a1[u], (unsigned long long)ld_pot(p.cv_h1 + t));
    return k + 1u >= kKMax ? kStOverflow : 0u;
}

// Pops the cycle of two nodes {u, ku} and its predecessor {w, kw}; returns the
// nodes popped (0: not, or no longer, a cycle of current arrows).
template <bool CV>
__device__ __forceinline__ uint32_t pop_pair(const Draws &d, uint32_t ctl, uint32_t u, uint32_t ku, uint32_t w,
                                             uint32_t kw, const LapSampleLaunch &p, unsigned &status)
{
    // By lock index: in any other order, two pairs whose locks coincide crosswise
    // could fail each other again and again.
    const bool first = (u & d.lmask) < (w & d.lmask);
    const uint32_t a = first ? u : w, b = first ? w : u;
    atoms_add(ctl + cInflight, 1u);
    __threadfence_block();
    bool ok = !lds(ctl + cExcl) && d.try_lock(a);
    if (ok) {
        const bool same = ((a ^ b) & d.lmask) == 0u;
        if (same || d.try_lock(b)) {
            const uint32_t k0 = d.k(u), k1 = d.k(w);
            ok = k0 == ku && k1 == kw;
            if (ok) {
                status |= pop_node<CV>(d, u, ku, w, p) | pop_node<CV>(d, w, kw, u, p);
                __threadfence_block();               // the new k's before the locks' release
            }
            if (!same) d.unlock(b);
        } else {
            ok = false;
        }
        d.unlock(a);
    }
    atoms_add(ctl + cInflight, 0xFFFFFFFFu);
    return ok ? 2u : 0u;
}

// Early phase of a sample, one lane per sample: Wilson's run as Alg. 2 states
// it (exact marks of the current path) until the tree holds `early_nodes`
// nodes, or a step budget is spent, for thousands of samples at once.  While
// the tree is small, a run is a long walk that more walkers cannot shorten, so
// it is left to lanes that wait on memory side by side.  State: an
// open-addressing table per sample of 4-byte entries {node + 1 : 21 | k : 9 |
// path | tree}; a sample that does not fit stops early.  Its entries with
// k > 0 or the tree mark are the sample's state for lewalk_block_kernel.
constexpr uint32_t kETree = 1u, kEPath = 2u, kEKShift = 2u, kEKMask = 511u, kEKeyShift = 11u, kEKMax = 500u;

template <bool CV, bool PACK>
__global__ void __launch_bounds__(128) lewalk_early_kernel(LapSampleLaunch p, LapBlockLaunch b)
{
    const uint32_t per_warp = b.early_lanes;
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t q = (blockIdx.x * (uint64_t)(blockDim.x >> 5) + (threadIdx.x >> 5)) * per_warp + lane;
    if (lane >= per_warp || q >= b.early_count) return;
    const Graph<PACK> g{p.g.rowinfo, p.g.col, b.arcs, b.bw, b.bo, policy_evict_last()};
    const uint32_t n = (uint32_t)p.g.n, v = (uint32_t)p.root, i = p.first + (uint32_t)q;
    const uint32_t key0 = (uint32_t)p.seed, key1 = (uint32_t)(p.seed >> 32);
    uint32_t *tbl = b.early + q * b.early_entries;
    uint32_t *stk = b.early_stacks + q * b.early_cap;            // slots of the path's entries
    const uint32_t mask = b.early_entries - 1u, shift = 32u - b.early_log2;
    uint32_t off, deg, droot;
    g.row(v, off, droot);
    // Expected steps: about 2m / d_v to the root, then a few per node.  A sample
    // that is left without a tree costs the block kernel far more than a lane here.
    const unsigned long long budget64 = 8ull * ((unsigned long long)p.g.arcs / droot) + 4ull * b.early_nodes;
    const uint32_t budget = budget64 > b.early_budget ? b.early_budget : (uint32_t)budget64;
    tbl[((v + 1u) * 2654435761u) >> shift] = (v + 1u) << kEKeyShift | kETree;
    uint32_t used = 1, done = 1, sp = 0, s = 0, u = 0, steps = 0, pops = 0;
    uint32_t com = 0xFFFFFFFFu;                                  // entries of the path still to be added to the tree
    uint32_t top = 0;                                            // CV: target of the entry added next
    g.row(0u, off, deg);
    for (;;) {
        if (com != 0xFFFFFFFFu) {
            // The path leads into the tree: a few entries per turn.
            for (int t = 0; t < 4 && com > 0u; ++t) {
                const uint32_t x = stk[--com];
                const uint32_t e = tbl[x];
                tbl[x] = (e & ~kEPath) | kETree;
                if (CV && p.cv_h1) {
                    const uint32_t node = (e >> kEKeyShift) - 1u;
                    atomicAdd(&p.cv_a1[node], (unsigned long long)ld_pot(p.cv_h1 + top));
                    top = node;
                }
            }
            if (com > 0u) continue;
            done += sp;
            sp = 0;
            com = 0xFFFFFFFFu;
            if (done >= b.early_nodes || s >= n) break;
            u = s;
            g.row(u, off, deg);
        }
        // The arrow of a first visit is asked for beside the node's entry.
        uint64_t a = g.arc(off + below32(lap::philox_r64(u, 0u, i, 0u, key0, key1), deg));
        uint32_t x = ((u + 1u) * 2654435761u) >> shift;
        uint32_t e = tbl[x];
        while (e && (e >> kEKeyShift) != u + 1u) {
            x = (x + 1u) & mask;
            e = tbl[x];
        }
        if (e & kETree) {
            com = sp;
            top = u;
            if (sp == 0u) ++s;                                   // the start itself is in the tree
            if (s >= n && sp == 0u) break;
            continue;
        }
        if (e & kEPath) {
            // The walk closed a cycle at u: pop it.
            uint32_t t = u;
            for (;;) {
                const uint32_t y = stk[--sp];
                const uint32_t f = tbl[y], node = (f >> kEKeyShift) - 1u;
                tbl[y] = (f & ~kEPath) + (1u << kEKShift);
                atomicAdd(&p.rep1[node], 1ull);
                if (CV && p.cv_h1) atomicAdd(&p.cv_a1[node], (unsigned long long)ld_pot(p.cv_h1 + t));
                t = node;
                ++pops;
                if (y == x) break;
            }
            e = tbl[x];
        }
        const uint32_t k = (e >> kEKShift) & kEKMask;
        if (!e) ++used;
        if (++steps > budget || used > b.early_entries / 2u || k >= kEKMax || sp >= b.early_cap) break;
        if (k) a = g.arc(off + below32(lap::philox_r64(u, k, i, 0u, key0, key1), deg));
        tbl[x] = (u + 1u) << kEKeyShift | k << kEKShift | kEPath;
        stk[sp++] = x;
        u = g.target(a);
        g.next_row(a, u, off, deg);
    }
    b.early_pops[q] = pops;
}

// LAP_OPT_WITHDRAW: whether sample q is withdrawn at its start (when 0), before its sweeps
// (1) or at its end (2).
__device__ __forceinline__ bool give_up(const LapBlockLaunch &b, uint32_t q, uint32_t when)
{
    return q % b.withdraw == 0u && q / b.withdraw % 3u == when;
}

// One sample per CTA at a time.  CHECK: with LAP_OPT_WITHDRAW (in the kernel of other calls
// its tests, once per sample, cost 3 % on 10^6 nodes, 205 -> 212 ms).
template <bool CV, bool PACK, bool CHECK>
__global__ void __launch_bounds__(1024, 1) lewalk_block_kernel(LapSampleLaunch p, LapBlockLaunch b)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t wilson = blockDim.x;
    const Graph<PACK> g{p.g.rowinfo, p.g.col, b.arcs, b.bw, b.bo, policy_evict_last()};
    const uint32_t n = (uint32_t)p.g.n, v = (uint32_t)p.root;
    const uint32_t j = threadIdx.x;                      // walker index
    const uint64_t slot = blockIdx.x;
    const uint32_t nwords = (n + 31u) >> 5;
    // Shared memory: control block, tree bits, lock bits, filter bits, and a
    // queue of nodes per warp.
    const uint32_t ctl = (uint32_t)__cvta_generic_to_shared(smem), tree = ctl + kCtlBytes;
    const uint32_t lock_words = (b.lmask + 1u) >> 5;
    Draws d;
    d.locks = tree + 4u * nwords;
    d.side = d.locks + 4u * lock_words;
    d.lmask = b.lmask;
    d.fshift = b.fshift;
    d.words = b.words + slot * (uint64_t)n;
    d.tag = 0;
    const uint32_t side_words = lock_words + (((n - 1u) >> b.fshift) >> 5) + 1u;
    const uint32_t queue = d.locks + 4u * side_words + (threadIdx.x >> 5) * (4u * kQueue);
    uint32_t *arrows = b.sweep + slot * 3ull * n, *list = arrows + n, *list2 = list + n;
    // Path stacks: the first 32 walkers of a sample walk while the tree is small
    // and get the larger ones.
    const uint32_t cap = j < 32u ? b.cap_a : b.cap_b;
    uint2 *stk = b.stacks + slot * (uint64_t)b.stack_entries +
                 (j < 32u ? (uint64_t)j * b.cap_a : 32ull * b.cap_a + (uint64_t)(j - 32u) * b.cap_b);
    const uint32_t key0 = (uint32_t)p.seed, key1 = (uint32_t)(p.seed >> 32);
    const unsigned long long pop_limit = p.step_limit > n - 1u ? p.step_limit - (n - 1u) : 0ull;
    const float grow = b.grow / (float)n;
    unsigned long long acc1 = 0;
    unsigned int bad = 0;

    // All threads of the CTA, their warps converged first (the aligned barrier
    // takes a warp as a whole).
    auto group_sync = [&]() {
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"r"(wilson) : "memory");
    };

    for (;;) {
        // Claim a sample and clear the shared memory; the root and the
        // bits beyond n count as in the tree.
        if (j == 0) sts(ctl + cClaim, atomicAdd(&p.acc->claim, 1u));
        group_sync();
        const uint32_t q = lds(ctl + cClaim);
        if (q >= p.count) break;
        const uint32_t i = p.first + q;
        d.tag = (unsigned long long)lap_word_tag(b.tag_base + q) << 32;
        const bool early = q < b.early_count;
        for (uint32_t x = j; x < nwords; x += wilson) {
            uint32_t t = x == v >> 5 ? 1u << (v & 31u) : 0u;
            if (x == nwords - 1u && (n & 31u)) t |= ~((1u << (n & 31u)) - 1u);
            sts(tree + 4u * x, t);
        }
        for (uint32_t x = j; x < side_words; x += wilson) sts(d.locks + 4u * x, 0u);
        if (j == 0) {
            const uint32_t e = early ? b.early_pops[q] : 0u;
            sts(ctl + cPops, e);
            sts(ctl + cPops + 4u, 0u);
            sts(ctl + cDone, 1u);
            sts(ctl + cCursor, 0u);
            sts(ctl + cExcl, 0u);
            sts(ctl + cInflight, 0u);
            sts(ctl + cStatus, p.step_limit < n - 1u || e > pop_limit ? kStLimit : 0u);
            if (CHECK && give_up(b, q, 0u)) reds_or(ctl + cStatus, kStWithdraw);
        }
        group_sync();
        if (early) {
            // The state that lewalk_early_kernel left.
            const uint4 *t = reinterpret_cast<const uint4 *>(b.early + (uint64_t)q * b.early_entries);
            uint32_t add = 0;
            for (uint32_t x = j; x < b.early_entries / 4u; x += wilson) {
                const uint4 f = t[x];
                const uint32_t e4[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const uint32_t e = e4[y];
                    if (!e) continue;
                    const uint32_t w = (e >> kEKeyShift) - 1u, k = (e >> kEKShift) & kEKMask;
                    if (k) d.set_k(w, k);
                    if ((e & kETree) && w != v) {
                        reds_or(word_of(tree, w), 1u << (w & 31u));
                        ++add;
                    }
                }
            }
            if (add) atoms_add(ctl + cDone, add);
            __threadfence_block();
            group_sync();
        }

        for (int stage = 0; stage < 2; ++stage) {
        // Walkers: first until the tree is large enough for the sweeps (or
        // complete), then on what the sweeps have left.
        const uint32_t goal = stage == 0 && b.sweep_nodes < n ? b.sweep_nodes : n;
        const uint32_t left = stage ? lds(ctl + cIn) : n;          // start nodes: the list's, or all
        const uint32_t units = (left + 31u) >> 5;
        uint32_t phase = lds(ctl + cDone) >= goal || lds(ctl + cStatus) ? (uint32_t)B_OFF : (uint32_t)B_SCAN;
        uint32_t u = 0, ku = 0, off = 0, deg = 1, sp = 0;
        uint32_t r0 = 0, r1 = 0, k0 = 0, k1 = 0;  // path entries sp-1 and sp-2 (valid below sp)
        uint32_t tort = kFull, tpos = 0, hops = 0;                 // Brent's cycle detection
        uint32_t wt = 0;                         // the target of u's arrow (B_COMMIT: in the tree; B_PAIR: entry sp-1)
        uint32_t run = 0;                        // B_COMMIT: entries added one by one
        uint32_t committed = 0;                  // additions to the tree not yet in done
        uint32_t cur = 0, cend = 0;              // units of start nodes taken by this warp
        uint32_t act = 0;                        // walkers j < act look for starts
        uint32_t iter = 0;
        unsigned long long t0 = 0, seen = ~0ull;
        auto update_act = [&](uint32_t done) {
            const float f = grow * (float)done * (float)done;
            act = f >= (float)wilson ? wilson : (uint32_t)f;
            if (act < b.walk_min) act = b.walk_min;
        };
        update_act(lds(ctl + cDone));

        while (!__all_sync(kFull, phase == B_OFF)) {
            ++iter;
            if ((iter & 31u) == 0u) {
                // Reached or given up elsewhere, or nothing has moved for too long.
                if (committed) atoms_add(ctl + cDone, committed);
                committed = 0;
                const uint32_t done = lds(ctl + cDone);
                if ((iter & 1023u) == 0u) {
                    const unsigned long long s = lds64(ctl + cPops) + done, t = now_ns();
                    if (s != seen) { seen = s; t0 = t; }
                    else if (phase != B_OFF && t - t0 > kStallNs) reds_or(ctl + cStatus, kStWithdraw);
                }
                if (done >= goal || lds(ctl + cStatus)) phase = B_OFF;
            }
            // ---- start nodes: lane l takes node l of a unit of 32, so starts
            // are neighbours and need no hand-out; a node whose lane is busy is
            // left to a later sweep.
            const unsigned idle = __ballot_sync(kFull, phase == B_SCAN && j < act);
            const unsigned busy = __ballot_sync(kFull, phase > B_SCAN);
            const bool poll = phase != B_OFF && (busy == 0u || (uint32_t)__popc(idle) >= b.idle_min);
            if (__any_sync(kFull, poll)) {
                // Publish this warp's additions and see whether the sample is
                // complete.
                if (poll && committed) {
                    atoms_add(ctl + cDone, committed);
                    committed = 0;
                }
                __syncwarp();
                if (poll) {
                    const uint32_t done = lds(ctl + cDone);
                    if (done >= goal || lds(ctl + cStatus)) phase = B_OFF;
                    else update_act(done);
                }
                if (__all_sync(kFull, phase == B_OFF)) break;
                const bool mine = poll && phase == B_SCAN && j < act;
                bool got = false;
                for (int t = 0; t < 8; ++t) {
                    const unsigned want = __ballot_sync(kFull, mine && !got);
                    if (!want || (t && (uint32_t)__popc(want) < b.idle_min)) break;
                    if (cur == cend) {
                        if (lane == 0u) cur = atoms_add(ctl + cCursor, b.unit_batch);
                        cur = __shfl_sync(kFull, cur, 0);
                        cur %= units;                    // past the last unit: sweeps
                        cend = cur + b.unit_batch;
                    }
                    const uint32_t x = cur * 32u + lane;
                    ++cur;
                    if (mine && !got && x < left) {
                        const uint32_t s = stage ? list[x] : x;
                        if (!test_bit(tree, s)) {
                            got = true;
                            u = s;
                        }
                    }
                }
                if (got) {
                    g.row(u, off, deg);
                    sp = 0;
                    tort = kFull;
                    hops = 0;
                    phase = B_STEP;
                } else if (poll && busy == 0u) {
                    __nanosleep(idle ? 50 : 400);        // a sweep's end, or not yet this warp's turn
                }
                __syncwarp();
            }
            // ---- one step: the current arrow of u
            uint32_t cpos = kFull, popped = 0;
            if (phase == B_STEP) {
                ku = d.k(u);
                const uint64_t a = g.arc(off + below32(lap::philox_r64(u, ku, i, 0u, key0, key1), deg));
                const uint32_t w = g.target(a);
                if (test_bit(tree, w)) {
                    wt = w;
                    run = 0;
                    phase = B_COMMIT;
                } else {
                    if (sp > 0u && w == r0) {
                        phase = B_PAIR;
                        wt = w;
                    } else {
                        if (sp > 1u && w == r1) cpos = sp - 2u;
                        else if (w == tort) cpos = tpos;
                        if (cpos != kFull) {
                            wt = w;
                        } else {
                            if (sp >= cap) {
                                // The stack is full: forget the path (a sweep
                                // finds its nodes again).
                                phase = B_SCAN;
                            } else {
                                stk[sp] = make_uint2(u, ku);
                                ++sp;
                                r1 = r0;
                                k1 = k0;
                                r0 = u;
                                k0 = ku;
                                ++hops;
                                if ((hops & (hops - 1u)) == 0u) {
                                    tort = w;
                                    tpos = sp;
                                }
                            }
                            u = w;
                        }
                    }
                    g.next_row(a, w, off, deg);
                }
            }
            // ---- cycles of two nodes: a few walkers at a time, since the whole
            // warp waits for one
            const unsigned pairs = __ballot_sync(kFull, phase == B_PAIR);
            if (pairs && ((uint32_t)__popc(pairs) >= b.pair_min || (iter & 3u) == 0u ||
                          !__any_sync(kFull, phase == B_STEP))) {
                if (phase == B_PAIR) {
                    unsigned st = 0;
                    popped = pop_pair<CV>(d, ctl, u, ku, wt, k0, p, st);
                    if (st) reds_or(ctl + cStatus, st);
                    // Popped or not, the walk goes on at the closing node with
                    // its current arrow and the path below it.
                    u = wt;
                    --sp;
                    r0 = r1;
                    k0 = k1;
                    if (sp > 1u) {
                        const uint2 e = stk[sp - 2u];
                        r1 = e.x;
                        k1 = e.y;
                    }
                    tort = kFull;
                    hops = 0;
                    phase = B_STEP;
                }
            }
            // ---- longer cycles, one after the other: all lanes of the warp
            // check and pop the entries
            for (unsigned todo = __ballot_sync(kFull, cpos != kFull); todo; todo &= todo - 1u) {
                const int o = __ffs(todo) - 1;
                const uint32_t oc = __shfl_sync(kFull, cpos, o), osp = __shfl_sync(kFull, sp, o), om = osp - oc + 1u;
                const uint32_t ou = __shfl_sync(kFull, u, o), oku = __shfl_sync(kFull, ku, o), ow = __shfl_sync(kFull, wt, o);
                const uint2 *ob = reinterpret_cast<const uint2 *>(__shfl_sync(kFull, (unsigned long long)stk, o));
                const uint2 *os = ob + oc;
                bool mayc = true;
                if (lane == 0u) {
                    mayc = atoms_cas(ctl + cExcl, 0u, 1u) == 0u;
                    __threadfence_block();
                    if (mayc) {
                        for (int t = 0; t < 100000 && lds(ctl + cInflight); ++t) {}
                        if (lds(ctl + cInflight)) {
                            sts(ctl + cExcl, 0u);
                            mayc = false;
                        }
                    }
                }
                mayc = __shfl_sync(kFull, (int)mayc, 0) != 0;
                if (mayc) {
                    bool valid = true;
                    for (uint32_t x = lane; x < om; x += 32u) {
                        const uint2 e = x + 1u < om ? os[x] : make_uint2(ou, oku);
                        valid = valid && d.k(e.x) == e.y;
                    }
                    if (__all_sync(kFull, valid)) {
                        unsigned st = 0;
                        for (uint32_t x = lane; x < om; x += 32u) {
                            const uint2 e = x + 1u < om ? os[x] : make_uint2(ou, oku);
                            const uint32_t t = x + 2u < om ? os[x + 1u].x : (x + 2u == om ? ou : ow);
                            st |= pop_node<CV>(d, e.x, e.y, t, p);
                        }
                        st = __reduce_or_sync(kFull, st);
                        if ((int)lane == o) {
                            popped = om;
                            if (st) reds_or(ctl + cStatus, st);
                        }
                    }
                    __threadfence_block();
                    __syncwarp();
                    if (lane == 0u) sts(ctl + cExcl, 0u);
                }
                // Cycles longer than the recent entries are seen a lap late: the
                // entries below oc that repeat the cycle backwards go too.
                uint32_t mu = oc;
                for (;;) {
                    const uint32_t x = oc - mu + lane;                // entry oc - 1 - x against position osp - x
                    const bool same = mu > lane && ob[mu - 1u - lane].x == (x ? ob[osp - x].x : ou);
                    const unsigned diff = ~__ballot_sync(kFull, same);
                    const uint32_t eq = diff ? (uint32_t)__ffs(diff) - 1u : 32u;
                    mu -= eq;
                    if (eq < 32u) break;
                }
                if ((int)lane == o) {
                    u = ow;
                    if (mu != oc) {
                        u = stk[mu].x;
                        g.row(u, off, deg);
                    }
                    sp = mu;
                    if (sp > 0u) {
                        const uint2 e = stk[sp - 1u];
                        r0 = e.x;
                        k0 = e.y;
                    }
                    if (sp > 1u) {
                        const uint2 e = stk[sp - 2u];
                        r1 = e.x;
                        k1 = e.y;
                    }
                    tort = kFull;
                    hops = 0;
                }
            }
            if (popped) {
                const unsigned long long before = atoms_add64(ctl + cPops, (unsigned long long)popped);
                if (before + popped > pop_limit) reds_or(ctl + cStatus, kStLimit);
            }
            // ---- long paths into the tree: all lanes of the warp check and
            // add 32 entries at a time.  An entry may be added when it is in the
            // tree already, or its k and those of all entries above it are the
            // ones seen: none has changed since the walker passed it, so all these
            // arrows are current together and lead into the tree.
            for (unsigned todo = __ballot_sync(kFull, phase == B_COMMIT && sp >= kLongPath && run >= kLongRun); todo;
                 todo &= todo - 1u) {
                const int o = __ffs(todo) - 1;
                const uint32_t osp = __shfl_sync(kFull, sp, o), ou = __shfl_sync(kFull, u, o), oku = __shfl_sync(kFull, ku, o);
                uint32_t above = __shfl_sync(kFull, wt, o);
                const uint2 *os = reinterpret_cast<const uint2 *>(__shfl_sync(kFull, (unsigned long long)stk, o));
                uint32_t x0 = 0, added = 0, good = 32u;     // entry 0 is the head, entry x the x-th below it
                for (; x0 <= osp; x0 += 32u) {
                    const uint32_t x = x0 + lane;
                    uint2 e = make_uint2(ou, oku);
                    if (x && x <= osp) e = os[osp - x];
                    const bool valid = x <= osp && (test_bit(tree, e.x) ||
                                                    (!d.locked(e.x) && !lds(ctl + cExcl) && d.k(e.x) == e.y));
                    const unsigned bad_lanes = ~__ballot_sync(kFull, valid);
                    good = bad_lanes ? (uint32_t)__ffs(bad_lanes) - 1u : 32u;
                    uint32_t t = __shfl_up_sync(kFull, e.x, 1);
                    if (lane == 0u) t = above;
                    bool fresh = false;
                    if (lane < good) {
                        const uint32_t bit = 1u << (e.x & 31u);
                        fresh = !(atoms_or(word_of(tree, e.x), bit) & bit);
                        if (CV && fresh && p.cv_h1) atomicAdd(&p.cv_a1[e.x], (unsigned long long)ld_pot(p.cv_h1 + t));
                    }
                    added += __popc(__ballot_sync(kFull, fresh));
                    if (good) above = __shfl_sync(kFull, e.x, (int)good - 1);
                    if (good < 32u) break;
                }
                if ((int)lane == o) {
                    committed += added;
                    const uint32_t x = x0 + good;           // first entry not added
                    if (x0 > osp || x > osp) {
                        sp = 0;
                        phase = B_SCAN;
                    } else if (x) {
                        sp = osp - x;
                        const uint2 e = os[sp];
                        u = e.x;
                        ku = e.y;
                        wt = above;
                        if (sp > 0u) {
                            const uint2 f = stk[sp - 1u];
                            r0 = f.x;
                            k0 = f.y;
                        }
                        if (sp > 1u) {
                            const uint2 f = stk[sp - 2u];
                            r1 = f.x;
                            k1 = f.y;
                        }
                    }
                }
            }
            // ---- u's arrow leads into the tree
            if (phase == B_COMMIT && !d.locked(u) && !lds(ctl + cExcl)) {
                const uint32_t k = d.k(u);
                const uint32_t bit = 1u << (u & 31u);
                if (k != ku && !(lds(word_of(tree, u)) & bit)) {
                    // Popped since: take its current arrow.
                    run = 0;
                    g.row(u, off, deg);
                    tort = kFull;
                    hops = 0;
                    phase = B_STEP;
                } else {
                    if (!(atoms_or(word_of(tree, u), bit) & bit)) {
                        ++committed;
                        if (CV && p.cv_h1) atomicAdd(&p.cv_a1[u], (unsigned long long)ld_pot(p.cv_h1 + wt));
                    }
                    if (sp == 0u) phase = B_SCAN;
                    else {
                        ++run;
                        wt = u;
                        u = r0;
                        ku = k0;
                        --sp;
                        r0 = r1;
                        k0 = k1;
                        if (sp > 1u) {
                            const uint2 e = stk[sp - 2u];
                            r1 = e.x;
                            k1 = e.y;
                        }
                    }
                }
            }
        }

        group_sync();
        if (stage || goal == n || lds(ctl + cDone) >= n || lds(ctl + cStatus) || (CHECK && give_up(b, q, 1u))) break;
        {
        uint32_t added = 0;
        // The node's arrow leads to w in the tree, seen with k = ku.
        auto join = [&](uint32_t u, uint32_t ku, uint32_t w) {
            if (d.locked(u) || d.k(u) != ku) return false;
            const uint32_t bit = 1u << (u & 31u);
            if (!(atoms_or(word_of(tree, u), bit) & bit)) {
                ++added;
                if (CV && p.cv_h1) atomicAdd(&p.cv_a1[u], (unsigned long long)ld_pot(p.cv_h1 + w));
            }
            return true;
        };
        auto publish = [&]() {
            const uint32_t sum = __reduce_add_sync(kFull, added);
            added = 0;
            if (lane == 0u && sum) atoms_add(ctl + cDone, sum);
            __syncwarp();
            return sum;
        };
        // The cycle of two nodes {node | k}, as seen.
        auto pop_two = [&](uint32_t x, uint32_t y) {
            unsigned st = 0;
            if (pop_pair<CV>(d, ctl, x >> kArrowK, x & kArrowKBits, y >> kArrowK, y & kArrowKBits, p, st)) {
                const unsigned long long before = atoms_add64(ctl + cPops, 2ull);
                if (before + 2ull > pop_limit) st |= kStLimit;
            }
            if (st) reds_or(ctl + cStatus, st);
        };
        // ---- sweeps: every node outside the tree looks whether its arrow leads
        // into the tree, again and again.  The first pass computes the arrows,
        // stores them and lists the nodes that stay outside; later passes read
        // list and arrows (a few instructions per node instead of a Philox draw
        // and a graph read), and where they gain little, a pass also pops the
        // cycles of two nodes.
        uint32_t qn = 0;                              // nodes in the warp's queue
        // Appends the lanes' nodes to the list being written.
        auto keep = [&](bool yes, uint32_t u) {
            const unsigned m = __ballot_sync(kFull, yes);
            if (!m) return;
            uint32_t at = 0;
            if (lane == 0u) at = atoms_add(ctl + cOut, (uint32_t)__popc(m));
            at = __shfl_sync(kFull, at, 0);
            if (yes) list2[at + __popc(m & ((1u << lane) - 1u))] = u;
        };
        // Computes the arrows of up to 32 queued nodes.
        auto flush = [&](uint32_t count) {
            const bool on = lane < count;
            const uint32_t u = on ? lds(queue + 4u * (qn - count + lane)) : 0u;
            const uint64_t r = g.row_if(u, on);
            const uint32_t k = d.k_of(d.k_load(u, on));
            const uint64_t a = g.arc_if((uint32_t)r + below32(lap::philox_r64(u, k, i, 0u, key0, key1), (uint32_t)(r >> 32)), on);
            qn -= count;
            __syncwarp();
            bool stay = on;
            if (on) {
                const uint32_t w = g.target(a);
                if (test_bit(tree, w) && join(u, k, w)) stay = false;
                else arrows[u] = k <= kArrowKMax ? w << kArrowK | k : kNoArrow;
            }
            keep(stay, u);
        };
        auto push = [&](bool yes, uint32_t u) {
            const unsigned m = __ballot_sync(kFull, yes);
            if (yes) sts(queue + 4u * (qn + __popc(m & ((1u << lane) - 1u))), u);
            qn += __popc(m);
            __syncwarp();
            if (qn >= 32u) flush(32u);
        };
        uint32_t in = nwords * 32u;                   // entries of this pass
        bool first = true, pops = false, stuck = false;
        for (int pass = 0; pass < 1000; ++pass) {
            if (j == 0) {
                sts(ctl + cTake, 0u);
                sts(ctl + cOut, 0u);
            }
            group_sync();
            for (;;) {
                uint32_t at = 0;
                if (lane == 0u) at = atoms_add(ctl + cTake, 128u);
                at = __shfl_sync(kFull, at, 0);
                if (at >= in) break;
                if (first) {
                    for (uint32_t c = at; c < at + 128u && c < in; c += 32u)
                        push(!((lds(tree + (c >> 3)) >> lane) & 1u), c + lane);
                    continue;
                }
                uint32_t u4[4], a4[4];
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const uint32_t c = at + 32u * y + lane;
                    u4[y] = ld_u32_if(list + c, c < in);
                }
#pragma unroll
                for (int y = 0; y < 4; ++y) a4[y] = ld_u32_if(arrows + u4[y], at + 32u * y + lane < in);
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const bool on = at + 32u * y + lane < in;
                    const uint32_t u = u4[y], a = a4[y], w = a >> kArrowK;
                    bool stay = on, renew = false;
                    if (on) {
                        if (a == kNoArrow) {
                            renew = true;
                            stay = false;
                        } else if (test_bit(tree, w)) {
                            stay = false;
                            renew = !join(u, a & kArrowKBits, w);
                        }
                    }
                    if (pops) {
                        // u -> w -> u: popped by the lower node.
                        const uint32_t back = ld_u32_if(arrows + w, stay && u < w);
                        const bool pair = stay && u < w && back != kNoArrow && back >> kArrowK == u;
                        if (__any_sync(kFull, pair)) {
                            if (pair) {
                                pop_two(u << kArrowK | (a & kArrowKBits), w << kArrowK | (back & kArrowKBits));
                                arrows[u] = kNoArrow;
                                arrows[w] = kNoArrow;
                                renew = true;
                                stay = false;
                            }
                            __syncwarp();
                        }
                    }
                    keep(stay, u);
                    push(renew, u);
                }
            }
            if (qn) flush(qn);
            publish();
            group_sync();
            const uint32_t out = lds(ctl + cOut);
            const bool over = out == 0u || lds(ctl + cStatus);
            group_sync();                             // (read before the next pass resets it)
            // The walkers take the rest when it is small, or when neither kind
            // of pass gets on.
            const bool slow = !first && out >= in - in / 8u;
            const bool hard = slow && pops && out >= in - in / 64u;
            uint32_t *t = list;
            list = list2;
            list2 = t;
            const bool small = out <= b.sweep_rest;
            in = out;
            if (over || small || (hard && stuck)) break;
            stuck = hard;
            pops = slow && !pops ? true : (slow && hard);
            first = false;
        }
        // Read before the barrier: beyond it the first warps' walkers change both words,
        // and a warp that saw them changed would leave with one barrier less than the
        // others.
        const bool complete = lds(ctl + cDone) >= n || lds(ctl + cStatus);
        if (j == 0) {
            sts(ctl + cIn, in);
            sts(ctl + cCursor, 0u);
        }
        group_sync();
        if (complete) break;
        }
        }

        if (CHECK && j == 0 && (give_up(b, q, 1u) || give_up(b, q, 2u))) reds_or(ctl + cStatus, kStWithdraw);
        group_sync();
        const unsigned st = lds(ctl + cStatus);
        if (st & kStLimit) bad |= LAP_DEV_STEP_LIMIT;
        if (st & kStOverflow) bad |= LAP_DEV_K_OVERFLOW;
        if (st & kStWithdraw) {
            // Withdraw the sample: subtract the pops counted so far and, with
            // the control variate, the potentials of the arrows popped and of
            // the last arrows of the nodes in the tree.
            for (uint32_t x = j; x < n; x += wilson) {
                const uint32_t k = d.k(x);
                if (k) atomicAdd(&p.rep1[x], (unsigned long long)(-(long long)k));
                if (CV && p.cv_h1 && x != v) {
                    const uint32_t draws = k + (test_bit(tree, x) ? 1u : 0u);
                    if (!draws) continue;
                    uint32_t o, dg;
                    g.row(x, o, dg);
                    long long sub = 0;
                    for (uint32_t y = 0; y < draws; ++y)
                        sub += ld_pot(p.cv_h1 + g.target(g.arc(o + below32(lap::philox_r64(x, y, i, 0u, key0, key1), dg))));
                    atomicAdd(&p.cv_a1[x], (unsigned long long)(-sub));
                }
            }
            if (j == 0) {
                const unsigned int ix = atomicAdd(&p.acc->ovf_count, 1u);
                if (p.ovf_ids && ix < b.ovf_cap) p.ovf_ids[ix] = i;
            }
        } else if (j == 0) {
            const unsigned long long y1 = (unsigned long long)(n - 1u) + lds64(ctl + cPops);
            acc1 += y1;
            if (p.y1_out) p.y1_out[q] = y1;
        }
        if (p.tree_out && !st) {
            // The tree: every node's current arrow.
            uint32_t *out = p.tree_out + (uint64_t)q * n;
            for (uint32_t x = j; x < n; x += wilson) {
                uint32_t o, dg;
                g.row(x, o, dg);
                out[x] = g.target(g.arc(o + below32(lap::philox_r64(x, d.k(x), i, 0u, key0, key1), dg)));
            }
        }
        group_sync();
        if (bad) break;
    }
    if (acc1) atomicAdd(&p.acc->sum_y1, acc1);
    if (bad) atomicOr(&p.acc->status, bad);
}

__global__ void pack_arcs_kernel(const int2 *__restrict__ rowinfo, const int32_t *__restrict__ col, int64_t arcs,
                                 uint32_t bw, uint32_t bo, unsigned long long *__restrict__ out)
{
    const uint32_t dmax = (uint32_t)((1ull << (64u - bw - bo)) - 1ull);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < arcs; e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t w = (uint32_t)col[e];
        const int2 r = rowinfo[w];
        const uint32_t d = (uint32_t)r.y < dmax ? (uint32_t)r.y : dmax;
        out[e] = (unsigned long long)w | (unsigned long long)(uint32_t)r.x << bw | (unsigned long long)d << (bw + bo);
    }
}

uint32_t bits_for(uint64_t x)          // smallest b with x < 2^b
{
    uint32_t b = 1;
    while (x >> b) ++b;
    return b;
}

constexpr uint64_t kSmemMax = 227ull << 10;
uint64_t align16(uint64_t x) { return (x + 15ull) & ~15ull; }

template <bool CHECK>
const void *kernel_of(bool cv, bool pack)
{
    if (cv) return pack ? (const void *)lewalk_block_kernel<true, true, CHECK> : (const void *)lewalk_block_kernel<true, false, CHECK>;
    return pack ? (const void *)lewalk_block_kernel<false, true, CHECK> : (const void *)lewalk_block_kernel<false, false, CHECK>;
}
const void *kernel_for(bool cv, bool pack, bool check = false) { return check ? kernel_of<true>(cv, pack) : kernel_of<false>(cv, pack); }

template <bool CV, bool PACK>
void launch_early(const LapSampleLaunch &p, const LapBlockLaunch &b, unsigned blocks, cudaStream_t st)
{
    lewalk_early_kernel<CV, PACK><<<blocks, 128, 0, st>>>(p, b);
}

}  // namespace

void lap_pack_bits(int32_t n, int64_t arcs, uint32_t *bw, uint32_t *bo)
{
    *bw = bits_for((uint64_t)n - 1ull);
    *bo = bits_for((uint64_t)arcs);
}

cudaError_t lap_launch_pack_arcs(const int2 *rowinfo, const int32_t *col, int32_t n, int64_t arcs,
                                 unsigned long long *out, cudaStream_t st)
{
    uint32_t bw, bo;
    lap_pack_bits(n, arcs, &bw, &bo);
    int64_t grid = (arcs + 255) / 256;
    if (grid > 152 * 16) grid = 152 * 16;
    pack_arcs_kernel<<<(unsigned)grid, 256, 0, st>>>(rowinfo, col, arcs, bw, bo, out);
    return cudaGetLastError();
}

// The launch of `count` samples in `ws_bytes` of workspace: threads, CTAs,
// shared memory and the workspace's layout (words, path words, stacks, sweep
// arrays, early tables).  False: the graph's tree bits exceed an SM's shared
// memory, or the workspace does not hold one sample.
bool lap_block_plan(int32_t n, int64_t arcs, int32_t root_degree, int32_t max_degree, uint64_t count, uint64_t slots_opt, uint64_t ws_bytes, int num_sms, bool paths, bool cv,
                    bool pack, LapBlockPlan *out)
{
    LapBlockPlan pl;
    const uint64_t nn = (uint64_t)n, tree = 4ull * ((nn + 31ull) / 32ull);
    if (num_sms < 1) num_sms = 1;
    uint64_t want = count;                                // samples in flight
    if (slots_opt && slots_opt < want) want = slots_opt;
    if (want == 0) want = 1;
    const uint64_t per_sm = (want + num_sms - 1) / num_sms;
    LapBlockLaunch &b = pl.b;
    // Threads: as many CTAs on an SM as registers and tree bits leave room for, and the
    // walkers a sample of that size uses.  Against the neighbouring counts: 20,000 nodes 96 /
    // 128 / 192 threads 13.4 / 13.3 / 13.0 ms, 50,000 nodes 128 / 224 / 288: 25.9 / 24.6 /
    // 24.7 ms, 100,000 nodes 288 / 480 / 672: 42.2 / 40.6 / 48.7 ms, 300,000 nodes 288 / 480 /
    // 992: 73.9 / 58.5 / 59.5 ms, 10^6 nodes 480 / 992: 126 / 85.5 ms (Barabasi-Albert, 8192
    // samples; 4096 and 1520 of the last two).  The lines lie between the measured sizes.
    pl.threads = nn < 24000 ? 128 : nn < 64000 ? 224 : nn < 400000 ? 480 : 992;
    if (per_sm * (uint64_t)(pl.threads + 32) <= 512ull) pl.threads *= 2;
    b.lmask = 8191u;
    const uint64_t fixed = kCtlBytes + tree + 1024ull + (uint64_t)pl.threads / 32ull * 4ull * kQueue;
    uint32_t fs = 0;
    while (fs < 8 && fixed + 4ull * ((((nn - 1ull) >> fs) >> 5) + 1ull) > kSmemMax) ++fs;
    pl.smem = align16(fixed + 4ull * ((((nn - 1ull) >> fs) >> 5) + 1ull));
    if (pl.smem > kSmemMax) return false;
    b.fshift = fs;
    // The same for every size: on the graphs above, an R-MAT graph of 31 million arcs and
    // Erdos-Renyi graphs of 15,000 and 50,000 nodes, other values are within 1 % or slower
    // but for walk_min 64 (3 and 5 % faster on the two graphs below 24,000 nodes) and grow 16
    // (2 to 4 % from 50,000 nodes on); idle_min 28 costs 8 to 23 %, grow 2 up to 5 %, sweeps from
    // 0.2 n up to 9 % (they gain 5 % on the R-MAT graph), unit_batch 1 up to 3 %.
    b.walk_min = 32u;
    b.grow = 4.0f;
    b.idle_min = 12u;
    b.pair_min = 4u;
    b.unit_batch = 4u;
    // Paths of first walks have about sqrt(n) nodes, on sparse graphs a few times that;
    // a sample whose path does not fit ends its early phase without a tree.  (With 4096
    // entries at every size, 256 samples of Erdos-Renyi graphs of 10^6 nodes took over a
    // minute; now 3.2 s, a lane per sample 11.9 s.)
    uint64_t path = 4096ull;
    while (path * path < 256ull * nn) path *= 2ull;
    b.cap_a = (uint32_t)(2ull * nn + 64ull < 2ull * path ? 2ull * nn + 64ull : 2ull * path);
    b.cap_b = 512u;
    b.sweep_nodes = (uint32_t)(nn * 35ull / 100ull);
    b.sweep_rest = (uint32_t)(nn / 200ull < 64ull ? 64ull : nn / 200ull);
    const void *kernel = kernel_for(cv, pack);
    int resident = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, kernel, pl.threads + 32, pl.smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (resident < 1) return false;
    // A warp of absorbed walks per CTA in flight, as counted for `resident`.
    pl.walk_ctas = (uint64_t)resident * num_sms;
    uint64_t slots = want < (uint64_t)resident * num_sms ? want : (uint64_t)resident * num_sms;
    // Early phase: until about twice sqrt(8 / n) of the nodes are in the tree,
    // where 32 walkers become useful.  A sample's table has four entries for each
    // of them, and two for each node that a long first walk passes: it reaches
    // the root after 2m / d_v steps on average, few beside a hub but 36,000 on an
    // Erdos-Renyi graph of 100,000 nodes.
    const uint64_t target = (uint64_t)(5.7 * sqrt((double)nn));
    uint64_t pass = 4ull * ((uint64_t)arcs / (uint64_t)(root_degree > 0 ? root_degree : 1));
    if (pass > nn) pass = nn;
    // A hub is drawn about d / d_v times on the way to the root.  Where that is more
    // than the tables' 9 bits count, samples reach the block kernel without a tree,
    // and its walkers do not shorten the rest.  It is still the faster kernel for few
    // samples (64 on a graph of 200,000 nodes, hub of degree 1823, rooted at degree 6:
    // 1.3 s, a lane per sample 3.7 s), but runs them some 300 at a time, where the
    // other kernels run all at once.
    if (pass > 16ull * target && max_degree / 64 > root_degree && count > 4ull * num_sms) return false;
    uint32_t lg = 10;
    while ((1ull << lg) < 4ull * target || (1ull << lg) < 2ull * pass) ++lg;
    b.early_log2 = lg;
    b.early_entries = 1u << lg;
    b.early_nodes = (uint32_t)target;
    b.early_cap = (uint32_t)path;
    b.early_budget = 1u << 22;
    const uint64_t early_per = 4ull * b.early_entries + 4ull * b.early_cap + 4ull;
    // The workspace: at most half for the early tables (none if no sample fits
    // beside them); then shorter stacks, then fewer samples in flight.
    const uint64_t node_bytes = (8ull + 12ull) * nn;
    const uint64_t path_bytes = paths ? 8ull * nn : 0ull;       // one walk's departures, at least
    const uint64_t slack = 2048ull;
    uint64_t reserve = early_per * count < ws_bytes / 2ull ? early_per * count : ws_bytes / 2ull;
    for (;;) {
        b.stack_entries = 32ull * b.cap_a + (uint64_t)(pl.threads - 32) * b.cap_b;
        const uint64_t per = node_bytes + 8ull * b.stack_entries, other = path_bytes + slack + reserve;
        if (slots * per + other <= ws_bytes) break;
        if (b.cap_a > 4096u || b.cap_b > 64u) {
            // Not below 4096 (or 2 n): a cycle longer than every stack is never found.
            if (b.cap_a > 4096u) b.cap_a = 4096u;
            if (b.cap_b > 64u) b.cap_b /= 2u;
        } else {
            const uint64_t fit = (ws_bytes > other ? ws_bytes - other : 0ull) / per;
            if (fit) slots = fit;
            else if (reserve) reserve = 0;
            else return false;
        }
    }
    pl.slots = slots;
    const uint64_t fixed_bytes = slots * (node_bytes + 8ull * b.stack_entries) + slack;
    if (paths) {
        // At most half of the rest: the early tables need some too.
        b.path_lanes = (ws_bytes - fixed_bytes + path_bytes) / 2ull / path_bytes;
        if (b.path_lanes < 1ull) b.path_lanes = 1ull;
        if (b.path_lanes > pl.walk_ctas * 32ull) b.path_lanes = pl.walk_ctas * 32ull;
    }
    auto up = [](uint64_t x) { return (x + 255ull) & ~255ull; };
    pl.path_offset = slots * 8ull * nn;
    pl.words_bytes = pl.path_offset + b.path_lanes * path_bytes;
    pl.stack_offset = up(pl.words_bytes);
    pl.sweep_offset = up(pl.stack_offset + 8ull * slots * b.stack_entries);
    pl.early_offset = up(pl.sweep_offset + 12ull * slots * nn);
    // Early tables from what the workspace has left.
    uint64_t m = ws_bytes > pl.early_offset + 64ull ? (ws_bytes - pl.early_offset - 64ull) / early_per : 0ull;
    if (m > count) m = count;
    b.early_count = (uint32_t)m;
    pl.bytes = fixed_bytes + b.path_lanes * path_bytes + early_per * m + 64ull;
    // Where the first walk is long, a call whose tables do not fit runs in parts.
    if (pass > 16ull * target) pl.table_bytes = early_per * count;
    b.part = pl.table_bytes && b.early_count > 0 && b.early_count < count ? b.early_count : (uint32_t)count;
    // Few samples per warp: a warp's lanes wait for each other.
    const uint64_t warps = 16ull * num_sms;
    const uint64_t l = (m + warps - 1) / warps;
    b.early_lanes = (uint32_t)(l < 1 ? 1 : l > 32 ? 32 : l);
    *out = pl;
    return true;
}

cudaError_t lap_launch_sample_block(const LapSampleLaunch &all, const LapBlockPlan &pl, cudaStream_t st)
{
    if (all.count == 0 || pl.slots == 0) return cudaSuccess;
    const bool cv = all.cv_h1 || all.cv_h2, pack = pl.b.arcs != nullptr;
    const void *kernel = kernel_for(cv, pack, pl.b.withdraw != 0u);
    if (pl.b.withdraw) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
        if (e != cudaSuccess) return e;
    }
    for (uint32_t done = 0; done < all.count; done += pl.b.part) {
        LapSampleLaunch p = all;
        LapBlockLaunch b = pl.b;
        p.first += done;
        p.count = all.count - done < b.part ? all.count - done : b.part;
        if (p.y1_out) p.y1_out += done;
        if (p.tree_out) p.tree_out += (uint64_t)done * (uint64_t)p.g.n;
        b.tag_base += done;
        b.ovf_cap = all.count;
        if (b.early_count > p.count) b.early_count = p.count;
        cudaError_t e = done ? cudaMemsetAsync(&p.acc->claim, 0, sizeof(unsigned int), st) : cudaSuccess;
        if (e != cudaSuccess) return e;
        if (b.early_count) {
            e = cudaMemsetAsync(b.early, 0, 4ull * b.early_entries * b.early_count, st);
            if (e != cudaSuccess) return e;
            const uint64_t per_block = 4ull * b.early_lanes;
            const unsigned blocks = (unsigned)((b.early_count + per_block - 1) / per_block);
            if (cv) pack ? launch_early<true, true>(p, b, blocks, st) : launch_early<true, false>(p, b, blocks, st);
            else pack ? launch_early<false, true>(p, b, blocks, st) : launch_early<false, false>(p, b, blocks, st);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        void *args[2] = {&p, &b};
        const uint64_t ctas = pl.slots < p.count ? pl.slots : p.count;
        e = cudaLaunchKernel(kernel, dim3((unsigned)ctas), dim3((unsigned)pl.threads), args, (size_t)pl.smem, st);
        if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}
