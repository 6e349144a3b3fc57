// Graph reads shared by the samplers that leave the absorbed walks to a kernel of
// their own (sampler_block.cu, sampler_small.cu), and these walks (launched by
// sampler_cta.cu).
#pragma once

#include "lap_internal.h"
#include "philox.cuh"

namespace lap_walks {

constexpr unsigned kFull = 0xFFFFFFFFu;

static __device__ __forceinline__ unsigned long long ld_word(const unsigned long long *a)
{
    unsigned long long v;
    asm volatile("ld.relaxed.cta.global.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
    return v;
}
static __device__ __forceinline__ void st_word(unsigned long long *a, unsigned long long v)
{
    asm volatile("st.relaxed.cta.global.u64 [%0], %1;" ::"l"(a), "l"(v) : "memory");
}
// Loads that happen only where `on` (0 otherwise), with no branch, so that
// several can be in flight.
static __device__ __forceinline__ unsigned long long ld_word_if(const unsigned long long *a, bool on)
{
    unsigned long long v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.u64 %0, 0;\n\t"
                 "@p ld.relaxed.cta.global.u64 %0, [%1];\n\t}" : "=l"(v) : "l"(a), "r"((uint32_t)on) : "memory");
    return v;
}
static __device__ __forceinline__ uint32_t ld_u32_if(const uint32_t *a, bool on)
{
    uint32_t v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.u32 %0, 0;\n\t"
                 "@p ld.relaxed.cta.global.u32 %0, [%1];\n\t}" : "=r"(v) : "l"(a), "r"((uint32_t)on) : "memory");
    return v;
}
static __device__ __forceinline__ uint64_t ld_graph64_if(const void *a, uint64_t pol, bool on)
{
    uint64_t v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.u64 %0, 0;\n\t"
                 "@p ld.global.nc.L2::cache_hint.u64 %0, [%1], %2;\n\t}" : "=l"(v) : "l"(a), "l"(pol), "r"((uint32_t)on));
    return v;
}
static __device__ __forceinline__ uint32_t ld_graph32_if(const int32_t *a, uint64_t pol, bool on)
{
    uint32_t v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.u32 %0, 0;\n\t"
                 "@p ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;\n\t}" : "=r"(v) : "l"(a), "l"(pol), "r"((uint32_t)on));
    return v;
}
static __device__ __forceinline__ uint64_t policy_evict_last()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
static __device__ __forceinline__ uint64_t ld_u64(const void *a, uint64_t pol)
{
    uint64_t v;
    asm volatile("ld.global.nc.L2::cache_hint.u64 %0, [%1], %2;" : "=l"(v) : "l"(a), "l"(pol));
    return v;
}
static __device__ __forceinline__ uint32_t ld_u32(const int32_t *a, uint64_t pol)
{
    uint32_t v;
    asm volatile("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(a), "l"(pol));
    return v;
}
static __device__ __forceinline__ long long ld_pot(const long long *a)
{
    long long v;
    asm volatile("ld.global.nc.s64 %0, [%1];" : "=l"(v) : "l"(a));
    return v;
}
// High 64 bits of x * r for a 32-bit r (lap::below).
static __device__ __forceinline__ uint32_t below32(uint64_t x, uint32_t r)
{
    const uint64_t t = (uint64_t)(uint32_t)x * r >> 32;
    return (uint32_t)(((x >> 32) * (uint64_t)r + t) >> 32);
}

// The graph as the kernels read it: row record {offset, degree} and the next
// node of draw x at a node.  PACK: one 8-byte entry per arc {target, its row
// offset, its degree}, so a step needs no row load.
template <bool PACK>
struct Graph {
    const int2 *rowinfo;
    const int32_t *col;
    const unsigned long long *arcs;
    uint32_t bw, bo;             // bits of the target and of the offset in a packed arc
    uint64_t pol;

    __device__ __forceinline__ void row(uint32_t u, uint32_t &off, uint32_t &deg) const
    {
        const uint64_t r = ld_u64(rowinfo + u, pol);
        off = (uint32_t)r;
        deg = (uint32_t)(r >> 32);
    }
    __device__ __forceinline__ uint64_t row_if(uint32_t u, bool on) const { return ld_graph64_if(rowinfo + u, pol, on); }
    __device__ __forceinline__ uint64_t arc_if(uint32_t e, bool on) const
    {
        return PACK ? ld_graph64_if(arcs + e, pol, on) : (uint64_t)ld_graph32_if(col + e, pol, on);
    }
    // The raw entry of arc e; split by target() and, for a node that is walked
    // on, next_row().
    __device__ __forceinline__ uint64_t arc(uint32_t e) const
    {
        return PACK ? ld_u64(arcs + e, pol) : (uint64_t)ld_u32(col + e, pol);
    }
    __device__ __forceinline__ uint32_t target(uint64_t a) const
    {
        return PACK ? (uint32_t)a & ((1u << bw) - 1u) : (uint32_t)a;
    }
    __device__ __forceinline__ void next_row(uint64_t a, uint32_t w, uint32_t &off, uint32_t &deg) const
    {
        if (PACK) {
            const uint32_t d = (uint32_t)(a >> (bw + bo));
            off = (uint32_t)(a >> bw) & (uint32_t)((1ull << bo) - 1ull);
            deg = d;
            if (d == (uint32_t)((1ull << (64u - bw - bo)) - 1ull)) row(w, off, deg);    // saturated
        } else {
            row(w, off, deg);
        }
    }
};

// The absorbed walks of the launch's samples, one lane per walk: task 2 q is
// the uniform-start (or fixed-start) walk of sample q with its passes, task
// 2 q + 1 its pi-start walk (Y2 and, with the control variate, M2).  Own draws
// depend on the step alone, so the next one is computed while the column load
// is in flight; loop-included paths count departures in 8-byte words
// {tag 32 | count 32} of the lane's region.
template <bool CV, bool PACK>
static __device__ void walk_tasks(const LapSampleLaunch &p, const LapBlockLaunch &b, const Graph<PACK> &g)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t wl = blockIdx.x * 32ull + lane;
    unsigned long long *pw = p.paths ? b.path_words + wl * (uint64_t)p.g.n : nullptr;
    const bool usable = !p.paths || wl < b.path_lanes;
    const uint32_t key0 = (uint32_t)p.seed, key1 = (uint32_t)(p.seed >> 32);
    const uint32_t v = (uint32_t)p.root;
    const uint64_t tasks = 2ull * p.count;
    const uint32_t ustart = p.ustart_dev ? *p.ustart_dev : p.ustart;
    bool open = usable, active = false;
    uint32_t kind = 0, q = 0, u = v, off = 0, deg = 1, i = 0;
    uint64_t t = 0, r = 0;
    unsigned long long tag = 0, acc2 = 0;
    double m2 = 0.0;
    unsigned int bad = 0;

    for (;;) {
        const unsigned want = __ballot_sync(kFull, open && !active);
        if (want) {
            unsigned int first = 0;
            const int leader = __ffs(want) - 1;
            if ((int)lane == leader) first = atomicAdd(&p.acc->walk_claim, (unsigned int)__popc(want));
            first = __shfl_sync(kFull, first, leader);
            if (open && !active) {
                const uint64_t id = (uint64_t)first + __popc(want & ((1u << lane) - 1u));
                if (id >= tasks) open = false;
                else {
                    q = (uint32_t)(id >> 1);
                    kind = (uint32_t)id & 1u;
                    i = p.first + q;
                    t = 0;
                    m2 = 0.0;
                    active = true;
                    tag = (unsigned long long)lap_path_tag(b.tag_base + q, kind) << 32;
                    if (kind == 0) {
                        u = ustart ? ustart - 1u
                                   : (uint32_t)lap::below(lap::philox_r64(0u, 0u, i, 1u, key0, key1), (uint64_t)p.g.n);
                        g.row(u, off, deg);
                    } else {
                        const uint64_t a = g.arc((uint32_t)lap::below(lap::philox_r64(0u, 0u, i, 2u, key0, key1), (uint64_t)p.g.arcs));
                        u = g.target(a);
                        g.next_row(a, u, off, deg);
                    }
                    if (!p.paths) r = lap::philox_r64(1u, 0u, i, 1u + kind, key0, key1);
                }
            }
        }
        if (!__any_sync(kFull, active)) break;
        if (!active) continue;
        if (u == v) {
            if (kind) {
                acc2 += t;
                if (p.y2_out) {
                    p.y2_out[q] = t;
                    if (CV && p.m2_out) p.m2_out[q] = m2;
                }
            }
            active = false;
        } else {
            if (++t > p.step_limit) {
                // The launch's results are void: leave the remaining walks.
                bad = LAP_DEV_STEP_LIMIT;
                active = false;
                open = false;
            }
            uint64_t x = r;
            if (p.paths) {
                const unsigned long long c = pw[u];
                const uint32_t j = (c ^ tag) >> 32 ? 0u : (uint32_t)c;
                x = lap::philox_r64(u, j, i, 0u, key0, key1);
                pw[u] = tag | (j + 1u);
            }
            const uint64_t a = g.arc(off + below32(x, deg));
            if (kind == 0) atomicAdd(&p.cnt2[u], 1ull);
            if (!p.paths) r = lap::philox_r64((uint32_t)t + 1u, 0u, i, 1u + kind, key0, key1);
            const uint32_t w = g.target(a);
            if (CV && kind && p.cv_h2) {
                const long long d = (long long)deg, hw = ld_pot(p.cv_h2 + w), s2 = ld_pot(p.cv_S2 + u);
                atomicAdd(&p.cv_a2[u], (unsigned long long)hw);
                atomicAdd(&p.cv_p2[u], 1ull);
                m2 = __dadd_rn(m2, __ddiv_rn((double)(d * hw - s2), (double)d));
            }
            u = w;
            g.next_row(a, w, off, deg);
        }
    }
    if (acc2) atomicAdd(&p.acc->sum_y2, acc2);
    if (bad) atomicOr(&p.acc->status, bad);
}

}  // namespace lap_walks
