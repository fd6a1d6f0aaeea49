// Units of work shared by groups of resident blocks: the two-pass scorers that read K twice in one launch.
//
// A unit is one (layer, sequence, KV head).  Its scores need a statistic of all of its keys first, so K is read twice.
// The blocks of a cooperative launch (one per SM, all resident) are split into groups; each group takes a unit at a
// time, each block a share of its pages.  A block works on "pass 1 of unit n, pass 2 of unit n - 1" in turn: while the blocks
// exchange the statistics of a unit they read the next one, and the second pass finds its keys in L2.  The groups are made as
// wide as that takes: their units together hold kGroupWindow bytes.  Measured without the exchange, one head of 32768
// tokens per group, 8.6 GB of K: read once 1.24 ms; twice with 17 / 25 / 34 / 42 MB of units 1.33 / 1.35 / 1.38 / 1.50 ms
// with the second read marked evict-first, 1.33 / 1.58 / 2.00 / 2.34 ms without the mark.  With the exchange, key scores of
// 512 units of 4096 tokens at a window of 26 / 34 / 42 / 50 / 64 MB: 131 / 136 / 148 / 149 / 175 us.
#pragma once
#include "ams_common.cuh"

namespace ams {

constexpr long long kGroupWindow = 26ll << 20;

struct Groups {
    int g, n;    // blocks per group, groups
    int id, me;  // this block's group (>= n: none) and its place in it
    unsigned from, to; // the block's share of a unit's pages, in 2^-32
    int dh, db, dl;    // n as a number of heads, sequences and layers: the step from a unit of the group to the next
};

// The split for the lengths of this call; the same in every block, computed by each warp for itself.
__device__ __forceinline__ Groups split_groups(const DevParams &p, int warps)
{
    const int lane = threadIdx.x & 31, nb = gridDim.x;
    int longest = 0, active = 0;
    for (int b = lane; b < p.B; b += 32) {
        const int T = p.seq_lens[b];
        if (T > p.Tk && T <= p.T_cap) { longest = max(longest, T); ++active; }
    }
    longest = __reduce_max_sync(0xffffffffu, longest);
    active = __reduce_add_sync(0xffffffffu, active);
    const int units = active * p.L * p.H, pages = (longest + kPage - 1) / kPage;
    Groups r;
    r.g = 1; r.n = 0; r.id = 1; r.me = 0;
    if (units <= 0) return r;
    const long long bytes = (long long)pages * kPage * kRowBytes;
    // two groups at least, so that one reads while the other waits (K of 80000 tokens, 32 units: 222 -> 132 us; of 131072,
    // where two units no longer fit L2: 388 -> 324 us); no group without work; no fewer units in the last round than need be
    int n = min(min(nb, units), (int)max(2ll, kGroupWindow / bytes));
    n = (units + (units + n - 1) / n - 1) / ((units + n - 1) / n);
    const int g = min(nb / n, (pages + warps - 1) / warps); // no warp without a page
    r.g = g;
    r.n = min(nb / g, units);
    r.id = blockIdx.x / g;
    r.me = blockIdx.x % g;
    r.from = (unsigned)(((unsigned long long)r.me << 32) / g);
    r.to = (unsigned)(((unsigned long long)(r.me + 1) << 32) / g); // (0 for the last block: wraps)
    r.dh = r.n % p.H;
    r.db = (r.n / p.H) % p.B;
    r.dl = r.n / (p.H * p.B);
    return r;
}

// The walk over a group's units: one after the other those that have something to evict, and the block's share of their
// pages.
struct GroupWalk {
    int l, b, h;
};
struct GroupUnit {
    int l, b, h, T, first, pages;
};
__device__ __forceinline__ GroupWalk group_walk(const DevParams &p, const Groups &gr)
{
    return GroupWalk{gr.id / (p.H * p.B), (gr.id / p.H) % p.B, gr.id % p.H};
}
__device__ __forceinline__ bool next_group_unit(const DevParams &p, const Groups &gr, GroupWalk &w, GroupUnit &u)
{
    while (w.l < p.L) {
        u.l = w.l; u.b = w.b; u.h = w.h;
        u.T = p.seq_lens[w.b];
        w.h += gr.dh;
        w.b += gr.db;
        w.l += gr.dl;
        if (w.h >= p.H) { w.h -= p.H; ++w.b; }
        if (w.b >= p.B) { w.b -= p.B; ++w.l; }
        if (u.T <= p.Tk || u.T > p.T_cap) continue;
        const int pages = (u.T + kPage - 1) / kPage;
        u.first = (int)__umulhi((unsigned)pages, gr.from);
        u.pages = (gr.me == gr.g - 1 ? pages : (int)__umulhi((unsigned)pages, gr.to)) - u.first;
        return true;
    }
    return false;
}

// Exchange of a block's statistics with its group.  Four slots in turn: a block publishes unit n + 4 only after its
// pass 2 of unit n + 2, which waited until every block of the group had published unit n + 2 and so was through with unit n.
// The counters only grow during a launch (the first kernel of the event clears them).
__device__ __forceinline__ int *group_counter(const DevParams &p, const Groups &gr, int n) { return p.group_count + (gr.id * 4 + (n & 3)) * 8; }
__device__ __forceinline__ float *group_slot(const DevParams &p, const Groups &gr, int member, int n)
{
    return p.group_part + (size_t)((gr.id * gr.g + member) * 4 + (n & 3)) * kGroupSlot;
}
// one lane, after the warp's stores to the slot and a __syncwarp
__device__ __forceinline__ void group_publish(int *counter)
{
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(counter) : "memory");
}
// one lane, before the warp's reads of the group's slots; false when the wait ran out or another role gave up
__device__ __forceinline__ bool group_wait(const int *counter, int want, volatile int *abort_flag)
{
    for (int i = 0; i < (1 << 21); ++i) {
        int have;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(have) : "l"(counter) : "memory");
        if (have >= want) return true;
        if ((i & 255) == 255 && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
// barrier over the first `threads` that arrive at it: true if `ok` holds in all
__device__ __forceinline__ bool named_barrier_all(int id, int threads, bool ok)
{
    int r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, %2, %3, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
                 : "=r"(r) : "r"(ok ? 1 : 0), "r"(id), "r"(threads) : "memory");
    return r != 0;
}

// L2 policies of the two passes
__device__ __forceinline__ unsigned long long l2_keep()
{
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ unsigned long long l2_done()
{
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
// Cooperative launch, one block per SM (fewer where the context does not have all of the device's SMs).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_groups(void (*kernel)(KArgs...), int blocks, int threads, size_t smem, cudaStream_t s, Args... args)
{
    for (;; blocks /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)blocks);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
        if (e != cudaErrorCooperativeLaunchTooLarge || blocks == 1) return e;
        (void)cudaGetLastError();
    }
}

} // namespace ams
