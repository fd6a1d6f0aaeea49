// Units of work shared by groups of resident blocks: scorers that need a statistic over all keys of a unit before they can score
// any of them, in one launch.
//
// A unit is one (layer, sequence, KV head).  The blocks of a cooperative launch (one per SM, all resident) are split into
// groups; each group takes a unit at a time, each block a share of its pages.  A block works on "pass 1 of unit n, pass 2
// of unit n - 1" in turn: while the blocks exchange the statistics of a unit they read the next one, and the second pass
// finds its keys in L2, or what it needs of them in shared memory.  The groups are made as wide as it takes for their
// units together to hold a window of so many bytes: small enough to be still there, large enough to hide the exchange.
// Measured without the exchange, one head of 32768 tokens per group, 8.6 GB of K: read once 1.24 ms; twice with 17 / 25 / 34 / 42
// MB of units 1.33 / 1.35 / 1.38 / 1.50 ms with the second read marked evict-first, 1.33 / 1.58 / 2.00 / 2.34 ms without.
#pragma once
#include "ams_common.cuh"
#include "ams_tc_ptx.cuh"
#include "ams_tc_tiles.cuh"

namespace ams {

struct Groups {
    int g, n;    // blocks per group, groups
    int id, me;  // this block's group (>= n: none) and its place in it
    unsigned from, to; // the block's share of a unit's pages, in 2^-32
    bool all;          // every sequence has something to evict
    int T;             // length of the lane's sequence, of the first 32
    int dh, db, dl;    // n as a number of heads, sequences with something to evict and layers: the step from a unit of the group to
                       // the next
};

// The split for the lengths of this call; the same in every block, computed by each warp for itself.  most_pages: of a unit that
// a block can hold.
__device__ __forceinline__ Groups split_groups(const DevParams &p, int warps, float window, int most_pages)
{
    const int lane = threadIdx.x & 31, nb = gridDim.x;
    int longest = 0, active = 0;
    float total = 0.0f;
    Groups r;
    r.T = 0;
    for (int b = lane; b < p.B; b += 32) {
        const int T = p.seq_lens[b];
        if (b == lane) r.T = T;
        if (T > p.Tk && T <= p.T_cap) { longest = max(longest, T); total += (float)T; ++active; }
    }
    longest = __reduce_max_sync(0xffffffffu, longest);
    active = __reduce_add_sync(0xffffffffu, active);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    const int units = active * p.L * p.H, pages = (longest + kPage - 1) / kPage;
    r.g = 1; r.n = 0; r.id = 1; r.me = 0;
    if (units <= 0) return r;
    const float fit = window * (float)active / (total * kRowBytes); // units in the window, of the average size
    // two groups at least, so that one reads while the other waits (K of 80000 tokens, 32 units: 222 -> 132 us; of 131072,
    // where two units no longer fit L2: 388 -> 324 us); no group without work; no fewer units in the last round than need be
    int n = min(min(nb, units), (int)fmaxf(2.0f, fit));
    n = (units + (units + n - 1) / n - 1) / ((units + n - 1) / n);
    n = max(1, min(n, nb / ((pages + most_pages - 2) / (most_pages - 1)))); // no share above what a block can hold (its ends are rounded)
    int g = min(nb / n, (pages + warps - 1) / warps); // no warp without a page
    if (p.group_size) g = p.group_size;
    r.g = g;
    r.n = min(nb / g, units);
    r.id = blockIdx.x / g;
    r.me = blockIdx.x % g;
    const unsigned share = g > 1 ? 0xffffffffu / g + 1 : 0u;
    r.from = r.me * share;
    r.to = r.from + share; // (the last block takes what is left)
    r.all = active == p.B;
    r.dh = r.n % p.H;
    r.db = (r.n / p.H) % active;
    r.dl = r.n / (p.H * active);
    return r;
}

// The walk over a group's units, each with the block's share of their pages.  Only what has something to evict is dealt out: in
// the numbers of all sequences, a stride of whole sequences can miss the active ones for half of the groups (32 layers of 16
// sequences of 6400 tokens, every other one within the budget, key scores: 1236 us, now 650, as for the eight alone).  The
// lengths of 32 sequences stay in the warp's registers: the exchange's acquiring loads empty L1, and a trip to L2 per unit shows
// (the eight alone 660 us, with two trips 676).  Called by whole warps.
struct GroupWalk {
    int l, b, h;   // the next unit; l >= L: none
    int base, T;   // first of the sequences at hand, the length of the lane's
    unsigned live; // which of them have something to evict
};
struct GroupUnit {
    int l, b, h, T, first, pages;
};
__device__ __forceinline__ void walk_lengths(const DevParams &p, const Groups &gr, GroupWalk &w, int base)
{
    const int b = base + (threadIdx.x & 31);
    w.base = base;
    w.T = base == 0 ? gr.T : b < p.B ? p.seq_lens[b] : 0;
    w.live = __ballot_sync(0xffffffffu, w.T > p.Tk && w.T <= p.T_cap);
}
// `count` sequences with something to evict further on, round the batch into the next layers
__device__ __forceinline__ void walk_sequences(const DevParams &p, const Groups &gr, GroupWalk &w, int count)
{
    if (gr.all) {
        for (w.b += count; w.b >= p.B; w.b -= p.B) ++w.l;
        const int base = w.b & ~31;
        if (base != w.base && w.l < p.L) walk_lengths(p, gr, w, base);
        return;
    }
    if (count <= 0 || w.l >= p.L) return;
    unsigned rest = w.b < w.base ? w.live : w.live & ~((2u << (w.b - w.base)) - 1u); // those after b
    for (int found; (found = __popc(rest)) < count;) {
        count -= found;
        int base = w.base + 32;
        if (base >= p.B) {
            base = 0;
            if (++w.l >= p.L) return;
        }
        if (base != w.base) walk_lengths(p, gr, w, base);
        rest = w.live;
    }
    const int lane = threadIdx.x & 31;
    w.b = w.base - 1 + __ffs(__ballot_sync(0xffffffffu, (rest >> lane & 1u) && __popc(rest & ((1u << lane) - 1u)) == count - 1));
}
__device__ __forceinline__ GroupWalk group_walk(const DevParams &p, const Groups &gr)
{
    GroupWalk w;
    w.l = 0; w.b = -1; w.h = gr.id % p.H;
    walk_lengths(p, gr, w, 0);
    walk_sequences(p, gr, w, gr.id / p.H + 1);
    return w;
}
__device__ __forceinline__ bool next_group_unit(const DevParams &p, const Groups &gr, GroupWalk &w, GroupUnit &u)
{
    if (w.l >= p.L) return false;
    u.l = w.l; u.b = w.b; u.h = w.h;
    u.T = __shfl_sync(0xffffffffu, w.T, w.b - w.base);
    const int pages = (u.T + kPage - 1) / kPage;
    u.first = (int)__umulhi((unsigned)pages, gr.from);
    u.pages = (gr.me == gr.g - 1 ? pages : (int)__umulhi((unsigned)pages, gr.to)) - u.first;
    w.h += gr.dh;
    w.l += gr.dl;
    const bool carry = w.h >= p.H;
    if (carry) w.h -= p.H;
    walk_sequences(p, gr, w, gr.db + (carry ? 1 : 0));
    return true;
}

// Exchange of a block's statistics with its group: slots of data, and a counter of the blocks that have filled theirs.  Four of
// each in turn: a block publishes unit n + 4 only after its pass 2 of unit n + 2, which waited until every block of the group
// had published unit n + 2 and so was through with unit n.  The counters only grow during a launch (the first kernel of the event
// clears them).  A warp waits for one word: a flag per block, or tags in the data themselves, cost more than the
// counter's extra trips, because a warp's acquiring loads of many words are not pipelined (2048 units of 32768 tokens in
// groups of 49 blocks: 3.47 ms with the counter, 5.84 with flags, 6.05 with tags).
constexpr int kGroupCollectors = 2; // warps that read a group's slots
template <typename T>
__device__ __forceinline__ T *group_slot(const DevParams &p, const Groups &gr, int member, int n)
{
    return reinterpret_cast<T *>(p.group_part + (size_t)((n & 3) * kGroupBlocks + gr.id * gr.g + member) * kGroupSlot);
}
__device__ __forceinline__ int *group_counter(const DevParams &p, const Groups &gr, int n) { return p.group_count + (gr.id * 4 + (n & 3)) * kGroupCounterPad; }
// after the warp's stores to the block's slot
__device__ __forceinline__ void group_publish(const DevParams &p, const Groups &gr, int n)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(group_counter(p, gr, n)) : "memory");
}
// before a warp's reads of the group's slots; false when the wait ran out or another role gave up.  All lanes load the one word, a
// single request: each has then acquired what it reads next.  (One lane for all needs a __syncwarp to pass its acquire on and is
// slower: 1792 units of 8192 to 32768 tokens at 16 rows, event 3531 us, this 3499; 2048 units of 6400 tokens, key scores, 1124 and 1109.)
__device__ __forceinline__ bool group_await(const DevParams &p, const Groups &gr, int n, volatile int *abort_flag)
{
    const int *counter = group_counter(p, gr, n);
    const int want = (n / 4 + 1) * gr.g + (p.expire_polls ? 1 : 0), limit = p.expire_polls ? (int)p.expire_polls : 1 << 21;
    for (int i = 0;; ++i) {
        int have;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(have) : "l"(counter) : "memory");
        if (__all_sync(0xffffffffu, have >= want)) return true;
        if (i == limit) *abort_flag = 1;
        if ((i & 255) == 255 && __any_sync(0xffffffffu, *abort_flag)) return false;
    }
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
// ------------------------------------------------------------------ the stream of pages
// kFeeders warps feed pages of 16 tokens by TMA to kWarps streaming warps, in turn and on across the ends of passes and
// units, into a ring of kRing pages per warp.  Page number q of this walk (pass 1 of unit 0, pass 1 of unit 1, pass 2 of unit
// 0, pass 1 of unit 2, ...) goes to streaming warp q % kWarps.
constexpr int kPageBytes = kPage * kRowBytes;
constexpr int kFeeders = 2;
constexpr uint32_t kFeedLimit = 1u << 25;
constexpr int kHeldIds = 128; // page ids of a unit that are fetched a unit ahead

// A unit as the streaming warps need it
struct GroupShare {
    float *scores;     // of the block's first page
    int tokens, pages; // of the sequence from there on; of the block's share, < 0: no more units
};

template <int kWarps, int kRing, int kUnits> // kUnits: units whose description is held
struct GroupPipe {
    unsigned char ring[kWarps * kRing * kPageBytes];              // first: aligned to 1024 bytes with the whole
    GroupShare unit[kUnits];
    int ids[kFeeders][2][kHeldIds];                               // page ids of a feeder's unit and the one before
    unsigned long long full[kWarps * kRing], empty[kWarps * kRing]; // page is there; page is used
    unsigned long long unit_full[kUnits], unit_empty[kUnits];       // unit is known; unit is done
    unsigned long long summed[2], ready[2];                         // statistics of the warps are there; of the group
    int abort_flag;
};

template <int kWarps, int kRing, int kUnits>
__device__ __forceinline__ void pipe_init(GroupPipe<kWarps, kRing, kUnits> &pipe)
{
    static_assert(kWarps * kRing <= 64, "a thread per barrier");
    const int i = threadIdx.x;
    if (i < kWarps * kRing) { tc::mbar_init(tc::smem_u32(&pipe.full[i]), 1); tc::mbar_init(tc::smem_u32(&pipe.empty[i]), 1); }
    if (i < kUnits) { tc::mbar_init(tc::smem_u32(&pipe.unit_full[i]), 1); tc::mbar_init(tc::smem_u32(&pipe.unit_empty[i]), kWarps); }
    if (i < 2) { tc::mbar_init(tc::smem_u32(&pipe.summed[i]), kWarps); tc::mbar_init(tc::smem_u32(&pipe.ready[i]), 1); }
    if (i == 0) pipe.abort_flag = 0;
    if (i < 64) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
}

// bounded, the same result in all lanes
__device__ __forceinline__ bool warp_wait(const unsigned long long *bar, uint32_t parity, volatile int *abort_flag)
{
    return __all_sync(0xffffffffu, tc::mbar_wait(tc::smem_u32(bar), parity, abort_flag));
}

// A feeder warp.  announce(n, u) is called by one lane with each unit's description in place and completes unit_full[n % kUnits]'s
// arrival.  A lane feeds one streaming warp throughout, so that the places of a ring are filled in turn by the same lane
// and no wait for a place can be a round of the ring off.  False after a wait that ran out, with the copies on their
// way landed.
template <int kPasses, int kWarps, int kRing, int kUnits, typename Announce>
__device__ __forceinline__ bool feed_pages(const DevParams &p, const Groups &gr, const CUtensorMap &k_map, GroupPipe<kWarps, kRing, kUnits> &pipe,
                                           int feeder, Announce announce)
{
    constexpr int kShare = kWarps / kFeeders, kSlots = kWarps * kRing;
    static_assert(kWarps % kFeeders == 0 && kShare <= 32, "a lane per streaming warp");
    const int lane = threadIdx.x & 31;
    const unsigned long long keep = l2_keep(), done = l2_done();
    const uint32_t ring = tc::smem_u32(pipe.ring), full = tc::smem_u32(pipe.full), empty = tc::smem_u32(pipe.empty);
    volatile int *abort_flag = &pipe.abort_flag;
    const bool feeds = lane < kShare;
    const int fed = feeder * kShare + (feeds ? lane : 0);
    GroupWalk walk = group_walk(p, gr);
    GroupUnit cur, old, nxt;
    cur.pages = old.pages = 0;
    unsigned at = 0; // walk number of the pass's first page
    int sent = 0;    // copies that this lane has started: all the pages of its streaming warp, in turn
    bool ok = true;
    // page ids come a unit ahead, so that no copy waits for one
    int ahead[kHeldIds / 32] = {};
    auto fetch_ids = [&]() {
#pragma unroll
        for (int i = 0; i < kHeldIds / 32; ++i)
            ahead[i] = lane + 32 * i < nxt.pages ? p.block_table[(size_t)nxt.b * p.bt_stride + nxt.first + lane + 32 * i] : 0;
    };
    bool more = next_group_unit(p, gr, walk, nxt);
    if (more) fetch_ids();
    int announced = 0;
    for (int n = 0, last = 0; !last && ok; ++n) {
        last = !more;
        cur = nxt;
        if (last) cur.pages = 0;
#pragma unroll
        for (int i = 0; i < kHeldIds / 32; ++i) pipe.ids[feeder][n & 1][lane + 32 * i] = ahead[i];
        __syncwarp();
        if (more) more = next_group_unit(p, gr, walk, nxt);
        if (more) fetch_ids();
        if (feeder == 0) {
            ok = warp_wait(&pipe.unit_empty[n % kUnits], (uint32_t)(((n / kUnits) & 1) ^ 1), abort_flag);
            if (!ok) break;
            if (lane == 0) {
                GroupShare &u = pipe.unit[n % kUnits];
                u.pages = last ? -1 : cur.pages;
                u.tokens = last ? 0 : cur.T - cur.first * kPage;
                u.scores = !last ? p.scores + (size_t)((cur.l * p.B + cur.b) * p.H + cur.h) * p.T_cap + (size_t)cur.first * kPage : nullptr;
                if (!last) announce(n, cur);
                else tc::mbar_arrive(tc::smem_u32(&pipe.unit_full[n % kUnits]));
            }
            ++announced;
            __syncwarp();
        }
#pragma unroll 1
        for (int pass = 0; pass < kPasses && ok; ++pass) {
            const GroupUnit u = pass ? old : cur;
            const int *ids = pipe.ids[feeder][(n - pass) & 1];
            const int layer = u.l * (int)p.num_pages;
            for (int k0 = -(int)(at % kWarps); k0 < u.pages && ok; k0 += kWarps) {
                const int k = k0 + fed;
                const bool mine = feeds && k >= 0 && k < u.pages;
                const int page = layer + (!mine ? 0 : k < kHeldIds ? ids[k] : p.block_table[(size_t)u.b * p.bt_stride + u.first + k]);
                const unsigned q = at + k;
                const int s = (int)(q % kSlots);
                bool todo = mine;
                for (uint32_t i = 0; ok; ++i) { // each page goes out as soon as its place is free
                    if (todo && tc::mbar_test_wait(empty + 8 * s, ((q / kSlots) & 1) ^ 1)) {
                        tc::mbar_expect_tx(full + 8 * s, kPageBytes);
                        tc::tma_load_5d_policy(ring + s * kPageBytes, &k_map, full + 8 * s, 0, 0, 2 * u.h, 0, page, pass == kPasses - 1 ? done : keep);
                        todo = false;
                        ++sent;
                    }
                    if (!__any_sync(0xffffffffu, todo)) break;
                    if (i == kFeedLimit) *abort_flag = 1;
                    if ((i & 1023u) == 1023u) ok = __all_sync(0xffffffffu, !*abort_flag);
                }
            }
            at += u.pages;
        }
        old = cur;
    }
    if (!ok) {
        for (int u = max(0, announced - kUnits); u < announced; ++u) // (a unit's description may come with a copy)
            for (int i = 0; i < (1 << 16) && !tc::mbar_try_wait(tc::smem_u32(&pipe.unit_full[u % kUnits]), (u / kUnits) & 1); ++i) {}
        for (int k = max(0, sent - kRing); k < sent; ++k) // (by what was started: a wait for a turn that was not would pass at once)
            for (int i = 0; i < (1 << 16) && !tc::mbar_try_wait(full + 8 * (k % kRing * kWarps + fed), (k / kRing) & 1); ++i) {}
    }
    return ok;
}

// A streaming warp's place in the stream.
template <int kWarps, int kRing, int kUnits>
struct PipeReader {
    GroupPipe<kWarps, kRing, kUnits> &pipe;
    int warp, slot, turn; // place in the ring; pages from the start of the pass until the warp's next one
    uint32_t phase;
    __device__ __forceinline__ PipeReader(GroupPipe<kWarps, kRing, kUnits> &pipe_, int warp_) : pipe(pipe_), warp(warp_), slot(0), turn(warp_), phase(0) {}
    __device__ __forceinline__ bool wait() { return warp_wait(&pipe.full[slot * kWarps + warp], phase, &pipe.abort_flag); }
    // Matrix loads of the page: chunk pair s (dimensions 16 s .. 16 s + 15), each lane from token 8 rows8 + lane % 8 and chunk 2 s + odd
    // at chunk(at(rows8, odd), s).  Tokens in eights lie at 2048, halves of a row at 1024, a 16-byte chunk of a half at its
    // number XOR the token, which leaves the loads free of bank conflicts (rows are 128 bytes, so the XOR can be taken of the address).
    __device__ __forceinline__ uint32_t at(int rows8, int odd) const
    {
        const int r = threadIdx.x & 7;
        return tc::smem_u32(pipe.ring) + (slot * kWarps + warp) * kPageBytes + (rows8 * 2048 + r * 128 + ((odd ^ r) << 4));
    }
    static __device__ __forceinline__ uint32_t chunk(uint32_t at, int s) { return (at ^ ((s & 3) << 5)) + (s >> 2) * 1024; }
    __device__ __forceinline__ void release()
    {
        __syncwarp();
        if ((threadIdx.x & 31) == 0) tc::mbar_arrive(tc::smem_u32(&pipe.empty[slot * kWarps + warp]));
        if (++slot == kRing) { slot = 0; phase ^= 1; }
    }
};

__device__ __forceinline__ void ldsm4(unsigned (&r)[4], unsigned addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4_trans(unsigned (&r)[4], unsigned addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}

// Cooperative launch, one block per SM (fewer, but not below `least`, the blocks that can hold a unit, where the context does not have
// all of the device's SMs).
template <typename... Maps>
inline cudaError_t launch_groups(void (*kernel)(DevParams, Maps...), int least, int threads, size_t smem, cudaStream_t s, DevParams p, Maps... maps)
{
    const long long units = (long long)p.L * p.B * p.H;
    // The blocks of a cluster are resident together as well, and unlike a cooperative launch one of clusters comes in behind the kernel
    // before it: few short units take a cluster each (one layer of 4096 tokens, event: 43.3 -> 41.1 us; 32 units of 4096 tokens at 32
    // rows 66.6 -> 63.5).  16 units in clusters of eight no longer fit at once (56 -> 63 us).
    const int cluster = units <= 8 && p.T_cap <= 8192 ? 8 : units <= 32 && p.T_cap <= 4096 ? 4 : 0;
    if (cluster && least <= cluster) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(units * cluster));
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cluster; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        p.group_size = cluster;
        if (cudaLaunchKernelEx(&cfg, kernel, p, maps...) == cudaSuccess) return cudaSuccess;
        (void)cudaGetLastError();
        p.group_size = 0;
    }
    int blocks = sm_count() < kGroupBlocks ? sm_count() : kGroupBlocks;
    for (;; blocks = (blocks + 1) / 2) {
        if (blocks < least || blocks < 1) return cudaErrorCooperativeLaunchTooLarge;
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
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, p, maps...);
        if (e != cudaErrorCooperativeLaunchTooLarge || blocks == 1) return e;
        (void)cudaGetLastError();
    }
}

} // namespace ams
