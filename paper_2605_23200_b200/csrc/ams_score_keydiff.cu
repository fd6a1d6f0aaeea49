// KeyDiff-style score: negative cosine similarity of each key to the mean key of its (sequence, KV head) cache.
//
// One cooperative launch over groups of blocks (ams_groups.cuh).  Pass 1 sums a unit's keys, pass 2 scores them, both on the
// tensor cores.  Two warps feed pages of 16 tokens by TMA to sixteen streaming warps, in turn and on across the ends
// of passes and units, into a ring of three pages per warp; two more warps exchange the sums, so that no streaming
// warp waits for another block unless that one is more than a unit's read behind.  Bound by the K stream, read once from HBM
// and once from L2, and by the spread of the blocks of a group at each exchange: 17.2 GB of K (2048 units of 32768
// tokens) 5.72 ms with one kernel per pass and both reads from HBM, now 3.47 ms (5.0 TB/s of HBM, 9.9 TB/s of L2); 256 units of 3000
// tokens 101 -> 68 us.  One warp to feed them all 4.07 ms (its copies go out one by one); thread-issued 16-byte copies, each
// warp for itself, 4.02 ms (half of the instructions were addresses).  Every wait is bounded; on
// expiry the block reports AMS_ERR_TIMEOUT, drains its copies and returns.
#include "ams_common.cuh"
#include "ams_groups.cuh"
#include "ams_tc_ptx.cuh"
#include "ams_tc_tiles.cuh"

namespace ams {

namespace {

using namespace tc;

constexpr int kKdWarps = 16;    // streaming warps
constexpr int kKdFeeders = 2, kKdCollectors = 2;
constexpr int kKdThreads = (kKdWarps + kKdFeeders + kKdCollectors) * 32;
constexpr int kKdRing = 3;      // pages per streaming warp in shared memory
constexpr int kKdSlots = kKdWarps * kKdRing;
constexpr int kKdTile = kPage * kRowBytes;
constexpr uint32_t kFeedLimit = 1u << 25;
constexpr int kKdUnits = 4;     // units the feeder may be ahead

// A unit as the streaming warps need it
struct KdUnit {
    float *scores;              // of the block's first page
    int tokens, pages;          // of the block's share; pages < 0: no more units
};

struct KdShared {
    unsigned char ring[kKdSlots * kKdTile];
    float sum[2][kKdWarps][kHeadDim];        // the warps' sums of a unit's keys
    float4 part[2][kKdCollectors][32];       // the collectors' shares of the group's sum
    __nv_bfloat16 mean[2][3][kHeadDim + 8];  // the mean key as a sum of three bf16 vectors
    float norm[2];
    KdUnit unit[kKdUnits];
    unsigned long long full[kKdSlots], empty[kKdSlots];           // page is there; page is used
    unsigned long long unit_full[kKdUnits], unit_empty[kKdUnits]; // unit is known; unit is done
    unsigned long long summed[2], ready[2];                       // sums of the warps are there; mean is there
    int abort_flag;
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
// both, the first or none of two neighbouring bf16 values
__device__ __forceinline__ unsigned tokens_mask(int n) { return n >= 2 ? 0xffffffffu : n == 1 ? 0xffffu : 0u; }

// all lanes or none
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag));
}

__global__ void __launch_bounds__(kKdThreads, 1) k_keydiff(DevParams p, const __grid_constant__ CUtensorMap k_map)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    KdShared &sh = *reinterpret_cast<KdShared *>(smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gq = lane >> 2, tq = lane & 3;
    const uint32_t full = smem_u32(sh.full), empty = smem_u32(sh.empty), unit_full = smem_u32(sh.unit_full), unit_empty = smem_u32(sh.unit_empty);
    const uint32_t summed = smem_u32(sh.summed), ready = smem_u32(sh.ready);
    volatile int *abort_flag = &sh.abort_flag;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kKdSlots; ++i) { mbar_init(full + 8 * i, 1); mbar_init(empty + 8 * i, 1); }
        for (int i = 0; i < kKdUnits; ++i) { mbar_init(unit_full + 8 * i, 1); mbar_init(unit_empty + 8 * i, kKdWarps); }
        for (int i = 0; i < 2; ++i) { mbar_init(summed + 8 * i, kKdWarps); mbar_init(ready + 8 * i, 1); }
        sh.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const Groups gr = split_groups(p, kKdWarps);
    if (gr.id >= gr.n) return;
    bool ok = true;
    if (warp < kKdWarps) {
        const uint32_t ring = smem_u32(sh.ring) + warp * kKdTile;
        int slot = 0, turn = warp; // the warp's place in its ring; pages until its next one
        uint32_t phase = 0;
        // rows of eight tokens lie at 2048, halves of a row at 1024, a 16-byte chunk of a half at its number XOR the row
        auto load = [&](auto ldsm, unsigned (&a)[8][4], int rows8, int chunk) {
            const uint32_t at = ring + slot * (kKdWarps * kKdTile) + rows8 * 2048 + (lane & 7) * 128;
#pragma unroll
            for (int s = 0; s < 8; ++s) ldsm(a[s], at + (s >> 2) * 1024 + (((2 * (s & 3) + chunk) ^ (lane & 7)) << 4));
        };
        auto release = [&]() {
            __syncwarp();
            if (lane == 0) mbar_arrive(empty + 8 * (slot * kKdWarps + warp));
            if (++slot == kKdRing) { slot = 0; phase ^= 1; }
        };
        KdUnit cur, old;
        old.pages = -1;
        for (int n = 0;; ++n) { // pass 1 of unit n, pass 2 of unit n - 1
            ok = warp_wait(unit_full + 8 * (n % kKdUnits), (uint32_t)((n / kKdUnits) & 1), abort_flag);
            if (!ok) break;
            cur = sh.unit[n % kKdUnits];
            if (cur.pages >= 0) {
                float acc[8][4]; // dimension 16 s + g: [s][0] and [s][1], dimension 16 s + 8 + g: [s][2] and [s][3]
#pragma unroll
                for (int s = 0; s < 8; ++s) acc[s][0] = acc[s][1] = acc[s][2] = acc[s][3] = 0.0f;
                int k = turn;
                for (; k < cur.pages; k += kKdWarps) {
                    ok = warp_wait(full + 8 * (slot * kKdWarps + warp), phase, abort_flag);
                    if (!ok) break;
                    // dimensions as rows, tokens as the contraction, against a matrix of ones
                    unsigned a[8][4];
                    load(ldsm4_trans, a, lane >> 4, (lane >> 3) & 1);
                    // the last page's rows past the end hold anything: they are taken as zeros
                    const int left = cur.tokens - k * kPage;
                    if (left < kPage) {
                        const unsigned m_lo = tokens_mask(left - 2 * tq), m_hi = tokens_mask(left - 2 * tq - 8);
#pragma unroll
                        for (int s = 0; s < 8; ++s) { a[s][0] &= m_lo; a[s][1] &= m_lo; a[s][2] &= m_hi; a[s][3] &= m_hi; }
                    }
#pragma unroll
                    for (int s = 0; s < 8; ++s) mma_bf16(acc[s], a[s][0], a[s][1], a[s][2], a[s][3], 0x3f803f80u, 0x3f803f80u);
                    release();
                }
                if (!ok) break;
                turn = k - cur.pages;
                // the four lanes of a row hold the same sums: each stores those of two steps
#pragma unroll
                for (int s = 0; s < 8; ++s)
                    if ((s >> 1) == tq) { sh.sum[n & 1][warp][16 * s + gq] = acc[s][0]; sh.sum[n & 1][warp][16 * s + 8 + gq] = acc[s][2]; }
                __syncwarp();
                if (lane == 0) mbar_arrive(summed + 8 * (n & 1));
            }
            if (n > 0) {
                const int m = n - 1;
                ok = warp_wait(ready + 8 * (m & 1), (uint32_t)((m >> 1) & 1), abort_flag);
                if (!ok) break;
                // column n of the second operand: part n of the mean (three), zeros beyond
                unsigned mu[8][2];
#pragma unroll
                for (int s = 0; s < 8; ++s)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        mu[s][i] = gq < 3 ? *reinterpret_cast<const unsigned *>(&sh.mean[m & 1][gq < 3 ? gq : 0][16 * s + 8 * i + 2 * tq]) : 0u;
                const float mu_norm = sh.norm[m & 1];
                int k = turn;
                for (; k < old.pages; k += kKdWarps) {
                    ok = warp_wait(full + 8 * (slot * kKdWarps + warp), phase, abort_flag);
                    if (!ok) break;
                    unsigned a[8][4];
                    load(ldsm4, a, (lane >> 3) & 1, lane >> 4);
                    float dot[4] = {0.0f, 0.0f, 0.0f, 0.0f}, lo[4] = {0.0f, 0.0f, 0.0f, 0.0f}, hi[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        // tokens as rows: k . mu, and k . k on the diagonals of the products with tokens 0-7 and 8-15,
                        // whose fragments are halves of the first operand's
                        mma_bf16(dot, a[s][0], a[s][1], a[s][2], a[s][3], mu[s][0], mu[s][1]);
                        mma_bf16(lo, a[s][0], a[s][1], a[s][2], a[s][3], a[s][0], a[s][2]);
                        mma_bf16(hi, a[s][0], a[s][1], a[s][2], a[s][3], a[s][1], a[s][3]);
                    }
                    release();
                    // lanes 0 and 1 of a row hold its products with the parts of the mean
                    float d0 = dot[0] + dot[1], d1 = dot[2] + dot[3];
                    d0 += __shfl_xor_sync(0xffffffffu, d0, 1);
                    d1 += __shfl_xor_sync(0xffffffffu, d1, 1);
                    d0 = __shfl_sync(0xffffffffu, d0, lane & ~3);
                    d1 = __shfl_sync(0xffffffffu, d1, lane & ~3);
                    // token g to lane g / 2 of its row, token g + 8 to that lane's neighbour
                    const float s0 = gq & 1 ? lo[1] : lo[0], s1 = __shfl_xor_sync(0xffffffffu, gq & 1 ? hi[3] : hi[2], 1);
                    const bool second = tq != gq >> 1;
                    const int t = k * kPage + gq + (second ? 8 : 0);
                    if ((tq ^ (gq >> 1)) < 2 && t < old.tokens) old.scores[t] = -(second ? d1 : d0) / fmaxf(sqrtf(second ? s1 : s0) * mu_norm, 1e-30f);
                }
                if (!ok) break;
                turn = k - old.pages;
                if (lane == 0) mbar_arrive(unit_empty + 8 * (m % kKdUnits));
            }
            if (cur.pages < 0) break;
            old = cur;
        }
    } else if (warp < kKdWarps + kKdFeeders) {
        // feeders: pages in the order pass 1 of unit 0, pass 1 of unit 1, pass 2 of unit 0, pass 1 of unit 2, ...; page number q of
        // this walk goes to streaming warp q % 16.  A lane feeds one streaming warp throughout, so that the places of a ring are
        // filled in turn by the same lane and no wait for a place can be a round of the ring off.
        const unsigned long long keep = l2_keep(), done = l2_done();
        const uint32_t ring = smem_u32(sh.ring);
        constexpr int kShare = kKdWarps / kKdFeeders;
        const bool feeds = lane < kShare;
        const int fed = (warp - kKdWarps) * kShare + (feeds ? lane : 0);
        GroupWalk walk = group_walk(p, gr);
        GroupUnit cur, old;
        cur.pages = old.pages = 0;
        unsigned at = 0; // walk number of the pass's first page
        bool more = true;
        auto page_id = [&](const GroupUnit &u, int k) {
            return feeds && k >= 0 && k < u.pages ? p.block_table[(size_t)u.b * p.bt_stride + u.first + k] : 0;
        };
        for (int n = 0; more && ok; ++n) {
            more = next_group_unit(p, gr, walk, cur);
            if (!more) cur.pages = 0;
            if (warp == kKdWarps) {
                ok = warp_wait(unit_empty + 8 * (n % kKdUnits), (uint32_t)(((n / kKdUnits) & 1) ^ 1), abort_flag);
                if (!ok) break;
                if (lane == 0) {
                    KdUnit &u = sh.unit[n % kKdUnits];
                    u.pages = more ? cur.pages : -1;
                    u.tokens = more ? cur.T - cur.first * kPage : 0;
                    u.scores = more ? p.scores + (size_t)((cur.l * p.B + cur.b) * p.H + cur.h) * p.T_cap + (size_t)cur.first * kPage : nullptr;
                    mbar_arrive(unit_full + 8 * (n % kKdUnits));
                }
                __syncwarp();
            }
            int id = page_id(cur, fed - (int)(at % kKdWarps));
            const int id_old = page_id(old, fed - (int)((at + cur.pages) % kKdWarps));
#pragma unroll 1
            for (int pass = 0; pass < 2 && ok; ++pass) {
                const GroupUnit u = pass ? old : cur;
                if (pass) id = id_old;
                const int layer = u.l * (int)p.num_pages;
                for (int k0 = -(int)(at % kKdWarps); k0 < u.pages && ok; k0 += kKdWarps) {
                    const int k = k0 + fed, page = layer + id;
                    id = page_id(u, k + kKdWarps);
                    const unsigned q = at + k;
                    const int s = (int)(q % kKdSlots);
                    bool todo = feeds && k >= 0 && k < u.pages;
                    for (uint32_t i = 0; ok; ++i) { // each page goes out as soon as its place is free
                        if (todo && mbar_test_wait(empty + 8 * s, ((q / kKdSlots) & 1) ^ 1)) {
                            mbar_expect_tx(full + 8 * s, kKdTile);
                            tma_load_5d_policy(ring + s * kKdTile, &k_map, full + 8 * s, 0, 0, 2 * u.h, 0, page, pass ? done : keep);
                            todo = false;
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
        // after a wait that ran out: the copies on their way land before the block ends
        if (!ok)
            for (int s = lane; s < kKdSlots; s += 32) {
                // the last walk number of this place below `at` (its copy may not have been started: the wait is bounded)
                if (at <= (unsigned)s) continue;
                const unsigned turns = (at - 1 - s) / kKdSlots;
                for (int i = 0; i < (1 << 16) && !mbar_try_wait(full + 8 * s, turns & 1); ++i) {}
            }
    } else {
        // exchange: one warp publishes the block's sum of each unit, both collect the group's, in the blocks' order
        const int w = warp - kKdWarps - kKdFeeders;
        GroupWalk walk = group_walk(p, gr);
        GroupUnit u;
        for (int n = 0; next_group_unit(p, gr, walk, u); ++n) {
            if (w == 0) {
                ok = warp_wait(summed + 8 * (n & 1), (uint32_t)((n >> 1) & 1), abort_flag);
                if (ok) {
                    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                    for (int i = 0; i < kKdWarps; ++i) {
                        const float4 v = reinterpret_cast<const float4 *>(sh.sum[n & 1][i])[lane];
                        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
                    }
                    __stcg(reinterpret_cast<float4 *>(group_slot(p, gr, gr.me, n)) + lane, s);
                    __syncwarp();
                    if (lane == 0) group_publish(group_counter(p, gr, n));
                }
            }
            if (lane == 0) ok = ok && group_wait(group_counter(p, gr, n), (n / 4 + 1) * gr.g, abort_flag);
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (ok) {
                constexpr int kAhead = 16; // loads in flight
                const float4 *src = reinterpret_cast<const float4 *>(group_slot(p, gr, 0, n)) + lane;
                for (int i0 = w; i0 < gr.g; i0 += kAhead * kKdCollectors) {
                    float4 v[kAhead];
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) {
                        const int j = i0 + i * kKdCollectors;
                        v[i] = j < gr.g ? __ldcg(src + (size_t)j * (4 * kGroupSlot / 4)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    }
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) { s.x += v[i].x; s.y += v[i].y; s.z += v[i].z; s.w += v[i].w; }
                }
            }
            sh.part[n & 1][w][lane] = s;
            ok = named_barrier_all(1, kKdCollectors * 32, ok);
            if (!ok) break;
            if (w == 0) {
#pragma unroll
                for (int i = 1; i < kKdCollectors; ++i) {
                    const float4 v = sh.part[n & 1][i][lane];
                    s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
                }
                const float T = (float)u.T;
                s.x /= T; s.y /= T; s.z /= T; s.w /= T;
                float sq = (s.x * s.x + s.y * s.y) + (s.z * s.z + s.w * s.w);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float rest = v[i];
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        const __nv_bfloat16 x = __float2bfloat16_rn(rest);
                        sh.mean[n & 1][j][lane * 4 + i] = x;
                        rest -= __bfloat162float(x);
                    }
                }
                if (lane == 0) sh.norm[n & 1] = sqrtf(sq);
                __syncwarp();
                if (lane == 0) mbar_arrive(ready + 8 * (n & 1));
            }
        }
    }
    if (!ok && lane == 0) set_status(p.status, AMS_ERR_TIMEOUT, blockIdx.x, 4, 0);
}

} // namespace

int launch_score_keydiff(const DevParams &p, LaunchCtx &ctx)
{
    const EncodeTiledFn enc = encode_fn();
    if (!enc) return AMS_ERR_CUDA;
    CUtensorMap k_map;
    const int rc = make_k_map(p, enc, &k_map);
    if (rc != AMS_OK) return rc;
    static SmemGrant grant;
    const int n_sm = sm_count();
    if (n_sm <= 0 || !grant_dynamic_smem(k_keydiff, sizeof(KdShared), grant)) return AMS_ERR_CUDA;
    if (launch_groups(k_keydiff, n_sm < kGroupBlocks ? n_sm : kGroupBlocks, kKdThreads, sizeof(KdShared), ctx.s, p, k_map) != cudaSuccess) return AMS_ERR_CUDA;
    ctx.mark(kKernScore1);
    return AMS_OK;
}

} // namespace ams
