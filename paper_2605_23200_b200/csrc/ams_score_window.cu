// Window scorer for up to 32 query rows per KV head (see ams_score.cu for the definition), both phases in one cooperative launch
// over groups of blocks (ams_groups.cuh).  Pass 1 finds each row's (max, sum of exponentials) over a unit's keys, pass 2 sums
// the normalised probabilities over the rows.
//
// Up to 16 rows pass 1 leaves the logits in shared memory and pass 2 works on those; above, they would take too much of it to
// hide the exchange, and pass 2 recomputes them with K from L2.  Before, 7 rows over 9.4 GB of K (1792 units of 8192 to
// 32768 tokens) took 1.87 ms in three launches, with the logits through HBM, now 1.66 (5.7 TB/s, bound by the K stream and by
// the spread of a group's blocks at each exchange); 16 rows, 256 units of 3000 tokens, 76 -> 49 us; 32 rows over 2.9 GB, with K
// twice from HBM, 1.04 ms, now 0.77 (bound by the latency of a page in a warp: loads, eight dependent products, exponentials).
#include <float.h>

#include "ams_common.cuh"
#include "ams_groups.cuh"

namespace ams {

namespace {

using namespace tc;

// (m, z) <- merge of (m, z) and all of v, with one maximum
template <int N>
__device__ __forceinline__ void stat_merge_all(float &m, float &z, const float2 (&v)[N])
{
    float mx = m;
#pragma unroll
    for (int i = 0; i < N; ++i) mx = fmaxf(mx, v[i].x);
    if (mx == -INFINITY) return;
    z *= ex2((m - mx) * kLogitScale);
#pragma unroll
    for (int i = 0; i < N; ++i) z += v[i].y * ex2((v[i].x - mx) * kLogitScale);
    m = mx;
}

// Wide windows, up to 32 rows
struct WideTraits {
    static constexpr int rows = 32;
    static constexpr int mt = 2;              // M operands of 16 rows
    // the queries take 64 registers: 12 streaming warps of 128 registers, three pages each
    static constexpr int warps = 12, ring = 3, units = 3;
    static constexpr int threads = (warps + kFeeders + kGroupCollectors) * 32;
};
// 2048 units of 1900 to 9001 tokens at 26 / 34 / 42 MB: 773 / 738 / 767 us (with other code around it; 769 at 34 as it is)
constexpr float kWideWindow = 34.0f * (1 << 20);

struct WideShared {
    using T = WideTraits;
    GroupPipe<T::warps, T::ring, T::units> pipe;
    alignas(1024) unsigned char q[T::units][T::rows * kRowBytes]; // the units' query rows, halves of 128 bytes, swizzled
    float2 stat[2][T::warps][T::rows];                            // the warps' (max, sum)
    float2 part[2][32];                                           // the second collector's share of the group's
    float b[2][T::rows];                                          // the rows' references
    float pmax[2];                                                // largest probability of the window
};
static_assert(sizeof(WideShared) <= 227 * 1024, "shared memory of a block");

// One lane: the arrival of a unit's description, together with its query rows.
template <int RP>
__device__ __forceinline__ void feed_queries(const DevParams &p, const CUtensorMap &q_map, const GroupUnit &u, uint32_t dst, uint32_t bar)
{
    const int row = ((u.l * p.B + u.b) * p.H + u.h) * p.rows;
    mbar_expect_tx(bar, RP * kRowBytes);
    tma_load_2d(dst, &q_map, bar, 0, row);
    tma_load_2d(dst + RP * 128, &q_map, bar, 64, row);
}

// The exchange warps: one publishes the block's statistics of each unit, a row per lane, both collect the group's, in the blocks'
// order.
template <int RP, int kWarps, typename Shared>
__device__ __forceinline__ bool exchange_stats(const DevParams &p, const Groups &gr, Shared &sh, int w)
{
    const int lane = threadIdx.x & 31;
    volatile int *abort_flag = &sh.pipe.abort_flag;
    bool ok = true;
    GroupWalk walk = group_walk(p, gr);
    GroupUnit u;
    for (int n = 0; next_group_unit(p, gr, walk, u); ++n) {
        if (w == 0) {
            ok = warp_wait(&sh.pipe.summed[n & 1], (uint32_t)((n >> 1) & 1), abort_flag);
            if (ok) {
                if (lane < RP) {
                    float2 v[kWarps];
#pragma unroll
                    for (int i = 0; i < kWarps; ++i) v[i] = sh.stat[n & 1][i][lane];
                    float m = -INFINITY, z = 0.0f;
                    stat_merge_all(m, z, v);
                    __stcg(group_slot<float2>(p, gr, gr.me, n) + lane, make_float2(m, z));
                }
                group_publish(p, gr, n);
            }
        }
        float m = -INFINITY, z = 0.0f;
        ok = ok && group_await(p, gr, n, abort_flag);
        if (ok) {
            // a row per lane of each kSub-th of the warp, which takes every kSub-th block
            constexpr int kSub = 32 / RP, kAhead = 8;
            const float2 *src = group_slot<float2>(p, gr, 0, n) + lane % RP;
            for (int i0 = w + lane / RP * kGroupCollectors; i0 < gr.g; i0 += kAhead * kSub * kGroupCollectors) {
                float2 v[kAhead];
#pragma unroll
                for (int i = 0; i < kAhead; ++i) {
                    const int member = i0 + i * kSub * kGroupCollectors;
                    v[i] = member < gr.g ? __ldcg(src + (size_t)member * (kGroupSlot / 8)) : make_float2(-INFINITY, 0.0f);
                }
                stat_merge_all(m, z, v);
            }
        }
#pragma unroll
        for (int o = RP; o < 32; o <<= 1) {
            const float m2 = __shfl_xor_sync(0xffffffffu, m, o), z2 = __shfl_xor_sync(0xffffffffu, z, o);
            stat_merge(m, z, m2, z2);
        }
        if (w == 1) sh.part[n & 1][lane] = make_float2(m, z);
        ok = named_barrier_all(1, kGroupCollectors * 32, ok);
        if (!ok) break;
        if (w == 0) {
            const float2 v = sh.part[n & 1][lane];
            stat_merge(m, z, v.x, v.y);
            const bool live = lane < p.rows && z > 0.0f;
            float best = live ? 1.0f / z : 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
            if (lane < RP) set_reference(sh.b[n & 1][lane], live, m, z); // padding rows contribute nothing
            if (lane == 0) sh.pmax[n & 1] = best;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.pipe.ready[n & 1]));
        }
    }
    return ok;
}

__global__ void __launch_bounds__(WideTraits::threads, 1) k_window(DevParams p, const __grid_constant__ CUtensorMap k_map,
                                                                   const __grid_constant__ CUtensorMap q_map)
{
    using T = WideTraits;
    constexpr int MT = T::mt, E = 2, RP = T::rows, kWarps = T::warps;
    extern __shared__ __align__(1024) unsigned char smem[];
    WideShared &sh = *reinterpret_cast<WideShared *>(smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, tq = lane & 3;
    volatile int *abort_flag = &sh.pipe.abort_flag;
    if (threadIdx.x == 0) { tma_prefetch_map(&k_map); tma_prefetch_map(&q_map); }
    pipe_init(sh.pipe);
    wait_for_previous_kernel(); // effective lengths; the exchange's counters
    const Groups gr = split_groups(p, kWarps, kWideWindow, 1 << 20);
    if (gr.id >= gr.n) return;
    bool ok = true;
    if (warp < kWarps) {
        constexpr float c = kLogitScale;
        PipeReader<T::warps, T::ring, T::units> in(sh.pipe, warp);
        unsigned q[MT][8][4];
        auto load_queries = [&](int n) {
            const uint32_t at = smem_u32(sh.q[n % T::units]) + (lane & 7) * 128;
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    const int half = s >> 2, ch = 2 * (s & 3) + (lane >> 4);
                    ldsm4(q[mt][s], at + half * (RP * 128) + (mt * 16 + ((lane >> 3) & 1) * 8) * 128 + ((ch ^ (lane & 7)) << 4));
                }
            if (p.rows < RP) // the copy goes on into the next unit's rows: they are taken as zeros
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        if (mt * 16 + g >= p.rows) q[mt][s][0] = q[mt][s][2] = 0u;
                        if (mt * 16 + 8 + g >= p.rows) q[mt][s][1] = q[mt][s][3] = 0u;
                    }
        };
        // logits of the page: v[mt][e][i] of row 16 mt + 8 e + g and token 2 tq + (i & 1) + 8 (i >> 1)
        auto logits = [&](float (&da)[MT][4], float (&db)[MT][4]) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int i = 0; i < 4; ++i) da[mt][i] = db[mt][i] = 0.0f;
            const uint32_t at = in.at(lane >> 4, (lane >> 3) & 1);
#pragma unroll
            for (int s = 0; s < 8; s += 2) {
                unsigned k[2][4];
                ldsm4(k[0], in.chunk(at, s));
                ldsm4(k[1], in.chunk(at, s + 1));
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        mma_bf16(da[mt], q[mt][s + i][0], q[mt][s + i][1], q[mt][s + i][2], q[mt][s + i][3], k[i][0], k[i][1]);
                        mma_bf16(db[mt], q[mt][s + i][0], q[mt][s + i][1], q[mt][s + i][2], q[mt][s + i][3], k[i][2], k[i][3]);
                    }
            }
        };
        // the last page start from which every row sees every token (padding rows are taken care of by their statistics)
        auto last_whole = [&](int tokens) { return tokens - (p.causal ? p.W : 1) - 15; };
        // pairs the window hides add nothing
        auto hide = [&](float (&da)[MT][4], float (&db)[MT][4], int tokens, int t0) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int r = mt * 16 + 8 * e + g;
                    const int last = (r < p.rows ? tokens - (p.causal ? p.W - r % p.W : 1) : -1) - t0 - 2 * tq; // that the row sees
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (i > last) da[mt][2 * e + i] = -INFINITY;
                        if (8 + i > last) db[mt][2 * e + i] = -INFINITY;
                    }
                }
        };
        GroupShare cur, old;
        old.pages = -1;
        for (int n = 0;; ++n) { // pass 1 of unit n, pass 2 of unit n - 1
            ok = warp_wait(&sh.pipe.unit_full[n % T::units], (uint32_t)((n / T::units) & 1), abort_flag);
            if (!ok) break;
            cur = sh.pipe.unit[n % T::units];
            if (cur.pages >= 0) {
                load_queries(n);
                const int whole = last_whole(cur.tokens);
                float st_a[MT][E], st_b[MT][E], st_m[MT][E]; // reference, sum of 2^(c (x - reference)), largest logit
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int e = 0; e < E; ++e) { st_a[mt][e] = -FLT_MAX; st_b[mt][e] = 0.0f; st_m[mt][e] = -INFINITY; }
                int k = in.turn;
                for (; k < cur.pages; k += kWarps) {
                    ok = in.wait();
                    if (!ok) break;
                    float da[MT][4], db[MT][4];
                    logits(da, db);
                    in.release();
                    const int t0 = k * kPage;
                    if (t0 > whole) hide(da, db, cur.tokens, t0);
                    // The sum's reference follows the largest logit at a distance of up to 2^32, so that rescaling is rare; the
                    // sum is put on the maximum at the end.  One branch for all rows: their exponentials then overlap.
                    bool far = false;
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            st_m[mt][e] = max3(max3(st_m[mt][e], da[mt][2 * e], da[mt][2 * e + 1]), db[mt][2 * e], db[mt][2 * e + 1]);
                            far |= st_m[mt][e] - st_a[mt][e] > 32.0f / c;
                        }
                    if (far) {
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                            for (int e = 0; e < E; ++e) {
                                const float mx = st_m[mt][e];
                                if (mx > st_a[mt][e]) { st_b[mt][e] *= ex2((st_a[mt][e] - mx) * c); st_a[mt][e] = mx; }
                            }
                    }
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            const float n = -st_a[mt][e];
                            const float2 s = ex2_from(da[mt][2 * e], da[mt][2 * e + 1], n, n), t = ex2_from(db[mt][2 * e], db[mt][2 * e + 1], n, n);
                            st_b[mt][e] += (s.x + s.y) + (t.x + t.y);
                        }
                }
                if (!ok) break;
                in.turn = k - cur.pages;
                // fold the four lanes of a row
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        float m = st_m[mt][e], z = m > -INFINITY ? st_b[mt][e] * ex2((st_a[mt][e] - m) * c) : 0.0f;
#pragma unroll
                        for (int o = 1; o < 4; o <<= 1) {
                            const float m2 = __shfl_xor_sync(0xffffffffu, m, o), z2 = __shfl_xor_sync(0xffffffffu, z, o);
                            stat_merge(m, z, m2, z2);
                        }
                        if (tq == 0) sh.stat[n & 1][warp][mt * 16 + 8 * e + g] = make_float2(m, z);
                    }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh.pipe.summed[n & 1]));
            }
            if (n > 0) {
                const int m = n - 1;
                ok = warp_wait(&sh.pipe.ready[m & 1], (uint32_t)((m >> 1) & 1), abort_flag);
                if (!ok) break;
                load_queries(m);
                const int whole = last_whole(old.tokens);
                float b[MT][E];
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int e = 0; e < E; ++e) b[mt][e] = sh.b[m & 1][mt * 16 + 8 * e + g];
                const float pmax = sh.pmax[m & 1];
                int k = in.turn;
                for (; k < old.pages; k += kWarps) {
                    ok = in.wait();
                    if (!ok) break;
                    float da[MT][4], db[MT][4];
                    logits(da, db);
                    in.release();
                    const int t0 = k * kPage;
                    if (t0 > whole) hide(da, db, old.tokens, t0);
                    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f}; // tokens 2 tq, 2 tq + 1, 8 + 2 tq, 9 + 2 tq
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            const float n = b[mt][e];
                            const float2 s = ex2_from(da[mt][2 * e], da[mt][2 * e + 1], n, n), t = ex2_from(db[mt][2 * e], db[mt][2 * e + 1], n, n);
                            acc[0] += s.x; acc[1] += s.y; acc[2] += t.x; acc[3] += t.y;
                        }
                    // sums over the eight lanes of a tq, four tokens at once: at each step a lane hands half of its values over
                    const bool up = lane & 16, odd = lane & 8;
                    float k0 = up ? acc[2] : acc[0], k1 = up ? acc[3] : acc[1];
                    k0 += __shfl_xor_sync(0xffffffffu, up ? acc[0] : acc[2], 16);
                    k1 += __shfl_xor_sync(0xffffffffu, up ? acc[1] : acc[3], 16);
                    float v = (odd ? k1 : k0) + __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, 8);
                    v += __shfl_xor_sync(0xffffffffu, v, 4);
                    const int t = t0 + (up ? 8 : 0) + 2 * tq + (odd ? 1 : 0);
                    if (!(lane & 4) && t < old.tokens) {
                        const int ninv = p.causal ? p.G * max(0, t - (old.tokens - p.W)) : 0;
                        old.scores[t] = (v + (float)ninv * pmax) * p.inv_rows;
                    }
                }
                if (!ok) break;
                in.turn = k - old.pages;
                if (lane == 0) mbar_arrive(smem_u32(&sh.pipe.unit_empty[m % T::units]));
            }
            if (cur.pages < 0) break;
            old = cur;
        }
    } else if (warp < kWarps + kFeeders) {
        ok = feed_pages<2>(p, gr, k_map, sh.pipe, warp - kWarps, [&](int n, const GroupUnit &u) {
            feed_queries<RP>(p, q_map, u, smem_u32(sh.q[n % T::units]), smem_u32(&sh.pipe.unit_full[n % T::units]));
        });
    } else {
        ok = exchange_stats<RP, kWarps>(p, gr, sh, warp - kWarps - kFeeders);
    }
    if (!ok && lane == 0) report_timeout(p, 5, 0);
}

// Up to sixteen query rows: a page's logits are an eighth or a quarter of its keys, so they stay in shared memory until the unit's
// statistics are there, and K is read once.  The page's tokens are the M operand, eight query rows an N operand; a lane gets the
// logits that it stored back from the same place.
template <int NB> // padded query rows / 8
struct OnceTraits {
    static constexpr int rows = NB * 8;
    // Places for two units' logits, the one being read and the one before, with what a ring of two pages per warp leaves:
    // enough for 131072 tokens spread over all SMs.
    static constexpr int warps = NB == 1 ? 16 : 10;
    static constexpr int held = NB == 1 ? 10 : 12;
    static constexpr int ring = 2, units = 3;
    static constexpr int pages = warps * (held / 2); // most of a unit that a block can take
    static constexpr int threads = (warps + kFeeders + kGroupCollectors) * 32;
};
// (no second read: as much as the places hold; 256 units of 20000 tokens at 36 / 44 MB: 249 / 225 us)
constexpr float kOnceWindow = 44.0f * (1 << 20);

template <int NB>
struct OnceShared {
    using T = OnceTraits<NB>;
    GroupPipe<T::warps, T::ring, T::units> pipe;
    alignas(1024) unsigned char q[T::units][T::rows * kRowBytes]; // the units' query rows, halves of 128 bytes, swizzled
    float4 logits[T::warps][T::held][NB][32];
    float2 stat[2][T::warps][T::rows];                            // the warps' (max, sum)
    float2 part[2][32];                                           // the second collector's share of the group's
    float2 b[2][T::rows];                                         // the rows' references
    float pmax[2];                                                // largest probability of the window
};
static_assert(sizeof(OnceShared<1>) <= 227 * 1024 && sizeof(OnceShared<2>) <= 227 * 1024, "shared memory of a block");

template <int NB>
__global__ void __launch_bounds__(OnceTraits<NB>::threads, 1) k_window_once(DevParams p, const __grid_constant__ CUtensorMap k_map,
                                                                            const __grid_constant__ CUtensorMap q_map)
{
    using T = OnceTraits<NB>;
    constexpr int kWarps = T::warps;
    extern __shared__ __align__(1024) unsigned char smem[];
    OnceShared<NB> &sh = *reinterpret_cast<OnceShared<NB> *>(smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, tq = lane & 3;
    volatile int *abort_flag = &sh.pipe.abort_flag;
    if (threadIdx.x == 0) { tma_prefetch_map(&k_map); tma_prefetch_map(&q_map); }
    pipe_init(sh.pipe);
    wait_for_previous_kernel(); // effective lengths; the exchange's counters
    const Groups gr = split_groups(p, kWarps, kOnceWindow, T::pages);
    if (gr.id >= gr.n) return;
    bool ok = true;
    if (warp < kWarps) {
        constexpr float c = kLogitScale;
        PipeReader<T::warps, T::ring, T::units> in(sh.pipe, warp);
        int see[NB][2]; // row 8 nb + 2 tq + e: the last token it sees, from the end of the sequence
#pragma unroll
        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int r = 8 * nb + 2 * tq + e;
                see[nb][e] = r < p.rows ? (p.causal ? (r % p.W) - p.W : -1) : -(1 << 30);
            }
        GroupShare cur, old;
        old.pages = -1;
        int kept = 0, first_old = 0, k_old = 0; // places of logits in turn; the unit before: its first place and page
        for (int n = 0;; ++n) {                 // pass 1 of unit n, pass 2 of unit n - 1
            ok = warp_wait(&sh.pipe.unit_full[n % T::units], (uint32_t)((n / T::units) & 1), abort_flag);
            if (!ok) break;
            cur = sh.pipe.unit[n % T::units];
            int k_cur = 0, first_cur = kept;
            if (cur.pages >= 0) {
                unsigned q[NB][8][2];
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int s = 0; s < 8; s += 2) { // two k-steps at a time
                        unsigned x[4];
                        ldsm4(x, smem_u32(sh.q[n % T::units]) + (nb * 8 + (lane & 7)) * 128 + (s >> 2) * (T::rows * 128) +
                                     (((2 * (s & 3) + (lane >> 3)) ^ (lane & 7)) << 4));
                        const bool row = nb * 8 + g < p.rows; // the copy goes on into the next unit's rows: they are taken as zeros
                        q[nb][s][0] = row ? x[0] : 0u; q[nb][s][1] = row ? x[1] : 0u;
                        q[nb][s + 1][0] = row ? x[2] : 0u; q[nb][s + 1][1] = row ? x[3] : 0u;
                    }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh.pipe.unit_empty[n % T::units]));
                float st_a[NB][2], st_b[NB][2], st_m[NB][2]; // reference, sum of 2^(c (x - reference)), largest logit
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int e = 0; e < 2; ++e) { st_a[nb][e] = -FLT_MAX; st_b[nb][e] = 0.0f; st_m[nb][e] = -INFINITY; }
                int k = in.turn;
                k_cur = k;
                for (; k < cur.pages; k += kWarps) {
                    ok = in.wait();
                    if (!ok) break;
                    float d[NB][4];
#pragma unroll
                    for (int nb = 0; nb < NB; ++nb) d[nb][0] = d[nb][1] = d[nb][2] = d[nb][3] = 0.0f;
                    const uint32_t at = in.at((lane >> 3) & 1, lane >> 4);
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        unsigned a[4];
                        ldsm4(a, in.chunk(at, s));
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb) mma_bf16(d[nb], a[0], a[1], a[2], a[3], q[nb][s][0], q[nb][s][1]);
                    }
                    in.release();
                    const int t0 = k * kPage;
                    if (t0 + 15 >= cur.tokens || (p.causal && t0 + 15 > cur.tokens - p.W)) { // pairs the window hides add nothing
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const int last = min(cur.tokens + see[nb][e], cur.tokens - 1) - t0 - g;
                                if (last < 0) d[nb][e] = -INFINITY;
                                if (last < 8) d[nb][2 + e] = -INFINITY;
                            }
                    }
                    // (references and sums as above)
                    bool far = false;
#pragma unroll
                    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            st_m[nb][e] = max3(st_m[nb][e], d[nb][e], d[nb][2 + e]);
                            far |= st_m[nb][e] - st_a[nb][e] > 32.0f / c;
                        }
                    if (far) {
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const float mx = st_m[nb][e];
                                if (mx > st_a[nb][e]) { st_b[nb][e] *= ex2((st_a[nb][e] - mx) * c); st_a[nb][e] = mx; }
                            }
                    }
#pragma unroll
                    for (int nb = 0; nb < NB; ++nb) {
                        const float2 s = ex2_from(d[nb][0], d[nb][1], -st_a[nb][0], -st_a[nb][1]);
                        const float2 t = ex2_from(d[nb][2], d[nb][3], -st_a[nb][0], -st_a[nb][1]);
                        st_b[nb][0] += s.x + t.x;
                        st_b[nb][1] += s.y + t.y;
                        sh.logits[warp][kept][nb][lane] = make_float4(d[nb][0], d[nb][1], d[nb][2], d[nb][3]);
                    }
                    kept = kept == T::held - 1 ? 0 : kept + 1;
                }
                if (!ok) break;
                in.turn = k - cur.pages;
                // fold the eight lanes of a row
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float m = st_m[nb][e], z = m > -INFINITY ? st_b[nb][e] * ex2((st_a[nb][e] - m) * c) : 0.0f;
#pragma unroll
                        for (int o = 4; o < 32; o <<= 1) {
                            const float m2 = __shfl_xor_sync(0xffffffffu, m, o), z2 = __shfl_xor_sync(0xffffffffu, z, o);
                            stat_merge(m, z, m2, z2);
                        }
                        if (g == 0) sh.stat[n & 1][warp][8 * nb + 2 * tq + e] = make_float2(m, z);
                    }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh.pipe.summed[n & 1]));
            }
            if (n > 0) {
                const int m = n - 1;
                ok = warp_wait(&sh.pipe.ready[m & 1], (uint32_t)((m >> 1) & 1), abort_flag);
                if (!ok) break;
                float2 b[NB][2];
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int e = 0; e < 2; ++e) b[nb][e] = sh.b[m & 1][8 * nb + 2 * tq + e];
                const float pmax = sh.pmax[m & 1];
                int at = first_old;
                for (int k = k_old; k < old.pages; k += kWarps) {
                    float lo = 0.0f, hi = 0.0f; // tokens g and g + 8
#pragma unroll
                    for (int nb = 0; nb < NB; ++nb) {
                        const float4 d = sh.logits[warp][at][nb][lane];
                        const float2 s = ex2_from(d.x, d.y, b[nb][0], b[nb][1]), t = ex2_from(d.z, d.w, b[nb][0], b[nb][1]);
                        lo += s.x + s.y;
                        hi += t.x + t.y;
                    }
                    at = at == T::held - 1 ? 0 : at + 1;
                    // sums over the four lanes of a token, both tokens at once
                    float v = (tq & 1 ? hi : lo) + __shfl_xor_sync(0xffffffffu, tq & 1 ? lo : hi, 1);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    const int t = k * kPage + g + (tq & 1 ? 8 : 0);
                    if (tq < 2 && t < old.tokens) {
                        const int ninv = p.causal ? p.G * max(0, t - (old.tokens - p.W)) : 0;
                        old.scores[t] = (v + (float)ninv * pmax) * p.inv_rows;
                    }
                }
            }
            if (cur.pages < 0) break;
            old = cur;
            first_old = first_cur; k_old = k_cur;
        }
    } else if (warp < kWarps + kFeeders) {
        ok = feed_pages<1>(p, gr, k_map, sh.pipe, warp - kWarps, [&](int n, const GroupUnit &u) {
            feed_queries<T::rows>(p, q_map, u, smem_u32(sh.q[n % T::units]), smem_u32(&sh.pipe.unit_full[n % T::units]));
        });
    } else {
        ok = exchange_stats<T::rows, kWarps>(p, gr, sh, warp - kWarps - kFeeders);
    }
    if (!ok && lane == 0) report_timeout(p, 5, 0);
}

template <int RP, typename Shared, typename Kernel>
int launch_window(Kernel kernel, int least, int threads, const DevParams &p_in, LaunchCtx &ctx)
{
    DevParams p = p_in;
    p.inv_rows = 1.0f / (float)p.rows;
    p.group_count += kGroupCounters * kGroupCounterPad; // (the event's other launch of this kind scores keys)
    const EncodeTiledFn enc = encode_fn();
    if (!enc) return AMS_ERR_CUDA;
    CUtensorMap k_map, q_map;
    int rc = make_k_map(p, enc, &k_map);
    if (rc == AMS_OK) rc = make_rows_map(p.q, (unsigned long long)p.L * p.B * p.H * p.rows, enc, &q_map, RP);
    if (rc != AMS_OK) return rc;
    static SmemGrant grant;
    if (!grant_dynamic_smem(kernel, sizeof(Shared), grant)) return AMS_ERR_CUDA;
    const cudaError_t e = launch_groups(kernel, least, threads, sizeof(Shared), ctx.s, p, k_map, q_map);
    if (e == cudaErrorCooperativeLaunchTooLarge) { (void)cudaGetLastError(); return AMS_ERR_UNSUPPORTED; }
    if (e != cudaSuccess) return AMS_ERR_CUDA;
    ctx.mark(kKernScore1);
    return AMS_OK;
}

} // namespace

int launch_score_window(const DevParams &p, LaunchCtx &ctx)
{
    // (a context with too few SMs to hold a unit's logits takes the kernel that reads K again)
    auto least = [&](int pages) { return (p.T_cap / kPage + pages - 2) / (pages - 1); };
    int rc = AMS_ERR_UNSUPPORTED;
    if (p.rows <= 8) rc = launch_window<8, OnceShared<1>>(k_window_once<1>, least(OnceTraits<1>::pages), OnceTraits<1>::threads, p, ctx);
    else if (p.rows <= 16) rc = launch_window<16, OnceShared<2>>(k_window_once<2>, least(OnceTraits<2>::pages), OnceTraits<2>::threads, p, ctx);
    return rc != AMS_ERR_UNSUPPORTED ? rc : launch_window<32, WideShared>(k_window, 1, WideTraits::threads, p, ctx);
}

} // namespace ams
