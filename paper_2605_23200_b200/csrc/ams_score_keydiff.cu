// KeyDiff-style score: negative cosine similarity of each key to the mean key of its (sequence, KV head) cache.
//
// One cooperative launch over groups of blocks (ams_groups.cuh).  Pass 1 sums a unit's keys, pass 2 scores them, both on the
// tensor cores.  Two warps feed sixteen streaming warps; two more exchange the sums, so that no streaming
// warp waits for another block unless that one is more than a unit's read behind.  Bound by the K stream, read once from HBM
// and once from L2, and by the spread of the blocks of a group at each exchange: 17.2 GB of K (2048 units of 32768
// tokens) 5.72 ms with one kernel per pass and both reads from HBM, now 3.47 ms (5.0 TB/s of HBM, 9.9 TB/s of L2); 256 units of 3000
// tokens 101 -> 68 us.  One warp to feed them all 4.07 ms (its copies go out one by one); thread-issued 16-byte copies, each
// warp for itself, 4.02 ms (half of the instructions were addresses).  Every wait is bounded; on
// expiry the block reports AMS_ERR_TIMEOUT, drains its copies and returns.
#include "ams_common.cuh"
#include "ams_groups.cuh"

namespace ams {

namespace {

using namespace tc;

constexpr int kKdWarps = 16, kKdRing = 3, kKdUnits = 4;
// 512 units of 4096 tokens at 26 / 34 / 42 / 50 / 64 MB: 131 / 136 / 148 / 149 / 175 us
constexpr float kKdWindow = 26.0f * (1 << 20);
constexpr int kKdThreads = (kKdWarps + kFeeders + kGroupCollectors) * 32;

struct KdShared {
    GroupPipe<kKdWarps, kKdRing, kKdUnits> pipe;
    alignas(16) float sum[2][kKdWarps][kHeadDim];        // the warps' sums of a unit's keys
    float4 part[2][32];                      // the second collector's share of the group's sum
    alignas(16) __nv_bfloat16 mean[2][3][kHeadDim + 8];  // the mean key as a sum of three bf16 vectors
    float norm[2];
};

// both, the first or none of two neighbouring bf16 values
__device__ __forceinline__ unsigned tokens_mask(int n) { return n >= 2 ? 0xffffffffu : n == 1 ? 0xffffu : 0u; }

__global__ void __launch_bounds__(kKdThreads, 1) k_keydiff(DevParams p, const __grid_constant__ CUtensorMap k_map)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    KdShared &sh = *reinterpret_cast<KdShared *>(smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gq = lane >> 2, tq = lane & 3;
    volatile int *abort_flag = &sh.pipe.abort_flag;
    if (threadIdx.x == 0) tma_prefetch_map(&k_map);
    pipe_init(sh.pipe);
    wait_for_previous_kernel(); // effective lengths; the exchange's counters
    const Groups gr = split_groups(p, kKdWarps, kKdWindow, 1 << 20);
    if (gr.id >= gr.n) return;
    bool ok = true;
    if (warp < kKdWarps) {
        PipeReader<kKdWarps, kKdRing, kKdUnits> in(sh.pipe, warp);
        GroupShare cur, old;
        old.pages = -1;
        for (int n = 0;; ++n) { // pass 1 of unit n, pass 2 of unit n - 1
            ok = warp_wait(&sh.pipe.unit_full[n % kKdUnits], (uint32_t)((n / kKdUnits) & 1), abort_flag);
            if (!ok) break;
            cur = sh.pipe.unit[n % kKdUnits];
            if (cur.pages >= 0) {
                float acc[8][4]; // dimension 16 s + g: [s][0] and [s][1], dimension 16 s + 8 + g: [s][2] and [s][3]
#pragma unroll
                for (int s = 0; s < 8; ++s) acc[s][0] = acc[s][1] = acc[s][2] = acc[s][3] = 0.0f;
                int k = in.turn;
                for (; k < cur.pages; k += kKdWarps) {
                    ok = in.wait();
                    if (!ok) break;
                    // dimensions as rows, tokens as the contraction, against a matrix of ones
                    unsigned a[8][4];
                    const uint32_t at = in.at(lane >> 4, (lane >> 3) & 1);
#pragma unroll
                    for (int s = 0; s < 8; ++s) ldsm4_trans(a[s], in.chunk(at, s));
                    // the last page's rows past the end hold anything: they are taken as zeros
                    const int left = cur.tokens - k * kPage;
                    if (left < kPage) {
                        const unsigned m_lo = tokens_mask(left - 2 * tq), m_hi = tokens_mask(left - 2 * tq - 8);
#pragma unroll
                        for (int s = 0; s < 8; ++s) { a[s][0] &= m_lo; a[s][1] &= m_lo; a[s][2] &= m_hi; a[s][3] &= m_hi; }
                    }
#pragma unroll
                    for (int s = 0; s < 8; ++s) mma_bf16(acc[s], a[s][0], a[s][1], a[s][2], a[s][3], 0x3f803f80u, 0x3f803f80u);
                    in.release();
                }
                if (!ok) break;
                in.turn = k - cur.pages;
                // the four lanes of a row hold the same sums: each stores those of two steps
#pragma unroll
                for (int s = 0; s < 8; ++s)
                    if ((s >> 1) == tq) { sh.sum[n & 1][warp][16 * s + gq] = acc[s][0]; sh.sum[n & 1][warp][16 * s + 8 + gq] = acc[s][2]; }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh.pipe.summed[n & 1]));
            }
            if (n > 0) {
                const int m = n - 1;
                ok = warp_wait(&sh.pipe.ready[m & 1], (uint32_t)((m >> 1) & 1), abort_flag);
                if (!ok) break;
                // column n of the second operand: part n of the mean (three), zeros beyond
                unsigned mu[8][2];
#pragma unroll
                for (int s = 0; s < 8; ++s)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        mu[s][i] = gq < 3 ? *reinterpret_cast<const unsigned *>(&sh.mean[m & 1][gq < 3 ? gq : 0][16 * s + 8 * i + 2 * tq]) : 0u;
                const float mu_norm = sh.norm[m & 1];
                int k = in.turn;
                for (; k < old.pages; k += kKdWarps) {
                    ok = in.wait();
                    if (!ok) break;
                    unsigned a[8][4];
                    const uint32_t at = in.at((lane >> 3) & 1, lane >> 4);
#pragma unroll
                    for (int s = 0; s < 8; ++s) ldsm4(a[s], in.chunk(at, s));
                    float dot[4] = {0.0f, 0.0f, 0.0f, 0.0f}, lo[4] = {0.0f, 0.0f, 0.0f, 0.0f}, hi[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        // tokens as rows: k . mu, and k . k on the diagonals of the products with tokens 0-7 and 8-15,
                        // whose fragments are halves of the first operand's
                        mma_bf16(dot, a[s][0], a[s][1], a[s][2], a[s][3], mu[s][0], mu[s][1]);
                        mma_bf16(lo, a[s][0], a[s][1], a[s][2], a[s][3], a[s][0], a[s][2]);
                        mma_bf16(hi, a[s][0], a[s][1], a[s][2], a[s][3], a[s][1], a[s][3]);
                    }
                    in.release();
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
                in.turn = k - old.pages;
                if (lane == 0) mbar_arrive(smem_u32(&sh.pipe.unit_empty[m % kKdUnits]));
            }
            if (cur.pages < 0) break;
            old = cur;
        }
    } else if (warp < kKdWarps + kFeeders) {
        ok = feed_pages<2>(p, gr, k_map, sh.pipe, warp - kKdWarps, [&](int n, const GroupUnit &) { mbar_arrive(smem_u32(&sh.pipe.unit_full[n % kKdUnits])); });
    } else {
        // exchange: one warp publishes the block's sum of each unit, both collect the group's, in the blocks' order
        const int w = warp - kKdWarps - kFeeders;
        GroupWalk walk = group_walk(p, gr);
        GroupUnit u;
        for (int n = 0; next_group_unit(p, gr, walk, u); ++n) {
            if (w == 0) {
                ok = warp_wait(&sh.pipe.summed[n & 1], (uint32_t)((n >> 1) & 1), abort_flag);
                if (ok) {
                    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                    for (int i = 0; i < kKdWarps; ++i) {
                        const float4 v = reinterpret_cast<const float4 *>(sh.sum[n & 1][i])[lane];
                        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
                    }
                    __stcg(group_slot<float4>(p, gr, gr.me, n) + lane, s);
                    group_publish(p, gr, n);
                }
            }
            float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            ok = ok && group_await(p, gr, n, abort_flag);
            if (ok) {
                constexpr int kAhead = 16; // loads in flight
                const float4 *src = group_slot<float4>(p, gr, 0, n) + lane;
                for (int i0 = w; i0 < gr.g; i0 += kAhead * kGroupCollectors) {
                    float4 v[kAhead];
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) {
                        const int member = i0 + i * kGroupCollectors;
                        v[i] = member < gr.g ? __ldcg(src + (size_t)member * (kGroupSlot / 16)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    }
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) { s.x += v[i].x; s.y += v[i].y; s.z += v[i].z; s.w += v[i].w; }
                }
            }
            if (w == 1) sh.part[n & 1][lane] = s;
            ok = named_barrier_all(1, kGroupCollectors * 32, ok);
            if (!ok) break;
            if (w == 0) {
                const float T = (float)u.T;
                const float4 o4 = sh.part[n & 1][lane];
                float v[4] = {(s.x + o4.x) / T, (s.y + o4.y) / T, (s.z + o4.z) / T, (s.w + o4.w) / T};
                float sq = (v[0] * v[0] + v[1] * v[1]) + (v[2] * v[2] + v[3] * v[3]);
#pragma unroll
                for (int part = 0; part < 3; ++part)
#pragma unroll
                    for (int i = 0; i < 4; i += 2) {
                        const __nv_bfloat162 x = __floats2bfloat162_rn(v[i], v[i + 1]);
                        *reinterpret_cast<__nv_bfloat162 *>(&sh.mean[n & 1][part][4 * lane + i]) = x;
                        v[i] -= __low2float(x); v[i + 1] -= __high2float(x);
                    }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                if (lane == 0) sh.norm[n & 1] = sqrtf(sq);
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh.pipe.ready[n & 1]));
            }
        }
    }
    if (!ok && lane == 0) report_timeout(p, 4, 0);
}

// The same score by blocks that never wait for one another, both passes from HBM, a kernel each (5.7 ms where k_keydiff takes 3.5):
// for callers that cannot give an event the whole device at once.  A sequence is cut by the capacity alone, so its scores do
// not depend on the others of the batch.
constexpr int kApartThreads = 256; // 16 token rows x 16 lanes of 16 bytes

__global__ void __launch_bounds__(kApartThreads) k_keydiff_sum(DevParams p)
{
    __shared__ float red[16][kHeadDim];
    wait_for_previous_kernel(); // effective lengths
    const int uid = blockIdx.y, slice = blockIdx.x;
    const int h = uid % p.H, b = (uid / p.H) % p.B, l = uid / (p.H * p.B);
    const int T = p.seq_lens[b];
    if (T <= p.Tk || T > p.T_cap) return;
    const int t_begin = slice * p.slice_len;
    if (t_begin >= T) return;
    const int t_end = min(T, t_begin + p.slice_len);
    const int lane = threadIdx.x & 15, r = threadIdx.x >> 4;
    const int *table = p.block_table + (size_t)b * p.bt_stride;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int t = t_begin + r; t < t_end; t += 16) {
        const uint4 v = ld_stream16(p.k_pages + row_offset(p, l, table[t >> 4], t & 15, h) + lane * 8);
        acc[0] += bf16_lo(v.x); acc[1] += bf16_hi(v.x); acc[2] += bf16_lo(v.y); acc[3] += bf16_hi(v.y);
        acc[4] += bf16_lo(v.z); acc[5] += bf16_hi(v.z); acc[6] += bf16_lo(v.w); acc[7] += bf16_hi(v.w);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) red[r][lane * 8 + i] = acc[i];
    __syncthreads();
    if (threadIdx.x < kHeadDim) {
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < 16; ++i) s += red[i][threadIdx.x];
        p.part[((size_t)uid * p.n_slices + slice) * kHeadDim + threadIdx.x] = s;
    }
}

__global__ void __launch_bounds__(kHeadDim) k_keydiff_combine(DevParams p)
{
    __shared__ float sq[kHeadDim];
    wait_for_previous_kernel(); // the slices' sums
    const int uid = blockIdx.x;
    const int b = (uid / p.H) % p.B;
    const int T = p.seq_lens[b];
    if (T <= p.Tk || T > p.T_cap) return;
    const int ns = (T + p.slice_len - 1) / p.slice_len;
    float s = 0.0f;
    for (int i = 0; i < ns; ++i) s += p.part[((size_t)uid * p.n_slices + i) * kHeadDim + threadIdx.x];
    const float mu = s / (float)T;
    float *fin = p.fin + (size_t)uid * (p.rows_pad + 8);
    fin[threadIdx.x] = mu;
    sq[threadIdx.x] = mu * mu;
    __syncthreads();
    if (threadIdx.x == 0) {
        float tot = 0.0f;
        for (int i = 0; i < kHeadDim; ++i) tot += sq[i];
        fin[kHeadDim] = sqrtf(tot);
    }
}

__global__ void __launch_bounds__(kApartThreads) k_keydiff_score(DevParams p)
{
    wait_for_previous_kernel(); // the mean key
    const int uid = blockIdx.y, slice = blockIdx.x;
    const int h = uid % p.H, b = (uid / p.H) % p.B, l = uid / (p.H * p.B);
    const int T = p.seq_lens[b];
    if (T <= p.Tk || T > p.T_cap) return;
    const int t_begin = slice * p.slice_len;
    if (t_begin >= T) return;
    const int t_end = min(T, t_begin + p.slice_len);
    const int lane = threadIdx.x & 15, r = threadIdx.x >> 4;
    const int *table = p.block_table + (size_t)b * p.bt_stride;
    const float *fin = p.fin + (size_t)uid * (p.rows_pad + 8);
    unsigned long long mu2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) mu2[i] = pack_f32x2(fin[lane * 8 + 2 * i], fin[lane * 8 + 2 * i + 1]);
    const float mu_norm = fin[kHeadDim];
    float *g_out = p.scores + (size_t)uid * p.T_cap;
    // four tokens per thread and round: their loads are issued together, so that enough bytes are in flight
    constexpr int kU = 4;
    const int n_iter = (t_end - t_begin + 16 * kU - 1) / (16 * kU);
    for (int it = 0; it < n_iter; ++it) {
        uint4 v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int t = t_begin + (it * kU + u) * 16 + r;
            v[u] = make_uint4(0, 0, 0, 0);
            if (t < t_end) v[u] = ld_stream16(p.k_pages + row_offset(p, l, table[t >> 4], t & 15, h) + lane * 8);
        }
        // a[2u] = this lane's part of k_t . mu, a[2u + 1] of |k_t|^2, for the four tokens u
        float a[2 * kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            // two dimensions per instruction: a bf16 pair widens to a packed fp32 pair (low half shifted up, high half
            // masked), and both running sums take packed multiply-adds
            const unsigned w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
            unsigned long long dot2 = 0ull, sq2 = 0ull; // (0.0f, 0.0f)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const unsigned long long k2 = pack_f32x2(bf16_lo(w[i]), bf16_hi(w[i]));
                dot2 = fma_f32x2(k2, mu2[i], dot2);
                sq2 = fma_f32x2(k2, k2, sq2);
            }
            a[2 * u] = sum_f32x2(dot2); a[2 * u + 1] = sum_f32x2(sq2);
        }
        // sums over the 16 lanes of a token row, all eight values at once: at each step a lane hands half of
        // its values to its partner and keeps the other half (9 shuffles instead of 32)
#pragma unroll
        for (int o = 8, n = 2 * kU; o >= 2; o >>= 1, n >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < n / 2; ++i) {
                const float send = up ? a[i] : a[i + n / 2];
                const float keep = up ? a[i + n / 2] : a[i];
                a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
        // lane holds value index 4 * bit3 + 2 * bit2 + bit1: even = dot of token (index / 2), odd = its |k|^2
        const float other = __shfl_xor_sync(0xffffffffu, a[0], 2);
        if ((lane & 3) == 0) {
            const int u = lane >> 2;
            const int t = t_begin + (it * kU + u) * 16 + r;
            if (t < t_end) g_out[t] = -a[0] / fmaxf(sqrtf(other) * mu_norm, 1e-30f);
        }
    }
}

int launch_apart(const DevParams &p, LaunchCtx &ctx)
{
    const dim3 grid((unsigned)p.n_slices, (unsigned)(p.L * p.B * p.H));
    launch_after(k_keydiff_sum, grid, dim3(kApartThreads), 0, ctx.s, p);
    ctx.mark(kKernScore1);
    launch_after(k_keydiff_combine, dim3((unsigned)(p.L * p.B * p.H)), dim3(kHeadDim), 0, ctx.s, p);
    ctx.mark(kKernScoreCombine);
    launch_after(k_keydiff_score, grid, dim3(kApartThreads), 0, ctx.s, p);
    ctx.mark(kKernScore2);
    return cudaGetLastError() == cudaSuccess ? AMS_OK : AMS_ERR_CUDA;
}

} // namespace

int launch_score_keydiff(const DevParams &p, LaunchCtx &ctx)
{
    if (p.independent) return launch_apart(p, ctx);
    const EncodeTiledFn enc = encode_fn();
    if (!enc) return AMS_ERR_CUDA;
    CUtensorMap k_map;
    const int rc = make_k_map(p, enc, &k_map);
    if (rc != AMS_OK) return rc;
    static SmemGrant grant;
    if (!grant_dynamic_smem(k_keydiff, sizeof(KdShared), grant)) return AMS_ERR_CUDA;
    if (launch_groups(k_keydiff, 1, kKdThreads, sizeof(KdShared), ctx.s, p, k_map) != cudaSuccess) return AMS_ERR_CUDA;
    ctx.mark(kKernScore1);
    return AMS_OK;
}

} // namespace ams
