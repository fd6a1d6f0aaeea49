// Window scorer of the AMS compression step.
//
// TOVA-style usage (Section 3.2 / Algorithm 1 step 1 of the paper): every query row
// r = (head of the GQA group, window query j) is a softmax of q_r.k_t/sqrt(D) over the
// tokens the row can see; the usage of a token is the mean over rows, where a
// (row, token) pair the row cannot see counts as the largest probability in the
// window.  Two phases over K: phase 1 finds each row's (max, sum of exponentials),
// phase 2 recomputes the logits and sums the normalised probabilities over rows.
// The largest probability of a row is 1/Z_r (its arg-max token), so the window
// maximum is 1/min_r Z_r and needs no third pass.  Up to 32 rows: ams_score_window.cu (here where the caller wants
// independent blocks); from 64: ams_score_tc.cu; the rest here.
#include <float.h>

#include "ams_common.cuh"
#include "ams_tc_ptx.cuh"

namespace ams {

namespace {

using namespace tc;

constexpr int kTovaThreads = 128;
constexpr int kRing = 3;       // 16-token K tiles per warp in shared memory: one worked on, two on their way
constexpr int kTileK = 16 * kRowBytes;
static_assert(kRing == 3, "the waits below count on two tiles in flight");

// One (unit, token slice, block of query rows) of work, and the warp's share of it.
struct TovaItem {
    int uid, slice, rb, b, h, l, T, t_begin, t_end, mine; // mine: tiles of this warp (warp, warp + 4, ...)
    int page[2];                                          // lane k: page ids of the warp's tiles k and 32 + k
    const __nv_bfloat16 *k, *q;                           // this lane's 16 bytes of the layer's first page; first query row
};

// The stream of K tiles of one warp, and the query rows of the block, across all the work the block takes.  A block takes
// (unit, token slice) pairs in turn, all units of a slice number before the next one: the blocks of neighbouring KV heads
// read the same pages at the same time, and the slices past a sequence's end cost a look at its length instead of a block.
// A tile is 16 tokens, one page.  Its rows come through a ring of tiles in shared memory (asynchronous copies, two
// tiles ahead; a chunk of 16 bytes lies at its number XOR 4 in odd rows, so that reads are free of bank conflicts).  The
// stream runs on across the ends of slices: the next slice's page ids, queries and first tiles are on their way while this
// one's last tiles are worked on.
template <int kQRows, int PHASE>
struct TovaStream {
    const DevParams &p;
    unsigned ring, qbuf;     // shared addresses: this warp's tiles, the block's query rows [kQRows][256 bytes], one or two of them
    int units, n_slices, n_rb, wslot, rslot;
    long long item;
    int next_rb;
    size_t page_stride, row2; // elements between pages, between every other slot of a page

    __device__ __forceinline__ TovaStream(const DevParams &p_, unsigned ring0, unsigned q0) : p(p_)
    {
        ring = ring0 + (threadIdx.x >> 5) * (kRing * kTileK);
        qbuf = q0;
        units = p.L * p.B * p.H;
        n_slices = (p.T_cap + p.slice_len - 1) / p.slice_len;
        n_rb = p.rows_pad / kQRows;
        wslot = rslot = next_rb = 0;
        item = blockIdx.x;
        page_stride = (size_t)kPage * p.H * kHeadDim;
        row2 = (size_t)2 * p.H * kHeadDim;
    }
    // the next piece of work; false at the end
    __device__ __forceinline__ bool next(TovaItem &it)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (; item < (long long)units * n_slices; item += gridDim.x, next_rb = 0) {
            it.uid = (int)(item % units);
            it.slice = (int)(item / units);
            it.h = it.uid % p.H; it.b = (it.uid / p.H) % p.B; it.l = it.uid / (p.H * p.B);
            it.T = p.seq_lens[it.b];
            it.t_begin = it.slice * p.slice_len;
            if (it.T <= p.Tk || it.T > p.T_cap) continue;
            if (p.W > it.T) { if (PHASE == 1 && it.slice == 0 && threadIdx.x == 0) set_status(p.status, AMS_ERR_INVALID_ARG, it.uid, p.W, it.T); continue; }
            if (it.t_begin >= it.T) continue;
            it.t_end = min(it.T, it.t_begin + p.slice_len);
            it.rb = next_rb;
            it.mine = max(0, (((it.t_end - it.t_begin + 15) >> 4) - warp + 3) >> 2);
            const int *table = p.block_table + (size_t)it.b * p.bt_stride + (it.t_begin >> 4) + warp;
#pragma unroll
            for (int j = 0; j < 2; ++j) it.page[j] = j * 32 + lane < it.mine ? table[4 * (j * 32 + lane)] : 0;
            it.k = p.k_pages + row_offset(p, it.l, 0, lane >> 4, it.h) + (lane & 15) * 8;
            it.q = p.q + ((((size_t)it.l * p.B + it.b) * p.H + it.h) * p.G) * (size_t)p.W * kHeadDim;
            if (++next_rb >= n_rb) { next_rb = 0; item += gridDim.x; }
            return true;
        }
        return false;
    }
    // starts the copy of the warp's tile k (none past the end) and with the first one that of the queries, as one group
    __device__ __forceinline__ void fetch(const TovaItem &it, bool live, int k, int buf)
    {
        if (live && k < it.mine) {
            const int lane = threadIdx.x & 31, page = __shfl_sync(0xffffffffu, k < 32 ? it.page[0] : it.page[1], k & 31);
            const __nv_bfloat16 *src = it.k + (size_t)page * page_stride;
            const unsigned dst = ring + wslot * kTileK + (lane >> 4) * kRowBytes + (((lane & 15) ^ ((lane >> 4) << 2)) << 4);
#pragma unroll
            for (int i = 0; i < 8; ++i, src += row2) cp_async16(dst + i * 2 * kRowBytes, src);
            wslot = wslot == kRing - 1 ? 0 : wslot + 1;
        }
        if (live && k == 0) {
#pragma unroll
            for (int j = 0; j < kQRows / 8; ++j) {
                const int i = j * kTovaThreads + threadIdx.x, r = i >> 4, ch = i & 15, row = it.rb * kQRows + r;
                cp_async16_or_zero(qbuf + (buf * kQRows + r) * kRowBytes + ((ch ^ ((r & 1) << 2)) << 4),
                                   it.q + (size_t)min(row, p.rows - 1) * kHeadDim + ch * 8, row < p.rows);
            }
        }
        cp_async_commit();
    }
    // waits for the stream's next tile and reads it: lane (g, tq) gets 16-byte pieces 4 j + tq of its rows g and g + 8
    __device__ __forceinline__ void read(uint4 (&x)[4], uint4 (&y)[4])
    {
        const int lane = threadIdx.x & 31, g = lane >> 2, tq = lane & 3;
        cp_async_wait<1>();
        __syncwarp();
        const unsigned at = ring + rslot * kTileK + g * kRowBytes;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned ch = ((4 * j + tq) ^ ((g & 1) << 2)) << 4; // (rows g and g + 8 are both odd or both even)
            x[j] = lds16(at + ch);
            y[j] = lds16(at + 8 * kRowBytes + ch);
        }
        rslot = rslot == kRing - 1 ? 0 : rslot + 1;
    }
};

// Windows of 33 to 63 rows (blocks of 128 rows where the tcgen05 form does not apply): 16 query rows are the
// M operand, the tile's tokens two N operands.  A token's piece of 16 bytes is then two consecutive registers per k-step,
// as the instruction wants them (with the tile as M operand every k-step interleaves two rows' pieces: 380 of 546
// instructions per tile were moves and their like), and a thread sees four logits of a row per tile.  The queries are laid
// out in shared
// memory as the fragments the lanes read.  3.0 GB of K at 32 query rows: statistics 0.70 -> 0.52 ms, usage 0.69 -> 0.51 ms (5.9
// TB/s).
template <int MT, int PHASE>
__global__ void __launch_bounds__(kTovaThreads) k_tova_wide(DevParams p)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ float red[4][MT * 16][2];
    const unsigned smem = (unsigned)__cvta_generic_to_shared(dyn);
    const unsigned Qb = smem + (kTovaThreads / 32) * kRing * kTileK;    // [MT * 16 rows][256 bytes] as they come
    const unsigned Fr = Qb + MT * 16 * kRowBytes;                   // [MT][8 k-steps][32 lanes] fragments of the current rows
    wait_for_previous_kernel(); // effective lengths; merged statistics
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, tq = lane & 3;
    constexpr float c = kLogitScale;
    const float inv_rows = 1.0f / (float)p.rows;
    TovaStream<MT * 16, PHASE> st(p, smem, Qb);
    const int n_rb = st.n_rb;

    TovaItem cur, nxt;
    bool live = st.next(cur);
    st.fetch(cur, live, 0, 0);
    st.fetch(cur, live, 1, 0);
    while (live) {
        const bool more = st.next(nxt);
        int ahead = 0; // tiles of the next piece of work whose copy has been started
        const int uid = cur.uid, T = cur.T, t_begin = cur.t_begin, t_end = cur.t_end, rb = cur.rb, row0 = rb * MT * 16;
        const float *fin = p.fin + (size_t)uid * (p.rows_pad + 8);
        float *u_out = p.scores + (size_t)uid * p.T_cap;
        const float pmax = PHASE == 2 ? fin[p.rows_pad] : 0.0f;
        // per thread: rows (mt, e) = row0 + 16 mt + g + 8 e
        float st_a[MT][2], st_b[MT][2], st_m[MT][2]; // phase 1: reference, sum of 2^(c (x - reference)), largest logit;
                                                     // phase 2: the row's reference in the first
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                st_a[mt][e] = PHASE == 1 ? -FLT_MAX : fin[row0 + mt * 16 + 8 * e + g];
                st_b[mt][e] = 0.0f;
                st_m[mt][e] = -INFINITY;
            }
        cp_async_wait<1>(); // the queries and the first tile
        __syncthreads();
        // fragments: k-step 2 j takes words 0 and 1 of piece 4 j + tq, k-step 2 j + 1 words 2 and 3 (the tiles' pieces alike)
        for (int i = threadIdx.x; i < MT * 4 * 32; i += kTovaThreads) {
            const int ln = i & 31, j = (i >> 5) & 3, mt = i >> 7, gg = ln >> 2, ch = ((4 * j + (ln & 3)) ^ ((gg & 1) << 2)) << 4;
            const unsigned row = Qb + (mt * 16 + gg) * kRowBytes + ch;
            const uint4 lo = lds16(row), hi = lds16(row + 8 * kRowBytes);
            const unsigned f = Fr + ((mt * 8 + 2 * j) * 32 + ln) * 16;
            asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(f), "r"(lo.x), "r"(hi.x), "r"(lo.y), "r"(hi.y) : "memory");
            asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(f + 512), "r"(lo.z), "r"(hi.z), "r"(lo.w), "r"(hi.w) : "memory");
        }
        __syncthreads();

        for (int kt = 0; kt < cur.mine; ++kt) {
            uint4 x[4], y[4];
            st.read(x, y);
            if (kt + 2 < cur.mine) st.fetch(cur, true, kt + 2, 0); // into the slot read in the round before
            else { st.fetch(nxt, more, ahead, 0); ++ahead; }
            const int t0 = t_begin + (warp + 4 * kt) * 16;
            // every row sees every token of the tile (padding rows are taken care of by their statistics)
            const bool plain = t0 + 15 < t_end && t0 + 15 <= (p.causal ? T - p.W : T - 1);
            float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f}; // tokens 2 tq, 2 tq + 1, 8 + 2 tq, 9 + 2 tq
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                float da[4] = {0.0f, 0.0f, 0.0f, 0.0f}, db[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint4 f0 = lds16(Fr + ((mt * 8 + 2 * j) * 32 + lane) * 16), f1 = lds16(Fr + ((mt * 8 + 2 * j + 1) * 32 + lane) * 16);
                    mma_bf16(da, f0.x, f0.y, f0.z, f0.w, x[j].x, x[j].y);
                    mma_bf16(db, f0.x, f0.y, f0.z, f0.w, y[j].x, y[j].y);
                    mma_bf16(da, f1.x, f1.y, f1.z, f1.w, x[j].z, x[j].w);
                    mma_bf16(db, f1.x, f1.y, f1.z, f1.w, y[j].z, y[j].w);
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float v[4] = {da[2 * e], da[2 * e + 1], db[2 * e], db[2 * e + 1]};
                    if (!plain) { // pairs the window hides add nothing
                        const int r = row0 + mt * 16 + 8 * e + g;
                        const int lv = min(r < p.rows ? (p.causal ? T - p.W + (r % p.W) : T - 1) : -1, t_end - 1) - t0 - 2 * tq;
#pragma unroll
                        for (int i = 0; i < 4; ++i) v[i] = (i >> 1) * 8 + (i & 1) <= lv ? v[i] : -INFINITY;
                    }
                    if (PHASE == 1) {
                        // The sum's reference follows the largest logit at a distance of up to 2^32, so that rescaling is
                        // rare; the sum is put on the maximum at the end.
                        st_m[mt][e] = max3(max3(st_m[mt][e], v[0], v[1]), v[2], v[3]);
                        if (st_m[mt][e] - st_a[mt][e] > 32.0f / c) {
                            const float mx = st_m[mt][e];
                            st_b[mt][e] *= ex2((st_a[mt][e] - mx) * c);
                            st_a[mt][e] = mx;
                        }
                        const float n = -st_a[mt][e];
                        const float2 s = ex2_from(v[0], v[1], n, n), t = ex2_from(v[2], v[3], n, n);
                        st_b[mt][e] += (s.x + s.y) + (t.x + t.y);
                    } else {
                        const float n = st_a[mt][e];
                        const float2 s = ex2_from(v[0], v[1], n, n), t = ex2_from(v[2], v[3], n, n);
                        acc[0] += s.x; acc[1] += s.y; acc[2] += t.x; acc[3] += t.y;
                    }
                }
            }
            if (PHASE == 2) {
                // sums over the eight lanes of a tq, four tokens at once: at each step a lane hands half of its values over
                const bool up = lane & 16, odd = lane & 8;
                float k0 = up ? acc[2] : acc[0], k1 = up ? acc[3] : acc[1];
                k0 += __shfl_xor_sync(0xffffffffu, up ? acc[0] : acc[2], 16);
                k1 += __shfl_xor_sync(0xffffffffu, up ? acc[1] : acc[3], 16);
                float v = (odd ? k1 : k0) + __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 4);
                const int t = t0 + (up ? 8 : 0) + 2 * tq + (odd ? 1 : 0);
                if (!(lane & 4) && t < t_end) {
                    if (rb > 0) v += u_out[t];
                    if (rb == n_rb - 1) {
                        const int ninv = p.causal ? p.G * max(0, t - (T - p.W)) : 0;
                        v = (v + (float)ninv * pmax) * inv_rows;
                    }
                    u_out[t] = v;
                }
            }
        }
        for (; ahead < 2; ++ahead) st.fetch(nxt, more, ahead, 0); // (fewer than two tiles for this warp)

        if (PHASE == 1) {
            // fold the four lanes of a row, then the four warps
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float m = st_m[mt][e], z = m > -INFINITY ? st_b[mt][e] * ex2((st_a[mt][e] - m) * c) : 0.0f;
#pragma unroll
                    for (int o = 1; o < 4; o <<= 1) {
                        const float m2 = __shfl_xor_sync(0xffffffffu, m, o), z2 = __shfl_xor_sync(0xffffffffu, z, o);
                        stat_merge(m, z, m2, z2);
                    }
                    if (tq == 0) {
                        red[warp][mt * 16 + 8 * e + g][0] = m;
                        red[warp][mt * 16 + 8 * e + g][1] = z;
                    }
                }
            __syncthreads();
            for (int r = threadIdx.x; r < MT * 16; r += kTovaThreads) {
                float m = red[0][r][0], z = red[0][r][1];
#pragma unroll
                for (int w = 1; w < 4; ++w) stat_merge(m, z, red[w][r][0], red[w][r][1]);
                float2 *out = reinterpret_cast<float2 *>(p.part) + ((size_t)uid * p.n_slices + cur.slice) * p.rows_pad + row0 + r;
                *out = make_float2(m, z);
            }
        }
        cur = nxt;
        live = more;
    }
    cp_async_wait<0>();
}

// Per unit: merge the slices' (max, sum) in slice order; the rows' references, and the window maximum 1 / min_r Z_r.
__global__ void __launch_bounds__(128) k_tova_combine(DevParams p)
{
    __shared__ u64 scratch[40];
    wait_for_previous_kernel(); // the slices' statistics
    const int uid = blockIdx.x;
    const int b = (uid / p.H) % p.B;
    const int T = p.seq_lens[b];
    if (T <= p.Tk || T > p.T_cap || p.W > T) return;
    const int ns = (T + p.slice_len - 1) / p.slice_len;
    float *fin = p.fin + (size_t)uid * (p.rows_pad + 8);
    float best = 0.0f;
    for (int r = threadIdx.x; r < p.rows_pad; r += blockDim.x) {
        float m = -INFINITY, z = 0.0f;
        for (int s = 0; s < ns; ++s) {
            const float2 v = reinterpret_cast<const float2 *>(p.part)[((size_t)uid * p.n_slices + s) * p.rows_pad + r];
            stat_merge(m, z, v.x, v.y);
        }
        const bool live = r < p.rows && z > 0.0f;
        set_reference(fin[r], live, m, z); // padding rows contribute nothing
        if (live) best = fmaxf(best, 1.0f / z);
    }
    best = block_max_f32(best, scratch);
    if (threadIdx.x == 0) fin[p.rows_pad] = best;
}

template <int MT>
int launch_tova_wide(const DevParams &p, LaunchCtx &ctx)
{
    constexpr size_t smem = (size_t)(kTovaThreads / 32) * kRing * kTileK + (size_t)2 * MT * 16 * kRowBytes;
    const auto k1 = k_tova_wide<MT, 1>, k2 = k_tova_wide<MT, 2>;
    static SmemGrant grant1, grant2;
    static int resident[2][kMaxDevices]; // blocks per SM
    const int dev = current_device(), n_sm = sm_count();
    if (dev < 0 || n_sm <= 0 || !grant_dynamic_smem(k1, smem, grant1) || !grant_dynamic_smem(k2, smem, grant2)) return AMS_ERR_CUDA;
    if (!resident[0][dev] && (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident[1][dev], k2, kTovaThreads, smem) != cudaSuccess ||
                              cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident[0][dev], k1, kTovaThreads, smem) != cudaSuccess))
        return AMS_ERR_CUDA;
    const long long units = (long long)p.L * p.B * p.H, items = units * ((p.T_cap + p.slice_len - 1) / p.slice_len);
    auto blocks = [&](int phase) {
        const long long r = (long long)n_sm * (resident[phase][dev] > 0 ? resident[phase][dev] : 1);
        return dim3((unsigned)(items < r ? items : r));
    };
    launch_after(k1, blocks(0), dim3(kTovaThreads), smem, ctx.s, p);
    ctx.mark(kKernScore1);
    launch_after(k_tova_combine, dim3((unsigned)units), dim3(128), 0, ctx.s, p);
    ctx.mark(kKernScoreCombine);
    launch_after(k2, blocks(1), dim3(kTovaThreads), smem, ctx.s, p);
    ctx.mark(kKernScore2);
    return cudaGetLastError() == cudaSuccess ? AMS_OK : AMS_ERR_CUDA;
}

} // namespace

int tova_rows_block(int rows)
{
    int ntb = 1;
    while (ntb < 16 && ntb * 8 < rows) ntb *= 2;
    return ntb * 8;
}

int launch_score_tova(const DevParams &p, LaunchCtx &ctx)
{
    if (tova_tc_supported(p)) return launch_score_tova_tc(p, ctx);
    if (p.rows <= 32 && !p.independent) return launch_score_window(p, ctx);
    if (p.rows <= 32) {
        DevParams q = p;
        q.rows_pad = 32; // (the workspace has room for 128 floats per slice and 136 per unit at least)
        return launch_tova_wide<2>(q, ctx);
    }
    return tova_rows_block(p.rows) == 64 ? launch_tova_wide<4>(p, ctx) : launch_tova_wide<8>(p, ctx);
}

} // namespace ams
