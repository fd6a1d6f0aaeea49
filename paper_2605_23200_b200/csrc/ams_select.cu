// Algorithm 1 steps 1-5 of the paper for all (layer, sequence, KV head) units of an event, in one kernel with one block per
// unit: Eq. 1 on fixed-point weights, the EMA credit update and the history-aware mass (Section 3.3, "EMA credit"; steps
// 1-2), the mass-quantile cuts b_k = min{t : c(t) >= k / S} (step 3), segments (merge, split) and their quotas (steps 3-4),
// per-segment top-q_i, must-keep prefix and suffix, backfill to exactly the budget, ordered kept positions and the credit
// rows that travel with them (step 5).
//
// Every decision is integer arithmetic on fixed-point images of the mass (kFixBits fractional bits) and every
// floating-point step a single round-to-nearest operation, so results do not depend on the order in which a block adds
// things up.
//
// The mass takes one walk over the unit's row per reduction that the arithmetic needs (largest weight, sum of the images,
// credit and its maximum, sum of the credit's images, mass), a warp taking 256-token pieces.  The last walk leaves one sum
// per 32-token window in shared memory; the cuts and the masses of the segments need the mass at a hundred positions or
// so, for which the tokens of one window are computed again.  (A prefix sum of every token in memory, 8 bytes each, cost
// three times the instructions, 290 MB of traffic on the ragged batch, and a kernel of its own.)
//
// Selection order is (score key descending, position ascending), a strict total order, so a segment and its quota have
// exactly one answer however it is found.  Finding the q-th largest key is what costs.  It is bound by latency and issue
// slots, not by memory (4 bytes per token, from L2):
//   * a segment of at most 256 tokens lives in the registers of one warp.  The lanes' extreme keys give a narrow range that
//     holds the q-th key; a histogram over it (128 bins, shared memory) leads to its bin, and the few keys in that bin are
//     taken apart one by one.  Exact fallbacks take over for ties, NaN and short segments.  Fixing key bits from the top
//     instead is a chain of 16 to 20 dependent warp-wide counts.
//   * longer segments are searched together by the whole block, in walks over their 256-token pieces: largest key (from a
//     quarter of the tokens), histogram per segment over the octaves below it, then keys above the threshold's bin are
//     kept and the few inside it go to a list in which every entry counts the entries of its segment before it.  (A bin
//     that is still crowded gets another histogram first; ties by the hundred end with a bin of one key.)  Every warp has
//     the same share of the walks whatever the lengths of the segments.
// The backfill takes its bound from the best keys that groups of lanes have seen rejected, and looks only at pieces whose best
// rejected key reaches it, instead of walking the sequence twice.
//
// us per event, three kernels of the mass, the quotas and the selection before / this one: 256 units of 16384 tokens
// 118 / 59, 1792 ragged units of 8192..32768 tokens 683 / 379, 1792 units of 4224 tokens 253 / 145, 2048 units of 32768 tokens in
// long segments 922 / 480, 640 units of 131072 tokens 1684 / 1130, 512 units of 7001..8191 tokens 127 / 54.
#include <algorithm>
#include <type_traits>

#include "ams_common.cuh"
#include "ams_move.cuh"
#include "ams_select.cuh"

namespace ams {

using namespace sel;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kPiece = 256;         // tokens a warp holds in registers, eight per lane
constexpr int kPer = kPiece / 32;
constexpr int kWarpBins = 128;      // bins of a warp's own histogram, four per lane
constexpr int kBatch = 64;          // long segments searched together
constexpr int kMaxBins = 1024;      // histogram bins per long segment
constexpr unsigned kOctaves = 12;   // octaves below a long segment's largest score that its histogram resolves
constexpr int kMoveLimit = 1 << 22; // polls of a move for the units that it needs: a second and more, as each goes to L2
constexpr int kBest = 512;          // entries of the table of the pieces' best rejected keys

// Working arrays of the search of long segments, one entry per segment of the batch.
struct SegTab {
    unsigned lo[kBatch];             // bin = (key - lo) >> shift, the first and last one taking what lies outside
    unsigned rl[kBatch], rw[kBatch]; // only the keys [rl, rl + rw] are counted
    unsigned L[kBatch], U[kBatch];   // keys >= U win, keys < L lose
    int above[kBatch];               // keys above the range of the histogram
    int r[kBatch], m[kBatch];        // r of the m keys in [L, U) win
    int base[kBatch], cnt[kBatch];   // part of the list
    unsigned short seg[kBatch];
    int piece0[kBatch + 1];          // first piece
    unsigned char shift[kBatch];
    unsigned char state[kBatch];
};
enum { kDone = 0, kSearch = 1, kTies = 2 };

template <int NT> struct Tune {
    static constexpr int kBins = NT <= 256 ? 8192 : 16384; // histogram bins of a batch
    static constexpr int kList = NT <= 256 ? 1024 : 2048;  // candidates, of the long segments and then of the backfill
};

struct SelSmem { size_t mask, ms, bounds, quota, best, list, hist, tab, total; };
template <int NT>
__host__ __device__ inline SelSmem sel_smem(int T_cap, int sc, int S, bool longs)
{
    SelSmem m;
    size_t o = 0;
    m.mask = o;   o += (size_t)((T_cap + 31) / 32 + 2) * 4;
    o = (o + 15) & ~(size_t)15;
    m.ms = o;     o += (size_t)sc * 8;
    m.bounds = o; o += (size_t)(sc + 1) * 4;
    m.quota = o;  o += (size_t)sc * 4;
    o = (o + 15) & ~(size_t)15;
    m.best = o;   o += (size_t)kBest * 4;
    o = (o + 15) & ~(size_t)15;
    const size_t wsum = (size_t)((T_cap + 31) / 32) * 8, list = (size_t)Tune<NT>::kList * 8;
    m.list = o;   o += wsum > list ? wsum : list; // the windows' sums of the mass, then candidates
    o = (o + 15) & ~(size_t)15;
    // one area in turn for: the quota computation, the warps' histograms, those of the long segments, the backfill's bound
    // and the pieces it looks at
    m.hist = o;
    const size_t q = (size_t)(S + 1) * 12 + (size_t)sc * 4, w = (size_t)(NT / 32) * kWarpBins * 4, l = longs ? (size_t)Tune<NT>::kBins * 4 : 0;
    o += q > w ? (q > l ? q : l) : (w > l ? w : l);
    o = (o + 15) & ~(size_t)15;
    m.tab = o;    o += longs ? sizeof(SegTab) : 0;
    m.total = (o + 15) & ~(size_t)15;
    return m;
}

struct SelShared {
    u64 scratch[40];
    int wc[2][32];   // per-warp counts of even / odd rounds of a block-wide count
    int n_list, n_look, n_long, total;
    unsigned bound, gbest[128];
    int n_merged, n_seg, level, rem;
};

__device__ __forceinline__ int warp_sum(int v) { return (int)__reduce_add_sync(kFull, v); }
__device__ __forceinline__ int warp_incl_scan(int v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(kFull, v, d);
        if (lane >= d) v += y;
    }
    return v;
}

// Sum of one count per thread over the block with one barrier per call: counts of consecutive calls land in
// alternating tables, so a table is rewritten only after every thread has passed the barrier that follows
// its last read.
template <int NT>
__device__ __forceinline__ int block_count(int c, int &round, SelShared &sh)
{
    const int lane = threadIdx.x & 31;
    c = warp_sum(c);
    int *mine = sh.wc[round++ & 1];
    if (lane == 0) mine[threadIdx.x >> 5] = c;
    __syncthreads();
    return warp_sum(lane < NT / 32 ? mine[lane] : 0);
}

// ------------------------------------------------------------------------------------------- the mass

// Calls f(a, room, full) for the 256-token pieces of [0, T): the lane's tokens are a + lane + 32 j for 32 j < room; full
// (a compile-time flag) says that all eight exist.
template <int NT, typename F>
__device__ __forceinline__ void walk_pieces(int T, F f)
{
    const int lane = threadIdx.x & 31;
    for (int a = (threadIdx.x >> 5) * kPiece; a < T; a += NT / 32 * kPiece) {
        if (a + kPiece <= T) f(a, kPiece, std::true_type{});
        else f(a, T - a - lane, std::false_type{});
    }
}

// Sum over a warp of integers below 2^51 whose total is below 2^53: two reductions of 32 bits, where five steps of two shuffles
// and an addition take five times as long.  (A credit that the caller restored with negative entries makes larger masses: their
// sum is some number then, and so are the cuts and shares, within the bounds that these keep for any.)
__device__ __forceinline__ u64 warp_sum_wide(u64 v)
{
    const unsigned lo = __reduce_add_sync(kFull, (unsigned)v & 0x3ffffffu), hi = __reduce_add_sync(kFull, (unsigned)(v >> 26));
    return ((u64)hi << 26) + lo;
}
// Block-wide sum of doubles v that are multiples of 1 / scale (a power of two) and whose sum has fewer than 53 bits of it, times
// scale: exact, hence independent of the order.  They are added as integers (the images of 131072 tokens below 2^53 in all)
// unless a credit that the caller restored is negative or not a number.
__device__ __forceinline__ double block_sum_images(double v, double scale, u64 *scratch)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = __dmul_rn(v, scale);
    const bool fits = v >= 0.0 && v < 1125899906842624.0; // 2^50
    const u64 w = warp_sum_wide(fits ? (u64)v : 0ull);
    __syncthreads();
    if (lane == 0) scratch[warp] = w;
    if (!__syncthreads_or(!fits)) return (double)warp_sum_wide(lane < nw ? scratch[lane] : 0ull);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    if (lane == 0) scratch[warp] = (u64)__double_as_longlong(v);
    __syncthreads();
    double x = lane < nw ? __longlong_as_double((long long)scratch[lane]) : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}
// Block-wide maximum of non-negative floats.
__device__ __forceinline__ float block_max_pos(float v, u64 *scratch)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned m = __reduce_max_sync(kFull, __float_as_uint(v));
    __syncthreads();
    if (lane == 0) scratch[warp] = m;
    __syncthreads();
    return __uint_as_float(__reduce_max_sync(kFull, lane < nw ? (unsigned)scratch[lane] : 0u));
}
// Sum over a warp of 37-bit integers.
__device__ __forceinline__ u64 warp_sum_mass(u64 h)
{
    const unsigned lo = __reduce_add_sync(kFull, (unsigned)h & 0xfffffu), hi = __reduce_add_sync(kFull, (unsigned)(h >> 20));
    return ((u64)hi << 20) + lo;
}

// What the integer mass of a token is made of.
struct Mass {
    const float *u, *credit;
    float eps, cut_w, cut_c;
    double inv_sa_w, inv_sc_c; // 2^(36 - e_w) / SA, 2^(36 - e_c) / SC
    double beta, omb;          // weights of the current and the past mass, times 2^36 (exactly)
    bool ema, have_credit;

    __device__ __forceinline__ double share(float x) const // Eq. 1 mass of a token with usage x
    {
        return __dmul_rn((double)fixed_trunc_by_add(weight_of(x, eps), cut_w), inv_sa_w);
    }
    // history-aware integer mass floor((beta m + (1 - beta) normalize(c)) 2^36)
    __device__ __forceinline__ u64 of(float x, float c) const
    {
        double r = __dmul_rn(beta, share(x)); // (beta is 2^36 where there is no credit)
        if (have_credit) r = __dadd_rn(r, __dmul_rn(omb, __dmul_rn((double)fixed_trunc_by_add(c, cut_c), inv_sc_c)));
        return floor_to_u64(r);
    }
    __device__ __forceinline__ u64 at(int t) const { return of(u[t], have_credit ? credit[t] : 0.0f); }
};

// Eq. 1, credit update, integer mass: exclusive sums of the 32-token windows into wsum; returns the total.
template <int NT>
__device__ u64 mass_of_unit(const DevParams &p, int uid, int T, float *credit, u64 *wsum, Mass &ms, SelShared &sh)
{
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t row = (size_t)uid * p.T_cap;
    const float *u = p.usage + row;
    float *mass_dbg = p.mass_dbg ? p.mass_dbg + row : nullptr;
    ms.u = u; ms.credit = credit; ms.eps = p.eps;
    ms.ema = p.beta != 1.0f;
    ms.have_credit = false;
    ms.cut_c = 0.0f; ms.inv_sc_c = 0.0;
    ms.beta = __dmul_rn((double)p.beta, (double)(1ull << kFixBits)); // (1 where there is no credit)
    ms.omb = __dmul_rn(__dsub_rn(1.0, (double)p.beta), (double)(1ull << kFixBits));
    // ---- largest Eq. 1 weight (that of the largest usage) -> exponent of the fixed-point images
    float umax = 0.0f;
    walk_pieces<NT>(T, [&](int a, int room, auto full) {
        float x[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) x[j] = decltype(full)::value || j * 32 < room ? u[a + j * 32 + lane] : 0.0f;
#pragma unroll
        for (int j = 0; j < kPer; ++j) umax = fmaxf(umax, x[j]);
    });
    const int ew = fix_exponent(weight_of(block_max_pos(umax, sh.scratch), p.eps));
    // ---- SA = sum of the images A_t = floor(w_t 2^(36 - ew)); the truncated weights are added unscaled (multiples of
    //      2^(ew - 36) below 2^(ew + 17): exact)
    const double scale_w = fix_scale_of(ew);
    ms.cut_w = fixed_trunc_threshold(ew); // weights below it lose their bits under the image's last one
    double sa = 0.0;
    walk_pieces<NT>(T, [&](int a, int room, auto full) {
        float x[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) x[j] = decltype(full)::value || j * 32 < room ? u[a + j * 32 + lane] : 0.0f;
#pragma unroll
        for (int j = 0; j < kPer; ++j)
            if (decltype(full)::value || j * 32 < room) sa += (double)fixed_trunc_by_add(weight_of(x[j], p.eps), ms.cut_w);
    });
    const double SA = block_sum_images(sa, scale_w, sh.scratch);
    ms.inv_sa_w = __dmul_rn(__ddiv_rn(1.0, SA), scale_w); // normalisations multiply by the rounded reciprocal; the scaling is exact

    // ---- EMA credit: c <- lambda c + (1 - lambda) m, updated in place (the block-wide reductions that follow
    //      make every thread's writes visible to the others before anybody reads them back)
    if (ms.ema) {
        const float oml = __fsub_rn(1.0f, p.lambda);
        float cmax = 0.0f;
        walk_pieces<NT>(T, [&](int a, int room, auto full) {
            float x[kPer], c[kPer];
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                x[j] = c[j] = 0.0f;
                if (decltype(full)::value || j * 32 < room) { x[j] = u[a + j * 32 + lane]; c[j] = credit[a + j * 32 + lane]; }
            }
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const float m = __double2float_rn(ms.share(x[j]));
                c[j] = __fadd_rn(__fmul_rn(p.lambda, c[j]), __fmul_rn(oml, m));
                if (decltype(full)::value || j * 32 < room) {
                    cmax = fmaxf(cmax, c[j]);
                    credit[a + j * 32 + lane] = c[j];
                    if (mass_dbg) mass_dbg[a + j * 32 + lane] = m;
                }
            }
        });
        cmax = block_max_pos(cmax, sh.scratch);
        if (cmax > 0.0f) {
            const int ec = fix_exponent(cmax);
            const double scale_c = fix_scale_of(ec);
            ms.cut_c = fixed_trunc_threshold(ec);
            double sc = 0.0;
            walk_pieces<NT>(T, [&](int a, int room, auto full) {
                float c[kPer];
#pragma unroll
                for (int j = 0; j < kPer; ++j) c[j] = decltype(full)::value || j * 32 < room ? credit[a + j * 32 + lane] : 0.0f;
#pragma unroll
                for (int j = 0; j < kPer; ++j) sc += (double)fixed_trunc_by_add(c[j], ms.cut_c);
            });
            const double SC = block_sum_images(sc, scale_c, sh.scratch);
            ms.have_credit = SC > 0.0 && SC < (double)INFINITY; // (a restored credit may be infinite: it has no shares)
            if (ms.have_credit) ms.inv_sc_c = __dmul_rn(__ddiv_rn(1.0, SC), scale_c);
        }
    } else if (mass_dbg) {
        for (int t = tid; t < T; t += NT) mass_dbg[t] = __double2float_rn(ms.share(u[t]));
    }

    // ---- integer mass, summed per window, and the windows' exclusive sums
    walk_pieces<NT>(T, [&](int a, int room, auto full) {
        float x[kPer], c[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            x[j] = c[j] = 0.0f;
            if (decltype(full)::value || j * 32 < room) {
                x[j] = u[a + j * 32 + lane];
                if (ms.have_credit) c[j] = credit[a + j * 32 + lane];
            }
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            u64 h = ms.of(x[j], c[j]);
            if (!(decltype(full)::value || j * 32 < room)) h = 0;
            const u64 sum = warp_sum_mass(h);
            if (lane == j && (a >> 5) + j < (T + 31) >> 5) wsum[(a >> 5) + j] = sum;
        }
    });
    __syncthreads();
    // a warp takes a run of windows, a lane eight at a time
    const int n_win = (T + 31) >> 5, per = (n_win + NW - 1) / NW, w0 = min(n_win, warp * per), w1 = min(n_win, w0 + per);
    u64 mine = 0;
    for (int w = w0 + lane; w < w1; w += 32) mine += wsum[w];
    mine = warp_sum_wide(mine);
    if (lane == 0) sh.scratch[warp] = mine; // (the reductions above ended with reads of this table two barriers ago)
    __syncthreads();
    const u64 tot = warp_sum_wide(lane < NW ? sh.scratch[lane] : 0ull);
    u64 run = warp_sum_wide(lane < warp ? sh.scratch[lane] : 0ull);
    for (int g = w0; g < w1; g += 32) {
        const u64 v = g + lane < w1 ? wsum[g + lane] : 0ull;
        u64 inc = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const u64 y = __shfl_up_sync(kFull, inc, d);
            if (lane >= d) inc += y;
        }
        if (g + lane < w1) wsum[g + lane] = run + inc - v;
        run += __shfl_sync(kFull, inc, 31);
    }
    __syncthreads();
    return tot;
}

// Sum of the integer mass before position b (0 <= b < T), by one warp.
__device__ __forceinline__ u64 mass_before(const Mass &ms, const u64 *wsum, int b)
{
    const int lane = threadIdx.x & 31;
    return wsum[b >> 5] + warp_sum_mass(lane < (b & 31) ? ms.at((b & ~31) + lane) : 0ull);
}

// Boundary after the token that reaches `thr` (at most the total), by one warp.  Always from 0 to the last window's end, whatever
// the sums are: a total of 0 (no credit and ema_beta = 0) has thresholds of 0, below which no window starts.
__device__ __forceinline__ int mass_cut(const Mass &ms, const u64 *wsum, int T, u64 thr)
{
    const int lane = threadIdx.x & 31;
    int w = 0; // the last window that starts below thr: a lane to each of 32 places at a time (the windows' sums ascend from 0)
    for (int n = (T + 31) >> 5; n > 1;) {
        const int step = (n + 31) >> 5, at = lane * step;
        const unsigned below = __ballot_sync(kFull, at < n && wsum[w + at] < thr);
        const int i = below ? 31 - __clz(below) : 0;
        w += i * step;
        n = min(step, n - i * step);
    }
    const int t = w * 32 + lane;
    u64 inc = t < T ? ms.at(t) : 0ull;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const u64 y = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += y;
    }
    return w * 32 + __ffs(__ballot_sync(kFull, wsum[w] + inc >= thr));
}

// ------------------------------------------------------------------------------- segments and quotas

// The cycling quota adjustment in closed form: `D` (> 0) tokens go to segments one per visit in the visiting order,
// segment i taking at most cap[i]; every segment receives min(cap, level) with `level` the largest whose total fits,
// and the first `rem` segments in visiting order that still have room receive one more.  sign = +1: order (M desc,
// i asc), the tokens are added to the quotas; sign = -1: order (M asc, i desc), they are taken off.  Returns what is
// left.  Counts of tokens fit 32 bits; the level is found by one warp.
template <int NT>
__device__ int block_distribute(int sign, int D, const int *cap, int *quota, const u64 *M, int n_seg, SelShared &sh)
{
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < 32) {
        constexpr int kC = 8; // room of the first 256 segments in registers
        int c[kC], cnt1 = 0, tot = 0, mx = 0;
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            c[j] = j * 32 + lane < n_seg ? cap[j * 32 + lane] : 0;
            cnt1 += c[j] >= 1; tot += c[j]; mx = max(mx, c[j]);
        }
        for (int i = kC * 32 + lane; i < n_seg; i += 32) { cnt1 += cap[i] >= 1; tot += cap[i]; mx = max(mx, cap[i]); }
        cnt1 = warp_sum(cnt1);
        tot = warp_sum(tot);
        mx = __reduce_max_sync(kFull, mx);
        int level = 0, used = 0; // F(k) = sum of min(cap, k) <= D < F(k + 1)
        if (tot <= D) {
            level = mx;
            used = tot;
        } else {
            // from F(level) <= D: as many whole rounds as the rest pays for if nobody else fills up, until it pays for none
            for (int n = cnt1; D - used >= n;) {
                level += (D - used) / n;
                int f = 0, o = 0;
#pragma unroll
                for (int j = 0; j < kC; ++j) { f += min(c[j], level); o += c[j] > level; }
                for (int i = kC * 32 + lane; i < n_seg; i += 32) { f += min(cap[i], level); o += cap[i] > level; }
                used = warp_sum(f);
                n = warp_sum(o);
            }
        }
        if (lane == 0) { sh.level = level; sh.rem = D - used; sh.total = tot <= D ? D - tot : 0; }
    }
    __syncthreads();
    const int level = sh.level, rem = sh.rem, left = sh.total;
    for (int i0 = 0; i0 < n_seg; i0 += NT / 8) { // eight lanes per segment: its rank in visiting order among those with room
        const int i = i0 + (tid >> 3);
        const bool in = i < n_seg;
        const int ci = in ? cap[i] : 0;
        int g = min(ci, level);
        if (rem > 0) {
            const long long Mx = in ? (long long)M[i] : 0ll;
            int rank = 0;
#pragma unroll 4
            for (int j = tid & 7; j < n_seg; j += 8) { // (M, position) as one strict order; masses stay far below 2^63
                const long long Mj = (long long)M[j];
                rank += cap[j] > level && (sign > 0 ? Mj + (j < i) > Mx : Mj < Mx + (j > i));
            }
#pragma unroll
            for (int d = 1; d < 8; d <<= 1) rank += __shfl_xor_sync(kFull, rank, d);
            g += ci > level && rank < rem;
        }
        if (in && (tid & 7) == 0) quota[i] += sign * g;
    }
    __syncthreads();
    return left;
}

// floor(x / y) for a quotient below 2^50 and x < 2^62, inv = 1 / y rounded: the product is off by less than one, the
// remainder corrects it.
__device__ __forceinline__ u64 quotient(u64 x, u64 y, double inv)
{
    u64 q = (u64)((double)x * inv);
    const long long rem = (long long)(x - q * y);
    if (rem < 0) --q;
    else if (rem >= (long long)y) ++q;
    return q;
}

// Merge of short and split of long segments, quotas with their adjustment (Section 3.3 of the paper; Algorithm 1 steps
// 3-4): bounds[0..n], quota[0..n).  Returns n, or -1 if the tables cannot hold the segments.  Bq: the budget less the
// must-keep positions.  SH: total of the integer mass.  `tmp`: 3 (S + 1) + seg_cap ints.
template <int NT>
__device__ int segments_and_quotas(const DevParams &p, int T, int Bq, const Mass &ms, const u64 *wsum, u64 SH, u64 *Ms, int *bounds,
                                   int *quota, int *tmp, SelShared &sh, int &round)
{
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int *merged = tmp, *poff = merged + p.S + 1, *raw = poff + p.S + 1, *cap = raw + p.S + 1;
    const u64 SHq = p.uniform_q ? (u64)T : max(SH, 1ull); // total of what the quotas are proportional to (no mass: nobody has a share)
    const double inv = 1.0 / (double)(2ull * SHq);
    const double inv_s = 1.0 / (double)p.S;
    // raw cuts, ascending: the token that reaches quantile k closes its segment, c(t) >= k / S <=> C(t) >= ceil(k SH / S)
    for (int k = warp + 1; k < p.S; k += NW) {
        const int e = p.fixed_seg ? (int)(((long long)k * T) / p.S) // component ablation: boundary k at floor(k T / S)
                                  : mass_cut(ms, wsum, T, quotient((u64)k * SH + (u64)p.S - 1, (u64)p.S, inv_s));
        if (lane == 0) raw[k] = e;
    }
    __syncthreads();
    if (warp == 0) {
        // short raw segments merge forward: the next boundary is the first cut at least l_min past the last one
        int nm = 0, start = 0;
        if (lane == 0) merged[0] = 0;
        bool plain = true; // no raw segment is short: every cut is a boundary
        for (int k0 = 1; k0 < p.S; k0 += 32) {
            const int k = k0 + lane, e = k < p.S ? raw[k] : 0, before = k > 1 && k < p.S ? raw[k - 1] : 0;
            plain = plain && (k >= p.S || (e < T && e - before >= p.l_min));
        }
        if (__all_sync(kFull, plain)) {
            for (int k = lane + 1; k < p.S; k += 32) merged[k] = raw[k];
            nm = p.S - 1;
            start = p.S > 1 ? raw[p.S - 1] : 0;
            __syncwarp();
        } else for (int k0 = 1; k0 < p.S; k0 += 32) {
            const int k = k0 + lane;
            const int e = k < p.S ? raw[k] : T;
            for (;;) {
                const unsigned can = __ballot_sync(kFull, e < T && e - start >= p.l_min);
                if (!can) break;
                start = __shfl_sync(kFull, e, __ffs(can) - 1);
                ++nm;
                if (lane == 0) merged[nm] = start;
            }
        }
        if (nm == 0 || T - start >= p.l_min) ++nm; // (otherwise the short tail folds left)
        if (lane == 0) merged[nm] = T;
        __syncwarp();
        int off = 0; // pieces of the segments before
        for (int i0 = 0; i0 < nm; i0 += 32) {
            const int i = i0 + lane;
            int c = 0;
            if (i < nm) {
                const int len = merged[i + 1] - merged[i];
                c = (p.l_max > 0 && len > p.l_max) ? (len + p.l_max - 1) / p.l_max : 1;
            }
            const int inc = warp_incl_scan(c);
            if (i < nm) poff[i] = off + inc - c;
            off += __shfl_sync(kFull, inc, 31);
        }
        if (lane == 0) { poff[nm] = off; sh.n_merged = nm; sh.n_seg = off; bounds[0] = 0; }
    }
    __syncthreads();
    const int n_merged = sh.n_merged, n_seg = sh.n_seg;
    if (n_seg > p.seg_cap) return -1;
    for (int i = warp; i < n_merged; i += NW) {
        const int a = merged[i], len = merged[i + 1] - a, o = poff[i], pieces = poff[i + 1] - o;
        const int bs = len / pieces, extra = len - bs * pieces;
        for (int j = lane; j < pieces; j += 32) bounds[o + j + 1] = a + (j + 1) * bs + min(j + 1, extra);
    }
    __syncthreads();
    // quotas: q_i = q_i^min + round(T_rem M_i / sum M), clipped, then adjusted
    if (!p.uniform_q) {
        for (int i = warp; i < n_seg; i += NW) { // mass before the segment
            const u64 c = mass_before(ms, wsum, bounds[i]);
            if (lane == 0) Ms[i] = c;
        }
        __syncthreads();
    }
    int smin = 0;
    for (int i = tid; i < n_seg; i += NT) smin += max(0, min(p.q_min, bounds[i + 1] - bounds[i]));
    const int Trem = Bq - block_count<NT>(smin, round, sh);
    int sq = 0;
    constexpr int kIn = 4096 / NT; // (at most 4096 segments)
    u64 M[kIn];
#pragma unroll
    for (int j = 0; j < kIn; ++j) {
        const int i = j * NT + tid;
        M[j] = 0;
        if (j > 0 && j * NT >= n_seg) break;
        if (i < n_seg) M[j] = p.uniform_q ? (u64)(bounds[i + 1] - bounds[i]) // ablation: share by length
                                          : (i + 1 < n_seg ? Ms[i + 1] : SH) - Ms[i];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kIn; ++j) {
        const int i = j * NT + tid;
        if (i >= n_seg) break;
        const int L = bounds[i + 1] - bounds[i];
        u64 qi = (u64)max(0, min(p.q_min, L));
        if (Trem >= 0) qi += quotient(2ull * (u64)Trem * M[j] + SHq, 2ull * SHq, inv);
        if (qi > (u64)L) qi = (u64)L; // (whatever the masses are)
        Ms[i] = M[j];
        quota[i] = (int)qi;
        sq += (int)qi;
    }
    const int Dq = Bq - block_count<NT>(sq, round, sh);
    if (Dq != 0) {
        for (int i = tid; i < n_seg; i += NT) {
            const int L = bounds[i + 1] - bounds[i];
            cap[i] = Dq > 0 ? L - quota[i] : quota[i] - max(0, min(p.q_min, L));
        }
        __syncthreads();
        const int left = block_distribute<NT>(Dq > 0 ? 1 : -1, abs(Dq), cap, quota, Ms, n_seg, sh);
        if (Dq < 0 && left > 0) { // the budget cannot cover the minima: go below them
            for (int i = tid; i < n_seg; i += NT) cap[i] = quota[i];
            __syncthreads();
            block_distribute<NT>(-1, left, cap, quota, Ms, n_seg, sh);
        }
    }
    return n_seg;
}

// ------------------------------------------------------------------------------------------ searches

struct Cut { unsigned key; int ties; }; // the keys above `key` win, and `ties` of those equal to it (-1: all of them)

// *word += 1 where d <= w, as a predicated instruction (a branch around each of a lane's increments costs more than they do).
__device__ __forceinline__ void count_if(unsigned *word, unsigned d, unsigned w)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %1, %2;\n\t@p red.shared.add.u32 [%0], 1;\n\t}"
                 ::"r"((unsigned)__cvta_generic_to_shared(word)), "r"(d), "r"(w) : "memory");
}

// Bin of a warp's histogram that holds the q-th key from the top (1 <= q <= number of keys counted, at most 1023 keys): bin,
// keys in it, keys above it.
__device__ __forceinline__ void find_bin(const unsigned *hist, int q, int &bin, int &m, int &above)
{
    const int lane = threadIdx.x & 31;
    const uint4 v = reinterpret_cast<const uint4 *>(hist)[31 - lane]; // lane 0 has the top four bins
    const int c0 = (int)v.w, c1 = c0 + (int)v.z, c2 = c1 + (int)v.y, c3 = c2 + (int)v.x;
    const int inc = warp_incl_scan(c3), exc = inc - c3, rest = q - exc;
    const int src = __ffs(__ballot_sync(kFull, inc >= q)) - 1; // the first lane that covers q
    const int i = (rest > c0) + (rest > c1) + (rest > c2);
    const int below = rest > c2 ? c2 : (rest > c1 ? c1 : (rest > c0 ? c0 : 0)), upto = rest > c2 ? c3 : (rest > c1 ? c2 : (rest > c0 ? c1 : c0));
    const unsigned mine = (unsigned)(127 - lane * 4 - i) | (unsigned)(upto - below) << 8 | (unsigned)(exc + below) << 18;
    const unsigned got = __shfl_sync(kFull, mine, src);
    bin = (int)(got & 255u); m = (int)((got >> 8) & 1023u); above = (int)(got >> 18);
}

// The q-th largest (0 < q < n) of n keys in a warp's registers, kPL per lane, key number j * 32 + lane in register j, unused
// registers 0.  hist: kWarpBins words of the warp's own.
template <int kPL>
__device__ __forceinline__ Cut warp_cut(const unsigned (&k)[kPL], int n, int q, unsigned *hist)
{
    const int lane = threadIdx.x & 31, room = n - lane;
    unsigned mx = 0u, mn = kFull;
#pragma unroll
    for (int j = 0; j < kPL; ++j) {
        mx = max(mx, k[j]);
        mn = min(mn, j * 32 < room ? k[j] : kFull);
    }
    mx = __reduce_max_sync(kFull, mx);
    mn = __reduce_min_sync(kFull, mn);
    if (mn == mx) return {mn, q};
    if (mn == 0u) { // NaN scores (and unused registers) stay out of the histogram
        int c = 0;
        mn = kFull;
#pragma unroll
        for (int j = 0; j < kPL; ++j) { c += k[j] > 0u; mn = min(mn, k[j] - 1u); }
        c = warp_sum(c);
        if (c < q) return {0u, q - c};
        mn = __reduce_min_sync(kFull, mn) + 1u;
    }
    unsigned lo = mn, w = mx - mn;
    for (;;) {
        const int shift = max(0, 25 - __clz(w)); // w >> shift < kWarpBins
        reinterpret_cast<uint4 *>(hist)[lane] = make_uint4(0, 0, 0, 0);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kPL; ++j) {
            const unsigned d = k[j] - lo;
            count_if(&hist[d >> shift], d, w);
        }
        __syncwarp();
        int bin, m, above;
        find_bin(hist, q, bin, m, above);
        q -= above;
        lo += (unsigned)bin << shift;
        if (q == m) return {lo, -1};
        w = min((1u << shift) - 1u, w - ((unsigned)bin << shift));
        if (w == 0u) return {lo, q};
        if (m <= 4) break;
        __syncwarp();
    }
    for (;;) { // few keys are left in [lo, lo + w]: from the largest down
        unsigned v = 0u;
#pragma unroll
        for (int j = 0; j < kPL; ++j) { const unsigned d = k[j] - lo; v = max(v, d <= w ? d : 0u); }
        v = __reduce_max_sync(kFull, v);
        int c = 0;
#pragma unroll
        for (int j = 0; j < kPL; ++j) c += k[j] - lo == v;
        c = warp_sum(c);
        if (c >= q) return {lo + v, c == q ? -1 : q};
        q -= c;
        w = v - 1u;
    }
}

// The usual case of the search: at least q keys are known to lie in [lo, lo + w], the range is narrow, and a histogram over it
// leaves few keys in the bin of the q-th one, of which the smallest are dropped one by one.  Returns the key from which on
// q keys lie, unless some are equal (the caller counts).  Unused registers must lie outside the range.
template <int kPL>
__device__ __forceinline__ unsigned warp_cut_fast(const unsigned (&k)[kPL], int q, unsigned lo, unsigned w, unsigned *hist)
{
    const int lane = threadIdx.x & 31;
    int bin, m, above;
    do {
        const int shift = max(0, 25 - __clz(w)); // w >> shift < kWarpBins
        __syncwarp();
        reinterpret_cast<uint4 *>(hist)[lane] = make_uint4(0, 0, 0, 0);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kPL; ++j) { const unsigned d = k[j] - lo; count_if(&hist[d >> shift], d, w); }
        __syncwarp();
        find_bin(hist, q, bin, m, above);
        lo += (unsigned)bin << shift;
        q -= above;
        w = min((1u << shift) - 1u, w - ((unsigned)bin << shift));
    } while (m - q > 4 && w > 0u); // crowded: another histogram over the bin
    for (; q < m; --m) {
        unsigned v = kFull;
#pragma unroll
        for (int j = 0; j < kPL; ++j) { const unsigned d = k[j] - lo; v = min(v, d <= w ? d : kFull); }
        v = __reduce_min_sync(kFull, v);
        if (v >= w) break; // (equal keys)
        lo += v + 1u;
        w -= v + 1u;
    }
    return lo;
}

// Kept bits of a piece of at most kPiece tokens from position a: lane j's word holds tokens a + 32 j .., shifted onto
// the words of the mask.
__device__ __forceinline__ void mask_or(unsigned *mask, int a, unsigned word)
{
    const int lane = threadIdx.x & 31;
    const unsigned prev = __shfl_up_sync(kFull, word, 1);
    const unsigned w = __funnelshift_l(lane ? prev : 0u, word, a & 31);
    if (lane <= kPer && w) atomicOr(&mask[(a >> 5) + lane], w);
}

// Best rejected key of a piece (slots beyond the table share entries), and of all that this lane has seen.
__device__ __forceinline__ void note_best(unsigned *best, int slot, unsigned key, unsigned &lane_best)
{
    lane_best = max(lane_best, key);
    key = __reduce_max_sync(kFull, key);
    if ((threadIdx.x & 31) == 0) atomicMax(&best[slot & (kBest - 1)], key);
}

__device__ __forceinline__ void load_piece(const float *g, int a, int len, float (&x)[kPer])
{
    const float *src = g + a + (threadIdx.x & 31);
    const int room = len - (int)(threadIdx.x & 31);
#pragma unroll
    for (int j = 0; j < kPer; ++j) x[j] = j * 32 < room ? src[j * 32] : 0.0f;
}

// One segment of at most kPiece tokens.
__device__ __forceinline__ void warp_segment(const float (&x)[kPer], unsigned *mask, unsigned *best, unsigned *hist, int slot, unsigned &lane_best,
                                             int a, int L, int q, int ns, int t_last)
{
    const int lane = threadIdx.x & 31, room = L - lane;
    const bool plain = a >= ns && a + L <= t_last; // no must-keep position in it
    auto may_fill = [&](int j) { return plain || (a + j * 32 + lane >= ns && a + j * 32 + lane < t_last); };
    unsigned k[kPer], word = 0, rej = 0, mine = 0u;
#pragma unroll
    for (int j = 0; j < kPer; ++j) { k[j] = __float_as_uint(x[j]); mine = max(mine, k[j]); }
    const bool pos = __reduce_max_sync(kFull, mine) <= 0x7f800000u; // no negative score, no NaN: the bit patterns ascend
    if (!pos) {
        mine = 0u;
#pragma unroll
        for (int j = 0; j < kPer; ++j) { k[j] = j * 32 < room ? score_key(x[j]) : 0u; mine = max(mine, k[j]); }
    }
    bool done = false;
    if (q >= L) { // all of it
        const int n = min(32, max(0, L - lane * 32));
        word = n > 0 ? kFull >> (32 - n) : 0u;
        done = true;
    } else if (q > 0 && L >= 2 * 32) {
        // A narrow range that holds the q-th key: 32 (64) keys lie at or above the smallest of the lanes' largest (second
        // largest) keys, and as many at or below the largest of their smallest (second smallest) ones.
        unsigned top = mine, lo, hi;
        int q_in = q; // its number from the top within the range
        if (q <= 2 * 32) {
            if (q > 32) {
                unsigned first = 0u;
                top = 0u;
#pragma unroll
                for (int j = 0; j < kPer; ++j) { top = max(top, min(first, k[j])); first = max(first, k[j]); }
            }
            lo = __reduce_min_sync(kFull, top);
            hi = __reduce_max_sync(kFull, mine);
        } else {
            unsigned first = kFull, second = kFull;
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const unsigned v = j * 32 < room ? k[j] : kFull;
                second = min(second, max(first, v));
                first = min(first, v);
            }
            lo = __reduce_min_sync(kFull, first);
            hi = __reduce_max_sync(kFull, L - q < 32 ? first : (L - q < 2 * 32 ? second : mine));
            int above = 0;
#pragma unroll
            for (int j = 0; j < kPer; ++j) above += k[j] > hi;
            q_in = q - warp_sum(above);
        }
        if (lo > 0u && lo < hi) {
            const unsigned key = warp_cut_fast<kPer>(k, q_in, lo, hi - lo, hist);
            unsigned b[kPer];
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const bool kept = k[j] >= key;
                b[j] = __ballot_sync(kFull, kept);
                if (!kept && may_fill(j)) rej = max(rej, k[j]);
            }
            const bool l0 = lane & 1, l1 = lane & 2, l2 = lane & 4;
            const unsigned w0 = l0 ? b[1] : b[0], w1 = l0 ? b[3] : b[2], w2 = l0 ? b[5] : b[4], w3 = l0 ? b[7] : b[6];
            const unsigned v0 = l1 ? w1 : w0, v1 = l1 ? w3 : w2;
            word = lane < kPer ? (l2 ? v1 : v0) : 0u;
            done = warp_sum(__popc(word)) == q;
            if (pos) {
                if (__any_sync(kFull, rej == 0u)) { // nothing rejected, or scores of 0, which unused registers look like
                    bool zero = false;
#pragma unroll
                    for (int j = 0; j < kPer; ++j) zero |= j * 32 < room && k[j] == 0u && may_fill(j);
                    rej = rej | (rej || zero ? 0x80000000u : 0u);
                } else {
                    rej |= 0x80000000u;
                }
            }
        }
    }
    if (!done) {
        if (pos) {
#pragma unroll
            for (int j = 0; j < kPer; ++j) k[j] = j * 32 < room ? k[j] | 0x80000000u : 0u;
        }
        Cut cut = {kFull, 0};                // none of it
        if (q > 0) cut = warp_cut<kPer>(k, L, q, hist);
        int seen = 0;
        word = 0; rej = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) { // ties: the first ones in position order
            const bool in = j * 32 < room, tie = in && k[j] == cut.key;
            const unsigned tb = __ballot_sync(kFull, tie);
            const bool kept = in && (k[j] > cut.key || (tie && (cut.ties < 0 || seen + __popc(tb & ((1u << lane) - 1u)) < cut.ties)));
            seen += __popc(tb);
            const unsigned bal = __ballot_sync(kFull, kept);
            if (lane == j) word = bal;
            if (!kept && may_fill(j)) rej = max(rej, k[j]);
        }
    }
    mask_or(mask, a, word);
    note_best(best, slot, rej, lane_best);
}

// Walks the pieces of the batch's long segments, a run of consecutive pieces per warp, the next piece's scores on their way
// while f(i, piece, a, len, x) works on this one's; i is the segment's entry in the table, enter(i) announces it.
template <int NT, typename Enter, typename F>
__device__ __forceinline__ void walk_long(const float *g, const int *bounds, const SegTab &tb, int n, Enter enter, F f)
{
    constexpr int NW = NT / 32;
    const int warp = threadIdx.x >> 5, n_piece = tb.piece0[n];
    const int p0 = (int)((long long)n_piece * warp / NW), p1 = (int)((long long)n_piece * (warp + 1) / NW);
    if (p0 >= p1) return;
    int i = 0;
    for (int hi = n; hi - i > 1;) {
        const int mid = (i + hi) >> 1;
        if (tb.piece0[mid] <= p0) i = mid; else hi = mid;
    }
    int next = tb.piece0[i + 1], e = bounds[tb.seg[i] + 1], a = bounds[tb.seg[i]] + (p0 - tb.piece0[i]) * kPiece;
    float x[kPer];
    load_piece(g, a, e - a, x);
    enter(i);
    for (int pc = p0; pc < p1; ++pc) {
        float y[kPer];
        const int ca = a, cl = min(kPiece, e - a), ci = i;
        if (pc + 1 < p1) {
            a += kPiece;
            if (pc + 1 == next) { ++i; next = tb.piece0[i + 1]; a = bounds[tb.seg[i]]; e = bounds[tb.seg[i] + 1]; }
            load_piece(g, a, e - a, y);
        }
        f(ci, pc, ca, cl, x);
        if (i != ci) enter(i);
#pragma unroll
        for (int j = 0; j < kPer; ++j) x[j] = y[j];
    }
}

// A warp finds the bin of long segment i that holds its q-th key and what is left to decide in it.
__device__ __forceinline__ void find_long_bin(SegTab &tb, const unsigned *hist, int nb, int i, int q)
{
    const int lane = threadIdx.x & 31;
    const uint4 *h4 = reinterpret_cast<const uint4 *>(hist + i * nb);
    int above = tb.above[i];
    uint4 v = make_uint4(0, 0, 0, 0);
    int c = (nb + 127) / 128 - 1, sum = 0;
    for (;; --c) { // 128 bins at a time from the top
        const int k = c * 32 + lane;
        v = k * 4 < nb ? h4[k] : make_uint4(0, 0, 0, 0);
        sum = (int)(v.x + v.y + v.z + v.w);
        above += warp_sum(sum);
        if (c == 0 || above >= q) break;
    }
    const int before = above - warp_incl_scan(sum); // keys in the lanes (bins) above this one's, and above the range
    if (before < q && q <= before + sum) {
        int run = before, bin = 0, m = 0;
        const int cnt[4] = {(int)v.w, (int)v.z, (int)v.y, (int)v.x};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (run < q && q <= run + cnt[j]) { bin = c * 128 + lane * 4 + 3 - j; m = cnt[j]; above = run; }
            run += cnt[j];
        }
        const unsigned sft = tb.shift[i], rl = tb.rl[i], rh = rl + tb.rw[i], first = tb.lo[i] + ((unsigned)bin << sft);
        const unsigned L = bin == 0 ? rl : first, w = bin == nb - 1 ? rh - L : min(rh - L, first - L + (1u << sft) - 1u);
        const int r = q - above;
        tb.above[i] = above;
        tb.r[i] = r;
        tb.m[i] = m;
        tb.L[i] = L;
        tb.U[i] = r == m ? L : L + w + 1u;
        tb.state[i] = r == m ? kDone : (w == 0u ? kTies : kSearch);
    }
}

__device__ __forceinline__ int bin_shift(unsigned w, int nb) // smallest shift with w >> shift < nb
{
    return max(0, __clz(nb) + 1 - __clz(w)); // nb a power of two: log2(nb) = 31 - clz(nb)
}

// Top-q_i of the n <= kBatch long segments of the table: kept bits into mask, best rejected keys (must-keep positions
// apart) into `best`, pieces taking the slots from slot0 on.
template <int NT>
__device__ void select_long(const float *g, const int *bounds, const int *quota, int n, unsigned *mask, unsigned *best, int slot0, unsigned &lane_best,
                            SegTab &tb, unsigned *hist, uint2 *list, int ns, int t_last, SelShared &sh)
{
    constexpr int NW = NT / 32, kList = Tune<NT>::kList;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int nb = Tune<NT>::kBins / n;
    nb = min(kMaxBins, 1 << (31 - __clz(nb)));

    // ---- walk 1: the bins of a segment cover the kOctaves octaves (2^23 keys each) below its largest key, judged by a
    //      quarter of the tokens: scores below that hardly ever hold the threshold, whatever their sign, and what does
    //      lie outside falls into the first or the last bin
    uint4 *h4 = reinterpret_cast<uint4 *>(hist);
    for (int i = tid; i < n * nb / 4; i += NT) h4[i] = make_uint4(0, 0, 0, 0);
    for (int i = warp; i < n; i += NW) { // (32 tokens of every 128, at most 64 such groups)
        const int a = bounds[tb.seg[i]], len = bounds[tb.seg[i] + 1] - a, q = quota[tb.seg[i]], step = max(128, (len >> 6) & ~31);
        unsigned hi = 0u;
        for (int t0 = lane; t0 < len; t0 += 8 * step) {
            float x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = t0 + j * step < len ? g[a + t0 + j * step] : __uint_as_float(0x7fffffffu);
#pragma unroll
            for (int j = 0; j < 8; ++j) hi = max(hi, score_key(x[j]));
        }
        hi = __reduce_max_sync(kFull, hi);
        if (lane == 0) {
            constexpr unsigned span = kOctaves << 23;
            const unsigned lo = hi > span ? hi - span : 0u;
            int state = kSearch;
            unsigned L = 0u, U = kFull; // (no key is as large as kFull)
            if (q <= 0) { state = kDone; L = kFull; }
            else if (q >= len) { state = kDone; U = 0u; }
            tb.L[i] = L; tb.U[i] = U;
            tb.lo[i] = lo; tb.rl[i] = 0u; tb.rw[i] = kFull - 1u;
            tb.above[i] = 0; tb.r[i] = q; tb.m[i] = len;
            tb.state[i] = (unsigned char)state;
            tb.shift[i] = (unsigned char)(state == kSearch ? bin_shift(hi - lo, nb) : 255);
        }
    }
    __syncthreads();

    // ---- walk 2: histograms, and again over the threshold's bin where that is still crowded
    for (;;) {
        {
            unsigned lo = 0u, rl = 0u, rw = 0u, sft = 255u;
            unsigned *mine = hist;
            walk_long<NT>(g, bounds, tb, n,
                          [&](int i) { lo = tb.lo[i]; rl = tb.rl[i]; rw = tb.rw[i]; sft = tb.shift[i]; mine = hist + i * nb; },
                          [&](int, int, int, int len, const float (&x)[kPer]) {
                              if (sft >= 32u) return;
#pragma unroll
                              for (int j = 0; j < kPer; ++j) {
                                  const unsigned k = score_key(x[j]), b = min((max(k, lo) - lo) >> sft, (unsigned)(nb - 1));
                                  count_if(&mine[b], j * 32 + lane < len ? k - rl : kFull, rw); // (rw < kFull)
                              }
                          });
        }
        __syncthreads();
        for (int i = warp; i < n; i += NW)
            if (tb.shift[i] < 32) find_long_bin(tb, hist, nb, i, quota[tb.seg[i]]);
        __syncthreads();
        // room in the list: segments in order, each with its m candidates
        if (warp == 0) {
            int tot = 0;
            for (int i0 = 0; i0 < n; i0 += 32) {
                const int i = i0 + lane, m = i < n && tb.state[i] == kSearch ? tb.m[i] : 0;
                const int inc = warp_incl_scan(m);
                if (i < n) tb.base[i] = tb.cnt[i] = tot + inc - m;
                tot += __shfl_sync(kFull, inc, 31);
            }
            if (lane == 0) sh.total = tot;
        }
        __syncthreads();
        const int limit = sh.total > kList ? kList / kBatch : 256; // most candidates of a segment that are ranked pairwise
        bool again = false;
        for (int i = tid; i < n; i += NT) {
            tb.shift[i] = 255;
            if (tb.state[i] == kSearch && tb.m[i] > limit) {
                const unsigned w = tb.U[i] - 1u - tb.L[i];
                tb.lo[i] = tb.rl[i] = tb.L[i]; tb.rw[i] = w;
                tb.shift[i] = (unsigned char)bin_shift(w, nb);
                again = true;
            }
        }
        if (!__syncthreads_or(again)) break;
        for (int i = warp; i < n; i += NW)
            if (tb.shift[i] < 32)
                for (int k = lane; k < nb; k += 32) hist[i * nb + k] = 0u;
        __syncthreads();
    }

    // ---- walk 3: kept bits, candidates, best rejected keys
    {
        unsigned L = 0u, U = 0u;
        bool search = false;
        walk_long<NT>(g, bounds, tb, n, [&](int i) { L = tb.L[i]; U = tb.U[i]; search = tb.state[i] == kSearch; },
                      [&](int i, int pc, int a, int len, const float (&x)[kPer]) {
                          const bool plain = a >= ns && a + len <= t_last; // no must-keep position in it
                          unsigned word = 0, rej = 0, cand = 0;
#pragma unroll
                          for (int j = 0; j < kPer; ++j) {
                              const bool in = j * 32 + lane < len;
                              const unsigned k = score_key(x[j]);
                              const unsigned bal = __ballot_sync(kFull, in && k >= U);
                              if (lane == j) word = bal;
                              if (k < L) {
                                  if (in && (plain || (a + j * 32 + lane >= ns && a + j * 32 + lane < t_last))) rej = max(rej, k);
                              } else if (in && k < U) {
                                  cand |= 1u << j;
                              }
                          }
                          if (search && __any_sync(kFull, cand)) {
#pragma unroll
                              for (int j = 0; j < kPer; ++j)
                                  if ((cand >> j) & 1u)
                                      list[atomicAdd(&tb.cnt[i], 1)] = make_uint2(score_key(x[j]), (unsigned)(a + j * 32 + lane) | ((unsigned)i << 24));
                          }
                          mask_or(mask, a, word);
                          note_best(best, slot0 + pc, rej, lane_best);
                      });
    }
    __syncthreads();
    auto rejected = [&](unsigned key, int i, int t) { // a candidate that did not make it
        const int slot = slot0 + tb.piece0[i] + (t - bounds[tb.seg[i]]) / kPiece;
        if (t >= ns && t < t_last) {
            atomicMax(&best[slot & (kBest - 1)], key);
            lane_best = max(lane_best, key);
        }
    };
    for (int c = tid; c < sh.total; c += NT) { // every candidate ranks itself
        const uint2 v = list[c];
        const int i = (int)(v.y >> 24), t = (int)(v.y & 0xffffffu);
        const int b = tb.base[i], e = b + tb.m[i];
        int rank = 0;
        for (int j = b; j < e; ++j) {
            const uint2 o = list[j];
            rank += o.x > v.x || (o.x == v.x && o.y < v.y); // (same segment: y orders by position)
        }
        if (rank < tb.r[i]) atomicOr(&mask[t >> 5], 1u << (t & 31));
        else rejected(v.x, i, t);
    }
    for (int i = warp; i < n; i += NW) { // ties across the threshold: the first r of them in position order
        if (tb.state[i] != kTies) continue;
        const unsigned key = tb.L[i];
        const int s = tb.seg[i], a = bounds[s], e = bounds[s + 1], r = tb.r[i];
        int seen = 0;
        for (int t0 = a; t0 < e; t0 += 32) {
            const int t = t0 + lane;
            const bool tie = t < e && score_key(g[t]) == key;
            const unsigned bal = __ballot_sync(kFull, tie);
            if (tie) {
                if (seen + __popc(bal & ((1u << lane) - 1u)) < r) atomicOr(&mask[t >> 5], 1u << (t & 31));
                else rejected(key, i, t);
            }
            seen += __popc(bal);
        }
    }
    __syncthreads();
}

// Top-q (q > 0) of the tokens for which ok(t) holds, by the whole block, with the scores read again in every round: the
// form that needs no room, for a backfill that the short list could not hold (ties by the hundred, NaN scores).
template <int NT, typename Ok, typename Keep>
__device__ void block_select_stream(const float *g, int T, int q, SelShared &sh, int &round, Ok ok, Keep keep)
{
    const int tid = threadIdx.x;
    unsigned P = 0; // the largest key with count(>= P) >= q, bit by bit
    bool exact = false;
    for (int bit = 31; bit >= 0; --bit) {
        const unsigned X = P | (1u << bit);
        int c = 0;
        for (int t = tid; t < T; t += NT) c += ok(t) && score_key(g[t]) >= X;
        const int tot = block_count<NT>(c, round, sh);
        if (tot >= q) {
            P = X;
            if (tot == q) { exact = true; break; }
        }
    }
    int last = T - 1; // ties at P count up to this position
    if (!exact) {
        int c = 0;
        for (int t = tid; t < T; t += NT) c += ok(t) && score_key(g[t]) > P;
        const int take = q - block_count<NT>(c, round, sh);
        int l = 0, r = T - 1;
        while (l < r) {
            const int mid = (l + r) >> 1;
            c = 0;
            for (int t = tid; t <= mid; t += NT) c += ok(t) && score_key(g[t]) == P;
            if (block_count<NT>(c, round, sh) >= take) r = mid; else l = mid + 1;
        }
        last = l;
    }
    for (int t = tid; t < T; t += NT) {
        if (!ok(t)) continue;
        const unsigned key = score_key(g[t]);
        if (key > P || (key == P && t <= last)) keep(t);
    }
}

// -------------------------------------------------------------------------------------- k_select_compact

// Steps 1-5 of one unit, by the block.
template <int NT>
__device__ __forceinline__ void select_unit(const DevParams &p, int longs, int uid, unsigned char *dyn, SelShared &sh)
{
    constexpr int NW = NT / 32, kList = Tune<NT>::kList;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int h = uid % p.H, bq = (uid / p.H) % p.B, l = uid / (p.H * p.B);
    const int T = seq_len_of(p, bq), bad = p.seq_lens ? p.seq_bad[bq] & kBadScores : 0; // (the allocation-free entry point has no scorer)
    if (T <= p.Tk || T > p.T_cap || bad) return; // (bad: no scores to go by)
    const int sc = p.seg_cap;
    const SelSmem mp = sel_smem<NT>(p.T_cap, sc, p.S, longs != 0);
    unsigned *mask = reinterpret_cast<unsigned *>(dyn + mp.mask);
    int *bounds = reinterpret_cast<int *>(dyn + mp.bounds);
    int *quota = reinterpret_cast<int *>(dyn + mp.quota);
    unsigned *best = reinterpret_cast<unsigned *>(dyn + mp.best);
    unsigned *hist = reinterpret_cast<unsigned *>(dyn + mp.hist) + warp * kWarpBins;
    uint2 *list = reinterpret_cast<uint2 *>(dyn + mp.list); // (key, position) of candidates
    SegTab &tb = *reinterpret_cast<SegTab *>(dyn + mp.tab);
    u64 *look_at = reinterpret_cast<u64 *>(dyn + mp.hist);  // pieces the backfill looks at: position, length
    const size_t row = (size_t)uid * p.T_cap;
    const float *g = p.scores + row;
    int *keep = p.keep_idx + (size_t)uid * p.Tk;
    const int n_words = (T + 31) >> 5;
    const int ns = max(0, min(p.n_sink, min(p.Tk, T)));           // must-keep prefix and suffix
    const int nl = max(0, min(p.n_last, min(p.Tk - ns, T - ns)));
    const int t_last = T - nl;
    int round = 0;
    for (int i = tid; i <= n_words; i += NT) mask[i] = 0u;
    for (int i = tid; i < kBest; i += NT) best[i] = 0u;
    if (tid == 0) { sh.n_list = 0; sh.n_look = 0; sh.bound = 0u; }
    float *credit = p.ema ? p.ema + (((size_t)l * p.Bmax + bq) * p.H + h) * (size_t)p.T_cap : nullptr;
    Mass ms;
    u64 *wsum = reinterpret_cast<u64 *>(dyn + mp.list);
    const u64 SH = mass_of_unit<NT>(p, uid, T, credit, wsum, ms, sh);
    const int n_seg = segments_and_quotas<NT>(p, T, p.Tk - ns - nl, ms, wsum, SH, reinterpret_cast<u64 *>(dyn + mp.ms), bounds, quota,
                                              reinterpret_cast<int *>(dyn + mp.hist), sh, round);
    if (n_seg < 0) { // cannot happen with the capacity formula of the header; reported all the same
        if (tid == 0) { set_status(p.status, AMS_ERR_CAPACITY, uid, sh.n_seg, sc); p.n_seg[uid] = -1; atomicOr(&p.seq_bad[bq], kBadUnit); }
        return;
    }
    __syncthreads();
    if (p.seg_out) { // inspection
        if (tid == 0) { p.n_seg[uid] = n_seg; p.seg_bounds[(size_t)uid * (sc + 1) + n_seg] = T; }
        for (int i = tid; i < n_seg; i += NT) {
            p.seg_bounds[(size_t)uid * (sc + 1) + i] = bounds[i];
            p.quotas[(size_t)uid * sc + i] = quota[i];
        }
    }

    // ---- per-segment top-q_i.  Slots of the table of best rejected keys: short segment sg takes sg, the pieces of long
    //      ones those behind.  The next segment's scores are fetched before the current one is searched.
    unsigned lane_best = 0u; // best key this lane has seen rejected
    {
        float xn[kPer];
        auto fetch = [&](int sg) {
            if (sg < n_seg) load_piece(g, bounds[sg], min(kPiece, bounds[sg + 1] - bounds[sg]), xn);
        };
        fetch(warp);
        for (int sg = warp; sg < n_seg; sg += NW) {
            const int a = bounds[sg], L = bounds[sg + 1] - a, q = quota[sg];
            float x[kPer];
#pragma unroll
            for (int j = 0; j < kPer; ++j) x[j] = xn[j];
            fetch(sg + NW);
            if (L <= kPiece) warp_segment(x, mask, best, hist, sg, lane_best, a, L, q, ns, t_last);
        }
    }
    int n_slot = n_seg;
    if (longs) {
        for (int s0 = 0; s0 < n_seg;) { // batches of long segments
            __syncthreads();
            if (warp == 0) {
                int n = 0, pc = 0, sg = s0;
                for (; sg < n_seg && n <= kBatch - 32; sg += 32) {
                    const int i = sg + lane, len = i < n_seg ? bounds[i + 1] - bounds[i] : 0;
                    const bool is = len > kPiece;
                    const unsigned bal = __ballot_sync(kFull, is);
                    const int c = is ? (len + kPiece - 1) / kPiece : 0, inc = warp_incl_scan(c), at = n + __popc(bal & ((1u << lane) - 1u));
                    if (is) { tb.seg[at] = (unsigned short)i; tb.piece0[at] = pc + inc - c; }
                    n += __popc(bal);
                    pc += __shfl_sync(kFull, inc, 31);
                }
                if (lane == 0) { tb.piece0[n] = pc; sh.n_long = n; sh.level = sg; }
            }
            __syncthreads();
            s0 = sh.level;
            const int n = sh.n_long;
            if (n > 0) {
                const int n_pc = tb.piece0[n];
                select_long<NT>(g, bounds, quota, n, mask, best, n_slot, lane_best, tb, reinterpret_cast<unsigned *>(dyn + mp.hist), list, ns, t_last, sh);
                n_slot += n_pc;
            }
        }
    }
    // groups of eight lanes: the tokens they have seen
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) lane_best = max(lane_best, __shfl_xor_sync(kFull, lane_best, d));
    if ((lane & 7) == 0) sh.gbest[warp * 4 + (lane >> 3)] = lane_best;
    __syncthreads();

    // ---- must-keep prefix and suffix; every must-keep position a segment already chose frees one slot,
    //      refilled by the best positions not yet kept (top r_fill of the unflagged tokens of the sequence)
    int already = 0;
    for (int i = tid; i < ns + nl; i += NT) {
        const int t = i < ns ? i : t_last + (i - ns);
        already += (atomicOr(&mask[t >> 5], 1u << (t & 31)) >> (t & 31)) & 1u;
    }
    const int r_fill = block_count<NT>(already, round, sh);
    if (r_fill > 0) {
        // At least r_fill unflagged tokens lie at or above the r_fill-th largest of the groups' best rejected keys, so
        // only pieces whose best one reaches that bound can hold a winner; their tokens at or above it go to a list.
        if (warp == 0) {
            unsigned k[NW / 8], M = 0u; // (0: too few groups, every token is looked at)
            int c = 0;
#pragma unroll
            for (int j = 0; j < NW / 8; ++j) { k[j] = sh.gbest[j * 32 + lane]; c += k[j] > 0u; }
            if (warp_sum(c) >= r_fill) M = warp_cut<NW / 8>(k, NW * 4, r_fill, hist).key;
            if (lane == 0) sh.bound = M;
        }
        __syncthreads();
        const unsigned M = sh.bound;
        auto raise = [&](int t) { atomicOr(&mask[t >> 5], 1u << (t & 31)); };
        auto unflagged = [&](int t) { return ((mask[t >> 5] >> (t & 31)) & 1u) == 0u; };
        const float least = M ? __uint_as_float((M & 0x80000000u) ? M ^ 0x80000000u : ~M) : -INFINITY;
        auto look = [&](int a, int len) { // a piece, by one warp
            float x[kPer];
            load_piece(g, a, len, x);
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const int t = a + j * 32 + lane;
                if (!(x[j] < least) && j * 32 + lane < len && unflagged(t)) { // (NaN too: a candidate that ranks last)
                    const int at = atomicAdd(&sh.n_list, 1);
                    if (at < kList) list[at] = make_uint2(score_key(x[j]), (unsigned)t);
                }
            }
        };
        // pieces that reach the bound go to a list of their own
        auto note = [&](int slot, int a, int len) {
            if (best[slot & (kBest - 1)] < M) return;
            const int at = atomicAdd(&sh.n_look, 1);
            if (at < kBest) look_at[at] = (u64)(unsigned)a << 32 | (unsigned)len;
        };
        if (!longs) {
            for (int sg = tid; sg < n_seg; sg += NT) note(sg, bounds[sg], bounds[sg + 1] - bounds[sg]);
        } else {
            int slot = n_seg;
            for (int sg = 0; sg < n_seg; ++sg) {
                const int a = bounds[sg], L = bounds[sg + 1] - a;
                if (L <= kPiece) {
                    if (sg % NT == tid) note(sg, a, L);
                } else {
                    const int n_pc = (L + kPiece - 1) / kPiece;
                    for (int i = tid; i < n_pc; i += NT) note(slot + i, a + i * kPiece, min(kPiece, L - i * kPiece));
                    slot += n_pc;
                }
            }
        }
        __syncthreads();
        const int n_look = sh.n_look;
        if (n_look <= kBest) {
            for (int i = warp; i < n_look; i += NW) look((int)(look_at[i] >> 32), (int)(unsigned)look_at[i]);
        } else { // (a bound of 0, or hundreds of pieces with equal keys)
            for (int a = warp * kPiece; a < T; a += NW * kPiece) look(a, min(kPiece, T - a));
        }
        __syncthreads();
        const int n_list = sh.n_list;
        if (n_list > kList) {
            block_select_stream<NT>(g, T, r_fill, sh, round, unflagged, raise);
        } else {
            for (int i = warp; i < n_list; i += NW) { // every candidate is ranked by a warp
                const uint2 v = list[i];
                int rank = 0;
                for (int j = lane; j < n_list; j += 32) {
                    const uint2 o = list[j];
                    rank += o.x > v.x || (o.x == v.x && o.y < v.y);
                }
                if (warp_sum(rank) < r_fill && lane == 0) raise((int)v.y);
            }
        }
    }
    __syncthreads();

    // ---- ordered compaction of the kept positions: a warp takes a run of mask words, a lane a bit of the current one
    const int wpw = (n_words + NW - 1) / NW, w0 = warp * wpw, w1 = min(n_words, w0 + wpw);
    int n_kept = 0;
    for (int w = w0 + lane; w < w1; w += 32) n_kept += __popc(mask[w]);
    n_kept = warp_sum(n_kept);
    if (lane == 0) sh.wc[0][warp] = n_kept;
    __syncthreads();
    int pos = warp_sum(lane < warp ? sh.wc[0][lane] : 0);
    const int total = warp_sum(lane < NW ? sh.wc[0][lane] : 0);
    if (total != p.Tk) {
        if (tid == 0) { set_status(p.status, AMS_ERR_INTERNAL, uid, total, p.Tk); atomicOr(&p.seq_bad[bq], kBadUnit); }
        return;
    }
    for (int g0 = w0; g0 < w1; g0 += 32) {
        const unsigned mine = g0 + lane < w1 ? mask[g0 + lane] : 0u;
        const int inc = warp_incl_scan(__popc(mine)), at = pos + inc - __popc(mine);
        if (__shfl_sync(kFull, inc, 31) > 256) { // dense: a word after the other, a bit per lane (coalesced)
            const int n = min(32, w1 - g0);
#pragma unroll 4
            for (int i = 0; i < n; ++i) {
                const unsigned m = __shfl_sync(kFull, mine, i);
                const int b = __shfl_sync(kFull, at, i);
                if ((m >> lane) & 1u) keep[b + __popc(m & ((1u << lane) - 1u))] = (g0 + i) * 32 + lane;
            }
        } else { // sparse: every lane its own word
            int to = at;
            for (unsigned m = mine; m; m &= m - 1u) keep[to++] = (g0 + lane) * 32 + __ffs(m) - 1;
        }
        pos += __shfl_sync(kFull, inc, 31);
    }
    // ---- credit rows travel with their tokens, in place: kept positions ascend and keep[j] >= j, so what a tile
    //      writes is never read by a later one.  Rows beyond the budget start from zero.  (As extra blocks of the gather
    //      kernel, "hidden" behind the K and V rows, the same moves cost that kernel 40 us more than they take here.)
    if (p.beta != 1.0f) {
        constexpr int kIn = 4; // rows in flight per thread
        __syncthreads();
        for (int base = 0; base < p.Tk; base += NT * kIn) {
            int from[kIn];
            float c[kIn];
#pragma unroll
            for (int i = 0; i < kIn; ++i) from[i] = keep[min(base + i * NT + tid, p.Tk - 1)];
#pragma unroll
            for (int i = 0; i < kIn; ++i) c[i] = credit[from[i]];
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kIn; ++i) {
                const int j = base + i * NT + tid;
                if (j < p.Tk) credit[j] = c[i];
            }
        }
        const int z0 = min(T, (p.Tk + 3) & ~3); // first whole group of four
        for (int j = p.Tk + tid; j < z0; j += NT) credit[j] = 0.0f;
        for (int j = z0 + 4 * tid; j < T; j += 4 * NT) {
            if (j + 3 < T) *reinterpret_cast<float4 *>(credit + j) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            else for (int i = j; i < T; ++i) credit[i] = 0.0f;
        }
    }
}

template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_select_compact(DevParams p, int longs)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ SelShared sh;
    wait_for_previous_kernel(); // scores, effective lengths
    select_unit<NT>(p, longs, blockIdx.x, dyn, sh);
}

// The rest of an event in one launch: selection, row moves, block table.  Selection is bound by instructions and latency, the moves by
// HBM, so blocks doing the one run beside blocks doing the other.  A block takes a ticket from a counter when it starts: the first
// `lag` are units to select, then units and parts of the moves in turn, the moves `lag` units behind, then what is left of
// the moves.  A move waits for the units of its (layer, sequence), whose tickets all came before its own, to
// blocks that are running or through: no wait needs a block that has not started.  Whoever finishes a sequence's last part rewrites
// its row of the table, beside the others' moves (one block that rewrites 128 rows of 8192 entries at the end: event of 2048 units of 600 to 900 tokens 472 us, so 310, apart 341).  (Blocks that stay and take one ticket after the other need 200 to 800 bytes of spills, as the compiler keeps
// what does not depend on the ticket in registers throughout; this form spills 64 to 68.  `longs` is 0 in every launch, but not for
// the compiler: with that known it spills 28 to 36 bytes and orders the moves' loads so that 1792 units of 4224 tokens, budget 4096,
// take 1789 instead of 1335 us.)
struct MovePlan { int lag, parts, rows; }; // parts of a (layer, sequence), rows in each

template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_select_move(DevParams p, int longs, MovePlan plan)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ SelShared sh;
    const int tid = threadIdx.x, groups = p.L * p.B, n_sel = groups * p.H, n_mov = groups * plan.parts;
    int *finished = p.move_count + 1, *done = finished + p.B;
    wait_for_previous_kernel(); // scores, effective lengths; the counters
    if (tid == 0) {
        const int t = atomicAdd(p.move_count, 1);
        int what = t; // a unit, or n_sel + a part
        if (t >= plan.lag) {
            const long long A = n_sel - plan.lag, mixed = A + A * n_mov / n_sel, m = t - plan.lag;
            if (m < mixed) {
                const long long s = m * A / mixed;
                what = (m + 1) * A / mixed > s ? plan.lag + (int)s : n_sel + (int)(m - s);
            } else {
                what = n_sel + (int)(m - A);
            }
        }
        sh.total = what;
    }
    __syncthreads();
    const int what = sh.total;
    if (what < n_sel) {
        select_unit<NT>(p, longs, what, dyn, sh);
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(done + what / p.H) : "memory");
        }
        return;
    }
    const int part = what - n_sel, group = part / plan.parts, b = group % p.B, T = p.seq_lens[b];
    if (T > p.Tk && T <= p.T_cap) {
        if (tid == 0) {
            const int want = p.H + (p.expire_polls ? 1 : 0), limit = p.expire_polls ? (int)p.expire_polls : kMoveLimit;
            int have = 0, bad = 0;
            for (int i = 0; i < limit && !bad; ++i) {
                asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(have) : "l"(done + group) : "memory");
                if (have >= want) break;
                __nanosleep(100);
                if ((i & 255) == 255) bad = __ldcg(p.seq_bad + b);
            }
            bad = __ldcg(p.seq_bad + b);
            if (have < want && !bad) { // (only where the device stood still, or as a test)
                set_status(p.status, AMS_ERR_TIMEOUT, group * p.H, have, want);
                atomicOr(&p.seq_bad[b], kBadUnit);
            }
            sh.level = have >= want && !bad;
        }
        __syncthreads();
        if (sh.level) {
            const int r0 = (part - group * plan.parts) * plan.rows;
            move_rows<NT>(p, group / p.B, b, r0, min(p.Tk * p.H, r0 + plan.rows));
        }
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            sh.level = atomicAdd(finished + b, 1) == p.L * plan.parts - 1;
            __threadfence();
            if (sh.level && __ldcg(p.seq_bad + b)) sh.level = 0; // (no unit of the sequence is under way any more, or a move has flagged it)
        }
        __syncthreads();
        if (sh.level) update_table(p, b);
    }
}

template <int NT>
cudaError_t launch_nt(const DevParams &p, int units, bool longs, LaunchCtx &ctx)
{
    static SmemGrant grant;
    const size_t smem = sel_smem<NT>(p.T_cap, p.seg_cap, p.S, longs).total;
    if (!grant_dynamic_smem(k_select_compact<NT>, smem, grant)) return cudaErrorInvalidValue;
    return launch_after(k_select_compact<NT>, dim3((unsigned)units), dim3(NT), smem, ctx.s, p, longs ? 1 : 0);
}

template <int NT>
cudaError_t launch_move_nt(const DevParams &p, int units, int fit, int n_sm, LaunchCtx &ctx)
{
    static SmemGrant grant;
    const size_t smem = sel_smem<NT>(p.T_cap, p.seg_cap, p.S, false).total;
    if (!grant_dynamic_smem(k_select_move<NT>, smem, grant)) return cudaErrorInvalidValue;
    const int blocks = fit * n_sm, n_rows = p.Tk * p.H;
    constexpr int kRound = NT / 4; // rows of one round of a block
    const long long per = (long long)p.L * p.B * n_rows / (2LL * blocks); // two parts for each block where there is little to move
    const int most = (int)std::min(1024LL, std::max((long long)kRound, per / kRound * kRound));
    MovePlan plan; // equal parts: with a remainder of its own (720 rows as 704 and 16), 2442 units of 400 tokens took 282 instead of 242 us
    plan.parts = (n_rows + most - 1) / most;
    plan.rows = (n_rows + plan.parts - 1) / plan.parts;
    plan.lag = std::min(units, std::max(blocks, 2 * p.H + 2));
    const long long tickets = units + (long long)p.L * p.B * plan.parts;
    if (tickets > 0x7fffffffLL) return cudaErrorInvalidValue;
    return launch_after(k_select_move<NT>, dim3((unsigned)tickets), dim3(NT), smem, ctx.s, p, 0, plan);
}

constexpr size_t kSmShared = 228 * 1024, kBlockReserve = 1024; // shared memory of an SM; what each block takes besides its own

bool long_segments(const DevParams &p) { return p.l_max == 0 || p.l_max > kPiece; }

} // namespace

bool segsel_supported(const DevParams &p) { return sel_smem<1024>(p.T_cap, p.seg_cap, p.S, long_segments(p)).total <= (size_t)224 * 1024; }

int launch_segsel(const DevParams &p, LaunchCtx &ctx, bool *moved)
{
    bool move = moved != nullptr;
    const int units = p.L * p.B * p.H, n_sm = sm_count();
    if (n_sm <= 0) return AMS_ERR_CUDA;
    const bool longs = long_segments(p);
    // Threads per unit: a unit costs about (T / threads + a fixed part worth 24 tokens a thread), and the SMs' 1024 slots of 64
    // registers and their shared memory (which grows with the capacity: 121 KB for 512 threads at 131072 tokens in long segments) make
    // ceil(units / resident blocks) rounds of it.  160 units of 125840 tokens, l_max 4096: 512 threads by the registers alone 500 us,
    // 1024 by both 384; 640 of 131072 take 1024 either way, since one block of 512 fits as well.  The host knows the
    // capacity, not the lengths: rows far below it take the capacity's size (640 of 8704 tokens under 131072: 230 us).
    auto fits = [&](int nt, size_t smem) { return (int)std::max(1LL, std::min(1024LL / nt, (long long)(kSmShared / (smem + sizeof(SelShared) + kBlockReserve)))); };
    const int f256 = fits(256, sel_smem<256>(p.T_cap, p.seg_cap, p.S, longs).total), f512 = fits(512, sel_smem<512>(p.T_cap, p.seg_cap, p.S, longs).total),
              f1024 = fits(1024, sel_smem<1024>(p.T_cap, p.seg_cap, p.S, longs).total);
    auto cost = [&](int nt, int fit) { return ((long long)units + fit * n_sm - 1) / (fit * n_sm) * (p.T_cap / nt + 24); };
    const long long c256 = cost(256, f256), c512 = cost(512, f512), c1024 = cost(1024, f1024);
    const int nt = c256 <= c512 && c256 <= c1024 ? 256 : c512 <= c1024 ? 512 : 1024, fit = nt == 256 ? f256 : nt == 512 ? f512 : f1024;
    // Selection and moves in one launch, by figures of events apart / together / (apart, before there was a joint launch), us.  The host
    // knows the capacity, not the lengths, so the line lies where lengths just above the budget, which leave least to run beside, do not lose:
    // - 12 units per SM: 1184 units of 4224 tokens, budget 4096, 874 / 904 / (876); 1776 of 4096, 2048: 716 / 701 / (719); 1792 of
    //   8192 to 32768, 4096: 1611 / 1485 / (1619); 2048 of 1900 to 9001, 1000: 497 / 456 / (506).
    // - Two blocks to an SM, so that both kinds are on it: 640 units under 131072 tokens take blocks of 1024, 8704 tokens, 8192: 970 / 1005 /
    //   (983); 444 of 65536, 512: 339 / 396 / (340); 640 of 131072, 8192, that gain (1848 / 1691) are given up for those.
    //   Long segments (2048 units, 1176 / 1224) leave room for one block as well.
    // - A budget that pays for the tickets: 600 tokens, 1792 units, four heads, 320: 184 / 171 / (190), one head: 192 / 174 / (195); 3584
    //   units, one head, 320: 353 / 380 / (360); 2664, four heads, 360: 273 / 281 / (280); 400: 292 / 286 / (299).
    // - The separate moves read a token's rows of all heads together, which from 8 heads on is 2 KB in a piece and as fast as copying;
    //   selection of few units then hides less than the joint moves lose: 2560 units of 4136 tokens, 8 heads, 4096: 1853 / 1875 /
    //   (1864); 2088, 2048: 972 / 969 / (979); 8704, 8192, 8 heads: 3651 / 3700 / (3666), 4 heads: 3778 / 3702 / (3784).
    move = move && !longs && fit >= 2 && units >= 12LL * n_sm && p.Tk >= (units < 16LL * n_sm ? 320 : 400) && (p.H <= 4 || p.Tk <= 128LL * units / n_sm);
    if (moved) *moved = move;
    const cudaError_t e = nt == 256 ? (move ? launch_move_nt<256>(p, units, fit, n_sm, ctx) : launch_nt<256>(p, units, longs, ctx))
                        : nt == 512 ? (move ? launch_move_nt<512>(p, units, fit, n_sm, ctx) : launch_nt<512>(p, units, longs, ctx))
                                    : launch_nt<1024>(p, units, longs, ctx);
    if (e != cudaSuccess) return AMS_ERR_CUDA;
    ctx.mark(kKernSelect);
    return AMS_OK;
}

} // namespace ams
