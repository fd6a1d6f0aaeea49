// Algorithm 1 steps 3-5 of the paper for all (layer, sequence, KV head) units of an event, from the prefix sums and
// mass-quantile cuts of k_mass_scan: segments (merge, split) and their quotas, per-segment top-q_i, must-keep prefix
// and suffix, backfill to exactly the budget, ordered kept positions and the credit rows that travel with them.  One
// block per unit, one kept bit per token in shared memory.
//
// Selection order is (score key descending, position ascending), a strict total order, so a segment and its quota have
// exactly one answer however it is found.  The block searches all segments at once, in three walks over the unit's
// scores (the first from L2, the others mostly from L1):
//   1. smallest and largest key of every segment;
//   2. a histogram per segment, its bins spread evenly over that range of keys;
//   3. a warp per segment has found the bin of the q-th key: keys above it are kept, the few inside it go to a list
//      in which every entry counts the entries of its segment before it.
// A segment whose bin holds too many keys gets another histogram over that bin first (ties by the hundred end with a
// bin of one key).  The work per token does not depend on how long the segments are, every warp has the same share of
// it, and the number of block-wide steps is fixed; fixing key bits segment by segment, as this kernel once did, is a
// chain of 16 to 20 dependent warp-wide counts per segment.
// The backfill takes its bound from the best rejected key of every chunk, which walk 3 leaves behind, instead of
// walking the sequence twice more.
#include "ams_common.cuh"
#include "ams_select.cuh"

namespace ams {

using namespace sel;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBatch = 256;         // segments searched together
constexpr int kMaxBins = 1024;      // histogram bins per segment
constexpr int kMaxChunks = 256;     // entries of the table of best rejected keys
constexpr int kGroup = 8;           // 32-token windows whose scores a warp fetches together

// Working arrays of the search, one entry per segment of the batch.
struct SegTab {
    unsigned lo[kBatch], hi[kBatch]; // range of keys of the histogram (hi inclusive)
    unsigned L[kBatch], U[kBatch];   // keys >= U win, keys < L lose
    int above[kBatch];               // keys above the range of the histogram
    int r[kBatch], m[kBatch];        // r of the m keys in [L, U) win
    int base[kBatch], cnt[kBatch];   // part of the list
    unsigned char shift[kBatch];     // bin = (key - lo) >> shift
    unsigned char state[kBatch];
};
enum { kDone = 0, kSearch = 1, kTies = 2 };

template <int NT> struct Tune {
    static constexpr int kBins = NT <= 256 ? 8192 : 16384; // histogram bins of a batch
    static constexpr int kList = NT <= 256 ? 1024 : 2048;  // candidates
};

struct SelSmem { size_t mask, ms, bounds, quota, tab, hist, list, total; };
template <int NT>
__host__ __device__ inline SelSmem sel_smem(int T_cap, int sc, int S)
{
    SelSmem m;
    size_t o = 0;
    m.mask = o;   o += (size_t)((T_cap + 31) / 32 + 1) * 4;
    o = (o + 15) & ~(size_t)15;
    m.ms = o;     o += (size_t)sc * 8;
    m.bounds = o; o += (size_t)(sc + 1) * 4;
    m.quota = o;  o += (size_t)sc * 4;
    o = (o + 15) & ~(size_t)15;
    m.tab = o;    o += sizeof(SegTab);
    o = (o + 15) & ~(size_t)15;
    m.hist = o;   // also: scratch of the quota computation, which comes before
    const size_t h = (size_t)Tune<NT>::kBins * 4, q = (size_t)(S + 1) * 12 + (size_t)sc * 4;
    o += (h > q ? h : q);
    o = (o + 15) & ~(size_t)15;
    m.list = o;   o += (size_t)Tune<NT>::kList * 8;
    m.total = (o + 15) & ~(size_t)15;
    return m;
}

struct SelShared {
    int wc[2][32];   // per-warp counts of even / odd rounds of a block-wide count
    unsigned cmax[kMaxChunks];
    int n_list, n_clist, total;
    unsigned bound;
    int n_merged, n_seg, level, rem;
    unsigned short clist[kMaxChunks];
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
        int cnt1 = 0, tot = 0, mx = 0;
        for (int i = lane; i < n_seg; i += 32) { cnt1 += cap[i] >= 1; tot += cap[i]; mx = max(mx, cap[i]); }
        cnt1 = warp_sum(cnt1);
        tot = warp_sum(tot);
        mx = __reduce_max_sync(kFull, mx);
        int level = 0, used = 0;
        if (tot <= D) {
            level = mx;
            used = tot;
        } else if (cnt1 <= D) {
            int lo = 1, hi = mx; // F(lo) <= D < F(hi), F(k) = sum of min(cap, k)
            used = cnt1;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                int f = 0;
                for (int i = lane; i < n_seg; i += 32) f += min(cap[i], mid);
                f = warp_sum(f);
                if (f <= D) { lo = mid; used = f; } else hi = mid;
            }
            level = lo;
        }
        if (lane == 0) { sh.level = level; sh.rem = D - used; sh.total = tot <= D ? D - tot : 0; }
    }
    __syncthreads();
    const int level = sh.level, rem = sh.rem, left = sh.total;
    for (int i = tid; i < n_seg; i += NT) {
        int g = min(cap[i], level);
        if (rem > 0 && cap[i] > level) {
            int rank = 0;
            const u64 Mi = M[i];
            for (int j = 0; j < n_seg; ++j) {
                if (cap[j] <= level) continue;
                const u64 Mj = M[j];
                rank += sign > 0 ? (Mj > Mi || (Mj == Mi && j < i)) : (Mj < Mi || (Mj == Mi && j > i));
            }
            g += rank < rem;
        }
        quota[i] += sign * g;
    }
    __syncthreads();
    return left;
}

// Merge of short and split of long segments, quotas with their adjustment (Section 3.3 of the paper; Algorithm 1 steps
// 3-4): bounds[0..n], quota[0..n).  Returns n, or -1 if the tables cannot hold the segments.  Bq: the budget less the
// must-keep positions.  `tmp`: 3 (S + 1) + seg_cap ints.
template <int NT>
__device__ int segments_and_quotas(const DevParams &p, int uid, int T, int Bq, u64 *Ms, int *bounds, int *quota, int *tmp,
                                   SelShared &sh, int &round)
{
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int *raw = tmp, *merged = raw + p.S + 1, *poff = merged + p.S + 1, *cap = poff + p.S + 1;
    const u64 *C = p.cbuf + (size_t)uid * p.T_cap;
    const u64 SH = C[T - 1];
    if (warp == 0) {
        // raw cuts of the mass quantiles, found by the scan kernel (a cut at or beyond T means "none")
        for (int k = lane + 1; k < p.S; k += 32)
            raw[k] = p.fixed_seg ? (int)(((long long)k * T) / p.S) // component ablation: boundary k at floor(k T / S)
                                 : p.raw_cuts[(size_t)uid * (p.S + 1) + k];
        __syncwarp();
        int nm = 0;
        if (lane == 0) { // merge short raw segments forward, fold a short tail left
            int last = 0, start = 0;
            merged[nm++] = 0;
            for (int k = 1; k < p.S; ++k) {
                const int e = raw[k];
                if (e <= last || e >= T) continue;
                last = e;
                if (e - start >= p.l_min) { merged[nm++] = e; start = e; }
            }
            if (nm > 1 && T - start < p.l_min) --nm;
            merged[nm] = T; // nm segments
        }
        __syncwarp();
        nm = __shfl_sync(kFull, nm, 0);
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
    const u64 SHq = p.uniform_q ? (u64)T : SH; // total of what the quotas are proportional to
    int smin = 0;
    for (int i = tid; i < n_seg; i += NT) {
        const int a = bounds[i], e = bounds[i + 1];
        Ms[i] = p.uniform_q ? (u64)(e - a) : C[e - 1] - (a > 0 ? C[a - 1] : 0ull); // ablation: share by length
        smin += max(0, min(p.q_min, e - a));
    }
    const int Trem = Bq - block_count<NT>(smin, round, sh);
    int sq = 0;
    for (int i = tid; i < n_seg; i += NT) {
        const int L = bounds[i + 1] - bounds[i];
        long long qi = max(0, min(p.q_min, L));
        if (Trem >= 0) qi += (long long)((2ull * (u64)Trem * Ms[i] + SHq) / (2ull * SHq));
        if (qi > L) qi = L;
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

// ------------------------------------------------------------------------------------------ walks

// Walks the tokens [bounds[0], bounds[n]) of the batch's segments in windows of 32 (one token per lane, aligned to words of
// the kept mask); a warp takes one run of consecutive windows, kGroup of them fetched ahead.  f(t, s, in, key, crossing):
// s is the lane's segment; `crossing` (warp-uniform) says that the lanes may differ in it or in `in`; enter(s) is called
// when the warp moves to segment s as a whole, done(w) after the last window of a run or of a chunk of 2^chunk_log windows.
template <int NT, typename Enter, typename F, typename Done>
__device__ __forceinline__ void walk(const float *g, const int *bounds, int n, int chunk_log, Enter enter, F f, Done done)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int A = bounds[0], E = bounds[n];
    const int w0 = A >> 5, n_win = ((E + 31) >> 5) - w0;
    const int per = ((n_win + NW - 1) / NW + kGroup - 1) / kGroup * kGroup;
    const int wb = w0 + warp * per, we = min(w0 + n_win, wb + per);
    if (wb >= we) return;
    int s = 0;
    { // the segment of the run's first token
        int hi = n;
        const int t = max(A, wb * 32);
        while (hi - s > 1) {
            const int mid = (s + hi) >> 1;
            if (bounds[mid] <= t) s = mid; else hi = mid;
        }
    }
    int next = bounds[s + 1];
    enter(s);
    for (int g0 = wb; g0 < we; g0 += kGroup) {
        float x[kGroup];
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
            const int t = (g0 + j) * 32 + lane;
            x[j] = (g0 + j < we && t >= A && t < E) ? g[t] : 0.0f;
        }
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
            const int w = g0 + j;
            if (w >= we) break;
            const int ts = w * 32, t = ts + lane;
            const unsigned key = score_key(x[j]);
            if (ts >= next) {
                while (ts >= next) next = bounds[++s + 1];
                enter(s);
            }
            if (ts >= A && ts + 32 <= next) {
                f(t, s, true, key, false);
            } else {
                const bool in = t >= A && t < E;
                int sl = s;
                if (in) while (t >= bounds[sl + 1]) ++sl;
                f(t, sl, in, key, true);
            }
            if ((((w + 1) >> chunk_log) << chunk_log) == w + 1 || w + 1 == we) done(w);
        }
    }
}

// A warp finds the bin of segment s that holds its q-th key and what is left to decide in it.
__device__ __forceinline__ void find_bin(SegTab &tb, const unsigned *hist, int nb, int s, int q)
{
    const int lane = threadIdx.x & 31;
    const uint4 *h4 = reinterpret_cast<const uint4 *>(hist + s * nb);
    int above = tb.above[s];
    uint4 v = make_uint4(0, 0, 0, 0);
    int c = (nb + 127) / 128 - 1, sum = 0;
    for (;; --c) { // 128 bins at a time from the top
        const int i = c * 32 + lane;
        v = i * 4 < nb ? h4[i] : make_uint4(0, 0, 0, 0);
        sum = (int)(v.x + v.y + v.z + v.w);
        above += warp_sum(sum);
        if (c == 0 || above >= q) break;
    }
    const int before = above - warp_incl_scan(sum); // keys in the lanes (bins) above this one's, and above the range
    if (before < q && q <= before + sum) {
        int run = before, bin = 0, m = 0;
        const int cnt[4] = {(int)v.w, (int)v.z, (int)v.y, (int)v.x};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (run < q && q <= run + cnt[i]) { bin = c * 128 + lane * 4 + 3 - i; m = cnt[i]; above = run; }
            run += cnt[i];
        }
        const unsigned lo = tb.lo[s], hi = tb.hi[s], sft = tb.shift[s];
        const unsigned L = lo + ((unsigned)bin << sft);
        const unsigned U = (unsigned)bin == (hi - lo) >> sft ? hi + 1u : lo + ((unsigned)(bin + 1) << sft);
        const int r = q - above;
        tb.above[s] = above;
        tb.r[s] = r;
        tb.m[s] = m;
        tb.U[s] = r == m ? L : U;
        tb.L[s] = L;
        tb.state[s] = r == m ? kDone : (U - L == 1u ? kTies : kSearch);
    }
}

__device__ __forceinline__ int bin_shift(unsigned width_less_1, int nb) // smallest shift with width_less_1 >> shift < nb
{
    const int bits = 32 - __clz(width_less_1), have = 31 - __clz(nb);
    return max(0, bits - have);
}

// Top-q_i of the n <= kBatch segments at `bounds`: kept bits into mask, best rejected keys (must-keep positions apart)
// into the chunk table.
template <int NT>
__device__ void select_batch(const float *g, const int *bounds, const int *quota, int n, unsigned *mask, SegTab &tb, unsigned *hist, uint2 *list,
                             int ns, int t_last, int chunk_log, SelShared &sh)
{
    constexpr int NW = NT / 32, kList = Tune<NT>::kList;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int nb = Tune<NT>::kBins / n;
    nb = min(kMaxBins, 1 << (31 - __clz(nb)));

    // ---- walk 1: range of keys
    for (int i = tid; i < n; i += NT) { tb.lo[i] = kFull; tb.hi[i] = 0u; }
    uint4 *h4 = reinterpret_cast<uint4 *>(hist);
    for (int i = tid; i < n * nb / 4; i += NT) h4[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    {
        int cur = 0;
        unsigned mn = kFull, mx = 0u;
        auto flush = [&]() {
            mn = __reduce_min_sync(kFull, mn);
            mx = __reduce_max_sync(kFull, mx);
            if (lane == 0 && mn <= mx) { atomicMin(&tb.lo[cur], mn); atomicMax(&tb.hi[cur], mx); }
            mn = kFull; mx = 0u;
        };
        walk<NT>(g, bounds, n, 30, [&](int s) { flush(); cur = s; },
                 [&](int, int s, bool in, unsigned key, bool crossing) {
                     if (!crossing) { mn = min(mn, key); mx = max(mx, key); }
                     else if (in) { atomicMin(&tb.lo[s], key); atomicMax(&tb.hi[s], key); }
                 },
                 [&](int) { flush(); });
    }
    __syncthreads();
    for (int i = tid; i < n; i += NT) {
        const int len = bounds[i + 1] - bounds[i], q = quota[i];
        const unsigned lo = tb.lo[i], hi = tb.hi[i];
        tb.above[i] = 0;
        tb.r[i] = q;
        tb.m[i] = len;
        tb.state[i] = kSearch;
        tb.L[i] = lo; tb.U[i] = hi + 1u;
        tb.shift[i] = (unsigned char)bin_shift(hi - lo, nb);
        if (q <= 0) { tb.state[i] = kDone; tb.L[i] = tb.U[i] = kFull; }
        else if (q >= len) { tb.state[i] = kDone; tb.L[i] = tb.U[i] = 0u; }
        else if (lo == hi) tb.state[i] = kTies;
        if (tb.state[i] != kSearch) tb.shift[i] = 255;
    }
    __syncthreads();

    // ---- walk 2: histograms, and again over the threshold's bin where that is still crowded
    for (;;) {
        {
            unsigned lo = 0u, hi = 0u, sft = 255u;
            int cur = 0;
            auto load = [&](int s) { cur = s; lo = tb.lo[s]; hi = tb.hi[s]; sft = tb.shift[s]; };
            walk<NT>(g, bounds, n, 30, load,
                     [&](int, int s, bool in, unsigned key, bool crossing) {
                         unsigned l = lo, h = hi, f = sft;
                         if (crossing && s != cur) { l = tb.lo[s]; h = tb.hi[s]; f = tb.shift[s]; }
                         if (in && f < 32u && key >= l && key <= h) atomicAdd(&hist[s * nb + ((key - l) >> f)], 1u);
                     },
                     [](int) {});
        }
        __syncthreads();
        for (int s = warp; s < n; s += NW)
            if (tb.shift[s] < 32) find_bin(tb, hist, nb, s, quota[s]);
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
        const int limit = sh.total > kList ? kList / kBatch : 384; // most candidates of a segment that are ranked pairwise
        bool again = false;
        for (int i = tid; i < n; i += NT) {
            tb.shift[i] = 255;
            if (tb.state[i] == kSearch && tb.m[i] > limit) {
                tb.lo[i] = tb.L[i]; tb.hi[i] = tb.U[i] - 1u;
                tb.shift[i] = (unsigned char)bin_shift(tb.U[i] - 1u - tb.L[i], nb);
                again = true;
            }
        }
        if (!__syncthreads_or(again)) break;
        for (int s = warp; s < n; s += NW)
            if (tb.shift[s] < 32)
                for (int i = lane; i < nb; i += 32) hist[s * nb + i] = 0u;
        __syncthreads();
    }

    // ---- walk 3: kept bits, candidates, best rejected keys
    {
        unsigned L = 0u, U = 0u, best = 0u;
        int cur = 0;
        walk<NT>(g, bounds, n, chunk_log, [&](int s) { cur = s; L = tb.L[s]; U = tb.U[s]; },
                 [&](int t, int s, bool in, unsigned key, bool crossing) {
                     unsigned l = L, u = U;
                     if (crossing && s != cur) { l = tb.L[s]; u = tb.U[s]; }
                     const unsigned bal = __ballot_sync(kFull, in && key >= u);
                     if (lane == 0 && bal) atomicOr(&mask[t >> 5], bal);
                     if (in && key < u) {
                         if (key >= l) {
                             if (tb.state[s] == kSearch) list[atomicAdd(&tb.cnt[s], 1)] = make_uint2(key, (unsigned)t | ((unsigned)s << 24));
                         } else if (t >= ns && t < t_last) {
                             best = max(best, key);
                         }
                     }
                 },
                 [&](int w) {
                     best = __reduce_max_sync(kFull, best);
                     if (lane == 0 && best) atomicMax(&sh.cmax[w >> chunk_log], best);
                     best = 0u;
                 });
    }
    __syncthreads();
    for (int i = tid; i < sh.total; i += NT) { // every candidate ranks itself
        const uint2 v = list[i];
        const int s = (int)(v.y >> 24), t = (int)(v.y & 0xffffffu);
        const int b = tb.base[s], e = b + tb.m[s];
        int rank = 0;
        for (int j = b; j < e; ++j) {
            const uint2 o = list[j];
            rank += o.x > v.x || (o.x == v.x && o.y < v.y); // (same segment: y orders by position)
        }
        if (rank < tb.r[s]) atomicOr(&mask[t >> 5], 1u << (t & 31));
        else if (t >= ns && t < t_last) atomicMax(&sh.cmax[(t >> 5) >> chunk_log], v.x);
    }
    for (int s = warp; s < n; s += NW) { // ties across the threshold: the first r of them in position order
        if (tb.state[s] != kTies) continue;
        const unsigned key = tb.L[s];
        const int a = bounds[s], e = bounds[s + 1], r = tb.r[s];
        int seen = 0;
        for (int t0 = a & ~31; t0 < e; t0 += 32) {
            const int t = t0 + lane;
            const bool tie = t >= a && t < e && score_key(g[t]) == key;
            const unsigned bal = __ballot_sync(kFull, tie);
            const bool kept = tie && seen + __popc(bal & ((1u << lane) - 1u)) < r;
            const unsigned kb = __ballot_sync(kFull, kept);
            if (lane == 0 && kb) atomicOr(&mask[t0 >> 5], kb);
            if (__any_sync(kFull, tie && !kept && t >= ns && t < t_last) && lane == 0) atomicMax(&sh.cmax[(t0 >> 5) >> chunk_log], key);
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

template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_select_compact(DevParams p)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ SelShared sh;
    constexpr int NW = NT / 32, kList = Tune<NT>::kList;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, uid = blockIdx.x;
    const int h = uid % p.H, bq = (uid / p.H) % p.B, l = uid / (p.H * p.B);
    const int T = p.seq_lens[bq];
    if (T <= p.Tk || T > p.T_cap) return;
    const int sc = p.seg_cap;
    const SelSmem mp = sel_smem<NT>(p.T_cap, sc, p.S);
    unsigned *mask = reinterpret_cast<unsigned *>(dyn + mp.mask);
    int *bounds = reinterpret_cast<int *>(dyn + mp.bounds);
    int *quota = reinterpret_cast<int *>(dyn + mp.quota);
    unsigned *hist = reinterpret_cast<unsigned *>(dyn + mp.hist);
    SegTab &tb = *reinterpret_cast<SegTab *>(dyn + mp.tab);
    uint2 *list = reinterpret_cast<uint2 *>(dyn + mp.list); // (key, position) of candidates
    const size_t row = (size_t)uid * p.T_cap;
    const float *g = p.scores + row;
    int *keep = p.keep_idx + (size_t)uid * p.Tk;
    const bool ema_on = p.beta != 1.0f;
    const int n_words = (T + 31) >> 5;
    const int ns = max(0, min(p.n_sink, min(p.Tk, T)));           // must-keep prefix and suffix
    const int nl = max(0, min(p.n_last, min(p.Tk - ns, T - ns)));
    const int t_last = T - nl;
    int chunk_log = 0; // chunks of 2^chunk_log windows, at most kMaxChunks of them
    while ((n_words - 1) >> chunk_log >= kMaxChunks) ++chunk_log;
    const int n_chunk = ((n_words - 1) >> chunk_log) + 1;
    int round = 0;
    for (int i = tid; i <= n_words; i += NT) mask[i] = 0u;
    for (int i = tid; i < kMaxChunks; i += NT) sh.cmax[i] = 0u;
    if (tid == 0) { sh.n_list = 0; sh.n_clist = 0; sh.bound = 0u; }
    wait_for_previous_kernel(); // prefix sums and cuts
    const int n_seg = segments_and_quotas<NT>(p, uid, T, p.Tk - ns - nl, reinterpret_cast<u64 *>(dyn + mp.ms), bounds, quota,
                                              reinterpret_cast<int *>(hist), sh, round);
    if (n_seg < 0) { // cannot happen with the capacity formula of the header; reported all the same
        if (tid == 0) { set_status(p.status, AMS_ERR_CAPACITY, uid, sh.n_seg, sc); p.n_seg[uid] = -1; p.seq_bad[bq] = 1; }
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

    // ---- per-segment top-q_i
    for (int s0 = 0; s0 < n_seg; s0 += kBatch)
        select_batch<NT>(g, bounds + s0, quota + s0, min(kBatch, n_seg - s0), mask, tb, hist, list, ns, t_last, chunk_log, sh);

    // ---- must-keep prefix and suffix; every must-keep position a segment already chose frees one slot,
    //      refilled by the best positions not yet kept (top r_fill of the unflagged tokens of the sequence)
    int already = 0;
    for (int i = tid; i < ns + nl; i += NT) {
        const int t = i < ns ? i : t_last + (i - ns);
        already += (atomicOr(&mask[t >> 5], 1u << (t & 31)) >> (t & 31)) & 1u;
    }
    const int r_fill = block_count<NT>(already, round, sh);
    if (r_fill > 0) {
        // At least r_fill unflagged tokens lie at or above the r_fill-th largest of the chunks' best rejected keys, so
        // only chunks whose best key reaches that bound can hold a winner; their tokens at or above it go to a list.
        for (int i = tid; i < n_chunk; i += NT) {
            const unsigned v = sh.cmax[i];
            int rank = 0;
            for (int j = 0; j < n_chunk; ++j) {
                const unsigned o = sh.cmax[j];
                rank += o > v || (o == v && j < i);
            }
            if (rank == r_fill - 1) sh.bound = v; // (none, or 0: too few chunks with a candidate, everything is looked at)
        }
        __syncthreads();
        const unsigned M = sh.bound;
        auto raise = [&](int t) { atomicOr(&mask[t >> 5], 1u << (t & 31)); };
        auto unflagged = [&](int t) { return ((mask[t >> 5] >> (t & 31)) & 1u) == 0u; };
        for (int i = tid; i < n_chunk; i += NT)
            if (sh.cmax[i] >= M) sh.clist[atomicAdd(&sh.n_clist, 1)] = (unsigned short)i;
        __syncthreads();
        const int n_w = sh.n_clist << chunk_log; // windows to look at
        for (int i0 = warp; i0 < n_w; i0 += NW * 4) {
            float x[4];
            int tt[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = i0 + j * NW;
                tt[j] = i < n_w ? (((int)sh.clist[i >> chunk_log] << chunk_log) + (i & ((1 << chunk_log) - 1))) * 32 + lane : T;
                x[j] = tt[j] < T ? g[tt[j]] : 0.0f;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const unsigned key = score_key(x[j]);
                if (tt[j] < T && key >= M && unflagged(tt[j])) {
                    const int at = atomicAdd(&sh.n_list, 1);
                    if (at < kList) list[at] = make_uint2(key, (unsigned)tt[j]);
                }
            }
        }
        __syncthreads();
        const int n_list = sh.n_list;
        if (n_list > kList) {
            block_select_stream<NT>(g, T, r_fill, sh, round, unflagged, raise);
        } else {
            for (int i = tid; i < n_list; i += NT) {
                const uint2 v = list[i];
                int rank = 0;
                for (int j = 0; j < n_list; ++j) {
                    const uint2 o = list[j];
                    rank += o.x > v.x || (o.x == v.x && o.y < v.y);
                }
                if (rank < r_fill) raise((int)v.y);
            }
        }
    }
    __syncthreads();

    // ---- ordered compaction of the kept positions: a warp takes a run of mask words, a lane a bit of the current one
    const int wpw = (n_words + NW - 1) / NW, w0 = warp * wpw, w1 = min(n_words, w0 + wpw);
    int n_kept = 0;
    for (int w = w0 + lane; w < w1; w += 32) n_kept += __popc(mask[w]);
    n_kept = warp_sum(n_kept);
    if (lane == 0) sh.cmax[warp] = (unsigned)n_kept;
    __syncthreads();
    int pos = warp_sum(lane < warp ? (int)sh.cmax[lane] : 0);
    const int total = warp_sum(lane < NW ? (int)sh.cmax[lane] : 0);
    if (total != p.Tk) {
        if (tid == 0) { set_status(p.status, AMS_ERR_INTERNAL, uid, total, p.Tk); p.seq_bad[bq] = 1; }
        return;
    }
    for (int g0 = w0; g0 < w1; g0 += 32) {
        const unsigned mine = g0 + lane < w1 ? mask[g0 + lane] : 0u;
        const int n = min(32, w1 - g0);
        for (int i = 0; i < n; ++i) {
            const unsigned m = __shfl_sync(kFull, mine, i);
            if ((m >> lane) & 1u) keep[pos + __popc(m & ((1u << lane) - 1u))] = (g0 + i) * 32 + lane;
            pos += __popc(m);
        }
    }
    // ---- credit rows travel with their tokens, in place: kept positions ascend and keep[j] >= j, so what a tile
    //      writes is never read by a later one.  Rows beyond the budget start from zero.
    if (ema_on) {
        float *credit = p.ema + (((size_t)l * p.Bmax + bq) * p.H + h) * (size_t)p.T_cap;
        constexpr int kPer = 8;
        __syncthreads();
        for (int base = 0; base < p.Tk; base += NT * kPer) {
            float c[kPer];
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int j = base + i * NT + tid;
                c[i] = j < p.Tk ? credit[keep[j]] : 0.0f;
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
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
cudaError_t launch_nt(const DevParams &p, int units, LaunchCtx &ctx)
{
    static SmemGrant grant;
    const size_t smem = sel_smem<NT>(p.T_cap, p.seg_cap, p.S).total;
    if (!grant_dynamic_smem(k_select_compact<NT>, smem, grant)) return cudaErrorInvalidValue;
    return launch_after(k_select_compact<NT>, dim3((unsigned)units), dim3(NT), smem, ctx.s, p);
}

} // namespace

size_t select_smem_bytes(const DevParams &p) { return sel_smem<512>(p.T_cap, p.seg_cap, p.S).total; }

int launch_select(const DevParams &p, LaunchCtx &ctx)
{
    const int units = p.L * p.B * p.H, n_sm = sm_count();
    if (n_sm <= 0) return AMS_ERR_CUDA;
    const cudaError_t e = units >= 6 * n_sm ? launch_nt<256>(p, units, ctx)
                        : units > n_sm ? launch_nt<512>(p, units, ctx) : launch_nt<1024>(p, units, ctx);
    if (e != cudaSuccess) return AMS_ERR_CUDA;
    ctx.mark(kKernSelect);
    return AMS_OK;
}

} // namespace ams
