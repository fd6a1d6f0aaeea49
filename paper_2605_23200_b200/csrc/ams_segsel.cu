// Algorithm 1 steps 1-3 of the paper over all (layer, sequence, KV head) units of an event (steps 3-5 follow in
// ams_select.cu):
//
//   k_mass_scan        Eq. 1 on fixed-point weights, the EMA credit update and the history-aware mass
//                      (Section 3.3, "EMA credit"; Algorithm 1 steps 1-2), and the inclusive prefix sum of
//                      the integer mass with the mass-quantile cuts b_k = min{t : c(t) >= k / S} (Algorithm 1
//                      step 3).  One block per unit streams the unit's usage row from L2 once per reduction
//                      that the arithmetic needs.
//
// Every decision is integer arithmetic on fixed-point images of the mass (kFixBits fractional bits) and
// every floating-point step a single round-to-nearest operation, so results do not depend on the order in
// which a block adds things up.
#include <type_traits>

#include "ams_common.cuh"
#include "ams_select.cuh"

namespace ams {

using namespace sel;

namespace {

constexpr int kScanVec = 8;                 // tokens per thread and round of the scan pass

struct UnitId { int l, b, h; };
__device__ __forceinline__ UnitId unit_of(const DevParams &p, int uid)
{
    UnitId u;
    u.h = uid % p.H; u.b = (uid / p.H) % p.B; u.l = uid / (p.H * p.B);
    return u;
}

// ------------------------------------------------------------------------------------------ k_mass_scan

// Walks the first `n` floats of a row (allocated to a multiple of 4) with float4 loads, four per thread in
// flight: f(t, v, full) gets the position of the group's first element and, as a compile-time flag, whether
// the whole group lies inside the row (then no per-element bound is needed).
template <int NT, typename F>
__device__ __forceinline__ void walk4(const float *row, int n, F f)
{
    const int n4 = (n + 3) & ~3;
    const int tid = threadIdx.x;
    for (int base = 0; base < n4; base += NT * 16) {
        float4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int t = base + (j * NT + tid) * 4;
            v[j] = t < n4 ? *reinterpret_cast<const float4 *>(row + t) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int t = base + (j * NT + tid) * 4;
            if (t + 3 < n) f(t, v[j], std::true_type{});
            else if (t < n) f(t, v[j], std::false_type{});
        }
    }
}

// The same over two rows at once (usage and credit).
template <int NT, typename F>
__device__ __forceinline__ void walk4x2(const float *row_a, const float *row_b, int n, F f)
{
    const int n4 = (n + 3) & ~3;
    const int tid = threadIdx.x;
    for (int base = 0; base < n4; base += NT * 16) {
        float4 va[4], vb[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int t = base + (j * NT + tid) * 4;
            va[j] = vb[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (t < n4) { va[j] = *reinterpret_cast<const float4 *>(row_a + t); vb[j] = *reinterpret_cast<const float4 *>(row_b + t); }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int t = base + (j * NT + tid) * 4;
            if (t + 3 < n) f(t, va[j], vb[j], std::true_type{});
            else if (t < n) f(t, va[j], vb[j], std::false_type{});
        }
    }
}

// Block-wide sum of doubles that are integers below 2^53 (exact, hence independent of the order).
__device__ __forceinline__ double block_sum_exact_f64(double v, u64 *scratch)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) scratch[warp] = (u64)__double_as_longlong(v);
    __syncthreads();
    if (warp == 0) {
        double x = lane < nw ? __longlong_as_double((long long)scratch[lane]) : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) scratch[32] = (u64)__double_as_longlong(x);
    }
    __syncthreads();
    return __longlong_as_double((long long)scratch[32]);
}

// raw_cuts: [units][S + 1] cut positions of the mass quantiles (entry k: boundary after the token that
// reaches k / S; T where no token before the last one does).
template <int NT>
__global__ void __launch_bounds__(NT) k_mass_scan(DevParams p)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ u64 scratch[40];
    u64 *qthr = reinterpret_cast<u64 *>(dyn); // [S]: prefix value at which quantile k is reached
    const int tid = threadIdx.x, uid = blockIdx.x;
    const UnitId un = unit_of(p, uid);
    const int T = p.seq_lens[un.b];
    if (T <= p.Tk || T > p.T_cap) return;
    const size_t row = (size_t)uid * p.T_cap;
    const float *u = p.usage + row;
    float *credit = p.ema + (((size_t)un.l * p.Bmax + un.b) * p.H + un.h) * (size_t)p.T_cap;
    u64 *C = p.cbuf + row;
    int *raw = p.raw_cuts + (size_t)uid * (p.S + 1);
    float *mass_dbg = p.mass_dbg ? p.mass_dbg + row : nullptr;
    const bool ema_on = p.beta != 1.0f;
    const double two_f = (double)(1ull << kFixBits);
    wait_for_previous_kernel(); // the usage scores
    for (int k = tid; k <= p.S; k += NT) raw[k] = T;

    // Rows are allocated to the capacity (a multiple of 16), so whole float4 groups may be read past the
    // sequence's end; what lies there is masked by position.
    // ---- largest Eq. 1 weight -> exponent of the fixed-point images
    float wmax = 0.0f;
    walk4<NT>(u, T, [&](int t, float4 v, auto full) {
        const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) if (decltype(full)::value || t + i < T) wmax = fmaxf(wmax, weight_of(w[i], p.eps));
    });
    wmax = block_max_f32(wmax, scratch);
    const int ew = fix_exponent(wmax);
    // ---- SA = sum of the images A_t = floor(w_t 2^(36 - ew)), held as doubles (integers below 2^53: exact)
    const double scale_w = fix_scale_of(ew);
    const float cut_w = fixed_trunc_threshold(ew); // weights below it lose their bits under the image's last one
    double sa = 0.0;
    walk4<NT>(u, T, [&](int t, float4 v, auto full) {
        const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (decltype(full)::value || t + i < T) sa = __dadd_rn(sa, __dmul_rn((double)fixed_trunc_by_add(weight_of(w[i], p.eps), cut_w), scale_w));
    });
    const double SA = block_sum_exact_f64(sa, scratch);
    const double inv_sa = __ddiv_rn(1.0, SA);          // normalisations multiply by the rounded reciprocal
    const double inv_sa_w = __dmul_rn(inv_sa, scale_w); // A_t / SA = trunc(w_t) * (2^(36 - ew) / SA): the scaling is exact

    // ---- EMA credit: c <- lambda c + (1 - lambda) m, updated in place (the block-wide reductions that follow
    //      make every thread's writes visible to the others before anybody reads them back)
    int ec = 0;
    float cut_c = 0.0f;
    double inv_sc_c = 0.0; // 2^(36 - ec) / SC
    bool have_credit = false;
    if (ema_on) {
        const float oml = __fsub_rn(1.0f, p.lambda);
        float cmax = 0.0f;
        walk4x2<NT>(u, credit, T, [&](int t, float4 v, float4 cv, auto full) {
            const float w[4] = {v.x, v.y, v.z, v.w};
            float c[4] = {cv.x, cv.y, cv.z, cv.w};
            float m[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                m[i] = __double2float_rn(__dmul_rn((double)fixed_trunc_by_add(weight_of(w[i], p.eps), cut_w), inv_sa_w));
                if (decltype(full)::value || t + i < T) {
                    c[i] = __fadd_rn(__fmul_rn(p.lambda, c[i]), __fmul_rn(oml, m[i]));
                    cmax = fmaxf(cmax, c[i]);
                }
            }
            if (decltype(full)::value) {
                *reinterpret_cast<float4 *>(credit + t) = make_float4(c[0], c[1], c[2], c[3]);
                if (mass_dbg) *reinterpret_cast<float4 *>(mass_dbg + t) = make_float4(m[0], m[1], m[2], m[3]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (t + i < T) { credit[t + i] = c[i]; if (mass_dbg) mass_dbg[t + i] = m[i]; }
            }
        });
        cmax = block_max_f32(cmax, scratch);
        double scsum = 0.0;
        double scale_c = 0.0;
        if (cmax > 0.0f) {
            ec = fix_exponent(cmax);
            scale_c = fix_scale_of(ec);
            cut_c = fixed_trunc_threshold(ec);
            walk4<NT>(credit, T, [&](int t, float4 cv, auto full) {
                const float c[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (decltype(full)::value || t + i < T) scsum = __dadd_rn(scsum, __dmul_rn((double)fixed_trunc_by_add(c[i], cut_c), scale_c));
            });
        }
        const double SC = block_sum_exact_f64(scsum, scratch);
        have_credit = SC > 0.0;
        if (have_credit) inv_sc_c = __dmul_rn(__ddiv_rn(1.0, SC), scale_c);
    }

    // ---- history-aware integer mass Hm_t = floor((beta m + (1 - beta) normalize(c)) 2^36) and its inclusive
    //      prefix sum, kScanVec consecutive tokens per thread and round; the next round's inputs are fetched
    //      before this round's block-wide scan
    const double bd = (double)p.beta, omb = __dsub_rn(1.0, (double)p.beta);
    u64 carry = 0;
    constexpr int kRound = NT * kScanVec;
    float4 wn[kScanVec / 4], cn[kScanVec / 4];
    auto fetch = [&](int base) {
#pragma unroll
        for (int q = 0; q < kScanVec / 4; ++q) {
            const int t = base + tid * kScanVec + 4 * q;
            wn[q] = cn[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (t < T) {
                wn[q] = *reinterpret_cast<const float4 *>(u + t);
                if (have_credit) cn[q] = *reinterpret_cast<const float4 *>(credit + t);
            }
        }
    };
    fetch(0);
    for (int base = 0; base < T; base += kRound) {
        const int t0 = base + tid * kScanVec;
        u64 Hm[kScanVec];
        u64 tot8 = 0;
        float4 wv[kScanVec / 4], cv[kScanVec / 4];
#pragma unroll
        for (int q = 0; q < kScanVec / 4; ++q) { wv[q] = wn[q]; cv[q] = cn[q]; }
        if (base + kRound < T) fetch(base + kRound);
#pragma unroll
        for (int q = 0; q < kScanVec / 4; ++q) {
            const int t = t0 + 4 * q;
            const float w[4] = {wv[q].x, wv[q].y, wv[q].z, wv[q].w}, c[4] = {cv[q].x, cv[q].y, cv[q].z, cv[q].w};
            float m[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                u64 h = 0;
                m[i] = 0.0f;
                if (t + i < T) {
                    const double r = __dmul_rn((double)fixed_trunc_by_add(weight_of(w[i], p.eps), cut_w), inv_sa_w);
                    if (ema_on) {
                        double hist = 0.0;
                        if (have_credit) hist = __dmul_rn(omb, __dmul_rn((double)fixed_trunc_by_add(c[i], cut_c), inv_sc_c));
                        h = floor_to_u64(__dmul_rn(__dadd_rn(__dmul_rn(bd, r), hist), two_f));
                    } else {
                        m[i] = __double2float_rn(r);
                        h = floor_to_u64(__dmul_rn(r, two_f));
                    }
                }
                Hm[4 * q + i] = h;
                tot8 += h;
            }
            if (!ema_on && mass_dbg && t < T) {
                if (t + 3 < T) *reinterpret_cast<float4 *>(mass_dbg + t) = make_float4(m[0], m[1], m[2], m[3]);
                else
#pragma unroll
                    for (int i = 0; i < 4; ++i) if (t + i < T) mass_dbg[t + i] = m[i];
            }
        }
        u64 tot;
        u64 run = carry + block_excl_scan_u64(tot8, scratch, &tot);
        carry += tot;
        if (t0 < T) { // rows have the capacity's length: whole pairs are written, positions past T are never read
#pragma unroll
            for (int q = 0; q < kScanVec / 2; ++q) {
                ulonglong2 o;
                run += Hm[2 * q]; o.x = run;
                run += Hm[2 * q + 1]; o.y = run;
                if (t0 + 2 * q < T) *reinterpret_cast<ulonglong2 *>(C + t0 + 2 * q) = o;
            }
        }
    }
    if (p.fixed_seg) return; // component ablation: the cuts do not depend on the mass (the next kernel places them)

    // ---- mass-quantile cuts: the token that reaches quantile k closes its segment, so the boundary is
    //      (position + 1).  c(t) >= k / S  <=>  C(t) S >= k SH  <=>  C(t) >= ceil(k SH / S).  A thread looks at
    //      the prefix before its first and at its last token of a round and walks its tokens only if a
    //      quantile lies between the two.
    const u64 SH = carry, S = (u64)p.S;
    for (int k = tid + 1; k < p.S; k += NT) qthr[k] = ((u64)k * SH + S - 1) / S;
    __syncthreads(); // (also orders the prefix sums written above before the reads below)
    auto quantile = [&](u64 c) -> int { // number of k in [1, S) with qthr[k] <= c
        int lo = 0, hi = p.S - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (qthr[mid] <= c) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    for (int base = 0; base < T; base += 4 * kRound) {
        u64 before[4], last[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int t0 = base + j * kRound + tid * kScanVec;
            before[j] = last[j] = 0;
            if (t0 < T) {
                before[j] = t0 > 0 ? C[t0 - 1] : 0ull;
                last[j] = C[min(t0 + kScanVec, T) - 1];
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int t0 = base + j * kRound + tid * kScanVec;
            if (t0 >= T) continue;
            int kprev = quantile(before[j]);
            const int klast = quantile(last[j]);
            if (klast == kprev) continue;
            for (int i = 0; i < kScanVec && t0 + i < T; ++i) {
                const int kc = quantile(C[t0 + i]);
                for (int k = kprev + 1; k <= kc; ++k) raw[k] = t0 + i + 1;
                kprev = kc;
            }
        }
    }
}

} // namespace

bool segsel_supported(const DevParams &p)
{
    return select_smem_bytes(p) <= (size_t)200 * 1024;
}

int launch_segsel(const DevParams &p, LaunchCtx &ctx)
{
    const int units = p.L * p.B * p.H;
    const int n_sm = sm_count();
    if (n_sm <= 0) return AMS_ERR_CUDA;
    const bool many_units = units >= 6 * n_sm; // several blocks per SM anyway: the smaller ones overlap their serial parts better
    const size_t smem_a = (size_t)(p.S + 1) * 8;
    // A unit's pass is a chain of block-wide reductions: with many units per SM, blocks of 256 threads (four per SM
    // instead of two) overlap those chains better; with few units the wider block finishes its unit sooner.
    const bool narrow_scan = many_units;
    if (ctx.launches <= 1) {
        // nothing but the validation kernel ran before (caller-supplied scores): its effective lengths are read
        // before this kernel's first wait, so this launch is fully ordered after it
        if (narrow_scan) k_mass_scan<256><<<units, 256, smem_a, ctx.s>>>(p);
        else k_mass_scan<512><<<units, 512, smem_a, ctx.s>>>(p);
        if (cudaGetLastError() != cudaSuccess) return AMS_ERR_CUDA;
    } else if ((narrow_scan ? launch_after(k_mass_scan<256>, dim3((unsigned)units), dim3(256), smem_a, ctx.s, p)
                            : launch_after(k_mass_scan<512>, dim3((unsigned)units), dim3(512), smem_a, ctx.s, p)) != cudaSuccess) {
        return AMS_ERR_CUDA;
    }
    ctx.mark(kKernSegmentSelect);
    return launch_select(p, ctx);
}

} // namespace ams
