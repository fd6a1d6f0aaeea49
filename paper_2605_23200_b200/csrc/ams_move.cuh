// Row moves of the compaction, shared by the kernel that only moves and the one that selects as well.
#pragma once
#include "ams_common.cuh"

namespace ams {

// Moves rows [r0, r1) of one (layer, sequence), by a block of NT threads; 16 lanes of 16 bytes to a row, K and V of four rows in
// flight per thread.  Rows are numbered r = j * H + h, so that consecutive rows are consecutive 256-byte pieces of the
// destination page.  The positions and page ids of the next rows are fetched while this round's are on their way: three
// trips to memory one after another otherwise leave a block idle for two of them.
template <int NT>
__device__ __forceinline__ void move_rows(const DevParams &p, int l, int b, int r0, int r1)
{
    constexpr int kUnroll = 4, kRows = NT / 16;
    const int lane = threadIdx.x & 15;
    const int *table = p.src_pages + (size_t)b * (p.T_cap / kPage);
    const int *dst = p.dst_pages + (size_t)b * p.n_dst;
    const int *keep = p.keep_idx + (size_t)(l * p.B + b) * p.H * p.Tk;
    const size_t base = (size_t)l * (size_t)p.num_pages * (size_t)(kPage * p.H) * kHeadDim + lane * 8;
    __nv_bfloat16 *k = p.k_pages + base, *v = p.v_pages + base;
    unsigned from[kUnroll], to[kUnroll]; // rows of the layer's pool (fewer than 2^32 rows of 256 bytes fit the device)
    const int dj = kRows / p.H, dh = kRows % p.H; // from a row of this thread to the next
    int r = r0 + (threadIdx.x >> 4), r_ahead = r;
    int j = r / p.H, h = r - j * p.H;
    auto locate = [&](unsigned &f, unsigned &t) {
        f = t = 0u;
        if (r_ahead < r1) {
            const int pos = __ldcg(keep + (size_t)h * p.Tk + j);
            f = ((unsigned)table[pos >> 4] * kPage + (pos & 15)) * p.H + h;
            t = ((unsigned)dst[j >> 4] * kPage + (j & 15)) * p.H + h;
        }
        r_ahead += kRows; j += dj; h += dh;
        if (h >= p.H) { h -= p.H; ++j; }
    };
#pragma unroll
    for (int i = 0; i < kUnroll; ++i) locate(from[i], to[i]);
    for (; r < r1; r += kRows * kUnroll) {
        uint4 kv[kUnroll], vv[kUnroll];
#pragma unroll
        for (int i = 0; i < kUnroll; ++i)
            if (r + i * kRows < r1) {
                kv[i] = ld_stream16(k + (size_t)from[i] * kHeadDim);
                vv[i] = ld_stream16(v + (size_t)from[i] * kHeadDim);
            }
        unsigned next[kUnroll];
#pragma unroll
        for (int i = 0; i < kUnroll; ++i) locate(from[i], next[i]);
#pragma unroll
        for (int i = 0; i < kUnroll; ++i) {
            if (r + i * kRows < r1) {
                st_stream16(k + (size_t)to[i] * kHeadDim, kv[i]);
                st_stream16(v + (size_t)to[i] * kHeadDim, vv[i]);
            }
            to[i] = next[i];
        }
    }
}

// Block-table row <- replacement pages followed by -1; length <- budget.  After every read of the old table.
__device__ __forceinline__ void update_table(const DevParams &p, int b)
{
    int *row = p.block_table + (size_t)b * p.bt_stride;
    for (int i = threadIdx.x; i < p.bt_stride; i += blockDim.x)
        row[i] = i < p.n_dst ? p.dst_pages[(size_t)b * p.n_dst + i] : -1;
    if (threadIdx.x == 0) p.seq_lens_out[b] = p.Tk;
}

} // namespace ams
