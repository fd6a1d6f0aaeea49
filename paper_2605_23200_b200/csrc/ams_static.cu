// Allocation-free selection entry point: steps 1-5 of Algorithm 1 on caller-supplied scores.
//
// Some callers cannot allocate device memory at all: code running while a stream is being
// captured into a CUDA graph (allocation calls are not permitted there), plug-ins loaded into
// a serving process whose memory pool is owned and fully reserved by the host framework, and
// callers on a hot path that must not take the allocator's locks.  For them the scratch the
// selection kernel needs lives in the fixed array below instead of a caller-supplied
// workspace.  Every GPU that loads the library holds the array (kStaticBytes) until the process
// exits.
//
// The kernel is that of ams_compress (k_select_compact), told the one length of all rows instead of reading lengths.
#include <string.h>

#include "ams_common.cuh"

namespace ams {
namespace {

constexpr int kStaticMaxUnits = 8;       // score rows per call
constexpr int kStaticMaxTokens = 32768;  // tokens per score row
constexpr int kStaticSegCap = 1024;      // segments per row after merge and split
constexpr int kStaticMaxDevices = 64;

struct StaticLayout {
    static constexpr size_t status = 0;                                                   // 4 x int32
    static constexpr size_t n_seg = 256;                                                  // [units] int32
    static constexpr size_t seq_bad = 512;                                                // [units] int32
    static constexpr size_t total = 768;
};
constexpr size_t kStaticBytes = StaticLayout::total;

// In host code this name is only a handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

struct PerDevice {
    bool ready;
    unsigned char *base;
};
PerDevice g_static_dev[kStaticMaxDevices];

} // namespace
} // namespace ams

extern "C" int ams_select_static(const ams_config *cfg, const float *scores, int32_t score_stride, int32_t n_units,
                                 int32_t seq_len, int32_t budget, int32_t n_segments, int32_t *keep_idx, void *stream)
{
    using namespace ams;
    if (!cfg || !scores || !keep_idx) return AMS_ERR_INVALID_ARG;
    if (n_units < 1 || n_units > kStaticMaxUnits) return AMS_ERR_CAPACITY;
    if (seq_len < 1 || seq_len > kStaticMaxTokens) return AMS_ERR_CAPACITY;
    if (score_stride < seq_len || score_stride > kStaticMaxTokens || score_stride % 16) return AMS_ERR_INVALID_ARG;
    if (budget < 1 || budget >= seq_len) return AMS_ERR_INVALID_ARG;
    if (n_segments < 1 || n_segments > 1024) return AMS_ERR_INVALID_ARG;
    if (cfg->l_min < 1 || cfg->l_max < 0 || cfg->q_min < 0 || cfg->n_sink < 0 || cfg->n_last < 0) return AMS_ERR_INVALID_ARG;
    if (!(cfg->eps > 0.0f) || !(cfg->eps < 1e30f)) return AMS_ERR_INVALID_ARG;
    const long long seg_cap = (long long)n_segments + (cfg->l_max > 0 ? 2LL * (seq_len / cfg->l_max) : 0) + 4;
    if (seg_cap > kStaticSegCap) return AMS_ERR_CAPACITY;

    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kStaticMaxDevices) return AMS_ERR_CUDA;
    PerDevice &pd = g_static_dev[dev];
    if (!pd.ready) {
        // once per device, with that device current: the array's address on this device
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) return AMS_ERR_CUDA;
        pd.base = (unsigned char *)ptr;
        pd.ready = true;
    }
    unsigned char *base = pd.base;

    DevParams p;
    memset(&p, 0, sizeof p);
    p.L = 1; p.B = n_units; p.Bmax = n_units; p.H = 1; p.G = 1; p.W = 0; p.rows = 1;
    p.T_cap = score_stride; p.seg_cap = (int)seg_cap; p.Tk = budget; p.S = n_segments; p.n_dst = (budget + kPage - 1) / kPage;
    p.l_min = cfg->l_min; p.l_max = cfg->l_max; p.q_min = cfg->q_min; p.n_sink = cfg->n_sink; p.n_last = cfg->n_last;
    p.lambda = 0.0f; p.beta = 1.0f; p.eps = cfg->eps; // no credit: the mass of the current scores alone
    p.seq_lens = nullptr;
    p.fixed_len = seq_len;
    p.usage = scores;
    p.scores = const_cast<float *>(scores);
    p.n_seg = (int *)(base + StaticLayout::n_seg);
    p.seq_bad = (int *)(base + StaticLayout::seq_bad);
    p.keep_idx = keep_idx;
    p.status = (int *)(base + StaticLayout::status);
    if (!segsel_supported(p)) return AMS_ERR_CAPACITY;
    LaunchCtx ctx;
    ctx.s = (cudaStream_t)stream;
    ctx.ev = nullptr;
    ctx.max_ev = 0;
    ctx.begin();
    return launch_segsel(p, ctx, nullptr);
}

// Device-side conditions of the calls above (a segment table that overflowed, a count that did not add up)
// land in a status word inside the same fixed array; this reads and clears it, like ams_get_status does
// for a handle.  Copies 16 bytes, allocates nothing, synchronises `stream`.
extern "C" int ams_select_static_status(int32_t *detail, void *stream)
{
    using namespace ams;
    int32_t host[4] = {0, 0, 0, 0};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kStaticMaxDevices) return AMS_ERR_CUDA;
    const PerDevice &pd = g_static_dev[dev];
    if (pd.ready) {
        cudaStream_t s = (cudaStream_t)stream;
        if (cudaMemcpyAsync(host, pd.base + StaticLayout::status, sizeof host, cudaMemcpyDeviceToHost, s) != cudaSuccess) return AMS_ERR_CUDA;
        if (cudaMemsetAsync(pd.base + StaticLayout::status, 0, sizeof host, s) != cudaSuccess) return AMS_ERR_CUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return AMS_ERR_CUDA;
    }
    if (detail) memcpy(detail, host, sizeof host);
    return host[0];
}
