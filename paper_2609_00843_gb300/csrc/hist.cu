// Range-tile histogram (Algorithm 5, all m tiles in one launch as in Section 3.3).
//
// CTA b works on tile t = b mod m and is the q-th (q = b / m) of the g CTAs of
// that tile -- the paper's interleaving, which keeps the m CTAs that read the
// same part of the input co-resident so that every read after the first is an
// L2 hit.  Each CTA keeps a private histogram S[0..w_t-1] of 32-bit counters
// in shared memory, sweeps the input grid-stride with 16-byte loads, adds 1 to
// S[y] for every key whose position y = key - minVal - b_t inside the tile is
// below w_t (one unsigned compare tests both ends; keys outside [minVal,
// maxVal) fall outside every tile), and finally adds each non-zero S[y] to
// H[b_t + y] with one global atomic.
//
// Out-of-range keys need no per-key test: they are counted by no tile, so the
// histogram total falls short of n, which the scan detects.
//
// On GB300 a single shared-memory copy per CTA sustains the HBM read rate for
// uniform, normal and all-equal inputs alike, so there is no replication.
// Bytes in flight come from unrolled 16-byte loads.  For one tile, bulk L2
// prefetches issued ahead of the loads gave nothing; for 2 to 8 tiles they are
// part of the adaptive form below.
#include <map>
#include <mutex>
#include <tuple>

#include "hist_tiles.cuh"

namespace rtcdf {

template <bool STREAMING, int UNROLL, bool ADAPT, bool FIXED = false>
__global__ void __launch_bounds__(1024) hist_kernel(HistArgs a) {
    extern __shared__ uint32_t S[];
    __shared__ uint32_t s_tc[8];
    hist_tiles<STREAMING, UNROLL, ADAPT, ADAPT, FIXED>(a, blockIdx.x, S, s_tc);
}

// One tile of a long input: one CTA per SM, whose 64 registers a thread hold six
// vectors in flight while six are counted.  Whole sorts one after another, us, against two
// CTAs of 32 registers: n = 1e9, R = 128 1116 / 1142, 4096 1132 / 1158, 16384 1136 / 1176, 49000
// 1124 / 1125; n = 2e8 246.0 / 246.9, 252.0 / 253.1, 252.3 / 255.8, 251.8 / 252.9; below 2e8 keys
// the two are within 1 % of each other either way (1e8: R = 128 125.5 / 126.5, 16384 129.8 /
// 129.2, 49000 134.4 / 133.5), and two leave room for other streams' kernels.
__global__ void __launch_bounds__(1024, 1) hist_long_kernel(HistArgs a) {
    extern __shared__ uint32_t S[];
    hist_tiles<true, 6, false, true, true>(a, blockIdx.x, S, nullptr);
}

// Kernel variant: streaming loads for one tile; the adaptive form for 2 to 8
// tiles; the plain predicated form beyond.  The first two also for launches that are
// not a sort's first (FIXED), which may have nothing to count.
enum HistVariant { kHistStreaming, kHistAdaptive, kHistPlain, kHistStreamingFixed, kHistAdaptiveFixed };
int hist_variant(bool streaming, uint32_t m, bool fixed) {
    if (streaming) return fixed ? kHistStreamingFixed : kHistStreaming;
    return m > 8 ? kHistPlain : fixed ? kHistAdaptiveFixed : kHistAdaptive;
}

const void *hist_fn(int variant, int unroll) {
    const bool deep = unroll == 8;
    switch (variant) {
        case kHistStreaming:
            return deep ? (const void *)hist_kernel<true, 8, false> : (const void *)hist_kernel<true, 4, false>;
        case kHistAdaptive:
            return deep ? (const void *)hist_kernel<false, 8, true> : (const void *)hist_kernel<false, 4, true>;
        case kHistStreamingFixed:
            return deep ? (const void *)hist_kernel<true, 8, false, true>
                        : (const void *)hist_kernel<true, 4, false, true>;
        case kHistAdaptiveFixed:
            return deep ? (const void *)hist_kernel<false, 8, true, true>
                        : (const void *)hist_kernel<false, 4, true, true>;
        default:
            return deep ? (const void *)hist_kernel<false, 8, false> : (const void *)hist_kernel<false, 4, false>;
    }
}

// The deep form (UNROLL = 8) when only one CTA fits on an SM: eight loads in
// flight per thread in the one-tile and plain forms, a six-deep pipeline in
// the 2-to-8-tile form.
int hist_unroll(size_t smem) { return smem > 114 * 1024 ? 8 : 4; }

constexpr uint64_t kHistFixedMinKeys = 500000000;  // (see launch_hist)

cudaError_t launch_hist(const HistArgs &a, int threads, size_t smem, bool streaming, HistLaunch how, cudaStream_t s) {
    // hist_max_ctas_per_sm() has raised the shared-memory limits for this size.
    dim3 grid(a.m * a.g);
    void *args[] = {const_cast<HistArgs *>(&a)};
    // Loads of a fixed input (ld.global.nc) are faster over long inputs of few values
    // (n = 3e8, R = 200000, 100 different keys: 467 us against 562).  The first launch of
    // a sort may overlap the kernel that writes its input, and gains by it up to about
    // 1e8 keys (n = 2e7, R = 2^18, whole sort 83 / 87); over longer inputs it does not.
    if (how == kHistFirst && !streaming && a.m <= 8 && a.n * a.m >= kHistFixedMinKeys) how = kHistAlone;
    const bool fixed = streaming ? a.only_if != nullptr : how != kHistFirst;
    const void *fn = hist_fn(hist_variant(streaming, a.m, fixed), hist_unroll(smem));
    if (a.long_form) fn = (const void *)hist_long_kernel;
    if (how == kHistFirst) return launch_first(fn, grid.x, threads, smem, args, s);
    if (how == kHistDependent) return launch_dependent(fn, grid.x, threads, smem, args, true, s);
    return cudaLaunchKernel(fn, grid, dim3(threads), args, smem, s);
}

// Occupancy of the histogram kernel for a launch shape, cached per device so
// that planning a sort inside CUDA graph capture makes no attribute calls.
cudaError_t hist_max_ctas_per_sm(int threads, size_t smem, bool streaming, int *ctas) {
    static std::mutex mu;
    static std::map<std::tuple<int, int, size_t, bool>, int> cache;
    static std::map<std::pair<int, bool>, size_t> smem_limit;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    auto key = std::make_tuple(dev, threads, smem, streaming);
    auto it = cache.find(key);
    if (it != cache.end()) {
        *ctas = it->second;
        return cudaSuccess;
    }
    // The adaptive and plain multi-tile variants share the same sizes.
    const void *f = hist_fn(streaming ? kHistStreaming : kHistAdaptive, hist_unroll(smem));
    size_t &lim = smem_limit[std::make_pair(dev, streaming)];
    if (smem > lim) {
        for (int v : {kHistStreaming, kHistAdaptive, kHistPlain, kHistStreamingFixed, kHistAdaptiveFixed}) {
            if ((v == kHistStreaming || v == kHistStreamingFixed) != streaming) continue;
            for (int u : {4, 8}) {
                e = cudaFuncSetAttribute(hist_fn(v, u), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (e != cudaSuccess) return e;
            }
        }
        if (streaming) {
            e = cudaFuncSetAttribute(hist_long_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        lim = smem;
    }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, f, threads, smem);
    if (e != cudaSuccess) return e;
    cache[key] = *ctas;
    return cudaSuccess;
}

}  // namespace rtcdf
