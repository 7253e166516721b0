// A whole sort in one CTA, for arrays of a few ten thousand keys over a narrow
// range: histogram (Algorithm 5), local CDF and runs (Algorithm 6) and output
// (Algorithm 7) in shared memory, with nothing but the status word in the
// workspace.
//
// What bounds such a sort is its chain of dependent steps, and as three launches
// also their latency and the host's submission of them.  One CTA's steps take
// longer with more keys, and pass the three launches' at about 32768 keys
// (replayed from a graph, us a sort, uniform keys, this kernel / the three
// launches): n = 100, R = 128 3.7 / 8.1; n = 10007, R = 1000 5.4 / 9.0; n = 16384,
// R = 16384 8.9 / 12.9; n = 32768, R = 128 7.4 / 7.3, R = 16384 11.6 / 12.9; and
// issued one by one from Python: n = 10007, R = 1000 8.2 / 11.7.
#include <atomic>

#include "fill_runs.cuh"

namespace rtcdf {

namespace {

constexpr int kSmallThreads = 1024;
constexpr uint32_t kSmallWarps = kSmallThreads / 32;

}  // namespace

__global__ void __launch_bounds__(kSmallThreads, 1) small_kernel(SmallArgs a) {
    extern __shared__ __align__(16) uint32_t S[];  // counters, then the output's blocks | run ends | run keys
    __shared__ uint32_t s_keys[kSmallWarps], s_runs[kSmallWarps];
    uint32_t *s_end = S + a.words;
    int32_t *s_val = reinterpret_cast<int32_t *>(s_end + a.max_runs);
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = a.n, R = a.R;
    // After a wait that ran out nothing is written until the status has been read.
    const uint32_t status = a.ctl->status;
    const uint32_t head = min(n, (uint32_t)((16 - ((uintptr_t)a.in & 15)) & 15) / 4), nv = (n - head) / 4;
    const int4 *vin = reinterpret_cast<const int4 *>(a.in + head);
    constexpr int V = kSmallMaxN / 4 / kSmallThreads;
    int4 k[V];
#pragma unroll
    for (int u = 0; u < V; u++)
        if (tid + u * kSmallThreads < nv) k[u] = __ldg(vin + tid + u * kSmallThreads);
    const uint32_t i = tid < head ? tid : head + 4 * nv + (tid - head);  // the keys outside whole vectors
    const int32_t extra = tid < n - 4 * nv ? __ldg(a.in + i) : 0;
    for (uint32_t b = tid; b < R; b += kSmallThreads) S[b] = 0;
    __syncthreads();
    const uint32_t s_base = (uint32_t)__cvta_generic_to_shared(S);
    auto count = [&](int32_t key) {
        const uint32_t y = (uint32_t)key - a.min_u;
        asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %0, %1;\n\t@p red.shared.add.u32 [%2], 1;\n\t}" ::"r"(y),
                     "r"(R), "r"(s_base + 4u * y));
    };
#pragma unroll
    for (int u = 0; u < V; u++)
        if (tid + u * kSmallThreads < nv) { count(k[u].x); count(k[u].y); count(k[u].z); count(k[u].w); }
    if (tid < n - 4 * nv) count(extra);
    __syncthreads();
    // Keys and non-empty values before each thread's bins (an odd number of
    // consecutive ones: the lanes of a warp step through 32 banks).
    const uint32_t per = ((R + kSmallThreads - 1) / kSmallThreads) | 1u;
    const uint32_t b0 = min(R, tid * per), b1 = min(R, b0 + per);
    uint32_t keys = 0, runs = 0;
    for (uint32_t b = b0; b < b1; b++) {
        keys += S[b];
        runs += S[b] > 0;
    }
    uint32_t ikeys = keys, iruns = runs;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, ikeys, d), y = __shfl_up_sync(0xffffffffu, iruns, d);
        if (lane >= (uint32_t)d) ikeys += x, iruns += y;
    }
    if (lane == 31) s_keys[warp] = ikeys, s_runs[warp] = iruns;
    __syncthreads();
    const uint32_t wk = s_keys[lane], wr = s_runs[lane];
    const uint32_t total = __reduce_add_sync(0xffffffffu, wk);
    const int nw = (int)__reduce_add_sync(0xffffffffu, wr);
    uint32_t end = __reduce_add_sync(0xffffffffu, lane < warp ? wk : 0u) + ikeys - keys;
    uint32_t r = __reduce_add_sync(0xffffffffu, lane < warp ? wr : 0u) + iruns - runs;
    for (uint32_t b = b0; b < b1; b++) {
        const uint32_t c = S[b];
        end += c;
        if (c) {
            s_end[r] = end;
            s_val[r] = (int32_t)(a.min_u + b);
            r++;
        }
    }
    if (tid == 0 && total != n) atomicOr(&a.ctl->status, kDevKeyOutOfRange);
    __syncthreads();
    if ((status & kDevTimeout) || nw == 0) return;
    // Positions [0, total): whole vectors by warps, at most three positions
    // before and after them one by one.
    const uint32_t oh = min(total, (uint32_t)((16 - ((uintptr_t)a.out & 15)) & 15) / 4);
    const uint32_t nvec = (total - oh) / 4;
    const uint32_t per_warp = ((nvec + kSmallWarps - 1) / kSmallWarps + 31) & ~31u;
    const uint32_t wb = warp * per_warp;
    int4 *vout = reinterpret_cast<int4 *>(a.out + oh);
    fill_short_runs(S + warp * kBlock, s_end, s_val, nw, oh, wb, min(nvec, wb + per_warp), (int32_t)(a.min_u - 1u),
                    [&](uint32_t v, int4 x) { vout[v] = x; });
    if (tid < total - 4 * nvec) {
        const uint32_t p = tid < oh ? tid : oh + 4 * nvec + (tid - oh);
        a.out[p] = s_val[first_run_after(s_end, 0, nw - 1, p)];
    }
}

cudaError_t launch_small(const int32_t *in, int32_t *out, uint32_t n, uint32_t min_u, uint32_t R, Ctl *ctl,
                         cudaStream_t s) {
    SmallArgs a;
    a.in = in; a.out = out; a.n = n; a.R = R; a.min_u = min_u; a.ctl = ctl;
    a.words = R > kSmallWarps * kBlock ? (R + 3) / 4 * 4 : kSmallWarps * kBlock;
    a.max_runs = R < n ? R : n;
    // The limit is raised once per device (a sort must not pay for it each time).
    static std::atomic<uint64_t> raised{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !(raised.load(std::memory_order_relaxed) >> dev & 1)) {
        constexpr int most = 4 * (kSmallMaxR + 2 * kSmallMaxR);
        e = cudaFuncSetAttribute(small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
        if (dev < 64) raised.fetch_or(1ull << dev, std::memory_order_relaxed);
    }
    small_kernel<<<1, kSmallThreads, 4 * ((size_t)a.words + 2 * (size_t)a.max_runs), s>>>(a);
    return cudaGetLastError();
}

}  // namespace rtcdf
