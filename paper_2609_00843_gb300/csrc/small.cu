// Sorts over narrow ranges with fewer launches.
//
// small_kernel: a whole sort in one CTA, for arrays of a few ten thousand keys over
// a narrow range: histogram (Algorithm 5), local CDF and runs (Algorithm 6) and
// output (Algorithm 7) in shared memory, with nothing but the status word in the
// workspace.
//
// What bounds such a sort is its chain of dependent steps, and as two launches
// also their latency and the host's submission of them.  One CTA's steps take
// longer with more keys, and pass the two launches' at about 24000 (issued one after
// another, us, this kernel / histogram, then scan and output, uniform keys): n = 100, R
// = 100 3.3 / 4.8; n = 8000, R = 1000 4.6 / 6.5; n = 16000, R = 16384 8.1 / 10.7; n = 24000, R =
// 100 6.3 / 5.9, R = 16384 10.1 / 10.6; n = 32000 6.8 / 5.5 and 11.0 / 10.9; before, as three
// launches, n = 10007, R = 1000 11.7.
#include <algorithm>

#include "fill_runs.cuh"

namespace rtcdf {

namespace {

constexpr int kSmallThreads = 1024;
constexpr uint32_t kSmallWarps = kSmallThreads / 32;
// The counters' words, which become a block per warp for the output.
constexpr uint32_t kSmallWords = kSmallWarps * kBlock;
static_assert(kSmallWords >= kSmallMaxR, "the blocks' words hold every counter");
constexpr size_t kSmallSmem = 4 * (kSmallWords + 2 * (size_t)kSmallMaxR);  // of both kernels, at most

// The run table of the R counts in S: run k's end (exclusive, the keys up to its
// value) and key.  Returns the number of keys; *num_runs values are not empty.
// s_keys, s_runs: a word per warp.  The caller synchronises before reading the
// runs.
__device__ __forceinline__ uint32_t runs_of_counts(const uint32_t *S, uint32_t R, uint32_t min_u, uint32_t *s_end,
                                                   int32_t *s_val, uint32_t *s_keys, uint32_t *s_runs,
                                                   int *num_runs) {
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
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
    *num_runs = (int)__reduce_add_sync(0xffffffffu, wr);
    uint32_t end = __reduce_add_sync(0xffffffffu, lane < warp ? wk : 0u) + ikeys - keys;
    uint32_t r = __reduce_add_sync(0xffffffffu, lane < warp ? wr : 0u) + iruns - runs;
    for (uint32_t b = b0; b < b1; b++) {
        const uint32_t c = S[b];
        end += c;
        if (c) {
            s_end[r] = end;
            s_val[r] = (int32_t)(min_u + b);
            r++;
        }
    }
    return total;
}

}  // namespace

__global__ void __launch_bounds__(kSmallThreads, 1) small_kernel(SmallArgs a) {
    extern __shared__ __align__(16) uint32_t S[];  // counters, then the output's blocks | run ends | run keys
    __shared__ uint32_t s_keys[kSmallWarps], s_runs[kSmallWarps];
    uint32_t *s_end = S + kSmallWords;
    int32_t *s_val = reinterpret_cast<int32_t *>(s_end + a.max_runs);
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = a.n, R = a.R;
    for (uint32_t b = tid; b < R; b += kSmallThreads) S[b] = 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    // After a wait that ran out nothing is written until the status has been read.
    const uint32_t status = a.ctl->status;
    const uint32_t head = min(n, (uint32_t)((16 - ((uintptr_t)a.in & 15)) & 15) / 4), nv = (n - head) / 4;
    const int4 *vin = reinterpret_cast<const int4 *>(a.in + head);
    constexpr int V = kSmallMaxN / 4 / kSmallThreads;
    int4 k[V];
#pragma unroll
    for (int u = 0; u < V; u++)
        if (tid + u * kSmallThreads < nv) k[u] = __ldcs(vin + tid + u * kSmallThreads);
    const uint32_t i = tid < head ? tid : head + 4 * nv + (tid - head);  // the keys outside whole vectors
    const int32_t extra = tid < n - 4 * nv ? __ldcs(a.in + i) : 0;
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
    int nw = 0;
    const uint32_t total = runs_of_counts(S, R, a.min_u, s_end, s_val, s_keys, s_runs, &nw);
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
    a.max_runs = R < n ? R : n;
    static std::atomic<uint64_t> raised{0};
    const cudaError_t e = raise_shared_limit((const void *)small_kernel, kSmallSmem, raised);
    if (e != cudaSuccess) return e;
    void *args[] = {&a};
    return launch_first((const void *)small_kernel, 1, kSmallThreads, 4 * (kSmallWords + 2 * (size_t)a.max_runs),
                        args, s);
}

// Scan and output in one launch, for counts H over a narrow range: every CTA (at
// most one per SM) forms the whole run table in its shared memory and writes its
// share of the positions [pos_base, pos_end).  The last CTA to have read H zeroes
// it.  What it saves is a launch of the chain and the run table's way through
// memory (n = 1e6, R = 4096, whole sort from a graph: 9.2 against 12.1 us); each
// CTA reads all of H, 64 KB at R = 16384, which keeps R small.
__global__ void __launch_bounds__(kSmallThreads, 1) finish_kernel(FinishArgs a) {
    extern __shared__ __align__(16) uint32_t S[];  // counts, then the output's blocks | run ends | run keys
    __shared__ uint32_t s_keys[kSmallWarps], s_runs[kSmallWarps], s_last;
    uint32_t *s_end = S + kSmallWords;
    int32_t *s_val = reinterpret_cast<int32_t *>(s_end + a.max_runs);
    const uint32_t tid = threadIdx.x, warp = tid >> 5, R = a.R;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const uint32_t status = a.ctl->status;
    // (H is padded to whole scan chunks of zeros, S to whole vectors)
    for (uint32_t i = tid; i < (R + 3) / 4; i += kSmallThreads)
        reinterpret_cast<uint4 *>(S)[i] = __ldcg(reinterpret_cast<const uint4 *>(a.H) + i);
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&a.ctl->finished, 1u) == gridDim.x - 1;
    int nw = 0;
    const uint32_t total = runs_of_counts(S, R, a.min_u, s_end, s_val, s_keys, s_runs, &nw);
    if (blockIdx.x == 0 && tid == 0 && total != a.n) atomicOr(&a.ctl->status, kDevKeyOutOfRange);
    __syncthreads();
    if (s_last) {  // every CTA has its copy
        for (uint32_t i = tid; i < (R + 3) / 4; i += kSmallThreads)
            reinterpret_cast<uint4 *>(a.H)[i] = make_uint4(0, 0, 0, 0);
        if (tid == 0) a.ctl->finished = 0;
    }
    if ((status & kDevTimeout) || nw == 0) return;
    const uint32_t end = min(a.pos_end, total);
    if (end <= a.pos_base) return;
    const uint32_t head = min(end - a.pos_base, (uint32_t)((16 - ((uintptr_t)a.out & 15)) & 15) / 4);
    const uint32_t hb = a.pos_base + head, nvec = (end - hb) / 4;
    // The CTA's vectors, and its warps' (multiples of 32 of them).
    const uint32_t per_cta = ((nvec + gridDim.x - 1) / gridDim.x + 31) & ~31u;
    const uint32_t v0 = min(nvec, blockIdx.x * per_cta), v1 = min(nvec, v0 + per_cta);
    const uint32_t per_warp = ((v1 - v0 + kSmallWarps - 1) / kSmallWarps + 31) & ~31u;
    const uint32_t wb = v0 + warp * per_warp;
    int4 *vout = reinterpret_cast<int4 *>(a.out + head);
    fill_short_runs(S + warp * kBlock, s_end, s_val, nw, hb, wb, min(v1, wb + per_warp), (int32_t)(a.min_u - 1u),
                    [&](uint32_t v, int4 x) { __stcs(vout + v, x); });
    if (blockIdx.x == 0 && tid < end - a.pos_base - 4 * nvec) {
        const uint32_t p = tid < head ? a.pos_base + tid : hb + 4 * nvec + (tid - head);
        a.out[p - a.pos_base] = s_val[first_run_after(s_end, 0, nw - 1, p)];
    }
}

cudaError_t launch_finish(const FinishArgs &args, int sms, cudaStream_t s) {
    FinishArgs a = args;
    a.max_runs = a.R;
    static std::atomic<uint64_t> raised{0};
    cudaError_t e = raise_shared_limit((const void *)finish_kernel, kSmallSmem, raised);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((uint32_t)std::min<uint64_t>(sms, ((uint64_t)a.pos_end - a.pos_base + 2047) / 2048));
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = 4 * (kSmallWords + 2 * (size_t)a.max_runs);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, finish_kernel, a);
}

}  // namespace rtcdf
