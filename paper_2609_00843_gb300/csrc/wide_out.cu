// Scan and output of a wide range in one launch, after a histogram by partition
// (part.cu), whose buckets' key counts say where each bucket's output begins.
//
// A tile is half a bucket (16384 values), an item a tile or a share of its
// positions: the CTA reads the tile's counts, forms their CDF in shared memory
// (Algorithm 6: the keys before the tile are its offset) and writes the item's
// positions from it (Algorithm 7's rule).  There is no run table in memory, and
// nothing waits on another CTA: the last of a tile's items to have read its counts
// zeroes them, the last CTA of the grid the tickets.
//
// It replaces a scan that reads H twice and writes 8 bytes a value, and an output
// kernel that reads those: at 6 keys a value and R = 2^24 that is 64 MB read
// and zeroed and 400 MB written, instead of 256 + 530 MB.  What bounds it is the
// output's stores, and an item's chain of reading and scanning its tile
// (about 3 us), which the SM's other CTA covers: two CTAs with tiles of 16384
// values against one with 32768 423 / 438 us (R = 2^24, n = 1e8, uniform, whole
// sort).  Tables of more than half the tile's values are kept as the plain CDF, an
// entry for every value; below that the empty values are left out (one warp that
// steps over them took 511 us for normal keys, 412 now, and 207 against 79 at n =
// 1e6).
#include <algorithm>

#include "fill_runs.cuh"

namespace rtcdf {

namespace {
constexpr int kThreads = 512;
constexpr uint32_t kWarps = kThreads / 32;
constexpr uint32_t kWidth = 1u << kPartShift >> 1;       // values of a tile: half a bucket
constexpr uint32_t kTiles = 2 * kPartMaxBuckets;
constexpr int kBlk = 256;                                // positions at a time
constexpr uint32_t kRow = 4 * kThreads;                  // values of a row
constexpr int kVecs = kWidth / 4 / kThreads;             // vectors of the counts per thread
// Up to so many values with keys: their runs (ends, and keys in the second half of
// the table's place), else the CDF of all values.
constexpr uint32_t kSparse = kWidth / 2;
constexpr size_t kSmem = 4 * (kWidth + kWarps * kBlk);  // the CDF, then a block per warp
static_assert(kPartMaxBuckets <= kThreads, "one thread per bucket");
constexpr uint32_t kDoneShift = 12;                      // (fewer CTAs than 4096, fewer items than 2^20)
}  // namespace

__global__ void __launch_bounds__(kThreads, 2) wide_out_kernel(WideOutArgs a) {
    extern __shared__ __align__(16) uint32_t S[];
    __shared__ uint32_t s_start[kTiles + 1];  // positions before each tile
    __shared__ uint32_t s_begin[kTiles + 1];  // items before each tile
    __shared__ uint32_t s_warp[kWarps], s_rows[kVecs * kWarps], s_tot[kVecs], s_runs[kVecs * kWarps], s_run_tot[kVecs];
    __shared__ uint32_t s_item, s_last;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, B = a.buckets;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (a.ctl->status & kDevTimeout) return;  // (part_kernel has written nothing)
    auto warp_incl = [&](uint32_t x) -> uint32_t {
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= (uint32_t)d) x += y;
        }
        return x;
    };
    auto block_incl = [&](uint32_t x, uint32_t *total) -> uint32_t {
        const uint32_t inc = warp_incl(x);
        if (lane == 31) s_warp[warp] = inc;
        __syncthreads();
        const uint32_t w = lane < kWarps ? s_warp[lane] : 0u;
        *total = __reduce_add_sync(0xffffffffu, w);
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
        __syncthreads();
        return before + inc;
    };
    // A thread has a bucket: its tiles' first positions, and their items from their
    // keys (in 16s) and the cost of a tile.  Every CTA computes the same numbers.
    uint32_t start = 0, t0 = 0, t1 = 0;
    if (tid < B) {
        start = a.starts[tid];
        t0 = a.half[tid];
        t1 = a.starts[tid + 1] - start - t0;
        // (keys past the last value, in no tile)
        if ((2 * tid + 1) * kWidth >= a.R && t1) t1 = 0, atomicOr(&a.ctl->status, kDevKeyOutOfRange);
    }
    uint32_t total = 0, items = 0;
    auto cost = [&](uint32_t t) { return t ? t / 16 + a.tile_cost : 0u; };
    block_incl(cost(t0) + cost(t1), &total);
    const uint32_t target = max(1u, total / a.target_items);
    auto share = [&](uint32_t t) { return t ? max(1u, t / 16 / target) : 0u; };
    const uint32_t incl = block_incl(share(t0) + share(t1), &items);
    if (tid < B) {
        s_start[2 * tid] = start;
        s_start[2 * tid + 1] = start + t0;
        s_start[2 * tid + 2] = start + t0 + t1;  // (the same from the next bucket)
        s_begin[2 * tid + 1] = incl - share(t1);
        s_begin[2 * tid + 2] = incl;
    }
    if (tid == 0) {
        s_begin[0] = 0;
        // (keys outside the range are in no bucket, or past the last one's values)
        if (blockIdx.x == 0 && a.starts[B] != a.n) atomicOr(&a.ctl->status, kDevKeyOutOfRange);
    }
    const uint32_t head = (uint32_t)((16 - ((uintptr_t)a.out & 15)) & 15) / 4;
    int4 *vout = reinterpret_cast<int4 *>(a.out + head);  // vector v: positions head + 4 v on
    uint32_t done = 0;  // items
    for (;; done++) {
        if (tid == 0) {
            s_item = done ? gridDim.x + atomicAdd(&a.ctl->scan_ticket, 1u) : blockIdx.x;
            s_last = 0;
        }
        __syncthreads();
        const uint32_t item = s_item;
        if (item >= items) break;
        const uint32_t b = (uint32_t)first_run_after(s_begin + 1, 0, 2 * (int)B - 1, item);
        const uint32_t sub = item - s_begin[b], k = s_begin[b + 1] - s_begin[b];
        const uint32_t base = s_start[b], keys = s_start[b + 1] - base;
        const uint32_t w = min(kWidth, a.R - b * kWidth);
        // The tile's counts: row r holds values kRow r on, a vector per thread.
        uint4 *H4 = reinterpret_cast<uint4 *>(a.H + (size_t)b * kWidth) + tid;
        uint4 c[kVecs];
        uint32_t inc[kVecs];
#pragma unroll
        for (int r = 0; r < kVecs; r++)  // (H is padded to whole rows of zeros)
            c[r] = kRow * r < w ? __ldcg(H4 + r * kThreads) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int r = 0; r < kVecs; r++) {
            inc[r] = warp_incl(c[r].x + c[r].y + c[r].z + c[r].w);
            const uint32_t runs =
                __reduce_add_sync(0xffffffffu, (c[r].x > 0) + (c[r].y > 0) + (c[r].z > 0) + (c[r].w > 0));
            if (lane == 31) s_rows[r * kWarps + warp] = inc[r], s_runs[r * kWarps + warp] = runs;
        }
        if (k == 1)
#pragma unroll
            for (int r = 0; r < kVecs; r++)
                if (kRow * r < w) H4[r * kThreads] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        if (k > 1 && tid == 0) s_last = atomicAdd(&a.read[b], 1u) == k - 1;
        if (warp < kVecs) {  // keys before each warp's part of row `warp`, and its total
            const uint32_t at = warp * kWarps + lane % kWarps;
            const uint32_t x = lane < kWarps ? s_rows[at] : 0u, i = warp_incl(x);
            const uint32_t y = lane < kWarps ? s_runs[at] : 0u, j = warp_incl(y);
            __syncwarp();
            if (lane < kWarps) s_rows[at] = i - x, s_runs[at] = j - y;
            if (lane == 31) s_tot[warp] = i, s_run_tot[warp] = j;
        }
        __syncthreads();
        const uint32_t ti = warp_incl(lane < kVecs ? s_tot[lane] : 0u);
        const uint32_t tr = warp_incl(lane < kVecs ? s_run_tot[lane] : 0u);
        const uint32_t sum = __shfl_sync(0xffffffffu, ti, kVecs - 1), runs = __shfl_sync(0xffffffffu, tr, kVecs - 1);
        const int32_t none = (int32_t)(a.min_u + b * kWidth - 1u);  // (no key of the tile)
        const bool sparse = runs <= kSparse;
        int32_t *s_val = reinterpret_cast<int32_t *>(S + kWidth / 2);
#pragma unroll
        for (int r = 0; r < kVecs; r++) {
            const uint32_t row = r ? __shfl_sync(0xffffffffu, ti, r - 1) : 0u;
            uint4 e;
            e.w = base + row + s_rows[r * kWarps + warp] + inc[r];
            e.z = e.w - c[r].w;
            e.y = e.z - c[r].z;
            e.x = e.y - c[r].y;
            if (!sparse) {
                reinterpret_cast<uint4 *>(S)[r * kThreads + tid] = e;
            } else {
                auto lanes_before = [&](uint32_t x) {
                    return __popc(__ballot_sync(0xffffffffu, x > 0) & ((1u << lane) - 1u));
                };
                uint32_t q = (r ? __shfl_sync(0xffffffffu, tr, r - 1) : 0u) + s_runs[r * kWarps + warp] +
                             lanes_before(c[r].x) + lanes_before(c[r].y) + lanes_before(c[r].z) + lanes_before(c[r].w);
                const int32_t v = (int32_t)((uint32_t)none + 1u + 4u * (r * kThreads + tid));
                if (c[r].x) S[q] = e.x, s_val[q++] = v;
                if (c[r].y) S[q] = e.y, s_val[q++] = v + 1;
                if (c[r].z) S[q] = e.z, s_val[q++] = v + 2;
                if (c[r].w) S[q] = e.w, s_val[q] = v + 3;
            }
        }
        if (tid == 0 && sum != keys) atomicOr(&a.ctl->status, kDevKeyOutOfRange);
        __syncthreads();
        // Positions [p0, p1) of the array (a tile's positions, evenly split).
        const uint32_t p0 = base + (uint32_t)((uint64_t)keys * sub / k);
        const uint32_t p1 = min(base + (uint32_t)((uint64_t)keys * (sub + 1) / k), base + min(sum, keys));
        if (p0 < p1) {
            const uint32_t w_lo = p0 > head ? (p0 - head + 3) / 4 : 0u, w_hi = p1 > head ? (p1 - head) / 4 : 0u;
            const uint32_t nvec = w_hi > w_lo ? w_hi - w_lo : 0u;
            const uint32_t per_warp = ((nvec + kWarps - 1) / kWarps + 31) & ~31u;
            const uint32_t wb = w_lo + warp * per_warp;
            const uint32_t we = min(w_hi, wb + per_warp);
            uint32_t *m = S + kWidth + warp * kBlk;
            const int nw = (int)(sparse ? runs : w);
            auto store = [&](uint32_t v, int4 x) { __stcs(vout + v, x); };
            if (sparse) fill_short_runs<false, kBlk>(m, S, s_val, nw, head, wb, we, none, store);
            else fill_short_runs<true, kBlk>(m, S, nullptr, nw, head, wb, we, none, store);
            // The positions outside whole vectors, at most three at each end.
            const uint32_t q_lo = nvec ? head + 4 * w_lo : p1, q_hi = nvec ? head + 4 * w_hi : p1;
            const uint32_t p = tid < q_lo - p0 ? p0 + tid : q_hi + (tid - (q_lo - p0));
            if (tid < 8 && p < p1) {
                const int j = first_run_after(S, 0, nw - 1, p);
                a.out[p] = sparse ? s_val[j] : (int32_t)((uint32_t)none + 1u + (uint32_t)j);
            }
        }
        if (s_last) {
#pragma unroll
            for (int r = 0; r < kVecs; r++)
                if (kRow * r < w) H4[r * kThreads] = make_uint4(0, 0, 0, 0);
            if (tid == 0) a.read[b] = 0;
        }
        __syncthreads();  // the CDF has been read
    }
    if (tid == 0) {
        s_last = 0;
        // CTAs that are done in the low bits, their items above.  The last one
        // leaves the tickets zero; items missing from the count (a workspace whose
        // ticket was not zero) were not written.
        const uint32_t before = atomicAdd(&a.ctl->finished, done << kDoneShift | 1u);
        if ((before & ((1u << kDoneShift) - 1)) == gridDim.x - 1) {
            if ((before >> kDoneShift) + done != items) atomicOr(&a.ctl->status, kDevTimeout);
            a.ctl->scan_ticket = a.ctl->part_ticket = a.ctl->finished = 0;
            s_last = 1;
        }
    }
    __syncthreads();
    if (s_last && tid < B) a.half[tid] = 0;  // (every CTA has read them)
}

cudaError_t launch_wide_out(const WideOutArgs &args, int sms, cudaStream_t s) {
    WideOutArgs a = args;
    a.buckets = (a.R + 2 * kWidth - 1) / (2 * kWidth);
    // Reading and scanning a tile takes about as long as writing 22000 positions.  One
    // item a CTA: with more of them the tiles' cost grows (n = 2e7, R = 2^20: 90 us,
    // with three items for two CTAs 95, with two items a CTA 97).
    a.tile_cost = 22000 / 16;
    a.target_items = 2 * (uint32_t)sms;
    cudaError_t e = cudaFuncSetAttribute(wide_out_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (uint32_t)sms);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, wide_out_kernel, a);
}

}  // namespace rtcdf
