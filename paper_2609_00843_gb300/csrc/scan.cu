// Local CDFs and tile offsets (Section 3.1 and Algorithm 6) in one pass.
//
// The paper scans each tile's slice of H in place (one CTA per tile), then a
// single thread accumulates the tile totals into O[t].  Here one scan over
// H[0..R-1] produces, for every value v,
//     O[t] + C_t[v - b_t] = sum_{u<=v} c_u,
// i.e. the tile offset plus the local CDF (Lemmas 1-2), which is exactly the
// exclusive end of v's output interval (Lemma 3).  In the same pass each value
// with c_v > 0 is given a run index k (a second prefix count) and the run table
//     run_end[k] = sum_{u<=v} c_u,   run_val[k] = minVal + v
// is written, so that output generation never walks empty values.
//
// Each output CTA needs the run holding its first position.  Every scan CTA
// has its chunk's runs in shared memory and, for the output CTAs whose first
// position falls inside the chunk's positions, finds that run with the rule of
// Algorithm 7 (first run whose end exceeds the position) by binary search -- a
// handful of steps per output CTA whatever the distribution.
//
// H is zeroed as it is read, leaving the workspace ready for the next sort.
// The bins go in chunks of kScanChunk, and each CTA takes a contiguous range of
// chunks (at most two CTAs per SM, so one chunk each up to R = 2^20).  It adds
// up its range, publishes the sum, and gets its prefix by adding the sums of
// all CTAs before it, read side by side; CTAs with several chunks then read
// their range again (from L2).  No CTA's sum waits for another's, so the
// exchange is one round trip whatever the number of CTAs.  Ranges are handed
// out by an atomic ticket so that a CTA only ever waits for CTAs that are
// running; every wait is bounded by kMaxSpin and records kDevTimeout when it
// gives up.
//
// What bounds it: the launch and the exchange up to R = 2^18 (n = 1e8, kernel
// alone: 9.0 us at 2^18, 13.9 with a lookback over 32 chunks at a time), memory
// beyond (2^24 with every value present: 82 us for 64 MB read twice, zeroed and
// 128 MB of runs written; 340 with one lookback chunk per CTA, whose chain and
// uncoalesced run stores bound it).
//
// The total count is compared with n: every in-range key is counted
// by exactly one tile, so a shortfall means some key lies outside
// [minVal, maxVal).
#include <algorithm>

#include "rtcdf_internal.h"

namespace rtcdf {

// Published sum: bits 0..31 count, bits 32..56 non-empty values, bit 62 set.
constexpr uint64_t kStatePublished = 1ull << 62;
constexpr uint64_t kValueMask = (1ull << 62) - 1;

__device__ __forceinline__ void store_release(uint64_t *p, uint64_t v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t load_acquire(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// A count of keys (mod 2^32) and of non-empty values, kept apart: counts that do
// not add up (a caller's own) never reach the run indices.
struct Pair {
    uint32_t keys, runs;
};
__device__ __forceinline__ Pair operator+(Pair x, Pair y) { return Pair{x.keys + y.keys, x.runs + y.runs}; }
__device__ __forceinline__ Pair bins_sum(const uint4 &h) {
    return Pair{h.x + h.y + h.z + h.w, (uint32_t)(h.x > 0) + (h.y > 0) + (h.z > 0) + (h.w > 0)};
}
__device__ __forceinline__ Pair warp_sum(Pair x) {
    return Pair{__reduce_add_sync(0xffffffffu, x.keys), __reduce_add_sync(0xffffffffu, x.runs)};
}

// Shared index of the chunk's r-th run: one padding word per 32, so that the
// four consecutive runs of each lane of a dense chunk fall in distinct banks.
__device__ __forceinline__ uint32_t run_slot(uint32_t r) { return r + (r >> 5); }

// One CTA per chunk range.  MULTI: some ranges hold several chunks.
template <bool MULTI>
__global__ void __launch_bounds__(kScanThreads, 2) scan_kernel(ScanArgs a) {
    __shared__ uint32_t s_slot;
    __shared__ Pair s_warp[kScanThreads / 32], s_part[kScanThreads / 32];
    __shared__ uint32_t s_end[kScanChunk + kScanChunk / 32];
    __shared__ int32_t s_val[kScanChunk + kScanChunk / 32];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // Launched as a programmatic dependent of the histogram.  The ticket does
    // not depend on it, so it is taken first: the counter was reset by the previous
    // sort's output kernel, which is done before any CTA here starts, because every
    // CTA of the launch before waits for its own predecessors before it lets this one
    // be scheduled or returns (as hist_tiles does).  Then wait until the histogram
    // grid has finished and its writes are visible, and let the output kernel be
    // scheduled (it waits for this grid in the same way).
    const bool single = (a.ctas == 1);  // no exchange at all
    if (!single) {
        if (tid == 0) s_slot = atomicAdd(&a.ctl->scan_ticket, 1u);
        __syncthreads();
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const uint32_t slot = single ? 0u : s_slot;
    // A ticket past the last CTA only happens with a workspace whose ticket
    // was not zero (not cleared, or shared by unordered calls): take no chunk
    // and record kDevTimeout, since the range that ticket stood for is never
    // published (its successors' waits would run out too) and the output
    // kernel must not trust this sort's run table.
    if (slot >= a.ctas) {
        if (tid == 0) atomicOr(&a.ctl->status, kDevTimeout);
        return;
    }
    const uint32_t c0 = (uint32_t)((uint64_t)slot * a.chunks / a.ctas);
    const uint32_t c1 = (uint32_t)((uint64_t)(slot + 1) * a.chunks / a.ctas);
    uint4 *H4 = reinterpret_cast<uint4 *>(a.H) + tid;  // (H is padded to whole chunks)
    constexpr uint32_t kVec = kScanChunk / 4;          // vectors of a chunk, one per thread

    // The range's sum, published; then the sums of the CTAs before.
    uint4 h = H4[(size_t)c0 * kVec];
    Pair before{0, 0};
    if (!single) {
        Pair sum = bins_sum(h);
        if (MULTI) {
#pragma unroll 8
            for (uint32_t c = c0 + 1; c < c1; c++) sum = sum + bins_sum(H4[(size_t)c * kVec]);
        }
        sum = warp_sum(sum);
        if (lane == 0) s_part[warp] = sum;
        __syncthreads();
        if (warp == 0) {
            const Pair total = warp_sum(s_part[lane]);
            if (lane == 0) store_release(&a.state[slot], kStatePublished | (uint64_t)total.runs << 32 | total.keys);
        }
        Pair mine{0, 0};
        bool timed_out = false;
        for (uint32_t i = tid; i < slot; i += kScanThreads) {
            uint64_t st = load_acquire(&a.state[i]);
            for (uint32_t spins = 0; st == 0 && !timed_out; spins++) {
                if (spins > kMaxSpin) timed_out = true;
                __nanosleep(64);
                st = load_acquire(&a.state[i]);
            }
            mine = mine + Pair{(uint32_t)st, (uint32_t)((st & kValueMask) >> 32)};
        }
        if (timed_out) atomicOr(&a.ctl->status, kDevTimeout);
        mine = warp_sum(mine);
        if (lane == 0) s_warp[warp] = mine;
        __syncthreads();
        before = warp_sum(s_warp[lane]);
        __syncthreads();  // s_warp is used again below
    }

    for (uint32_t chunk = c0; chunk < c1; chunk++) {
        const uint32_t base = chunk * kScanChunk + tid * kScanItems;
        // Four counts, zeroed behind us; the next chunk's are on their way.
        uint4 next = make_uint4(0, 0, 0, 0);
        if (MULTI && chunk + 1 < c1) next = H4[(size_t)(chunk + 1) * kVec];
        H4[(size_t)chunk * kVec] = make_uint4(0, 0, 0, 0);
        const uint32_t c[kScanItems] = {h.x, h.y, h.z, h.w};
        if (a.dbg_hist) {
#pragma unroll
            for (int i = 0; i < kScanItems; i++)
                if (base + i < a.R) a.dbg_hist[base + i] = c[i];
        }
        // Block scan.
        const Pair own = bins_sum(h);
        Pair inc = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const Pair y{__shfl_up_sync(0xffffffffu, inc.keys, d), __shfl_up_sync(0xffffffffu, inc.runs, d)};
            if (lane >= d) inc = inc + y;
        }
        if (lane == 31) s_warp[warp] = inc;
        __syncthreads();  // (also: the previous chunk's runs have been read)
        const Pair wt = s_warp[lane];
        const Pair total = warp_sum(wt), ahead = warp_sum(lane < warp ? wt : Pair{0, 0});
        // Keys of the array and runs of the chunk before this thread's bins.
        uint32_t end = before.keys + ahead.keys + inc.keys - own.keys;
        uint32_t runs = ahead.runs + inc.runs - own.runs;
#pragma unroll
        for (int i = 0; i < kScanItems; i++) {
            const uint32_t v = base + i;
            end += c[i];  // sum_{u<=v} c_u
            if (c[i] > 0) {
                s_end[run_slot(runs)] = end;
                s_val[run_slot(runs)] = (int32_t)((uint32_t)a.minVal + v);
                runs++;
            }
            if (a.dbg_cdf && v < a.R) a.dbg_cdf[v] = end;
            if (a.dbg_offset && v < a.R && (v % a.T) == 0) a.dbg_offset[v / a.T] = end - c[i];
            if (v == a.R - 1) {
                a.ctl->num_runs = before.runs + runs;
                if (end != (uint32_t)a.n) atomicOr(&a.ctl->status, kDevKeyOutOfRange);
            }
        }
        __syncthreads();
        // The chunk's runs, written out coalesced.
        const uint32_t chunk_runs = total.runs, run_base = before.runs;
        for (uint32_t r = tid; r < chunk_runs; r += kScanThreads) {
            a.run_end[run_base + r] = s_end[run_slot(r)];
            a.run_val[run_base + r] = s_val[run_slot(r)];
        }
        // Output CTA j starts at P0(j): P0(0) = pos_base, P0(j) = pos_base +
        // head + j * fill_chunk, all inside [pos_base, pos_end).  The chunk's
        // values cover positions [pos_lo, pos_hi); only the part inside the
        // written window can hold a CTA's first position.
        const uint32_t pos_lo = max(before.keys, a.pos_base);
        const uint32_t pos_hi = min(before.keys + total.keys, a.pos_end);
        if (pos_hi > pos_lo) {
            const uint32_t fc = (uint32_t)a.fill_chunk, head = a.head, pb = a.pos_base;
            // First CTA j with P0(j) >= pb + l (P0 is increasing in j).
            auto first_cta_at_or_after = [&](uint32_t l) -> uint32_t {
                if (l == 0) return 0u;
                if ((uint64_t)l <= (uint64_t)head + fc) return 1u;
                return (uint32_t)(((uint64_t)l - head + fc - 1) / fc);
            };
            const uint32_t j_lo = first_cta_at_or_after(pos_lo - pb);
            const uint32_t j_hi = min(first_cta_at_or_after(pos_hi - pb), a.fill_ctas);
            for (uint32_t j = j_lo + tid; j < j_hi; j += kScanThreads) {
                const uint32_t p0 = pb + ((j == 0) ? 0u : head + j * fc);
                // First run of the chunk whose end exceeds p0 (Algorithm 7's rule).
                uint32_t lo = 0, hi = chunk_runs - 1;
                while (lo < hi) {
                    const uint32_t mid = (lo + hi) >> 1;
                    if (s_end[run_slot(mid)] > p0) hi = mid; else lo = mid + 1;
                }
                a.start_run[j] = run_base + lo;
            }
        }
        before = before + total;
        h = next;
    }
}

cudaError_t launch_scan(const ScanArgs &args, int sms, cudaStream_t s) {
    ScanArgs a = args;
    a.ctas = std::min<uint32_t>(a.chunks, 2u * (uint32_t)sms);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.ctas);
    cfg.blockDim = dim3(kScanThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return a.ctas < a.chunks ? cudaLaunchKernelEx(&cfg, scan_kernel<true>, a)
                             : cudaLaunchKernelEx(&cfg, scan_kernel<false>, a);
}

}  // namespace rtcdf
