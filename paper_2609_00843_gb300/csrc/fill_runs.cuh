// Output positions from a window of the run table in shared memory, for the
// single-array and the segmented output kernels.
#pragma once

#include "rtcdf_internal.h"

namespace rtcdf {

// Vectors of four positions that begin before position p, p = 2^32 - 1 included.
__device__ __forceinline__ uint32_t vec_ceil(uint32_t p) { return (p >> 2) + ((p & 3) != 0); }

// Smallest j in [lo, hi] with s_end[j] > p, given s_end[hi] > p.
__device__ __forceinline__ int first_run_after(const uint32_t *s_end, int lo, int hi, uint32_t p) {
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (s_end[mid] > p) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// The same when the answer is expected close to lo: probes lo, lo + 1,
// lo + 3, lo + 7, ... until s_end exceeds p, then a binary search inside the
// last step -- O(log(j - lo)) reads, so a lane that crosses a few short runs
// between its vectors does not pay a search over the whole window.
__device__ __forceinline__ int next_run_after(const uint32_t *s_end, int lo, int hi, uint32_t p) {
    int probe = lo, step = 1;
    while (s_end[probe] <= p) {  // s_end[hi] > p ends it
        lo = probe + 1;
        probe = min(hi, probe + step);
        step <<= 1;
    }
    return first_run_after(s_end, lo, probe, p);
}

// Short runs: a warp's vectors [wb, we) (positions from `frame` on, four a
// vector), BLK positions at a time.  The warp writes the key of every run
// that begins in the block to its first position in `m` (kBlock words of shared
// memory, `none` elsewhere: no key of the array), reads it back as vectors and
// carries the last key before it into every position without one: a ballot
// finds the lane that holds it.  The same rule as the searches (Algorithm 7),
// at a cost that hardly depends on the runs' lengths: the searches take 47 to 129
// instructions for 128 positions, bound by issue below about 200 positions a
// run.  Measured (n = 1e8, output kernel, us, uniform / normal, with the
// searches before that): R = 2^20 59 / 61 (86 / 72), 2^22 64 / 72 (117 / 109), 2^24
// 107 / 94 (172 / 143; 134 MB of runs are read besides); n = 3e7, R = 1e6: 29 (57).
constexpr int kBlock = 512;

//
// CDF: the table has an entry for every value (s_val unused, the first value's key
// is none + 1); a value without keys, whose entry repeats the one before, begins
// no run.
template <bool CDF = false, int BLK = kBlock, class Store>
__device__ __forceinline__ void fill_short_runs(uint32_t *m, const uint32_t *s_end, const int32_t *s_val, int nw,
                                                uint32_t frame, uint32_t wb, uint32_t we, int32_t none, Store store) {
    const int lane = threadIdx.x & 31;
    auto key = [&](int r) { return CDF ? (int32_t)((uint32_t)none + 1u + (uint32_t)r) : s_val[r]; };
    if (wb >= we) return;
    int4 *m4 = reinterpret_cast<int4 *>(m);
    int j = first_run_after(s_end, 0, nw - 1, frame + 4 * wb);  // the run of the block's first position
    for (uint32_t w = wb; w < we; w += BLK / 4) {
        // The block's last position: q0 + BLK passes 2^32 in an array of nearly as many keys.
        const uint32_t q0 = frame + 4 * w, q_last = q0 + (min((uint32_t)BLK, 4 * (we - w)) - 1);
#pragma unroll
        for (int k = 0; k < BLK / 128; k++) m4[lane + 32 * k] = make_int4(none, none, none, none);
        int32_t carry = key(j);
        __syncwarp();
        for (int r = j + 1 + lane;; r += 32) {
            const uint32_t start = r < nw ? s_end[r - 1] : 0xffffffffu;
            const bool begins = start <= q_last;  // (2^32 - 1 is no position)
            // (start < q0 only where a caller's counts pass 2^32: any place in the block)
            if (begins && (!CDF || s_end[r] > start)) m[min(start - q0, (uint32_t)BLK - 1)] = (uint32_t)key(r);
            const unsigned b = __ballot_sync(0xffffffffu, begins);
            j += __popc(b);
            if (b != 0xffffffffu) break;
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < BLK / 128; k++) {
            int4 x = m4[lane + 32 * k];
            const int32_t last = x.w != none ? x.w : x.z != none ? x.z : x.y != none ? x.y : x.x;
            const unsigned has = __ballot_sync(0xffffffffu, last != none);
            const unsigned before = has & ((1u << lane) - 1u);
            const int32_t from = __shfl_sync(0xffffffffu, last, before ? 31 - __clz(before) : 0);
            const int32_t next = __shfl_sync(0xffffffffu, last, has ? 31 - __clz(has) : 0);
            if (x.x == none) x.x = before ? from : carry;
            if (x.y == none) x.y = x.x;
            if (x.z == none) x.z = x.y;
            if (x.w == none) x.w = x.z;
            if (has) carry = next;
            const uint32_t v = w + lane + 32 * k;
            if (v < we) store(v, x);
        }
        __syncwarp();  // the block has been read
    }
}

}  // namespace rtcdf
