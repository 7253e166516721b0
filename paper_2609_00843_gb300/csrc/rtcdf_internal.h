// Internal declarations shared by the RT-CDF kernels and the C-ABI host code.
// Not installed; the public interface is include/rtcdf.h.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/rtcdf.h"

namespace rtcdf {

// Launch parameters of the tuning table for (n, R), if it has an entry
// (tune.cu) that sets any of them; whether the table is the compiled-in one.
bool tune_lookup(uint64_t n, uint32_t R, rtcdf_params *out, bool *builtin);
// Whether the tuning table is the compiled-in one.
bool tune_is_builtin();

// rtcdf_sort_ex by the built-in rules, whatever the tuning table holds (rtcdf_api.cu).
rtcdf_status sort_by_rules(const int32_t *in, int32_t *out, uint64_t n, int64_t minVal, int64_t maxVal, void *ws,
                           size_t ws_bytes, cudaStream_t s);

// Device status bits (mirror RTCDF_DEV_* in rtcdf.h).
constexpr uint32_t kDevKeyOutOfRange = 0x1;
constexpr uint32_t kDevTimeout = 0x2;
constexpr uint32_t kDevBadSegment = 0x4;

// The library-owned workspace of rtcdf_sort_batched for `s` on the current
// device, or null (devplan.cu).
void *batch_stream_workspace(cudaStream_t s);

// Local-CDF scan: a CTA of kScanThreads threads scans kScanChunk histogram bins at a
// time (kScanItems per thread), one chunk or a range of them; the CTAs exchange their
// ranges' sums.
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanChunk = kScanThreads * kScanItems;

// Upper bound on output-generation CTAs (the start-run table has this many slots).
constexpr int kMaxFillCtas = 4096;

// Iteration cap of every device-side wait; a wait that runs out records
// kDevTimeout and the kernel carries on without hanging.
constexpr uint32_t kMaxSpin = 1u << 21;

// Control block at the start of every workspace.
struct Ctl {
    uint32_t status;       // RTCDF_DEV_* bits, sticky until read
    uint32_t scan_ticket;  // chunk ranges of the scan handed out so far (zero between sorts)
    uint32_t num_runs;     // number of values with c_v > 0 (written by the scan)
    uint32_t part_ticket;  // items of bucket_kernel taken so far (zero between sorts)
    uint32_t pack_copies;  // written-out counters of pack_kernel (written before it is read)
    uint32_t finished;     // CTAs of finish_kernel that have read H (zero between sorts)
    uint32_t pack_tiles;   // whether pack_kernel has left the keys to range tiles (written before it is read)
    uint32_t pad[57];
};
static_assert(sizeof(Ctl) == 256, "control block is 256 bytes");

// Most scan chunks any sort can have (RTCDF_MAX_R / kScanChunk).
constexpr uint32_t kMaxScanChunks = (1u << 24) / kScanChunk;

// Byte offsets of the workspace regions for a sort with range size R in a
// workspace of `total` bytes.  Regions that must be zero when a sort starts
// (control block, the scan's published sums, histogram H) sit at fixed offsets from the
// bottom, so they stay zero whatever R the previous sort had; regions that
// each sort writes before reading (run table, start-run table) are anchored
// at the top and may overlap what a previous sort left behind.
struct WsLayout {
    size_t ctl, scan_state, hist, run_end, run_val, start_run, total;
    uint32_t scan_chunks;
    size_t zero_bytes;  // [0, zero_bytes) must be zero when a sort starts
};

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

constexpr size_t kWsHistOffset = 256 + (size_t)kMaxScanChunks * 8;

// H is padded to whole scan chunks.  Its size never decreases as R grows, so a
// sort's run table (anchored at the top) never reaches the part of H
// (anchored at the bottom) that a sort with a smaller range expects zeroed.
inline size_t hist_region_bytes(uint64_t R) {
    return (size_t)((R + kScanChunk - 1) / kScanChunk) * kScanChunk * 4;
}

inline size_t ws_required(uint64_t R) {
    return kWsHistOffset + hist_region_bytes(R) + align_up((size_t)kMaxFillCtas * 4, 256) +
           2 * align_up((size_t)R * 4, 256);
}

inline WsLayout ws_layout(uint64_t R, size_t total) {
    WsLayout L;
    L.scan_chunks = (uint32_t)((R + kScanChunk - 1) / kScanChunk);
    L.ctl = 0;
    L.scan_state = 256;
    L.hist = kWsHistOffset;
    L.zero_bytes = L.hist + hist_region_bytes(R);
    size_t top = total / 256 * 256;
    L.run_val = top - align_up((size_t)R * 4, 256);
    L.run_end = L.run_val - align_up((size_t)R * 4, 256);
    L.start_run = L.run_end - align_up((size_t)kMaxFillCtas * 4, 256);
    L.total = total;
    return L;
}

// Raises a kernel's shared-memory limit to `bytes`, the most that any of its launches
// takes, once per device (bits of `raised`).  Never to one launch's own size: the limit
// belongs to the kernel, and another thread's smaller launch would lower it between
// this thread's raise and launch.
inline cudaError_t raise_shared_limit(const void *kernel, size_t bytes, std::atomic<uint64_t> &raised) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 64 && (raised.load(std::memory_order_relaxed) >> dev & 1)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && dev < 64) raised.fetch_or(1ull << dev, std::memory_order_relaxed);
    return e;
}

inline cudaError_t launch_dependent(const void *fn, uint32_t grid, int threads, size_t smem, void **args,
                                    bool dependent, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

// The first launch of a sort: a programmatic dependent of whatever kernel is before
// it in the stream, unless the stream is being captured (whose last node may be of
// another kind).  The kernel waits for that one before it reads or writes anything
// but its shared memory, and reads its input with loads that are coherent from then
// on (no ld.global.nc); the output kernels let it be scheduled in their tails.
// Sorts issued one after another, us each, before / now: n = 1e4, R = 1000 6.3 / 4.8; 1e6,
// R = 128 8.2 / 6.5, R = 350000 28.3 / 25.0; 3.1e6, R = 50021 28.7 / 25.5; 1e7, R = 200000 44.8 /
// 41.5; 1e8, R = 2^14 133.5 / 131.5.  Used for all range tiles and the one-CTA sort;
// part_kernel and pack_kernel take the shared memory that the output kernel's tail runs
// in and got slower (n = 3e7, R = 1e6 122 / 129; n = 1e8, R = 2^18 158.5 / 166.7).
inline cudaError_t launch_first(const void *fn, uint32_t grid, int threads, size_t smem, void **args, cudaStream_t s) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(s, &cap);
    if (e != cudaSuccess) return e;
    return launch_dependent(fn, grid, threads, smem, args, cap == cudaStreamCaptureStatusNone, s);
}

// ---------------------------------------------------------------- histogram
struct HistArgs {
    const int32_t *in;
    uint64_t n;
    uint64_t nvec;         // 16-byte vectors after the unaligned head
    uint32_t head;         // elements before the first 16-byte aligned address
    uint32_t min_u;        // (uint32_t)minVal
    uint32_t R, T, m, g;   // range size, tile width, tiles, CTAs per tile
    uint32_t *H;           // global histogram, R entries (added to)
    bool long_form = false;  // one tile, one CTA per SM: hist_long_kernel
    const uint32_t *only_if = nullptr;  // nothing is counted when this word is 0
};
// How the histogram is launched: after all earlier work in the stream, as the first
// launch of a whole sort (launch_first), or as a programmatic dependent of the sort's
// launch before it.
enum HistLaunch { kHistAlone, kHistFirst, kHistDependent };
cudaError_t launch_hist(const HistArgs &a, int threads, size_t smem, bool streaming, HistLaunch how, cudaStream_t s);
cudaError_t hist_max_ctas_per_sm(int threads, size_t smem, bool streaming, int *ctas);

// ---------------------------------------------------------------- small arrays
constexpr uint32_t kSmallMaxN = 24576, kSmallMaxR = 16384;
struct SmallArgs {
    const int32_t *in;
    int32_t *out;
    uint32_t n, R, min_u;
    uint32_t max_runs;     // that shared memory has room for
    Ctl *ctl;
};
// The whole sort of n <= kSmallMaxN keys over R <= kSmallMaxR values in one CTA.
cudaError_t launch_small(const int32_t *in, int32_t *out, uint32_t n, uint32_t min_u, uint32_t R, Ctl *ctl,
                         cudaStream_t s);

// Scan and output of counts H over R <= kSmallMaxR values in one launch.
struct FinishArgs {
    uint32_t *H;           // R counts, zeroed
    int32_t *out;          // out[0] holds position pos_base
    uint32_t n, pos_base, pos_end, R, min_u;
    uint32_t max_runs;     // (set by launch_finish)
    Ctl *ctl;
};
cudaError_t launch_finish(const FinishArgs &a, int sms, cudaStream_t s);

// ---------------------------------------------------------------- packed histogram
struct PackArgs {
    HistArgs h;            // (T, m, g: the range tiles of inputs that packed counters cannot hold)
    uint32_t words, fields, magic;
    uint32_t coarse_shift; // the sample's stretches of the range
    float limit;           // expected keys of the fullest field in a round
    uint32_t max_rounds;
    uint32_t *dump;        // written-out counters, or null: added to H by pairs of CTAs
    Ctl *ctl;              // (with dump)
    uint32_t *tiles_later; // written: whether the keys are left to range tiles; null: counted by them here
};
struct PackPlan {
    uint32_t words, fields, magic, max_rounds, ctas, tile, m, g;
    float limit;
    size_t smem;
    uintptr_t dump;
};
// The plan for n keys over R values; scratch: n words, or 0.  False when the
// range does not fit.
bool pack_plan(uint64_t n, uint32_t R, uint64_t nvec, uintptr_t scratch, int sms, PackPlan *p);
// ctl: the control block of a whole sort, or null (no scratch).  tiles_later: keys that
// packed counters cannot hold are left to a launch of the range tiles that follows
// (Ctl::pack_tiles).
cudaError_t launch_pack(const PackPlan &p, const HistArgs &hist, Ctl *ctl, bool tiles_later, cudaStream_t s);

// ---------------------------------------------------------------- histogram by partition
constexpr int kPartShift = 15;  // values per bucket, log2
constexpr uint32_t kPartMaxBuckets = 512;

struct PartArgs {
    const int32_t *in;
    uint64_t n, nvec;      // keys; 16-byte vectors after the unaligned head
    uint32_t head, min_u, R;
    uint32_t buckets;      // ranges of 2^15 values
    uint32_t slabs, slab_keys;
    uint32_t slab_units;   // 16-byte units between the slabs in `payload`
    uint32_t part_ctas;    // CTAs of part_kernel
    uint32_t tile_cost;    // of an item, in 16 keys, beside its keys
    uint32_t target_items; // items bucket_kernel aims at
    int4 *payload;         // per slab: its buckets' keys, 16 bits each
    uint16_t *starts;      // per slab: buckets + 1 starts (units)
    uint32_t *rows;        // per CTA of part_kernel: its keys of each bucket
    uint32_t *H;           // global histogram, R entries (zero on entry)
    uint32_t *bucket_start;  // written: keys before each bucket, buckets + 1
    uint32_t *half;        // null, or added to: keys in the lower half of each bucket (zero on entry)
    Ctl *ctl;
};
struct PartPlan {
    uint32_t buckets, slabs, slab_keys, slab_units, ctas;
    size_t smem;
    uintptr_t payload, starts, rows;  // in the scratch
};
// The plan for n keys over R values with the n words at out_addr as scratch;
// false when they cannot hold it.
bool part_plan(uint64_t n, uint32_t R, uint32_t head, uint64_t nvec, uintptr_t out_addr, int sms, PartPlan *p);
cudaError_t launch_part(const PartPlan &p, const int32_t *in, uint64_t n, uint32_t head, uint64_t nvec, uint32_t min_u,
                        uint32_t R, uint32_t *H, uint32_t *bucket_start, uint32_t *half, Ctl *ctl, int sms,
                        cudaStream_t s);

// Scan and output after it in one launch.
struct WideOutArgs {
    uint32_t *H;           // R counts, zeroed
    int32_t *out;
    uint32_t n, R, min_u;
    uint32_t buckets, tile_cost, target_items;  // (set by launch_wide_out)
    const uint32_t *starts;  // keys before each bucket
    uint32_t *half;        // keys in the lower half of each bucket, zeroed
    uint32_t *read;        // per half bucket: items that have read its counts (zero between sorts)
    Ctl *ctl;
};
cudaError_t launch_wide_out(const WideOutArgs &a, int sms, cudaStream_t s);

// ---------------------------------------------------------------- scan
struct ScanArgs {
    uint32_t *H;           // histogram, zeroed as it is consumed
    uint64_t *state;       // per scan CTA: the sum of its range, published (zero on entry)
    Ctl *ctl;
    uint32_t *run_end;     // inclusive CDF at each non-empty value (exclusive end of its run)
    int32_t *run_val;      // the key of each non-empty value
    uint32_t *start_run;   // per output CTA: run containing its first position
    uint64_t n;            // keys of the whole array (the counts must add up to it)
    uint64_t fill_chunk;   // positions per output CTA (multiple of 4)
    uint32_t head;         // first output CTA boundary is pos_base + head + fill_chunk
    uint32_t fill_ctas;
    uint32_t pos_base;     // the output CTAs cover positions [pos_base, pos_end) of
    uint32_t pos_end;      // the sorted array (0 and n for a whole sort)
    uint32_t R, T, chunks;
    uint32_t ctas;         // scan CTAs (set by launch_scan)
    int32_t minVal;
    uint32_t *dbg_hist, *dbg_cdf, *dbg_offset;  // optional exports
};
cudaError_t launch_scan(const ScanArgs &a, int sms, cudaStream_t s);

// ---------------------------------------------------------------- output
struct FillArgs {
    int32_t *out;          // out[0] holds position pos_base of the sorted array
    uint64_t n;            // end of the positions written (pos_end)
    uint32_t pos_base;     // first position written (0 for a whole sort)
    uint64_t fill_chunk;
    uint32_t head;
    uint32_t fill_ctas;
    const uint32_t *run_end;
    const int32_t *run_val;
    const uint32_t *start_run;
    Ctl *ctl;
    uint64_t *scan_state;  // reset here for the next call
    uint32_t scan_chunks;
    uint32_t R;            // entries of run_end / run_val
    int32_t none;          // a value no key of the array has (minVal - 1)
};
cudaError_t launch_fill(const FillArgs &a, int threads, bool short_runs, cudaStream_t s);

}  // namespace rtcdf
