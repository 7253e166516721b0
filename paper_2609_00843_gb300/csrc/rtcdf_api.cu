// Host side of the C ABI (include/rtcdf.h): argument checks, launch planning,
// workspace management and the pipeline of Algorithm 4.
//
//   1. histogram -- Algorithm 5: one shared-memory tile or several (hist.cu), packed
//                   counters for ranges of a few tiles (pack.cu), by partition for
//                   wider ones (part.cu)
//   2. scan      -- local CDFs + tile offsets (Algorithm 6) as one scan (scan.cu)
//   3. output    -- Algorithm 7 for all tiles in one launch (fill.cu)
//
// 2 and 3 are one launch over narrow ranges (small.cu) and over wide ones with few
// keys a value (wide_out.cu), and a small array takes one launch in all (small.cu).
//
// Unlike the paper's host driver there is no device-to-host copy of the tile
// offsets and no per-tile launch loop: every launch size is known from (n, R)
// alone, so a sort is one to five stream-ordered launches with no host
// synchronisation and can be captured in a CUDA graph.
#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <utility>

#include "../../include/rtcdf.h"
#include "rtcdf_internal.h"

using namespace rtcdf;

namespace {

struct DeviceInfo {
    int sms = 0;
    size_t smem_optin = 0;
};

std::mutex g_mu;
std::map<int, DeviceInfo> g_dev;

rtcdf_status device_info(DeviceInfo *out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return RTCDF_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_dev.find(dev);
    if (it == g_dev.end()) {
        DeviceInfo d;
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return RTCDF_ERR_CUDA;
        d.sms = v;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
            return RTCDF_ERR_CUDA;
        d.smem_optin = (size_t)v;
        try {
            it = g_dev.emplace(dev, d).first;
        } catch (...) {
            return RTCDF_ERR_NO_MEMORY;
        }
    }
    *out = it->second;
    return RTCDF_OK;
}

struct Plan {
    uint32_t R, T, m, g;
    int hist_threads;
    size_t hist_smem;
    bool streaming;
    bool hist_long;     // one tile of a long input (hist_long_kernel)
    bool shape_given;   // the histogram's shape comes from the caller or the tuning table
    bool given;         // parameters of the caller or of an entry in the caller's tuning table
    int sms;
    uint32_t head;
    uint64_t nvec;
    int fill_threads;
    uint32_t fill_ctas;
    uint64_t fill_chunk;
};

rtcdf_status check_range(int64_t minVal, int64_t maxVal, uint32_t *R) {
    if (minVal < INT32_MIN || maxVal > (int64_t)1 << 31) return RTCDF_ERR_RANGE;
    if (maxVal <= minVal) return RTCDF_ERR_RANGE;
    int64_t r = maxVal - minVal;
    if (r > RTCDF_MAX_R) return RTCDF_ERR_RANGE;
    *R = (uint32_t)r;
    return RTCDF_OK;
}

// Few keys per value: the output kernel's form for short runs.  (R = 2^19, n =
// 1e8, 190 keys per value: 65.5 against 71.7 us; 381 keys: 73.7 against 63.5.)
bool short_runs(uint64_t n, uint32_t R) { return n < 256ull * R; }

constexpr uint64_t kHistLongMinN = 200000000;  // (see hist_long_kernel)

// Choose the launch shape (Section 3.3): tile width T from shared memory, CTAs
// per tile from occupancy, output CTAs from n.
rtcdf_status make_plan_with(uint64_t n, uint32_t R, uintptr_t in_addr, uintptr_t out_addr,
                            const rtcdf_params *p, bool alone, Plan *pl) {
    DeviceInfo dev;
    rtcdf_status st = device_info(&dev);
    if (st) return st;
    rtcdf_params q;
    memset(&q, 0, sizeof(q));
    if (p) q = *p;

    pl->R = R;
    pl->sms = dev.sms;
    pl->shape_given = q.tile_width > 0 || q.hist_ctas_per_tile > 0 || q.hist_threads > 0;
    pl->hist_threads = q.hist_threads ? q.hist_threads : 1024;
    if (pl->hist_threads != 256 && pl->hist_threads != 512 && pl->hist_threads != 1024)
        return RTCDF_ERR_INVALID_ARG;
    // Largest tile whose 32-bit histogram fits the opt-in shared memory.
    const uint32_t t_max = (uint32_t)(dev.smem_optin / 4) & ~1023u;
    uint32_t T = q.tile_width > 0 ? (uint32_t)q.tile_width : 0;
    if (T == 0) {
        // Fewest tiles that fit, then equal widths (rounded up to 1024 values):
        // every tile costs a full input scan, and balanced tiles leave more
        // shared memory per SM for L1.
        const uint32_t m = (R + t_max - 1) / t_max;
        T = m == 1 ? R : std::min(t_max, ((R + m - 1) / m + 1023) & ~1023u);
        // Small arrays just past one tile: four, whose clearing and merging is less
        // than the keys' extra passes (n = 1e5, R = 60000 16.5 us against 18.5).
        const bool small = rtcdf_tune_n_class(n) == RTCDF_TUNE_N_SMALL;
        if (m == 2 && R <= 65536 && small) T = 16384;
        // A histogram alone: so too where a tile would hold the range, since its clearing
        // overlaps no earlier launch (n = 1e4 ... 1e6, R = 30000 6.2 us against 8.2, 50000 8.2
        // against 10.3).
        if (m == 1 && R > 16384 && small && alone) T = R > 32768 ? 16384 : 11264;
    }
    if (T > t_max) return RTCDF_ERR_INVALID_ARG;
    if (T > R) T = R;
    pl->T = T;
    pl->m = (R + T - 1) / T;
    pl->streaming = (pl->m == 1);
    // Several tiles: one more word after the tile (out-of-tile keys counted
    // into it, kept to 16 bytes).
    pl->hist_smem = (size_t)T * 4 + (pl->streaming ? 0 : 16);

    // Input split: unaligned head elements, 16-byte vectors, ragged tail.
    uint32_t head_in = (uint32_t)(((16 - (in_addr & 15)) & 15) / 4);
    if (head_in > n) head_in = (uint32_t)n;
    pl->head = head_in;
    pl->nvec = (n - head_in) / 4;

    int occ = 0;
    try {  // the occupancy cache may need memory for a new entry
        if (hist_max_ctas_per_sm(pl->hist_threads, pl->hist_smem, pl->streaming, &occ) != cudaSuccess)
            return RTCDF_ERR_CUDA;
    } catch (...) {
        return RTCDF_ERR_NO_MEMORY;
    }
    if (occ < 1) return RTCDF_ERR_INVALID_ARG;
    // g_hist = min(max(1, floor(a_hist * S / m)), ceil(n / (16 * threads)))
    uint64_t g = std::max<uint64_t>(1, (uint64_t)occ * dev.sms / pl->m);
    uint64_t g_n = std::max<uint64_t>(1, (n + 16ull * pl->hist_threads - 1) / (16ull * pl->hist_threads));
    g = std::min(g, g_n);
    pl->hist_long = pl->streaming && !pl->shape_given && n >= kHistLongMinN;
    if (pl->hist_long) g = dev.sms;
    if (q.hist_ctas_per_tile > 0) g = (uint64_t)q.hist_ctas_per_tile;
    pl->g = (uint32_t)g;

    // Output: contiguous position ranges, CTA boundaries on 16-byte vectors of `out`.
    // Not clamped to n: positions below head_out are written one by one, and
    // the vector frame must stay 16-byte aligned.
    const uint32_t head_out = (uint32_t)(((16 - (out_addr & 15)) & 15) / 4);
    pl->given = p != nullptr;
    const bool short_fill = short_runs(n, R) && !q.fill_threads && !q.fill_ctas && !q.fill_chunk;
    pl->fill_threads = q.fill_threads ? q.fill_threads : short_fill ? 256 : 512;
    if (pl->fill_threads != 256 && pl->fill_threads != 512 && pl->fill_threads != 1024)
        return RTCDF_ERR_INVALID_ARG;
    // Many more CTAs than fit at once (about 32K positions each, at least four
    // waves' worth): the block scheduler then balances CTAs whose positions
    // cross many short runs against CTAs inside one long run.  Where all runs
    // are short (few keys per value) small CTAs with 4096 positions, or as few
    // as kMaxFillCtas allows, are best (R = 2^20 normal, output kernel, us, for
    // 256 threads with 4K / 8K / 16K / 32K positions and 512 threads with 4K /
    // 16K: n = 1e7 16 / 23 / 35 / 55 and 27 / 23; 3e6 14 / 21 / 35 / 55 and 12 / 21).
    uint64_t body = n > head_out ? n - head_out : 0;
    uint64_t chunk;
    if (q.fill_chunk < 0 || q.fill_ctas < 0) return RTCDF_ERR_INVALID_ARG;
    if (q.fill_chunk > 0) {
        chunk = std::max<uint64_t>((uint64_t)q.fill_chunk,
                                   (body + kMaxFillCtas - 1) / kMaxFillCtas);
        chunk = std::max<uint64_t>(chunk, 4 * (uint64_t)pl->fill_threads);
    } else if (short_fill) {
        // (fewer than 4096 when that makes less than four CTAs per SM)
        chunk = std::min<uint64_t>(4096, std::max<uint64_t>(1024, body / (4 * (uint64_t)dev.sms)));
        chunk = std::max<uint64_t>(chunk, (body + kMaxFillCtas - 1) / kMaxFillCtas);
    } else {
        uint64_t want = q.fill_ctas > 0 ? (uint64_t)q.fill_ctas
                                        : std::max<uint64_t>((uint64_t)dev.sms * 4, body / 32768);
        want = std::min<uint64_t>(want, kMaxFillCtas);
        chunk = std::max<uint64_t>(4 * (uint64_t)pl->fill_threads, (body + want - 1) / want);
    }
    chunk = (chunk + 3) / 4 * 4;
    pl->fill_chunk = chunk;
    pl->fill_ctas = (uint32_t)(1 + (n > head_out ? (n - head_out - 1) / chunk : 0));
    if (pl->fill_ctas > kMaxFillCtas) return RTCDF_ERR_INVALID_ARG;
    pl->head = head_in;
    return RTCDF_OK;
}

// Explicit parameters are used as given; without them the tuning table is
// tried first and the built-in rules cover what it lacks (or what does not fit
// this device).
// alone: for a histogram that no sort follows at once.
rtcdf_status make_plan(uint64_t n, uint32_t R, uintptr_t in_addr, uintptr_t out_addr,
                       const rtcdf_params *p, Plan *pl, bool alone = false) {
    if (p) return make_plan_with(n, R, in_addr, out_addr, p, alone, pl);
    rtcdf_params t;
    bool builtin = false;
    const bool found = tune_lookup(n, R, &t, &builtin);
    // (the compiled-in table's output shapes are those of the kernel's form for long runs)
    if (found && builtin && short_runs(n, R)) t.fill_ctas = t.fill_threads = t.fill_chunk = 0;
    if (!(found && make_plan_with(n, R, in_addr, out_addr, &t, alone, pl) == RTCDF_OK))
        return make_plan_with(n, R, in_addr, out_addr, nullptr, alone, pl);
    pl->given = !builtin;
    return RTCDF_OK;
}

bool overlaps(const void *a, const void *b, uint64_t n) {
    uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    uint64_t bytes = n * 4;
    return x < y + bytes && y < x + bytes;
}

rtcdf_status check_args(const int32_t *in, int32_t *out, uint64_t n) {
    if (n >= (1ull << 32)) return RTCDF_ERR_INVALID_ARG;
    if (!in || !out) return RTCDF_ERR_INVALID_ARG;
    if (((uintptr_t)in & 3) || ((uintptr_t)out & 3)) return RTCDF_ERR_INVALID_ARG;
    if ((const void *)in != (const void *)out && overlaps(in, out, n)) return RTCDF_ERR_INVALID_ARG;
    return RTCDF_OK;
}

// The arguments of rtcdf_sort_ex (nothing beyond the range for an empty array).
rtcdf_status check_sort_ex(const int32_t *in, int32_t *out, uint64_t n, int64_t minVal, int64_t maxVal,
                           const void *workspace, size_t ws_bytes, uint32_t *R) {
    rtcdf_status st = check_range(minVal, maxVal, R);
    if (st || n == 0) return st;
    st = check_args(in, out, n);
    if (st) return st;
    if (!workspace || ((uintptr_t)workspace & 255)) return RTCDF_ERR_INVALID_ARG;
    return ws_bytes < ws_required(*R) ? RTCDF_ERR_NO_MEMORY : RTCDF_OK;
}

constexpr uint32_t kWideOutMinR = 1000000;  // (use_wide_out)

// Histogram by packed counters (pack.cu) or by range tiles (hist.cu): one pass
// over the input against one per tile, and about 10 us more (the sample and a
// second launch; without scratch, the counters added to H by pairs of CTAs: packed
// / tiles, us, n = 2e7, R = 200000, four tiles 46 / 48, 1.5e7 over 2^18, five, 46 /
// 44, 4e7 over 100000, two, 50 / 58, 3.5e7 over 150000, three, 50 / 62).
bool use_pack(uint64_t n, const Plan &pl, uintptr_t scratch, PackPlan *pp) {
    if (pl.shape_given || pl.R <= 49152 || n * pl.m < (scratch ? 70000000u : 80000000u)) return false;
    return pack_plan(n, pl.R, pl.nvec, scratch, pl.sms, pp);
}

// Histogram by partition (part.cu) or by range tiles (hist.cu).  Partition
// takes about 9 us more (two launches) and reads the input once where the
// tiles read it m times, so it needs several tiles and enough keys; fewer where
// wide_out.cu follows, whose launch takes the place of two that grow with R.  Whole
// sorts one after another, us, partition / tiles, uniform, normal, one value: R = 2^22, n =
// 3000 27 27 25 / 32 32 27, n = 3e5 33 32 29 / 45 47 34; R = 2^21, n = 1e6 35 33 31 / 46 49 33, n
// = 1e5 29 27 27 / 31 32 24; R = 1e6, n = 3e6 43 43 31 / 51 55 39, n = 1e6 35 34 29 / 35 36 26.
bool use_part(uint64_t n, const Plan &pl, uintptr_t scratch, PartPlan *pp) {
    const uint64_t keys = pl.R >= 1u << 22 ? 0 : pl.R >= kWideOutMinR ? 20000000 : 40000000;
    if (!scratch || pl.shape_given || pl.m <= 5 || n * (pl.m - 5) < keys) return false;
    return part_plan(n, pl.R, pl.head, pl.nvec, scratch, pl.sms, pp);
}

// Inputs that packed counters cannot hold (frequent keys, sorted ones) are counted by range
// tiles: over long inputs by a launch of their own, with the widest tiles, which finds
// nothing to do otherwise.  In pack_kernel's launch a tile is no wider than the packed
// counters, so that more passes are needed: whole sorts, us, there / own launch / range
// tiles from the start, n = 3e8, R = 200000 log-uniform keys 895 / 834 / 820, 100 different
// keys 762 / 648 / 641, sorted 647 / 633 / 630; but n = 1e8, R = 2^18 359 / 344 / 336, 286 / 274
// / 264 and 259 / 267 / 260, R = 350000 multiples of 1024 499 / 583 / 625.  The launch costs
// the others 0.7 us at n = 1e8 (uniform, 160.2 / 160.9), 3 us at 2e7 (69.9 / 73.0) and at n =
// 1e9, R = 2^16 (1139 / 1142), whose tiles are two either way.
constexpr uint64_t kPackTilesLaunchMin = 1000000000;

// Algorithm 5 (all tiles) into H (R counters).  H accumulates, so several calls
// over slices of one array add up to the array's histogram.  ctl and scratch (n
// words, 0 if there are none): of a whole sort, as bucket_start and half (or null)
// of a histogram by partition, which *parted says was made.
rtcdf_status hist_phase(const int32_t *in, uint64_t n, int64_t minVal, uint32_t R, const Plan &pl, uint32_t *H,
                        Ctl *ctl, uintptr_t scratch, uint32_t *bucket_start, uint32_t *half, bool *parted,
                        cudaStream_t s) {
    HistArgs h;
    h.in = in; h.n = n; h.nvec = pl.nvec; h.head = pl.head;
    h.min_u = (uint32_t)(int32_t)minVal; h.R = R; h.T = pl.T; h.m = pl.m; h.g = pl.g;
    h.H = H; h.long_form = pl.hist_long;
    PackPlan pack;
    PartPlan part;
    cudaError_t e;
    if (use_pack(n, pl, scratch, &pack)) {
        const bool tiles_later = ctl && pack.m > pl.m && n * pl.m >= kPackTilesLaunchMin;
        e = launch_pack(pack, h, ctl, tiles_later, s);
        if (tiles_later && e == cudaSuccess) {
            h.only_if = &ctl->pack_tiles;
            e = launch_hist(h, pl.hist_threads, pl.hist_smem, pl.streaming, kHistDependent, s);
        }
    } else if (ctl && (*parted = use_part(n, pl, scratch, &part)))
        e = launch_part(part, in, n, pl.head, pl.nvec, h.min_u, R, H, bucket_start, half, ctl, pl.sms, s);
    else
        e = launch_hist(h, pl.hist_threads, pl.hist_smem, pl.streaming, ctl ? kHistFirst : kHistAlone, s);
    return e == cudaSuccess ? RTCDF_OK : RTCDF_ERR_CUDA;
}

// After a histogram by partition: scan and output in one launch (wide_out.cu)
// where the run table's way through memory is a large part of both, at few keys a
// value, and there are enough tiles.  Whole sorts replayed from a graph, us, one
// launch / two, uniform, normal and one value: n = 1e8, R = 2^24 423 412 306 / 506 482
// 333; n = 1e6 81 79 43 / 111 109 73; n = 2e7, R = 2^20 90 96 73 / 102 106 76; n = 1.2e7
// 67 70 55 / 72 75 55; beyond the lines, n = 5e7, R = 2^21 184 196 144 / 187 195 140;
// n = 1e8, R = 2^20 302 331 248 / 287 307 236; n = 6e6, R = 7e5 47 51 40 / 50 56 38.
bool use_wide_out(uint64_t n, uint32_t R) { return R >= kWideOutMinR && n <= 20ull * R; }

// Most positions that scan and output in one launch serve (small.cu).  Whole
// sorts replayed from a graph, us, one launch / two, uniform keys over R = 128 and
// 16384: n = 1e6 6.4 / 7.9 and 11.9 / 15.3, 1e7 17.5 / 17.9 and 24.5 / 25.9, 3e7
// 45.1 / 46.3 and 50.8 / 53.4, 6e7 85.1 / 84.8 and 89.2 / 91.0, 1e8 140 / 137 and
// 143 / 140: one CTA per SM stores a little slower than the output kernel's many.
constexpr uint64_t kFinishMaxN = 40000000;

// Local CDFs + offsets (Algorithm 6) and output generation (Algorithm 7)
// for an n-key array whose histogram is in H: positions [pos_base, pos_end)
// of the sorted array are written, position p to out[p - pos_base] (the
// plan's output CTAs are sized for pos_end - pos_base positions).
rtcdf_status finish_phase(int32_t *out, uint64_t n, int64_t minVal, uint32_t R, const Plan &pl,
                          const WsLayout &L, char *base, const rtcdf_debug *dbg,
                          cudaEvent_t ev_scan, cudaEvent_t ev_fill, cudaStream_t s,
                          uint64_t pos_base, uint64_t pos_end) {
    Ctl *ctl = (Ctl *)(base + L.ctl);
    uint64_t *state = (uint64_t *)(base + L.scan_state);
    uint32_t *run_end = (uint32_t *)(base + L.run_end);
    int32_t *run_val = (int32_t *)(base + L.run_val);
    uint32_t *start_run = (uint32_t *)(base + L.start_run);
    // Positions before the first whole vector: all of them in a window without one,
    // since pos_base + head must not pass 2^32 (with no vector to store, the frame's
    // alignment does not matter).
    const uint32_t head_out =
        (uint32_t)std::min<uint64_t>(((16 - ((uintptr_t)out & 15)) & 15) / 4, pos_end - pos_base);
    if (!dbg && !pl.given && R <= kSmallMaxR && pos_end - pos_base <= kFinishMaxN) {
        FinishArgs f;
        f.H = (uint32_t *)(base + L.hist); f.out = out; f.n = (uint32_t)n;
        f.pos_base = (uint32_t)pos_base; f.pos_end = (uint32_t)pos_end;
        f.R = R; f.min_u = (uint32_t)(int32_t)minVal; f.ctl = ctl;
        return launch_finish(f, pl.sms, s) == cudaSuccess ? RTCDF_OK : RTCDF_ERR_CUDA;
    }
    ScanArgs sc;
    sc.H = (uint32_t *)(base + L.hist); sc.state = state; sc.ctl = ctl; sc.run_end = run_end;
    sc.run_val = run_val; sc.start_run = start_run; sc.n = n; sc.fill_chunk = pl.fill_chunk;
    sc.head = head_out; sc.fill_ctas = pl.fill_ctas; sc.R = R; sc.T = pl.T; sc.chunks = L.scan_chunks;
    sc.pos_base = (uint32_t)pos_base; sc.pos_end = (uint32_t)pos_end;
    sc.minVal = (int32_t)minVal;
    sc.dbg_hist = dbg ? dbg->tile_hist : nullptr;
    sc.dbg_cdf = dbg ? dbg->cdf : nullptr;
    sc.dbg_offset = dbg ? dbg->tile_offset : nullptr;
    if (launch_scan(sc, pl.sms, s) != cudaSuccess) return RTCDF_ERR_CUDA;
    if (ev_scan && cudaEventRecord(ev_scan, s) != cudaSuccess) return RTCDF_ERR_CUDA;

    FillArgs f;
    f.out = out; f.n = pos_end; f.pos_base = (uint32_t)pos_base; f.fill_chunk = pl.fill_chunk;
    f.head = head_out;
    f.fill_ctas = pl.fill_ctas; f.run_end = run_end; f.run_val = run_val;
    f.start_run = start_run; f.ctl = ctl; f.scan_state = state; f.scan_chunks = L.scan_chunks;
    f.R = R; f.none = (int32_t)((uint32_t)minVal - 1u);
    if (launch_fill(f, pl.fill_threads, short_runs(n, R), s) != cudaSuccess) return RTCDF_ERR_CUDA;
    if (ev_fill && cudaEventRecord(ev_fill, s) != cudaSuccess) return RTCDF_ERR_CUDA;
    return RTCDF_OK;
}

rtcdf_status run_pipeline(const int32_t *in, int32_t *out, uint64_t n, int64_t minVal,
                          uint32_t R, const Plan &pl, void *ws, size_t ws_bytes,
                          const rtcdf_debug *dbg, cudaStream_t s) {
    const WsLayout L = ws_layout(R, ws_bytes);
    char *base = (char *)ws;
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
    if (dbg)
        for (int i = 0; i < 4; i++) ev[i] = (cudaEvent_t)dbg->stage_events[i];
    if (ev[0] && cudaEventRecord(ev[0], s) != cudaSuccess) return RTCDF_ERR_CUDA;
    // (a sort in place has no scratch)
    bool parted = false;
    const bool wide = !dbg && !pl.given && use_wide_out(n, R);
    uint32_t *half = (uint32_t *)(base + L.scan_state) + 2 * kPartMaxBuckets;
    rtcdf_status st = hist_phase(in, n, minVal, R, pl, (uint32_t *)(base + L.hist), (Ctl *)(base + L.ctl),
                                 in == out ? 0 : (uintptr_t)out, (uint32_t *)(base + L.start_run),
                                 wide ? half : nullptr, &parted, s);
    if (st) return st;
    if (parted && wide) {
        WideOutArgs w;
        w.H = (uint32_t *)(base + L.hist); w.out = out; w.n = (uint32_t)n; w.R = R;
        w.min_u = (uint32_t)(int32_t)minVal; w.starts = (uint32_t *)(base + L.start_run);
        w.half = half; w.read = (uint32_t *)(base + L.scan_state); w.ctl = (Ctl *)(base + L.ctl);
        return launch_wide_out(w, pl.sms, s) == cudaSuccess ? RTCDF_OK : RTCDF_ERR_CUDA;
    }
    if (ev[1] && cudaEventRecord(ev[1], s) != cudaSuccess) return RTCDF_ERR_CUDA;
    return finish_phase(out, n, minVal, R, pl, L, base, dbg, ev[2], ev[3], s, 0, n);
}

// One sort with checked arguments in a workspace of at least ws_required(R) bytes.
// rules: by the built-in rules whatever the tuning table holds (params is null).
rtcdf_status sort_checked(const int32_t *in, int32_t *out, uint64_t n, int64_t minVal, uint32_t R,
                          const rtcdf_params *params, void *ws, size_t ws_bytes, const rtcdf_debug *dbg,
                          cudaStream_t s, bool rules = false) {
    // Small arrays in one launch (small.cu), unless the caller asks for launch
    // parameters, intermediates or stage events.  (The compiled-in table has no say in
    // them: no plan is made to find that out.)
    const bool small = n <= kSmallMaxN && R <= kSmallMaxR && !params && !dbg;
    Plan pl;
    if (!(small && (rules || tune_is_builtin()))) {
        const rtcdf_status st = rules ? make_plan_with(n, R, (uintptr_t)in, (uintptr_t)out, nullptr, false, &pl)
                                      : make_plan(n, R, (uintptr_t)in, (uintptr_t)out, params, &pl);
        if (st) return st;
        if (!small || pl.given) return run_pipeline(in, out, n, minVal, R, pl, ws, ws_bytes, dbg, s);
    }
    return launch_small(in, out, (uint32_t)n, (uint32_t)(int32_t)minVal, R, (Ctl *)ws, s) == cudaSuccess
               ? RTCDF_OK
               : RTCDF_ERR_CUDA;
}

// ---------------------------------------------------------------- workspace cache
struct CachedWs {
    void *ptr = nullptr;
    size_t bytes = 0;
};
std::map<std::pair<int, cudaStream_t>, CachedWs> g_ws;

rtcdf_status cached_workspace(cudaStream_t s, size_t need, void **ptr, size_t *bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return RTCDF_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_mu);
    CachedWs *wp = nullptr;
    try {
        wp = &g_ws[std::make_pair(dev, s)];
    } catch (...) {
        return RTCDF_ERR_NO_MEMORY;
    }
    CachedWs &w = *wp;
    if (w.bytes < need) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) return RTCDF_ERR_CUDA;
        if (cap != cudaStreamCaptureStatusNone) return RTCDF_ERR_NO_MEMORY;
        size_t grow = std::max(need, w.bytes * 2);
        void *p = nullptr;
        if (cudaMallocAsync(&p, grow, s) != cudaSuccess) return RTCDF_ERR_NO_MEMORY;
        if (cudaMemsetAsync(p, 0, grow, s) != cudaSuccess) {
            cudaFreeAsync(p, s);
            return RTCDF_ERR_CUDA;
        }
        void *old = w.ptr;
        w.ptr = p;
        w.bytes = grow;
        if (old && cudaFreeAsync(old, s) != cudaSuccess) return RTCDF_ERR_CUDA;
    }
    *ptr = w.ptr;
    *bytes = w.bytes;
    return RTCDF_OK;
}

// The status code for a status word: a wait that ran out makes every other
// finding unreliable, so it comes first.
rtcdf_status status_of_bits(uint32_t v) {
    if (v & kDevTimeout) return RTCDF_ERR_TIMEOUT;
    if (v & kDevBadSegment) return RTCDF_ERR_INVALID_ARG;
    if (v & kDevKeyOutOfRange) return RTCDF_ERR_KEY_OUT_OF_RANGE;
    return RTCDF_OK;
}

rtcdf_status read_status(void *ws, cudaStream_t s, int32_t *out) {
    uint32_t v = 0;
    Ctl *ctl = (Ctl *)ws;
    if (cudaMemcpyAsync(&v, &ctl->status, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess) return RTCDF_ERR_CUDA;
    if (cudaMemsetAsync(&ctl->status, 0, 4, s) != cudaSuccess) return RTCDF_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return RTCDF_ERR_CUDA;
    if (out) *out = (int32_t)v;
    return status_of_bits(v);
}

}  // namespace

namespace rtcdf {

// Sort in a workspace whose previous contents are unknown: the regions that
// must start at zero (control block, the scan's sums, histogram) are cleared
// on `s` first.  Used by rtcdf_sort_static.
rtcdf_status sort_with_workspace(const int32_t *in, int32_t *out, uint64_t n, int64_t minVal,
                                 int64_t maxVal, void *ws, size_t ws_bytes, cudaStream_t s) {
    uint32_t R = 0;
    rtcdf_status st = check_range(minVal, maxVal, &R);
    if (st) return st;
    if (n == 0) return RTCDF_OK;
    st = check_args(in, out, n);
    if (st) return st;
    if (!ws || ws_bytes < ws_required(R)) return RTCDF_ERR_NO_MEMORY;
    const WsLayout L = ws_layout(R, ws_bytes);
    if (cudaMemsetAsync(ws, 0, L.zero_bytes, s) != cudaSuccess) return RTCDF_ERR_CUDA;
    return sort_checked(in, out, n, minVal, R, nullptr, ws, ws_bytes, nullptr, s);
}

// A sort with checked arguments by the built-in rules, for rtcdf_autotune.
rtcdf_status sort_by_rules(const int32_t *in, int32_t *out, uint64_t n, int64_t minVal, int64_t maxVal, void *ws,
                           size_t ws_bytes, cudaStream_t s) {
    uint32_t R = 0;
    const rtcdf_status st = check_sort_ex(in, out, n, minVal, maxVal, ws, ws_bytes, &R);
    if (st || n == 0) return st;
    return sort_checked(in, out, n, minVal, R, nullptr, ws, ws_bytes, nullptr, s, true);
}

// The two halves of a sort, for rtcdf_sort_host: histogram of a slice (may be
// called once per uploaded chunk), then scan + output for the whole array.
rtcdf_status host_pipeline_hist(const int32_t *in, uint64_t n, int64_t minVal, uint32_t R, void *ws,
                                size_t ws_bytes, cudaStream_t s) {
    if (n == 0) return RTCDF_OK;
    Plan pl;
    rtcdf_status st = make_plan(n, R, (uintptr_t)in, 0, nullptr, &pl, true);
    if (st) return st;
    return hist_phase(in, n, minVal, R, pl, (uint32_t *)((char *)ws + ws_layout(R, ws_bytes).hist), nullptr, 0, nullptr,
                      nullptr, nullptr, s);
}

rtcdf_status host_pipeline_finish(int32_t *out, uint64_t n, int64_t minVal, uint32_t R, void *ws,
                                  size_t ws_bytes, cudaStream_t s) {
    Plan pl;
    rtcdf_status st = make_plan(n, R, 0, (uintptr_t)out, nullptr, &pl);
    if (st) return st;
    return finish_phase(out, n, minVal, R, pl, ws_layout(R, ws_bytes), (char *)ws, nullptr,
                        nullptr, nullptr, s, 0, n);
}

}  // namespace rtcdf

extern "C" {

const char *rtcdf_version(void) { return "rtcdf 0.1 (sm_103a)"; }

const char *rtcdf_status_str(rtcdf_status s) {
    switch (s) {
        case RTCDF_OK: return "ok";
        case RTCDF_ERR_INVALID_ARG: return "invalid argument";
        case RTCDF_ERR_RANGE: return "range size outside [1, RTCDF_MAX_R] or outside int32";
        case RTCDF_ERR_KEY_OUT_OF_RANGE: return "a key lies outside [minVal, maxVal)";
        case RTCDF_ERR_CUDA: return "CUDA runtime error";
        case RTCDF_ERR_NO_MEMORY: return "workspace allocation failed or workspace too small";
        case RTCDF_ERR_TIMEOUT: return "a bounded device wait gave up";
    }
    return "unknown status";
}

rtcdf_status rtcdf_workspace_size(int64_t R, size_t *bytes) {
    if (!bytes) return RTCDF_ERR_INVALID_ARG;
    if (R <= 0 || R > RTCDF_MAX_R) return RTCDF_ERR_RANGE;
    *bytes = ws_required((uint64_t)R);
    return RTCDF_OK;
}

rtcdf_status rtcdf_plan(uint64_t n, int64_t R, rtcdf_params *params) {
    if (!params) return RTCDF_ERR_INVALID_ARG;
    if (R <= 0 || R > RTCDF_MAX_R) return RTCDF_ERR_RANGE;
    Plan pl;
    rtcdf_status st = make_plan(n, (uint32_t)R, 0, 0, nullptr, &pl);
    if (st) return st;
    memset(params, 0, sizeof(*params));
    params->tile_width = (int32_t)pl.T;
    params->hist_ctas_per_tile = (int32_t)pl.g;
    params->hist_threads = pl.hist_threads;
    params->fill_ctas = (int32_t)pl.fill_ctas;
    params->fill_threads = pl.fill_threads;
    params->fill_chunk = (int32_t)std::min<uint64_t>(pl.fill_chunk, INT32_MAX);
    return RTCDF_OK;
}

rtcdf_status rtcdf_sort_ex(const int32_t *in, int32_t *out, uint64_t n, int64_t minVal,
                           int64_t maxVal, const rtcdf_params *params, void *workspace,
                           size_t ws_bytes, const rtcdf_debug *debug, rtcdf_stream_t stream) {
    uint32_t R = 0;
    const rtcdf_status st = check_sort_ex(in, out, n, minVal, maxVal, workspace, ws_bytes, &R);
    if (st || n == 0) return st;
    return sort_checked(in, out, n, minVal, R, params, workspace, ws_bytes, debug, (cudaStream_t)stream);
}

rtcdf_status rtcdf_sort_ws(const int32_t *in, int32_t *out, uint64_t n, int64_t minVal,
                           int64_t maxVal, void *workspace, size_t ws_bytes,
                           rtcdf_stream_t stream) {
    return rtcdf_sort_ex(in, out, n, minVal, maxVal, nullptr, workspace, ws_bytes, nullptr, stream);
}

rtcdf_status rtcdf_reserve(int64_t max_R, rtcdf_stream_t stream) {
    if (max_R <= 0 || max_R > RTCDF_MAX_R) return RTCDF_ERR_RANGE;
    void *ws = nullptr;
    size_t bytes = 0;
    return cached_workspace((cudaStream_t)stream, ws_required((uint64_t)max_R), &ws, &bytes);
}

rtcdf_status rtcdf_sort(const int32_t *in, int32_t *out, uint64_t n, int64_t minVal,
                        int64_t maxVal, rtcdf_stream_t stream) {
    uint32_t R = 0;
    rtcdf_status st = check_range(minVal, maxVal, &R);
    if (st) return st;
    if (n == 0) return RTCDF_OK;
    st = check_args(in, out, n);
    if (st) return st;
    void *ws = nullptr;
    size_t ws_bytes = 0;
    st = cached_workspace((cudaStream_t)stream, ws_required(R), &ws, &ws_bytes);
    if (st) return st;
    return sort_checked(in, out, n, minVal, R, nullptr, ws, ws_bytes, nullptr, (cudaStream_t)stream);
}

rtcdf_status rtcdf_hist_accumulate(const int32_t *in, uint64_t n, int64_t minVal, int64_t maxVal,
                                   uint32_t *counts, rtcdf_stream_t stream) {
    uint32_t R = 0;
    rtcdf_status st = check_range(minVal, maxVal, &R);
    if (st) return st;
    if (!counts || ((uintptr_t)counts & 3)) return RTCDF_ERR_INVALID_ARG;
    if (n == 0) return RTCDF_OK;
    if (n >= (1ull << 32) || !in || ((uintptr_t)in & 3)) return RTCDF_ERR_INVALID_ARG;
    {
        const uintptr_t x = (uintptr_t)in, y = (uintptr_t)counts;
        if (x < y + (uint64_t)R * 4 && y < x + n * 4) return RTCDF_ERR_INVALID_ARG;
    }
    Plan pl;
    st = make_plan(n, R, (uintptr_t)in, 0, nullptr, &pl, true);
    if (st) return st;
    // Algorithm 5 for every tile, added straight into the caller's counts.
    return hist_phase(in, n, minVal, R, pl, counts, nullptr, 0, nullptr, nullptr, nullptr, (cudaStream_t)stream);
}

rtcdf_status rtcdf_fill_from_counts(const uint32_t *counts, uint64_t total_n, int64_t minVal,
                                    int64_t maxVal, uint64_t pos_begin, uint64_t pos_end, int32_t *out,
                                    void *workspace, size_t ws_bytes, rtcdf_stream_t stream) {
    uint32_t R = 0;
    rtcdf_status st = check_range(minVal, maxVal, &R);
    if (st) return st;
    if (total_n >= (1ull << 32) || pos_begin > pos_end || pos_end > total_n) return RTCDF_ERR_INVALID_ARG;
    if (!counts || ((uintptr_t)counts & 3)) return RTCDF_ERR_INVALID_ARG;
    if (pos_end == pos_begin) return RTCDF_OK;
    if (!out || ((uintptr_t)out & 3)) return RTCDF_ERR_INVALID_ARG;
    if (!workspace || ((uintptr_t)workspace & 255)) return RTCDF_ERR_INVALID_ARG;
    if (ws_bytes < ws_required(R)) return RTCDF_ERR_NO_MEMORY;
    const uint64_t len = pos_end - pos_begin;
    {
        const uintptr_t x = (uintptr_t)out, y = (uintptr_t)counts, w = (uintptr_t)workspace;
        if (x < y + (uint64_t)R * 4 && y < x + len * 4) return RTCDF_ERR_INVALID_ARG;
        if (x < w + ws_bytes && w < x + len * 4) return RTCDF_ERR_INVALID_ARG;
    }
    Plan pl;
    st = make_plan(len, R, 0, (uintptr_t)out, nullptr, &pl);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const WsLayout L = ws_layout(R, ws_bytes);
    // The global counts become the workspace's H (zero between sorts; the scan
    // zeroes it again as it reads it).
    if (cudaMemcpyAsync((char *)workspace + L.hist, counts, (size_t)R * 4, cudaMemcpyDeviceToDevice, s) !=
        cudaSuccess)
        return RTCDF_ERR_CUDA;
    return finish_phase(out, total_n, minVal, R, pl, L, (char *)workspace, nullptr, nullptr, nullptr, s,
                        pos_begin, pos_end);
}

rtcdf_status rtcdf_status_get(rtcdf_stream_t stream, int32_t *device_status) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return RTCDF_ERR_CUDA;
    void *ws = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        auto it = g_ws.find(std::make_pair(dev, (cudaStream_t)stream));
        if (it != g_ws.end()) ws = it->second.ptr;
    }
    // The single-array sorts' workspace and the segmented sorts' one (both
    // start with their status word).
    void *bws = batch_stream_workspace((cudaStream_t)stream);
    int32_t bits = 0, b2 = 0;
    if (ws) {
        const rtcdf_status st = read_status(ws, (cudaStream_t)stream, &bits);
        if (st == RTCDF_ERR_CUDA) return st;
    }
    if (bws) {
        const rtcdf_status st = read_status(bws, (cudaStream_t)stream, &b2);
        if (st == RTCDF_ERR_CUDA) return st;
    }
    if (device_status) *device_status = bits | b2;
    return status_of_bits((uint32_t)(bits | b2));
}

rtcdf_status rtcdf_ws_status_get(void *workspace, rtcdf_stream_t stream, int32_t *device_status) {
    if (!workspace) return RTCDF_ERR_INVALID_ARG;
    return read_status(workspace, (cudaStream_t)stream, device_status);
}

}  // extern "C"
