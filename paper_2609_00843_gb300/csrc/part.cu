// Histogram of a wide range (more values than one shared-memory tile holds) by
// partition: every key is read from HBM once and counted once, where the
// range-tile kernel (hist.cu) reads and examines every key once per tile.
//
//   part_kernel   cuts the input into slabs (32768 keys), partitions each slab
//                 in shared memory by bucket (value >> 15, at most 512 buckets)
//                 and writes the 15-bit positions inside the buckets to scratch,
//                 two bytes a key: the slab's buckets one after another, each
//                 padded to 16 bytes, and a table of their starts.  A slab goes
//                 to its own place whatever its keys are, so there is no count
//                 pass over the input, no global offset and no overflow.
//   bucket_kernel counts one bucket at a time (Algorithm 5 on a tile of 32768
//                 values, 32-bit counters in 128 KB of shared memory): an item
//                 is a bucket and every k-th slab, k from the buckets' sizes,
//                 so that heavy buckets are shared by several CTAs.
//
// The scratch is the sort's own output buffer, which nothing reads before the
// output kernel fills it (2 bytes a key plus padding, of its 4); a sort in
// place has none and keeps the range-tile kernel.
//
// Measured (n = 1e8, uniform / normal / one value, both kernels, us; the range
// tiles before that): R = 2^19 214 / 225 / 167 (459 / 424 / 400), 2^20 218 / 236 / 170
// (771 / 777 / 717), 2^22 282 / 269 / 201 (2394 / 2699 / 2718), 2^24 340 / 333 / 249
// (8144 / 8353 / 9810).
#include <algorithm>

#include "rtcdf_internal.h"

namespace rtcdf {

namespace {

constexpr uint32_t kPartWidth = 1u << kPartShift;  // values per bucket
constexpr int kPartThreads = 1024;
constexpr uint32_t kPartSlabMax = 32768;           // keys per slab: 32 a thread, in registers
constexpr uint32_t kPartSlabMin = 4096;
static_assert(kPartSlabMax % (4 * kPartThreads) == 0, "slabs are whole vectors of the CTA");
static_assert(kPartMaxBuckets <= kPartThreads, "one thread per bucket");
constexpr int kBucketThreads = 1024;
constexpr uint32_t kPartList = 4096;               // slabs listed at once
// A bucket's tile (zeroed, and its counts added to H) costs about as much as
// counting this many keys, and looking up the bucket in a slab as counting 2.
constexpr uint32_t kPartTileKeys = 32768;
static_assert(RTCDF_MAX_R >> kPartShift == kPartMaxBuckets, "buckets of the widest range");

// Counters per bucket, log2: lane l of a warp counts in copy l mod copies.
// With 32 copies (up to 128 buckets) the lanes of a warp never meet in a bank or
// on a word, whatever the keys.  With more buckets the passes over the counters
// cost as much as the conflicts they save (n = 1e8, part_kernel, us, 8 / 16 / 32
// copies: 512 buckets 195 / 194 / 222, 256 187 / 175 / 182, 128 180 / 167 / 162).
__host__ __device__ constexpr int part_log_copies(uint32_t B) { return B <= 128 ? 5 : 4; }

// Words of part_kernel's shared memory before the staged slab (which starts on
// 128 bytes, see stage_slot).
__host__ __device__ inline uint32_t part_head_words(uint32_t B) {
    return (((B + 1) << part_log_copies(B)) + 2 * (B + 1) + 31) / 32 * 32;
}

// 16-byte units of a staged slab: its keys (and up to six outside whole vectors),
// each bucket padded to 8.
__host__ __device__ inline uint32_t part_slab_units(uint32_t B, uint32_t slab_keys) { return (slab_keys + 8 + 8 * B) / 8; }
// Bytes of part_kernel's shared memory.
inline size_t part_smem(uint32_t B, uint32_t slab_keys) {
    return 4 * (size_t)part_head_words(B) + align_up(16 * (size_t)part_slab_units(B, slab_keys), 128);
}

__device__ __forceinline__ uint32_t atom_inc(uint32_t s_addr) {
    uint32_t r;
    asm volatile("atom.shared.add.u32 %0, [%1], 1;" : "=r"(r) : "r"(s_addr));
    return r;
}
__device__ __forceinline__ void sts_u16(uint32_t s_addr, uint32_t v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(s_addr), "h"((unsigned short)v));
}
__device__ __forceinline__ void red_inc(uint32_t s_addr) {
    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(s_addr));
}

// Shared address of the staged key that belongs at address p: each 2048 bytes
// are permuted by a number of their own, in whole words inside 128 bytes,
// because the copies of one bucket often start 2048 bytes apart (a slab of one
// value: all of them), in one bank.  A 16-byte unit stays one, in another
// place and with its words in another order.
__device__ __forceinline__ uint32_t stage_slot(uint32_t p) { return p ^ ((p >> 9) & 0x7cu); }

// The 16 bits kept of a key's position y in the range: its position in the
// bucket, and the bucket's parity.  Pads carry the other parity's next value, so
// that they fall on the word after (even buckets) or before the tile.
__device__ __forceinline__ uint32_t pad_of(uint32_t bucket) { return bucket & 1 ? kPartWidth - 1 : kPartWidth; }

}  // namespace

// One CTA per SM with a slab in registers (32 keys a thread, so the input is read
// once), whose next slab's loads are in flight while the staged one is written
// out.  What bounds it (n = 1e8, R = 2^20, 149 us; the 4 + 2 bytes a key take 88):
// about 18 instructions a key, the shared-memory pipe, 7 wavefronts for 32 keys,
// of which the two-byte stores' bank conflicts are four, and seven barriers a
// slab.  Two CTAs per SM with half the slab each take the same time, but shorter
// runs slow bucket_kernel down (R = 2^24: 139 us against 202; 2^20: 71 against 80);
// the keys read a second time from L2 instead, at four CTAs per SM, took 157 us.
template <int LOGC>
__global__ void __launch_bounds__(kPartThreads, 1) part_kernel(PartArgs a) {
    extern __shared__ __align__(128) uint32_t sm[];
    constexpr uint32_t C = 1u << LOGC;
    constexpr int V = kPartSlabMax / 4 / kPartThreads;  // vectors of a slab per thread
    // Bucket B takes the keys outside the range: they are staged after the
    // others and not written out.  (Those of the last bucket's values that lie
    // past the range count into the part of its tile that is not read.)
    const uint32_t B = a.buckets, E = (B + 1) * C;
    uint32_t *cnt = sm;                  // [bucket][copy]: keys, then the copy's next place in the staged slab
    uint32_t *s_tot = sm + E;            // keys of each bucket
    uint32_t *s_off = s_tot + (B + 1);   // start of each bucket in the staged slab (keys, multiples of 8)
    __shared__ uint32_t s_warp[kPartThreads / 32];
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t cnt_base = (uint32_t)__cvta_generic_to_shared(cnt) + 4u * (lane & (C - 1));
    const uint32_t stage = (uint32_t)__cvta_generic_to_shared(sm + part_head_words(B));
    const uint32_t svec = a.slab_keys / 4;
    // After a wait that ran out nothing is written to the output (nor to its
    // use as scratch) until the status has been read.
    if (a.ctl->status & kDevTimeout) return;

    // The positions in the range of the thread's keys of slab s; the vectors
    // past its end hold keys of bucket B.
    uint32_t k[V][4];
    uint32_t nv = 0;
    auto load = [&](uint32_t s) {
        const uint64_t v0 = (uint64_t)s * svec;
        nv = s < a.slabs ? (uint32_t)min((uint64_t)svec, a.nvec - v0) : 0u;
        const int4 *vs = reinterpret_cast<const int4 *>(a.in + a.head) + v0 + tid;
#pragma unroll
        for (int u = 0; u < V; u++) {
            const int none = (int)(a.min_u - 1u);
            const int4 q = tid + u * kPartThreads < nv ? __ldcs(vs + u * kPartThreads) : make_int4(none, none, none, none);
            k[u][0] = (uint32_t)q.x, k[u][1] = (uint32_t)q.y, k[u][2] = (uint32_t)q.z, k[u][3] = (uint32_t)q.w;
        }
    };
    auto counter = [&](uint32_t y) -> uint32_t { return cnt_base + (min(y >> kPartShift, B) << (LOGC + 2)); };

    load(blockIdx.x);
    uint32_t row = 0;  // the CTA's keys of bucket `tid`
    for (uint32_t e = tid; e < E; e += kPartThreads) cnt[e] = 0;
    __syncthreads();
    for (uint32_t s = blockIdx.x; s < a.slabs; s += gridDim.x) {
        // The first slab also takes the keys before the first vector, the
        // last one those after the last (at most three each).
        const uint32_t front = s == 0 ? a.head : 0u;
        const uint32_t extra = front + (s + 1 == a.slabs ? (uint32_t)(a.n - a.head - 4 * a.nvec) : 0u);
        const int32_t *extra_in = tid < front ? a.in + tid : a.in + a.head + 4 * a.nvec + (tid - front);
#pragma unroll
        for (int u = 0; u < V; u++)
            if (u * kPartThreads < nv) {
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    k[u][e] -= a.min_u;
                    red_inc(counter(k[u][e]));
                }
            }
        if (tid < extra) red_inc(counter((uint32_t)*extra_in - a.min_u));
        __syncthreads();
        // Copies of a bucket: exclusive prefix within the bucket, and its total.
        for (uint32_t e0 = tid & ~31u; e0 < E; e0 += kPartThreads) {
            const uint32_t e = e0 + lane, c = lane & (C - 1);
            const uint32_t x = e < E ? cnt[e] : 0u;
            uint32_t inc = x;
#pragma unroll
            for (uint32_t d = 1; d < C; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
                if (c >= d) inc += y;
            }
            if (e < E) {
                cnt[e] = inc - x;
                if (c == C - 1) s_tot[e >> LOGC] = inc;
            }
        }
        __syncthreads();
        // Buckets (one per thread): starts in the staged slab, each rounded up
        // to 8 keys, and pads up to there.
        const uint32_t t = tid < B ? s_tot[tid] : 0u, room = (t + 7) & ~7u;
        uint32_t inc = room;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) s_warp[tid >> 5] = inc;
        __syncthreads();
        uint32_t w = lane < kPartThreads / 32 ? s_warp[lane] : 0u;
        if (lane >= tid >> 5) w = 0;
        const uint32_t off = __reduce_add_sync(0xffffffffu, w) + inc - room;
        if (tid <= B) s_off[tid] = off;
        row += t;
        for (uint32_t p = off + t; p < off + room; p++) sts_u16(stage_slot(stage + 2 * p), pad_of(tid));
        __syncthreads();
        for (uint32_t e = tid; e < E; e += kPartThreads) cnt[e] += s_off[e >> LOGC];
        __syncthreads();
#pragma unroll
        for (int u = 0; u < V; u++)
            if (u * kPartThreads < nv) {
                uint32_t p[4];
#pragma unroll
                for (int e = 0; e < 4; e++) p[e] = atom_inc(counter(k[u][e]));
#pragma unroll
                for (int e = 0; e < 4; e++) sts_u16(stage_slot(stage + 2 * p[e]), k[u][e]);
            }
        if (tid < extra) {
            const uint32_t y = (uint32_t)*extra_in - a.min_u;
            sts_u16(stage_slot(stage + 2 * atom_inc(counter(y))), y);
        }
        load(s + gridDim.x);
        __syncthreads();
        int4 *dst = a.payload + (size_t)s * a.slab_units;
        const uint32_t units = s_off[B] / 8;
        for (uint32_t i = tid; i < units; i += kPartThreads) {
            int4 q;
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                         : "r"(stage_slot(stage + 16 * i) & ~15u));
            dst[i] = q;
        }
        for (uint32_t b = tid; b <= B; b += kPartThreads) a.starts[(size_t)s * (B + 1) + b] = (uint16_t)(s_off[b] / 8);
        for (uint32_t e = tid; e < E; e += kPartThreads) cnt[e] = 0;
        __syncthreads();
    }
    asm volatile("griddepcontrol.launch_dependents;");
    if (tid < B) a.rows[(size_t)blockIdx.x * B + tid] = row;
}

// One CTA per SM taking items by ticket.  An item is a bucket and every k-th of
// its slabs (strided, so that the items of a bucket are even when the keys are
// sorted already), k from the bucket's keys.
//
// A bucket with few keys in a slab (less than 32 units): a group of lanes reads
// its run in one slab after another, up to four units a lane.  Longer runs: the
// item's slabs, 4096 at a time, are listed in shared memory as pieces of up to
// 128 units and the warps take the pieces in turn.  Either way each thread has
// the next four units in flight while it counts four, and the runs' ends are
// looked up one step earlier still.  n = 1e8, R = 2^20: 71 us uniform, 89 normal
// (30 for the reads alone): bound by its shared-memory reductions and, for
// buckets of a few keys a slab, by the latency of their many short runs (one run
// at a time instead of the groups of lanes: 206 us for the normal keys).
__global__ void __launch_bounds__(kBucketThreads, 1) bucket_kernel(PartArgs a) {
    extern __shared__ __align__(16) uint32_t s_mem[];
    uint32_t *S = s_mem + 4;                       // the tile, with a word for pads on both sides
    uint32_t *s_piece = S + kPartWidth + 4;        // pieces before each listed slab
    uint32_t *s_units = s_piece + kPartList;      // its units of the bucket: start | end << 16
    __shared__ uint32_t s_begin[kPartMaxBuckets + 1];  // items before each bucket
    __shared__ uint32_t s_keys[kPartMaxBuckets];
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_item;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t B = a.buckets;
    for (uint32_t b = tid; b < B; b += kBucketThreads) s_keys[b] = 0;
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (a.ctl->status & kDevTimeout) return;  // part_kernel has written nothing
    // The buckets' keys, from the totals of part_kernel's CTAs.
    {
        uint32_t cols = 32;
        while (cols < B) cols <<= 1;
        const uint32_t b = tid & (cols - 1), step = kBucketThreads / cols;
        uint32_t t = 0;
        if (b < B) {
#pragma unroll 16
            for (uint32_t r = tid / cols; r < a.part_ctas; r += step) t += a.rows[(size_t)r * B + b];
            if (t) atomicAdd(&s_keys[b], t);
        }
    }
    __syncthreads();
    auto block_incl = [&](uint32_t x, uint32_t *total) -> uint32_t {
        uint32_t inc = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) s_warp[warp] = inc;
        __syncthreads();
        uint32_t w = s_warp[lane], wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, d);
            if (lane >= d) wi += y;
        }
        *total = __shfl_sync(0xffffffffu, wi, 31);
        const uint32_t before = __shfl_sync(0xffffffffu, wi - w, warp);
        __syncthreads();
        return before + inc;
    };
    // Items of each bucket: none for an empty one, else its keys (in 16s) over
    // the keys and tiles of an even share.  Every CTA computes the same numbers.
    const uint32_t t = tid < B ? s_keys[tid] : 0u;
    const uint32_t weight = t ? t / 16 + a.tile_cost : 0u;
    uint32_t total = 0, items = 0;
    if (blockIdx.x == 0) {  // (for wide_out.cu)
        const uint32_t end = block_incl(t, &total);
        if (tid < B) a.bucket_start[tid + 1] = end;
        if (tid == 0) a.bucket_start[0] = 0;
    }
    block_incl(weight, &total);
    const uint32_t target = max(1u, total / a.target_items);
    const uint32_t incl = block_incl(t ? min(a.slabs, max(1u, t / 16 / target)) : 0u, &items);
    if (tid < B) s_begin[tid + 1] = incl;
    if (tid == 0) s_begin[0] = 0;
    for (;;) {
        if (tid == 0) s_item = atomicAdd(&a.ctl->part_ticket, 1u);
        __syncthreads();  // also: the items are placed, the previous item's tile has been read
        const uint32_t item = s_item;
        if (item >= items) break;
        uint32_t b = 0, bh = B - 1;  // last bucket whose first item is at or before it
        while (b < bh) {
            const uint32_t mid = (b + bh + 1) >> 1;
            if (s_begin[mid] <= item) b = mid; else bh = mid - 1;
        }
        const uint32_t sub = item - s_begin[b], k = s_begin[b + 1] - s_begin[b];
        const uint32_t ns = (a.slabs - sub + k - 1) / k;  // slabs sub, sub + k, ...
        const uint32_t w = min(kPartWidth, a.R - b * kPartWidth);
        for (uint32_t i = tid; i < kPartWidth / 4; i += kBucketThreads)
            reinterpret_cast<uint4 *>(S)[i] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        // (the keys of an odd bucket carry its parity in bit 15)
        const uint32_t s_base = (uint32_t)__cvta_generic_to_shared(S) - (b & 1 ? 4 * kPartWidth : 0u);
        auto count2 = [&](uint32_t x) {
            red_inc(s_base + 4u * (x & 0xffffu));
            red_inc(s_base + 4u * (x >> 16));
        };
        auto count8 = [&](const int4 q) {
            count2((uint32_t)q.x); count2((uint32_t)q.y); count2((uint32_t)q.z); count2((uint32_t)q.w);
        };
        const uint16_t *st = a.starts + b;
        int4 q[4];
        const uint32_t avg = s_keys[b] / 8 / a.slabs + 1;  // units of a run
        if (avg < 32) {
            const uint32_t log_g = avg <= 3 ? 0 : avg <= 6 ? 1 : avg <= 12 ? 2 : 3;
            const uint32_t G = 1u << log_g, gl = lane & (G - 1), ng = kBucketThreads >> log_g;
            const uint32_t g = (lane >> log_g) * 32 + warp;  // consecutive slabs go to different warps
            const uint32_t rounds = (ns + ng - 1) / ng;      // (the same for every lane)
            uint32_t no0 = 0, no1 = 0;
            auto ends = [&](uint32_t r) {
                const uint32_t i = g + r * ng;
                no0 = no1 = 0;
                if (i < ns) {
                    const uint16_t *ss = st + (size_t)(sub + k * i) * (B + 1);
                    no0 = ss[0];
                    no1 = ss[1];
                }
            };
            uint32_t o = 0, e = 0;  // this lane's units of q: o + u * G below e
            auto load = [&](uint32_t r) {
                const int4 *pl = a.payload + (size_t)(sub + k * (g + r * ng)) * a.slab_units;
                o = no0 + gl;
                e = no1;
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (o + u * G < e) q[u] = __ldcs(pl + o + u * G);
            };
            ends(0);
            load(0);
            ends(1);
            for (uint32_t r = 0; r < rounds; r++) {
                int4 c[4];
                const uint32_t co = o, ce = e;
#pragma unroll
                for (int u = 0; u < 4; u++) c[u] = q[u];
                load(r + 1);  // (no units past the last round)
                ends(r + 2);
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (co + u * G < ce) count8(c[u]);
                // The rest of a run much longer than the others: the whole warp.
                uint32_t more = __ballot_sync(0xffffffffu, co - gl + 4 * G < ce);
                while (more) {
                    const int src = __ffs(more) - 1;  // its group's first lane
                    const uint32_t x0 = __shfl_sync(0xffffffffu, co, src) + 4 * G, x1 = __shfl_sync(0xffffffffu, ce, src);
                    const int4 *pl = a.payload +
                                     (size_t)(sub + k * (__shfl_sync(0xffffffffu, g, src) + r * ng)) * a.slab_units;
                    for (uint32_t p = x0 + lane; p < x1; p += 32) count8(__ldcs(pl + p));
                    more &= ~(((1u << G) - 1u) << src);
                }
            }
        } else {
            for (uint32_t j0 = 0; j0 < ns; j0 += kPartList) {
                constexpr int L = kPartList / kBucketThreads;
                uint32_t o0[L], o1[L], mine = 0;
#pragma unroll
                for (int u = 0; u < L; u++) {
                    const uint32_t j = j0 + tid * L + u;
                    o0[u] = o1[u] = 0;
                    if (j < ns) {
                        const uint16_t *ss = st + (size_t)(sub + k * j) * (B + 1);
                        o0[u] = ss[0];
                        o1[u] = ss[1];
                    }
                }
#pragma unroll
                for (int u = 0; u < L; u++) mine += (o1[u] - o0[u] + 127) / 128;
                uint32_t pieces = 0;
                uint32_t pin = block_incl(mine, &pieces) - mine;  // (also: the previous list is no longer read)
#pragma unroll
                for (int u = 0; u < L; u++) {
                    s_piece[tid * L + u] = pin;
                    s_units[tid * L + u] = o0[u] | (o1[u] << 16);
                    pin += (o1[u] - o0[u] + 127) / 128;
                }
                __syncthreads();
                // Lane l finds the warp's l-th piece of 32 rounds at a time.
                uint32_t my_o = 0, my_e = 0, my_s = 0;
                auto find = [&](uint32_t pc) {
                    uint32_t x = 0, xh = kPartList - 1;  // last slab with s_piece <= pc
                    while (x < xh) {
                        const uint32_t mid = (x + xh + 1) >> 1;
                        if (s_piece[mid] <= pc) x = mid; else xh = mid - 1;
                    }
                    const uint32_t un = s_units[x];
                    my_s = sub + k * (j0 + x);
                    my_o = (un & 0xffffu) + 128 * (pc - s_piece[x]);
                    my_e = min(un >> 16, my_o + 128);
                    if (pc >= pieces) my_o = my_e = 0;
                };
                uint32_t left = 0;  // this lane's units of q: those u with 32 u < left
                auto load = [&](uint32_t r) {
                    const uint32_t o = __shfl_sync(0xffffffffu, my_o, r & 31) + lane;
                    const uint32_t e = __shfl_sync(0xffffffffu, my_e, r & 31);
                    const int4 *pl = a.payload + (size_t)__shfl_sync(0xffffffffu, my_s, r & 31) * a.slab_units;
                    left = e > o ? e - o : 0u;
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (32 * u < left) q[u] = __ldcs(pl + o + 32 * u);
                };
                const uint32_t rounds = pieces > warp ? (pieces - warp + 31) / 32 : 0u;
                if (rounds) {
                    find(warp + 32 * lane);
                    load(0);
                }
                for (uint32_t r = 0; r < rounds; r++) {
                    int4 c[4];
                    const uint32_t cl = left;
#pragma unroll
                    for (int u = 0; u < 4; u++) c[u] = q[u];
                    if (r + 1 < rounds) {
                        if (((r + 1) & 31) == 0) find(warp + 32 * (r + 1 + lane));
                        load(r + 1);
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (32 * u < cl) count8(c[u]);
                }
            }
        }
        __syncthreads();
        uint32_t *H = a.H + (size_t)b * kPartWidth;
        uint32_t lower = 0;
        for (uint32_t i = tid; i < w; i += kBucketThreads) {
            const uint32_t c = S[i];
            if (c) atomicAdd(&H[i], c);
            if (i < kPartWidth / 2) lower += c;
        }
        if (a.half) {
            lower = __reduce_add_sync(0xffffffffu, lower);
            if (lane == 0 && lower) atomicAdd(&a.half[b], lower);
        }
    }
    asm volatile("griddepcontrol.launch_dependents;");
}

bool part_plan(uint64_t n, uint32_t R, uint32_t head, uint64_t nvec, uintptr_t out_addr, int sms, PartPlan *p) {
    p->buckets = (R + kPartWidth - 1) >> kPartShift;
    const uint32_t B = p->buckets;
    // Slabs of up to 32768 keys, as even over the SMs as whole vectors of the
    // CTA allow.
    const uint64_t want = (n + sms - 1) / sms;
    // (in whole vectors of the CTA: its threads' vectors past a slab's end are
    // staged too, as keys outside the range)
    const uint64_t step = 4 * kPartThreads;
    const uint64_t rounds = (want + kPartSlabMax - 1) / kPartSlabMax;
    const uint64_t keys = std::max<uint64_t>({kPartSlabMin, 16ull * B, (want + rounds - 1) / rounds});
    p->slab_keys = (uint32_t)std::min<uint64_t>(kPartSlabMax, (keys + step - 1) / step * step);
    const uint64_t slabs = std::max<uint64_t>(1, (nvec + p->slab_keys / 4 - 1) / (p->slab_keys / 4));
    p->slabs = (uint32_t)slabs;
    p->slab_units = part_slab_units(B, p->slab_keys);
    p->ctas = (uint32_t)std::min<uint64_t>(slabs, sms);
    p->smem = part_smem(B, p->slab_keys);
    const uintptr_t base = (out_addr + 15) & ~(uintptr_t)15;
    const uint64_t payload = slabs * p->slab_units * 16;
    const uint64_t starts = (slabs * (B + 1) * 2 + 15) / 16 * 16;
    const uint64_t rows = (uint64_t)p->ctas * B * 4;
    p->payload = base;
    p->starts = base + payload;
    p->rows = base + payload + starts;
    return p->rows + rows <= out_addr + 4 * n;
}

cudaError_t launch_part(const PartPlan &p, const int32_t *in, uint64_t n, uint32_t head, uint64_t nvec, uint32_t min_u,
                        uint32_t R, uint32_t *H, uint32_t *bucket_start, uint32_t *half, Ctl *ctl, int sms,
                        cudaStream_t s) {
    PartArgs a;
    a.in = in; a.n = n; a.nvec = nvec; a.head = head; a.min_u = min_u; a.R = R;
    a.buckets = p.buckets; a.slabs = p.slabs; a.slab_keys = p.slab_keys; a.slab_units = p.slab_units;
    a.part_ctas = p.ctas;
    a.tile_cost = (kPartTileKeys + 2 * p.slabs) / 16;
    a.target_items = (p.buckets > 64 ? 4 : 2) * (uint32_t)sms;
    a.payload = reinterpret_cast<int4 *>(p.payload);
    a.starts = reinterpret_cast<uint16_t *>(p.starts);
    a.rows = reinterpret_cast<uint32_t *>(p.rows);
    a.H = H; a.bucket_start = bucket_start; a.half = half; a.ctl = ctl;
    void *args[] = {&a};
    static std::atomic<uint64_t> raised[2] = {};
    const bool few = p.buckets <= 128;
    const void *pf = few ? (const void *)part_kernel<part_log_copies(128)>
                         : (const void *)part_kernel<part_log_copies(kPartMaxBuckets)>;
    cudaError_t e = raise_shared_limit(pf, part_smem(few ? 128 : kPartMaxBuckets, kPartSlabMax), raised[few]);
    if (e != cudaSuccess) return e;
    if ((e = cudaLaunchKernel(pf, dim3(p.ctas), dim3(kPartThreads), args, p.smem, s)) != cudaSuccess) return e;
    const void *fn = (const void *)bucket_kernel;
    const size_t smem = 4 * ((size_t)kPartWidth + 8 + 2 * kPartList);
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((uint32_t)sms);
    cfg.blockDim = dim3(kBucketThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace rtcdf
