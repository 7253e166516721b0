// Histogram of a range of a few shared-memory tiles (R up to about 360000) in
// one pass over the input, with several counters in a 32-bit word.
//
// The range-tile kernel (hist.cu) reads and examines every key once per tile of
// 57344 32-bit counters.  Here one CTA per SM holds the whole range: F values
// share a word, b = 32 / F bits each (value y in word y mod W, field y / W), and
// every key is one shared-memory reduction of 1 << (b * field).  A field that
// overflows carries into the next, or out of the word: either way the sum of
// the CTA's fields falls short of the keys it has counted, so the overflow is
// found exactly, and the CTA then counts its keys of that round again, by range
// tiles with 32-bit counters.
//
// What keeps overflows rare is a sample of the input (8192 keys, the same ones
// in every CTA, so that all decide alike):
//   - its most frequent key, when it holds 64 of them (0.8 %), is counted in a
//     register instead of a field (a column of one value, or with many zeros);
//   - the densest stretch of the range, and the next most frequent key, give
//     the rounds after which the fields are written out and cleared;
//   - an input that would need too many rounds (several frequent keys, or a
//     range of which only a small part is used), or whose neighbours are alike
//     (sorted or clustered keys: they fill a field within one block of the
//     input, and the lanes of a warp meet on a word) is counted by range tiles,
//     here or by a launch of hist.cu of its own (kPackTilesLaunchMin).
//
// The fields leave the CTA as they are, 32 MB for R = 2^18, into the sort's
// output buffer (which nothing reads before the output kernel fills it), and
// pack_sum_kernel adds them up.  Without that scratch the two CTAs of a cluster
// add up their fields over distributed shared memory, half each, and the sums to
// H: an SM passes on about 20 bytes of reductions a cycle, so its own counters,
// 1 MB for R = 2^18, take it 28 us however many SMs there are, half of them 14
// (n = 5e7, R = 2^18, histogram alone: 70 us against 78.5; clusters of four do not
// fit all SMs: 119).
//
// Measured (n = 1e8, uniform / normal / one value, histogram of a sort, us; the
// range tiles before that): R = 2^16 82 / 82 / 81 (92 / 92 / 85), 2^17 85 / 86 / 85
// (129 / 162 / 107), 2^18 92 / 92 / 92 (200 / 244 / 189), 350000 95 / 132 / 95 (259 /
// 308 / 244); n = 1e9, R = 2^18 680 / 770 (2189 / 2640).  Reading 4n bytes takes 59:
// the input's stream bounds it, together with writing back the 25 MB that the
// previous sort's output left dirty in L2, the sample (about 4 us) and the sum
// (7 to 13 us).  Three, four and six vectors in flight a thread are the same up
// to 128 KB of counters; six are slower at 176 KB (the L1 that is left).
#include <algorithm>

#include "hist_tiles.cuh"

namespace rtcdf {

namespace {

constexpr int kPackThreads = 1024;
constexpr int kSampleVecs = 2;                      // vectors each thread samples
constexpr uint32_t kSampleKeys = kPackThreads * kSampleVecs * 4;
constexpr uint32_t kHashBits = 14;                  // sample hash table, in the counters' shared memory
constexpr uint32_t kCoarse = 256;                   // stretches of the range
constexpr int kPackCluster = 2;                     // CTAs that add up their fields before H (without scratch)
constexpr uint32_t kHotMin = 64;                    // sampled keys that make a key hot
constexpr uint32_t kPackMaxWords = 45056 + 1024, kPackMaxTile = 45056;  // of pack_plan
constexpr size_t kPackSmem = 4 * (size_t)kPackMaxWords + 16;
constexpr uint32_t kSingleNoise = 12;               // hash counts that uniform and normal keys reach

__device__ __forceinline__ uint32_t sample_hash(uint32_t y) { return (y * 0x9E3779B1u) >> (32 - kHashBits); }

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
// The word at `s_addr` of the cluster's CTA c.
__device__ __forceinline__ uint32_t cluster_word(uint32_t s_addr, uint32_t c) {
    uint32_t x;
    asm volatile(
        "{\n\t.reg .u32 r;\n\t"
        "mapa.shared::cluster.u32 r, %1, %2;\n\t"
        "ld.shared::cluster.u32 %0, [r];\n\t}"
        : "=r"(x) : "r"(s_addr), "r"(c) : "memory");
    return x;
}

}  // namespace

__global__ void __launch_bounds__(kPackThreads, 1) pack_kernel(PackArgs a) {
    extern __shared__ __align__(16) uint32_t S[];
    __shared__ uint32_t s_coarse[kCoarse];
    __shared__ unsigned long long s_best;
    __shared__ uint32_t s_single, s_dense, s_near, s_alike, s_smooth, s_keys, s_diff, s_hot, s_tc[8];
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const HistArgs &h = a.h;
    const int4 *vin = reinterpret_cast<const int4 *>(h.in + h.head);
    const uint64_t nvec = h.nvec;
    const uint32_t min_u = h.min_u, R = h.R;

    // After a wait that ran out nothing is written to the output (nor to its
    // use as scratch) until the status has been read.
    if (a.dump && (a.ctl->status & kDevTimeout)) {
        if (blockIdx.x == 0 && tid == 0) {
            a.ctl->pack_copies = 0;
            if (a.tiles_later) *a.tiles_later = 0;
        }
        return;
    }

    // ---- the sample
    for (uint32_t i = tid; i < (1u << kHashBits); i += kPackThreads) S[i] = 0;
    if (tid < kCoarse) s_coarse[tid] = 0;
    if (tid == 0) {
        s_best = 0;
        s_single = s_dense = s_near = s_alike = s_smooth = s_keys = s_diff = s_hot = 0;
    }
    uint32_t y[4 * kSampleVecs];
#pragma unroll
    for (int u = 0; u < kSampleVecs; u++) {
        const int4 k = __ldg(vin + (uint64_t)(tid + u * kPackThreads) * nvec / (kPackThreads * kSampleVecs));
        y[4 * u] = (uint32_t)k.x - min_u, y[4 * u + 1] = (uint32_t)k.y - min_u;
        y[4 * u + 2] = (uint32_t)k.z - min_u, y[4 * u + 3] = (uint32_t)k.w - min_u;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4 * kSampleVecs; i++)
        if (y[i] < R) {
            atomicAdd(&S[sample_hash(y[i])], 1u);
            atomicAdd(&s_coarse[y[i] >> a.coarse_shift], 1u);
        }
    __syncthreads();
    {
        unsigned long long best = 0;
#pragma unroll
        for (int i = 0; i < 4 * kSampleVecs; i++)
            if (y[i] < R) best = max(best, (unsigned long long)S[sample_hash(y[i])] << 32 | y[i]);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, d));
        if (lane == 0) atomicMax(&s_best, best);
    }
    __syncthreads();
    const bool has_hot = (uint32_t)(s_best >> 32) >= kHotMin;
    const uint32_t hot = has_hot ? (uint32_t)s_best : 0xffffffffu;
    {
        uint32_t single = 0, n_hot = 0, alike = 0, keys = 0;
#pragma unroll
        for (int i = 0; i < 4 * kSampleVecs; i++) {
            if (y[i] == hot) n_hot++;
            else if (y[i] < R) {
                const uint32_t c = S[sample_hash(y[i])];
                single = max(single, c);
                alike += c - 1;
                keys++;
            }
        }
        if (has_hot && n_hot) atomicSub(&s_coarse[hot >> a.coarse_shift], n_hot);
        single = __reduce_max_sync(0xffffffffu, single);
        if (lane == 0) atomicMax(&s_single, single);
        // Keys close to each other: inside a vector (+1), and between the
        // thread's two vectors, half the input apart (-4 a pair: twice as
        // many of the others expected, and as many again allowed).
        auto near = [&](uint32_t p, uint32_t q) -> bool {
            return p < R && q < R && p != hot && (p > q ? p - q : q - p) <= R / 512;
        };
        const int close = (int)near(y[0], y[3]) + (int)near(y[4], y[7]) - 4 * (int)near(y[0], y[4]);
        const uint32_t sum = __reduce_add_sync(0xffffffffu, (uint32_t)close);
        alike = __reduce_add_sync(0xffffffffu, alike);
        keys = __reduce_add_sync(0xffffffffu, keys);
        if (lane == 0) {
            atomicAdd(&s_near, sum);
            atomicAdd(&s_alike, alike);
            atomicAdd(&s_keys, keys);
        }
    }
    __syncthreads();
    {
        const uint32_t c = tid < kCoarse ? s_coarse[tid] : 0u;
        const uint32_t dense = __reduce_max_sync(0xffffffffu, c), smooth = __reduce_add_sync(0xffffffffu, c * c);
        if (lane == 0) {
            atomicMax(&s_dense, dense);
            atomicAdd(&s_smooth, smooth);
        }
    }
    __syncthreads();
    // Expected keys of one CTA in its fullest field, and the rounds that keep
    // them below the limit.  The densest stretch of the range gives them when
    // its values are all in use; more pairs of sampled keys that are alike than
    // such stretches have (and than the hash makes alike, with three standard
    // deviations) raise the estimate by as much: keys that are multiples of
    // something, or many moderately frequent ones.
    const float stretch = 1.f / (float)(1u << a.coarse_shift);
    const float hashed = (float)s_keys * (float)s_keys / (float)(1u << kHashBits);
    const float spike = ((float)s_alike - hashed - 3.f * sqrtf(2.f * hashed)) / ((float)s_smooth * stretch + 1.f);
    const float dense = ((float)s_dense - sqrtf((float)s_dense)) * stretch * fmaxf(1.f, spike);
    const float single = s_single > kSingleNoise ? (float)s_single : 0.f;
    const float fullest = fmaxf(dense, single) * ((float)h.n / (float)gridDim.x / (float)kSampleKeys);
    const float want = ceilf(fullest / a.limit);
    const bool tiles = want > (float)a.max_rounds || (int)s_near > (int)(kSampleVecs * kPackThreads / 16);
    const uint32_t rounds = tiles ? 0u : max(1u, (uint32_t)want);
    if (blockIdx.x == 0 && tid == 0) {
        if (a.dump) a.ctl->pack_copies = rounds * gridDim.x;
        if (a.tiles_later) *a.tiles_later = tiles;
    }
    if (tiles) {
        if (!a.tiles_later && blockIdx.x < h.m * h.g) hist_tiles<false, 8, true>(h, blockIdx.x, S, s_tc);
        return;
    }

    // ---- packed counters
    const uint32_t W = a.words, F = a.fields, bits = 32 / F, mask = (1u << bits) - 1u;
    uint4 *S4 = reinterpret_cast<uint4 *>(S);
    for (uint32_t i = tid; i < W / 4; i += kPackThreads) S4[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    const uint32_t s_base = (uint32_t)__cvta_generic_to_shared(S);
    const uint32_t minus_4w = 0u - 4u * W, magic = a.magic;
    uint32_t n_hot = 0;
    // A key: its field y / W by multiplication (exact, see pack_plan), its
    // word, and one reduction; the hot key is only counted.
    auto count = [&](int32_t key) {
        const uint32_t yy = (uint32_t)key - min_u;
        const uint32_t f = __umulhi(yy, magic);
        const uint32_t addr = s_base + 4u * yy + f * minus_4w;
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "setp.eq.u32 q, %1, %2;\n\t"
            "@q add.u32 %0, %0, 1;\n\t"
            "setp.lt.and.u32 p, %1, %3, !q;\n\t"
            "@p red.shared.add.u32 [%4], %5;\n\t}"
            : "+r"(n_hot)
            : "r"(yy), "r"(hot), "r"(R), "r"(addr), "r"(1u << (f * bits)));
    };
    auto count4 = [&](const int4 k) { count(k.x); count(k.y); count(k.z); count(k.w); };

    const uint64_t stride = (uint64_t)gridDim.x * kPackThreads;
    const uint64_t first = (uint64_t)blockIdx.x * kPackThreads + tid;
    const uint64_t per_round = ((nvec + stride - 1) / stride + rounds - 1) / rounds * stride;  // vectors of all CTAs
    const uint32_t tail = (uint32_t)(h.n - h.head - 4 * nvec);
    uint32_t hot_total = 0;
    for (uint32_t r = 0; r < rounds; r++) {
        const uint64_t v0 = first + r * per_round;
        const uint64_t v1 = r + 1 < rounds ? min(nvec, (r + 1) * per_round) : nvec;
        // The last round also takes the keys outside whole vectors (CTA 0).
        const uint32_t extra = r + 1 == rounds && blockIdx.x == 0 ? h.head + tail : 0u;
        const int32_t *extra_in = tid < h.head ? h.in + tid : h.in + h.head + 4 * nvec + (tid - h.head);
        uint4 *dump = a.dump ? reinterpret_cast<uint4 *>(a.dump + ((size_t)r * gridDim.x + blockIdx.x) * W) : nullptr;
        bool recount;
        {
            n_hot = 0;
            constexpr int P = 4;
            uint64_t v = v0;
            if (v + (P - 1) * stride < v1) {
                int4 kn[P];
#pragma unroll
                for (int u = 0; u < P; u++) kn[u] = __ldcs(vin + v + u * stride);
                v += P * stride;
                for (; v + (P - 1) * stride < v1; v += P * stride) {
                    int4 kc[P];
#pragma unroll
                    for (int u = 0; u < P; u++) kc[u] = kn[u];
#pragma unroll
                    for (int u = 0; u < P; u++) kn[u] = __ldcs(vin + v + u * stride);
#pragma unroll
                    for (int u = 0; u < P; u++) count4(kc[u]);
                }
#pragma unroll
                for (int u = 0; u < P; u++) count4(kn[u]);
            }
            for (; v < v1; v += stride) count4(__ldcs(vin + v));
            if (tid < extra) count(*extra_in);
            __syncthreads();
            // Keys of the fields and hot keys against the keys read.
            uint32_t diff = n_hot - (tid < extra ? 1u : 0u);
            if (v0 < v1) diff -= 4u * (uint32_t)((v1 - v0 + stride - 1) / stride);
            for (uint32_t i = tid; i < W / 4; i += kPackThreads) {
                const uint4 x = S4[i];
                for (uint32_t f = 0, sh = 0; f < F; f++, sh += bits)
                    diff += ((x.x >> sh) & mask) + ((x.y >> sh) & mask) + ((x.z >> sh) & mask) + ((x.w >> sh) & mask);
                if (dump) {
                    __stcg(dump + i, x);
                    S4[i] = make_uint4(0, 0, 0, 0);
                }
            }
            diff = __reduce_add_sync(0xffffffffu, diff);
            const uint32_t hots = __reduce_add_sync(0xffffffffu, n_hot);
            if (lane == 0) {
                atomicAdd(&s_diff, diff);
                atomicAdd(&s_hot, hots);
            }
            __syncthreads();
            recount = s_diff != 0;
            if (!recount) hot_total += s_hot;
            __syncthreads();
            if (tid == 0) s_diff = s_hot = 0;
        }
        if (recount) {
            // An overflow (or a key outside the range, which the scan
            // reports): this CTA's keys of the round again, by range tiles.
            if (dump)
                for (uint32_t i = tid; i < W / 4; i += kPackThreads) __stcg(dump + i, make_uint4(0, 0, 0, 0));
            for (uint32_t b = 0; b < R; b += h.T) {
                const uint32_t w = min(h.T, R - b), base = min_u + b;
                for (uint32_t i = tid; i < w; i += kPackThreads) S[i] = 0;
                __syncthreads();
                auto tile4 = [&](const int4 k) {
                    count_key(s_base, (uint32_t)k.x - base, w);
                    count_key(s_base, (uint32_t)k.y - base, w);
                    count_key(s_base, (uint32_t)k.z - base, w);
                    count_key(s_base, (uint32_t)k.w - base, w);
                };
                uint64_t v = v0;
                for (; v + 3 * stride < v1; v += 4 * stride) {
                    int4 k[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) k[u] = __ldg(vin + v + u * stride);
#pragma unroll
                    for (int u = 0; u < 4; u++) tile4(k[u]);
                }
                for (; v < v1; v += stride) tile4(__ldg(vin + v));
                if (tid < extra) count_key(s_base, (uint32_t)*extra_in - base, w);
                __syncthreads();
                for (uint32_t i = tid; i < w; i += kPackThreads) {
                    const uint32_t c = S[i];
                    if (c) atomicAdd(&h.H[b + i], c);
                }
                __syncthreads();
            }
            for (uint32_t i = tid; i < W / 4; i += kPackThreads) S4[i] = make_uint4(0, 0, 0, 0);
        }
        __syncthreads();
        if (!dump) {
            // The CTAs of a cluster add up their fields, each a share of the
            // words, and every cluster starts at another word of the share, so
            // that they do not meet.
            constexpr uint32_t cs = kPackCluster;
            const uint32_t rank = blockIdx.x % cs;
            cluster_sync();
            const uint32_t w0 = (uint32_t)((uint64_t)W * rank / cs);
            const uint32_t len = (uint32_t)((uint64_t)W * (rank + 1) / cs) - w0;
            const uint32_t rot = (uint32_t)((uint64_t)len * blockIdx.x / gridDim.x);
            constexpr int P = 4;
            for (uint32_t i0 = tid; i0 < len; i0 += P * kPackThreads) {
                uint32_t w[P], x[P][kPackCluster];
#pragma unroll
                for (int u = 0; u < P; u++) {
                    const uint32_t i = i0 + u * kPackThreads;
                    w[u] = w0 + (i + rot < len ? i + rot : i + rot - len);
#pragma unroll
                    for (int c = 0; c < kPackCluster; c++) x[u][c] = i < len ? cluster_word(s_base + 4 * w[u], c) : 0u;
                }
                for (uint32_t f = 0, sh = 0; f < F; f++, sh += bits)
#pragma unroll
                    for (int u = 0; u < P; u++) {
                        uint32_t sum = 0;
#pragma unroll
                        for (int c = 0; c < kPackCluster; c++) sum += (x[u][c] >> sh) & mask;
                        if (sum) atomicAdd(&h.H[f * W + w[u]], sum);
                    }
            }
            cluster_sync();
            for (uint32_t i = tid; i < W / 4; i += kPackThreads) S4[i] = make_uint4(0, 0, 0, 0);
            __syncthreads();
        }
    }
    asm volatile("griddepcontrol.launch_dependents;");
    if (has_hot && tid == 0 && hot_total) atomicAdd(&h.H[hot], hot_total);
}

// H += the fields of all copies: a block adds up 16 x 4 words, its 16 groups of
// 16 lanes taking the copies in turn.
template <int F>
__global__ void __launch_bounds__(256) pack_sum_kernel(PackArgs a) {
    __shared__ uint32_t s_sum[16][F * 64];
    const uint32_t tid = threadIdx.x, l = tid & 15, grp = tid >> 4;
    constexpr uint32_t bits = 32 / F, mask = (1u << bits) - 1u;
    const uint32_t q = blockIdx.x * 16 + l, quads = a.words / 4;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const uint32_t copies = a.ctl->pack_copies;
    if (copies == 0) return;
    uint32_t acc[F][4] = {};
    if (q < quads) {
        const uint4 *d = reinterpret_cast<const uint4 *>(a.dump) + q;
#pragma unroll 4
        for (uint32_t c = grp; c < copies; c += 16) {
            const uint4 x = __ldcg(d + (size_t)c * quads);
#pragma unroll
            for (int f = 0; f < F; f++) {
                acc[f][0] += (x.x >> (f * bits)) & mask;
                acc[f][1] += (x.y >> (f * bits)) & mask;
                acc[f][2] += (x.z >> (f * bits)) & mask;
                acc[f][3] += (x.w >> (f * bits)) & mask;
            }
        }
    }
#pragma unroll
    for (int f = 0; f < F; f++)
#pragma unroll
        for (int e = 0; e < 4; e++) s_sum[grp][f * 64 + 4 * l + e] = acc[f][e];
    __syncthreads();
    for (uint32_t i = tid; i < F * 64; i += 256) {
        uint32_t c = 0;
#pragma unroll
        for (int g = 0; g < 16; g++) c += s_sum[g][i];
        const uint32_t y = (i >> 6) * a.words + blockIdx.x * 64 + (i & 63);
        if (c && blockIdx.x * 64 + (i & 63) < a.words && y < a.h.R) atomicAdd(&a.h.H[y], c);
    }
}

bool pack_plan(uint64_t n, uint32_t R, uint64_t nvec, uintptr_t scratch, int sms, PackPlan *p) {
    // The fewest fields that keep the counters near 128 KB: above about 176 KB
    // the L1 cache is too small for the loads in flight.
    const uint32_t fields = R <= 2 * 32768 ? 2 : R <= 4 * 32768 ? 4 : R <= 5 * 32768 ? 5 : R <= 6 * 45056 ? 6 : 8;
    p->fields = fields;
    // Words, so that y / W == umulhi(y, magic) for every y < fields * W: with
    // e = magic * W - 2^32 that holds when y * e < 2^32.
    uint32_t W = std::max<uint32_t>((R + fields - 1) / fields, 1u << kHashBits);
    for (W = (W + 3) / 4 * 4;; W += 4) {
        if (W > kPackMaxWords) return false;
        p->magic = (uint32_t)(((1ull << 32) + W - 1) / W);
        if (((uint64_t)p->magic * W - (1ull << 32)) * fields * W < (1ull << 32)) break;
    }
    p->words = W;
    // Expected keys of the fullest field that overflow with a chance below 1e-7
    // (Poisson tails).
    p->limit = fields == 2 ? 30000.f : fields == 4 ? 140.f : fields == 5 ? 24.f : fields == 6 ? 10.f : 2.5f;
    p->ctas = (uint32_t)std::min<uint64_t>(sms, nvec / (4 * kPackThreads)) / kPackCluster * kPackCluster;
    if (p->ctas == 0) return false;
    // Range tiles: as few as kPackMaxTile values allow, and the trash word.
    p->m = (R + kPackMaxTile - 1) / kPackMaxTile;
    p->tile = (R + p->m - 1) / p->m;
    p->smem = (size_t)std::max(W, p->tile) * 4 + 16;
    p->g = std::max(1u, p->ctas / p->m);
    if (p->m > 8 || p->m * p->g > p->ctas) return false;
    // A round (the fields written out and added up) takes about 7 us, as much as
    // counting 150000 keys of a CTA once, and a range tile's pass over the keys
    // three fifths of the packed pass: twice that, for inputs whose few values
    // also meet in few banks.
    p->max_rounds = 1 + (uint32_t)std::min<uint64_t>(1000, n / p->ctas * (p->m - 1) / 500000);
    p->dump = 0;
    if (scratch) {
        const uintptr_t base = (scratch + 15) & ~(uintptr_t)15;
        const uint64_t room = (scratch + 4 * n - base) / (4ull * W * p->ctas);
        if (room >= 1) {
            p->dump = base;
            p->max_rounds = (uint32_t)std::min<uint64_t>(p->max_rounds, room);
        }
    }
    return true;
}

cudaError_t launch_pack(const PackPlan &p, const HistArgs &hist, Ctl *ctl, bool tiles_later, cudaStream_t s) {
    PackArgs a;
    a.h = hist;
    a.h.T = p.tile; a.h.m = p.m; a.h.g = p.g;
    a.words = p.words; a.fields = p.fields; a.magic = p.magic; a.limit = p.limit; a.max_rounds = p.max_rounds;
    a.coarse_shift = 0;
    while (((hist.R - 1) >> a.coarse_shift) >= kCoarse) a.coarse_shift++;
    a.dump = ctl ? reinterpret_cast<uint32_t *>(p.dump) : nullptr;
    a.ctl = ctl;
    a.tiles_later = tiles_later ? &ctl->pack_tiles : nullptr;
    void *args[] = {&a};
    static std::atomic<uint64_t> raised{0};
    cudaError_t e = raise_shared_limit((const void *)pack_kernel, kPackSmem, raised);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.blockDim = dim3(kPackThreads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(p.ctas);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = a.dump ? 1 : kPackCluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    if ((e = cudaLaunchKernelExC(&cfg, (const void *)pack_kernel, args)) != cudaSuccess) return e;
    if (!a.dump) return cudaSuccess;
    const void *fn = p.fields == 2   ? (const void *)pack_sum_kernel<2>
                     : p.fields == 4 ? (const void *)pack_sum_kernel<4>
                     : p.fields == 5 ? (const void *)pack_sum_kernel<5>
                     : p.fields == 6 ? (const void *)pack_sum_kernel<6>
                                     : (const void *)pack_sum_kernel<8>;
    cfg.gridDim = dim3((p.words / 4 + 15) / 16);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = 0;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace rtcdf
