// One CTA's share of the range-tile histogram (Algorithm 5), for the kernels
// that count by range tiles: hist.cu, and pack.cu for the inputs its packed
// counters cannot hold.
#pragma once

#include "rtcdf_internal.h"

namespace rtcdf {

// FIXED: not the first launch of a sort, so that the input does not change while the
// kernel is resident.
template <bool STREAMING, bool FIXED = false>
__device__ __forceinline__ int4 load_vec(const int4 *p) {
    if (STREAMING) return __ldcs(p);  // read once: evict first
    if (FIXED) return __ldg(p);       // re-read by the other tiles' CTAs: keep in L2
    return __ldcg(p);
}

// S[y] += 1 when y < w, as a predicated shared-memory reduction (no branch).
// No "memory" clobber: S is only otherwise touched on the far side of a
// __syncthreads(), and the clobber would stop the next loads from being
// scheduled early.
__device__ __forceinline__ void count_key(uint32_t s_base, uint32_t y, uint32_t w) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.lt.u32 p, %0, %1;\n\t"
        "@p red.shared.add.u32 [%2], 1;\n\t}"
        ::"r"(y), "r"(w), "r"(s_base + 4u * y));
}

// S[min(y, w)] += 1: a key outside the tile adds to the trash word S[w]
// instead of being predicated off; all such lanes of a warp hit one address
// with an immediate increment and are combined.
__device__ __forceinline__ void count_key_trash(uint32_t s_base, uint32_t y, uint32_t w) {
    const uint32_t yy = y < w ? y : w;
    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(s_base + 4u * yy));
}

__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// ADAPT (2 to 8 tiles): out-of-tile keys go to a trash word, and the m CTAs
// that read the same vectors prefetch them into L2 two iterations ahead --
// unless the input is long (more than 2^28 keys) and a sample of it (one
// vector per warp) shows one tile holding more than 2/m of the keys without
// holding nearly all of them: the CTAs of such tiles then run at unequal
// speeds, over a long input the heavy tile's CTAs fall so far behind that
// the lines prefetched for them are gone, and the prefetches cost more than
// they save (n = 1e9, R = 2^18, normal keys: 3.04 ms with them against 2.93
// without; n = 1e8: 0.312 against 0.322 ms, measured).  The choice changes
// only the speed, never the counts.
// CTA `cta` of m * g: tile cta mod m, the (cta / m)-th of the tile's g CTAs.  S is
// the tile's shared memory (the tile, and the trash word if ADAPT), s_tc eight
// words of it.
template <bool STREAMING, int UNROLL, bool ADAPT, bool PIPE = ADAPT, bool FIXED = false>
__device__ __forceinline__ void hist_tiles(const HistArgs &a, uint32_t cta, uint32_t *S, uint32_t *s_tc) {
    const uint32_t t = cta % a.m;
    const uint32_t q = cta / a.m;
    const uint32_t b = t * a.T;
    const uint32_t w = min(a.T, a.R - b);
    const int tid = threadIdx.x, nt = blockDim.x;

    for (uint32_t i = tid; i < w + (ADAPT ? 1u : 0u); i += nt) S[i] = 0;  // + the trash word
    if (ADAPT && tid < 8) s_tc[tid] = 0;
    __syncthreads();
    // The kernels before are done (launch_first).  Before anything else: the scan
    // launched after this kernel relies on every CTA here having waited (scan.cu).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (FIXED && a.only_if && __ldcg(a.only_if) == 0) return;

    const uint32_t base = a.min_u + b;  // key - base = position inside the tile
    const uint32_t s_base = (uint32_t)__cvta_generic_to_shared(S);

    // Grid-stride over 16-byte vectors: the g CTAs of a tile sweep the input
    // together, and the CTAs of the other tiles with the same q read the same
    // addresses at the same time (served from L2 after the first).
    const int4 *vin = reinterpret_cast<const int4 *>(a.in + a.head);
    const uint64_t stride = (uint64_t)a.g * nt;
    const uint64_t nvec = a.nvec;
    uint64_t v = (uint64_t)q * nt + tid;
    bool pf = false;
    if (ADAPT) {
        if ((tid & 31) == 0 && v < nvec) {
            const int4 k = __ldcg(vin + v);
            const uint32_t y[4] = {(uint32_t)k.x - a.min_u, (uint32_t)k.y - a.min_u,
                                   (uint32_t)k.z - a.min_u, (uint32_t)k.w - a.min_u};
#pragma unroll
            for (int e = 0; e < 4; e++)
                if (y[e] < a.R) atomicAdd(&s_tc[min(y[e] / a.T, 7u)], 1u);
        }
        __syncthreads();
        uint32_t tot = 0, mx = 0;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            tot += s_tc[i];
            mx = max(mx, s_tc[i]);
        }
        pf = tot > 0 && (a.nvec <= (1ull << 26) || mx * a.m <= 2 * tot || mx * 10 >= 9 * tot);
    }
    uint64_t vb = (uint64_t)q * nt;  // thread 0's vector of the iteration
    auto count_vec = [&](const int4 k) {
        if (ADAPT) {
            count_key_trash(s_base, (uint32_t)k.x - base, w);
            count_key_trash(s_base, (uint32_t)k.y - base, w);
            count_key_trash(s_base, (uint32_t)k.z - base, w);
            count_key_trash(s_base, (uint32_t)k.w - base, w);
        } else {
            count_key(s_base, (uint32_t)k.x - base, w);
            count_key(s_base, (uint32_t)k.y - base, w);
            count_key(s_base, (uint32_t)k.z - base, w);
            count_key(s_base, (uint32_t)k.w - base, w);
        }
    };
    if (!PIPE) {
        // One tile: UNROLL vectors loaded, then counted (32 registers, so
        // that two CTAs fit an SM: with the pipeline below these CTAs took 64
        // registers and the 12-array step on three streams got slower).
        for (; v + (UNROLL - 1) * stride < nvec; v += UNROLL * stride) {
            int4 k[UNROLL];
#pragma unroll
            for (int u = 0; u < UNROLL; u++) k[u] = load_vec<STREAMING, FIXED>(vin + v + u * stride);
#pragma unroll
            for (int u = 0; u < UNROLL; u++) count_vec(k[u]);
        }
    } else {
        // Several tiles (one CTA per SM, its shared memory being the tile), or a
        // long input over one tile (hist_long_kernel):
        // software pipelined, the next P vectors in flight while the last P
        // are counted (R = 2^18 uniform, n = 1e8: 0.272 against 0.281 ms per
        // sort, measured).
        constexpr int P = UNROLL < 6 ? UNROLL : 6;
        if (v + (P - 1) * stride < nvec) {
            int4 kn[P];
#pragma unroll
            for (int u = 0; u < P; u++) kn[u] = load_vec<STREAMING, FIXED>(vin + v + u * stride);
            v += P * stride;
            vb += P * stride;
            for (; v + (P - 1) * stride < nvec; v += P * stride, vb += P * stride) {
                if (pf && tid == 0) {
                    // This CTA's share (u = t, t + m, ...) of the vectors its
                    // group loads two stages from now.
                    const uint64_t ahead = vb + 2ull * P * stride;
                    for (uint32_t u = t; u < (uint32_t)P; u += a.m) {
                        const uint64_t s0 = ahead + (uint64_t)u * stride;
                        if (s0 + nt <= nvec) prefetch_l2(vin + s0, 16u * nt);
                    }
                }
                int4 kc[P];
#pragma unroll
                for (int u = 0; u < P; u++) kc[u] = kn[u];
#pragma unroll
                for (int u = 0; u < P; u++) kn[u] = load_vec<STREAMING, FIXED>(vin + v + u * stride);
#pragma unroll
                for (int u = 0; u < P; u++) count_vec(kc[u]);
            }
#pragma unroll
            for (int u = 0; u < P; u++) count_vec(kn[u]);
        }
    }
    for (; v < nvec; v += stride) {
        int4 k0 = load_vec<STREAMING, FIXED>(vin + v);
        count_key(s_base, (uint32_t)k0.x - base, w);
        count_key(s_base, (uint32_t)k0.y - base, w);
        count_key(s_base, (uint32_t)k0.z - base, w);
        count_key(s_base, (uint32_t)k0.w - base, w);
    }
    if (q == 0) {
        // Unaligned head and ragged tail, scalar.
        if ((uint32_t)tid < a.head) count_key(s_base, (uint32_t)a.in[tid] - base, w);
        for (uint64_t i = a.head + 4 * nvec + tid; i < a.n; i += nt)
            count_key(s_base, (uint32_t)a.in[i] - base, w);
    }
    // The scan may be scheduled now; it waits for this grid to finish before
    // reading H.
    asm volatile("griddepcontrol.launch_dependents;");

    __syncthreads();
    uint32_t *H = a.H + b;
    for (uint32_t i = tid; i < w; i += nt) {
        uint32_t c = S[i];
        if (c) atomicAdd(&H[i], c);
    }
}


}  // namespace rtcdf
