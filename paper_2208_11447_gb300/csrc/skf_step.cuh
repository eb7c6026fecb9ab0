// Device helpers shared by the Arnoldi step kernels (FP64 and reduced-precision
// variants): exact and fixed-order cross-CTA reductions, the arrival ticket and
// the sparse-sign pattern load.
#pragma once

#include "skf_internal.cuh"

namespace skf {

constexpr int kNoExp = -100000;

// Exact sum of G int64 partials by one warp (lanes strided over G, 128-bit
// butterfly); every lane returns the same double.
__device__ __forceinline__ double warp_sum_i64_exact(const long long *p, int G, size_t stride) {
    const int lane = threadIdx.x & 31;
    unsigned long long lo = 0;
    long long hi = 0;
    for (int g = lane; g < G; g += 32) {
        const long long v = __ldcg(p + (size_t)g * stride);
        const unsigned long long nlo = lo + (unsigned long long)v;
        hi += (v < 0 ? -1 : 0) + (nlo < lo ? 1 : 0);
        lo = nlo;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long olo = __shfl_xor_sync(0xffffffffu, lo, o);
        const long long ohi = __shfl_xor_sync(0xffffffffu, hi, o);
        const unsigned long long nlo = lo + olo;
        hi += ohi + (nlo < lo ? 1 : 0);
        lo = nlo;
    }
    const bool neg = hi < 0;
    unsigned long long uhi = (unsigned long long)hi;
    if (neg) {
        lo = ~lo + 1ull;
        uhi = ~uhi + (lo == 0ull ? 1ull : 0ull);
    }
    const double r = (double)uhi * 18446744073709551616.0 + (double)lo;
    return neg ? -r : r;
}

// Fixed-order reduction of G partials by one warp (sum or max).
__device__ __forceinline__ double warp_reduce_partials(const double *p, int G, int stride, bool is_max) {
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
    for (int g = lane; g < G; g += 32) {
        const double v = __ldcg(p + (size_t)g * stride);
        acc = is_max ? fmax(acc, v) : acc + v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double t = __shfl_xor_sync(0xffffffffu, acc, o);
        acc = is_max ? fmax(acc, t) : acc + t;
    }
    return acc;
}

// The zeta pattern entries of column r (one 16-byte load for zeta = 8).
template <int ZCAP>
__device__ __forceinline__ void load_pattern(const uint16_t *pattern, int zeta, int64_t r, uint16_t (&e)[ZCAP]) {
    if (ZCAP == 8 && zeta == 8) {
        const uint4 v = __ldg((const uint4 *)(pattern + r * 8));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) e[q] = (uint16_t)(w[q >> 1] >> (16 * (q & 1)));
    } else {
#pragma unroll
        for (int q = 0; q < ZCAP; ++q) e[q] = q < zeta ? __ldg(pattern + r * zeta + q) : (uint16_t)0;
    }
}

// Sketch of one value of a row with the compact pattern (zeta = 8): its limbs
// into bins laid out [limb][stripe][sign][BLK] in 1 << LC copies (copy index in
// the low bits, the caller's lane in `base`, a shared-memory address), so that a
// pattern byte is a bin offset and everything else an immediate: four
// instructions per nonzero.  The kernels that scatter are bound by instruction
// issue or by these atomics, not by memory.
template <int OFF>
__device__ __forceinline__ void red_shared(unsigned addr, int v) {
    asm volatile("red.shared.add.s32 [%0+%2], %1;" ::"r"(addr), "r"(v), "n"(OFF) : "memory");
}
template <int BLK, int LC, int Q = 0>
__device__ __forceinline__ void scatter8(uint2 pv, unsigned base, int l0, int l1) {
    if constexpr (Q < 8) {
        const unsigned e = __byte_perm(Q < 4 ? pv.x : pv.y, 0u, 0x4440u + (Q & 3));
        const unsigned a = base + (e << (LC + 2));
        red_shared<(Q * 2 * BLK) << (LC + 2)>(a, l0);
        red_shared<((Q * 2 + 16) * BLK) << (LC + 2)>(a, l1);
        scatter8<BLK, LC, Q + 1>(pv, base, l0, l1);
    }
}
// The same with the copies of both limbs side by side: a bin is 2 << LC words
// [limb][copy], and of two lanes that share a copy of their limb's words one
// adds limb 0 first and the other limb 1 (a1, v1 first, then a2, v2: see
// PairedLane).  With LC = 4 a warp's 32 adds fall into 32 banks whatever the
// rows; with the limbs in separate arrays two lanes shared each bank (reduced-
// precision update at N = 16.8M, from the solves: 87 -> 79 us).  One instruction
// more per nonzero: with fewer copies, where lanes still collide, it is the slower
// form (sketch apply, 4 copies: 226 -> 280 us).
template <int BLK, int LC, int Q = 0>
__device__ __forceinline__ void scatter8_paired(uint2 pv, unsigned a1, unsigned a2, int v1, int v2) {
    if constexpr (Q < 8) {
        const unsigned e = __byte_perm(Q < 4 ? pv.x : pv.y, 0u, 0x4440u + (Q & 3)) << (LC + 3);
        red_shared<(Q * 2 * BLK) << (LC + 3)>(a1 + e, v1);
        red_shared<(Q * 2 * BLK) << (LC + 3)>(a2 + e, v2);
        scatter8_paired<BLK, LC, Q + 1>(pv, a1, a2, v1, v2);
    }
}
// one limb only
template <int BLK, int LC, int Q = 0>
__device__ __forceinline__ void scatter8_one(uint2 pv, unsigned base, int l0) {
    if constexpr (Q < 8) {
        const unsigned e = __byte_perm(Q < 4 ? pv.x : pv.y, 0u, 0x4440u + (Q & 3));
        red_shared<(Q * 2 * BLK) << (LC + 2)>(base + (e << (LC + 2)), l0);
        scatter8_one<BLK, LC, Q + 1>(pv, base, l0);
    }
}
__device__ __forceinline__ unsigned shared_address(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
// A lane's place in paired bins of 1 << LC copies.
template <int LC> struct PairedLane {
    unsigned a1, a2;
    bool swap;   // limb 1 first
    __device__ __forceinline__ PairedLane(const void *bins, int lane) {
        constexpr unsigned C = 1u << LC;
        swap = ((unsigned)lane & C) != 0u;
        const unsigned a = shared_address(bins) + 4u * ((unsigned)lane & (C - 1u));
        a1 = a + (swap ? 4u * C : 0u);
        a2 = a + (swap ? 0u : 4u * C);
    }
};
// Limb sums (positive minus negative bin) of a row of S from paired bins, by one
// warp; exact in 32 bits, since all contributions of the row fit together.
template <int LC>
__device__ __forceinline__ void paired_sums(const int *bins, int pos, int neg, int &v0, int &v1) {
    constexpr int C = 1 << LC;
    const int lane = threadIdx.x & 31;
    int v = lane < 2 * C ? bins[(pos << (LC + 1)) + lane] - bins[(neg << (LC + 1)) + lane] : 0;
#pragma unroll
    for (int o = C / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    v0 = __shfl_sync(0xffffffffu, v, 0);
    v1 = __shfl_sync(0xffffffffu, v, C);
}

// Arrival ticket: true in exactly one CTA, the last to finish its partials.
__device__ __forceinline__ bool last_to_arrive(unsigned *cnt) {
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(cnt, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Offset of basis column j in V: column-major with leading dimension ldv,
// or, when the basis is kept as a ring of vring slots (two-pass mode, only
// the columns the recurrence still reads are alive), slot j mod vring.
template <class Ctx>
__host__ __device__ __forceinline__ size_t vcol(const Ctx &c, int j) {
    return (size_t)(c.vring ? j % c.vring : j) * (size_t)c.ldv;
}

// Host: the window columns i0 .. j of step j (i0 = max(0, j - k + 1)) as
// element offsets into V, in the launch's copy of the context.
template <class Ctx>
inline void window_offsets(Ctx &c, int j) {
    const int i0 = j - c.k + 1 > 0 ? j - c.k + 1 : 0;
    for (int a = 0; a < kMaxK; ++a) {
        const int col = i0 + a <= j ? i0 + a : j;
        c.woff[a] = (int64_t)(c.vring ? col % c.vring : col) * c.ldv;
    }
}

}  // namespace skf
