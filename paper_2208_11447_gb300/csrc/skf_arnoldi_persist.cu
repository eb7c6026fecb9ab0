// Persistent single-launch form of the k-truncated Arnoldi process
// (Algorithm 2, Sec. 2.2) for sparse-sign sketches, with an FP64 basis or
// (k <= 2) an FP32 one: the kernel is instantiated on the value type T of the
// operator, the basis and the on-chip rows; with T = float the SpMV, the
// update and the per-thread sums run in FP32 (block and grid sums, scalars,
// sketches and H stay FP64), and the update applies the FP32 values of sigma_j
// and of its coefficients, which H and the relation for S A v_j then use.
//
// The whole recurrence (all m steps) runs in one cooperative launch of one
// CTA per SM at most (of a small problem two launches fit side by side, see
// kShortRows).  CTA g owns R consecutive rows (whole SELL-32 slices) and keeps
// its rows of the k window vectors w_{j-k+1} .. w_j and of y~ = A w_j in
// shared memory for the whole process.  Per step HBM therefore sees the
// operator, the gathered entries of w_j and the store of w_{j+1}: the window
// is never re-read and y~ never leaves the SM.  A step has two phases, each
// closed by a grid-wide barrier:
//   A  y~ = A w_j on the CTA's rows (gathers from V[:, j]), partial window
//      dots <w_i, y~> and max|y~|;
//   B  MGS coefficients from the reduced dots and the window Gram matrix
//      (identical to MGS in exact arithmetic), w_{j+1} = sigma_j y~ -
//      sum_i h_ij sigma_i w_i, partial ||w_{j+1}||^2, Gram entries of the
//      next window and max|w_{j+1}|; exact fixed-point sketch of w_j.
// Storage is that of the two-kernel path: column j of V holds w_j, a
// positive multiple of v_j, and vscale[j] = 1 / ||w_j||.  When the rows of the
// window and of y~ do not fit in shared memory together but the window does
// (FP64, k <= 2), y~ lives in a global array instead, written in phase A and
// read back in phase B by the same CTA (L2-resident).
//
// S A v_j is not scattered row by row.  The update of step j applied
//   w_{j+1} = sigma_j y~_j - sum_i c_i w_i,
// so S A v_j = sigma_j S y~_j = S w_{j+1} + sum_i c_i S w_i, the sketched
// Arnoldi relation S A V_m = S V_{m+1} H, evaluated with the very
// coefficients c_i the update used.  It differs from a direct sketch of
// A v_j only by the sketch of the update's own rounding (about one unit
// roundoff of ||A v_j||).  The last column (and the column at a happy
// breakdown, where no further vector is formed) is sketched directly.
//
// Cross-CTA sums: integer sums of the dots and sketch partials, added with
// 64-bit global atomics (the order does not matter; see flush_sums).  Every
// barrier wait is bounded by a clock64 budget: past it the kernel records
// SKF_ERR_TIMEOUT, and every CTA returns at its next barrier.
#include <math.h>

#include <algorithm>

#include "skf_internal.cuh"
#include "skf_step.cuh"

namespace skf {

namespace {

constexpr int kPT = 512;                      // threads per CTA
constexpr int kPNW = kPT / 32;                // warps per CTA
// Rows per CTA below which CTAs are left out.  Alone, 10^4 rows take 12.4 / 9.6 /
// 9.6 us per step at 512 / 256 / 128 rows, 25600 rows 13.7 / 10.6 / 10.9 us.  The
// solves of a batch on three or more lanes share the card: they take the first
// level at which those of all lanes leave a quarter of it (at two CTAs per SM) to
// each other's tails, else the last.  16 solves with m = 40, ms per batch with
// 1024 rows and one CTA per SM / 256 rows and one CTA per SM / the levels: 1e4 rows
// on 8 lanes 2.56 / 3.02 / 2.16, 25600 on 4 lanes 4.43 / 6.90 / 4.00 and on 8 3.13 /
// 6.97 / 2.73, 4e4 on 8 4.39 / 7.46 / 3.69, four operators of 1e4 to 1e5 rows on 8
// 4.90 / 7.00 / 3.91.
constexpr int kPersistMinRows[kPersistLevels] = {256, 384, 768};
// Rows per CTA up to which a partition takes the short form of the kernel: two
// CTAs per SM (64 registers; a warp has at most three slices, so nothing is
// loaded ahead), and sums that do not depend on the partition (a summand is a
// lane's share of one or two slices, see persist_group), so that a solve gives the
// same bits alone and in a batch.
constexpr int kShortRows = 1024;
constexpr int kFlushAll = 64;                 // slices per CTA up to which all warps add up the sketch bins
constexpr long long kBarrierBudget = 1ll << 31;   // SM cycles (about one second)

struct PCtx {
    int64_t n;
    int R;                     // rows per CTA (multiple of 32)
    const int64_t *sell_off;
    const int32_t *sell_w;
    const void *sell_val;      // T values (T = double, or float for an FP32 basis)
    const int32_t *sell_col;
    DiagOp dg;                 // diagonal copy of the operator (dg.w = W, or 0: none)
    int group;                 // (short form) slices per summand of the grid sums, 1 or 2 (persist_group)
    float l2_frac;             // share of the operator's lines kept in L2 from step to step (not with y~ in global memory)
    SparseSign sp;
    const uint16_t *pattern;   // [n][zeta]
    const uint8_t *pattern8;   // [n][8] or nullptr
    int p8_block;
    int L, frac;               // fixed-point limb width and fraction bits (sketch)
    double sk_scale;           // 1 / sqrt(zeta)
    int m, k;
    const double *b;
    void *V;                   // T [m][ldv]
    int64_t ldv;
    double *vscale, *SV, *SAV, *H;
    int *iscal;
    double *pB;                // [2][G]: partial ||b||^2, max|b| (short form: [2][slices])
    unsigned long long *slot;  // [3 m + 1][kSlot]: exact sums of the window dots and max|y~| of step j at
                               // 2 j, of ||w_j||^2, the Gram entries and max|w_j| at 2 j - 1 (see push_sums),
                               // of the dots below a tighter bound at 2 m + 1 + j
    int e_row;                 // |(A x)_r| < 2^e_row max|x|
    unsigned long long *accw;  // [m][2][s]: limb sums of S w_j
    unsigned long long *accy;  // [2][s]: limb sums of the directly sketched y~
    double *Sw;                // s x m: S w_j (unnormalised)
    void *ysg;                 // T y~ in global memory ([G][R]) when the rows do not fit with it on chip
    unsigned *bar;             // barrier arrival counter (zeroed before launch)
    int *flag;                 // 1 once a barrier wait ran out
    long long budget;
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int ld_volatile_i32(const int *p) {
    return *(const volatile int *)p;
}

// Operator loads.  A is read once per step by the same CTA, so what decides is
// whether it stays in L2 (129 MB) from one step to the next: `pol` keeps the
// fraction l2_frac of its lines (evict_last) and streams the rest
// (evict_first), so that an operator beyond the budget still finds that
// fraction there instead of evicting itself.  A fraction lies in (0, 1]; an
// operator of which nothing is kept (KEEP false) is streamed by a policy of its own.
template <bool KEEP>
__device__ __forceinline__ unsigned long long operator_policy(float frac) {
    unsigned long long p;
    if constexpr (KEEP)
        asm("createpolicy.fractional.L2::evict_last.L2::evict_first.b64 %0, %1;" : "=l"(p) : "f"(frac));
    else
        asm("createpolicy.fractional.L2::evict_first.b64 %0, 0f3F800000;" : "=l"(p));
    return p;
}
__device__ __forceinline__ double ld_op(const double *a, unsigned long long pol) {
    double v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(a), "l"(pol));
    return v;
}
__device__ __forceinline__ float ld_op(const float *a, unsigned long long pol) {
    float v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(a), "l"(pol));
    return v;
}
__device__ __forceinline__ int ld_op(const int32_t *a, unsigned long long pol) {
    int v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(v) : "l"(a), "l"(pol));
    return v;
}

// Wait (one thread) until *cnt reaches target; 0 if the wait ran out of budget
// or another CTA's did, and then *flag is set.
__device__ __forceinline__ int spin_until(const unsigned *cnt, unsigned target, int *flag, long long budget) {
    const long long t0 = clock64();
    while (ld_acquire_u32(cnt) < target) {
        if (ld_volatile_i32(flag) != 0 || clock64() - t0 > budget) {
            atomicExch(flag, 1);
            return 0;
        }
    }
    return 1;
}

// Grid-wide barrier number `nb` (1, 2, ...) of a co-resident grid: arrive,
// then wait until nb * gridDim.x arrivals are visible.  Returns false (in
// every thread of the CTA) if the wait ran out of budget or another CTA's
// did; the first CTA to give up sets *flag.  The arrival is a release and the
// poll an acquire at GPU scope, and the block barriers on both sides extend
// them to the whole CTA (cumulativity), so no further fence is needed; a
// __threadfence() on each side cost 0.3 us per barrier (1.34 -> 1.12 us with
// 10 CTAs, 2.45 -> 2.14 us with 152) and made the reduction before it wait
// for the service warp's sketch atomics (5.5 -> 3.5 us at s = 960).
__device__ __forceinline__ void grid_arrive(unsigned *bar) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}
__device__ bool grid_barrier(unsigned *bar, int *flag, unsigned nb, long long budget) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        grid_arrive(bar);
        ok = spin_until(bar, nb * gridDim.x, flag, budget);   // one thread per CTA polls one L2 line
    }
    __syncthreads();
    return ok != 0;
}

// Exact value of a * 2^L + b for int64 a, b (|a| 2^L < 2^94), rounded to
// double (two roundings at most, as warp_sum_i64_exact).
__device__ __forceinline__ double limbs_to_double(long long a1, long long a0, int L) {
    // 128-bit two's complement: hi:lo = a1 << L, then + a0
    unsigned long long lo = (unsigned long long)a1 << L;
    long long hi = (L == 0) ? (a1 < 0 ? -1 : 0) : (a1 >> (64 - L));
    const unsigned long long nlo = lo + (unsigned long long)a0;
    hi += (a0 < 0 ? -1 : 0) + (nlo < lo ? 1 : 0);
    lo = nlo;
    const bool neg = hi < 0;
    unsigned long long uhi = (unsigned long long)hi;
    if (neg) {
        lo = ~lo + 1ull;
        uhi = ~uhi + (lo == 0ull ? 1ull : 0ull);
    }
    const double r = (double)uhi * 18446744073709551616.0 + (double)lo;
    return neg ? -r : r;
}

constexpr int kMaxG = 160;   // partial-table rows one warp reduces with hoisted loads (G <= SMs)

// Sum (or max) of p[0 .. G) in a fixed order, by one warp: every lane loads
// its (at most five) entries at once, adds them in index order, then a
// butterfly; the result is returned to every lane.  The same order in every
// CTA, so all CTAs obtain bitwise the same total.
__device__ __forceinline__ double reduce_slot(const double *p, int G, bool is_max) {
    const int lane = threadIdx.x & 31;
    double v[kMaxG / 32];
#pragma unroll
    for (int i = 0; i < kMaxG / 32; ++i) v[i] = (lane + 32 * i < G) ? __ldcg(p + lane + 32 * i) : 0.0;
    double acc = v[0];
#pragma unroll
    for (int i = 1; i < kMaxG / 32; ++i) acc = is_max ? fmax(acc, v[i]) : acc + v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double t = __shfl_xor_sync(0xffffffffu, acc, o);
        acc = is_max ? fmax(acc, t) : acc + t;
    }
    return acc;
}

// Block sums of NV values (one per thread) and the block max of a magnitude
// key, delivered to thread 0.  The FP64 pipe of this part retires one warp
// instruction per 16 SM cycles whatever the active lanes, so the sums use
// full-width adds: values are parked in shared memory and four warps per
// value (one per SM sub-partition) add 128 of them each (4 per lane in index
// order, then a butterfly); thread 0 adds the four quarter sums in order.
// smem: NV * kPT + 4 * NV doubles + kPNW keys.
template <int NV>
__device__ __forceinline__ unsigned long long block_reduce_t0(double (&v)[NV], unsigned long long key, double *smem) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double *qs = smem + NV * kPT;
    unsigned long long *ks = (unsigned long long *)(qs + 4 * NV);
#pragma unroll
    for (int i = 0; i < NV; ++i) smem[i * kPT + tid] = v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
    if (lane == 0) ks[warp] = key;
    __syncthreads();
    if (warp < 4 * NV) {
        const double *p = smem + (warp >> 2) * kPT + (warp & 3) * 128 + lane;
        double a = ((p[0] + p[32]) + p[64]) + p[96];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) qs[warp] = a;
    }
    __syncthreads();
    if (tid == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = ((qs[4 * i] + qs[4 * i + 1]) + qs[4 * i + 2]) + qs[4 * i + 3];
        key = ks[0];
#pragma unroll
        for (int w = 1; w < kPNW; ++w) key = max(key, ks[w]);
    }
    return key;
}

// Grid-wide sums without floating-point additions.  The per-thread partials of
// a phase (window dots; ||w||^2 and Gram entries) are cut into kCh chunks of 22
// bits (short form: 21) of a field below an exponent bound that every CTA knows, and
// the chunks are added as integers: a warp reduction per chunk, a shared
// atomic per warp, one 64-bit global atomic per CTA and chunk, issued just
// before the CTA's barrier arrival.  Integer sums do not depend on the order,
// so after the barrier one 7-word load replaces the read and fixed-order sum
// of G partials, and no FP64 addition (65 dependent cycles each on this part,
// 16 more of the SM's FP64 pipe) is left on the path from the last row to the
// coefficients.  A partial is cut off 2^-154 (2^-147) below its bound and the sum
// 2^-132 (2^-126) below it (pull_sums carries the lowest chunk and drops the rest).  The bound of
// the dots holds ||A||_inf, which one row can set far above the y~ of the others:
// where it lies more than kMaxSlack bits above max|y~|, known after the barrier,
// the dots are summed once more below that.  Measured per step
// from the last row to the coefficients: 7.3 -> 5.9 us (100^3 grid, 152 CTAs),
// 7.0 -> 4.2 us (10^4 rows; 10 -> 40 CTAs).
// The short form has up to kShortRows summands per CTA: 21-bit chunks there, so
// that a CTA's sum stays below 2^31.
constexpr int kCh = 7;                                   // chunks of a sum
constexpr int chunk_bits(bool sh) { return sh ? 21 : 22; }
constexpr int kMaxSlack = 54;                // bits by which the bound of the dots may lie above max|w_i| max|y~|
constexpr int kSlot = 32;                    // words of a slot: kCh per sum (at most 4), [30] not finite, [31] max key

// x as signed chunks of CB bits of x / 2^(E - kCh CB); false if x is not finite
// or not below 2^E in magnitude.
template <int CB>
__device__ __forceinline__ bool chunks_of(double x, int E, int (&ch)[kCh]) {
    constexpr int kField = kCh * CB;
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int be = (int)((bits >> 52) & 0x7FFull);
    const unsigned long long frac = bits & 0xFFFFFFFFFFFFFull, mant = be ? frac | 0x10000000000000ull : frac;
    const int p = max(be, 1) - 1075 - (E - kField);   // position of the mantissa's lowest bit in the field
    const bool ok = be != 0x7FF && (mant == 0ull || p + 64 - __clzll((long long)mant) <= kField);
    const bool neg = (bits >> 63) != 0ull;
#pragma unroll
    for (int i = 0; i < kCh; ++i) {
        const int sh = CB * i - p;
        unsigned long long v;
        asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(mant), "r"(max(sh, 0)));   // shifts of 64 and more give 0
        asm("shl.b64 %0, %1, %2;" : "=l"(v) : "l"(v), "r"(max(-sh, 0)));
        const int d = (int)((unsigned)v & ((1u << CB) - 1u));
        ch[i] = ok ? (neg ? -d : d) : 0;
    }
    return ok;
}
template <int CB>
__device__ __forceinline__ bool chunks_of(float x, int E, int (&ch)[kCh]) {
    constexpr int kField = kCh * CB;
    const unsigned bits = __float_as_uint(x);
    const int be = (int)((bits >> 23) & 0xFFu);
    const unsigned frac = bits & 0x7FFFFFu, mant = be ? frac | 0x800000u : frac;
    const int p = max(be, 1) - 150 - (E - kField);
    const bool ok = be != 0xFF && (mant == 0u || p + 32 - __clz((int)mant) <= kField);
    const bool neg = (bits >> 31) != 0u;
#pragma unroll
    for (int i = 0; i < kCh; ++i) {
        const int sh = CB * i - p;
        unsigned v;
        asm("shr.u32 %0, %1, %2;" : "=r"(v) : "r"(mant), "r"(max(sh, 0)));
        asm("shl.b32 %0, %1, %2;" : "=r"(v) : "r"(v), "r"(max(-sh, 0)));
        const int d = (int)(v & ((1u << CB) - 1u));
        ch[i] = ok ? (neg ? -d : d) : 0;
    }
    return ok;
}

// Magnitudes as ordered 32-bit keys (the high word of a double), and the
// exponent bound |x| < 2^E of the largest: only its exponent is needed.
__device__ __forceinline__ unsigned mag_key(double x) {
    return (unsigned)((unsigned long long)__double_as_longlong(x) >> 32) & 0x7FFFFFFFu;
}
__device__ __forceinline__ unsigned mag_key(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }
template <typename T>
__device__ __forceinline__ int key_exponent(unsigned key) {
    constexpr bool F32 = sizeof(T) == 4;
    const int be = (int)(key >> (F32 ? 23 : 20));
    if (key == 0u || be == (F32 ? 0xFF : 0x7FF)) return kNoExp;   // zero (or below 2^-1042), or not finite
    return max(be, 1) - (F32 ? 126 : 1022);
}
// E with |x| < 2^E (x finite)
__device__ __forceinline__ int exponent_above(double x) {
    return (int)(mag_key(x) >> 20) - 1022;
}

// One value of every thread of the warp (|v| < 2^E) into value a's chunk sums:
// lane a kCh + i holds the warp's sum of chunk i in `mine`, `bad` a value that
// is not finite.
template <int CB, typename T>
__device__ __forceinline__ void add_chunks(T v, int E, int a, int &mine, bool &bad) {
    const int lane = threadIdx.x & 31;
    int ch[kCh];
    bad |= !chunks_of<CB>(v, E, ch);
#pragma unroll
    for (int i = 0; i < kCh; ++i) {
        const int t = __reduce_add_sync(0xffffffffu, ch[i]);   // |t| < 2^(CB + 5)
        if (lane == a * kCh + i) mine += t;
    }
}

// Adds the warps' chunk sums of nv values and the maximum of the keys to this
// CTA's share of `slot`: shared atomics (at most 2^(31 - CB) summands per CTA),
// then one global atomic per chunk from warp 0, whose lane 0 may arrive at the
// barrier after a __syncwarp().  sch: kSlot ints, zero on entry and left zero.
__device__ __forceinline__ void flush_sums(int mine, bool bad, int nv, unsigned key, int *sch,
                                           unsigned long long *slot) {
    const int lane = threadIdx.x & 31;
    key = __reduce_max_sync(0xffffffffu, key);
    bad = __any_sync(0xffffffffu, bad);
    if (lane < nv * kCh) atomicAdd(sch + lane, mine);
    if (lane == 30 && bad) sch[30] = 1;
    if (lane == 31) atomicMax((unsigned *)sch + 31, key);
    __syncthreads();
    if (threadIdx.x < 32) {
        const int t = sch[lane];
        if (lane < nv * kCh || (lane == 30 && t != 0))
            atomicAdd(slot + lane, (unsigned long long)(long long)t);
        if (lane == 31) atomicMax(slot + lane, (unsigned long long)(unsigned)t);
        sch[lane] = 0;
    }
}

// The first nv of the per-thread values v[] (|v[i]| < 2^E[i]).
template <int CB, int KW, typename T>
__device__ __forceinline__ void push_sums(const T (&v)[KW], int nv, const int *E, unsigned key, int *sch,
                                          unsigned long long *slot) {
    int mine = 0;
    bool bad = false;
#pragma unroll
    for (int a = 0; a < KW; ++a)
        if (a < nv) add_chunks<CB>(v[a], E[a], a, mine, bad);
    flush_sums(mine, bad, nv, key, sch, slot);
}

// The sums of a slot (after the barrier): lane i < nv returns value i (carries
// from the lowest chunk up, then the digits as three integers and two FMAs;
// NaN when a partial was not finite), every lane the slot's maximum key.  One
// load per chunk and lane: a single coalesced load of the slot and shuffles
// took 3.4 instead of 1.8 us with 152 CTAs reading it (1.9 / 1.3 with 40).
template <int CB>
__device__ __forceinline__ double pull_sums(const unsigned long long *slot, int nv, const int *E, unsigned &key) {
    const int lane = threadIdx.x & 31;
    const unsigned long long *p = slot + (lane < nv ? lane : 0) * kCh;
    long long t[kCh];
#pragma unroll
    for (int q = 0; q < kCh; ++q) t[q] = (long long)__ldcg(p + q);
    key = (unsigned)__ldcg(slot + 31);
    const bool bad = __ldcg(slot + 30) != 0ull;
    if (lane >= nv) return 0.0;
    constexpr long long mask = (1ll << CB) - 1;
#pragma unroll
    for (int q = 0; q + 1 < kCh; ++q) {
        t[q + 1] += t[q] >> CB;
        t[q] &= mask;
    }
    const long long hi = t[6] * (1ll << CB) + t[5];
    const long long mid = (t[4] << CB) | t[3], lo = (t[2] << CB) | t[1];
    constexpr double two = (double)(1ull << (2 * CB));
    const double r = fma(fma((double)hi, two, (double)mid), two, (double)lo);
    return bad ? __longlong_as_double(0x7FF8000000000000ll) : scale_pow2(r, E[lane] - (kCh - 1) * CB);
}

// Fixed-point limbs of one value into the shared bins of the sparse-sign
// rows of row r.  With the compact pattern (p8: one 8-byte entry per row,
// prefetched) the bins are laid out [stripe][sign][p8_block], so that a pattern
// byte is a bin offset and no sign has to be applied: 4 instructions per
// nonzero instead of 9 (the update is issue- and shared-atomic-bound beside its
// FP64 work; 100^3 grid: 10.5 -> 10.1 us in FP64, 8.8 -> 7.8 us in FP32).
template <int ZCAP>
__device__ __forceinline__ void scatter_row(const PCtx &c, int64_t r, uint2 pv, bool p8, int *b0, int *b1, int l0,
                                            int l1) {
    if (p8) {   // (b1 follows b0 by 16 p8_block bins)
        const unsigned base = shared_address(b0);
        if (c.p8_block == 64) scatter8<64, 0>(pv, base, l0, l1);
        else scatter8<128, 0>(pv, base, l0, l1);
    } else {
        uint16_t e[ZCAP];
        load_pattern<ZCAP>(c.pattern, c.sp.zeta, r, e);
#pragma unroll
        for (int q = 0; q < ZCAP; ++q) {
            if (q < c.sp.zeta) {
                int row;
                bool neg;
                pattern_entry(c.sp, e[q], q, row, neg);
                red_limbs(b0, b1, row, l0, l1, neg);
            }
        }
    }
}

// y~ = A w on this CTA's rows into ys[] by the kSpmvWarps SpMV warps, warp
// w taking slices w, w + kSpmvWarps, ... (a fixed assignment, so every lane
// accumulates the same rows in every run: the dot products are bitwise
// reproducible), with the window dots acc[a] = <w_{i0+a}, y~> (soff: slot
// offsets of the window in win[], nw of them) and the magnitude key of
// max|y~|.  Entries of one row are summed in their SELL (= CSR) order.
constexpr int kSpmvWarps = kPNW - 1;   // the last warp serves the reductions
template <int KW, int W, bool KEEP, bool SHORT, typename T>
__device__ __forceinline__ void spmv_rows(const PCtx &c, const T *__restrict__ wsrc, const T *win,
                                          const int (&soff)[KW], int nw, T *ys, const long long *meta_o,
                                          const int *meta_w, uint2 dmask, int nsl, int nr, T (&acc)[KW],
                                          unsigned &ykey) {
    const T *sell_val = (const T *)c.sell_val;
    const unsigned long long pol = operator_policy<KEEP>(c.l2_frac);
    const int lane = threadIdx.x & 31;
    int next_t = threadIdx.x >> 5;
    auto grab = [&]() {
        const int t = next_t;
        next_t += kSpmvWarps;
        return t;
    };
    if constexpr (SHORT) {   // y~ alone: the dots follow from shared memory
        for (int t = next_t; t < nsl; t += kSpmvWarps) {
            T y = T(0);
            if (W > 0 && c.dg.w != 0) {
                constexpr int WD = W > 0 ? W : 1;
                const int64_t r0 = (int64_t)blockIdx.x * c.R + 32 * t + lane;
                const unsigned m = t == next_t ? dmask.x : t == next_t + kSpmvWarps ? dmask.y
                                                                                   : (unsigned)__ldg(c.dg.mask + r0);
                const T *dv = (const T *)c.dg.val + (r0 - lane) * W + lane;
                const T *wr = wsrc + r0;
                T av[WD], xv[WD];
#pragma unroll
                for (int d = 0; d < W; ++d) {
                    av[d] = ld_op(dv + 32 * d, pol);
                    xv[d] = (m >> d) & 1u ? __ldcg(wr + c.dg.off[d]) : T(0);
                }
#pragma unroll
                for (int d = 0; d < W; ++d) y = fma(av[d], xv[d], y);
            } else {
                const int wt = meta_w[t];
                const T *pv = sell_val + meta_o[t] + lane;
                const int32_t *pc = c.sell_col + meta_o[t] + lane;
                if constexpr (W > 0) {
                    T av[W], xv[W];
                    int cv[W];
#pragma unroll
                    for (int p = 0; p < W; ++p) cv[p] = p < wt ? ld_op(pc + 32 * p, pol) : 0;
#pragma unroll
                    for (int p = 0; p < W; ++p) av[p] = p < wt ? ld_op(pv + 32 * p, pol) : T(0);
#pragma unroll
                    for (int p = 0; p < W; ++p) xv[p] = p < wt ? __ldcg(wsrc + cv[p]) : T(0);
#pragma unroll
                    for (int p = 0; p < W; ++p)
                        if (p < wt) y = fma(av[p], xv[p], y);
                } else {
                    for (int p = 0; p < wt; ++p)
                        y = fma(ld_op(pv + 32 * p, pol), __ldcg(wsrc + ld_op(pc + 32 * p, pol)), y);
                }
            }
            if (t * 32 + lane < nr) ys[t * 32 + lane] = y;
        }
        return;
    }
    if (W > 0 && c.dg.w != 0) {
        // diagonal copy: values and gathers of slice tn and the masks of slice
        // tnn in flight while slice t is computed (a row past nr is present in no
        // mask); the first two masks are the same in every step (dmask), so the
        // gathers start with the phase.  Per step, slices / this copy: 100^3 grid
        // FP64 37.0 / 34.5 us, FP32 25.1 / 23.6; 25600 rows 9.8 / 9.6; 10^4 rows
        // 9.9 / 10.0.  (A guard around the whole load instead of one per value: 35.8
        // and 25.2 us.)
        constexpr int WD = W > 0 ? W : 1;
        const int64_t r0 = (int64_t)blockIdx.x * c.R;
        const T *dv = (const T *)c.dg.val + r0 * W + lane;
        const T *wr = wsrc + r0 + lane;
        const uint8_t *mk = c.dg.mask + r0 + lane;
        struct Stage {
            T av[WD], xv[WD];
        };
        auto load = [&](int t, unsigned m, Stage &q) {
#pragma unroll
            for (int d = 0; d < W; ++d) {
                q.av[d] = t < nsl ? ld_op(dv + t * (32 * W) + 32 * d, pol) : T(0);
                q.xv[d] = (m >> d) & 1u ? __ldcg(wr + 32 * t + c.dg.off[d]) : T(0);
            }
        };
        auto mask_of = [&](int t) { return t < nsl ? (unsigned)__ldg(mk + 32 * t) : 0u; };
        Stage cur, nxt;
        int t = next_t;
        load(t, dmask.x, cur);
        unsigned mn = dmask.y;
        for (; t < nsl; t += kSpmvWarps) {
            load(t + kSpmvWarps, mn, nxt);
            mn = mask_of(t + 2 * kSpmvWarps);
            const int lr = t * 32 + lane;
            if (lr < nr) {
                T y = T(0);
#pragma unroll
                for (int d = 0; d < W; ++d) y = fma(cur.av[d], cur.xv[d], y);   // an absent entry adds 0
                ys[lr] = y;
#pragma unroll
                for (int a = 0; a < KW; ++a)
                    if (a < nw) acc[a] = fma(win[soff[a] + lr], y, acc[a]);
                ykey = max(ykey, mag_key(y));
            }
            cur = nxt;
        }
        return;
    }
    if constexpr (W > 0) {
        // three-stage pipeline: values and gathers of slice tn and column
        // indices of slice tnn are in flight while slice t is computed
        int t = grab();
        int wt = t < nsl ? meta_w[t] : 0;
        int cv[W];
        {
            const int32_t *pc = c.sell_col + (t < nsl ? meta_o[t] : 0) + lane;
#pragma unroll
            for (int p = 0; p < W; ++p) cv[p] = p < wt ? ld_op(pc + 32 * p, pol) : 0;
        }
        T av[W], xv[W];
        {
            const T *pv = sell_val + (t < nsl ? meta_o[t] : 0) + lane;
#pragma unroll
            for (int p = 0; p < W; ++p) {
                av[p] = p < wt ? ld_op(pv + 32 * p, pol) : T(0);
                xv[p] = p < wt ? __ldcg(wsrc + cv[p]) : T(0);
            }
        }
        int tn = t < nsl ? grab() : nsl;
        int wtn = tn < nsl ? meta_w[tn] : 0;
        int cvn[W];
        {
            const int32_t *pc = c.sell_col + (tn < nsl ? meta_o[tn] : 0) + lane;
#pragma unroll
            for (int p = 0; p < W; ++p) cvn[p] = p < wtn ? ld_op(pc + 32 * p, pol) : 0;
        }
        while (t < nsl) {
            T avn[W], xvn[W];
            {
                const T *pv = sell_val + (tn < nsl ? meta_o[tn] : 0) + lane;
#pragma unroll
                for (int p = 0; p < W; ++p) {
                    avn[p] = p < wtn ? ld_op(pv + 32 * p, pol) : T(0);
                    xvn[p] = p < wtn ? __ldcg(wsrc + cvn[p]) : T(0);
                }
            }
            const int tnn = tn < nsl ? grab() : nsl;
            const int wtnn = tnn < nsl ? meta_w[tnn] : 0;
            int cvnn[W];
            {
                const int32_t *pc = c.sell_col + (tnn < nsl ? meta_o[tnn] : 0) + lane;
#pragma unroll
                for (int p = 0; p < W; ++p) cvnn[p] = p < wtnn ? ld_op(pc + 32 * p, pol) : 0;
            }
            const int lr = t * 32 + lane;
            if (lr < nr) {
                T y = T(0);
#pragma unroll
                for (int p = 0; p < W; ++p)
                    if (p < wt) y = fma(av[p], xv[p], y);
                ys[lr] = y;
#pragma unroll
                for (int a = 0; a < KW; ++a)
                    if (a < nw) acc[a] = fma(win[soff[a] + lr], y, acc[a]);
                ykey = max(ykey, mag_key(y));
            }
            t = tn;
            wt = wtn;
            tn = tnn;
            wtn = wtnn;
#pragma unroll
            for (int p = 0; p < W; ++p) {
                av[p] = avn[p];
                xv[p] = xvn[p];
                cvn[p] = cvnn[p];
            }
        }
    } else {
        // slices wider than 8: one row per lane, entries in a loop
        for (int t = grab(); t < nsl; t = grab()) {
            const int lr = t * 32 + lane;
            const int wt = meta_w[t];
            const long long o = meta_o[t] + lane;
            T y = T(0);
            for (int p = 0; p < wt; ++p)
                y = fma(ld_op(sell_val + o + 32 * p, pol), __ldcg(wsrc + ld_op(c.sell_col + o + 32 * p, pol)), y);
            if (lr < nr) {
                ys[lr] = y;
#pragma unroll
                for (int a = 0; a < KW; ++a)
                    if (a < nw) acc[a] = fma(win[soff[a] + lr], y, acc[a]);
                ykey = max(ykey, mag_key(y));
            }
        }
    }
}

// T = double: the FP64 basis; T = float: an FP32 basis with FP32 SpMV,
// orthogonalisation and accumulation, the update applying the FP32 values of
// sigma_j and of the MGS coefficients (H and S A v_j are those of the relation
// with the applied values), everything else FP64.
template <int KW, int W, int ZCAP, bool YG, bool SHORT, typename T>
__global__ void __launch_bounds__(kPT, SHORT ? 2 : 1) k_arnoldi_persist(PCtx c) {
    constexpr bool F32 = sizeof(T) == 4;
    constexpr int CB = chunk_bits(SHORT);
    extern __shared__ __align__(16) unsigned char psm[];
    constexpr int kRed = kPT + 4 + kPNW;             // block_reduce_t0<1>
    constexpr int kSvc = kPNW - 1;                   // the service warp
    const int G = gridDim.x, g = blockIdx.x;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R = c.R, k = c.k, m = c.m, s = c.sp.s;
    const int64_t r0 = (int64_t)g * R;
    const int nr = (int)min((int64_t)R, c.n - r0);          // rows of this CTA (>= 1)
    const int nsl = (nr + 31) >> 5;                          // slices of this CTA
    T *win = (T *)psm;                                       // [k][R]: w_i at slot i % k
    T *Vb = (T *)c.V;
    // [R] y~ of this CTA's rows: shared memory, or (YG) this CTA's slice of a
    // global array, read back by the same CTA after a block barrier (L2)
    T *ys = YG ? (T *)c.ysg + r0 : win + (size_t)k * R;
    double *red = (double *)(YG ? win + (size_t)k * R : ys + R);   // block reductions (R: multiple of 32)
    long long *meta_o = (long long *)(red + kRed);           // [nsl] slice offsets
    int *meta_w = (int *)(meta_o + R / 32);                  // [nsl] slice widths
    const bool p8 = ZCAP == 8 && c.pattern8 != nullptr;
    const int nbin = p8 ? 16 * c.p8_block : s;               // bins of one limb
    int *bins = meta_w + R / 32;                             // [2][2][nbin]: limbs of S w_j in buffer j & 1
    const long long lmask = (1ll << c.L) - 1;

    // per-step scalars, in rings indexed by step & 3 (k <= 4)
    __shared__ double sig[4];                // sigma_i = 1 / ||w_i||
    __shared__ double sap[4];                // the sigma_i the update of step i applied (FP32: rounded)
    __shared__ double grm[4][kMaxK];         // grm[i & 3][d] = <w_i, w_{i-d}>
    __shared__ double coef[4][kMaxK];        // c_b for w_{i-b} (newest first) of the update of step i
    __shared__ int cnw[4];                   // window length of step i
    __shared__ int ews[4];                   // exponent bound of max|w_i| (its sketch)
    __shared__ int eys[4];                   // exponent bound of max|y~_i|
    __shared__ double sh[kMaxK];             // MGS coefficients h_ij of the current step
    __shared__ double sb[2];                 // reduced ||b||^2, max|b|
    __shared__ double fd[kMaxK], fg[KW][KW]; // MGS factors of the current step (phase A)
    __shared__ int ea[KW], eb[KW];           // exponent bounds of the per-thread sums of phases A and B
    __shared__ int sch[kSlot];               // this CTA's chunk sums (push_sums)
    __shared__ int bar_ok;                   // the last grid barrier was passed (2: the dots are to be summed again)
    __shared__ int sbreak;                   // w_j is a happy breakdown
    unsigned nb = 0;                         // barriers passed
    const int nh = max(0, kSpmvWarps - nsl); // SpMV warps without a slice
    // (short form) slices per group less one, and this thread's row at its turn q:
    // warp w takes the groups w, w + kPNW, ..., slice by slice
    const int gl = SHORT ? c.group - 1 : 0;
    auto row_of = [&](int q) { return ((((warp + kPNW * (q >> gl)) << gl) | (q & gl)) << 5) | lane; };
    const int lg_rows = SHORT ? gl : 32 - __clz(R / 256); // log2 of a bound of the products in one summand

    // Column i of S V and column i-1 of S A V from the integer sums of S w_i
    // (rows is = g + G t of S): S w_i, S v_i = sigma_i S w_i and, by the
    // relation, S A v_{i-1} = S w_i + sum_b c_b S w_{i-1-b}.
    auto finalize_col = [&](int i, int t) {
        const int is = g + G * t;
        if (is >= s) return;
        const unsigned long long *aw = c.accw + (size_t)i * 2 * s;
        const int ew = ews[i & 3];
        double swv = 0.0;
        if (ew != kNoExp)
            swv = scale_pow2(limbs_to_double((long long)__ldcg(aw + s + is), (long long)__ldcg(aw + is), c.L),
                             ew - c.frac) * c.sk_scale;
        c.Sw[is + (size_t)i * s] = swv;
        c.SV[is + (size_t)i * s] = sig[i & 3] * swv;
        if (i >= 1) {
            const int pn = cnw[(i - 1) & 3];
            double v = swv;
            for (int b2 = pn - 1; b2 >= 0; --b2)
                v = fma(coef[(i - 1) & 3][b2], __ldcg(c.Sw + is + (size_t)(i - 1 - b2) * s), v);
            // the update applied sap y~ (= sigma y~ in FP64): S A v = (sigma / sap) (...)
            if constexpr (F32) v *= sig[(i - 1) & 3] / sap[(i - 1) & 3];
            c.SAV[is + (size_t)(i - 1) * s] = v;
        }
    };
    // S A v_i sketched directly from y~_i (limb sums in accy)
    auto finalize_direct = [&](int i, int t) {
        const int is = g + G * t;
        if (is >= s) return;
        const int ey = eys[i & 3];
        double v = 0.0;
        if (ey != kNoExp)
            v = scale_pow2(limbs_to_double((long long)__ldcg(c.accy + s + is), (long long)__ldcg(c.accy + is), c.L),
                           ey - c.frac) * c.sk_scale * sig[i & 3];
        c.SAV[is + (size_t)i * s] = v;
    };
    // add this CTA's S w_i limb bins (buffer i & 1) to accw[i], then clear them
    // (split layout: x enumerates the bins of one sign, so that a warp stays within a stripe)
    auto flush_bins = [&](int buf, unsigned long long *aw, int t0, int dt) {
        int *b0 = bins + (buf & 1) * 2 * nbin, *b1 = b0 + nbin;
        if (p8) {
            const int blk = c.p8_block, lb = blk == 64 ? 6 : 7;
#pragma unroll 4
            for (int x = t0; x < 8 * blk; x += dt) {
                const int q = x >> lb, i = x & (blk - 1);
                if (i < c.sp.size[q]) {
                    const int row = c.sp.start[q] + i, o = x + q * blk;
                    atomicAdd(aw + row, (unsigned long long)(long long)(b0[o] - b0[o + blk]));
                    atomicAdd(aw + s + row, (unsigned long long)(long long)(b1[o] - b1[o + blk]));
                    b0[o] = b0[o + blk] = 0;
                    b1[o] = b1[o + blk] = 0;
                }
            }
        } else {
            for (int x = t0; x < s; x += dt) {
                atomicAdd(aw + x, (unsigned long long)(long long)b0[x]);
                atomicAdd(aw + s + x, (unsigned long long)(long long)b1[x]);
                b0[x] = 0;
                b1[x] = 0;
            }
        }
    };
    auto flush_w = [&](int i, int t0, int dt) { flush_bins(i, c.accw + (size_t)i * 2 * s, t0, dt); };

    // FP32 basis: H of the relation with the applied sigma_j and coefficients,
    // A v_j = (sigma_j / sap_j) (v_{j+1} ||w_{j+1}|| + sum_i c_i v_i / sigma_i), from the
    // stored c_i and ||w_{j+1}|| of columns 0 .. nc - 1 (an FP64 division is too slow
    // for the recurrence's critical path)
    auto finish_h = [&](int nc) {
        if (!F32 || g != 0) return;
        __syncthreads();
        for (int x = tid; x < nc * (k + 1); x += kPT) {
            const int jc = x / (k + 1), i = jc + 1 - x % (k + 1);
            if (i < 0) continue;
            const double sj = __ldcg(c.vscale + jc), f = (double)(float)sj;
            double *h = c.H + i + (size_t)jc * (m + 1);
            const double v = __ldcg(h);
            *h = i == jc + 1 ? sj * v / f : sj * v / (f * __ldcg(c.vscale + i));
        }
    };

    // ---- set-up: slice metadata, bins, H = 0, iscal, w_0 = b
    for (int t = tid; t < nsl; t += kPT) {
        meta_o[t] = c.sell_off[r0 / 32 + t];
        meta_w[t] = c.sell_w[r0 / 32 + t];
    }
    uint2 dmask = make_uint2(0u, 0u);   // masks of this warp's first two slices (diagonal copy)
    if (W > 0 && c.dg.w != 0 && warp < kSpmvWarps) {
        if (warp < nsl) dmask.x = c.dg.mask[r0 + 32 * warp + lane];
        if (warp + kSpmvWarps < nsl) dmask.y = c.dg.mask[r0 + 32 * (warp + kSpmvWarps) + lane];
    }
    for (int i = tid; i < 4 * nbin; i += kPT) bins[i] = 0;
    for (int64_t i = (int64_t)g * kPT + tid; i < (int64_t)(m + 1) * m; i += (int64_t)G * kPT) c.H[i] = 0.0;
    if (g == 0 && tid == 0) {
        c.iscal[0] = 0;
        c.iscal[1] = m;
        c.iscal[2] = SKF_OK;
        c.iscal[3] = m;
    }
    if (tid == 0) sbreak = 0;
    if (tid < kSlot) sch[tid] = 0;
    if constexpr (SHORT) {
        // sums of b^2 by slice, which the partition does not change
        const int64_t ns = (c.n + 31) >> 5;
        for (int t = warp; t < nsl; t += kPNW) {
            const int lr = t * 32 + lane;
            double v = 0.0, mx = 0.0;
            if (lr < nr) {
                const T xt = (T)c.b[r0 + lr];
                const double x = (double)xt;
                Vb[r0 + lr] = xt;
                win[lr] = xt;    // slot 0
                v = x * x;
                mx = key_to_abs(abs_key(x));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                v += __shfl_xor_sync(0xffffffffu, v, o);
                mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            }
            if (lane == 0) {
                c.pB[r0 / 32 + t] = v;
                c.pB[ns + r0 / 32 + t] = mx;
            }
        }
    } else {
        double nrm[1] = {0.0};
        unsigned long long key = 0;
        for (int lr = tid; lr < nr; lr += kPT) {
            const T xt = (T)c.b[r0 + lr];
            const double x = (double)xt;
            Vb[r0 + lr] = xt;
            win[lr] = xt;    // slot 0
            nrm[0] = fma(x, x, nrm[0]);
            key = max(key, abs_key(x));
        }
        key = block_reduce_t0<1>(nrm, key, red);
        if (tid == 0) {
            c.pB[g] = nrm[0];
            c.pB[G + g] = key_to_abs(key);
        }
    }
    if (!grid_barrier(c.bar, c.flag, ++nb, c.budget)) goto timeout;
    if constexpr (SHORT) {
        // by 128 threads, whatever the grid
        const int ns = (int)((c.n + 31) >> 5);
        if (warp < 4) {
            double v = 0.0, mx = 0.0;
#pragma unroll 4
            for (int t = tid; t < ns; t += 128) {
                v += __ldcg(c.pB + t);
                mx = fmax(mx, __ldcg(c.pB + ns + t));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                v += __shfl_xor_sync(0xffffffffu, v, o);
                mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            }
            if (lane == 0) {
                red[warp] = v;
                red[4 + warp] = mx;
            }
        }
        __syncthreads();
        if (tid == 0) {
            sb[0] = ((red[0] + red[1]) + red[2]) + red[3];
            sb[1] = fmax(fmax(red[4], red[5]), fmax(red[6], red[7]));
        }
    } else if (warp < 2) {
        const double v = reduce_slot(c.pB + (size_t)warp * G, G, warp == 1);
        if (lane == 0) sb[warp] = v;
    }
    __syncthreads();
    if (!(sb[0] > 0.0)) {   // zero right-hand side: x = 0
        if (g == 0 && tid == 0) {
            c.iscal[0] = 1;
            c.iscal[1] = 0;
            c.iscal[2] = SKF_ERR_ZERO_RHS;
            c.iscal[3] = 0;
        }
        return;
    }
    if (tid == 0) {
        sig[0] = rsqrt(sb[0]);
        sap[0] = F32 ? (double)(float)sig[0] : sig[0];
        ews[0] = positive_finite(sb[1]) ? bound_exponent(sb[1]) : kNoExp;
        if (g == 0) c.vscale[0] = sig[0];
    }
    __syncthreads();

    for (int j = 0; j < m; ++j) {
        const int i0 = max(0, j - k + 1);
        const int nw = j - i0 + 1;
        const bool last = j == m - 1;
        const int ngj = min(j, k - 1);       // Gram distances of w_j
        // ---- phase A: y~ = A w_j and the window dots (kSpmvWarps warps).
        // Phase A does not need the norm of w_j (stored unnormalised): meanwhile
        // the service warp turns the sums of phase B of the previous step into
        // sigma_j, the breakdown test and the factors of the MGS recurrence, so
        // that after the barrier only the products with the dots are left; the
        // CTA's S w_{j-1} bins are added to the global sums and the sketch
        // columns of step j - 2 finalised (none of it is needed before that).
        T acc[KW];
#pragma unroll
        for (int a = 0; a < KW; ++a) acc[a] = T(0);
        unsigned ykey = 0;
        if (warp == kSvc && j >= 1) {
            // lane 0: ||w_j||^2, lane d: <w_j, w_{j-d}>
            unsigned wk;
            const double tot = pull_sums<CB>(c.slot + (size_t)(2 * j - 1) * kSlot, 1 + ngj, eb, wk);
            double gr[KW];
#pragma unroll
            for (int d = 1; d < KW; ++d) gr[d] = __shfl_sync(0xffffffffu, tot, d);
            if (lane == 0) {
                // H column j - 1 (FP32: c_i and h_{j,j-1} unscaled, finish_h turns them
                // into the coefficients of the relation with the applied values)
                const int jp = j - 1, ip0 = max(0, jp - k + 1), np = jp - ip0 + 1;
                double hs = 0.0;
                for (int a = 0; a < np; ++a) {
                    hs = fma(sh[a], sh[a], hs);
                    if (g == 0) c.H[ip0 + a + (size_t)jp * (m + 1)] = F32 ? coef[jp & 3][np - 1 - a] : sh[a];
                }
                // ||A v_{j-1}||^2 = sum_i h_i^2 + ||w_j||^2 for the orthonormal window;
                // happy breakdown when ||w_j|| <= 1e-12 ||A v_{j-1}||
                // (compared in squares, and sigma = 1/||w_j|| from one rsqrt: an FP64
                // square root or division is ~650 dependent cycles on this part)
                // (FP32: ||w_j|| <= 2^-17 ||A v_{j-1}||, 64 FP32 unit roundoffs)
                sbreak = (tot > (F32 ? 5.820766091346741e-11 : 1e-24) * (hs + tot)) ? 0 : 1;
                const double sgm = tot > 0.0 ? rsqrt(tot) : 0.0;
                if (g == 0) {
                    c.H[j + (size_t)jp * (m + 1)] = tot * sgm;
                    if (!sbreak) c.vscale[j] = sgm;
                }
                if (!sbreak) {   // w_j enters the window
                    sig[j & 3] = sgm;
                    sap[j & 3] = F32 ? (double)(float)sgm : sgm;
#pragma unroll
                    for (int d = 1; d < KW; ++d)
                        if (d <= ngj) grm[j & 3][d] = gr[d];
                    ews[j & 3] = key_exponent<T>(wk);
                }
            }
            __syncwarp();
        }
        if (warp == kSvc) {
            // factors of the MGS recurrence that do not depend on the dots
            // (h_i = fd_i <w_i, y> - sum_{i' < i} fg_ii' h_i'), one per lane
            if (lane < nw) {
                fd[lane] = sig[(i0 + lane) & 3] * sig[j & 3];
                ea[lane] = ews[(i0 + lane) & 3] + ews[j & 3] + c.e_row + lg_rows;
            }
            if (lane >= 16 && lane < 16 + KW * KW) {
                const int a = (lane - 16) / KW, b2 = (lane - 16) % KW;
                if (a < nw && b2 < a)
                    fg[a][b2] = sig[(i0 + a) & 3] * sig[(i0 + b2) & 3] * grm[(i0 + a) & 3][a - b2];
            }
        }
        // S w_{j-1}: by the warps that have no slice; by all warps after their
        // slices where phase A is short (kFlushAll: the service warp alone needs
        // longer than that, 3.0 of 14.7 us per step with 45 slices; 13.8 with all warps); else by the
        // service warp, beside phase A
        const bool flush_all = nh == 0 && nsl <= kFlushAll;
        if (j >= 1 && (nh > 0 ? (warp >= nsl && warp < kSpmvWarps) : warp == kSvc)) {
            const int ht = nh > 0 ? tid - 32 * nsl : lane, nt = nh > 0 ? 32 * nh : 32;
            if (!flush_all) flush_w(j - 1, ht, nt);
            if (j >= 2)
                for (int t = ht; g + G * t < s; t += nt) finalize_col(j - 2, t);
        }
        int soff[KW];   // window slot offsets, oldest first
#pragma unroll
        for (int a = 0; a < KW; ++a) soff[a] = a < nw ? ((i0 + a) % k) * R : 0;
        if (warp < kSpmvWarps)
            spmv_rows<KW, W, !YG, SHORT, T>(c, Vb + (size_t)j * c.ldv, win, soff, nw, ys, meta_o, meta_w, dmask, nsl,
                                            nr, acc, ykey);
        if (flush_all && j >= 1) flush_w(j - 1, tid, kPT);
        __syncthreads();   // the bounds ea[] of the service warp
        // grid sums of the dots and, by warp 0, the coefficients of the step; bar_ok
        // becomes 2 where a first pass finds its bound too far above max|y~|
        auto sum_dots = [&](unsigned long long *sl, bool first) {
            if constexpr (SHORT) {
                int mine = 0;
                bool bad = false;
                unsigned key = 0;
                for (int q = 0; row_of(q) - lane < nr; ++q) {   // a summand per lane and turn
                    T v[KW];
#pragma unroll
                    for (int a = 0; a < KW; ++a) v[a] = T(0);
                    for (int u = 0; u <= gl; ++u, q += u <= gl) {
                        const int lr = row_of(q);
                        const T y = lr < nr ? ys[lr] : T(0);
#pragma unroll
                        for (int a = 0; a < KW; ++a)
                            if (a < nw && lr < nr) v[a] = fma(win[soff[a] + lr], y, v[a]);
                        key = max(key, mag_key(y));
                    }
#pragma unroll
                    for (int a = 0; a < KW; ++a)
                        if (a < nw) add_chunks<CB>(v[a], ea[a], a, mine, bad);
                }
                flush_sums(mine, bad, nw, key, sch, sl);
            } else {
                push_sums<CB, KW, T>(acc, nw, ea, ykey, sch, sl);
            }
            ++nb;
            if (warp == 0) {
                __syncwarp();
                if (lane == 0) {
                    grid_arrive(c.bar);
                    bar_ok = spin_until(c.bar, nb * (unsigned)G, c.flag, c.budget);
                }
                __syncwarp();
                // totals of this step (every CTA, identically): lane a the dot with
                // w_{i0+a}; MGS in the window, ascending, from the dots and the Gram
                // matrix: h_i = <v_i, y> - sum_{i' < i} h_i' <v_i, v_i'>
                unsigned yk;
                double dot = pull_sums<CB>(sl, nw, ea, yk);
                if (lane < nw) dot *= fd[lane];
                double h[KW];
#pragma unroll
                for (int a = 0; a < KW; ++a) h[a] = __shfl_sync(0xffffffffu, dot, a);
                if (lane == 0 && !sbreak) {
                    int ew1 = -2000;   // |w_{j+1}| < 2^ew1: the largest term's exponent, for up to 5 terms
                    const int ey = key_exponent<T>(yk);
                    if (ey != kNoExp) ew1 = max(ew1, exponent_above(sap[j & 3]) + ey);
#pragma unroll
                    for (int a = 0; a < KW; ++a) {
                        if (a < nw) {
#pragma unroll
                            for (int b2 = 0; b2 < KW; ++b2)
                                if (b2 < a) h[a] = fma(-h[b2], fg[a][b2], h[a]);
                            sh[a] = h[a];
                            double cc = h[a] * sig[(i0 + a) & 3];
                            if constexpr (F32) cc = (double)(float)cc;
                            coef[j & 3][nw - 1 - a] = cc;
                            if (ews[(i0 + a) & 3] != kNoExp) ew1 = max(ew1, exponent_above(cc) + ews[(i0 + a) & 3]);
                        }
                    }
                    cnw[j & 3] = nw;
                    eys[j & 3] = ey;
                    ew1 += 3;
                    eb[0] = 2 * ew1 + lg_rows;
#pragma unroll
                    for (int d = 1; d < KW; ++d)   // <w_{j+1}, w_{j+1-d}>
                        if (d <= nw) eb[d] = ew1 + ews[(j + 1 - d) & 3] + lg_rows;
                    if (first && bar_ok && ey != kNoExp && ews[j & 3] + c.e_row - ey > kMaxSlack) bar_ok = 2;
                }
            }
            __syncthreads();
        };
        sum_dots(c.slot + (size_t)(2 * j) * kSlot, true);
        if (bar_ok != 1) {
            if (bar_ok == 0) goto timeout;
            // (rare) ||A||_inf says nothing about this y~: the dots once more, below
            // max|y~|, from y~ and the window into the step's second slot
            if (tid < nw) ea[tid] = ews[(i0 + tid) & 3] + eys[j & 3] + lg_rows;
            if constexpr (!SHORT) {
#pragma unroll
                for (int a = 0; a < KW; ++a) acc[a] = T(0);
                ykey = 0;
                for (int lr = tid; lr < nr; lr += kPT) {
                    const T y = ys[lr];
#pragma unroll
                    for (int a = 0; a < KW; ++a)
                        if (a < nw) acc[a] = fma(win[soff[a] + lr], y, acc[a]);
                    ykey = max(ykey, mag_key(y));
                }
            }
            __syncthreads();
            sum_dots(c.slot + (size_t)(2 * m + 1 + j) * kSlot, false);
            if (!bar_ok) goto timeout;
        }

        if (sbreak) {
            // happy breakdown: w_j is rounding noise, the basis ends at m_eff = j.
            // S A v_{j-1} is sketched directly from y~_{j-1} = A w_{j-1}, computed
            // again (bitwise the same: fixed per-row order) into ys[].
            const int jb = j - 1, i0b = max(0, jb - k + 1), nwb = jb - i0b + 1;
            int soff[KW];
#pragma unroll
            for (int a = 0; a < KW; ++a) soff[a] = a < nwb ? ((i0b + a) % k) * R : 0;
            T accb[KW];
#pragma unroll
            for (int a = 0; a < KW; ++a) accb[a] = T(0);
            unsigned kb = 0;
            if (warp < kSpmvWarps)
                spmv_rows<KW, W, !YG, SHORT, T>(c, Vb + (size_t)jb * c.ldv, win, soff, 0, ys, meta_o, meta_w, dmask, nsl, nr,
                                         accb, kb);
            __syncthreads();
            const int ey = eys[jb & 3];
            const int shift_y = c.frac - (ey == kNoExp ? 0 : ey);
            // (both bin buffers are empty: S w_{j-1} was added up in phase A)
            int *by0 = bins, *by1 = bins + nbin;
            for (int lr = tid; lr < nr; lr += kPT) {
                const int64_t r = r0 + lr;
                const long long vy = ey == kNoExp ? 0 : fixed_point(ys[lr], shift_y);
                const uint2 pv = p8 ? __ldg((const uint2 *)(c.pattern8 + r * 8)) : make_uint2(0u, 0u);
                scatter_row<ZCAP>(c, r, pv, p8, by0, by1, (int)(vy & lmask), (int)(vy >> c.L));
            }
            __syncthreads();
            flush_bins(0, c.accy, tid, kPT);
            if (!grid_barrier(c.bar, c.flag, ++nb, c.budget)) goto timeout;
            // S v_{j-1}, S A v_{j-2} (S w_{j-1} was added up before the last barrier) and S A v_{j-1}
            for (int t = tid; g + G * t < s; t += kPT) {
                finalize_col(jb, t);
                finalize_direct(jb, t);
            }
            if (g == 0 && tid == 0) {
                c.iscal[0] = 1;
                c.iscal[1] = j;
                c.iscal[3] = j;
            }
            finish_h(j);
            return;
        }

        // ---- phase B: w_{j+1} and this thread's partials of its norm, Gram
        // entries and max; sketch of w_j (and of y~ in the last step)
        {
            const T sj = (T)sap[j & 3];   // sigma_j as applied
            const int ew = ews[j & 3], ey = eys[j & 3];
            const int shift_w = c.frac - (ew == kNoExp ? 0 : ew);
            const int shift_y = c.frac - (ey == kNoExp ? 0 : ey);
            const int ng = min(j + 1, k - 1);
            int *bw0 = bins + (j & 1) * 2 * nbin, *bw1 = bw0 + nbin;
            int *by0 = bins + ((j + 1) & 1) * 2 * nbin, *by1 = by0 + nbin;   // S y~ of the last step: the empty buffer
            T cf[KW];        // c_b for w_{j-b} (as applied)
            int soffr[KW];   // slot offsets, newest first
#pragma unroll
            for (int b2 = 0; b2 < KW; ++b2) {
                cf[b2] = b2 < nw ? (T)coef[j & 3][b2] : T(0);
                soffr[b2] = b2 < nw ? ((j - b2) % k) * R : 0;
            }
            const int snew = ((j + 1) % k) * R;
            T *wn = Vb + (size_t)(j + 1) * c.ldv;
            T part[KW];
#pragma unroll
            for (int a = 0; a < KW; ++a) part[a] = T(0);
            unsigned nkey = 0;
            uint2 pv_next = make_uint2(0u, 0u);
            int mine = 0;      // (short form: chunk sums)
            bool bad = false;
            // rows of this thread; in the short form whole groups, lanes past nr without a row
            int lr = SHORT ? row_of(0) : tid;
            if (p8 && lr < nr) pv_next = __ldg((const uint2 *)(c.pattern8 + (r0 + lr) * 8));
            for (int q = 0; SHORT ? lr - lane < nr || (q & gl) != 0 : lr < nr; ++q) {
                const int64_t r = r0 + lr;
                const int lrn = SHORT ? row_of(q + 1) : lr + kPT;
                const uint2 pv = pv_next;
                if (p8 && lrn < nr) pv_next = __ldg((const uint2 *)(c.pattern8 + (r0 + lrn) * 8));
                if (!SHORT || lr < nr) {
                    const T y = ys[lr];
                    T wv[KW];
#pragma unroll
                    for (int b2 = 0; b2 < KW; ++b2) wv[b2] = b2 < nw ? win[soffr[b2] + lr] : T(0);
                    if (!last) {
                        T w = sj * y;
#pragma unroll
                        for (int b2 = KW - 1; b2 >= 0; --b2)
                            if (b2 < nw) w = fma(-cf[b2], wv[b2], w);   // oldest first
                        wn[r] = w;
                        win[snew + lr] = w;
                        nkey = max(nkey, mag_key(w));
                        part[0] = fma(w, w, part[0]);
#pragma unroll
                        for (int d = 1; d < KW; ++d)
                            if (d <= ng) part[d] = fma(w, wv[d - 1], part[d]);
                    }
                    const long long vw = ew == kNoExp ? 0 : fixed_point(wv[0], shift_w);
                    scatter_row<ZCAP>(c, r, pv, p8, bw0, bw1, (int)(vw & lmask), (int)(vw >> c.L));
                    if (last) {
                        const long long vy = ey == kNoExp ? 0 : fixed_point(y, shift_y);
                        scatter_row<ZCAP>(c, r, pv, p8, by0, by1, (int)(vy & lmask), (int)(vy >> c.L));
                    }
                }
                if (SHORT && !last && (q & gl) == gl) {   // the group's summands
#pragma unroll
                    for (int d = 0; d < KW; ++d) {
                        if (d <= ng) add_chunks<CB>(part[d], eb[d], d, mine, bad);
                        part[d] = T(0);
                    }
                }
                lr = lrn;
            }
            if (!last) {
                unsigned long long *sl = c.slot + (size_t)(2 * j + 1) * kSlot;
                if constexpr (SHORT) flush_sums(mine, bad, 1 + ng, nkey, sch, sl);
                else push_sums<CB, KW, T>(part, 1 + ng, eb, nkey, sch, sl);
            } else {
                __syncthreads();
                flush_w(j, tid, kPT);
                flush_bins(j + 1, c.accy, tid, kPT);
                __syncthreads();
            }
        }
        ++nb;
        if (warp == 0) {
            __syncwarp();
            if (lane == 0) {
                grid_arrive(c.bar);
                bar_ok = spin_until(c.bar, nb * (unsigned)G, c.flag, c.budget);
            }
        }
        __syncthreads();
        if (!bar_ok) goto timeout;
        if (last) {
            // S v_{m-2}, S v_{m-1}, S A v_{m-3}, S A v_{m-2} (relation), S A v_{m-1} (direct)
            for (int t = tid; g + G * t < s; t += kPT) {
                if (j >= 1) finalize_col(j - 1, t);
                finalize_col(j, t);
                finalize_direct(j, t);
            }
        }
    }
    finish_h(m - 1);
    return;
timeout:
    if (g == 0 && tid == 0) {
        c.iscal[0] = 1;
        c.iscal[1] = 0;
        c.iscal[2] = SKF_ERR_TIMEOUT;
        c.iscal[3] = 0;
    }
}

// | ||S v_j||^2 - 1 | for column j (one CTA per column), folded into a
// maximum with an integer atomic on the bit pattern (non-negative doubles
// order like their bits, so the result does not depend on the order).
__global__ void __launch_bounds__(128) k_persist_eps(const double *__restrict__ SV, int s,
                                                    const int *__restrict__ iscal, unsigned long long *epsmax) {
    __shared__ double red[4];
    const int j = blockIdx.x;
    if (j >= iscal[1]) return;
    double a = 0.0;
    for (int i = threadIdx.x; i < s; i += 128) a = fma(SV[i + (size_t)j * s], SV[i + (size_t)j * s], a);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        const double e = fabs(((red[0] + red[1]) + red[2]) + red[3] - 1.0);
        atomicMax(epsmax, (unsigned long long)__double_as_longlong(e));
    }
}

__global__ void k_persist_info(const double *__restrict__ vscale, const int *__restrict__ iscal,
                               const unsigned long long *epsmax, skf_info *info) {
    if (threadIdx.x != 0 || info == nullptr) return;
    const int me = iscal[1];
    info->status = iscal[2];
    info->m_eff = me;
    info->breakdown = (iscal[0] == 1 && me > 0) ? 1 : 0;
    info->beta = me > 0 ? 1.0 / vscale[0] : 0.0;
    info->eps_est = __longlong_as_double((long long)*epsmax);
}

// The short form (kShortRows) and its slices per summand, by the size alone,
// whatever the partition of a call: with one slice per summand the cutting into
// chunks, about 100 instructions per warp and value, would come twice per phase
// beyond 512 rows per CTA (N = 1e5, m = 40: 858 us, 801 with two slices and the
// window offsets taken out of the loop; alone on the card at one CTA per SM, 781).
bool persist_short(int64_t n) { return n <= (int64_t)kShortRows * num_sms(); }
int persist_group(int64_t n) { return n <= (int64_t)kPT * num_sms() ? 1 : 2; }

// A barrier that can never complete (it waits for one CTA more than the
// grid has), with the given budget: the self-test of the bounded wait.
__global__ void __launch_bounds__(32) k_barrier_selftest(unsigned *bar, int *flag, long long budget, int *status) {
    // barrier number 2 needs 2 G arrivals; the grid makes G
    const bool ok = grid_barrier(bar, flag, 2, budget);
    if (blockIdx.x == 0 && threadIdx.x == 0) *status = ok ? SKF_OK : SKF_ERR_TIMEOUT;
}

template <int KW, int W, int ZCAP, bool YG, typename T>
cudaError_t launch_persist(const PCtx &c, int G, size_t smem, cudaStream_t st) {
    auto kern = k_arnoldi_persist<KW, W, ZCAP, YG, false, T>;
    if constexpr (!YG)
        if (persist_short(c.n)) kern = k_arnoldi_persist<KW, W, ZCAP, false, true, T>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPT, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1 || G > per_sm * num_sms()) return cudaErrorCooperativeLaunchTooLarge;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)G);
    cfg.blockDim = dim3(kPT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, c);
}

template <int KW, int W, bool YG, typename T>
cudaError_t launch_persist_z(const PCtx &c, int G, size_t smem, cudaStream_t st) {
    return c.sp.zeta <= 8 ? launch_persist<KW, W, 8, YG, T>(c, G, smem, st)
                          : launch_persist<KW, W, 16, YG, T>(c, G, smem, st);
}

template <int KW>
cudaError_t launch_persist_w(const PCtx &c, int maxw, int G, size_t smem, cudaStream_t st) {
    if (maxw <= 5) return launch_persist_z<KW, 5, false, double>(c, G, smem, st);
    if (maxw <= 7) return launch_persist_z<KW, 7, false, double>(c, G, smem, st);
    if (maxw <= 8) return launch_persist_z<KW, 8, false, double>(c, G, smem, st);
    return launch_persist_z<KW, 0, false, double>(c, G, smem, st);
}

// y~ in global memory: instantiated for k <= 2 and slices at most 7 wide (the
// 5- and 7-point stencils) only
cudaError_t launch_persist_yg(const PCtx &c, int maxw, int G, size_t smem, cudaStream_t st) {
    if (maxw <= 5) return launch_persist_z<2, 5, true, double>(c, G, smem, st);
    return launch_persist_z<2, 7, true, double>(c, G, smem, st);
}

// FP32 basis: k <= 2, slices at most 7 wide, y~ on chip
cudaError_t launch_persist_f32(const PCtx &c, int maxw, int G, size_t smem, cudaStream_t st) {
    if (maxw <= 5) return launch_persist_z<2, 5, false, float>(c, G, smem, st);
    return launch_persist_z<2, 7, false, float>(c, G, smem, st);
}

// Dynamic shared memory of the persistent kernel for R rows per CTA with
// elements of vb bytes (yg: y~ kept in global memory instead).
size_t persist_smem(int R, int k, int nbin, bool yg, size_t vb = sizeof(double)) {
    const size_t red = (size_t)kPT + 4 + kPNW;
    return vb * (size_t)(k + (yg ? 0 : 1)) * R + sizeof(double) * red +
           (sizeof(long long) + sizeof(int)) * (size_t)(R / 32) + sizeof(int) * 4 * (size_t)nbin;
}

}  // namespace

// Persistent partition of a level: G = min(SMs, ceil(n / kPersistMinRows)) CTAs
// of R rows (whole slices).  The sketch tables record the bin-load maximum over
// the levels.
void persist_partition(int64_t n, int level, int *G, int64_t *rows) {
    const int64_t mr = kPersistMinRows[level];
    int64_t g = (n + mr - 1) / mr;
    if (g > num_sms()) g = num_sms();
    if (g < 1) g = 1;
    const int64_t u = persist_short(n) ? 32 * persist_group(n) : 32;   // whole groups
    const int64_t R = ((n + g - 1) / g + u - 1) / u * u;
    *rows = R;
    *G = (int)((n + R - 1) / R);
}

int64_t persist_max_rows_f64() {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int R = 32;
    while (persist_smem(R + 32, 1, 16 * 64, true) + 4096 <= (size_t)optin) R += 32;
    return (int64_t)R * num_sms();
}

// The level of a solve on one of `lanes` lanes (beyond kShortRows all levels are one).
static int persist_level(int64_t n, int lanes) {
    if (lanes <= 2) return 0;   // (two of any size fit side by side)
    for (int l = 0; l + 1 < kPersistLevels; ++l) {
        int G;
        int64_t rows;
        persist_partition(n, l, &G, &rows);
        if (2ll * lanes * G <= 3ll * num_sms()) return l;
    }
    return kPersistLevels - 1;
}

static int g_step_mode = 0;   // 0 auto, 1 two-kernel path only, 2 persistent path required
void set_step_mode(int mode) { g_step_mode = mode; }
int step_mode() { return g_step_mode; }

// The persistent form for an FP64 basis (f32 = false) or an FP32 one (f32:
// FP32 values, k <= 2, slices at most 7 wide, the window and y~ both on chip:
// N up to about 2e6).
static skf_status run_persistent(const skf_csr *A, const skf_sketch *S, const double *b, int m, int k, void *V,
                                 int64_t ldv, double *vscale, double *SV, double *SAV, double *H, int *iscal,
                                 skf_info *info, cudaStream_t st, bool f32, int lanes) {
    if (S->kind != SKF_SKETCH_SPARSE_SIGN || S->binmax_persist == nullptr || k > 4 ||
        A->vdtype != (f32 ? SKF_F32 : SKF_F64) || A->nlong > 0 ||
        A->perm != nullptr)   // a row split or sorted slices take the two-kernel form
        return SKF_ERR_NOT_SUPPORTED;
    if (f32 && (k > 2 || A->max_width > 7)) return SKF_ERR_NOT_SUPPORTED;
    const size_t vb = f32 ? sizeof(float) : sizeof(double);
    int G;
    int64_t R64;
    persist_partition(A->n, persist_level(A->n, lanes), &G, &R64);
    if (G > kMaxG) return SKF_ERR_NOT_SUPPORTED;
    const int R = (int)R64;
    const int KW = k <= 2 ? 2 : 4;
    const int s = S->s;
    const bool p8 = S->zeta == 8 && S->pattern8 != nullptr;
    const int nbin = p8 ? 16 * S->p8_block : s;
    size_t smem = persist_smem(R, k, nbin, false, vb);
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return SKF_ERR_NOT_SUPPORTED;
    }
    // static shared arrays of the kernel take about 3 KB; past the per-CTA
    // shared memory the window alone may still fit, with y~ in global memory
    bool yg = false;
    if (smem + 4096 > (size_t)optin) {
        if (f32) return SKF_ERR_NOT_SUPPORTED;   // an FP32 basis keeps y~ on chip
        yg = true;
        smem = persist_smem(R, k, nbin, true, vb);
        if (KW != 2 || A->max_width > 7 || smem + 4096 > (size_t)optin) return SKF_ERR_NOT_SUPPORTED;
    }
    int coop = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
        cudaGetLastError();
        return SKF_ERR_NOT_SUPPORTED;
    }

    PCtx c{};
    c.n = A->n;
    c.R = R;
    c.group = persist_group(A->n);
    c.sell_off = A->sell_off;
    c.sell_w = A->sell_w;
    c.sell_val = A->sell_val;
    c.sell_col = A->sell_col;
    // 8 diagonals of rows at most 7 wide: only the general FP64 form has 8 slots
    if (A->dia_w <= (f32 || yg ? 7 : 8)) c.dg = diag_of(A);
    const double opb = c.dg.w != 0 ? 32.0 * (double)A->nslices * (double)(vb * c.dg.w + 1)
                                   : (double)A->sell_entries * (double)(vb + 4);
    c.l2_frac = l2_keep_fraction(opb);
    c.sp = make_sparse_sign(S);
    c.pattern = S->pattern;
    if (p8) {
        c.pattern8 = S->pattern8;
        c.p8_block = S->p8_block;
    }
    c.L = limb_bits(S->binmax_persist_host);
    c.frac = sketch_fraction_bits_from_limb(c.L);
    c.e_row = positive_finite(A->norm_inf) ? bound_exponent(A->norm_inf) + 1 : 0;
    c.sk_scale = 1.0 / sqrt((double)S->zeta);
    c.m = m;
    c.k = k;
    c.b = b;
    c.V = V;
    c.ldv = ldv;
    c.vscale = vscale;
    c.SV = SV;
    c.SAV = SAV;
    c.H = H;
    c.iscal = iscal;
    c.budget = kBarrierBudget;

    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t szP = sizeof(double) * 2 * (size_t)(persist_short(A->n) ? (A->n + 31) / 32 : G);
    const size_t szSlot = sizeof(unsigned long long) * (size_t)(3 * m + 1) * kSlot;
    const size_t szAw = sizeof(unsigned long long) * (size_t)m * 2 * s;
    const size_t szAy = sizeof(unsigned long long) * 2 * (size_t)s;
    const size_t szSw = sizeof(double) * (size_t)s * m;
    const size_t szBar = 2 * sizeof(int) + sizeof(unsigned long long);   // counter, flag, eps maximum
    const size_t szYs = yg ? vb * (size_t)G * R : 0;
    const size_t total = al(szP) + al(szSlot) + al(szAw) + al(szAy) + al(szSw) + al(szBar) + al(szYs);
    char *ws = nullptr;
    skf_status stt = dalloc((void **)&ws, total, st);
    if (stt != SKF_OK) return stt;
    size_t off = 0;
    auto take = [&](size_t sz) {
        char *p = ws + off;
        off += al(sz);
        return p;
    };
    c.pB = (double *)take(szP);
    c.slot = (unsigned long long *)take(szSlot);
    c.accw = (unsigned long long *)take(szAw);
    c.accy = (unsigned long long *)take(szAy);
    c.Sw = (double *)take(szSw);
    c.bar = (unsigned *)take(szBar);
    c.ysg = yg ? (void *)take(szYs) : nullptr;
    c.flag = (int *)(c.bar + 1);
    unsigned long long *epsmax = (unsigned long long *)(c.bar + 2);
    // accumulators and the barrier start at zero (one memset: they are adjacent)
    cudaMemsetAsync(c.slot, 0, (size_t)((char *)c.Sw - (char *)c.slot), st);
    cudaMemsetAsync(c.bar, 0, szBar, st);
    cudaError_t e;
    const int slots = c.dg.w != 0 ? c.dg.w : A->max_width;   // product slots of the kernel
    if (f32) e = launch_persist_f32(c, slots, G, smem, st);
    else if (yg) e = launch_persist_yg(c, slots, G, smem, st);
    else if (KW == 2) e = launch_persist_w<2>(c, slots, G, smem, st);
    else e = launch_persist_w<4>(c, slots, G, smem, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        dfree(ws, st);
        if (e == cudaErrorCooperativeLaunchTooLarge) return SKF_ERR_NOT_SUPPORTED;
        return cuda_fail(e, "persistent Arnoldi launch");
    }
    k_persist_eps<<<m, 128, 0, st>>>(SV, s, iscal, epsmax);
    k_persist_info<<<1, 32, 0, st>>>(vscale, iscal, epsmax, info);
    count_launches(3);
    e = cudaGetLastError();
    dfree(ws, st);
    if (e != cudaSuccess) return cuda_fail(e, "persistent Arnoldi kernels");
    return SKF_OK;
}

skf_status arnoldi_run_persistent(const skf_csr *A, const skf_sketch *S, const double *b, int m, int k, double *V,
                                  int64_t ldv, double *vscale, double *SV, double *SAV, double *H, int *iscal,
                                  skf_info *info, cudaStream_t st, int lanes) {
    return run_persistent(A, S, b, m, k, V, ldv, vscale, SV, SAV, H, iscal, info, st, false, lanes);
}

skf_status arnoldi_run_persistent_f32(const skf_csr *A, const skf_sketch *S, const double *b, int m, int k, float *V,
                                      int64_t ldv, double *vscale, double *SV, double *SAV, double *H, int *iscal,
                                      skf_info *info, cudaStream_t st, int lanes) {
    return run_persistent(A, S, b, m, k, V, ldv, vscale, SV, SAV, H, iscal, info, st, true, lanes);
}

// Self-test of the bounded barrier wait: a grid of `ctas` co-resident CTAs
// waits at a barrier that can never complete; the wait must give up after
// `budget` SM cycles and report SKF_ERR_TIMEOUT in *status_out (device int).
skf_status barrier_selftest(int ctas, long long budget, int *status_out, cudaStream_t st) {
    char *ws = nullptr;
    skf_status stt = dalloc((void **)&ws, 256, st);
    if (stt != SKF_OK) return stt;
    unsigned *bar = (unsigned *)ws;
    int *flag = (int *)(ws + 4);
    cudaMemsetAsync(ws, 0, 8, st);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(32);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_barrier_selftest, bar, flag, budget, status_out);
    count_launches(1);
    dfree(ws, st);
    if (e != cudaSuccess) return cuda_fail(e, "barrier self-test launch");
    return SKF_OK;
}

}  // namespace skf
