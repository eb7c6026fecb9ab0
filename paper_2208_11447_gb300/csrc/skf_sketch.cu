// The subspace embedding S (eq. (1.1)): expansion of the sparse-sign pattern
// from its SplitMix64 definition, the per-partition bin-load maxima that
// size the fixed-point limbs, and S X for general X (column maxima,
// fixed-point scatter into per-CTA shared-memory bins, exact cross-CTA
// reduction).  The Arnoldi kernels use the same pattern and accumulation.
#include <math.h>

#include <algorithm>
#include <mutex>

#include "skf_internal.cuh"
#include "skf_step.cuh"

namespace skf {

SparseSign make_sparse_sign(const skf_sketch *S) {
    SparseSign sp{};
    sp.s = S->s;
    sp.zeta = S->zeta;
    sp.words = (S->zeta + 3) / 4;
    sp.seed = S->seed;
    for (int q = 0; q < S->zeta; ++q) {
        const int a = (int)(((long long)q * S->s) / S->zeta);
        const int b = (int)(((long long)(q + 1) * S->s) / S->zeta);
        sp.start[q] = a;
        sp.size[q] = b - a;
    }
    return sp;
}

void row_partition(int64_t n, int *G, int64_t *rows) {
    int g = 2 * num_sms();
    const int64_t min_rows = 512;
    if ((n + min_rows - 1) / min_rows < g) g = (int)((n + min_rows - 1) / min_rows);
    if (g < 1) g = 1;
    *G = g;
    *rows = ((n + g - 1) / g + 31) / 32 * 32;   // whole SELL slices per CTA
}

void chunk_partition(int64_t n, int *G) {
    const int64_t chunks = (n + kChunkRows - 1) / kChunkRows;
    int g = num_sms();
    if (chunks < g) g = (int)chunks;
    *G = g < 1 ? 1 : g;
}

namespace {

// pattern[c * zeta + q] = (row of nonzero q of column c within stripe q) | sign << 15
__global__ void k_build_pattern(SparseSign sp, int64_t n, uint16_t *__restrict__ pattern) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (int64_t)gridDim.x * blockDim.x) {
        uint64_t word = 0;
        for (int q = 0; q < sp.zeta; ++q) {
            if ((q & 3) == 0) word = splitmix_word(sp.seed, (uint64_t)c * sp.words + (q >> 2));
            int row;
            bool neg;
            sparse_sign_entry(sp, word, q, row, neg);
            pattern[c * sp.zeta + q] = (uint16_t)((row - sp.start[q]) | (neg ? 0x8000 : 0));
        }
    }
}

// The same pattern in bytes (row within stripe + block * sign, block = 64 or
// 128), eight per column.
__global__ void k_build_pattern8(SparseSign sp, int64_t n, int block, const uint16_t *__restrict__ pattern,
                                 uint8_t *__restrict__ p8) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (int64_t)gridDim.x * blockDim.x)
        for (int q = 0; q < 8; ++q) {
            uint8_t v = 0;
            if (q < sp.zeta) {
                const uint16_t e = pattern[c * sp.zeta + q];
                v = (uint8_t)((e & 0x7FFFu) + ((e >> 15) ? block : 0));
            }
            p8[c * 8 + q] = v;
        }
}

// Largest number of nonzeros that one CTA's rows put into one row of S.  CTA
// g owns the chunks g, g + G, g + 2G, ... of `chunk` rows (one chunk per CTA
// for the contiguous partition).
__global__ void k_bin_max(SparseSign sp, int64_t n, int64_t chunk, const uint16_t *__restrict__ pattern,
                          int *binmax) {
    extern __shared__ int cnt[];
    for (int i = threadIdx.x; i < sp.s; i += blockDim.x) cnt[i] = 0;
    __syncthreads();
    for (int64_t r0 = (int64_t)blockIdx.x * chunk; r0 < n; r0 += (int64_t)gridDim.x * chunk) {
        const int64_t r1 = min(n, r0 + chunk);
        for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x)
            for (int q = 0; q < sp.zeta; ++q) {
                int row;
                bool neg;
                pattern_entry(sp, pattern[r * sp.zeta + q], q, row, neg);
                atomicAdd(cnt + row, 1);
            }
    }
    __syncthreads();
    int mx = 0;
    for (int i = threadIdx.x; i < sp.s; i += blockDim.x) mx = max(mx, cnt[i]);
    atomicMax(binmax, mx);
}

// Sketch of a block of columns in three launches (skf_sketch_apply): column
// maxima, scatter into per-CTA fixed-point bins, reduction.  16 columns of
// 1e6 rows, s = 800, zeta = 8: 388 -> 218 us (maxima 68 -> 26, scatter 242 -> 171,
// reduction 78 -> 21); X is read twice, 2 x 19 us at the measured copy rate, and
// the 2.6e8 shared atomics take 83 us at 3.3 cycles each.

// Magnitude key of each column: the high word of max |X[:, col]| (NaN
// skipped), of which only the exponent is used.  blockIdx.y = column; with more
// than one CTA per column the keys start at zero.
__global__ void __launch_bounds__(kThreads) k_colmax(const double *__restrict__ X, int64_t ldx, int64_t n,
                                                     unsigned *__restrict__ key) {
    const double *x = X + (int64_t)blockIdx.y * ldx;
    unsigned mx = 0;
    // integer maxima: an FP64 comparison holds the SM's FP64 pipe for 16 cycles
    for (int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x; r < n; r += (int64_t)gridDim.x * kThreads) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(x[r]) & 0x7FFFFFFFFFFFFFFFull;
        if (b <= 0x7FF0000000000000ull) mx = max(mx, (unsigned)(b >> 32));
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (gridDim.x == 1) {
        __shared__ unsigned wmx[kThreads / 32];
        if ((threadIdx.x & 31) == 0) wmx[threadIdx.x >> 5] = mx;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < kThreads / 32; ++w) mx = max(mx, wmx[w]);
            key[blockIdx.y] = mx;
        }
    } else if ((threadIdx.x & 31) == 0 && mx != 0u) {
        atomicMax(key + blockIdx.y, mx);
    }
}

constexpr int64_t kShortColumn = 8192;   // rows of a column that one CTA of k_colmax takes

// Exponent bound of a column from its key (key != 0; a key of a subnormal
// maximum gives the bound 2^-1022: its entries round to zero either way).
__device__ __forceinline__ int key_bound(unsigned key) { return max((int)(key >> 20), 1) - 1022; }

// Scatter of the rows of this CTA into fixed-point limb bins; writes the
// int64 partial sums [ncols][G][s].  With the compact pattern (BLK = 64 or 128)
// the bins are those of scatter8 in 1 << LC copies by lane; BLK = 0: any
// pattern, bins [limb][s].  Bound by instruction issue (IPC 3.2 of 4 before the
// immediates: 249 -> 171 us for 16 columns of 1e6 rows, s = 800).
constexpr int kScatterThreads = 512;
template <int BLK> struct ScatterGeom {
    static constexpr int kLc = BLK == 64 ? 3 : BLK == 128 ? 2 : 0;   // 64 KB of bins either way: three CTAs per SM
    static constexpr size_t bytes(int s) { return sizeof(int) * 2 * (BLK ? (size_t)(16 * BLK) << kLc : (size_t)s); }
};
template <int BLK>
__global__ void __launch_bounds__(kScatterThreads, BLK ? 3 : 1) k_sparse_sign_scatter(
    const double *__restrict__ X, int64_t ldx, int64_t n, int ncols, int64_t rows_per_cta, SparseSign sp,
    const uint16_t *__restrict__ pattern, const uint8_t *__restrict__ pattern8, const int *__restrict__ binmax,
    const unsigned *__restrict__ key, long long *__restrict__ out) {
    extern __shared__ __align__(16) int bins[];
    constexpr int LC = ScatterGeom<BLK>::kLc, C = 1 << LC;
    const int G = gridDim.x, s = sp.s, ns = BLK ? (16 * BLK) << LC : s;
    const int L = limb_bits(*binmax);
    const int frac = sketch_fraction_bits_from_limb(L);
    const long long lmask = (1ll << L) - 1;
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_cta;
    const int rn = (int)max((int64_t)0, min(n - r0, rows_per_cta));   // rows of this CTA
    const int tid = threadIdx.x, lane = tid & 31;
    const unsigned base = shared_address(bins) + 4u * (unsigned)(lane & (C - 1));
    const uint2 *p8 = (const uint2 *)pattern8 + r0;
    for (int i = tid; i < 2 * ns; i += kScatterThreads) bins[i] = 0;
    __syncthreads();
    // kBatch rows of a thread are loaded together, the next batch (or the next
    // column's first) before the atomics of this one
    constexpr int kBatch = 2;
    struct Rows {
        double x[kBatch];
        uint2 pv[kBatch];
    };
    auto load = [&](int c, int r, Rows &q) {
        const double *x = X + c * ldx + r0;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int ru = r + u * kScatterThreads;
            const bool ok = c < ncols && ru < rn;
            q.x[u] = ok ? x[ru] : 0.0;
            q.pv[u] = (BLK && ok) ? __ldg(p8 + ru) : make_uint2(0u, 0u);
        }
    };
    Rows cur, nxt;
    load(0, tid, cur);
    for (int c = 0; c < ncols; ++c) {
        const unsigned k = key[c];
        const int shift = frac - key_bound(k);
        for (int rb = 0; rb < rn; rb += kBatch * kScatterThreads) {
            const bool more = rb + kBatch * kScatterThreads < rn;
            load(more ? c : c + 1, (more ? rb + kBatch * kScatterThreads : 0) + tid, nxt);
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const long long v = k ? fixed_point(cur.x[u], shift) : 0;
                if (v == 0) continue;
                const int l0 = (int)(v & lmask), l1 = (int)(v >> L);
                if constexpr (BLK != 0) {
                    scatter8<BLK, LC>(cur.pv[u], base, l0, l1);
                } else {
                    const int64_t ru = r0 + rb + tid + u * kScatterThreads;
                    for (int q = 0; q < sp.zeta; ++q) {
                        int row;
                        bool neg;
                        pattern_entry(sp, pattern[ru * sp.zeta + q], q, row, neg);
                        red_limbs(bins, bins + s, row, l0, l1, neg);
                    }
                }
            }
            cur = nxt;
        }
        __syncthreads();
        // the copies of both signs summed (exact: all contributions of a row of S
        // together fit in 32 bits by the limb-width rule), bins cleared
        long long *o = out + ((size_t)c * G + blockIdx.x) * s;
        if constexpr (BLK != 0) {
            for (int x = tid; x < 8 * BLK; x += kScatterThreads) {
                const int q = x / BLK, i = x % BLK;
                int a[2] = {0, 0};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    int *p = bins + (((16 * h + 2 * q) * BLK + i) << LC), *m = p + (BLK << LC);
#pragma unroll
                    for (int d = 0; d < C; ++d) {   // (copies in rotated order: distinct banks for the lanes)
                        const int dd = (d + x) & (C - 1);
                        a[h] += p[dd] - m[dd];
                        p[dd] = 0;
                        m[dd] = 0;
                    }
                }
                if (i < sp.size[q]) o[sp.start[q] + i] = combine_limbs(a[0], a[1], L);
            }
        } else {
            for (int i = tid; i < s; i += kScatterThreads) {
                o[i] = combine_limbs(bins[i], bins[s + i], L);
                bins[i] = 0;
                bins[s + i] = 0;
            }
        }
        __syncthreads();
    }
}

// SX[i, c] = 2^(E_c - frac) zeta^-1/2 sum_g partial[c][g][i], summed exactly:
// 32 rows of S per CTA (coalesced loads), the partials dealt out over its
// warps, 128-bit sums combined through shared memory.
__global__ void __launch_bounds__(kThreads) k_sparse_sign_reduce(const long long *__restrict__ part,
                                                                 const unsigned *__restrict__ key, int G, int s,
                                                                 int zeta, const int *__restrict__ binmax,
                                                                 double *__restrict__ SX) {
    __shared__ unsigned long long slo[kThreads];
    __shared__ long long shi[kThreads];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.y, i = blockIdx.x * 32 + lane;
    unsigned long long lo = 0;
    long long hi = 0;
    if (i < s) {
        const long long *p = part + (size_t)c * G * s + i;
#pragma unroll 8
        for (int g = warp; g < G; g += kThreads / 32) {
            const long long v = p[(size_t)g * s];
            const unsigned long long nlo = lo + (unsigned long long)v;
            hi += (v < 0 ? -1 : 0) + (nlo < lo ? 1 : 0);
            lo = nlo;
        }
    }
    slo[threadIdx.x] = lo;
    shi[threadIdx.x] = hi;
    __syncthreads();
    if (warp != 0 || i >= s) return;
    for (int w = 1; w < kThreads / 32; ++w) {
        const unsigned long long nlo = lo + slo[w * 32 + lane];
        hi += shi[w * 32 + lane] + (nlo < lo ? 1 : 0);
        lo = nlo;
    }
    const unsigned k = key[c];
    double r = 0.0;
    if (k != 0u) {
        const bool neg = hi < 0;
        unsigned long long uhi = (unsigned long long)hi;
        if (neg) {
            lo = ~lo + 1ull;
            uhi = ~uhi + (lo == 0ull ? 1ull : 0ull);
        }
        r = (double)uhi * 18446744073709551616.0 + (double)lo;
        const int frac = sketch_fraction_bits_from_limb(limb_bits(*binmax));
        r = scale_pow2(neg ? -r : r, key_bound(k) - frac) / sqrt((double)zeta);
    }
    SX[i + (size_t)c * s] = r;
}

// The three launches: keys [ncols] and part [ncols][G][s] are the caller's.
void sketch_block_launch(const skf_sketch *S, const double *X, int64_t ldx, int ncols, int G, int64_t rows,
                         unsigned *key, long long *part, double *SX, cudaStream_t st) {
    const SparseSign sp = make_sparse_sign(S);
    const int64_t n = S->n;
    // a short column takes one CTA, and the keys need no clearing: such a call is
    // bound by the host (5000 rows, one column, called from Python, against three
    // launches and two allocations: 0.94 of the speed with a clearing and two
    // allocations, 1.02 with neither and one)
    const int64_t wide = std::min<int64_t>((n + 4 * kThreads - 1) / (4 * kThreads), (8ll * num_sms() + ncols - 1) / ncols);
    const unsigned gx = n <= kShortColumn ? 1u : (unsigned)std::max<int64_t>(1, wide);
    if (gx > 1) cudaMemsetAsync(key, 0, sizeof(unsigned) * (size_t)ncols, st);
    for (int c0 = 0; c0 < ncols; c0 += 32768) {   // grid.y limit
        const unsigned nc = (unsigned)std::min(ncols - c0, 32768);
        k_colmax<<<dim3(gx, nc), kThreads, 0, st>>>(X + c0 * ldx, ldx, n, key + c0);
    }
    const int blk = S->zeta == 8 && S->pattern8 != nullptr ? S->p8_block : 0;
    auto kern = blk == 64 ? k_sparse_sign_scatter<64> : blk == 128 ? k_sparse_sign_scatter<128> : k_sparse_sign_scatter<0>;
    const size_t smem = blk == 64 ? ScatterGeom<64>::bytes(S->s) : blk == 128 ? ScatterGeom<128>::bytes(S->s)
                                                                              : ScatterGeom<0>::bytes(S->s);
    if (smem > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<G, kScatterThreads, smem, st>>>(X, ldx, n, ncols, rows, sp, S->pattern, S->pattern8, S->binmax, key, part);
    for (int c0 = 0; c0 < ncols; c0 += 32768) {
        const unsigned nc = (unsigned)std::min(ncols - c0, 32768);
        k_sparse_sign_reduce<<<dim3((unsigned)((S->s + 31) / 32), nc), kThreads, 0, st>>>(
            part + (size_t)c0 * G * S->s, key + c0, G, S->s, S->zeta, S->binmax, SX + (size_t)c0 * S->s);
    }
    count_launches(3);
}

__global__ void k_copy_cols(const double *__restrict__ X, int64_t ldx, int64_t n, int ncols, double *__restrict__ Y) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * ncols) return;
    const int64_t c = idx / n, r = idx % n;
    Y[idx] = X[r + c * ldx];
}

}  // namespace

// Expand the sparse-sign pattern and its bin-load maximum (once per sketch).
skf_status build_sparse_sign_tables(skf_sketch *S, cudaStream_t st) {
    const SparseSign sp = make_sparse_sign(S);
    const size_t bytes = sizeof(uint16_t) * (size_t)S->n * S->zeta;
    cudaError_t e = cudaMalloc(&S->pattern, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        S->pattern = nullptr;
        return fail(SKF_ERR_OOM, "sketch pattern allocation");
    }
    e = cudaMalloc(&S->binmax, 3 * sizeof(int));
    if (e != cudaSuccess) {
        cudaGetLastError();
        S->binmax = nullptr;
        return fail(SKF_ERR_OOM, "sketch table allocation");
    }
    S->binmax_chunk = S->binmax + 1;
    S->binmax_persist = S->binmax + 2;
    int G;
    int64_t rows;
    row_partition(S->n, &G, &rows);
    const int blocks = (int)std::min<int64_t>((S->n + 255) / 256, 16ll * num_sms());
    k_build_pattern<<<blocks, 256, 0, st>>>(sp, S->n, S->pattern);
    cudaMemsetAsync(S->binmax, 0, 3 * sizeof(int), st);
    const size_t smem = sizeof(int) * S->s;
    if (smem > 48 * 1024) cudaFuncSetAttribute(k_bin_max, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_bin_max<<<G, 256, smem, st>>>(sp, S->n, rows, S->pattern, S->binmax);
    int Gc;
    chunk_partition(S->n, &Gc);
    k_bin_max<<<Gc, 256, smem, st>>>(sp, S->n, kChunkRows, S->pattern, S->binmax_chunk);
    int64_t last_rows = 0;   // the persistent partitions, where they differ
    for (int level = 0; level < kPersistLevels; ++level) {
        int Gp;
        int64_t rows_p;
        persist_partition(S->n, level, &Gp, &rows_p);
        if (rows_p == last_rows) continue;
        last_rows = rows_p;
        k_bin_max<<<Gp, 256, smem, st>>>(sp, S->n, rows_p, S->pattern, S->binmax_persist);
        count_launches(1);
    }
    count_launches(3);
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "sketch table build");
    int hmax[3] = {0, 0, 0};
    cudaMemcpy(hmax, S->binmax, 3 * sizeof(int), cudaMemcpyDeviceToHost);
    if (limb_bits(hmax[0]) < 13 || limb_bits(hmax[1]) < 13)
        return fail(SKF_ERR_NOT_SUPPORTED, "sketch too dense for the fixed-point accumulators");
    // the persistent Arnoldi kernel is simply not used for a denser partition
    S->binmax_persist_host = hmax[2];
    if (limb_bits(hmax[2]) < 13) S->binmax_persist = nullptr;
    int max_stripe = 0;
    for (int q = 0; q < sp.zeta; ++q) max_stripe = std::max(max_stripe, sp.size[q]);
    if (max_stripe <= 128 && S->zeta <= 8) {
        if (cudaMalloc(&S->pattern8, (size_t)S->n * 8) == cudaSuccess) {
            S->p8_block = max_stripe <= 64 ? 64 : 128;
            k_build_pattern8<<<blocks, 256, 0, st>>>(sp, S->n, S->p8_block, S->pattern, S->pattern8);
            count_launches(1);
            e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) return cuda_fail(e, "sketch table build");
        } else {
            cudaGetLastError();   // no compact table: the kernels read the 16-bit one
            S->pattern8 = nullptr;
        }
    }
    return SKF_OK;
}

skf_status sketch_apply_f64(const skf_sketch *S, const double *X, int64_t ldx, int ncols, double *SX,
                            cudaStream_t st) {
    const int64_t n = S->n;
    if (ncols <= 0) return SKF_OK;
    if (S->kind == SKF_SKETCH_IDENTITY) {
        const int64_t tot = n * ncols;
        k_copy_cols<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(X, ldx, n, ncols, SX);
        count_launches(1);
        SKF_LAUNCH_CHECK("k_copy_cols");
        return SKF_OK;
    }
    if (S->kind == SKF_SKETCH_SRHT) return srht_apply_f64(S, X, ldx, ncols, SX, st);
    if (S->kind == SKF_SKETCH_SRDCT) return srdct_apply_f64(S, X, ldx, ncols, SX, st);
    if (S->kind != SKF_SKETCH_SPARSE_SIGN) return fail(SKF_ERR_NOT_SUPPORTED, "sketch kind not implemented");
    int G;
    int64_t rows;
    row_partition(n, &G, &rows);
    const size_t szKey = (sizeof(unsigned) * (size_t)ncols + 255) & ~(size_t)255;
    char *ws = nullptr;
    const skf_status stt = dalloc((void **)&ws, szKey + sizeof(long long) * (size_t)G * ncols * S->s, st);
    if (stt != SKF_OK) return stt;
    sketch_block_launch(S, X, ldx, ncols, G, rows, (unsigned *)ws, (long long *)(ws + szKey), SX, st);
    cudaError_t e = cudaGetLastError();
    dfree(ws, st);
    if (e != cudaSuccess) return cuda_fail(e, "sketch_apply kernels");
    return SKF_OK;
}

// ---------------------------------------------------------------------
// Allocation-free variant of sketch_apply_f64.
//
// Some callers cannot allocate device memory at the point where they need a
// sketch: code running inside a memory-budgeted runtime that owns every
// allocation, or code paths that must not touch the allocator or its memory
// pools at all (the allocating path goes through cudaMallocAsync and
// cudaFreeAsync on the library's pool; this one makes no allocator or pool
// call of any kind).  For them the scratch of the column-max / scatter /
// reduce pipeline (a key per column and per-CTA integer partial sums)
// lives in the fixed array below instead of coming from cudaMallocAsync.
//
// kNoAllocScratchBytes bounds G * ncols * (s + 1) * 8 bytes, where G is the
// number of CTAs of the row partition (at most 2 per SM).  The array is a
// module global: every GPU that loads this library keeps it for the life of
// the process, and all calls on a device share it, so calls whose kernels
// may overlap on the GPU (different streams, or different host threads)
// race on it.  Every word a call reads is first written by the same call, so
// nothing has to be cleared between calls.
constexpr size_t kNoAllocScratchBytes = 4u << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_addr[kMaxDevices] = {};

// Device address of g_noalloc_scratch on the current device (set-up once per
// device; cudaGetSymbolAddress is not valid inside a stream capture).
skf_status noalloc_scratch(void **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= kMaxDevices) return fail(SKF_ERR_NOT_SUPPORTED, "device ordinal too large");
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (g_noalloc_addr[dev] == nullptr) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(no-alloc scratch)");
        g_noalloc_addr[dev] = p;
    }
    *out = g_noalloc_addr[dev];
    return SKF_OK;
}

}  // namespace

skf_status sketch_apply_f64_noalloc(const skf_sketch *S, const double *X, int64_t ldx, int ncols, double *SX,
                                    cudaStream_t st) {
    if (S->kind != SKF_SKETCH_SPARSE_SIGN)
        return fail(SKF_ERR_NOT_SUPPORTED, "the allocation-free sketch apply supports the sparse-sign sketch only");
    if (ncols <= 0) return SKF_OK;
    const int64_t n = S->n;
    int G;
    int64_t rows;
    row_partition(n, &G, &rows);
    const size_t need = sizeof(long long) * (size_t)G * ncols * ((size_t)S->s + 1);
    if (need > kNoAllocScratchBytes)
        return fail(SKF_ERR_INVALID_ARG, "allocation-free sketch apply needs " + std::to_string(need) +
                                             " bytes of scratch, more than its fixed " +
                                             std::to_string(kNoAllocScratchBytes) +
                                             " (reduce ncols or s, or use skf_sketch_apply)");
    void *base = nullptr;
    skf_status stt = noalloc_scratch(&base);
    if (stt != SKF_OK) return stt;
    unsigned *key = (unsigned *)base;                                                     // [ncols]
    long long *part = (long long *)((char *)base + sizeof(double) * (size_t)G * ncols);   // [ncols][G][s]
    sketch_block_launch(S, X, ldx, ncols, G, rows, key, part, SX, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "allocation-free sketch_apply kernels");
    return SKF_OK;
}

}  // namespace skf
