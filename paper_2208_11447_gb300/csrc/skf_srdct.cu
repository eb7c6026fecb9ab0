// Subsampled randomized discrete cosine transform (the sketch of the paper's
// experiments, Sec. 5.1: S = P F E with F a DCT):
//   (S x)_i = sqrt(N/s) (F E x)_{P_i},  F the orthonormal DCT-II,
//   (F y)_k = a_k sum_n y_n cos(pi k (2n + 1) / (2N)),  a_0 = 1/sqrt(N), a_k = sqrt(2/N),
// E the signs of the SRHT definition and P the first s entries of its partial
// Fisher-Yates shuffle, of [0, N).
//
// Fast form (N with no prime factor above 7).  Makhoul's reordering (IEEE
// Trans. ASSP 28, 1980) turns the DCT-II into one DFT of length N: with
// v_n = y_{2n} for n < ceil(N/2) and v_{N-1-n} = y_{2n+1} for n < N/2,
// V = DFT_N(v) and (F y)_k = a_k Re(e^{-i pi k / (2N)} V_k), for any N.  v is
// real, so for even N it is packed two to a complex entry, z_n = v_{2n} +
// i v_{2n+1} (n < M = N/2), and only Z = DFT_M(z) is computed: the DFTs of
// the even and odd entries are E_k = (Z_k + conj Z_{M-k}) / 2 and
// O_k = (Z_k - conj Z_{M-k}) / (2i) (indices mod M), V_k = E_k +
// e^{-2 pi i k / N} O_k.  The DFT runs as Stockham autosort passes (one
// launch each, radices 4, 2, 3, 5, 7): pass with radix R and span Ns (the
// product of the earlier radices) reads x_{j + r L/R}, multiplies by
// e^{-2 pi i (j mod Ns) r / (Ns R)}, takes the R-point DFT (radix 3 and 5 in
// the symmetric form: sums and differences of the entries r and R - r) and
// writes it to (j div Ns) Ns R + (j mod Ns) + r Ns, so the output comes out
// in natural order.  Only the s sampled V_k are then formed.  Work per
// vector about 2.5 N log2 N flops instead of 2 s N; the complex buffers
// (2 per column) are the caller's scratch.
//
// Direct form (any other N): each output is a dot product of length N
// against a cosine table of period 4N (cos(pi j / (2N)), j = k (2n + 1) mod
// 4N, advanced by additions): O(s N) work per vector, one CTA per sampled
// row, fixed summation order.
#include <math.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "skf_internal.cuh"

namespace skf {

namespace {

constexpr int kSrdctThreads = 256;
constexpr int kFftThreads = 256;

__device__ __forceinline__ bool srdct_stopped(const SrdctCols &cols) {
    return cols.iscal && cols.iscal[0] && cols.iscal[3] <= cols.step;   // the Arnoldi process stopped
}

// entry r of column q, widened exactly from F32 where the columns are F32
__device__ __forceinline__ double srdct_ld(const SrdctCols &cols, int q, int64_t r) {
    return cols.f32 ? (double)((const float *)cols.x[q])[r] : ((const double *)cols.x[q])[r];
}

__global__ void __launch_bounds__(kSrdctThreads) k_srdct(SrdctDev d, SrdctCols cols) {
    __shared__ double red[64];
    if (srdct_stopped(cols)) return;
    const int i = blockIdx.x;
    const int64_t k = d.P[i];
    const int64_t M4 = 4 * d.n;
    int64_t idx = (k * (2 * (int64_t)threadIdx.x + 1)) % M4;
    const int64_t stp = (2 * k * (int64_t)blockDim.x) % M4;
    double acc[2] = {0.0, 0.0};
    for (int64_t n = threadIdx.x; n < d.n; n += blockDim.x) {
        const double cs = d.costab[idx] * d.E[n];
        acc[0] = fma(srdct_ld(cols, 0, n), cs, acc[0]);
        if (cols.ncols > 1) acc[1] = fma(srdct_ld(cols, 1, n), cs, acc[1]);
        idx += stp;
        if (idx >= M4) idx -= M4;
    }
    block_sum<2>(acc, red);
    if (threadIdx.x == 0) {
        const double sk = sqrt((k == 0 ? 1.0 : 2.0) / (double)d.s);
        for (int q = 0; q < cols.ncols; ++q)
            cols.out[q][i] = acc[q] * sk * (cols.colscale[q] ? *cols.colscale[q] : 1.0);
    }
}

// entry t of Makhoul's reordering v of E x (column q)
__device__ __forceinline__ double makhoul(const SrdctDev &d, const SrdctCols &cols, int q, int64_t t) {
    const int64_t src = t < (d.n + 1) / 2 ? 2 * t : 2 * (d.n - 1 - t) + 1;
    return d.E[src] * srdct_ld(cols, q, src);
}

// the FFT input of column blockIdx.y: z_t = v_{2t} + i v_{2t+1} (even n) or
// v_t (odd n)
__global__ void __launch_bounds__(kFftThreads) k_dct_permute(SrdctDev d, SrdctCols cols, double2 *dst) {
    if (srdct_stopped(cols)) return;
    const int q = blockIdx.y;
    const int64_t L = d.fft_len;
    const bool packed = 2 * L == d.n;
    double2 *z = dst + (size_t)q * L;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < L; t += (int64_t)gridDim.x * blockDim.x)
        z[t] = packed ? make_double2(makhoul(d, cols, q, 2 * t), makhoul(d, cols, q, 2 * t + 1))
                      : make_double2(makhoul(d, cols, q, t), 0.0);
}

// cos and sin of 2 pi k / R, k < R (host-computed)
struct RootTable {
    double c[8], s[8];
};

// R-point DFT o_t = sum_r v_r e^{-2 pi i r t / R}
template <int R>
__device__ __forceinline__ void dft_point(const double2 (&v)[R], double2 (&o)[R], const RootTable &rt) {
    if constexpr (R == 2) {
        o[0] = make_double2(v[0].x + v[1].x, v[0].y + v[1].y);
        o[1] = make_double2(v[0].x - v[1].x, v[0].y - v[1].y);
    } else if constexpr (R == 4) {
        const double2 t0 = make_double2(v[0].x + v[2].x, v[0].y + v[2].y);
        const double2 t1 = make_double2(v[0].x - v[2].x, v[0].y - v[2].y);
        const double2 t2 = make_double2(v[1].x + v[3].x, v[1].y + v[3].y);
        const double2 t3 = make_double2(v[1].x - v[3].x, v[1].y - v[3].y);
        o[0] = make_double2(t0.x + t2.x, t0.y + t2.y);
        o[2] = make_double2(t0.x - t2.x, t0.y - t2.y);
        o[1] = make_double2(t1.x + t3.y, t1.y - t3.x);   // t1 - i t3
        o[3] = make_double2(t1.x - t3.y, t1.y + t3.x);   // t1 + i t3
    } else if constexpr (R == 3) {
        // o_0 = v0 + t1, o_{1,2} = (v0 - t1 / 2) -/+ i sin(2 pi / 3) t2, t1 = v1 + v2, t2 = v1 - v2
        const double2 t1 = make_double2(v[1].x + v[2].x, v[1].y + v[2].y);
        const double2 t2 = make_double2(v[1].x - v[2].x, v[1].y - v[2].y);
        const double2 a = make_double2(fma(-0.5, t1.x, v[0].x), fma(-0.5, t1.y, v[0].y));
        const double2 b = make_double2(rt.s[1] * t2.x, rt.s[1] * t2.y);
        o[0] = make_double2(v[0].x + t1.x, v[0].y + t1.y);
        o[1] = make_double2(a.x + b.y, a.y - b.x);   // a - i b
        o[2] = make_double2(a.x - b.y, a.y + b.x);   // a + i b
    } else if constexpr (R == 5) {
        // t1 = v1 + v4, t2 = v2 + v3, t3 = v1 - v4, t4 = v2 - v3;
        // o_{1,4} = v0 + c1 t1 + c2 t2 -/+ i (s1 t3 + s2 t4),
        // o_{2,3} = v0 + c2 t1 + c1 t2 -/+ i (s2 t3 - s1 t4)  (c_k, s_k: cos, sin of 2 pi k / 5)
        const double2 t1 = make_double2(v[1].x + v[4].x, v[1].y + v[4].y);
        const double2 t2 = make_double2(v[2].x + v[3].x, v[2].y + v[3].y);
        const double2 t3 = make_double2(v[1].x - v[4].x, v[1].y - v[4].y);
        const double2 t4 = make_double2(v[2].x - v[3].x, v[2].y - v[3].y);
        const double c1 = rt.c[1], c2 = rt.c[2], s1 = rt.s[1], s2 = rt.s[2];
        const double2 a1 = make_double2(fma(c2, t2.x, fma(c1, t1.x, v[0].x)), fma(c2, t2.y, fma(c1, t1.y, v[0].y)));
        const double2 a2 = make_double2(fma(c1, t2.x, fma(c2, t1.x, v[0].x)), fma(c1, t2.y, fma(c2, t1.y, v[0].y)));
        const double2 b1 = make_double2(fma(s2, t4.x, s1 * t3.x), fma(s2, t4.y, s1 * t3.y));
        const double2 b2 = make_double2(fma(-s1, t4.x, s2 * t3.x), fma(-s1, t4.y, s2 * t3.y));
        o[0] = make_double2(v[0].x + t1.x + t2.x, v[0].y + t1.y + t2.y);
        o[1] = make_double2(a1.x + b1.y, a1.y - b1.x);
        o[4] = make_double2(a1.x - b1.y, a1.y + b1.x);
        o[2] = make_double2(a2.x + b2.y, a2.y - b2.x);
        o[3] = make_double2(a2.x - b2.y, a2.y + b2.x);
    } else {
        // direct R-point DFT: o_t = sum_q v_q e^{-2 pi i q t / R}
    #pragma unroll
        for (int t = 0; t < R; ++t) {
            double re = v[0].x, im = v[0].y;
    #pragma unroll
            for (int q = 1; q < R; ++q) {
                const int e = (q * t) % R;
                re = fma(v[q].x, rt.c[e], fma(v[q].y, rt.s[e], re));
                im = fma(v[q].y, rt.c[e], fma(-v[q].x, rt.s[e], im));
            }
            o[t] = make_double2(re, im);
        }
    }
}

// one Stockham pass of radix R over each column (blockIdx.y)
// (length n; the twiddle table holds e^{-2 pi i t / (n twstride)})
template <int R>
__global__ void __launch_bounds__(kFftThreads) k_fft_pass(int64_t n, int64_t ns, const double2 *__restrict__ tw,
                                                         int64_t twstride, RootTable rt,
                                                         const double2 *__restrict__ src, double2 *__restrict__ dst,
                                                         SrdctCols cols) {
    if (srdct_stopped(cols)) return;
    src += (size_t)blockIdx.y * n;
    dst += (size_t)blockIdx.y * n;
    const int64_t nr = n / R;
    // twiddle index step: e^{-2 pi i k r / (ns R)} = tw[k r tstep]
    const int64_t tstep = n / (ns * R) * twstride;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nr; j += (int64_t)gridDim.x * blockDim.x) {
        double2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = src[j + r * nr];
        const int64_t k = j % ns;
#pragma unroll
        for (int r = 1; r < R; ++r) {
            const double2 w = tw[k * r * tstep];   // k r < ns R: the index stays below n twstride
            const double re = fma(v[r].x, w.x, -v[r].y * w.y);
            const double im = fma(v[r].x, w.y, v[r].y * w.x);
            v[r] = make_double2(re, im);
        }
        double2 o[R];
        dft_point<R>(v, o, rt);
        const int64_t base = (j / ns) * ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) dst[base + r * ns] = o[r];
    }
}

// V_k = E_k + e^{-2 pi i k / n} O_k from z1 = Z_{k mod M}, z2 = Z_{M - k mod M} (even n)
__device__ __forceinline__ double2 unpack_v(double2 z1, double2 z2, double2 w) {
    const double2 e = make_double2(0.5 * (z1.x + z2.x), 0.5 * (z1.y - z2.y));    // z2 enters conjugated
    const double2 o = make_double2(0.5 * (z1.y + z2.y), -0.5 * (z1.x - z2.x));   // (z1 - conj z2) / (2i)
    return make_double2(e.x + fma(w.x, o.x, -w.y * o.y), e.y + fma(w.x, o.y, w.y * o.x));
}

// out[q][i] = colscale Re(twist_i V_k), k = P_i; V_k from the FFT output Z
// (even n: V_k = E_k + e^{-2 pi i k / n} O_k from Z_{k mod M} and Z_{M - k mod M})
__global__ void __launch_bounds__(kFftThreads) k_dct_gather(SrdctDev d, SrdctCols cols, const double2 *Zall) {
    if (srdct_stopped(cols)) return;
    const int q = blockIdx.y;
    const int64_t L = d.fft_len;
    const double2 *Z = Zall + (size_t)q * L;
    const double cscale = cols.colscale[q] ? *cols.colscale[q] : 1.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.s; i += gridDim.x * blockDim.x) {
        const int64_t k = d.P[i];
        double2 V;
        if (2 * L == d.n) {
            const int64_t kk = k % L, kc = (L - kk) % L;
            V = unpack_v(Z[kk], Z[kc], d.tw[k]);
        } else {
            V = Z[k];
        }
        const double2 t = d.twist[i];
        cols.out[q][i] = fma(t.x, V.x, -t.y * V.y) * cscale;
    }
}

// Pruned form (fft_p1 > 0): only s outputs of the transform are wanted, so its
// passes stop at span P1 = fft_p1 (the product of the first radices) and the
// remaining P2 = L / P1 terms of each wanted output are summed directly:
//   Z_k = sum_{q < P2} Y_{(k mod P1) + q P1} e^{-2 pi i q k / L},
// Y the array after the passes of span P1.  Those passes run in shared memory,
// one CTA per T residues j (the P1-point DFTs of the entries j + r P2), with
// the reordering on load: one launch and 16 L bytes written instead of a
// launch and 32 L bytes per radix, and about log P1 / log L of the flops.
// N = 3.6e5, s = 240, one column: 11 launches, 57 us, before; 23 + 12 us now.
constexpr int kGroupThreads = 256;
constexpr size_t kGroupSmem = 72 * 1024;    // of one CTA (three per SM)
constexpr int kGroupMax = 1024;             // largest P1
struct RootTables {
    RootTable r[8];   // by radix
};

template <int R>
__device__ __forceinline__ void group_pass(const double2 *__restrict__ src, double2 *__restrict__ dst, int P, int T,
                                           int ns, const double2 *__restrict__ tw, int64_t twn, const RootTable &rt) {
    const int nr = P / R;
    const int64_t tstep = twn / ((int64_t)ns * R);   // e^{-2 pi i k r / (ns R)} = tw[k r tstep]
    for (int x = threadIdx.x; x < nr * T; x += kGroupThreads) {
        const int jj = x / T, tj = x - jj * T;
        const int hi = jj / ns, k = jj - hi * ns;
        double2 v[R], o[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = src[(jj + r * nr) * T + tj];
        if (ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                const double2 w = __ldg(tw + (int64_t)(k * r) * tstep);
                v[r] = make_double2(fma(v[r].x, w.x, -v[r].y * w.y), fma(v[r].x, w.y, v[r].y * w.x));
            }
        }
        dft_point<R>(v, o, rt);
#pragma unroll
        for (int r = 0; r < R; ++r) dst[(hi * ns * R + k + r * ns) * T + tj] = o[r];
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kGroupThreads) k_dct_group(SrdctDev d, SrdctCols cols, int T, RootTables rts,
                                                             double2 *__restrict__ Yall) {
    extern __shared__ __align__(16) double2 gsm[];
    if (srdct_stopped(cols)) return;
    const int q = blockIdx.y;
    const int P = d.fft_p1;
    const int64_t L = d.fft_len, P2 = L / P;
    const bool packed = 2 * L == d.n;
    const int64_t j0 = (int64_t)blockIdx.x * T;
    const int tn = (int)min((int64_t)T, P2 - j0);
    double2 *a = gsm, *b = gsm + (size_t)P * T;
    for (int x = threadIdx.x; x < P * T; x += kGroupThreads) {
        const int r = x / T, tj = x - r * T;
        double2 z = make_double2(0.0, 0.0);
        if (tj < tn) {
            const int64_t t = j0 + tj + (int64_t)r * P2;
            z = packed ? make_double2(makhoul(d, cols, q, 2 * t), makhoul(d, cols, q, 2 * t + 1))
                       : make_double2(makhoul(d, cols, q, t), 0.0);
        }
        a[x] = z;
    }
    __syncthreads();
    int ns = 1;
    for (int p = 0; ns < P; ++p) {
        const int R = d.rad[p];
        switch (R) {
            case 2: group_pass<2>(a, b, P, T, ns, d.tw, d.n, rts.r[2]); break;
            case 3: group_pass<3>(a, b, P, T, ns, d.tw, d.n, rts.r[3]); break;
            case 4: group_pass<4>(a, b, P, T, ns, d.tw, d.n, rts.r[4]); break;
            case 5: group_pass<5>(a, b, P, T, ns, d.tw, d.n, rts.r[5]); break;
            default: group_pass<7>(a, b, P, T, ns, d.tw, d.n, rts.r[7]); break;
        }
        ns *= R;
        double2 *t = a;
        a = b;
        b = t;
    }
    double2 *Y = Yall + (size_t)q * L + j0 * P;
    for (int x = threadIdx.x; x < P * tn; x += kGroupThreads) {
        const int tj = x / P, r = x - tj * P;
        Y[x] = a[r * T + tj];
    }
}

// out[q][i] from Y, one CTA per sampled row: Z_k and, packed, Z_{L-k}.  The
// P2 terms are dealt out over the CTA's threads (gathers of one 16-byte entry
// of Y and one of the table each; a warp per row took 31 us, latency-bound).
constexpr int kDotThreads = 128;
__global__ void __launch_bounds__(kDotThreads) k_dct_dots(SrdctDev d, SrdctCols cols, const double2 *__restrict__ Yall) {
    __shared__ double red[4][kDotThreads / 32];
    if (srdct_stopped(cols)) return;
    const int i = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = blockIdx.y, P = d.fft_p1;
    const int64_t L = d.fft_len, P2 = L / P, tws = d.n / L;
    const double2 *Y = Yall + (size_t)q * L;
    const bool packed = 2 * L == d.n;
    const int64_t k = d.P[i], kk = k % L, kc = packed ? (L - kk) % L : kk;
    const double2 *y0 = Y + kk % P, *y1 = Y + kc % P;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    int64_t e = (kk * threadIdx.x) % L;
    const int64_t de = (kk * kDotThreads) % L;
#pragma unroll 4
    for (int64_t p = threadIdx.x; p < P2; p += kDotThreads) {
        // the table entry of L - k is the conjugate of that of k
        const double2 a = __ldg(y0 + p * P), b = __ldg(y1 + p * P), w = __ldg(d.tw + e * tws);
        v[0] = fma(a.x, w.x, fma(-a.y, w.y, v[0]));
        v[1] = fma(a.x, w.y, fma(a.y, w.x, v[1]));
        v[2] = fma(b.x, w.x, fma(b.y, w.y, v[2]));
        v[3] = fma(-b.x, w.y, fma(b.y, w.x, v[3]));
        e += de;
        if (e >= L) e -= L;
    }
#pragma unroll
    for (int h = 0; h < 4; ++h) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[h] += __shfl_xor_sync(0xffffffffu, v[h], o);
        if (lane == 0) red[h][warp] = v[h];
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
#pragma unroll
    for (int h = 0; h < 4; ++h) v[h] = (red[h][0] + red[h][1]) + (red[h][2] + red[h][3]);
    double2 V = make_double2(v[0], v[1]);
    if (packed) V = unpack_v(V, make_double2(v[2], v[3]), d.tw[k]);
    const double2 t = d.twist[i];
    cols.out[q][i] = fma(t.x, V.x, -t.y * V.y) * (cols.colscale[q] ? *cols.colscale[q] : 1.0);
}

RootTable root_table(int R) {
    RootTable rt{};
    for (int k = 0; k < R; ++k) {
        const double a = 2.0 * M_PI * (double)k / (double)R;
        rt.c[k] = cos(a);
        rt.s[k] = sin(a);
    }
    return rt;
}

void fft_launch(const SrdctDev &d, const SrdctCols &cols, cudaStream_t st) {
    const int64_t n = d.fft_len;
    const int64_t twstride = d.n / n;
    double2 *a = d.work, *b = d.work + 2 * (size_t)n;
    const unsigned ny = (unsigned)cols.ncols;
    if (d.fft_p1 > 0) {
        // T residues per CTA: about three CTAs per SM (their passes are latency-bound),
        // within kGroupSmem of shared memory
        const int64_t p2 = n / d.fft_p1;
        const int64_t fit = (int64_t)(kGroupSmem / (2 * sizeof(double2) * (size_t)d.fft_p1));
        const int T = (int)std::max<int64_t>(1, std::min<int64_t>(fit, (p2 * ny + 3 * num_sms() - 1) / (3 * num_sms())));
        const size_t smem = 2 * sizeof(double2) * (size_t)d.fft_p1 * T;
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(k_dct_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        RootTables rts{};
        for (int R : {2, 3, 4, 5, 7}) rts.r[R] = root_table(R);
        k_dct_group<<<dim3((unsigned)((p2 + T - 1) / T), ny), kGroupThreads, smem, st>>>(d, cols, T, rts, a);
        k_dct_dots<<<dim3((unsigned)d.s, ny), kDotThreads, 0, st>>>(d, cols, a);
        count_launches(2);
        return;
    }
    auto grid = [&](int64_t items) {
        return dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>((items + kFftThreads - 1) / kFftThreads,
                                                                       8ll * num_sms())), ny);
    };
    k_dct_permute<<<grid(n), kFftThreads, 0, st>>>(d, cols, a);
    int64_t ns = 1;
    for (int p = 0; p < d.nrad; ++p) {
        const int R = d.rad[p];
        const RootTable rt = root_table(R);
        const dim3 g = grid(n / R);
        switch (R) {
            case 2: k_fft_pass<2><<<g, kFftThreads, 0, st>>>(n, ns, d.tw, twstride, rt, a, b, cols); break;
            case 3: k_fft_pass<3><<<g, kFftThreads, 0, st>>>(n, ns, d.tw, twstride, rt, a, b, cols); break;
            case 4: k_fft_pass<4><<<g, kFftThreads, 0, st>>>(n, ns, d.tw, twstride, rt, a, b, cols); break;
            case 5: k_fft_pass<5><<<g, kFftThreads, 0, st>>>(n, ns, d.tw, twstride, rt, a, b, cols); break;
            default: k_fft_pass<7><<<g, kFftThreads, 0, st>>>(n, ns, d.tw, twstride, rt, a, b, cols); break;
        }
        ns *= R;
        std::swap(a, b);
    }
    k_dct_gather<<<grid(d.s), kFftThreads, 0, st>>>(d, cols, a);
    count_launches(2 + d.nrad);
}

}  // namespace

size_t srdct_work_bytes(const skf_sketch *S) {
    return S->fft_len > 0 ? sizeof(double2) * 4 * (size_t)S->fft_len : 0;
}

SrdctDev make_srdct(const skf_sketch *S) {
    SrdctDev d{};
    d.n = S->n;
    d.s = S->s;
    d.P = S->P;
    d.E = S->E;
    d.costab = S->costab;
    d.fft_len = S->fft_len;
    d.nrad = S->nrad;
    d.fft_p1 = S->fft_p1;
    for (int i = 0; i < S->nrad; ++i) d.rad[i] = S->rad[i];
    d.tw = S->tw;
    d.twist = S->twist;
    d.work = nullptr;
    return d;
}

skf_status build_srdct_tables(skf_sketch *S) {
    if ((int64_t)S->s > S->n) return fail(SKF_ERR_INVALID_ARG, "SRDCT needs s <= N");
    S->np = S->n;
    skf_status st = build_sampled_rows(S, S->n);
    if (st != SKF_OK) return st;
    const int64_t n = S->n;
    std::vector<double> E((size_t)n);
    for (int64_t c = 0; c < n; ++c) E[c] = (splitmix_word(S->seed, (uint64_t)c) & 1ull) ? -1.0 : 1.0;
    if (cudaMalloc(&S->E, sizeof(double) * n) != cudaSuccess) {
        cudaGetLastError();
        return fail(SKF_ERR_OOM, "SRDCT table allocation");
    }
    if (cudaMemcpy(S->E, E.data(), sizeof(double) * n, cudaMemcpyHostToDevice) != cudaSuccess)
        return cuda_fail(cudaGetLastError(), "SRDCT table upload");
    // FFT length (real input packed two to an entry for even n); radices 4
    // first, then 2, 3, 5, 7; the FFT form if nothing is left over
    const int64_t len = (n % 2 == 0) ? n / 2 : n;
    int64_t rest = len;
    int nrad = 0;
    int rad[64];
    for (int p : {4, 2, 3, 5, 7})
        while (rest % p == 0 && rest > 1 && nrad < 64) {
            rad[nrad++] = p;
            rest /= p;
        }
    if (rest == 1 && n >= 2) {
        S->fft_len = len;
        S->nrad = nrad;
        for (int i = 0; i < nrad; ++i) S->rad[i] = rad[i];
        // pruned form: P1 = the most leading radices whose product stays within
        // kGroupMax, where summing the rest directly (8 s P2 FMAs with the pair of
        // outputs) costs less than the passes it replaces (about 2.5 L log2 P2 FMAs).
        // 20 Arnoldi steps, full passes / pruned: N = 4e4 1.83 / 1.15 ms at s = 240,
        // 1.89 / 1.30 at s = 800 (1200: full); N = 3.6e5 2.54 / 1.56 and 2.55 / 1.79;
        // N = 1e6 4.38 / 2.88 and 4.41 / 3.14, at s = 2000 4.45 / 3.56
        int64_t p1 = 1;
        for (int i = 0; i < nrad && p1 * rad[i] <= kGroupMax; ++i) p1 *= rad[i];
        const int64_t p2 = len / p1;
        if (p2 == 1 || 8.0 * S->s * (double)p2 <= 2.5 * (double)len * std::log2((double)p2)) S->fft_p1 = (int)p1;
        std::vector<double2> tw((size_t)n), twist((size_t)S->s);
        for (int64_t t = 0; t < n; ++t) {
            const double a = 2.0 * M_PI * ((double)t / (double)n);
            tw[t] = make_double2(cos(a), -sin(a));
        }
        std::vector<int32_t> P((size_t)S->s);
        if (cudaMemcpy(P.data(), S->P, sizeof(int32_t) * S->s, cudaMemcpyDeviceToHost) != cudaSuccess)
            return cuda_fail(cudaGetLastError(), "SRDCT sampled rows");
        for (int i = 0; i < S->s; ++i) {
            const int64_t k = P[i];
            const double a = M_PI * (double)k / (2.0 * (double)n);
            const double sc = sqrt((k == 0 ? 1.0 : 2.0) / (double)S->s);   // a_k sqrt(N / s)
            twist[i] = make_double2(cos(a) * sc, -sin(a) * sc);
        }
        if (cudaMalloc(&S->tw, sizeof(double2) * n) != cudaSuccess ||
            cudaMalloc(&S->twist, sizeof(double2) * S->s) != cudaSuccess) {
            cudaGetLastError();
            return fail(SKF_ERR_OOM, "SRDCT FFT table allocation");
        }
        if (cudaMemcpy(S->tw, tw.data(), sizeof(double2) * n, cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(S->twist, twist.data(), sizeof(double2) * S->s, cudaMemcpyHostToDevice) != cudaSuccess)
            return cuda_fail(cudaGetLastError(), "SRDCT FFT table upload");
        return SKF_OK;
    }
    std::vector<double> tab((size_t)(4 * n));
    for (int64_t j = 0; j < 4 * n; ++j) tab[j] = cos(M_PI * (double)j / (2.0 * (double)n));
    if (cudaMalloc(&S->costab, sizeof(double) * 4 * n) != cudaSuccess) {
        cudaGetLastError();
        return fail(SKF_ERR_OOM, "SRDCT table allocation");
    }
    if (cudaMemcpy(S->costab, tab.data(), sizeof(double) * 4 * n, cudaMemcpyHostToDevice) != cudaSuccess)
        return cuda_fail(cudaGetLastError(), "SRDCT table upload");
    return SKF_OK;
}

void srdct_launch(const SrdctDev &d, const SrdctCols &cols, cudaStream_t st) {
    if (d.fft_len > 0 && d.work != nullptr) {
        fft_launch(d, cols, st);
        return;
    }
    k_srdct<<<d.s, kSrdctThreads, 0, st>>>(d, cols);
    count_launches(1);
}

skf_status srdct_apply_f64(const skf_sketch *S, const double *X, int64_t ldx, int ncols, double *SX,
                           cudaStream_t st) {
    SrdctDev d = make_srdct(S);
    const size_t wb = srdct_work_bytes(S);
    if (wb > 0) {
        skf_status e = dalloc((void **)&d.work, wb, st);
        if (e != SKF_OK) return e;
    }
    for (int c0 = 0; c0 < ncols; c0 += 2) {
        SrdctCols cols{};
        cols.ncols = ncols - c0 < 2 ? ncols - c0 : 2;
        for (int q = 0; q < cols.ncols; ++q) {
            cols.x[q] = X + (size_t)(c0 + q) * ldx;
            cols.out[q] = SX + (size_t)(c0 + q) * S->s;
        }
        srdct_launch(d, cols, st);
    }
    if (d.work) dfree(d.work, st);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "SRDCT kernels");
    return SKF_OK;
}

}  // namespace skf
