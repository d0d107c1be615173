// fc_kernels.cu -- CUDA kernels of the Feldman-Cousins grid fit (all steps but
// the tensor-core screen, which lives in fc_screen.cu).
//
// Method (§2, Algorithm 1, Algorithm 2, Eq. 1): per universe, fluctuate the
// true point's spectrum, scan every grid spectrum with chi2 = r^T A r
// (r = s_g - d, A = M^-1), keep the first minimum, refit M at the minimum and
// rescan until the minimum repeats, then dchi2 = chi2(p) - chi2_min under the
// last scan's A.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cooperative_groups.h>
#include <float.h>
#include <math_constants.h>

#include <algorithm>
#include <cstdint>

#include "fc_df.cuh"
#include "fc_internal.cuh"
#include "fc_sampler.cuh"
#include "fc_spec.cuh"

namespace fcdev {

namespace {

constexpr int kThreads = 256;
constexpr int kResolveMaxN = 64;  // a fit-space matrix is staged in shared memory up to this N_fit

inline unsigned blocks_for(int64_t n, int t = kThreads) {
    int64_t b = (n + t - 1) / t;
    if (b < 1) b = 1;
    if (b > 2147483647LL) b = 2147483647LL;
    return (unsigned)b;
}

// (value, index) lexicographic minimum across a warp
__device__ __forceinline__ void warp_argmin(double& v, int32_t& g) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int32_t og = __shfl_xor_sync(0xffffffffu, g, o);
        if (ov < v || (ov == v && og < g)) {
            v = ov;
            g = og;
        }
    }
}

// The plain path's residual form ||W r||^2 (r = s - d, A = W^T W, W lower
// triangular) in binary64, spread over a warp: lanes form the row dot products
// t_i = sum_{j<=i} W_ij r_j (each summed over j in increasing order with fma),
// lane 0 sums t_i^2 in row order with fma.
// r and t are this warp's shared-memory vectors; the result is lane 0's.
__device__ double resid_chi2_warp(const double* __restrict__ W, int n, const double* r, double* t, int lane) {
    for (int i = lane; i < n; i += 32) {
        const double* Wi = W + i * n;
        double x = 0.0;
        for (int j = 0; j <= i; ++j) x = fma(Wi[j], r[j], x);
        t[i] = x;
    }
    __syncwarp();
    double acc = 0.0;
    if (lane == 0)
        for (int i = 0; i < n; ++i) acc = fma(t[i], t[i], acc);
    __syncwarp();
    return acc;
}

// The mixed path's residual chi2 = |W (s - d)|^2 in double-float (fc_df.cuh):
// r_j = s_j - d_j, t_i = sum_j W_ij r_j, chi2 = sum_i t_i^2 in increasing i.
// Every mixed-path kernel evaluates it in this order, so a universe's result
// has the same bits whichever certified round decided it.  W and s are
// double-float copies of the binary64 arrays; the value is returned as
// binary64.
// Row i of W r: four interleaved partial sums (j = 0, 1, 2, 3 mod 4, each in
// increasing j), combined as (p0 + p1) + (p2 + p3) and renormalised.  A row
// runs over whole blocks of four columns; W is lower triangular and W and r
// are zero past N_fit, so columns past the diagonal add exact zeros and it
// does not matter how many of them a kernel takes.
// Sums 0 and 2 share a packed pair and so do 1 and 3 (df2x): a block of four
// columns is two packed multiply-adds, and (p0 + p1, p2 + p3) is one packed
// add.  Both operands are stored for that, eight floats per block of columns
// j..j+3: (hi_j, hi_j+2), (lo_j, lo_j+2), (hi_j+1, hi_j+3), (lo_j+1, lo_j+3).
__host__ __device__ __forceinline__ int df_blocks(int n) { return (n + 3) / 4; }
// float position of column j's hi half inside a blocked row (the lo half is two floats on)
__device__ __forceinline__ int df_pos(int j) { return (j >> 2) * 8 + (j & 1) * 4 + ((j >> 1) & 1); }

// W of a slot: block jb of row i at float4 index (jb n + i) 2 (k_wdf), so the
// lanes of a warp that hold consecutive rows read consecutive memory.
__device__ __forceinline__ size_t wdf_floats(int n) { return (size_t)df_blocks(n) * n * 8; }

// (p0 + p1) + (p2 + p3) of the packed sums (0, 2) and (1, 3)
__device__ __forceinline__ float2 df_row_sum(df2x s02, df2x s13) {
    const df2x h = df2_add(df2_norm(s02), df2_norm(s13));
    return df_add(make_float2(x2_lo(h.x), x2_lo(h.y)), make_float2(x2_hi(h.x), x2_hi(h.y)));
}

// One thread per residual, N_fit <= NR, the residual vector in registers
// (every index of it a compile-time constant; a block of columns runs only
// when the row reaches it, a branch that is uniform across the warp because
// all its lanes walk the same rows).  W: the slot's blocked W in shared
// memory, read as one broadcast of 16 bytes per packed multiply-add.
template <int NR, class SRow>
__device__ __forceinline__ double resid_df_reg(const ulonglong2* __restrict__ W, int n, const SRow& s,
                                               const float* __restrict__ du) {
    static_assert(NR % 4 == 0, "NR is a multiple of 4");
    f32x2 rx[NR / 2], ry[NR / 2];  // [2 jb + h]: columns 4 jb + h and 4 jb + h + 2
#pragma unroll
    for (int k = 0; k < NR / 2; ++k) {
        const int j = (k >> 1) * 4 + (k & 1);
        const float2 a = (j < n) ? df_sub_f(s[j], du[j]) : make_float2(0.0f, 0.0f);
        const float2 b = (j + 2 < n) ? df_sub_f(s[j + 2], du[j + 2]) : make_float2(0.0f, 0.0f);
        rx[k] = x2_pack(a.x, b.x);
        ry[k] = x2_pack(a.y, b.y);
    }
    float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        const ulonglong2* Wi = W + 2 * i;
        const int last = i >> 2;
        df2x s02{0ull, 0ull}, s13{0ull, 0ull};
#pragma unroll
        for (int jb = 0; jb < NR / 4; ++jb) {
            if (jb <= last) {
                const ulonglong2 w0 = Wi[jb * 2 * n], w1 = Wi[jb * 2 * n + 1];
                s02 = df2_fma(s02, w0.x, w0.y, rx[2 * jb], ry[2 * jb]);
                s13 = df2_fma(s13, w1.x, w1.y, rx[2 * jb + 1], ry[2 * jb + 1]);
            }
        }
        const float2 t = df_row_sum(s02, s13);
        acc = df_fma(acc, t, t);
    }
    return df_to(df_norm(acc.x, acc.y));
}

// One warp per group of up to B residuals under one W (any N_fit): each lane
// owns a row of W, 32 rows at a time, and every W block it loads meets the B
// residual vectors, which wait in the warp's shared memory; lane k then sums
// residual k's t_i^2.  This is the form for few residuals, for covariances
// with few residuals each and for N_fit > 64: a residual is spread over the
// warp, W is read coalesced and once per group, and nothing lives in local
// memory.  Bound by the binary32 pipe (63 % active at N = 120) when there are
// enough groups, else by the latency of one group.  Against one thread per residual everywhere: a
// scan of 4096 data sets on 141x141 1.15 -> 0.76 ms, one point of 25x25 x 1000
// universes 2.59 -> 1.88 ms, 4 points of 27^3 with N = 200 61.3 -> 49.6 ms.
constexpr int kRowsB = 4;       // residuals of a group
constexpr int kRowsWarps = 4;   // warps of a CTA of the row kernels
// shared memory of one warp, in floats: kRowsB blocked residual vectors and row sums
__host__ __device__ __forceinline__ int rows_floats(int n) { return kRowsB * df_blocks(n) * 8 + kRowsB * df_blocks(n) * 8; }
__host__ __forceinline__ size_t rows_smem(int n) { return (size_t)kRowsWarps * rows_floats(n) * sizeof(float); }

// residual vector k of a group into the warp's shared memory sr (zero past N_fit)
template <class SRow>
__device__ __forceinline__ void rows_stage(float* sr, int k, int n, const SRow& s, const float* __restrict__ du,
                                           int lane) {
    float* r = sr + k * df_blocks(n) * 8;
    for (int j = lane; j < df_blocks(n) * 4; j += 32) {
        const float2 v = (j < n) ? df_sub_f(s[j], du[j]) : make_float2(0.0f, 0.0f);
        r[df_pos(j)] = v.x;
        r[df_pos(j) + 2] = v.y;
    }
}

template <int B>
__device__ __forceinline__ void rows_products(const ulonglong2* __restrict__ W, int n, const ulonglong2* sr, float4* st,
                                              int lane) {
    const int nb = df_blocks(n);
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const ulonglong2* Wi = W + 2 * (i < n ? i : n - 1);
        const int nblk = min(nb, (i0 + 31) / 4 + 1);
        constexpr int kAhead = B > 2 ? 2 : 4;
        df2x s02[B], s13[B];
#pragma unroll
        for (int k = 0; k < B; ++k) s02[k] = s13[k] = df2x{0ull, 0ull};
        // kAhead blocks of W are on their way while as many are used (past the last one, the last again):
        // a warp alone on its scheduler waits for W, not for the pipe (a block ahead only: residuals of the
        // 25x25 point 28 instead of 17 us a launch, of N = 200 289 instead of 134)
        ulonglong2 w[2 * kAhead];
        auto fetch = [&](int jb) {
#pragma unroll
            for (int h = 0; h < kAhead; ++h) {
                const ulonglong2* p = Wi + (size_t)min(jb + h, nblk - 1) * 2 * n;
                w[2 * h] = __ldg(p);
                w[2 * h + 1] = __ldg(p + 1);
            }
        };
        fetch(0);
        for (int jb = 0; jb < nblk; jb += kAhead) {
            ulonglong2 c[2 * kAhead];
#pragma unroll
            for (int h = 0; h < 2 * kAhead; ++h) c[h] = w[h];
            if (jb + kAhead < nblk) fetch(jb + kAhead);
#pragma unroll
            for (int h = 0; h < kAhead; ++h) {
                if (jb + h >= nblk) break;
#pragma unroll
                for (int k = 0; k < B; ++k) {
                    const ulonglong2 r0 = sr[(k * nb + jb + h) * 2], r1 = sr[(k * nb + jb + h) * 2 + 1];
                    s02[k] = df2_fma(s02[k], c[2 * h].x, c[2 * h].y, r0.x, r0.y);
                    s13[k] = df2_fma(s13[k], c[2 * h + 1].x, c[2 * h + 1].y, r1.x, r1.y);
                }
            }
        }
        if (i < n) {
            // t_i^2 as the product and its error term, the part of df_fma that needs no order
#pragma unroll
            for (int k = 0; k < B; ++k) {
                const float2 t = df_row_sum(s02[k], s13[k]);
                const float p = __fmul_rn(t.x, t.x);
                float e = __fmaf_rn(t.x, t.x, -p);
                e = __fmaf_rn(t.x, t.y, e);
                e = __fmaf_rn(t.y, t.x, e);
                reinterpret_cast<float2*>(st)[k * nb * 4 + i] = make_float2(p, e);
            }
        }
    }
}

// chi2 of the m <= kRowsB staged residuals; residual k's value is lane k's
// result.  sm: the warp's shared memory (rows_floats), its vectors staged.
__device__ __forceinline__ double rows_chi2(const float* __restrict__ Wslot, int n, float* sm, int m, int lane) {
    const int nb = df_blocks(n);
    const ulonglong2* W = reinterpret_cast<const ulonglong2*>(Wslot);
    const ulonglong2* sr = reinterpret_cast<const ulonglong2*>(sm);
    float4* st = reinterpret_cast<float4*>(sm + kRowsB * nb * 8);
    __syncwarp();
    if (m <= 1)
        rows_products<1>(W, n, sr, st, lane);
    else if (m <= 2)
        rows_products<2>(W, n, sr, st, lane);
    else
        rows_products<kRowsB>(W, n, sr, st, lane);
    __syncwarp();
    float2 acc = make_float2(0.0f, 0.0f);
    if (lane < m) {
        const float2* t = reinterpret_cast<const float2*>(st) + lane * nb * 4;
#pragma unroll 4
        for (int i = 0; i < n; ++i) {
            const float2 pe = t[i];
            float s, err;
            two_sum(acc.x, pe.x, s, err);
            acc = make_float2(s, __fadd_rn(acc.y, __fadd_rn(err, pe.y)));
        }
    }
    __syncwarp();  // the shared memory may be staged again
    return df_to(df_norm(acc.x, acc.y));
}

// Row g of s for the residual routines (g = -1: the centre).  The kernels that
// score residuals are instantiated twice: MODEL = false reads the stored
// double-float rows through a plain pointer, MODEL = true (a recomputed grid)
// evaluates the shape model through a DfRow.  Both feed the same routines, so
// the bits agree and the stored path carries none of the model's registers.
template <bool MODEL>
__device__ __forceinline__ auto srow(const GridSpec& gs, const float2* centre_df, int64_t g) {
    if constexpr (MODEL)
        return df_row_of(gs, centre_df, g);
    else
        return (g < 0) ? centre_df : gs.Sdf + g * gs.nfit;
}

// blocked double-float copies of W for a list of slots
__global__ void k_wdf(const double* __restrict__ W64, const int32_t* __restrict__ slots, int nfit,
                      float* __restrict__ Wdf) {
    const double* W = W64 + (size_t)slots[blockIdx.x] * nfit * nfit;
    float* o = Wdf + (size_t)slots[blockIdx.x] * wdf_floats(nfit);
    const int np = df_blocks(nfit) * 4;
    for (int e = threadIdx.x; e < nfit * np; e += blockDim.x) {
        const int i = e / np, j = e % np;
        const float2 v = (j <= i) ? df_from(W[i * nfit + j]) : make_float2(0.0f, 0.0f);
        float* w = o + ((size_t)(j >> 2) * nfit + i) * 8 + (j & 1) * 4 + ((j >> 1) & 1);
        w[0] = v.x;
        w[2] = v.y;
    }
}

__global__ void k_to_df(const double* __restrict__ x, int64_t n, float2* __restrict__ y) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) y[i] = df_from(x[i]);
}

// ---------------------------------------------------------------- ingest ---

__global__ void k_collapse(const double* __restrict__ S, int64_t G, int nf, const int32_t* __restrict__ coll,
                           int nfit, double* __restrict__ out) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= G) return;
    double acc[kMaxBins];
    for (int j = 0; j < nfit; ++j) acc[j] = 0.0;
    for (int i = 0; i < nf; ++i) {
        const int j = coll ? coll[i] : i;
        acc[j] = __dadd_rn(acc[j], S[g * nf + i]);
    }
    for (int j = 0; j < nfit; ++j) out[g * nfit + j] = acc[j];
}

// Sine table of an oscillation shape model: for each term t and each value k
// of its dm2 axis, sin(1.27 dm2_k L_i / E_i) for every full bin i, with the
// products and the quotient in that order.
__global__ void k_osc_sin(SpecModel m, int rows, const double* __restrict__ L, const double* __restrict__ E,
                          double* __restrict__ sinT) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)rows * m.nf) return;
    const int row = (int)(e / m.nf), i = (int)(e % m.nf);
    int t = 0;
    while (t + 1 < m.n_terms && row >= m.sin_off[t + 1]) ++t;
    const int a = m.dm2_ax[t];
    const double dm2 = m.axis_val[m.axis_off[a] + (row - m.sin_off[t])];
    sinT[e] = sin(__ddiv_rn(__dmul_rn(__dmul_rn(1.27, dm2), L[i]), E[i]));
}

// Grid spectra from an oscillation shape model, one thread per (grid point,
// full bin): s_i(p) = b_i + sum_t amp_t(p) sin^2(1.27 dm2_t(p) L_i / E_i) f_ti,
// the terms added in order t = 0, 1, ... to b_i (model_full).  Grid point p is
// the row-major index over the axes (axis 0 slowest); term t reads its
// amplitude from axis amp_ax[t] and its dm2 from axis dm2_ax[t].  S null: the
// spectra are only checked.  bad counts entries that are not finite and >= 0.
__global__ void k_osc_spectra(SpecModel m, int64_t G, double* __restrict__ S, int* __restrict__ bad) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= G * m.nf) return;
    const int64_t g = e / m.nf;
    const int i = (int)(e % m.nf);
    const double v = model_full(m, model_row(m, g), i);
    if (S) S[e] = v;
    if (!(v >= 0.0) || !isfinite(v)) atomicAdd(bad, 1);
}

// Approximate per-bin median of the grid spectra by two rounds of a 4096-bucket
// histogram; it only chooses the centring vector of the screen, any value works.
__global__ void k_centre(GridSpec gs, int64_t G, double* __restrict__ centre) {
    constexpr int NB = 4096;
    __shared__ unsigned hist[NB];
    __shared__ double red_lo[kThreads / 32], red_hi[kThreads / 32];
    __shared__ double s_lo, s_hi;
    __shared__ int64_t s_rank;
    __shared__ int s_bucket;
    const int j = blockIdx.x;
    double lo = DBL_MAX, hi = -DBL_MAX;
    for (int64_t g = threadIdx.x; g < G; g += blockDim.x) {
        const double x = row_fit(gs, fit_row(gs, g), j);
        lo = fmin(lo, x);
        hi = fmax(hi, x);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        red_lo[threadIdx.x >> 5] = lo;
        red_hi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = red_lo[0], b = red_hi[0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
            a = fmin(a, red_lo[w]);
            b = fmax(b, red_hi[w]);
        }
        s_lo = a;
        s_hi = b;
        s_rank = (G - 1) / 2;
    }
    __syncthreads();
    double blo = s_lo, bhi = s_hi;
    for (int round = 0; round < 2; ++round) {
        for (int b = threadIdx.x; b < NB; b += blockDim.x) hist[b] = 0;
        __syncthreads();
        const double w = (bhi - blo) / NB;
        for (int64_t g = threadIdx.x; g < G; g += blockDim.x) {
            const double x = row_fit(gs, fit_row(gs, g), j);
            if (x < blo || x > bhi) continue;
            int b = (w > 0.0) ? (int)((x - blo) / w) : 0;
            b = b < 0 ? 0 : (b >= NB ? NB - 1 : b);
            atomicAdd(&hist[b], 1u);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int64_t acc = 0;
            int b = 0;
            for (; b < NB; ++b) {
                if (acc + hist[b] > s_rank) break;
                acc += hist[b];
            }
            if (b >= NB) b = NB - 1;
            s_bucket = b;
            s_rank -= acc;
        }
        __syncthreads();
        const double nlo = blo + w * s_bucket;
        const double nhi = (s_bucket == NB - 1) ? bhi : blo + w * (s_bucket + 1);
        __syncthreads();
        blo = nlo;
        bhi = nhi;
    }
    if (threadIdx.x == 0) centre[j] = 0.5 * (blo + bhi);
}

__device__ __forceinline__ int64_t btile_offset(int64_t g, int c, int K) {
    // B-operand image of one BN-row tile: [2K/8 chunks][BN/8 row groups][8 rows][8 cols] bf16
    const int64_t t = g / kBN;
    const int r = (int)(g % kBN);
    return t * (int64_t)(2 * K * kBN) + (int64_t)(c >> 3) * (kBN * 8) + (r >> 3) * 64 + (r & 7) * 8 + (c & 7);
}

// The screen's bf16 hi/lo image of s~ = s - centre and the norms of its split,
// one thread per grid point; the binary64 and binary32 centred rows are stored
// when Sc / Sc32 are given.
__global__ void k_centred(GridSpec gs, int64_t G, int K, double* __restrict__ Sc, float* __restrict__ Sc32,
                          float4* __restrict__ gnorm, uint16_t* __restrict__ Bt) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= G) return;
    const int nfit = gs.nfit;
    const FitRow fr = fit_row(gs, g);
    double ss = 0.0, sl = 0.0, sr = 0.0;
    for (int j = 0; j < nfit; ++j) {
        const double x = __dsub_rn(row_fit(gs, fr, j), gs.centre[j]);
        if (Sc) Sc[g * nfit + j] = x;
        if (Sc32) Sc32[g * nfit + j] = (float)x;
        ss = fma(x, x, ss);
        const __nv_bfloat16 h = __double2bfloat16(x);
        const double rem = x - (double)__bfloat162float(h);
        const __nv_bfloat16 l = __double2bfloat16(rem);
        const double lo = (double)__bfloat162float(l);
        const double res = rem - lo;  // r_S: what hi + lo leave out
        sl = fma(lo, lo, sl);
        sr = fma(res, res, sr);
        Bt[btile_offset(g, j, K)] = __bfloat16_as_ushort(h);
        Bt[btile_offset(g, K + j, K)] = __bfloat16_as_ushort(l);
    }
    // norms rounded up (double sqrt, then float), carried by the spare columns of the lo half
    const float n = __double2float_ru(__dsqrt_ru(ss) * (1.0 + 1e-12));
    const float nl = __double2float_ru(__dsqrt_ru(sl) * (1.0 + 1e-12));
    const float nr = __double2float_ru(__dsqrt_ru(sr) * (1.0 + 1e-12));
    gnorm[g] = make_float4(n, nl, nr, 0.0f);
    Bt[btile_offset(g, K + nfit, K)] = __bfloat16_as_ushort(__float2bfloat16_ru(n));
    Bt[btile_offset(g, K + nfit + 1, K)] = __bfloat16_as_ushort(__float2bfloat16_ru(nl));
    Bt[btile_offset(g, K + nfit + 2, K)] = __bfloat16_as_ushort(__float2bfloat16_ru(nr));
}

// ------------------------------------------------------------ covariances ---

__host__ __device__ __forceinline__ int tri(int n) { return n * (n + 1) / 2; }

// e -> (a, b) with 0 <= b <= a and e = a(a+1)/2 + b
__device__ __forceinline__ void tri_decode(int e, int& a, int& b) {
    a = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
    while ((a + 1) * (a + 2) / 2 <= e) ++a;
    while (a * (a + 1) / 2 > e) --a;
    b = e - a * (a + 1) / 2;
}

// Systematic Cholesky factor of a true point, in binary64.  Each element's
// terms are subtracted in increasing k with a separately rounded multiply and
// subtract, then divided by the pivot, so the factor is reproducible bit for
// bit; any blocking that keeps that order gives it.  Bound by the chain of roots
// and divisions when points are few, by the narrow binary64 pipe (a multiply
// and a subtract a term) when they are many.
// Panels of kCholPanel columns: the panel is gathered into P, factored there
// column by column (the thread that makes the next pivot takes its root while
// the others update), and its terms are then subtracted from the trailing
// triangle in one visit of each element.  The matrix is a packed lower triangle
// in shared memory (161 KB at N_full = 200).
// A cluster of CTAs shares one point when points are few: row i belongs to CTA
// i mod C, which updates it; every CTA gathers the next panel from the owners'
// shared memory and factors it for itself, so one cluster barrier a panel is
// all they exchange.
// Three forms, by what bounds the launch (us measured at points x N_full, the
// form above the line against the one below):
//  cluster   N_full >= 40 and at most 1.5 CTAs an SM: the chain decides, and
//            eight CTAs shorten it (against a CTA a point: 30 x 90 155 / 188, 30
//            x 200 858 / 1062; 38 x 130, where CTAs wait for one another, 477 /
//            390; 4 x 20 28.0 / 24.5 with the columns below)
//  panels    N_full >= 64 and a point an SM at most: the chain again (152 x 90
//            188 / 212, 152 x 200 1064 / 1705; 152 x 40 58.6 / 55.7)
//  columns   else (k_chol_columns): enough points keep the pipe busy, and the
//            panel's gathering is work on top (500 x 90 429 / 413, 9000 x 40 980
//            / 899, 2000 x 200 14853 / 12903; 500 x 120, just above one round of
//            CTAs, is the exception: 985 / 1035)
constexpr int kCholPanel = 8;
constexpr int kCholThreads = 256;
constexpr int kCholCluster = 8;        // CTAs a point when points are few

constexpr int kCholLonePanel = 4;      // panel of a lone CTA

enum { kCholColumnsForm, kCholPanelForm, kCholClusterForm };
inline int chol_form(int P, int nf, int n_sm) {
    if (nf >= 40 && 2 * (int64_t)P * kCholCluster <= 3 * (int64_t)n_sm) return kCholClusterForm;
    return nf >= 64 && P <= n_sm ? kCholPanelForm : kCholColumnsForm;
}

inline size_t chol_sys_smem(int nf, int C) {
    return (size_t)(tri(nf) + (C > 1 ? kCholPanel : kCholLonePanel) * nf) * sizeof(double);
}

__global__ void __launch_bounds__(kCholThreads, 6) k_chol_sys(FullSrc src, int nf, const double* __restrict__ F,
                                                           const int64_t* __restrict__ ps, int gauss,
                                                           double* __restrict__ L64, float* __restrict__ L32,
                                                           float* __restrict__ s32, int* __restrict__ status) {
    extern __shared__ double sT[];
    __shared__ double s_row[kMaxBins];
    __shared__ double s_d;
    __shared__ int s_bad;
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int ip = blockIdx.x / C;
    const int n = nf, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int kWarps = kCholThreads / 32;
    double* Lg = L64 + (size_t)ip * nf * nf;
    float* Lf = L32 + (size_t)ip * nf * nf;
    double* T = sT;             // packed; this CTA's rows (i % C == rank) are kept up to date
    double* P = sT + tri(n);    // [kCholPanel][n]: column c of the panel by row
    stage_full_row(src, nf, ps[ip], s_row);
    const double* s = s_row;
    if (tid == 0) s_bad = 0;
    // element (i, j), j <= i, of diag(s) F diag(s) (+ diag(s) in the Gaussian mode)
    for (int i = rank + C * warp; i < n; i += C * kWarps)
        for (int j = lane; j <= i; j += 32) {
            double v = __dmul_rn(__dmul_rn(s[i], F[i * nf + j]), s[j]);
            if (gauss && i == j) v = __dadd_rn(v, s[i]);
            T[tri(i) + j] = v;
        }
    auto meet = [&]() {
        if (C > 1)
            cluster.sync();
        else
            __syncthreads();
    };
    meet();
    auto pivot = [&](double acc) {
        if (!(acc > 0.0)) {
            s_bad = 1;
            acc = 1.0;
        }
        s_d = __dsqrt_rn(acc);
    };
    const int W = C > 1 ? kCholPanel : kCholLonePanel;
    for (int p0 = 0; p0 < n; p0 += W) {
        const int w = min(W, n - p0);
        for (int e = tid; e < (n - p0) * W; e += kCholThreads) {
            const int i = p0 + e / W, c = e % W;
            if (c < w && p0 + c <= i) {
                const double* own = C > 1 ? cluster.map_shared_rank(T, i % C) : T;
                const double v = own[tri(i) + p0 + c];
                P[c * n + i] = v;
                if (e == 0) pivot(v);
            }
        }
        __syncthreads();
        for (int c = 0; c < w; ++c) {
            const int k = p0 + c;
            const double dk = s_d;
            double* Pc = P + c * n;
            for (int i = k + tid; i < n; i += kCholThreads) Pc[i] = i == k ? dk : __ddiv_rn(Pc[i], dk);
            __syncthreads();
            // columns c + 1 .. w - 1 of the panel: rows on and below their diagonal
            const int below = n - k - 1;
            for (int e = tid; e < (w - c - 1) * below; e += kCholThreads) {
                const int c2 = c + 1 + e / below, i = k + 1 + e % below;
                if (p0 + c2 > i) continue;
                const double v = __dsub_rn(P[c2 * n + i], __dmul_rn(Pc[i], Pc[p0 + c2]));
                P[c2 * n + i] = v;
                if (e == 0) pivot(v);  // (k + 1, k + 1)
            }
            __syncthreads();
        }
        // the finished columns of this CTA's rows go straight out (T keeps what the others may still gather)
        for (int e = tid; e < n * W; e += kCholThreads) {
            const int i = e / W, c = e % W;
            if (i % C != rank || c >= w) continue;
            const double v = p0 + c <= i ? P[c * n + i] : 0.0;
            Lg[i * n + p0 + c] = v;
            Lf[i * n + p0 + c] = __double2float_rn(v);
        }
        // trailing triangle
        const int q0 = p0 + w;
        auto update = [&](int i, int j) {
            double x = T[tri(i) + j];
#pragma unroll
            for (int c = 0; c < kCholPanel; ++c)
                if (c < w) x = __dsub_rn(x, __dmul_rn(P[c * n + i], P[c * n + j]));
            T[tri(i) + j] = x;
        };
        if (C == 1) {
            for (int e = tid; e < tri(n - q0); e += kCholThreads) {
                int a, b;
                tri_decode(e, a, b);
                update(q0 + a, q0 + b);
            }
        } else {
            // this CTA's rows from q0 on, a row per warp
            for (int i = q0 + (rank - q0 % C + C) % C + C * warp; i < n; i += C * kWarps)
                for (int j = q0 + lane; j <= i; j += 32) update(i, j);
        }
        meet();
    }
    if (rank == 0) {
        if (s_bad && tid == 0) atomicOr(status, kDevNotSpd);
        for (int i = tid; i < nf; i += kCholThreads) s32[(size_t)ip * nf + i] = __double2float_rn(s[i]);
    }
}

// The same factor for many points, one CTA a point and a column at a time: after
// column k is final, every trailing element (i >= j > k) subtracts L_ik L_jk.
// Bound by the binary64 pipe.  The triangle is packed in shared memory up to
// kCholPackN (98 KB; 33 KB at N_full = 90, so six points share an SM), beyond it
// lies in the output, row-major, where the several points of an SM hide one
// another's latency better than the one that 161 KB leave room for.
constexpr int kCholPackN = 155;

template <bool PACKED>
__global__ void __launch_bounds__(kCholThreads) k_chol_columns(FullSrc src, int nf, const double* __restrict__ F,
                                                              const int64_t* __restrict__ ps, int gauss,
                                                              double* __restrict__ L64, float* __restrict__ L32,
                                                              float* __restrict__ s32, int* __restrict__ status) {
    extern __shared__ double sT[];
    __shared__ double s_row[kMaxBins];
    __shared__ double s_d;
    __shared__ int s_bad;
    const int ip = blockIdx.x, n = nf, tid = threadIdx.x;
    double* Lg = L64 + (size_t)ip * n * n;
    float* Lf = L32 + (size_t)ip * n * n;
    double* L = PACKED ? sT : Lg;
    auto at = [n](int i, int j) { return PACKED ? tri(i) + j : i * n + j; };
    stage_full_row(src, n, ps[ip], s_row);
    const double* s = s_row;
    if (tid == 0) s_bad = 0;
    for (int e = tid; e < tri(n); e += kCholThreads) {
        int i, j;
        tri_decode(e, i, j);
        double v = __dmul_rn(__dmul_rn(s[i], F[i * n + j]), s[j]);
        if (gauss && i == j) v = __dadd_rn(v, s[i]);
        L[at(i, j)] = v;
    }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (tid == 0) {
            double acc = L[at(k, k)];
            if (!(acc > 0.0)) {
                s_bad = 1;
                acc = 1.0;
            }
            s_d = __dsqrt_rn(acc);
            L[at(k, k)] = s_d;
        }
        __syncthreads();
        const double dk = s_d;
        for (int i = k + 1 + tid; i < n; i += kCholThreads) L[at(i, k)] = __ddiv_rn(L[at(i, k)], dk);
        __syncthreads();
        for (int e = tid; e < tri(n - k - 1); e += kCholThreads) {
            int a, b;
            tri_decode(e, a, b);
            const int i = k + 1 + a, j = k + 1 + b;
            L[at(i, j)] = __dsub_rn(L[at(i, j)], __dmul_rn(L[at(i, k)], L[at(j, k)]));
        }
        __syncthreads();
    }
    for (int e = tid; e < n * n; e += kCholThreads) {
        const int i = e / n, j = e % n;
        const double v = j <= i ? L[at(i, j)] : 0.0;
        Lg[e] = v;
        Lf[e] = __double2float_rn(v);
    }
    if (s_bad && tid == 0) atomicOr(status, kDevNotSpd);
    for (int i = tid; i < n; i += kCholThreads) s32[(size_t)ip * n + i] = __double2float_rn(s[i]);
}

// One CTA per (slot, q): M(q) = C [diag(s) F diag(s) + diag(s)] C^T, L = chol(M),
// W = L^-1, A = W^T W.  Bound by this GPU's narrow binary64 pipe (two
// multiply-adds a cycle and SM, whatever the active lanes of a warp), so every
// phase packs its elements onto full warps and the matrix lives in shared
// memory as one packed triangle.  Factorisation and inversion are one pass over
// it: step k scales column k of L and row k of W by the pivot's reciprocal and
// then takes one rank-1 update of every row below,
//     T_ij -= L_ik v_j,   v_j = L_jk for j > k, W_kj for j <= k
// (j > k: L's trailing triangle; j < k: W's rows; j = k: column k of L is done
// with and becomes -L_ik W_kk), a contiguous range of the packed triangle.  The
// thread that makes the next pivot takes its root while the others update.
// Every element sees the operations of the separate right-looking passes, in
// their order.  These factors feed the fit, not the fake data, so they need not
// repeat the oracle's rounding bit for bit.  Against separate passes over full
// squares (in global memory above N_fit = 64): 597 covariances of N = 200 in
// four launches 18.1 -> 11.3 ms, 10 500 of N = 120 30.1 -> 22.4 ms (their
// multiply-adds alone take 4.1 and 15.7 ms), 10 000 of N = 45 2.8 -> 1.8 ms.
inline size_t build_cov_smem(int nfit) { return (size_t)(tri(nfit) + 2 * nfit) * sizeof(double); }
// 512 threads while an SM holds three CTAs at most, for want of matrices or of shared memory (above N = 112):
// with four, 256 keep more of the pipe for the phases that need few threads.  Measured, us with 256 / 512
// threads: 152 matrices of N = 90 314 / 231, 400 431 / 413, 500 516 / 618; 400 of N = 40 84 / 77, 500 97 / 137;
// 2000 of N = 112 3242 / 3298, of N = 114 3673 / 3440.
inline int build_cov_threads(int nfit, int n, int n_sm) {
    constexpr size_t kStatic = 5 * 1024, kSmSmem = 228 * 1024;  // static arrays and what the system keeps, a CTA
    return n <= 3 * (int64_t)n_sm || 4 * (build_cov_smem(nfit) + kStatic) > kSmSmem ? 512 : 256;
}

__global__ void k_build_cov(FullSrc src, int nf, int nfit, const int32_t* __restrict__ coll,
                            const double* __restrict__ F, const int32_t* __restrict__ q_list,
                            const int32_t* __restrict__ slot_list, int cov_mode, double* __restrict__ A64,
                            double* __restrict__ W64, float* __restrict__ A32, float* __restrict__ rho,
                            int* __restrict__ status) {
    extern __shared__ double sT[];
    __shared__ int s_moff[kMaxBins + 1], s_mem[kMaxBins], s_cur[kMaxBins];
    __shared__ double s_row[kMaxBins];
    __shared__ double s_inv;
    __shared__ int s_bad, s_rho;
    const int e0 = blockIdx.x;
    const int q = q_list[e0];
    const int slot = slot_list[e0];
    const int n = nfit;
    double* T = sT;              // packed lower triangle: M, then L / W
    double* sl = sT + tri(n);    // column k of L below the diagonal
    double* sv = sl + n;         // v
    double* Wg = W64 + (size_t)slot * n * n;
    double* A = A64 + (size_t)slot * n * n;
    float* Af = A32 + (size_t)slot * n * n;
    stage_full_row(src, nf, q, s_row);
    const double* s = s_row;
    if (cov_mode == 2) {  // identity test mode
        for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
            const double v = (e / n == e % n) ? 1.0 : 0.0;
            Wg[e] = v;
            A[e] = v;
            Af[e] = (float)v;
        }
        if (threadIdx.x == 0) rho[slot] = 1.0f;
        return;
    }
    // full bins of each fit bin, in increasing order (counting sort by one thread)
    if (threadIdx.x == 0) {
        s_bad = 0;
        s_rho = 0;
        if (coll) {
            for (int j = 0; j <= n; ++j) s_moff[j] = 0;
            for (int i = 0; i < nf; ++i) ++s_moff[coll[i] + 1];
            for (int j = 0; j < n; ++j) s_moff[j + 1] += s_moff[j];
            for (int j = 0; j < n; ++j) s_cur[j] = s_moff[j];
            for (int i = 0; i < nf; ++i) s_mem[s_cur[coll[i]]++] = i;
        }
    }
    __syncthreads();
    auto pivot = [&](double d) {  // 1 / sqrt(d) for the step to come
        if (!(d > 0.0)) {
            s_bad = 1;
            d = 1.0;
        }
        s_inv = 1.0 / __dsqrt_rn(d);
    };
    // 1. M in fit space: element (j, l) sums (s_a F_ab) s_b (+ s_a when a == b) over full bins a -> j,
    //    b -> l in increasing (a, b)
    for (int e = threadIdx.x; e < tri(n); e += blockDim.x) {
        int j, l;
        tri_decode(e, j, l);
        double v = 0.0;
        if (coll == nullptr) {
            v = (s[j] * F[j * nf + l]) * s[l];
            if (j == l) v += s[j];
        } else {
            for (int ia = s_moff[j]; ia < s_moff[j + 1]; ++ia) {
                const int a = s_mem[ia];
                for (int ib = s_moff[l]; ib < s_moff[l + 1]; ++ib) {
                    const int b = s_mem[ib];
                    double t = (s[a] * F[a * nf + b]) * s[b];
                    if (a == b) t += s[a];
                    v += t;
                }
            }
        }
        T[e] = v;
        if (e == 0) pivot(v);
    }
    __syncthreads();
    // 2. L and W
    for (int k = 0; k < n; ++k) {
        const double inv = s_inv;
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
            if (j > k) {
                const double l = T[tri(j) + k] * inv;
                sl[j] = l;
                sv[j] = l;
            } else {
                const double w = j < k ? T[tri(k) + j] * inv : inv;
                sv[j] = w;
                T[tri(k) + j] = w;
            }
        }
        __syncthreads();
        const int next = tri(k + 1) + k + 1;  // the next pivot's element
        for (int e = tri(k + 1) + threadIdx.x; e < tri(n); e += blockDim.x) {
            int i, j;
            tri_decode(e, i, j);
            const double t = fma(-sl[i], sv[j], j == k ? 0.0 : T[e]);
            T[e] = t;
            if (e == next) pivot(t);
        }
        __syncthreads();
    }
    if (s_bad) {
        if (threadIdx.x == 0) atomicOr(status, kDevNotSpd);
        return;
    }
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const int i = e / n, j = e % n;
        Wg[e] = j <= i ? T[tri(i) + j] : 0.0;
    }
    // 3. A_ij = sum_{k >= i} W_ki W_kj for j <= i
    for (int e = threadIdx.x; e < tri(n); e += blockDim.x) {
        int i, j;
        tri_decode(e, i, j);
        double acc = 0.0;
        const double *wi = T + tri(i) + i, *wj = T + tri(i) + j;
        for (int k = i; k < n; ++k) {
            acc = fma(*wi, *wj, acc);
            wi += k + 1;
            wj += k + 1;
        }
        A[i * n + j] = acc;
        A[j * n + i] = acc;
        Af[i * n + j] = (float)acc;
        Af[j * n + i] = (float)acc;
    }
    __syncthreads();
    // rho >= max_i sum_j |A_ij| (an upper bound of the spectral norm of |A|): the binary32 sums, raised by
    // their rounding
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < n; i += blockDim.x >> 5) {
        float r = 0.0f;
        for (int j = lane; j < n; j += 32) r += fabsf(Af[i * n + j]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        if (lane == 0) atomicMax(&s_rho, __float_as_int(r));
    }
    __syncthreads();
    if (threadIdx.x == 0) rho[slot] = __fmul_ru(__int_as_float(s_rho), 1.0f + (float)(n + 4) * 1.1920929e-07f);
}

// q_g = s~_g^T A s~_g in binary64, one thread per g
// q_g = s~_g^T A s~_g = |W s~_g|^2 (A = W^T W, W lower triangular): t_i = sum_{j<=i}
// W_ij s~_j and q = sum_i t_i^2, each an fma chain in increasing index, so
// N (N + 3) / 2 DFMA per point instead of the N^2 + N of s~^T (A s~).
__global__ void k_qvec64(GridSpec gs, int64_t G, int nfit, const double* __restrict__ W64,
                         const int32_t* __restrict__ slots, int64_t ldq, double* __restrict__ Q64) {
    const int slot = slots[blockIdx.y];
    const double* W = W64 + (size_t)slot * nfit * nfit;
    double sl[kMaxBins];  // the row, when it is recomputed rather than stored
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < G; g += (int64_t)gridDim.x * blockDim.x) {
        const double* s = gs.Sc ? gs.Sc + g * nfit : sl;
        if (!gs.Sc) {
            const FitRow fr = fit_row(gs, g);
            for (int j = 0; j < nfit; ++j) sl[j] = row_sc(gs, fr, j);
        }
        double q = 0.0;
        for (int i = 0; i < nfit; ++i) {
            const double* Wi = W + i * nfit;
            double t = 0.0;
            for (int j = 0; j <= i; ++j) t = fma(Wi[j], s[j], t);
            q = fma(t, t, q);
        }
        Q64[(size_t)slot * ldq + g] = q;
    }
}

// binary32 q_g with its rounding bound; s~_g held in registers (NMAX >= nfit,
// NMAX a multiple of 4), A staged in shared memory with rows padded to NMAX.
template <int NMAX>
__global__ void k_qvec32(GridSpec gs, const float4* __restrict__ gnorm, int64_t G, int64_t G_pad,
                         int nfit, const float* __restrict__ A32, const float* __restrict__ rho,
                         const int32_t* __restrict__ slots, float* __restrict__ Qc, float* __restrict__ Qb,
                         uint16_t* __restrict__ Qb3) {
    __shared__ __align__(16) float sA[NMAX * NMAX];
    const int slot = slots[blockIdx.y];
    const float* A = A32 + (size_t)slot * nfit * nfit;
    for (int e = threadIdx.x; e < NMAX * NMAX; e += blockDim.x) {
        const int i = e / NMAX, j = e % NMAX;
        sA[e] = (i < nfit && j < nfit) ? A[i * nfit + j] : 0.0f;
    }
    __syncthreads();
    const float r = rho[slot];
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < G_pad; g += (int64_t)gridDim.x * blockDim.x) {
        float qc = 0.0f, qb = 3.0e38f;
        if (g < G) {
            float s[NMAX];
            if (gs.Sc32) {
#pragma unroll
                for (int j = 0; j < NMAX; ++j) s[j] = (j < nfit) ? gs.Sc32[g * nfit + j] : 0.0f;
            } else {
                const FitRow fr = fit_row(gs, g);
#pragma unroll
                for (int j = 0; j < NMAX; ++j) s[j] = (j < nfit) ? row_sc32(gs, fr, j) : 0.0f;
            }
            float q = 0.0f;
#pragma unroll
            for (int i = 0; i < NMAX; ++i) {
                const float4* Ai = reinterpret_cast<const float4*>(sA + i * NMAX);
                float t = 0.0f;
#pragma unroll
                for (int j4 = 0; j4 < NMAX / 4; ++j4) {
                    const float4 a4 = Ai[j4];
                    t = fmaf(a4.x, s[4 * j4 + 0], t);
                    t = fmaf(a4.y, s[4 * j4 + 1], t);
                    t = fmaf(a4.z, s[4 * j4 + 2], t);
                    t = fmaf(a4.w, s[4 * j4 + 3], t);
                }
                q = fmaf(s[i], t, q);
            }
            const float n = gnorm[g].x;
            // |q^ - q| <= (nfit+4) 2^-24 rho |s|^2 + 2^-23 |q^|   (A rounded to binary32, dot products, final rounding)
            const float beta = 1.02f * ((float)(nfit + 4) * 5.9604645e-08f * r * n * n + q_rel_slack(nfit) * fabsf(q));
            qc = q;
            qb = __fsub_rd(q, beta);
        }
        Qc[(size_t)slot * G_pad + g] = qc;
        Qb[(size_t)slot * G_pad + g] = qb;
        store_qb3(Qb3 + ((size_t)slot * G_pad + g) * 8, qb);
    }
}

__global__ void k_qvec32_generic(GridSpec gs, const float4* __restrict__ gnorm, int64_t G,
                                 int64_t G_pad, int nfit, const float* __restrict__ A32, const float* __restrict__ rho,
                                 const int32_t* __restrict__ slots, float* __restrict__ Qc, float* __restrict__ Qb,
                                 uint16_t* __restrict__ Qb3) {
    const int slot = slots[blockIdx.y];
    const float* A = A32 + (size_t)slot * nfit * nfit;
    const float r = rho[slot];
    float sl[kMaxBins];  // the row, when it is recomputed rather than stored
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < G_pad; g += (int64_t)gridDim.x * blockDim.x) {
        float qc = 0.0f, qb = 3.0e38f;
        if (g < G) {
            const float* s = gs.Sc32 ? gs.Sc32 + g * nfit : sl;
            if (!gs.Sc32) {
                const FitRow fr = fit_row(gs, g);
                for (int j = 0; j < nfit; ++j) sl[j] = row_sc32(gs, fr, j);
            }
            float q = 0.0f;
            for (int i = 0; i < nfit; ++i) {
                float t = 0.0f;
                for (int j = 0; j < nfit; ++j) t = fmaf(A[i * nfit + j], s[j], t);
                q = fmaf(s[i], t, q);
            }
            const float n = gnorm[g].x;
            const float beta = 1.02f * ((float)(nfit + 4) * 5.9604645e-08f * r * n * n + q_rel_slack(nfit) * fabsf(q));
            qc = q;
            qb = __fsub_rd(q, beta);
        }
        Qc[(size_t)slot * G_pad + g] = qc;
        Qb[(size_t)slot * G_pad + g] = qb;
        store_qb3(Qb3 + ((size_t)slot * G_pad + g) * 8, qb);
    }
}

// -------------------------------------------------------------- fake data ---

// One CTA per kFakeU universes of a point: z from Philox/Box-Muller, lam_i =
// max(0, s_i + sum_{j<=i} L_ij z_j) accumulated with fma in j order, n_i =
// Poisson(lam_i) from bin i's own stream, fit bin = sum of its full bins in i
// order.  Bound by instruction issue, so the four parts are laid out for full
// warps, with z, lam and the counts in shared memory:
//  - normals: one thread per (block of four, universe);
//  - lam: a warp per eight rows of L, two universes per lane, so each L_ij (one
//    broadcast) and z_j feed 16 multiply-adds;
//  - counts: one thread per (bin, universe): lam below ten by inversion, else
//    only the quick acceptance of the rejection sampler's first trial (about
//    seven draws of ten); the others are queued and tested by full warps, trial
//    by trial, instead of by the few lanes of every warp that need the
//    logarithms;
//  - fit bins: two or four threads per universe, each its part of the fit bins.
// One thread per universe did all of it with 16 of 32 lanes active: 500 points
// x 1000 universes of 90 bins 1.56 -> 0.95 ms, of 16 bins 236 -> 168 us, one
// point x 1000 universes of 40 bins 100 -> 25 us.
constexpr int kFakeU = 64;        // universes of a CTA
constexpr int kFakeLd = kFakeU + 2;
constexpr int kFakeRows = 8;      // rows of L per warp
constexpr int kFakePasses = 3;    // trials tested by full warps
constexpr int kFakeFewBins = 8;   // bins a thread can hold by itself

// A thread per universe (k_fake_few) from there on: with few bins a CTA's phases are shorter than its barriers.
// Measured, us, a thread / a CTA of 64 universes: 500 points x 1000 universes of 1 bin 25 / 46, of 5 bins 79 / 78
// (85 / 102 with counts below ten), of 8 bins 115 / 101 (110 / 123); 1216 points x 64 of 5 bins 20.8 / 15.8, of
// 1 bin 9.1 / 11.1.  From nine bins on the CTA is the faster but for counts below ten in 1500 CTAs and more
// (9 bins 130 / 134, 12 bins 154 / 152).
inline bool fake_few(int nf, int64_t ctas, int n_sm) {
    return nf <= 2 || (nf <= kFakeFewBins && ctas > 8 * (int64_t)n_sm);
}
// 128 threads a CTA, eight an SM, when there are more CTAs than four an SM (256 threads) take at once and
// eight fit in shared memory (N_full = 52): 500 x 1000 of 16 bins 218 -> 185 us, of 48 bins 502 -> 468; 310 x 64
// of 24 bins, one round either way, 22.6 with 256 and 28.0 with 128.
inline int fake_threads(int nf, int64_t ctas, int n_sm) { return nf <= 52 && ctas > 4 * (int64_t)n_sm ? 128 : 256; }
inline size_t fake_smem(int nf) { return (size_t)(2 * nf + 3) * kFakeLd * sizeof(float); }

template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) k_fake_data(const float* __restrict__ L32,
                                                               const float* __restrict__ s32, int nf,
                                                               const int32_t* __restrict__ coll, int nfit,
                                                               const int64_t* __restrict__ ps, int U, uint32_t k0,
                                                               uint32_t k1, int gauss, float* __restrict__ d) {
    extern __shared__ float4 s_fake[];
    __shared__ int s_queued[kFakePasses];
    float* lam = reinterpret_cast<float*>(s_fake);       // [nf][kFakeLd]: lam, then the counts
    float* z = lam + nf * kFakeLd;                       // [nf + 3][kFakeLd]; later the queue, then the fit bins
    uint16_t* queue = reinterpret_cast<uint16_t*>(z);    // two of [nf * kFakeU]: bin * kFakeU + universe
    const int ip = blockIdx.y;
    const int u0 = blockIdx.x * kFakeU;
    const int nu = min(kFakeU, U - u0);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t p = (uint32_t)ps[ip];
    const float* L = L32 + (size_t)ip * nf * nf;
    const float* s = s32 + (size_t)ip * nf;
    if (tid < kFakePasses) s_queued[tid] = 0;
    for (int e = tid; e < (nf + 3) / 4 * kFakeU; e += THREADS) {
        const int j = e / kFakeU, u = e % kFakeU;
        float zz[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (u < nu) normal_block((uint32_t)j, (uint32_t)(u0 + u), p, k0, k1, zz);
#pragma unroll
        for (int h = 0; h < 4; ++h) z[(4 * j + h) * kFakeLd + u] = zz[h];
    }
    __syncthreads();
    // the row blocks, longest first, dealt to the warps back and forth
    const int nb = (nf + kFakeRows - 1) / kFakeRows;
    constexpr int kWarps = THREADS / 32;
    for (int pass = 0; pass * kWarps < nb; ++pass) {
        const int b = nb - 1 - (pass * kWarps + ((pass & 1) ? kWarps - 1 - warp : warp));
        if (b < 0) continue;
        const int i0 = b * kFakeRows, jn = min(i0 + kFakeRows, nf);
        float a0[kFakeRows], a1[kFakeRows];
        const float* Lb = L + (size_t)i0 * nf;
        int off[kFakeRows];
#pragma unroll
        for (int r = 0; r < kFakeRows; ++r) {
            a0[r] = a1[r] = 0.0f;
            off[r] = min(r, nf - 1 - i0) * nf;
        }
        // L is zero above its diagonal: the columns past a row's own add exact zeros
#pragma unroll 2
        for (int j = 0; j < jn; ++j) {
            const float2 zj = *reinterpret_cast<const float2*>(z + j * kFakeLd + 2 * lane);
#pragma unroll
            for (int r = 0; r < kFakeRows; ++r) {
                const float l = __ldg(Lb + off[r] + j);
                a0[r] = __fmaf_rn(l, zj.x, a0[r]);
                a1[r] = __fmaf_rn(l, zj.y, a1[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < kFakeRows; ++r) {
            const int i = i0 + r;
            if (i >= nf) break;
            const float si = __ldg(s + i);
            float x = __fadd_rn(si, a0[r]), y = __fadd_rn(si, a1[r]);
            if (!gauss) {
                if (!(x > 0.0f)) x = 0.0f;
                if (!(y > 0.0f)) y = 0.0f;
            }
            *reinterpret_cast<float2*>(lam + i * kFakeLd + 2 * lane) = make_float2(x, y);
        }
    }
    __syncthreads();
    if (!gauss) {
        // appends the lanes' items; every lane of the warp is here
        auto push = [&](uint16_t* to, int* n, bool mine, int e) {
            const unsigned m = __ballot_sync(0xffffffffu, mine);
            if (!m) return;
            int at = 0;
            if (lane == 0) at = atomicAdd(n, __popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (mine) to[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)e;
        };
        // kFakeU is a multiple of the warp: a warp's lanes share the bin and are in the loop together
        for (int e = tid; e < nf * kFakeU; e += THREADS) {
            const int i = e / kFakeU, u = e % kFakeU;
            const float l = lam[i * kFakeLd + u];
            bool wait = u < nu && l > 0.0f;  // lam = 0: the count is 0
            if (wait) {
                BinUniforms un;
                un.init(k0, k1, (uint32_t)(u0 + u), p, (uint32_t)i);
                float ua, ub;
                un.pair(0, ua, ub);
                int32_t k = 0;
                if (l < 10.0f) {  // a bin of few counts has few in most universes: the warp is full as it is
                    k = poisson_inversion(l, ua);
                    wait = false;
                } else {
                    Ptrs t;
                    t.init(l);
                    wait = !t.propose(ua, ub);
                    k = (int32_t)t.kf;
                }
                if (!wait) lam[i * kFakeLd + u] = (float)k;
            }
            push(queue, &s_queued[0], wait, e);
        }
        __syncthreads();
        // trial by trial: the logarithms of trial t, then the quick acceptance of t + 1; what is left after
        // kFakePasses trials goes on alone
        uint16_t* from = queue;
        for (int t = 0; t < kFakePasses; ++t) {
            const int n = s_queued[t];
            if (n == 0) break;  // the same for every thread
            uint16_t* to = (t & 1) ? queue : queue + nf * kFakeU;
            const bool last = t + 1 == kFakePasses;
            for (int q0 = 0; q0 < n; q0 += THREADS) {  // the same trip count for every thread
                const bool have = q0 + tid < n;
                bool again = false;
                int e = 0;
                if (have) {
                    e = from[q0 + tid];
                    const int i = e / kFakeU, u = e % kFakeU;
                    const float l = lam[i * kFakeLd + u];
                    BinUniforms un;
                    un.init(k0, k1, (uint32_t)(u0 + u), p, (uint32_t)i);
                    float ua, ub;
                    un.pair(t, ua, ub);
                    Ptrs tr;
                    tr.init(l);
                    tr.propose(ua, ub);
                    const float loglam = ln32(l);
                    again = !tr.accept(loglam);
                    if (again) {
                        un.pair(t + 1, ua, ub);
                        again = !tr.propose(ua, ub);
                    }
                    if (again && last) {
                        int it = t + 1;
                        while (!tr.accept(loglam) && ++it < kPtrsTrials) {
                            un.pair(it, ua, ub);
                            if (tr.propose(ua, ub)) break;
                        }
                        if (it >= kPtrsTrials) tr.kf = floorf(l);
                        again = false;
                    }
                    if (!again) lam[i * kFakeLd + u] = (float)(int32_t)tr.kf;
                }
                if (!last) push(to, &s_queued[t + 1], again, e);
            }
            __syncthreads();
            from = to;
        }
    }
    const float* out = lam;
    if (coll) {
        out = z;
        for (int e = tid; e < nfit * kFakeLd; e += THREADS) z[e] = 0.0f;
        __syncthreads();
        constexpr int kParts = THREADS / kFakeU;  // a power of two
        const int u = tid % kFakeU, part = tid / kFakeU;  // fit bins part, part + kParts, ... of universe u
        for (int i = 0; i < nf; ++i) {
            const int jf = __ldg(coll + i);
            if ((jf & (kParts - 1)) == part) z[jf * kFakeLd + u] = __fadd_rn(z[jf * kFakeLd + u], lam[i * kFakeLd + u]);
        }
        __syncthreads();
    }
    float* o = d + ((size_t)ip * U + u0) * nfit;
    if (nfit < 32) {  // several universes a warp
        for (int e = tid; e < nu * nfit; e += THREADS) o[e] = out[e % nfit * kFakeLd + e / nfit];
    } else {
        for (int u = warp; u < nu; u += kWarps)
            for (int j = lane; j < nfit; j += 32) o[(size_t)u * nfit + j] = out[j * kFakeLd + u];
    }
}

// The same for at most kFakeFewBins bins: one thread per universe, everything
// in registers.
__global__ void __launch_bounds__(128) k_fake_few(const float* __restrict__ L32, const float* __restrict__ s32, int nf,
                                                  const int32_t* __restrict__ coll, int nfit,
                                                  const int64_t* __restrict__ ps, int U, uint32_t k0, uint32_t k1,
                                                  int gauss, float* __restrict__ d) {
    const int ip = blockIdx.y;
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= U) return;
    const uint32_t p = (uint32_t)ps[ip];
    const float* L = L32 + (size_t)ip * nf * nf;
    const float* s = s32 + (size_t)ip * nf;
    float z[kFakeFewBins], v[kFakeFewBins];
#pragma unroll
    for (int j = 0; j < kFakeFewBins; j += 4) {
        float zz[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (j < nf) normal_block((uint32_t)(j / 4), (uint32_t)u, p, k0, k1, zz);
#pragma unroll
        for (int h = 0; h < 4; ++h) z[j + h] = zz[h];
    }
#pragma unroll
    for (int r = 0; r < kFakeFewBins; ++r) {
        v[r] = 0.0f;
        if (r >= nf) continue;
        float acc = 0.0f;
#pragma unroll
        for (int j = 0; j <= r; ++j) acc = __fmaf_rn(__ldg(L + r * nf + j), z[j], acc);
        v[r] = __fadd_rn(__ldg(s + r), acc);
    }
    if (!gauss) {
        // not unrolled: the draw's code once, with the bins shifted through v
#pragma unroll 1
        for (int r = 0; r < nf; ++r) {
            BinUniforms un;
            un.init(k0, k1, (uint32_t)u, p, (uint32_t)r);
            const float n = (float)poisson(v[0], un);
#pragma unroll
            for (int k = 0; k + 1 < kFakeFewBins; ++k) v[k] = v[k + 1];
            v[kFakeFewBins - 1] = n;
        }
        // bin r is at kFakeFewBins - nf + r now
#pragma unroll 1
        for (int r = nf; r < kFakeFewBins; ++r) {
#pragma unroll
            for (int k = 0; k + 1 < kFakeFewBins; ++k) v[k] = v[k + 1];
        }
    }
    float* o = d + ((size_t)ip * U + u) * nfit;
    for (int j = 0; j < nfit; ++j) {
        float sum = 0.0f;
#pragma unroll
        for (int r = 0; r < kFakeFewBins; ++r)
            if (r < nf && (coll ? __ldg(coll + r) : r) == j) sum = coll ? __fadd_rn(sum, v[r]) : v[r];
        o[j] = sum;
    }
}

// ------------------------------------------------------- bookkeeping -------

__global__ void k_fill_i32(int32_t* p, int64_t n, int32_t v) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

__global__ void k_mark_used(const int32_t* __restrict__ active, int64_t n, const int32_t* __restrict__ cur,
                            uint8_t* __restrict__ flag) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) flag[cur[active[i]]] = 1;
}

__global__ void k_compact_flags(uint8_t* __restrict__ flag, int64_t G, int32_t* __restrict__ list,
                                int32_t* __restrict__ count) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= G) return;
    if (flag[g]) {
        flag[g] = 0;
        list[atomicAdd(count, 1)] = (int32_t)g;
    }
}

__global__ void k_lookup_slots(const int32_t* __restrict__ active, int64_t n, const int32_t* __restrict__ cur,
                               const int32_t* __restrict__ slot_of, int32_t* __restrict__ uslot) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) uslot[i] = slot_of[cur[active[i]]];
}

__global__ void k_set_slots(const int32_t* __restrict__ q, const int32_t* __restrict__ s, int n,
                            int32_t* __restrict__ slot_of) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) slot_of[q[i]] = s[i];
}

// ------------------------------------------------------ plain fp64 scan -----

// Plain binary64 scan: chi2_g - c = q_g - 2 y.s~_g with y = A (d - v) for every
// g, the first minimum in index order.  The y.s~ products of 16 universes x 64
// grid points are a small dense contraction on the FP64 pipe: y and a tile of
// s~ (transposed to [j][g]) sit in shared memory and every thread keeps a 4 x 2
// block of dot products in registers (the binary64 pipe is narrow, so operand
// loads are never the limit).  Every dot product is one fma chain over j in
// increasing order, as in a per-pair loop, so the minimum found does not depend
// on the blocking.  Grid (16 universes, split): few universes leave SMs idle,
// so the grid's tiles are then dealt to gridDim.y CTAs, which read y (k_y64)
// and write their minima for k_scan_resid_reduce.  One point of 25x25 x 1000
// universes: 2.00 ms a job unsplit, 1.54 ms split with every CTA forming y.
constexpr int kS64U = 16;   // universes per CTA
constexpr int kS64G = 64;   // grid points per staged tile
constexpr int kS64LdS = kS64G + 2;  // row stride of the staged tile (fewer bank conflicts, 16-byte rows)
constexpr int kS64Threads = 128;

// y = A (d - v) of each universe in list order, each component one fma chain
// over j in increasing order (A is symmetric: its columns are read, coalesced)
__global__ void __launch_bounds__(64) k_y64(const int32_t* __restrict__ list, const int32_t* __restrict__ uslot,
                                            const float* __restrict__ d, const double* __restrict__ centre, int nfit,
                                            const double* __restrict__ A64, double* __restrict__ y) {
    __shared__ double sd[kMaxBins];
    const int64_t i = blockIdx.x;
    const float* du = d + (size_t)list[i] * nfit;
    for (int j = threadIdx.x; j < nfit; j += blockDim.x) sd[j] = (double)du[j] - centre[j];
    __syncthreads();
    const double* A = A64 + (size_t)uslot[i] * nfit * nfit;
    for (int r = threadIdx.x; r < nfit; r += blockDim.x) {
        double t = 0.0;
#pragma unroll 4
        for (int j = 0; j < nfit; ++j) t = fma(A[(size_t)j * nfit + r], sd[j], t);
        y[i * nfit + r] = t;
    }
}

__global__ void __launch_bounds__(kS64Threads) k_scan64(const int32_t* __restrict__ list, int64_t n,
                                                         const int32_t* __restrict__ uslot,
                                                         const float* __restrict__ d, GridSpec gs, int64_t G,
                                                         int nfit, const double* __restrict__ A64,
                                                         const double* __restrict__ Q64, int64_t ldq,
                                                         int32_t* __restrict__ best, const double* __restrict__ ysrc,
                                                         double* __restrict__ part_v, int32_t* __restrict__ part_g) {
    extern __shared__ double2 sm64v[];
    double* sy = reinterpret_cast<double*>(sm64v);   // [nfit][kS64U]
    double* ss = sy + (size_t)nfit * kS64U;          // [nfit][kS64LdS]
    __shared__ double s_bv[kS64Threads / 4][kS64U];
    __shared__ int32_t s_bg[kS64Threads / 4][kS64U];
    __shared__ int s_slot[kS64U];
    const int tid = threadIdx.x;
    const int64_t u0 = (int64_t)blockIdx.x * kS64U;
    const int nu = (int)((n - u0) < kS64U ? (n - u0) : kS64U);
    if (tid < kS64U) s_slot[tid] = (tid < nu) ? uslot[u0 + tid] : 0;
    // d - v of the CTA's universes, [j][u] (in the tile buffer, free until the first tile)
    for (int e = tid; !ysrc && e < nfit * kS64U; e += kS64Threads) {
        const int j = e / kS64U, uu = e - (e / kS64U) * kS64U;
        ss[e] = (uu < nu) ? (double)d[(size_t)list[u0 + uu] * nfit + j] - gs.centre[j] : 0.0;
    }
    __syncthreads();
    // y_r = sum_j A_rj (d - v)_j, one fma chain in j order
    for (int e = tid; e < nfit * kS64U; e += kS64Threads) {
        const int r = e / kS64U, uu = e - (e / kS64U) * kS64U;
        double t = 0.0;
        if (uu < nu && ysrc) {
            t = ysrc[(u0 + uu) * nfit + r];
        } else if (uu < nu) {
            const double* A = A64 + (size_t)s_slot[uu] * nfit * nfit + (size_t)r * nfit;
            for (int j = 0; j < nfit; ++j) t = fma(A[j], ss[j * kS64U + uu], t);
        }
        sy[r * kS64U + uu] = t;
    }
    const int tu = tid & 3, tg = tid >> 2;  // universes 4 tu .. 4 tu + 3, tile points 2 tg, 2 tg + 1
    double bv[4];
    int32_t bg[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        bv[a] = DBL_MAX;
        bg[a] = INT32_MAX;
    }
    for (int64_t g0 = (int64_t)blockIdx.y * kS64G; g0 < G; g0 += (int64_t)gridDim.y * kS64G) {
        __syncthreads();  // y complete / the previous tile's readers done
        if (gs.Sc) {
            for (int e = tid; e < kS64G * nfit; e += kS64Threads) {
                const int gg = e / nfit, j = e - (e / nfit) * nfit;
                const int64_t g = g0 + gg;
                ss[j * kS64LdS + gg] = (g < G) ? gs.Sc[g * nfit + j] : 0.0;
            }
        } else {
            // recomputed rows: one point per thread, decoded once
            for (int gg = tid; gg < kS64G; gg += kS64Threads) {
                const int64_t g = g0 + gg;
                if (g < G) {
                    const FitRow fr = fit_row(gs, g);
                    for (int j = 0; j < nfit; ++j) ss[j * kS64LdS + gg] = row_sc(gs, fr, j);
                } else {
                    for (int j = 0; j < nfit; ++j) ss[j * kS64LdS + gg] = 0.0;
                }
            }
        }
        __syncthreads();
        double acc[4][2];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) acc[a][b] = 0.0;
        for (int j = 0; j < nfit; ++j) {
            const double2 y01 = *reinterpret_cast<const double2*>(sy + j * kS64U + 4 * tu);
            const double2 y23 = *reinterpret_cast<const double2*>(sy + j * kS64U + 4 * tu + 2);
            const double2 s01 = *reinterpret_cast<const double2*>(ss + j * kS64LdS + 2 * tg);
            const double y[4] = {y01.x, y01.y, y23.x, y23.y};
            const double sv[2] = {s01.x, s01.y};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) acc[a][b] = fma(y[a], sv[b], acc[a][b]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int uu = 4 * tu + a;
            if (uu >= nu) continue;
            const double* Q = Q64 + (size_t)s_slot[uu] * ldq;
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int64_t g = g0 + 2 * tg + b;
                if (g >= G) continue;
                const double v = fma(-2.0, acc[a][b], Q[g]);
                if (v < bv[a] || (v == bv[a] && (int32_t)g < bg[a])) {
                    bv[a] = v;
                    bg[a] = (int32_t)g;
                }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        s_bv[tg][4 * tu + a] = bv[a];
        s_bg[tg][4 * tu + a] = bg[a];
    }
    __syncthreads();
    if (tid < nu) {
        double v = DBL_MAX;
        int32_t g = INT32_MAX;
        for (int k = 0; k < kS64Threads / 4; ++k) {
            const double x = s_bv[k][tid];
            const int32_t xg = s_bg[k][tid];
            if (x < v || (x == v && xg < g)) {
                v = x;
                g = xg;
            }
        }
        if (gridDim.y == 1) {
            best[list[u0 + tid]] = g;
        } else {
            part_v[(u0 + tid) * gridDim.y + blockIdx.y] = v;
            part_g[(u0 + tid) * gridDim.y + blockIdx.y] = g;
        }
    }
}

// Exact residual-form scan (Algorithm 2 for every g) of the universes in
// `list`, used when all certified screen rounds failed, so it never needs
// binary64 q-vectors.  Grid (universe, split): the warps of a CTA walk groups
// of kRowsB grid points of its share (rows_chi2); k_scan_resid_reduce takes the
// first minimum over the splits.
template <bool MODEL>
__global__ void __launch_bounds__(32 * kRowsWarps) k_scan_resid(const int32_t* __restrict__ list,
                                                                const int32_t* __restrict__ uslot,
                                                                const float* __restrict__ d, GridSpec gs, int64_t G,
                                                                int nfit, const float* __restrict__ Wdf,
                                                                double* __restrict__ part_v,
                                                                int32_t* __restrict__ part_g) {
    extern __shared__ float4 s_rows[];
    __shared__ double rv[kRowsWarps];
    __shared__ int32_t rg[kRowsWarps];
    const int i = blockIdx.x, sp = blockIdx.y, nsp = gridDim.y;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* sm = reinterpret_cast<float*>(s_rows) + warp * rows_floats(nfit);
    const int u = list[i];
    const float* W = Wdf + (size_t)uslot[i] * wdf_floats(nfit);
    const float* du = d + (size_t)u * nfit;
    double bv = DBL_MAX;
    int32_t bg = INT32_MAX;
    const int64_t step = (int64_t)nsp * kRowsWarps * kRowsB;
    for (int64_t g0 = ((int64_t)sp * kRowsWarps + warp) * kRowsB; g0 < G; g0 += step) {
        const int m = (int)(G - g0 < kRowsB ? G - g0 : kRowsB);
        for (int k = 0; k < m; ++k) rows_stage(sm, k, nfit, srow<MODEL>(gs, nullptr, g0 + k), du, lane);
        const double c = rows_chi2(W, nfit, sm, m, lane);
        if (lane < m && c < bv) {
            bv = c;
            bg = (int32_t)(g0 + lane);
        }
    }
    warp_argmin(bv, bg);
    if (lane == 0) {
        rv[warp] = bv;
        rg[warp] = bg;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        bv = threadIdx.x < kRowsWarps ? rv[threadIdx.x] : DBL_MAX;
        bg = threadIdx.x < kRowsWarps ? rg[threadIdx.x] : INT32_MAX;
        warp_argmin(bv, bg);
        if (threadIdx.x == 0) {
            part_v[(size_t)i * nsp + sp] = bv;
            part_g[(size_t)i * nsp + sp] = bg;
        }
    }
}

__global__ void k_scan_resid_reduce(const int32_t* __restrict__ list, int64_t n, int nsp,
                                    const double* __restrict__ part_v, const int32_t* __restrict__ part_g,
                                    int32_t* __restrict__ best) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double bv = DBL_MAX;
    int32_t bg = INT32_MAX;
    for (int sp = 0; sp < nsp; ++sp) {
        const double v = part_v[i * nsp + sp];
        const int32_t g = part_g[i * nsp + sp];
        if (v < bv || (v == bv && g < bg)) {
            bv = v;
            bg = g;
        }
    }
    best[list[i]] = bg;
}

// ------------------------------------------------------ mixed: grouping -----

// Universes of one job sit next to each other and mostly share a slot, so the
// lanes of a warp that hold the same slot add their count with one atomic.
__global__ void k_count_slots(const int32_t* __restrict__ uslot, int64_t n, int32_t* __restrict__ cnt) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const unsigned act = __ballot_sync(0xffffffffu, i < n);
    if (i >= n) return;
    const int s = uslot[i];
    const unsigned peers = __match_any_sync(act, s);
    if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&cnt[s], __popc(peers));
}

// exclusive scan of ceil(cnt / 32) over slots (single CTA): each slot's first
// quadrant in base[s], the quadrant total in base[n_slots], the tile count
// (quadrants rounded up to whole tiles) in *n_tiles
__global__ void k_tile_scan(const int32_t* __restrict__ cnt, int n_slots, int slot_rows, int32_t* __restrict__ base,
                            int32_t* __restrict__ n_tiles) {
    __shared__ int32_t warp_tot[32];
    __shared__ int32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int start = 0; start < n_slots; start += blockDim.x) {
        const int s = start + threadIdx.x;
        // quadrants of the slot: its rows in granules of slot_rows (32: a quadrant, 128: a tile)
        const int32_t v = (s < n_slots) ? (cnt[s] + slot_rows - 1) / slot_rows * (slot_rows / kQuadRows) : 0;
        int32_t x = v;
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_tot[w] = x;
        __syncthreads();
        if (w == 0) {
            int32_t t = (lane < (int)(blockDim.x >> 5)) ? warp_tot[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += y;
            }
            warp_tot[lane] = t;
        }
        __syncthreads();
        const int32_t excl = carry + (w > 0 ? warp_tot[w - 1] : 0) + x - v;
        if (s < n_slots) base[s] = excl;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = excl + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        base[n_slots] = carry;
        *n_tiles = (carry + kQuads - 1) / kQuads;
    }
}

// quadrant -> slot; the quadrants that pad the last tile take the slot of the
// last used quadrant, so a tile whose used quadrants share a slot stays uniform
__global__ void k_tile_slots(const int32_t* __restrict__ cnt, const int32_t* __restrict__ base, int n_slots,
                             const int32_t* __restrict__ n_tiles, int32_t* __restrict__ quad_slot) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_slots) return;
    const int nq = base[s + 1] - base[s];
    for (int q = 0; q < nq; ++q) quad_slot[base[s] + q] = s;
    // the slot that owns the last used quadrant also pads the last tile
    const int used = base[n_slots];
    if (nq > 0 && base[s] + nq == used)
        for (int q = used; q < *n_tiles * kQuads; ++q) quad_slot[q] = s;
}

__global__ void k_scatter_tiles(const int32_t* __restrict__ active, int64_t n, const int32_t* __restrict__ uslot,
                                const int32_t* __restrict__ base, int32_t* __restrict__ fill,
                                int32_t* __restrict__ tile_univ) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const unsigned act = __ballot_sync(0xffffffffu, i < n);
    if (i >= n) return;
    const int s = uslot[i];
    // one atomic per slot per warp; the lanes of a slot take consecutive positions
    const unsigned peers = __match_any_sync(act, s);
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    int first = 0;
    if (lane == leader) first = atomicAdd(&fill[s], __popc(peers));
    first = __shfl_sync(peers, first, leader);
    const int pos = first + __popc(peers & ((1u << lane) - 1u));
    // quadrant base[s] + pos / 32, row pos % 32 of it: rows are numbered quadrant * 32 + row
    tile_univ[(int64_t)(base[s] + pos / kQuadRows) * kQuadRows + pos % kQuadRows] = active[i];
}

// ---------------------------------------------------------- mixed: y prep ---

__device__ __forceinline__ int64_t ytile_offset(int64_t t, int r, int c, int K) {
    // A-operand image of one BM-row tile: [2K/8 chunks][BM/8 row groups][8 rows][8 cols] bf16
    return t * (int64_t)(2 * K * kBM) + (int64_t)(c >> 3) * (kBM * 8) + (r >> 3) * 64 + (r & 7) * 8 + (c & 7);
}

// One CTA per tile quadrant (32 rows of one covariance slot): y^ = A (d - v) in
// binary32, Y = -2 y^ split into bf16 hi + lo, and the error-bound coefficient
// alpha in the spare column so that the screen directly yields a lower bound
// of chi2_g - c_u.  It also evaluates the row's screen value at its own
// covariance point q (= cur[u]) with an upper bound UB_q: no grid point with
// LB >= UB_q can be the minimum, so tau0 = UB_q seeds the screen's top-k
// threshold.
// The product is a 32 x K x N_fit contraction: lane = row, warp = 16 columns
// of the image (one after another when K has more of them than the CTA has
// warps), A in shared memory kYJ rows at a time, read as broadcasts of four
// columns, d - v transposed beside it; two columns share a packed
// multiply-add, and each column keeps one chain over j in increasing order.
// Bound by instruction issue where tiles are many (staging and the bf16 split
// cost as much as the products); where they are few, a quadrant per CTA and 16
// columns per warp keep its latency to a few microseconds (one thread per row
// walked all N^2 products alone).  Loads are asynchronous copies, all in flight
// at once: with plain loads a CTA spent 20 of 22 us waiting for them in turn.
// Prep stage against one thread per row: full 100x100 job 14.2 -> 10.6 ms,
// 128 points of 64^3 21.1 -> 3.2 ms, 4 points with N = 200 18.1 -> 2.0 ms.
constexpr int kYJ = 32;         // rows of A staged at a time above N_fit = 64 (all of them up to it)
constexpr int kYPad = kQuadRows + 1;  // row stride of the transposed vectors (conflict-free both ways)
constexpr int kYSums = 7;       // per-row sums that cross warps

__host__ __device__ inline int yprep_warps(int K) { return K / 16 <= 8 ? K / 16 : (K / 16 + 1) / 2; }
__host__ __device__ inline int yprep_rows(int nfit) { return nfit <= kResolveMaxN ? nfit : kYJ; }
inline size_t yprep_smem(int nfit, int K) {
    return (size_t)(yprep_rows(nfit) * K + 2 * nfit * kYPad + yprep_warps(K) * kYSums * kQuadRows) * sizeof(float);
}
// 4-byte asynchronous copy to shared memory: the CTA's loads are all in flight at once
__device__ __forceinline__ void copy4_async(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__global__ void k_yprep(const int32_t* __restrict__ quad_slot, const int32_t* __restrict__ tile_univ,
                        const float* __restrict__ d, const float2* __restrict__ centre, int nfit, int K,
                        const float* __restrict__ A32, const float* __restrict__ rho, const int32_t* __restrict__ cur,
                        GridSpec gs, const float4* __restrict__ gnorm, const float* __restrict__ Qc,
                        const float* __restrict__ Qb, int64_t G_pad, uint16_t* __restrict__ Yt,
                        float4* __restrict__ alpha, float* __restrict__ tau0, int32_t* __restrict__ tile_j0) {
    extern __shared__ float4 s_yprep[];
    const int jc = yprep_rows(nfit);
    float* sA = reinterpret_cast<float*>(s_yprep);       // [jc][K] rows of A
    float* sd = sA + jc * K;                             // [nfit][kYPad] d - v
    float* sq = sd + nfit * kYPad;                       // [nfit][kYPad] probe rows
    float* sred = sq + nfit * kYPad;                     // [warps][kYSums][32]
    const int64_t t = blockIdx.x / kQuads;
    const int quad = blockIdx.x % kQuads;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int r = quad * kQuadRows + lane;               // row of the tile
    const int u = tile_univ[t * kBM + r];
    const int q = u >= 0 ? cur[u] : -1;
    // the screen walks this tile's grid tiles starting at the one holding row 0's q
    if (quad == 0 && threadIdx.x == 0) tile_j0[t] = (u >= 0) ? q / kBN : 0;
    if (!__any_sync(0xffffffffu, u >= 0)) {  // the same in every warp: a quadrant of padding
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        for (int c8 = warp; c8 < 2 * K / 8; c8 += nw) *reinterpret_cast<uint4*>(Yt + ytile_offset(t, r, c8 * 8, K)) = z;
        if (warp == 0) {
            alpha[t * kBM + r] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            tau0[t * kBM + r] = -FLT_MAX;  // padding rows keep no candidate
        }
        return;
    }
    const int slot = quad_slot[t * kQuads + quad];
    const float* A = A32 + (size_t)slot * nfit * nfit;
    auto stage_A = [&](int j0) {  // A is symmetric: row j is column j
        const int nj = min(jc, nfit - j0);
        for (int j = warp; j < nj; j += nw)
            for (int i = lane; i < K; i += 32) {
                if (i < nfit)
                    copy4_async(sA + j * K + i, A + (size_t)(j0 + j) * nfit + i);
                else
                    sA[j * K + i] = 0.0f;
            }
    };
    // data and probe rows, one row per warp at a time (coalesced), stored transposed
    for (int k = warp; k < kQuadRows; k += nw) {
        const int uk = __shfl_sync(0xffffffffu, u, k), qk = __shfl_sync(0xffffffffu, q, k);
        for (int j = lane; j < nfit; j += 32) {
            if (uk >= 0)
                copy4_async(sd + j * kYPad + k, d + (size_t)uk * nfit + j);
            else
                sd[j * kYPad + k] = 0.0f;
            if (uk >= 0 && gs.Sc32)
                copy4_async(sq + j * kYPad + k, gs.Sc32 + (size_t)qk * nfit + j);
            else
                sq[j * kYPad + k] = 0.0f;
        }
    }
    stage_A(0);
    if (!gs.Sc32) {  // rows evaluated from the model
        for (int k = warp; k < kQuadRows; k += nw) {
            const int qk = __shfl_sync(0xffffffffu, q, k);
            if (qk < 0) continue;
            const FitRow fr = fit_row(gs, qk);
            for (int j = lane; j < nfit; j += 32) sq[j * kYPad + k] = row_sc32(gs, fr, j);
        }
    }
    copy_async_wait();
    // d - v by the thread that copied the value; v as double-float keeps the difference off the narrow
    // binary64 pipe.  Its error is at most 1.5 2^-24 |d - v|: one half unit from rounding the result, and what
    // v loses as hi + lo, at most 2^-24 |lo|, where |lo| is below |d - v| unless d = hi (then the result is -lo
    // itself), and where it comes near |d - v| hi - d + lo loses at most the bit that makes up the sum.
    for (int k = warp; k < kQuadRows; k += nw) {
        const bool used = __shfl_sync(0xffffffffu, u, k) >= 0;
        for (int j = lane; j < nfit; j += 32)
            if (used) sd[j * kYPad + k] = -df_sub_f(centre[j], sd[j * kYPad + k]).x;
    }
    __syncthreads();
    float yn2 = 0.0f, yl2 = 0.0f, yhl2 = 0.0f, ry2 = 0.0f, dot = 0.0f, adot = 0.0f, dn2 = 0.0f;
    for (int c0 = warp * 16; c0 - warp * 16 < K; c0 += nw * 16) {  // the same trip count for every warp
        f32x2 y[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) y[k] = 0ull;
        for (int j0 = 0; j0 < nfit; j0 += jc) {
            const int nj = min(jc, nfit - j0);
            if (jc < nfit && (j0 > 0 || c0 >= nw * 16)) {  // rows past the first ones staged above
                __syncthreads();
                stage_A(j0);
                copy_async_wait();
                __syncthreads();
            }
            if (c0 < K) {
#pragma unroll 4
                for (int j = 0; j < nj; ++j) {
                    const float v = sd[(j0 + j) * kYPad + lane];
                    const f32x2 vv = x2_pack(v, v);
                    const ulonglong2* a4 = reinterpret_cast<const ulonglong2*>(sA + j * K + c0);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const ulonglong2 a = a4[k];
                        y[2 * k] = x2_fma(a.x, vv, y[2 * k]);
                        y[2 * k + 1] = x2_fma(a.y, vv, y[2 * k + 1]);
                    }
                }
            }
        }
        if (c0 < K) {
            uint32_t vh[8], vl[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                vh[k] = vl[k] = 0u;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int i = c0 + 2 * k + h;
                    const float Y = -2.0f * (h ? x2_hi(y[k]) : x2_lo(y[k]));
                    const float sv = i < nfit ? sq[i * kYPad + lane] : 0.0f;
                    yn2 = fmaf(Y, Y, yn2);
                    dot = fmaf(Y, sv, dot);
                    adot = fmaf(fabsf(Y), fabsf(sv), adot);
                    const __nv_bfloat16 hi = __float2bfloat16_rn(Y);
                    const float rem = Y - __bfloat162float(hi);           // exact
                    const __nv_bfloat16 l = __float2bfloat16_rn(rem);
                    const float lo = __bfloat162float(l), hl = __bfloat162float(hi) + lo;
                    const float ry = rem - lo;                            // exact: r_Y = Y - hi - lo
                    yl2 = fmaf(lo, lo, yl2);
                    yhl2 = fmaf(hl, hl, yhl2);
                    ry2 = fmaf(ry, ry, ry2);
                    if (i < nfit) {
                        vh[k] |= (uint32_t)__bfloat16_as_ushort(hi) << (16 * h);
                        vl[k] |= (uint32_t)__bfloat16_as_ushort(l) << (16 * h);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                *reinterpret_cast<uint4*>(Yt + ytile_offset(t, r, c0 + 8 * k, K)) =
                    make_uint4(vh[4 * k], vh[4 * k + 1], vh[4 * k + 2], vh[4 * k + 3]);
                *reinterpret_cast<uint4*>(Yt + ytile_offset(t, r, K + c0 + 8 * k, K)) =
                    make_uint4(vl[4 * k], vl[4 * k + 1], vl[4 * k + 2], vl[4 * k + 3]);
            }
        }
    }
    for (int j = warp; j < nfit; j += nw) {
        const float v = sd[j * kYPad + lane];
        dn2 = fmaf(v, v, dn2);
    }
    const float sums[kYSums] = {yn2, yl2, yhl2, ry2, dot, adot, dn2};
#pragma unroll
    for (int k = 0; k < kYSums; ++k) sred[(warp * kYSums + k) * kQuadRows + lane] = sums[k];
    __syncthreads();
    if (warp != 0) return;
    float tot[kYSums];
#pragma unroll
    for (int k = 0; k < kYSums; ++k) {
        tot[k] = 0.0f;
        for (int w = 0; w < nw; ++w) tot[k] += sred[(w * kYSums + k) * kQuadRows + lane];
    }
    if (u < 0) {  // its Y is zero already
        alpha[t * kBM + r] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        tau0[t * kBM + r] = -FLT_MAX;
        return;
    }
    yn2 = tot[0], yl2 = tot[1], yhl2 = tot[2], ry2 = tot[3], dot = tot[4], adot = tot[5], dn2 = tot[6];
    // -2 y.s~_g - (hi*hi + lo*hi + hi*lo products)  =  -2 (y - y^).s~ + Y_lo.S_lo + (Y_hi + Y_lo).r_S + r_Y.s~
    // and the binary32 accumulation of the 3K products (each add bounded as truncated, Sum|products| <= 1.02 |Y||s~|):
    //   |error| <= [2 |y - y^| + |r_Y| + (3K+2) 1.02 2^-23 |Y|] |s~| + |Y_lo| |S_lo| + |Y_hi+Y_lo| |r_S|
    // with |y - y^| <= (nfit+2.5) 2^-24 rho |d~| (A rounded to binary32, d~ as above, binary32 dot products).
    const float dn = sqrtf(dn2) * 1.0001f, yn = sqrtf(yn2) * 1.0001f;
    const float a_acc = 1.02f * (2.0f * ((float)nfit + 2.5f) * 5.9604645e-08f * rho[slot] * dn +
                                 (float)(3 * K + 2) * 1.1920929e-07f * 1.02f * yn + sqrtf(ry2));
    const float4 al = make_float4(a_acc, 1.0001f * sqrtf(yl2), 1.0001f * sqrtf(yhl2), 0.0f);
    alpha[t * kBM + r] = al;
    // the spare columns nfit .. nfit+2 of the hi half (written as zero above, before the barrier)
    Yt[ytile_offset(t, r, nfit, K)] = __bfloat16_as_ushort(__float2bfloat16_rd(-al.x));
    Yt[ytile_offset(t, r, nfit + 1, K)] = __bfloat16_as_ushort(__float2bfloat16_rd(-al.y));
    Yt[ytile_offset(t, r, nfit + 2, K)] = __bfloat16_as_ushort(__float2bfloat16_rd(-al.z));
    // probe at q: sigma^ = q^_q + Y.s~_q (binary32), |sigma^ - sigma| <= 2|y - y^||s~_q| + |q^ - q|
    //   + (nfit+1) 2^-24 (sum |Y_i s~_i| + |q^|) + 2^-24 |sigma^|   (all inside eps below)
    const int64_t qi = (int64_t)slot * G_pad + q;
    const float qc = Qc[qi];
    const float sig = qc + dot;
    const float eps = bound_dot(al, gnorm[q]) + (qc - Qb[qi]) +
                      (float)(nfit + 2) * 5.9604645e-08f * (adot + fabsf(qc)) + 1.1920929e-07f * (fabsf(sig) + 1.0f);
    tau0[t * kBM + r] = (sig + 2.0f * eps) * 1.0000005f + 1.0e-6f + 4.7683716e-07f * fabsf(sig);
}

// ------------------------------------------------------- mixed: resolution --

constexpr int kItemCu = kMaxTopK;     // item codes beyond the candidates
constexpr int kItemP = kMaxTopK + 1;
constexpr int kItemMin = kMaxTopK + 2;
constexpr int kItemCodes = kMaxTopK + 3;

// Resolution of a top-k round, as five flat launches (launch_resolve): the
// residuals are the work, and a tile's rows need very different numbers of
// them, so they are evaluated from flat lists that keep every lane busy
// instead of inside the tile's CTA (where the lanes of rows with few residuals
// waited at barriers for the rows with many).
//  k_resolve_emit     per row: the screen certificate (decide_row); the
//                     residual items the row needs, appended in tile order;
//  k_resid_tiles/rows every item's double-float residual chi2 under the row's
//                     covariance slot: a thread per item in well-filled tiles,
//                     a warp per group of items else (launch_resolve);
//  k_resolve_conclude per row: the same decision again, then the rescored
//                     minimum and its certificate; finish (dchi2) / advance /
//                     hand on, exactly as one kernel did before; rescored rows
//                     that finish with p != best list their chi2_p;
//  k_resid_tiles/rows those chi2_p;
//  k_resolve_tail     their dchi2.
// Decision per row (§2 steps 3-4 with the screen's certificate):
//  1. from the screen's lower bounds LB and upper bounds UB = LB + 2 eps of
//     its candidates, accept the first candidate when it is the only one that
//     can still be the minimum and its UB is below every outside bound tau;
//  2. otherwise the residual-form chi2 of every candidate that can still be
//     the minimum (and c_u = |W (d - v)|^2 when the certificate needs it):
//     the first minimum, certified against tau, else the universe is handed
//     to the next round;
//  3. universes whose minimum repeats their covariance index (or that used
//     their last scan) finish with dchi2 = chi2_p - chi2_min; the others
//     move their covariance index to the minimum.
struct RowDecision {
    int state;  // 0 padding, 1 certified by the bounds, 2 rescoring, 3 nothing below the seed
    bool full;
    float tau, min_ub;
    int ncodes;                      // residual items of the row, in emission order
    uint8_t code[kMaxTopK + 1];      // candidate j < topk, kItemCu, kItemP, kItemMin
    int32_t g[kMaxTopK];
    float lb[kMaxTopK];
};

__device__ __forceinline__ void decide_row(const ResolveArgs& a, int64_t row, int slot, int u, RowDecision& D) {
    const int topk = a.topk;
    D.state = 0;
    D.ncodes = 0;
    D.full = false;
    D.tau = FLT_MAX;
    D.min_ub = FLT_MAX;
    if (u < 0) return;
    const float4 al = a.alpha[row];
    float ub[kMaxTopK];
    int nvalid = 0;
    for (int j = 0; j < topk; ++j) {
        const int32_t gj = a.cidx[row * topk + j];
        D.g[j] = gj;
        D.lb[j] = a.cval[row * topk + j];
        ub[j] = FLT_MAX;
        if (gj < 0) continue;
        ++nvalid;
        const int64_t q = (int64_t)slot * a.G_pad + gj;
        const float eps = bound_dot(al, a.gnorm[gj]) + (a.Qc[q] - a.Qb[q]);
        ub[j] = D.lb[j] + 2.0f * eps + 4.7683716e-07f * (fabsf(D.lb[j]) + fabsf(a.Qc[q]) + 1.0f);
        D.min_ub = fminf(D.min_ub, ub[j]);
    }
    // every grid point outside the list has LB >= the k-th kept value; an empty slot holds the
    // seed tau0 = UB of the row's probe, so a list that is not full holds every point that can
    // be the minimum
    D.full = (nvalid == topk);
    D.tau = D.lb[topk - 1] - 4.7683716e-07f * (fabsf(D.lb[topk - 1]) + 1.0f);
    int nR = 0;
    for (int j = 0; j < topk; ++j)
        if (D.g[j] >= 0 && D.lb[j] <= D.min_ub) ++nR;
    if (nvalid == 0) {
        D.state = 3;  // nothing below the seed: only possible with non-finite data
    } else if (nR == 1 && ub[0] < D.tau) {
        D.state = 1;
        // a universe that finishes on this certificate needs chi2_p and chi2_min in residual form
        if (D.g[0] == a.cur[u] || a.nscan[u] + 1 >= a.maxit[u]) {
            if (a.pt[u] != D.g[0]) D.code[D.ncodes++] = (uint8_t)kItemP;
            D.code[D.ncodes++] = (uint8_t)kItemMin;
        }
    } else {
        D.state = 2;
        for (int j = 0; j < topk; ++j)
            if (D.g[j] >= 0 && D.lb[j] <= D.min_ub) D.code[D.ncodes++] = (uint8_t)j;
        if (D.full && !(D.min_ub < D.tau)) D.code[D.ncodes++] = (uint8_t)kItemCu;
    }
}

// exclusive prefix sum of v over a CTA of kBM threads; *total receives the sum
__device__ __forceinline__ int block_excl_scan(int v, int* s_warp, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    int before = 0, sum = 0;
    for (int w = 0; w < kBM / 32; ++w) {
        before += (w < warp) ? s_warp[w] : 0;
        sum += s_warp[w];
    }
    *total = sum;
    return before + x - v;
}

__global__ void __launch_bounds__(kBM) k_resolve_emit(ResolveArgs a) {
    __shared__ int s_warp[kBM / 32];
    __shared__ int s_base;
    const int64_t t = blockIdx.x;
    const int64_t row = t * kBM + threadIdx.x;
    const int slot = a.quad_slot[row / kQuadRows];
    const int u = a.tile_univ[row];
    // an aborted screen's candidates are incomplete (and may be unwritten): nothing is read of them
    const bool aborted = (*a.status & kDevTimeout) != 0;
    RowDecision D;
    decide_row(a, row, slot, aborted ? -1 : u, D);
    int total = 0;
    const int off = block_excl_scan(D.ncodes, s_warp, &total);
    if (threadIdx.x == 0) {
        s_base = total ? atomicAdd(&a.counts[0], total) : 0;
        // a warp is a quadrant (one covariance): its rows' items are one contiguous range
        int q0 = s_base;
        for (int w = 0; w < kQuads; ++w) {
            a.tile_items[t * kQuads + w] = make_int2(q0, s_warp[w]);
            q0 += s_warp[w];
        }
        if (total) atomicAdd(a.n_resid, (unsigned long long)total);
    }
    __syncthreads();
    const int base = s_base + off;
    a.item_base[row] = base;
    for (int k = 0; k < D.ncodes; ++k) {
        const int c = D.code[k];
        const int32_t g = (c < kMaxTopK) ? D.g[c] : (c == kItemCu ? -1 : (c == kItemP ? a.pt[u] : D.g[0]));
        a.items[base + k] = make_int2((int32_t)row, g);
    }
}

// Residual chi2 of one tile's items, for launches whose tiles are well filled
// (N_fit <= 64, stored rows).  The items of each quadrant are a contiguous
// range (tile_items[4t + w]) and the tile's quadrants follow each other; a run
// of quadrants with one covariance slot shares one W, staged in shared memory
// (every lane reads the same element at once), and the lanes stride over the
// run's items with no barrier but the staging's.  A tile whose quadrants share
// one slot stages once.  Small CTAs (two warps) keep the last, partly filled
// round of a run cheap.  Bound by the binary32 pipe (52 % active at N = 45) and
// the latency of ten warps an SM, all that 140 registers leave: the packed
// multiply-add takes 14 instructions for two (24 unpacked) and one 16-byte
// broadcast of W instead of two 8-byte ones; scan 1 of 1000 points x 1000
// universes of N = 45 1.12 -> 0.88 ms, the full 100x100 job 178.1 -> 171.1.
constexpr int kResidThreads = 64;

template <int NR>
__global__ void __launch_bounds__(kResidThreads, 6) k_resid_tiles(const ResolveArgs a, const int2* __restrict__ items,
                                                                 const int2* __restrict__ tile_items,
                                                                 double* __restrict__ res) {
    extern __shared__ ulonglong2 sWd[];
    const int n = a.nfit;
    const int nw = df_blocks(n) * n * 2;
    const int64_t t = blockIdx.x;
    int w0 = 0;
    while (w0 < kQuads) {  // every bound below is the same for all lanes
        const int slot = a.quad_slot[t * kQuads + w0];
        int w1 = w0 + 1;
        while (w1 < kQuads && a.quad_slot[t * kQuads + w1] == slot) ++w1;
        const int64_t i0 = tile_items[t * kQuads + w0].x;
        const int2 last = tile_items[t * kQuads + w1 - 1];
        const int64_t i1 = (int64_t)last.x + last.y;
        w0 = w1;
        if (i1 <= i0) continue;
        const ulonglong2* Wg = reinterpret_cast<const ulonglong2*>(a.Wdf + (size_t)slot * wdf_floats(n));
        __syncthreads();  // the previous run's reads of sWd are done
        for (int e = threadIdx.x; e < nw; e += blockDim.x) sWd[e] = Wg[e];
        __syncthreads();
        for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            const int2 it = items[i];
            const int u = a.tile_univ[it.x];
            res[i] = resid_df_reg<NR>(sWd, n, srow<false>(a.gs, a.centre_df, it.y), a.d + (size_t)u * n);
        }
    }
}

// Every other launch: groups of kRowsB consecutive items per warp, grid-stride
// over the device count.  A row's items follow each other and the rows of a
// tile quadrant share a slot, so a group mostly has one W; where the slot
// changes inside a group, its runs go one after the other.
template <bool MODEL>
__global__ void __launch_bounds__(32 * kRowsWarps) k_resid_rows(const ResolveArgs a, const int2* __restrict__ items,
                                                                const int32_t* __restrict__ count,
                                                                double* __restrict__ res) {
    extern __shared__ float4 s_rows[];
    const int n = a.nfit;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* sm = reinterpret_cast<float*>(s_rows) + warp * rows_floats(n);
    const int64_t total = *count;
    const int64_t step = (int64_t)gridDim.x * kRowsWarps * kRowsB;
    for (int64_t e = ((int64_t)blockIdx.x * kRowsWarps + warp) * kRowsB; e < total; e += step) {
        const int m = (int)(total - e < kRowsB ? total - e : kRowsB);
        for (int k0 = 0; k0 < m;) {
            const int slot = a.quad_slot[items[e + k0].x / kQuadRows];
            int k1 = k0;
            for (; k1 < m; ++k1) {
                const int2 it = items[e + k1];
                if (a.quad_slot[it.x / kQuadRows] != slot) break;
                rows_stage(sm, k1 - k0, n, srow<MODEL>(a.gs, a.centre_df, it.y), a.d + (size_t)a.tile_univ[it.x] * n,
                           lane);
            }
            const double c = rows_chi2(a.Wdf + (size_t)slot * wdf_floats(n), n, sm, k1 - k0, lane);
            if (lane < k1 - k0) res[e + k0 + lane] = c;
            k0 = k1;
        }
    }
}

__global__ void __launch_bounds__(kBM) k_resolve_conclude(ResolveArgs a) {
    if (*a.status & kDevTimeout) {  // an aborted screen decides nothing, and leaves no items to k_resid_tiles
        if (threadIdx.x < kQuads) a.tile_items2[blockIdx.x * (int64_t)kQuads + threadIdx.x] = make_int2(0, 0);
        return;
    }
    __shared__ int s_nnext, s_nfb, s_n2[kQuads], s_cnt[3];
    __shared__ int s_base_next, s_base_fb, s_base2;
    const int64_t t = blockIdx.x;
    const int r = threadIdx.x;
    const int64_t row = t * kBM + r;
    const int slot = a.quad_slot[row / kQuadRows];
    const int u = a.tile_univ[row];
    if (r == 0) {
        s_nnext = 0;
        s_nfb = 0;
        for (int w = 0; w < kQuads; ++w) s_n2[w] = 0;
        s_cnt[0] = s_cnt[1] = s_cnt[2] = 0;
    }
    __syncthreads();
    RowDecision D;
    decide_row(a, row, slot, u, D);
    const int base = a.item_base[row];
    const int topk = a.topk;
    int state = D.state;
    int32_t g_best = -1;
    double chi2_min = 0.0, chi2_p = 0.0;
    bool have_min = false, have_p = false;
    if (state == 1) {
        g_best = D.g[0];
        for (int k = 0; k < D.ncodes; ++k) {
            if (D.code[k] == kItemMin) {
                chi2_min = a.res[base + k];
                have_min = true;
            } else if (D.code[k] == kItemP) {
                chi2_p = a.res[base + k];
                have_p = true;
            }
        }
        atomicAdd(&s_cnt[0], 1);
    } else if (state == 2) {
        double bchi = DBL_MAX, cu = 0.0;
        int32_t bg = INT32_MAX;
        for (int k = 0; k < D.ncodes; ++k) {
            const int c = D.code[k];
            const double v = a.res[base + k];
            if (c == kItemCu) {
                cu = v;
            } else if (v < bchi || (v == bchi && D.g[c] < bg)) {
                bchi = v;
                bg = D.g[c];
            }
        }
        bool ok = (!D.full || (D.min_ub < D.tau)) && bg != INT32_MAX;
        if (!ok && bg != INT32_MAX) ok = (double)D.tau > (bchi - cu) + 1e-9 * (fabs(bchi) + fabs(cu));
        if (ok) {
            state = 1;
            g_best = bg;
            chi2_min = bchi;
            have_min = true;
            atomicAdd(&s_cnt[1], 1);
        } else {
            state = 3;
            atomicAdd(&s_cnt[2], 1);
            // every grid point that can still be the minimum has LB <= sigma* = chi2_min - c_u of the
            // best candidate found: a list screen seeded with sigma* (rounded up) lists all of them
            if (a.thr) {
                const double sig = (bchi - cu) + 1e-9 * (fabs(bchi) + fabs(cu));
                a.thr[u] = __double2float_ru(sig) + 4.7683716e-07f * (fabsf((float)sig) + 1.0f);
            }
        }
    } else if (state == 3) {
        atomicAdd(&s_cnt[2], 1);
        if (a.thr) a.thr[u] = FLT_MAX;
    }
    (void)topk;
    if (state == 1 && a.rmask)
        a.rmask[u] |= a.round_bit ? a.round_bit : (D.state == 2 ? kDecidedRescored : kDecidedCert);
    // finish converged / exhausted universes, advance the others
    bool finishing = false, tail = false;
    int32_t p = -1;
    if (state == 1) {
        a.best[u] = g_best;
        finishing = (g_best == a.cur[u]) || (a.nscan[u] + 1 >= a.maxit[u]);
        if (finishing) {
            p = a.pt[u];
            // a rescored row that finishes still needs chi2_p (the certified ones listed it already)
            tail = (p != g_best) && !have_p;
        } else {
            a.cur[u] = g_best;
            a.nscan[u] = (int8_t)(a.nscan[u] + 1);
        }
    }
    const bool to_next = (state == 1 && !finishing);
    const int my_next = to_next ? atomicAdd(&s_nnext, 1) : -1;
    const int my_fb = (state == 3) ? atomicAdd(&s_nfb, 1) : -1;
    // chi2_p items stay grouped by quadrant (one W per residual CTA)
    const int quad = r / kQuadRows;
    const int my_2 = tail ? atomicAdd(&s_n2[quad], 1) : -1;
    __syncthreads();
    if (r == 0) {
        s_base_next = s_nnext ? atomicAdd(a.n_next, s_nnext) : 0;
        s_base_fb = s_nfb ? atomicAdd(a.n_fb, s_nfb) : 0;
        const int n2 = s_n2[0] + s_n2[1] + s_n2[2] + s_n2[3];
        s_base2 = n2 ? atomicAdd(&a.counts[1], n2) : 0;
        int q0 = s_base2;
        for (int w = 0; w < kQuads; ++w) {
            a.tile_items2[t * kQuads + w] = make_int2(q0, s_n2[w]);
            q0 += s_n2[w];
        }
        if (n2) atomicAdd(a.n_resid, (unsigned long long)n2);
        if (s_cnt[0]) atomicAdd(&a.counters[0], (unsigned long long)s_cnt[0]);
        if (s_cnt[1]) atomicAdd(&a.counters[1], (unsigned long long)s_cnt[1]);
        if (s_cnt[2]) atomicAdd(&a.counters[2], (unsigned long long)s_cnt[2]);
    }
    __syncthreads();
    if (to_next) a.next[s_base_next + my_next] = u;
    if (state == 3) a.fb[s_base_fb + my_fb] = u;
    if (tail) {
        int pos = s_base2 + my_2;
        for (int w = 0; w < quad; ++w) pos += s_n2[w];
        a.items2[pos] = make_int2((int32_t)row, p);
        a.cmin2[pos] = chi2_min;
    } else if (finishing) {
        a.dchi2[u] = (p == g_best) ? 0.0 : chi2_p - chi2_min;
        if (a.chi2min) a.chi2min[u] = chi2_min;
        a.nscan[u] = (int8_t)(a.nscan[u] + 1);
        atomicSub(&a.job_left[a.job_of[u]], 1);
    }
}

__global__ void k_resolve_tail(ResolveArgs a) {
    const int64_t total = a.counts[1];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int u = a.tile_univ[a.items2[i].x];
        const double cmin = a.cmin2[i];
        a.dchi2[u] = a.res2[i] - cmin;
        if (a.chi2min) a.chi2min[u] = cmin;
        a.nscan[u] = (int8_t)(a.nscan[u] + 1);
        atomicSub(&a.job_left[a.job_of[u]], 1);
    }
}

// List rounds: every grid point whose screen lower bound is at or below the
// row's seed (an upper bound of the minimum) is listed, so the residual-form
// minimum over a complete list is the minimum of the scan.  A row's list is
// cut into chunks of lp.pts points, a warp each, so a long list spreads over
// many warps.  k_list_plan checks each listed row (rows[] holds
// the round's occupied tile rows) and reserves its chunks; rows whose list
// overflowed go to the exact scan (their counts size the next, exact-size list
// round).
__global__ void k_list_plan(ResolveArgs a, const int32_t* __restrict__ cand_count, const int32_t* __restrict__ rows,
                            int64_t n_rows, const int32_t* __restrict__ n_rows_dev, ListPlan lp) {
    const int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (w >= n_rows || w >= *n_rows_dev) return;
    if (*a.status & kDevTimeout) return;  // an aborted screen's counts are not read: no chunks, nothing handed on
    const int64_t row = rows[w];
    const int u = a.tile_univ[row];
    const int n0 = cand_count[row * 2], n1 = cand_count[row * 2 + 1];
    bool complete;
    if (a.list_off) {
        const int2 want = a.list_n[u];
        complete = (n0 == want.x && n1 == want.y);
    } else {
        complete = (n0 >= 0 && n1 >= 0 && n0 <= kListCap && n1 <= kListCap);
    }
    lp.row_nc[w] = 0;
    if (complete && n0 + n1 > 0) {
        const int nc = (n0 + n1 + lp.pts - 1) / lp.pts;
        const int base = atomicAdd(lp.n_chunk, nc);
        if ((int64_t)base + nc <= lp.max_chunks) {
            lp.row_base[w] = base;
            lp.row_done[w] = 0;
            lp.row_nc[w] = nc;
            for (int k = 0; k < nc; ++k) lp.chunk[base + k] = make_int2((int32_t)w, k);
            return;
        }
        // no room (the host's bound makes this unreachable): void the reservation, take the exact scan
        for (int64_t k = base; k < lp.max_chunks && k < (int64_t)base + nc; ++k) lp.chunk[k] = make_int2(-1, 0);
    }
    if (a.lcount) a.lcount[u] = (n0 >= 0 && n1 >= 0) ? make_int2(n0, n1) : make_int2(-1, -1);
    a.fb[atomicAdd(a.n_fb, 1)] = u;
    atomicAdd(&a.counters[1], 1ull);
}

// One warp per chunk (grid-stride over the device count): the warp scores the
// chunk's points in groups of kRowsB with the canonical residual (rows_chi2),
// takes the first minimum (lowest index among equal values) and publishes it.
// The warp that completes a row's last chunk takes the first minimum over the
// row's chunks and finishes (dchi2) or advances the row.
// Four CTAs an SM where rows are stored: the lists of 128 points of 64^3 take
// 38.4 ms, with the registers of three 40.6.
template <bool MODEL>
__global__ void __launch_bounds__(32 * kRowsWarps, MODEL ? 3 : 4) k_list_chunks(ResolveArgs a, const int32_t* __restrict__ cand_count,
                                                                 const int32_t* __restrict__ rows, ListPlan lp) {
    extern __shared__ float4 s_rows[];
    const int n = a.nfit;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* sm = reinterpret_cast<float*>(s_rows) + warp * rows_floats(n);
    const int64_t total = *lp.n_chunk < lp.max_chunks ? (int64_t)*lp.n_chunk : lp.max_chunks;
    const int64_t stride = (int64_t)gridDim.x * kRowsWarps;
    for (int64_t e = (int64_t)blockIdx.x * kRowsWarps + warp; e < total; e += stride) {
        const int2 ck = lp.chunk[e];
        if (ck.x < 0) continue;
        const int w = ck.x;
        const int64_t row = rows[w];
        const int u = a.tile_univ[row];
        const float* W = a.Wdf + (size_t)a.quad_slot[row / kQuadRows] * wdf_floats(n);
        const int n0 = cand_count[row * 2], n1 = cand_count[row * 2 + 1];
        int64_t base0, base1;
        if (a.list_off) {
            base0 = a.list_off[u];
            base1 = base0 + a.list_n[u].x;
        } else {
            base0 = row * 2 * (int64_t)kListCap;
            base1 = base0 + kListCap;
        }
        const float* du = a.d + (size_t)u * n;
        double bv = DBL_MAX;
        int32_t bg = INT32_MAX;
        const int k_end = min((ck.y + 1) * lp.pts, n0 + n1);
        for (int k0 = ck.y * lp.pts; k0 < k_end; k0 += kRowsB) {
            const int m = min(kRowsB, k_end - k0);
            int32_t mine = INT32_MAX;  // lane k: the group's point k
            for (int k = 0; k < m; ++k) {
                const int32_t g = a.cidx[(k0 + k < n0) ? base0 + k0 + k : base1 + (k0 + k - n0)];
                if (lane == k) mine = g;
                rows_stage(sm, k, n, srow<MODEL>(a.gs, nullptr, g), du, lane);
            }
            const double c = rows_chi2(W, n, sm, m, lane);
            if (lane < m && (c < bv || (c == bv && mine < bg))) {
                bv = c;
                bg = mine;
            }
        }
        warp_argmin(bv, bg);
        int last = 0;
        if (lane == 0) {
            const int pos = lp.row_base[w] + ck.y;
            lp.pv[pos] = bv;
            lp.pg[pos] = bg;
            __threadfence();
            last = (atomicAdd(&lp.row_done[w], 1) == lp.row_nc[w] - 1);
        }
        if (!__shfl_sync(0xffffffffu, last, 0)) continue;
        __threadfence();
        bv = DBL_MAX;
        bg = INT32_MAX;
        const int nc = lp.row_nc[w], rb = lp.row_base[w];
        for (int j = lane; j < nc; j += 32) {
            const double v = __ldcg(&lp.pv[rb + j]);
            const int32_t gg = __ldcg(&lp.pg[rb + j]);
            if (v < bv || (v == bv && gg < bg)) {
                bv = v;
                bg = gg;
            }
        }
        warp_argmin(bv, bg);
        if (lane == 0 && a.rmask) a.rmask[u] |= a.round_bit;
        if (lane == 0 && a.n_resid) atomicAdd(a.n_resid, (unsigned long long)(n0 + n1));
        const int32_t cur_u = a.cur[u];
        const bool none = bg == INT32_MAX;  // no chi2 of the list compares: best -1, NaN (as k_finish)
        const bool finishing = none || (bg == cur_u) || (a.nscan[u] + 1 >= a.maxit[u]);
        if (finishing) {
            const int p = a.pt[u];
            double cp = 0.0;
            if (none) {
                bg = -1;
                bv = CUDART_NAN;
            } else if (p != bg) {
                rows_stage(sm, 0, n, srow<MODEL>(a.gs, nullptr, p), du, lane);
                cp = rows_chi2(W, n, sm, 1, lane);
                if (lane == 0 && a.n_resid) atomicAdd(a.n_resid, 1ull);
            }
            if (lane == 0) {
                a.best[u] = bg;
                a.dchi2[u] = (p == bg) ? 0.0 : cp - bv;
                if (a.chi2min) a.chi2min[u] = bv;
                a.nscan[u] = (int8_t)(a.nscan[u] + 1);
                atomicSub(&a.job_left[a.job_of[u]], 1);
                atomicAdd(&a.counters[0], 1ull);
            }
        } else if (lane == 0) {
            a.best[u] = bg;
            a.cur[u] = bg;
            a.nscan[u] = (int8_t)(a.nscan[u] + 1);
            a.next[atomicAdd(a.n_next, 1)] = u;
            atomicAdd(&a.counters[0], 1ull);
        }
    }
}

__global__ void k_or_mask(const int32_t* __restrict__ list, int64_t n, uint8_t bit, uint8_t* __restrict__ rmask) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) rmask[list[i]] |= bit;
}

__global__ void k_min_tau(const int32_t* __restrict__ tile_univ, int64_t n_rows, const float* __restrict__ thr,
                          float* __restrict__ tau0) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n_rows) return;
    const int u = tile_univ[i];
    if (u >= 0) tau0[i] = fminf(tau0[i], thr[u]);
}

// ---------------------------------------------------------- finishing -------

// One warp per finishing universe (*count of list): chi2_p and chi2_min in residual form under
// the last scan's covariance (A = W^T W), dchi2 = chi2_p - chi2_min.
template <bool MODEL>
__global__ void __launch_bounds__(128) k_finish(const int32_t* __restrict__ list, const int32_t* __restrict__ count,
                                                 int ident_slot, const int32_t* __restrict__ slot_of,
                                                 int32_t* __restrict__ best, UniverseState us, const float* __restrict__ d, GridSpec gs,
                                                 int nfit, const double* __restrict__ W64,
                                                 const float* __restrict__ Wdf, double* __restrict__ dchi2,
                                                 double* __restrict__ chi2min) {
    extern __shared__ float4 s_rows[];  // mixed path
    __shared__ double rp[4][kMaxBins], rm[4][kMaxBins], tt[4][kMaxBins];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = blockIdx.x * 4LL + w;
    if (i >= *count || *us.status) return;
    const int u = list[i];
    if (best[u] < 0 || best[u] >= us.G) {  // no row to read
        if (lane == 0) {
            best[u] = -1;
            dchi2[u] = CUDART_NAN;
            if (chi2min) chi2min[u] = CUDART_NAN;
            atomicSub(&us.job_left[us.job_of[u]], 1);
        }
        return;
    }
    const int slot = ident_slot >= 0 ? ident_slot : slot_of[us.cur[u]];
    const int p = us.pt[u];
    const int g = best[u];
    const float* du = d + (size_t)u * nfit;
    double cp = 0.0, cm = 0.0;
    if (Wdf) {
        // mixed path: the double-float residual of every other mixed-path kernel
        float* sm = reinterpret_cast<float*>(s_rows) + w * rows_floats(nfit);
        rows_stage(sm, 0, nfit, srow<MODEL>(gs, nullptr, g), du, lane);
        if (p != g) rows_stage(sm, 1, nfit, srow<MODEL>(gs, nullptr, p), du, lane);
        const double c = rows_chi2(Wdf + (size_t)slot * wdf_floats(nfit), nfit, sm, p == g ? 1 : 2, lane);
        cm = __shfl_sync(0xffffffffu, c, 0);
        cp = (p == g) ? 0.0 : __shfl_sync(0xffffffffu, c, 1);
    } else {
        // plain path: binary64, in the summation order of resid_chi2_warp
        const FitRow rowp = fit_row(gs, p), rowg = fit_row(gs, g);
        for (int j = lane; j < nfit; j += 32) {
            rp[w][j] = __dsub_rn(row_fit(gs, rowp, j), (double)du[j]);
            rm[w][j] = __dsub_rn(row_fit(gs, rowg, j), (double)du[j]);
        }
        __syncwarp();
        const double* W = W64 + (size_t)slot * nfit * nfit;
        cp = (p == g) ? 0.0 : resid_chi2_warp(W, nfit, rp[w], tt[w], lane);
        cm = resid_chi2_warp(W, nfit, rm[w], tt[w], lane);
    }
    if (lane == 0) {
        dchi2[u] = (p == g) ? 0.0 : cp - cm;
        if (chi2min) chi2min[u] = cm;
        atomicSub(&us.job_left[us.job_of[u]], 1);
    }
}

// exact-path bookkeeping: a universe finishes when its minimum repeats its
// covariance index, when it has none, or when it used its last scan; the
// others move on
__global__ void k_advance(const int32_t* __restrict__ active, int64_t n, const int32_t* __restrict__ best,
                          UniverseState us, int32_t* __restrict__ next_active, int32_t* __restrict__ n_next,
                          int32_t* __restrict__ fin, int32_t* __restrict__ n_fin) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n || *us.status) return;
    const int u = active[i];
    const int done = us.nscan[u] + 1;
    us.nscan[u] = (int8_t)done;
    const bool none = best[u] < 0 || best[u] >= us.G;
    if (none || best[u] == us.cur[u] || done >= us.maxit[u]) {
        fin[atomicAdd(n_fin, 1)] = u;
    } else {
        us.cur[u] = best[u];
        next_active[atomicAdd(n_next, 1)] = u;
    }
}

// ---------------------------------------------------------- quantiles -------

// One CTA per row: counts[row] += #{u < n : x[row][u] < thr[row]} (the empirical
// distribution of the row's dchi2 at the data's value).
__global__ void k_count_below(const double* __restrict__ x, int n, const double* __restrict__ thr,
                              int64_t* __restrict__ counts) {
    __shared__ int s_cnt;
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    const double t = thr[blockIdx.x];
    const double* xr = x + (size_t)blockIdx.x * n;
    int c = 0;
    for (int u = threadIdx.x; u < n; u += blockDim.x) c += (xr[u] < t) ? 1 : 0;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&s_cnt, c);
    __syncthreads();
    if (threadIdx.x == 0) counts[blockIdx.x] += s_cnt;
}


// Order of binary64 values as unsigned integers (comparing integers keeps the
// narrow binary64 pipe out of a sort); -0 before +0, NaN by its bits (rows that
// hold any are sorted, where every NaN comes last).
// It takes the bits, loaded as an integer: of a value that was a binary64
// before, the compiler may set the sign by negating it, which a NaN ignores.
__device__ __forceinline__ unsigned long long f64_key(unsigned long long b) {
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double f64_of_key(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7fffffffffffffffull) : ~k));
}

// numpy's "linear" rule between two order statistics
__device__ __forceinline__ void quantile_ranks(int n, double prob, int& lo, int& hi, double& f) {
    const double h = (double)(n - 1) * prob;
    lo = (int)floor(h);
    if (lo < 0) lo = 0;
    if (lo > n - 1) lo = n - 1;
    hi = lo + 1 < n ? lo + 1 : n - 1;
    f = h - lo;
}

// Whole row by a bitonic sort of its keys in shared memory (npow2 of them).
__device__ void quantiles_by_sort(unsigned long long* key, int n, int npow2, const double* __restrict__ probs, int nq,
                                  double* __restrict__ out) {
    for (int i = n + threadIdx.x; i < npow2; i += blockDim.x) key[i] = ~0ull;
    // keys below -infinity's are the NaN with the sign set: last, like the others (thread i wrote key i)
    const unsigned long long first = f64_key(0xfff0000000000000ull);
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        if (key[i] < first) key[i] = ~0ull;
    __syncthreads();
    for (int k = 2; k <= npow2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < npow2; i += blockDim.x) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const bool up = ((i & k) == 0);
                    const unsigned long long a = key[i], b = key[ixj];
                    if ((a > b) == up) {
                        key[i] = b;
                        key[ixj] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int q = threadIdx.x; q < nq; q += blockDim.x) {
        int lo, hi;
        double f;
        quantile_ranks(n, probs[q], lo, hi, f);
        const double a = f64_of_key(key[lo]), b = f64_of_key(key[hi]);
        out[q] = a + f * (b - a);
    }
}

// One CTA per row.  A few quantiles need a few order statistics, not a sorted
// row: the values are counted into BINS buckets by a monotone function
// (their binary32 rounding, linear between the row's extremes), the running
// count finds the buckets that hold each quantile's two ranks, the values of
// those buckets go to a short list, and their ranks in it are counted.  Rows
// that this does not suit (a crowded bucket, infinities, NaN) and calls with
// many quantiles sort the row; so do rows whose lists are long enough that
// counting ranks, a list's square, takes longer than the sort's steps (a call of
// 10000 rows of 100 values, 63 of them in one bucket: lists 82, 96 and 160 us
// for 1, 3 and 8 quantiles, a sort 98; 99 in one: 99, 172 and 375).  Bound by the
// binary64 pipe (72 % active: three conversions of each value to binary32), then
// by shared memory (61 %: three passes over the row and its counting atomics).
// 10000 rows of 1000 values, three quantiles: 1.04 -> 0.12 ms a call (the sort
// compared on the binary64 pipe and its rows were copied first).
constexpr int kQuantSelect = 8;   // quantiles of a call that selects
constexpr int kQuantList = 128;   // values of a quantile's list
constexpr int kQuantMaxRow = 16384;  // values of a row (the entry points refuse longer ones)

template <int BINS>
__global__ void k_quantiles(const double* __restrict__ x, int n, int npow2, const double* __restrict__ probs,
                            int nq, double* __restrict__ out) {
    extern __shared__ unsigned long long s_key[];  // [npow2], then the lists [min(nq, kQuantSelect)][kQuantList]
    __shared__ int s_bin[BINS];
    __shared__ int s_warp[16];
    __shared__ float s_lo[16], s_hi[16];
    __shared__ int s_b0[kQuantSelect], s_b1[kQuantSelect], s_before[kQuantSelect], s_len[kQuantSelect], s_n[kQuantSelect];
    __shared__ double s_v[kQuantSelect][2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const unsigned long long* xr = reinterpret_cast<const unsigned long long*>(x) + (size_t)blockIdx.x * n;
    double* o = out + (size_t)blockIdx.x * nq;
    const bool select = nq <= kQuantSelect;
    float lo = FLT_MAX, hi = -FLT_MAX;
    bool odd = false;  // a value whose binary32 rounding is not an ordinary number
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const unsigned long long v = xr[i];
        s_key[i] = f64_key(v);
        const float f = (float)__longlong_as_double((long long)v);
        odd = odd || !(fabsf(f) < 1.0e38f);
        lo = fminf(lo, f);
        hi = fmaxf(hi, f);
    }
    if (!select || __syncthreads_or(odd)) {
        quantiles_by_sort(s_key, n, npow2, probs, nq, o);
        return;
    }
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, k));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, k));
    }
    if (lane == 0) {
        s_lo[warp] = lo;
        s_hi[warp] = hi;
    }
    for (int b = threadIdx.x; b < BINS; b += blockDim.x) s_bin[b] = 0;
    if (threadIdx.x < kQuantSelect) s_n[threadIdx.x] = 0;
    __syncthreads();
    for (int w = 0; w < nw; ++w) {
        lo = fminf(lo, s_lo[w]);
        hi = fmaxf(hi, s_hi[w]);
    }
    const float scale = hi > lo ? (float)BINS / (hi - lo) : 0.0f;
    // monotone in the value, whatever the roundings
    auto bin = [&](unsigned long long k) {
        const float v = ((float)f64_of_key(k) - lo) * scale;
        return v < (float)(BINS - 1) ? (int)v : BINS - 1;
    };
    for (int i = threadIdx.x; i < n; i += blockDim.x) atomicAdd(&s_bin[bin(s_key[i])], 1);
    __syncthreads();
    // running count up to and including each bucket
    const int per = BINS / blockDim.x;
    int sum = 0;
    for (int k = 0; k < per; ++k) sum += s_bin[threadIdx.x * per + k];
    int run = sum;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, run, k);
        if (lane >= k) run += y;
    }
    if (lane == 31) s_warp[warp] = run;
    __syncthreads();
    run -= sum;
    for (int w = 0; w < warp; ++w) run += s_warp[w];
    for (int k = 0; k < per; ++k) {
        run += s_bin[threadIdx.x * per + k];
        s_bin[threadIdx.x * per + k] = run;
    }
    __syncthreads();
    if (threadIdx.x < nq) {  // the buckets of ranks r0 and r1
        int r0, r1;
        double f;
        quantile_ranks(n, probs[threadIdx.x], r0, r1, f);
        auto find = [&](int r) {  // first bucket whose running count exceeds r
            int a = 0, b = BINS - 1;
            while (a < b) {
                const int m = (a + b) >> 1;
                if (s_bin[m] > r) b = m; else a = m + 1;
            }
            return a;
        };
        const int b0 = find(r0), b1 = find(r1);
        s_b0[threadIdx.x] = b0;
        s_b1[threadIdx.x] = b1;
        s_before[threadIdx.x] = b0 ? s_bin[b0 - 1] : 0;
        s_len[threadIdx.x] = s_bin[b1] - s_before[threadIdx.x];
    }
    __syncthreads();
    int most = 0;  // the longest list
    for (int q = 0; q < nq; ++q) most = max(most, s_len[q]);
    // trips of a warp in all: of the rank loop, and of the sort's steps, each worth three of those
    const int lg = 31 - __clz(npow2), sort_work = 3 * lg * (lg + 1) / 2 * ((npow2 + 31) / 32);
    const int rank_work = nq * most * ((most + 31) / 32);
    if (most > kQuantList || rank_work > sort_work) {  // the same for every thread
        quantiles_by_sort(s_key, n, npow2, probs, nq, o);
        return;
    }
    // the values of those buckets (the buckets between them are empty)
    unsigned long long* list = s_key + npow2;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const unsigned long long k = s_key[i];
        const int b = bin(k);
        for (int q = 0; q < nq; ++q)
            if (b >= s_b0[q] && b <= s_b1[q]) {
                const int at = atomicAdd(&s_n[q], 1);
                if (at < kQuantList) list[q * kQuantList + at] = k;
            }
    }
    __syncthreads();
    for (int q = warp; q < nq; q += nw) {
        int r0, r1;
        double f;
        quantile_ranks(n, probs[q], r0, r1, f);
        r0 -= s_before[q];
        r1 -= s_before[q];
        const int m = s_len[q];
        const unsigned long long* l = list + q * kQuantList;
        for (int e = lane; e < m; e += 32) {
            const unsigned long long k = l[e];
            int rank = 0;  // equal values take their places in list order
            for (int j = 0; j < m; ++j) rank += (l[j] < k || (l[j] == k && j < e)) ? 1 : 0;
            if (rank == r0) s_v[q][0] = f64_of_key(k);
            if (rank == r1) s_v[q][1] = f64_of_key(k);
        }
        __syncwarp();
        if (lane == 0) o[q] = s_v[q][0] + f * (s_v[q][1] - s_v[q][0]);
    }
}

}  // namespace

// ---------------------------------------------------------- peak probes -----

namespace {

// Eight independent fma chains per thread, x <- x a + b with |a| < 1 (values
// stay normal): 16 flops per iteration, no memory traffic.
template <typename T>
__global__ void k_fma_peak(T* out, int iters, T a, T b) {
    T x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = (T)(threadIdx.x + k);
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = fma(x[k], a, b);
    }
    T sum = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) sum += x[k];
    if (sum == (T)-1) out[blockIdx.x] = sum;  // never true; keeps the chains live
}

}  // namespace

// TFLOP/s of one fma probe: best of three timed launches after a warm-up.
template <typename T>
static double fma_peak_tflops(int n_sm, int iters, cudaStream_t st) {
    T* out = nullptr;
    if (cudaMalloc(&out, 4096 * sizeof(T)) != cudaSuccess) return 0.0;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const unsigned blocks = (unsigned)n_sm * 8;
    const int threads = 256;
    double best = 0.0;
    for (int rep = 0; rep < 4; ++rep) {
        cudaEventRecord(e0, st);
        k_fma_peak<T><<<blocks, threads, 0, st>>>(out, iters, (T)0.999999, (T)1e-3);
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        const double flops = 16.0 * iters * (double)blocks * threads;
        if (rep > 0 && ms > 0.0f) best = std::max(best, flops / (ms * 1e-3) / 1e12);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(out);
    return best;
}

bool measure_fma_peaks(int n_sm, double* fp64_tflops, double* fp32_tflops, cudaStream_t st) {
    count_launch(8);
    *fp64_tflops = fma_peak_tflops<double>(n_sm, 20000, st);
    *fp32_tflops = fma_peak_tflops<float>(n_sm, 400000, st);
    return cudaGetLastError() == cudaSuccess && *fp64_tflops > 0.0 && *fp32_tflops > 0.0;
}

// ------------------------------------------------------------- launchers ----

namespace {
// Shared memory of `bytes`, beyond the 48 KB default, which also holds a kernel's static arrays.  The limit
// belongs to the kernel on the current device, which every thread and context shares: it is set to what the
// kernel's largest size takes, the same value at every launch, so that no thread lowers it between another's
// setting and launch.
template <class K>
void allow_smem(K kern, size_t bytes, size_t largest) {
    if (bytes > 24 * 1024)
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)largest);
}
}  // namespace

void launch_collapse(const double* S, int64_t G, int nf, const int32_t* coll, int nfit, double* out,
                     cudaStream_t st) {
    count_launch();
    k_collapse<<<blocks_for(G, 128), 128, 0, st>>>(S, G, nf, coll, nfit, out);
}

void launch_centre(const GridSpec& gs, int64_t G, double* centre, cudaStream_t st) {
    count_launch();
    k_centre<<<gs.nfit, kThreads, 0, st>>>(gs, G, centre);
}

void launch_centred(const GridSpec& gs, int64_t G, int64_t G_pad, int K, double* Sc, float* Sc32, float4* gnorm,
                    uint16_t* Bt, cudaStream_t st) {
    cudaMemsetAsync(Bt, 0, (size_t)G_pad * 2 * K * sizeof(uint16_t), st);
    count_launch();
    k_centred<<<blocks_for(G, 128), 128, 0, st>>>(gs, G, K, Sc, Sc32, gnorm, Bt);
}

void launch_chol_sys(const FullSrc& src, int nf, const double* F, const int64_t* ps, int P, int gauss, double* L64,
                     float* L32, float* s32, int n_sm, int* status, cudaStream_t st) {
    if (P <= 0) return;
    count_launch();
    const int form = chol_form(P, nf, n_sm);
    if (form == kCholColumnsForm) {
        const bool packed = nf <= kCholPackN;
        const size_t smem = packed ? (size_t)tri(nf) * sizeof(double) : 0;
        auto kern = packed ? k_chol_columns<true> : k_chol_columns<false>;
        allow_smem(kern, smem, (size_t)tri(kCholPackN) * sizeof(double));
        kern<<<P, kCholThreads, smem, st>>>(src, nf, F, ps, gauss, L64, L32, s32, status);
        return;
    }
    const int C = form == kCholClusterForm ? kCholCluster : 1;
    const size_t smem = chol_sys_smem(nf, C);
    allow_smem(k_chol_sys, smem, chol_sys_smem(kMaxBins, kCholCluster));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)P * C);
    cfg.blockDim = dim3(kCholThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)C;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_chol_sys, src, nf, F, ps, gauss, L64, L32, s32, status);
}

void launch_build_cov(const FullSrc& src, int nf, int nfit, const int32_t* coll, const double* F, const int32_t* q_list,
                      const int32_t* slot_list, int n, int cov_mode, double* A64, double* W64, float* A32,
                      float* rho, int n_sm, int* status, cudaStream_t st) {
    if (n <= 0) return;
    count_launch();
    const size_t smem = build_cov_smem(nfit);
    allow_smem(k_build_cov, smem, build_cov_smem(kMaxBins));
    const int threads = build_cov_threads(nfit, n, n_sm);
    k_build_cov<<<n, threads, smem, st>>>(src, nf, nfit, coll, F, q_list, slot_list, cov_mode, A64, W64, A32, rho,
                                          status);
}

void launch_qvec64(const GridSpec& gs, int64_t G, int nfit, const double* W64, const int32_t* slots, int n,
                   int64_t ldq, double* Q64, cudaStream_t st) {
    // blockIdx.y is the slot within a launch: chunks of at most gridDim.y's limit
    for (int s0 = 0; s0 < n; s0 += 65535) {
        const int ns = n - s0 < 65535 ? n - s0 : 65535;
        dim3 grid(blocks_for(G, 128) < 64 ? blocks_for(G, 128) : 64, ns);
        count_launch();
        k_qvec64<<<grid, 128, 0, st>>>(gs, G, nfit, W64, slots + s0, ldq, Q64);
    }
}

void launch_qvec32(const GridSpec& gs, const float4* gnorm, int64_t G, int64_t G_pad, int nfit, const float* A32,
                   const float* rho, const int32_t* slots, int n, float* Qc, float* Qb, uint16_t* Qb3,
                   cudaStream_t st) {
    if (n <= 0) return;
    if (n > 65535) {
        // blockIdx.y is the slot within a launch: chunks of at most gridDim.y's limit
        for (int s0 = 0; s0 < n; s0 += 65535)
            launch_qvec32(gs, gnorm, G, G_pad, nfit, A32, rho, slots + s0, n - s0 < 65535 ? n - s0 : 65535, Qc, Qb,
                          Qb3, st);
        return;
    }
    // ~16 grid points per thread so each block's staging of A is amortised
    unsigned gx = blocks_for(G_pad, 128 * 16);
    if (gx > 128) gx = 128;
    dim3 grid(gx, n);
    count_launch();
    if (nfit <= 16)
        k_qvec32<16><<<grid, 128, 0, st>>>(gs, gnorm, G, G_pad, nfit, A32, rho, slots, Qc, Qb, Qb3);
    else if (nfit <= 32)
        k_qvec32<32><<<grid, 128, 0, st>>>(gs, gnorm, G, G_pad, nfit, A32, rho, slots, Qc, Qb, Qb3);
    else if (nfit <= 48)
        k_qvec32<48><<<grid, 128, 0, st>>>(gs, gnorm, G, G_pad, nfit, A32, rho, slots, Qc, Qb, Qb3);
    else if (nfit <= 64)
        k_qvec32<64><<<grid, 128, 0, st>>>(gs, gnorm, G, G_pad, nfit, A32, rho, slots, Qc, Qb, Qb3);
    else
        k_qvec32_generic<<<grid, 128, 0, st>>>(gs, gnorm, G, G_pad, nfit, A32, rho, slots, Qc, Qb, Qb3);
}

void launch_fake_data(const float* L32, const float* s32, int nf, const int32_t* coll, int nfit, const int64_t* ps,
                      int P, int U, uint64_t seed, int gauss, float* d, int n_sm, cudaStream_t st) {
    if (P <= 0 || U <= 0) return;
    // blockIdx.y is the point within a launch; more points than gridDim.y allows take several launches
    constexpr int kMaxGridY = 65535;
    const int64_t ctas = (int64_t)P * ((U + kFakeU - 1) / kFakeU);
    const bool few = fake_few(nf, ctas, n_sm);
    const int threads = few ? std::min(128, (U + 31) / 32 * 32) : fake_threads(nf, ctas, n_sm);
    const int per = few ? threads : kFakeU;
    const size_t smem = few ? 0 : fake_smem(nf);
    auto kern = few ? k_fake_few : threads == 128 ? k_fake_data<128> : k_fake_data<256>;
    allow_smem(kern, smem, fake_smem(kMaxBins));
    for (int p0 = 0; p0 < P; p0 += kMaxGridY) {
        const int np = P - p0 < kMaxGridY ? P - p0 : kMaxGridY;
        const dim3 grid((U + per - 1) / per, np);
        count_launch();
        kern<<<grid, threads, smem, st>>>(L32 + (size_t)p0 * nf * nf, s32 + (size_t)p0 * nf, nf, coll, nfit, ps + p0, U,
                                          (uint32_t)seed, (uint32_t)(seed >> 32), gauss, d + (size_t)p0 * U * nfit);
    }
}

void launch_fill_i32(int32_t* p, int64_t n, int32_t v, cudaStream_t st) {
    if (n <= 0) return;
    unsigned b = blocks_for(n);
    if (b > 4096) b = 4096;
    count_launch();
    k_fill_i32<<<b, kThreads, 0, st>>>(p, n, v);
}

void launch_mark_used(const int32_t* active, int64_t n, const int32_t* cur, uint8_t* flag, cudaStream_t st) {
    if (n <= 0) return;
    count_launch();
    k_mark_used<<<blocks_for(n), kThreads, 0, st>>>(active, n, cur, flag);
}

void launch_compact_flags(uint8_t* flag, int64_t G, int32_t* list, int32_t* count, cudaStream_t st) {
    count_launch();
    k_compact_flags<<<blocks_for(G), kThreads, 0, st>>>(flag, G, list, count);
}

void launch_lookup_slots(const int32_t* active, int64_t n, const int32_t* cur, const int32_t* slot_of,
                         int32_t* uslot, cudaStream_t st) {
    if (n <= 0) return;
    count_launch();
    k_lookup_slots<<<blocks_for(n), kThreads, 0, st>>>(active, n, cur, slot_of, uslot);
}

void launch_set_slots(const int32_t* q, const int32_t* s, int n, int32_t* slot_of, cudaStream_t st) {
    if (n <= 0) return;
    count_launch();
    k_set_slots<<<blocks_for(n), kThreads, 0, st>>>(q, s, n, slot_of);
}

// CTAs per group of universes: up to eight for every SM, each with at least
// one tile of the grid.
int scan64_splits(int64_t n, int64_t G, int n_sm) {
    const int64_t groups = (n + kS64U - 1) / kS64U, tiles = (G + kS64G - 1) / kS64G;
    return (int)std::max<int64_t>(1, std::min<int64_t>(8 * (int64_t)n_sm / groups, tiles));
}

void launch_scan64(const int32_t* list, int64_t n, const int32_t* uslot, const float* d, const GridSpec& gs,
                   int64_t G, int nfit, const double* A64, const double* Q64, int64_t ldq, int32_t* best, int nsp,
                   double* y, double* part_v, int32_t* part_g, cudaStream_t st) {
    if (n <= 0) return;
    const size_t smem = (size_t)nfit * (kS64U + kS64LdS) * sizeof(double);
    allow_smem(k_scan64, smem, (size_t)kMaxBins * (kS64U + kS64LdS) * sizeof(double));
    const bool split = nsp > 1;
    if (split) {
        count_launch();
        k_y64<<<(unsigned)n, 64, 0, st>>>(list, uslot, d, gs.centre, nfit, A64, y);
    }
    count_launch();
    const dim3 grid((unsigned)((n + kS64U - 1) / kS64U), (unsigned)nsp);
    k_scan64<<<grid, kS64Threads, smem, st>>>(list, n, uslot, d, gs, G, nfit, A64, Q64, ldq, best, split ? y : nullptr,
                                              part_v, part_g);
    if (split) {
        count_launch();
        k_scan_resid_reduce<<<blocks_for(n), kThreads, 0, st>>>(list, n, nsp, part_v, part_g, best);
    }
}

void launch_scan_resid(const int32_t* list, int64_t n, const int32_t* uslot, const float* d, const GridSpec& gs,
                       int64_t G, int nfit, const float* Wdf, double* part_v, int32_t* part_g, int nsp,
                       int32_t* best, cudaStream_t st) {
    if (n <= 0) return;
    const size_t smem = rows_smem(nfit);
    count_launch(2);
    const dim3 grid((unsigned)n, (unsigned)nsp);
    auto kern = gs.Sdf ? k_scan_resid<false> : k_scan_resid<true>;
    allow_smem(kern, smem, rows_smem(kMaxBins));
    kern<<<grid, 32 * kRowsWarps, smem, st>>>(list, uslot, d, gs, G, nfit, Wdf, part_v, part_g);
    k_scan_resid_reduce<<<blocks_for(n), kThreads, 0, st>>>(list, n, nsp, part_v, part_g, best);
}

void launch_group(const int32_t* active, int64_t n, const int32_t* uslot, int n_slots, int32_t* cnt,
                  int32_t* tile_base, int32_t* fill, int32_t* n_tiles_dev, int32_t* quad_slot, int32_t* tile_univ,
                  int64_t max_tiles, int slot_rows, cudaStream_t st) {
    cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (size_t)n_slots, st);
    cudaMemsetAsync(fill, 0, sizeof(int32_t) * (size_t)n_slots, st);
    launch_fill_i32(tile_univ, max_tiles * kBM, -1, st);
    if (n > 0) {
        count_launch();
        k_count_slots<<<blocks_for(n), kThreads, 0, st>>>(uslot, n, cnt);
    }
    count_launch();
    k_tile_scan<<<1, 1024, 0, st>>>(cnt, n_slots, slot_rows, tile_base, n_tiles_dev);
    count_launch();
    k_tile_slots<<<blocks_for(n_slots), kThreads, 0, st>>>(cnt, tile_base, n_slots, n_tiles_dev, quad_slot);
    if (n > 0) {
        count_launch();
        k_scatter_tiles<<<blocks_for(n), kThreads, 0, st>>>(active, n, uslot, tile_base, fill, tile_univ);
    }
}

void launch_yprep(const int32_t* quad_slot, const int32_t* tile_univ, int64_t n_tiles, const float* d,
                  const float2* centre, int nfit, int K, const float* A32, const float* rho, const int32_t* cur,
                  const GridSpec& gs, const float4* gnorm, const float* Qc, const float* Qb, int64_t G_pad,
                  uint16_t* Yt, float4* alpha, float* tau0, int32_t* tile_j0, cudaStream_t st) {
    if (n_tiles <= 0) return;
    const size_t smem = yprep_smem(nfit, K);
    allow_smem(k_yprep, smem, yprep_smem(kMaxBins, kMaxScreenK));  // grows with N_fit
    count_launch();
    k_yprep<<<(unsigned)(n_tiles * kQuads), 32 * yprep_warps(K), smem, st>>>(quad_slot, tile_univ, d, centre, nfit, K,
                                                                            A32, rho, cur, gs, gnorm, Qc, Qb, G_pad,
                                                                            Yt, alpha, tau0, tile_j0);
}

void launch_or_mask(const int32_t* list, int64_t n, uint8_t bit, uint8_t* rmask, cudaStream_t st) {
    if (n <= 0 || !rmask) return;
    count_launch();
    k_or_mask<<<blocks_for(n), kThreads, 0, st>>>(list, n, bit, rmask);
}

void launch_min_tau(const int32_t* tile_univ, int64_t n_tiles, const float* thr, float* tau0, cudaStream_t st) {
    if (n_tiles <= 0) return;
    count_launch();
    k_min_tau<<<blocks_for(n_tiles * kBM), kThreads, 0, st>>>(tile_univ, n_tiles * kBM, thr, tau0);
}

// rows[] <- the indices t * BM + r of the tile rows that hold a universe (any order)
__global__ void k_list_rows(const int32_t* __restrict__ tile_univ, int64_t n, int32_t* __restrict__ rows,
                            int32_t* __restrict__ n_rows) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool have = e < n && tile_univ[e] >= 0;
    const unsigned m = __ballot_sync(0xffffffffu, have);
    if (!m) return;
    const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    int first = 0;
    if (lane == leader) first = atomicAdd(n_rows, __popc(m));
    first = __shfl_sync(0xffffffffu, first, leader);
    if (have) rows[first + __popc(m & ((1u << lane) - 1u))] = (int32_t)e;
}

void launch_resolve_list(const ResolveArgs& a, const int32_t* cand_count, int64_t n_tiles, int64_t n_rows,
                         int32_t* rows, int32_t* n_rows_dev, const ListPlan& lp, cudaStream_t st) {
    if (n_tiles <= 0 || n_rows <= 0) return;
    cudaMemsetAsync(n_rows_dev, 0, 4, st);
    cudaMemsetAsync(lp.n_chunk, 0, 4, st);
    count_launch();
    k_list_rows<<<blocks_for(n_tiles * kBM), kThreads, 0, st>>>(a.tile_univ, n_tiles * kBM, rows, n_rows_dev);
    count_launch();
    k_list_plan<<<blocks_for(n_rows), kThreads, 0, st>>>(a, cand_count, rows, n_rows, n_rows_dev, lp);
    // grid-stride over the chunks the plan reserved
    const int64_t want = (lp.max_chunks + kRowsWarps - 1) / kRowsWarps, cap = (int64_t)a.n_sm * 8;
    count_launch();
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min(want, cap));
    const size_t smem = rows_smem(a.nfit);
    auto kern = a.gs.Sdf ? k_list_chunks<false> : k_list_chunks<true>;
    allow_smem(kern, smem, rows_smem(kMaxBins));
    kern<<<grid, 32 * kRowsWarps, smem, st>>>(a, cand_count, rows, lp);
}

void launch_resolve(const ResolveArgs& a, int64_t n_tiles, int64_t n_rows, cudaStream_t st) {
    if (n_tiles <= 0) return;
    cudaMemsetAsync(a.counts, 0, 2 * sizeof(int32_t), st);
    // the tail loops over its device-side count
    const unsigned g3 = (unsigned)std::min<int64_t>(n_tiles, (int64_t)a.n_sm * 8);
    // One thread per residual (k_resid_tiles) is the faster form when its lanes are full: at least a
    // tile per SM and a quarter of the tile rows in use.  Below that a residual spread over a warp
    // ends sooner, and above N_fit = 64 its vector does not fit a thread's registers.
    const bool tiles = a.nfit <= 64 && a.gs.Sdf && n_tiles >= a.n_sm && 4 * n_rows >= n_tiles * kBM;
    auto resid = [&](const int2* items, const int2* tile_items, const int32_t* count, int64_t max_items, double* res) {
        if (!tiles) {
            const int64_t per = kRowsWarps * kRowsB;
            const int64_t want = (max_items + per - 1) / per, cap = (int64_t)a.n_sm * 8;
            const unsigned grid = (unsigned)std::max<int64_t>(1, std::min(want, cap));
            const size_t smem = rows_smem(a.nfit);
            auto kern = a.gs.Sdf ? k_resid_rows<false> : k_resid_rows<true>;
            allow_smem(kern, smem, rows_smem(kMaxBins));
            kern<<<grid, 32 * kRowsWarps, smem, st>>>(a, items, count, res);
            return;
        }
        const size_t smem = (size_t)df_blocks(a.nfit) * a.nfit * 8 * sizeof(float);
        auto run = [&](auto kern) { kern<<<(unsigned)n_tiles, kResidThreads, smem, st>>>(a, items, tile_items, res); };
        if (a.nfit <= 16)
            run(k_resid_tiles<16>);
        else if (a.nfit <= 32)
            run(k_resid_tiles<32>);
        else if (a.nfit <= 48)
            run(k_resid_tiles<48>);
        else
            run(k_resid_tiles<64>);
    };
    count_launch(5);
    k_resolve_emit<<<(unsigned)n_tiles, kBM, 0, st>>>(a);
    resid(a.items, a.tile_items, a.counts, n_rows * (a.topk + 1), a.res);
    k_resolve_conclude<<<(unsigned)n_tiles, kBM, 0, st>>>(a);
    resid(a.items2, a.tile_items2, a.counts + 1, n_rows, a.res2);
    k_resolve_tail<<<g3, 256, 0, st>>>(a);
}

void launch_finish(const int32_t* list, int64_t n, const int32_t* count, int ident_slot, const int32_t* slot_of,
                   int32_t* best, const UniverseState& us, const float* d, const GridSpec& gs, int nfit, const double* W64, const float* Wdf, double* dchi2,
                   double* chi2min, cudaStream_t st) {
    if (n <= 0) return;
    count_launch();
    const unsigned grid = (unsigned)((n + 3) / 4);
    static_assert(kRowsWarps == 4, "a warp of k_finish has one warp's row storage");
    const size_t smem = Wdf ? rows_smem(nfit) : 0;
    auto kern = gs.Sdf || !Wdf ? k_finish<false> : k_finish<true>;
    allow_smem(kern, smem, rows_smem(kMaxBins));
    kern<<<grid, 128, smem, st>>>(list, count, ident_slot, slot_of, best, us, d, gs, nfit, W64, Wdf, dchi2, chi2min);
}

size_t wdf_bytes(int nfit) { return (size_t)df_blocks(nfit) * nfit * 8 * sizeof(float); }

void launch_wdf(const double* W64, const int32_t* slots, int n, int nfit, float* Wdf, cudaStream_t st) {
    if (n <= 0) return;
    count_launch();
    k_wdf<<<n, 256, 0, st>>>(W64, slots, nfit, Wdf);
}

void launch_to_df(const double* x, int64_t n, float2* y, cudaStream_t st) {
    if (n <= 0) return;
    count_launch();
    k_to_df<<<blocks_for(n), kThreads, 0, st>>>(x, n, y);
}

void launch_advance(const int32_t* active, int64_t n, const int32_t* best, const UniverseState& us,
                    int32_t* next_active, int32_t* n_next, int32_t* fin, int32_t* n_fin, cudaStream_t st) {
    if (n <= 0) return;
    count_launch();
    k_advance<<<blocks_for(n), kThreads, 0, st>>>(active, n, best, us, next_active, n_next, fin, n_fin);
}

void launch_count_below(const double* x, int rows, int n, const double* thr, int64_t* counts, cudaStream_t st) {
    if (rows <= 0 || n <= 0) return;
    count_launch();
    k_count_below<<<rows, 256, 0, st>>>(x, n, thr, counts);
}

void launch_osc_sin(const SpecModel& m, int rows, const double* L, const double* E, double* sinT, cudaStream_t st) {
    const int64_t n = (int64_t)rows * m.nf;
    if (n <= 0) return;
    count_launch();
    k_osc_sin<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(m, rows, L, E, sinT);
}

void launch_osc_spectra(const SpecModel& m, int64_t G, double* S, int* bad, cudaStream_t st) {
    const int64_t n = G * m.nf;
    if (n <= 0) return;
    count_launch();
    k_osc_spectra<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(m, G, S, bad);
}

void launch_quantiles(const double* x, int rows, int n, const double* probs, int nq, double* out, int n_sm,
                      cudaStream_t st) {
    int p2 = 1;
    while (p2 < n) p2 <<= 1;
    const auto smem_of = [](size_t keys, int lists) {
        return (keys + (size_t)lists * kQuantList) * sizeof(unsigned long long);
    };
    const size_t smem = smem_of(p2, nq <= kQuantSelect ? nq : 0);
    count_launch();
    // short rows: small CTAs, many rows in flight; long rows (and a sort of many quantiles) a wide CTA,
    // with as many buckets as keep a bucket of a smooth distribution below the list's length.  A row an SM
    // at most gets the wide one too: 10 rows of 1000 values that have to be sorted 61 us a call with 128
    // threads, 46 with 512 (rows that select 34 either way)
    const bool small = n <= 2048 && nq <= kQuantSelect && rows > n_sm;
    auto kern = small ? k_quantiles<1024> : k_quantiles<4096>;
    allow_smem(kern, smem, smem_of(small ? 2048 : kQuantMaxRow, kQuantSelect));
    kern<<<rows, small ? 128 : 512, smem, st>>>(x, n, p2, probs, nq, out);
}

}  // namespace fcdev
