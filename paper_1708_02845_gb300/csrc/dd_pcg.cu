// Poisson-kernel preprocessing, Section IV Eq. (32)-(33), in FP64 on the GPU.
//
// Solves (-L_II) X = L_IB for all k boundary columns at once: one
// preconditioned conjugate-gradient recurrence per column, run in lock-step
// over a block of columns so that every sparse product streams the whole
// row-major [m][kc] block.  The preconditioner is a smoothed-aggregation
// multigrid V-cycle (dd_amg.cpp builds the hierarchy on the host); the
// diagonal (Jacobi) preconditioner remains for tiny meshes and as the
// fallback when no hierarchy can be built.  -L_II is a symmetric positive-definite
// M-matrix, so CG converges; its iterates are kept in FP64 because the
// small entries of P (shadowed boundary parts) need many correct digits for
// the logarithms of Eq. (35).  The block stops when every column's residual
// satisfies ||r|| <= rtol ||b||; only columns with b = 0 (no interior
// support) are skipped.  Columns are processed in chunks that fit a
// workspace budget; the result is written as FP32 P (row pitch k_pad).
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <cstdlib>
#include <utility>
#include <vector>

#include "dd_amg.h"
#include "dd_f32x2.cuh"
#include "dd_internal.h"
#include "dd_pairs.h"

namespace {

constexpr int kColsPerBlock = 128;   // columns (threads) of one CTA

struct Work {
    int64_t m = 0, kc = 0, nrb = 0;
    double *X = nullptr, *R = nullptr, *Pd = nullptr, *AP = nullptr;
    double *part0 = nullptr, *part1 = nullptr;   // [nrb][kc] partial column sums
    double *alpha = nullptr, *beta = nullptr, *rz = nullptr, *bnorm = nullptr, *dinv = nullptr;
    int *done = nullptr;
    unsigned long long *maxres = nullptr;        // bits of a non-negative double
};

// AP = A Pd over one row block; partial column sums of Pd . AP
__global__ void spmm_dot_kernel(int64_t m, int64_t kc, const int64_t *__restrict__ a_off,
                                const int32_t *__restrict__ a_col, const double *__restrict__ a_val,
                                const double *__restrict__ Pd, double *__restrict__ AP,
                                double *__restrict__ part, int rpb) {
    const int64_t c = (int64_t)blockIdx.y * kColsPerBlock + threadIdx.x;
    if (c >= kc) return;
    const int64_t r0 = (int64_t)blockIdx.x * rpb;
    const int64_t r1 = r0 + rpb < m ? r0 + rpb : m;
    double acc = 0.0;
    for (int64_t r = r0; r < r1; ++r) {
        double s = 0.0;
        for (int64_t q = a_off[r]; q < a_off[r + 1]; ++q) s += a_val[q] * Pd[(int64_t)a_col[q] * kc + c];
        AP[r * kc + c] = s;
        acc += Pd[r * kc + c] * s;
    }
    part[(int64_t)blockIdx.x * kc + c] = acc;
}

// X += alpha Pd, R -= alpha AP; partial sums of R.Z (Z = D^-1 R) and R.R
__global__ void update_xr_kernel(int64_t m, int64_t kc, const double *__restrict__ alpha,
                                 const double *__restrict__ dinv, double *__restrict__ X,
                                 double *__restrict__ R, const double *__restrict__ Pd,
                                 const double *__restrict__ AP, double *__restrict__ part_rz,
                                 double *__restrict__ part_rr, int rpb) {
    const int64_t c = (int64_t)blockIdx.y * kColsPerBlock + threadIdx.x;
    if (c >= kc) return;
    const int64_t r0 = (int64_t)blockIdx.x * rpb;
    const int64_t r1 = r0 + rpb < m ? r0 + rpb : m;
    const double a = alpha[c];
    double srz = 0.0, srr = 0.0;
    for (int64_t r = r0; r < r1; ++r) {
        const int64_t i = r * kc + c;
        double rr = R[i];
        if (a != 0.0) {
            X[i] += a * Pd[i];
            rr -= a * AP[i];
            R[i] = rr;
        }
        srz += rr * rr * dinv[r];
        srr += rr * rr;
    }
    part_rz[(int64_t)blockIdx.x * kc + c] = srz;
    part_rr[(int64_t)blockIdx.x * kc + c] = srr;
}

// Pd = D^-1 R + beta Pd
__global__ void update_p_kernel(int64_t m, int64_t kc, const double *__restrict__ beta,
                                const double *__restrict__ dinv, const double *__restrict__ R,
                                double *__restrict__ Pd, int rpb) {
    const int64_t c = (int64_t)blockIdx.y * kColsPerBlock + threadIdx.x;
    if (c >= kc) return;
    const int64_t r0 = (int64_t)blockIdx.x * rpb;
    const int64_t r1 = r0 + rpb < m ? r0 + rpb : m;
    const double b = beta[c];
    for (int64_t r = r0; r < r1; ++r) {
        const int64_t i = r * kc + c;
        Pd[i] = R[i] * dinv[r] + b * Pd[i];
    }
}

// Sum the [nrb][kc] partials of each column: blockDim (32, 32) (with 8 rows of
// threads the two sums of beta took 28 us an iteration on grid140, a chain of
// loads on 33 blocks)
constexpr int kSumRows = 32;
__device__ __forceinline__ double column_sum(const double *part, int64_t nrb, int64_t kc, int64_t c,
                                             double (*sh)[33]) {
    double s = 0.0;
    if (c < kc)
        for (int64_t b = threadIdx.y; b < nrb; b += blockDim.y) s += part[b * kc + c];
    sh[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0) {
        for (int y = 1; y < (int)blockDim.y; ++y) s += sh[y][threadIdx.x];
    }
    __syncthreads();
    return s;   // valid in threadIdx.y == 0
}

__global__ void alpha_kernel(int64_t nrb, int64_t kc, const double *__restrict__ part,
                             const double *__restrict__ rz, const int *__restrict__ done,
                             double *__restrict__ alpha) {
    __shared__ double sh[kSumRows][33];
    const int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.x;
    double pAp = column_sum(part, nrb, kc, c, sh);
    if (threadIdx.y == 0 && c < kc) alpha[c] = (!done[c] && pAp > 0.0) ? rz[c] / pAp : 0.0;
}

// (nrz, nrb: how many partials part_rz and part_rr hold a column; shift: null, or
// the columns' exponents for the next residual)
__global__ void beta_kernel(int64_t nrz, int64_t nrb, int64_t kc, const double *__restrict__ part_rz,
                            const double *__restrict__ part_rr, const double *__restrict__ bnorm,
                            double *__restrict__ rz, const int *__restrict__ done,
                            double *__restrict__ beta, unsigned long long *__restrict__ maxres,
                            int *__restrict__ shift) {
    __shared__ double sh[kSumRows][33];
    const int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.x;
    double rz_new = column_sum(part_rz, nrz, kc, c, sh);
    double rr = column_sum(part_rr, nrb, kc, c, sh);
    if (threadIdx.y == 0 && c < kc) {
        double res = bnorm[c] > 0.0 ? sqrt(rr) / bnorm[c] : 0.0;
        // columns are not frozen at rtol: every column keeps iterating until the
        // slowest one converges, which drives the small entries of P (shadowed
        // boundary parts, whose logarithms enter Eq. 35) far below rtol
        const int d = done[c];
        beta[c] = (!d && rz[c] > 0.0) ? rz_new / rz[c] : 0.0;
        rz[c] = rz_new;
        if (shift) shift[c] = shift_of_square(rr);
        atomicMax(maxres, (unsigned long long)__double_as_longlong(res));
    }
}

// R = L_IB[:, c0:c0+kc] (scatter of the edge weights to boundary columns); top:
// null, or the largest biased exponent of each column's entries (0 before)
__global__ void scatter_rhs_kernel(int64_t n_rb, const int32_t *__restrict__ rb_row,
                                   const int32_t *__restrict__ rb_col, const double *__restrict__ rb_val,
                                   int64_t c0, int64_t ncols, int64_t ld, double *__restrict__ R,
                                   int *__restrict__ top) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_rb) return;
    int64_t c = (int64_t)rb_col[i] - c0;
    if (c < 0 || c >= ncols) return;
    R[(int64_t)rb_row[i] * ld + c] += rb_val[i];   // one edge per (row, column): no race
    if (top) atomicMax(top + c, (int)((unsigned long long)__double_as_longlong(rb_val[i]) >> 52) & 0x7ff);
}

// the right-hand side's exponents (beta_kernel) from the largest biased one, in place
__global__ void first_shift_kernel(int64_t kc, int *__restrict__ shift) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < kc) shift[c] = shift_of_top(shift[c]);
}

__global__ void dinv_kernel(int64_t m, const double *__restrict__ diag, double *__restrict__ dinv) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) dinv[i] = 1.0 / diag[i];
}

// initial Pd = Z = D^-1 R and per-column partials of R.Z and R.R
__global__ void init_p_kernel(int64_t m, int64_t kc, const double *__restrict__ dinv,
                              const double *__restrict__ R, double *__restrict__ Pd,
                              double *__restrict__ part_rz, double *__restrict__ part_rr, int rpb) {
    const int64_t c = (int64_t)blockIdx.y * kColsPerBlock + threadIdx.x;
    if (c >= kc) return;
    const int64_t r0 = (int64_t)blockIdx.x * rpb;
    const int64_t r1 = r0 + rpb < m ? r0 + rpb : m;
    double srz = 0.0, srr = 0.0;
    for (int64_t r = r0; r < r1; ++r) {
        const int64_t i = r * kc + c;
        double rr = R[i], z = rr * dinv[r];
        Pd[i] = z;
        srz += rr * z;
        srr += rr * rr;
    }
    part_rz[(int64_t)blockIdx.x * kc + c] = srz;
    part_rr[(int64_t)blockIdx.x * kc + c] = srr;
}

__global__ void init_scalars_kernel(int64_t nrb, int64_t kc, const double *__restrict__ part_rz,
                                    const double *__restrict__ part_rr, double *__restrict__ rz,
                                    double *__restrict__ bnorm, int *__restrict__ done) {
    __shared__ double sh[kSumRows][33];
    const int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.x;
    double s_rz = column_sum(part_rz, nrb, kc, c, sh);
    double s_rr = column_sum(part_rr, nrb, kc, c, sh);
    if (threadIdx.y == 0 && c < kc) {
        rz[c] = s_rz;
        bnorm[c] = sqrt(s_rr);
        done[c] = s_rr > 0.0 ? 0 : 1;   // a column with no interior support is exactly zero
    }
}

// P[I[r], c0 + c] = X[r, c] as FP32, negatives clamped to 0 and values below FLT_MIN flushed
__global__ void pack_chunk_kernel(int64_t m, int64_t ncols, int64_t ld, int64_t c0, int64_t k_pad,
                                  const int32_t *__restrict__ interior, const double *__restrict__ X,
                                  float *__restrict__ P, int rpb) {
    const int64_t c = (int64_t)blockIdx.y * kColsPerBlock + threadIdx.x;
    if (c >= ncols) return;
    const int64_t r0 = (int64_t)blockIdx.x * rpb;
    const int64_t r1 = r0 + rpb < m ? r0 + rpb : m;
    for (int64_t r = r0; r < r1; ++r) {
        double v = X[r * ld + c];
        float f = v < (double)FLT_MIN ? 0.0f : (float)v;
        P[(int64_t)interior[r] * k_pad + c0 + c] = f;
    }
}

__global__ void boundary_identity_kernel(int64_t k, int64_t k_pad, const int32_t *__restrict__ boundary,
                                         float *__restrict__ P) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < k) P[(int64_t)boundary[j] * k_pad + j] = 1.0f;
}

__global__ void store_host_p_kernel(int64_t n_v, int64_t k, int64_t k_pad, const double *__restrict__ src,
                                    float *__restrict__ P) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_v * k) return;
    int64_t v = i / k, c = i % k;
    double x = src[i];
    P[v * k_pad + c] = x < (double)FLT_MIN ? 0.0f : (float)x;
}

// ---------------------------------------------------------------- multigrid V-cycle kernels
// The V-cycle's two sparse products a level (dd_amg.h: AmgLevel).  This part
// does about one FP64 multiply-add for every 60 in FP32, and in FP64 the
// cycle's 17 to 21 multiply-adds per fine entry took two thirds of the solve.
// It is the preconditioner, a fixed symmetric operator that only steers the
// iteration, so its numbers are unevaluated sums of two floats (about 48
// bits) and its sums compensated in the same form (Dekker, "A floating-point
// technique for extending the available precision", Numerische Mathematik
// 1971); the iteration itself -- residual, products, steps, stopping test --
// stays in FP64.  One term costs 12 FP32 operations, packed over the two
// columns of a thread.
//
// A block [rows][kc] of such numbers keeps the columns of a pair side by
// side: (hi0, hi1, lo0, lo1) in 16 bytes (kc is even).
struct Df2 {
    f2_t hi, lo;
};

__device__ __forceinline__ Df2 df_load(const float4 *p) {
    const float4 v = *p;
    return Df2{pk(v.x, v.y), pk(v.z, v.w)};
}
__device__ __forceinline__ f2_t sub2(f2_t a, f2_t b) { return fma2(b, pk(-1.0f, -1.0f), a); }

// (s, c) += a x: the product's leading part with its rounding error, added by a two-sum
__device__ __forceinline__ void df_fma(f2_t &s, f2_t &c, float2 a, const Df2 &x) {
    const f2_t ah = pk(a.x, a.x), al = pk(a.y, a.y);
    const f2_t p = mul2(ah, x.hi);
    f2_t e = fma2(ah, x.hi, p ^ 0x8000000080000000ULL);
    e = fma2(ah, x.lo, e);
    e = fma2(al, x.hi, e);
    const f2_t t = add2(s, p), b = sub2(t, s);
    const f2_t err = add2(sub2(s, sub2(t, b)), sub2(p, b));
    s = t;
    c = add2(c, add2(err, e));
}
// the sum as a normalised pair
__device__ __forceinline__ Df2 df_norm(f2_t s, f2_t c) {
    const f2_t h = add2(s, c);
    return Df2{h, sub2(c, sub2(h, s))};
}
__device__ __forceinline__ float4 df_pack(const Df2 &v) {
    float4 r;
    upk(v.hi, r.x, r.y);
    upk(v.lo, r.z, r.w);
    return r;
}

constexpr int kPairs = 64;      // column pairs (threads) of one CTA

// The sparse products' CTAs: 16 pairs of columns (256 bytes of a row) x 32
// rows at a time, down a band of consecutive rows.  A row of X is read by
// every row of its stencil, grid lines apart; a CTA that holds 64 pairs and
// eight rows reads most of them from L2 again (Q^T of grid140's finest level
// 180 us, L2's bandwidth), a narrow band keeps the last few lines in L1
// (the four Q^T of grid140 together 238 -> 117 us a cycle).
constexpr int kBandPairs = 16, kBandRows = 32;

// Y = M X
__global__ void __launch_bounds__(kBandPairs *kBandRows, 2)
    df_spmm_kernel(int64_t rows, int64_t kp, const int32_t *__restrict__ off, const int32_t *__restrict__ col,
                   const float2 *__restrict__ val, const float4 *__restrict__ X, float4 *__restrict__ Y, int band) {
    const int64_t c = (int64_t)blockIdx.y * kBandPairs + threadIdx.x;
    if (c >= kp) return;
    const int64_t r0 = (int64_t)blockIdx.x * band;
    const int64_t r1 = r0 + band < rows ? r0 + band : rows;
    for (int64_t r = r0 + threadIdx.y; r < r1; r += kBandRows) {
        f2_t s = 0ULL, cc = 0ULL;
#pragma unroll 4
        for (int q = off[r]; q < off[r + 1]; ++q) df_fma(s, cc, val[q], df_load(X + (int64_t)col[q] * kp + c));
        Y[r * kp + c] = df_pack(df_norm(s, cc));
    }
}

// Z = G B + Q E (E: rows of the next level).  FINE: Z in FP64 without the
// columns' exponents, with partial column sums of R . Z; else Z in pairs like B.
template <bool FINE>
__global__ void __launch_bounds__(kBandPairs *kBandRows, 2)
    df_up_kernel(int64_t rows, int64_t kp, const int32_t *__restrict__ goff, const int32_t *__restrict__ gcol,
                 const float2 *__restrict__ gval, const int32_t *__restrict__ qoff, const int32_t *__restrict__ qcol,
                 const float2 *__restrict__ qval, const float4 *__restrict__ B, const float4 *__restrict__ E,
                 const double2 *__restrict__ R, const int2 *__restrict__ shift, void *__restrict__ Z,
                 double2 *__restrict__ part, int band) {
    __shared__ double2 sum[FINE ? kBandRows : 1][kBandPairs];
    const int64_t c = (int64_t)blockIdx.y * kBandPairs + threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * band;
    const int64_t r1 = r0 + band < rows ? r0 + band : rows;
    double d0 = 0.0, d1 = 0.0;
    if (c < kp) {
        const int2 sh = FINE ? shift[c] : make_int2(0, 0);
        for (int64_t r = r0 + threadIdx.y; r < r1; r += kBandRows) {
            f2_t s = 0ULL, cc = 0ULL;
#pragma unroll 4
            for (int q = goff[r]; q < goff[r + 1]; ++q)
                df_fma(s, cc, gval[q], df_load(B + (int64_t)gcol[q] * kp + c));
#pragma unroll 4
            for (int q = qoff[r]; q < qoff[r + 1]; ++q)
                df_fma(s, cc, qval[q], df_load(E + (int64_t)qcol[q] * kp + c));
            const float4 z = df_pack(df_norm(s, cc));
            if (FINE) {
                const double2 v = R[r * kp + c];
                const double z0 = widen(z.x, sh.x) + widen(z.z, sh.x), z1 = widen(z.y, sh.y) + widen(z.w, sh.y);
                static_cast<double2 *>(Z)[r * kp + c] = make_double2(z0, z1);
                d0 += v.x * z0;
                d1 += v.y * z1;
            } else {
                static_cast<float4 *>(Z)[r * kp + c] = z;
            }
        }
    }
    if (FINE) {
        sum[threadIdx.y][threadIdx.x] = make_double2(d0, d1);
        __syncthreads();
        if (threadIdx.y == 0 && c < kp) {
            for (int y = 1; y < kBandRows; ++y) {
                d0 += sum[y][threadIdx.x].x;
                d1 += sum[y][threadIdx.x].y;
            }
            part[(int64_t)blockIdx.x * kp + c] = make_double2(d0, d1);
        }
    }
}

// X = Ainv B on the coarsest level (Ainv dense n x n, row-major)
__global__ void __launch_bounds__(kPairs) df_coarse_kernel(int64_t n, int64_t kp, const float2 *__restrict__ ainv,
                                                           const float4 *__restrict__ B, float4 *__restrict__ X) {
    const int64_t c = (int64_t)blockIdx.x * kPairs + threadIdx.x;
    const int64_t i = blockIdx.y;
    if (c >= kp || i >= n) return;
    f2_t s = 0ULL, cc = 0ULL;
#pragma unroll 4
    for (int64_t j = 0; j < n; ++j) df_fma(s, cc, ainv[i * n + j], df_load(B + j * kp + c));
    X[i * kp + c] = df_pack(df_norm(s, cc));
}

// a block as pairs (the first V-cycle's right-hand side), with partial column sums of R . R
__global__ void __launch_bounds__(kPairs) df_first_kernel(int64_t rows, int64_t kp, const double2 *__restrict__ R,
                                                          const int2 *__restrict__ shift, float4 *__restrict__ B, double2 *__restrict__ part,
                                                          int rpb) {
    const int64_t c = (int64_t)blockIdx.y * kPairs + threadIdx.x;
    if (c >= kp) return;
    const int64_t r0 = (int64_t)blockIdx.x * rpb;
    const int64_t r1 = r0 + rpb < rows ? r0 + rpb : rows;
    const int2 sh = shift[c];
    double d0 = 0.0, d1 = 0.0;
    for (int64_t r = r0; r < r1; ++r) {
        const double2 v = R[r * kp + c];
        float4 b;
        df_split(v.x, sh.x, b.x, b.z);
        df_split(v.y, sh.y, b.y, b.w);
        B[r * kp + c] = b;
        d0 += v.x * v.x;
        d1 += v.y * v.y;
    }
    part[(int64_t)blockIdx.x * kp + c] = make_double2(d0, d1);
}

// R -= alpha AP, also as pairs into B; partial column sums of R . R (a column
// with alpha = 0 keeps its residual)
__global__ void __launch_bounds__(kPairs) update_r_kernel(int64_t rows, int64_t kp,
                                                          const double2 *__restrict__ alpha,
                                                          double2 *__restrict__ R, const double2 *__restrict__ AP,
                                                          const int2 *__restrict__ shift, float4 *__restrict__ B, double2 *__restrict__ part,
                                                          int rpb) {
    const int64_t c = (int64_t)blockIdx.y * kPairs + threadIdx.x;
    if (c >= kp) return;
    const int64_t r0 = (int64_t)blockIdx.x * rpb;
    const int64_t r1 = r0 + rpb < rows ? r0 + rpb : rows;
    const double2 a = alpha[c];
    const int2 sh = shift[c];
    double d0 = 0.0, d1 = 0.0;
#pragma unroll 2
    for (int64_t r = r0; r < r1; ++r) {
        const int64_t i = r * kp + c;
        double2 v = R[i];
        const double2 w = AP[i];
        v.x -= a.x * w.x;
        v.y -= a.y * w.y;
        R[i] = v;
        float4 b;
        df_split(v.x, sh.x, b.x, b.z);
        df_split(v.y, sh.y, b.y, b.w);
        B[i] = b;
        d0 += v.x * v.x;
        d1 += v.y * v.y;
    }
    part[(int64_t)blockIdx.x * kp + c] = make_double2(d0, d1);
}

// X += alpha Pd, then Pd = Z + beta Pd: one read of Pd for both
__global__ void __launch_bounds__(kPairs) update_xp_kernel(int64_t rows, int64_t kp,
                                                           const double2 *__restrict__ alpha,
                                                           const double2 *__restrict__ beta,
                                                           const double2 *__restrict__ Z, double2 *__restrict__ X,
                                                           double2 *__restrict__ Pd, int rpb) {
    const int64_t c = (int64_t)blockIdx.y * kPairs + threadIdx.x;
    if (c >= kp) return;
    const int64_t r0 = (int64_t)blockIdx.x * rpb;
    const int64_t r1 = r0 + rpb < rows ? r0 + rpb : rows;
    const double2 a = alpha[c], b = beta[c];
#pragma unroll 2
    for (int64_t r = r0; r < r1; ++r) {
        const int64_t i = r * kp + c;
        double2 x = X[i], p = Pd[i];
        const double2 z = Z[i];
        x.x += a.x * p.x;
        x.y += a.y * p.y;
        p.x = z.x + b.x * p.x;
        p.y = z.y + b.y * p.y;
        X[i] = x;
        Pd[i] = p;
    }
}

// X = Ainv B in FP64, where the whole problem is the coarsest level
__global__ void coarse_solve_kernel(int64_t n, int64_t kc, const double *__restrict__ ainv,
                                    const double *__restrict__ B, double *__restrict__ X) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = blockIdx.y;
    if (c >= kc || i >= n) return;
    double s = 0.0;
    for (int64_t j = 0; j < n; ++j) s += ainv[i * n + j] * B[j * kc + c];
    X[i * kc + c] = s;
}

// rz = column sums of part_rz, bnorm from part_rr, done flags (first iteration)
__global__ void amg_init_scalars_kernel(int64_t nrz, int64_t nrb, int64_t kc, const double *__restrict__ part_rz,
                                        const double *__restrict__ part_rr, double *__restrict__ rz,
                                        double *__restrict__ bnorm, int *__restrict__ done) {
    __shared__ double sh[kSumRows][33];
    const int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.x;
    double s_rz = column_sum(part_rz, nrz, kc, c, sh);
    double s_rr = column_sum(part_rr, nrb, kc, c, sh);
    if (threadIdx.y == 0 && c < kc) {
        rz[c] = s_rz;
        bnorm[c] = sqrt(s_rr);
        done[c] = s_rr > 0.0 ? 0 : 1;   // a column with no interior support is exactly zero
    }
}

// One step of the power iteration for the largest eigenvalue of D^-1 A
// (dd_amg.cpp: spectral_radius, from the same start), the fine level's: y =
// D^-1 A x / |x|, with y's squared norm as one partial a CTA.  On
// the host its 24 steps took a third of the hierarchy's setup (3 ms on
// grid140).  part_x null: x is the start vector, formed here.
constexpr int kPowerCtas = 128, kPowerSteps = 24;
__device__ __forceinline__ double power_start(int64_t i) { return 1.0 + 0.5 * sin(0.7 * (double)i); }
__global__ void __launch_bounds__(256) power_kernel(int64_t m, const int64_t *__restrict__ off,
                                                    const int32_t *__restrict__ col, const double *__restrict__ val,
                                                    const double *__restrict__ diag, const double *__restrict__ x,
                                                    const double *__restrict__ part_x, double *__restrict__ y,
                                                    double *__restrict__ part_y) {
    __shared__ double sh[8];
    const int tid = threadIdx.x, lane = tid & 31;
    auto block_sum = [&](double v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        __syncthreads();
        if (lane == 0) sh[tid >> 5] = v;
        __syncthreads();
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += sh[w];
        return t;
    };
    double scale = 1.0;
    if (part_x) scale = rsqrt(block_sum(tid < kPowerCtas ? part_x[tid] : 0.0));
    double ny = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * 256 + tid; i < m; i += (int64_t)gridDim.x * 256) {
        double s = 0.0;
        for (int64_t p = off[i]; p < off[i + 1]; ++p) s += val[p] * (part_x ? x[col[p]] : power_start(col[p]));
        const double v = s * scale / diag[i];
        y[i] = v;
        ny += v * v;
    }
    ny = block_sum(ny);
    if (tid == 0) part_y[blockIdx.x] = ny;
}

// rho(D^-1 A) of the mesh's operator, or 0 where that fails (the host then forms it)
double device_spectral_radius(const DevMesh &M, cudaStream_t s) {
    double *w = nullptr;
    const size_t n = (size_t)M.m;
    if (cudaMalloc((void **)&w, (2 * n + 2 * kPowerCtas) * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        return 0.0;
    }
    double *part = w + 2 * n, h[kPowerCtas];
    for (int it = 0; it < kPowerSteps; ++it)
        power_kernel<<<kPowerCtas, 256, 0, s>>>(M.m, M.a_off, M.a_col, M.a_val, M.a_diag, w + (it & 1 ? 0 : n),
                                                it ? part + (it & 1 ? 0 : kPowerCtas) : nullptr, w + (it & 1 ? n : 0),
                                                part + (it & 1 ? kPowerCtas : 0));
    // the last step's x has norm 1, so |y| is the estimate
    const bool ok = cudaMemcpyAsync(h, part + ((kPowerSteps - 1) & 1 ? kPowerCtas : 0), sizeof h,
                                    cudaMemcpyDeviceToHost, s) == cudaSuccess &&
                    cudaStreamSynchronize(s) == cudaSuccess;
    cudaFree(w);
    if (!ok) {
        cudaGetLastError();
        return 0.0;
    }
    double t = 0.0;
    for (double v : h) t += v;
    return t > 0.0 && std::isfinite(t) ? std::sqrt(t) : 0.0;
}

template <typename T>
cudaError_t alloc(T **p, size_t count) {
    return cudaMalloc((void **)p, count * sizeof(T));
}

// rows per CTA for a [rows][kc] block: enough CTAs (about 16 per SM), at most 256 rows
int sm_count() {
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}
int rows_per_block(int64_t rows, int64_t kc) {
    const int sms = sm_count();
    const int64_t colblocks = (kc + kColsPerBlock - 1) / kColsPerBlock;
    const int64_t want = rows * colblocks / (16LL * sms);
    int rpb = 256;
    while (rpb > 4 && rpb > want) rpb >>= 1;
    return rpb;
}

struct DevCsr {
    int32_t *off = nullptr, *col = nullptr;
    float2 *val = nullptr;         // (hi, lo)
};

float2 split_pair(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}

// Block CG with the smoothed-aggregation V-cycle as preconditioner (one
// Jacobi pre- and post-sweep per level, exact coarsest solve): symmetric and
// positive definite, so CG applies.  Returns DD_ENOTCONV with *fallback set
// when the hierarchy cannot be built (the caller then uses Jacobi).
dd_status run_pcg_amg(DevMesh &M, double rtol, int32_t max_iter, cudaStream_t s, int32_t *iters_out,
                      double *resid_out, std::string &err, bool *fallback) {
    *fallback = false;
    const int64_t m = M.m, k = M.k;
    // host copy of A = -L_II and the hierarchy
    AmgCsr A0;
    A0.rows = A0.cols = m;
    A0.off.resize(m + 1);
    DD_CUDA_TRY(cudaMemcpy(A0.off.data(), M.a_off, (m + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost), err);
    const int64_t nnz = A0.off[m];
    A0.col.resize(nnz);
    A0.val.resize(nnz);
    DD_CUDA_TRY(cudaMemcpy(A0.col.data(), M.a_col, nnz * sizeof(int32_t), cudaMemcpyDeviceToHost), err);
    DD_CUDA_TRY(cudaMemcpy(A0.val.data(), M.a_val, nnz * sizeof(double), cudaMemcpyDeviceToHost), err);
    AmgHierarchy H;
    std::string why;
    if (!build_amg(A0, H, why, device_spectral_radius(M, s))) {
        *fallback = true;
        err = why;
        return DD_ENOTCONV;
    }
    const int nl = (int)H.levels.size();

    // chunk width: six FP64 [m][kc] vectors on the fine level (five and the
    // pairs), two of pairs per coarser level, within a 24 GB workspace budget
    double per_col = 6.0 * 8.0 * (double)m;
    for (int l = 1; l < nl; ++l) per_col += 2.0 * 8.0 * (double)H.levels[l].A.rows;
    int64_t kc = (int64_t)(24e9 / per_col);
    kc = kc / 128 * 128;
    if (kc < 128) kc = 128;
    if (kc > ((k + 3) / 4) * 4) kc = ((k + 3) / 4) * 4;
    const int64_t kp = kc / 2;
    const int rpb0 = rows_per_block(m, kc);
    const int64_t nrb = (m + rpb0 - 1) / rpb0;
    // rows of a sparse product's band: two CTAs an SM over all columns, at least 32 rows
    std::vector<int> band(nl);
    const int64_t colb = (kp + kBandPairs - 1) / kBandPairs;
    for (int l = 0; l < nl; ++l) {
        const int64_t nb = std::max<int64_t>(1, 2LL * sm_count() / colb), rows = H.levels[l].A.rows;
        band[l] = (int)std::max<int64_t>(kBandRows, (rows + nb - 1) / nb);
    }
    const int64_t nbands = (m + band[0] - 1) / band[0];

    // one device allocation for the hierarchy and the small arrays (a solve has
    // dozens; allocated and freed one by one they cost 2 ms), the hierarchy's
    // part filled from one host buffer in one copy; the six fine-level blocks
    // apart (as one block with the rest, its release left the next
    // allocations, and the first pass over P, up to 2 ms slower)
    size_t total = 0;
    auto take = [&](size_t bytes) {
        const size_t o = total;
        total += (bytes + 255) / 256 * 256;
        return o;
    };
    struct Plan {
        const AmgCsr *h;
        DevCsr *d;
        size_t off, col, val;
    };
    std::vector<DevCsr> dG(nl), dQ(nl), dQt(nl);
    std::vector<Plan> plans;
    for (int l = 0; l + 1 < nl; ++l) {
        AmgLevel &L = H.levels[l];
        for (auto pr : {std::make_pair(&L.G, &dG[l]), std::make_pair(&L.Q, &dQ[l]), std::make_pair(&L.Qt, &dQt[l])}) {
            if (pr.first->col.size() > (size_t)INT32_MAX) {
                *fallback = true;
                err = "multigrid operators exceed 32-bit offsets";
                return DD_ENOMEM;
            }
            const size_t o = take((size_t)(pr.first->rows + 1) * sizeof(int32_t));
            const size_t cl = take(pr.first->col.size() * sizeof(int32_t));
            plans.push_back(Plan{pr.first, pr.second, o, cl, take(pr.first->val.size() * sizeof(float2))});
        }
    }
    const size_t o_ainv = take(H.coarse_inv.size() * sizeof(double));
    const size_t filled = total;
    const size_t vec = (size_t)m * kc * sizeof(double);
    std::vector<size_t> o_b(nl), o_x(nl);
    for (int l = 1; l < nl; ++l) {
        const size_t lv = (size_t)H.levels[l].A.rows * kc * sizeof(float2);
        o_b[l] = take(lv);
        o_x[l] = take(lv);
    }
    const size_t o_p0 = take((size_t)std::max(nrb, nbands) * kc * sizeof(double)), o_p1 = take((size_t)nrb * kc * sizeof(double));
    const size_t o_al = take(kc * sizeof(double)), o_be = take(kc * sizeof(double)), o_rz = take(kc * sizeof(double));
    const size_t o_bn = take(kc * sizeof(double)), o_dn = take(kc * sizeof(int));
    const size_t o_mr = take(sizeof(unsigned long long)), o_sh = take(kc * sizeof(int));
    std::vector<uint8_t> host(filled);
    for (const Plan &q : plans) {
        int32_t *off = reinterpret_cast<int32_t *>(host.data() + q.off);
        for (int64_t i = 0; i <= q.h->rows; ++i) off[i] = (int32_t)q.h->off[i];
        std::memcpy(host.data() + q.col, q.h->col.data(), q.h->col.size() * sizeof(int32_t));
        float2 *val = reinterpret_cast<float2 *>(host.data() + q.val);
        for (size_t i = 0; i < q.h->val.size(); ++i) val[i] = split_pair(q.h->val[i]);
    }
    // the coarsest inverse: FP64 where it solves the whole problem, else pairs
    if (nl == 1) {
        std::memcpy(host.data() + o_ainv, H.coarse_inv.data(), H.coarse_inv.size() * sizeof(double));
    } else {
        float2 *val = reinterpret_cast<float2 *>(host.data() + o_ainv);
        for (size_t i = 0; i < H.coarse_inv.size(); ++i) val[i] = split_pair(H.coarse_inv[i]);
    }
    uint8_t *ws = nullptr;
    double *fine[6] = {};
    cudaError_t ce = cudaMalloc((void **)&ws, total);
    for (double *&v : fine)
        if (ce == cudaSuccess) ce = cudaMalloc((void **)&v, vec);
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(ws, host.data(), filled, cudaMemcpyHostToDevice, s);
    auto drop = [&]() {
        if (ws) cudaFree(ws);
        for (double *v : fine)
            if (v) cudaFree(v);
    };
    if (ce != cudaSuccess) {
        drop();
        cudaGetLastError();
        *fallback = true;
        err = std::string("multigrid workspace allocation failed: ") + cudaGetErrorString(ce);
        return DD_ENOMEM;
    }
    auto release = [&]() {
        cudaStreamSynchronize(s);
        drop();
    };
    for (const Plan &q : plans)
        *q.d = DevCsr{reinterpret_cast<int32_t *>(ws + q.off), reinterpret_cast<int32_t *>(ws + q.col),
                      reinterpret_cast<float2 *>(ws + q.val)};
    auto at = [&](size_t o) { return reinterpret_cast<double *>(ws + o); };
    double *X = fine[0], *R = fine[1], *Z = fine[2], *Pd = fine[3], *AP = fine[4];
    double *part0 = at(o_p0), *part1 = at(o_p1), *alpha = at(o_al), *beta = at(o_be), *rz = at(o_rz), *bnorm = at(o_bn);
    int *done = reinterpret_cast<int *>(ws + o_dn), *shift = reinterpret_cast<int *>(ws + o_sh);
    const int2 *shift2 = reinterpret_cast<const int2 *>(shift);
    unsigned long long *maxres = reinterpret_cast<unsigned long long *>(ws + o_mr);
    auto lb = [&](int l) {
        return l == 0 ? reinterpret_cast<float4 *>(fine[5]) : reinterpret_cast<float4 *>(ws + o_b[l]);
    };
    auto lx = [&](int l) { return reinterpret_cast<float4 *>(ws + o_x[l]); };
    auto d2 = [](double *p) { return reinterpret_cast<double2 *>(p); };

    auto grid = [&](int64_t rows, int rb) {
        return dim3((unsigned)((rows + rb - 1) / rb), (unsigned)((kc + kColsPerBlock - 1) / kColsPerBlock));
    };
    auto grid2 = [&](int64_t rows, int rb) {
        return dim3((unsigned)((rows + rb - 1) / rb), (unsigned)((kp + kPairs - 1) / kPairs));
    };
    auto bands = [&](int l) {
        return dim3((unsigned)((H.levels[l].A.rows + band[l] - 1) / band[l]), (unsigned)colb);
    };
    const dim3 bb(kBandPairs, kBandRows);
    // Z = V(the fine level's pairs lb(0)), partial sums of R . Z into part0
    auto vcycle = [&]() {
        for (int l = 0; l + 1 < nl; ++l)
            df_spmm_kernel<<<bands(l + 1), bb, 0, s>>>(H.levels[l + 1].A.rows, kp, dQt[l].off, dQt[l].col, dQt[l].val,
                                                      lb(l), lb(l + 1), band[l + 1]);
        const int64_t nc = H.levels[nl - 1].A.rows;
        df_coarse_kernel<<<dim3((unsigned)((kp + kPairs - 1) / kPairs), (unsigned)nc), kPairs, 0, s>>>(
            nc, kp, reinterpret_cast<const float2 *>(ws + o_ainv), lb(nl - 1), lx(nl - 1));
        for (int l = nl - 2; l >= 0; --l) {
            const int64_t n = H.levels[l].A.rows;
            if (l > 0)
                df_up_kernel<false><<<bands(l), bb, 0, s>>>(n, kp, dG[l].off, dG[l].col, dG[l].val, dQ[l].off,
                                                            dQ[l].col, dQ[l].val, lb(l), lx(l + 1), nullptr, nullptr,
                                                            lx(l), nullptr, band[l]);
            else
                df_up_kernel<true><<<bands(l), bb, 0, s>>>(n, kp, dG[l].off, dG[l].col, dG[l].val, dQ[l].off,
                                                           dQ[l].col, dQ[l].val, lb(l), lx(l + 1), d2(R), shift2, Z,
                                                           d2(part0), band[l]);
        }
    };

    dd_status st = DD_OK;
    int32_t iters_max = 0;
    double res_max = 0.0;
    const int check_every = 4;
    const dim3 g0 = grid(m, rpb0), gc((unsigned)((kc + 31) / 32)), bc(32, kSumRows);
    for (int64_t c0 = 0; c0 < k && st == DD_OK; c0 += kc) {
        const int64_t kcur = (k - c0) < kc ? (k - c0) : kc;
        cudaMemsetAsync(X, 0, vec, s);
        cudaMemsetAsync(shift, 0, kc * sizeof(int), s);
        cudaMemsetAsync(R, 0, vec, s);
        if (M.n_rb > 0)
            scatter_rhs_kernel<<<(unsigned)((M.n_rb + 255) / 256), 256, 0, s>>>(M.n_rb, M.rb_row, M.rb_col, M.rb_val,
                                                                                c0, kcur, kc, R, shift);
        if (nl == 1) {   // the whole problem is the coarsest level: one exact solve
            coarse_solve_kernel<<<dim3((unsigned)((kc + 127) / 128), (unsigned)m), 128, 0, s>>>(m, kc, at(o_ainv), R, X);
            pack_chunk_kernel<<<dim3((unsigned)nrb, (unsigned)((kcur + kColsPerBlock - 1) / kColsPerBlock)),
                                kColsPerBlock, 0, s>>>(m, kcur, kc, c0, M.k_pad, M.interior, X, M.P, rpb0);
            iters_max = std::max(iters_max, 1);
            continue;
        }
        first_shift_kernel<<<(unsigned)((kc + 255) / 256), 256, 0, s>>>(kc, shift);
        df_first_kernel<<<grid2(m, rpb0), kPairs, 0, s>>>(m, kp, d2(R), shift2, lb(0), d2(part1), rpb0);
        vcycle();
        amg_init_scalars_kernel<<<gc, bc, 0, s>>>(nbands, nrb, kc, part0, part1, rz, bnorm, done);
        cudaMemcpyAsync(Pd, Z, vec, cudaMemcpyDeviceToDevice, s);
        int32_t it = 0;
        double res = 1.0;
        for (it = 1; it <= max_iter; ++it) {
            spmm_dot_kernel<<<g0, kColsPerBlock, 0, s>>>(m, kc, M.a_off, M.a_col, M.a_val, Pd, AP, part0, rpb0);
            alpha_kernel<<<gc, bc, 0, s>>>(nrb, kc, part0, rz, done, alpha);
            update_r_kernel<<<grid2(m, rpb0), kPairs, 0, s>>>(m, kp, d2(alpha), d2(R), d2(AP), shift2, lb(0), d2(part1),
                                                              rpb0);
            vcycle();
            cudaMemsetAsync(maxres, 0, sizeof(unsigned long long), s);
            beta_kernel<<<gc, bc, 0, s>>>(nbands, nrb, kc, part0, part1, bnorm, rz, done, beta, maxres, shift);
            update_xp_kernel<<<grid2(m, rpb0), kPairs, 0, s>>>(m, kp, d2(alpha), d2(beta), d2(Z), d2(X), d2(Pd), rpb0);
            if (it % check_every == 0 || it == max_iter) {
                unsigned long long bits = 0;
                cudaError_t e1 = cudaMemcpyAsync(&bits, maxres, sizeof bits, cudaMemcpyDeviceToHost, s);
                cudaError_t e2 = cudaStreamSynchronize(s);
                if (e1 != cudaSuccess || e2 != cudaSuccess) {
                    err = std::string("PCG iteration failed: ") + cudaGetErrorString(e1 != cudaSuccess ? e1 : e2);
                    st = DD_ECUDA;
                    break;
                }
                std::memcpy(&res, &bits, sizeof res);
                if (res <= rtol) break;
            }
        }
        if (st != DD_OK) break;
        if (it > max_iter) it = max_iter;
        iters_max = std::max(iters_max, it);
        res_max = std::max(res_max, res);
        pack_chunk_kernel<<<dim3((unsigned)nrb, (unsigned)((kcur + kColsPerBlock - 1) / kColsPerBlock)),
                            kColsPerBlock, 0, s>>>(m, kcur, kc, c0, M.k_pad, M.interior, X, M.P, rpb0);
    }
    cudaError_t e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = cudaGetLastError();
    release();
    if (st != DD_OK) return st;
    if (e != cudaSuccess) {
        err = std::string("PCG failed: ") + cudaGetErrorString(e);
        return DD_ECUDA;
    }
    if (iters_out) *iters_out = iters_max;
    if (resid_out) *resid_out = res_max;
    M.has_P = true;
    if (!(res_max <= rtol)) {
        char buf[160];
        std::snprintf(buf, sizeof buf, "PCG stopped at %d iterations with relative residual %.3e > %.3e",
                      iters_max, res_max, rtol);
        err = buf;
        return DD_ENOTCONV;
    }
    return DD_OK;
}

bool use_multigrid(int64_t m) {
    static int mode = -1;
    if (mode < 0) {
        const char *e = getenv("DD_PCG_PRECOND");
        mode = (e && !strcmp(e, "jacobi")) ? 0 : 1;
    }
    return mode == 1 && m >= 256;
}

}  // namespace

dd_status run_pcg(DevMesh &M, double rtol, int32_t max_iter, cudaStream_t s, int32_t *iters_out,
                  double *resid_out, std::string &err) {
    const int64_t m = M.m, k = M.k;
    if (!M.P) {
        DD_CUDA_TRY(cudaMalloc((void **)&M.P, (size_t)M.n_v * M.k_pad * sizeof(float)), err);
        M.owned.push_back(M.P);
        M.bytes += (int64_t)M.n_v * M.k_pad * sizeof(float);
    }
    DD_CUDA_TRY(cudaMemsetAsync(M.P, 0, (size_t)M.n_v * M.k_pad * sizeof(float), s), err);
    if (k > 0)
        boundary_identity_kernel<<<(unsigned)((k + 255) / 256), 256, 0, s>>>(k, M.k_pad, M.boundary, M.P);
    int32_t iters_max = 0;
    double res_max = 0.0;
    if (m == 0) {
        M.has_P = true;
        if (iters_out) *iters_out = 0;
        if (resid_out) *resid_out = 0.0;
        return DD_OK;
    }

    if (use_multigrid(m)) {
        bool fallback = false;
        const dd_status sa = run_pcg_amg(M, rtol, max_iter, s, iters_out, resid_out, err, &fallback);
        if (!fallback) return sa;
        err.clear();   // the hierarchy could not be built: the diagonal preconditioner below
    }

    // chunk width: four FP64 [m][kc] vectors within a 24 GB workspace budget
    const double budget = 24e9;
    int64_t kc = (int64_t)(budget / (4.0 * 8.0 * (double)m));
    kc = kc / 128 * 128;
    if (kc < 128) kc = 128;
    if (kc > ((k + 3) / 4) * 4) kc = ((k + 3) / 4) * 4;

    Work w;
    w.m = m;
    w.kc = kc;
    // rows per CTA: enough CTAs (about 16 per SM) for small meshes, 256 rows for large ones
    int rpb = 256;
    {
        int sms = 0, dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
        const int64_t colblocks = (kc + kColsPerBlock - 1) / kColsPerBlock;
        const int64_t want = m * colblocks / (16LL * sms);
        while (rpb > 8 && rpb > want) rpb >>= 1;
    }
    w.nrb = (m + rpb - 1) / rpb;
    std::vector<void *> tmp;
    cudaError_t ce = cudaSuccess;
    size_t vec = (size_t)m * kc;
    if ((ce = alloc(&w.X, vec)) == cudaSuccess) tmp.push_back(w.X);
    if (ce == cudaSuccess && (ce = alloc(&w.R, vec)) == cudaSuccess) tmp.push_back(w.R);
    if (ce == cudaSuccess && (ce = alloc(&w.Pd, vec)) == cudaSuccess) tmp.push_back(w.Pd);
    if (ce == cudaSuccess && (ce = alloc(&w.AP, vec)) == cudaSuccess) tmp.push_back(w.AP);
    if (ce == cudaSuccess && (ce = alloc(&w.part0, (size_t)w.nrb * kc)) == cudaSuccess) tmp.push_back(w.part0);
    if (ce == cudaSuccess && (ce = alloc(&w.part1, (size_t)w.nrb * kc)) == cudaSuccess) tmp.push_back(w.part1);
    if (ce == cudaSuccess && (ce = alloc(&w.alpha, (size_t)kc)) == cudaSuccess) tmp.push_back(w.alpha);
    if (ce == cudaSuccess && (ce = alloc(&w.beta, (size_t)kc)) == cudaSuccess) tmp.push_back(w.beta);
    if (ce == cudaSuccess && (ce = alloc(&w.rz, (size_t)kc)) == cudaSuccess) tmp.push_back(w.rz);
    if (ce == cudaSuccess && (ce = alloc(&w.bnorm, (size_t)kc)) == cudaSuccess) tmp.push_back(w.bnorm);
    if (ce == cudaSuccess && (ce = alloc(&w.dinv, (size_t)m)) == cudaSuccess) tmp.push_back(w.dinv);
    if (ce == cudaSuccess && (ce = alloc(&w.done, (size_t)kc)) == cudaSuccess) tmp.push_back(w.done);
    if (ce == cudaSuccess && (ce = alloc(&w.maxres, 1)) == cudaSuccess) tmp.push_back(w.maxres);
    auto release = [&]() {
        for (void *p : tmp) cudaFree(p);
        tmp.clear();
    };
    if (ce != cudaSuccess) {
        release();
        cudaGetLastError();
        err = std::string("PCG workspace allocation failed: ") + cudaGetErrorString(ce);
        return DD_ENOMEM;
    }

    dd_status st = DD_OK;
    const int check_every = 16;
    dinv_kernel<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(m, M.a_diag, w.dinv);
    for (int64_t c0 = 0; c0 < k && st == DD_OK; c0 += kc) {
        const int64_t kcur = (k - c0) < kc ? (k - c0) : kc;   // columns in this chunk
        // vectors keep pitch kc; columns beyond kcur stay zero and converge at once
        dim3 g2((unsigned)w.nrb, (unsigned)((kc + kColsPerBlock - 1) / kColsPerBlock));
        dim3 gc((unsigned)((kc + 31) / 32));
        dim3 bc(32, kSumRows);
        cudaMemsetAsync(w.X, 0, vec * sizeof(double), s);
        cudaMemsetAsync(w.R, 0, vec * sizeof(double), s);
        if (M.n_rb > 0)
            scatter_rhs_kernel<<<(unsigned)((M.n_rb + 255) / 256), 256, 0, s>>>(M.n_rb, M.rb_row, M.rb_col,
                                                                                M.rb_val, c0, kcur, kc, w.R, nullptr);
        init_p_kernel<<<g2, kColsPerBlock, 0, s>>>(m, kc, w.dinv, w.R, w.Pd, w.part0, w.part1, rpb);
        init_scalars_kernel<<<gc, bc, 0, s>>>(w.nrb, kc, w.part0, w.part1, w.rz, w.bnorm, w.done);
        int32_t it = 0;
        double res = 1.0;
        for (it = 1; it <= max_iter; ++it) {
            spmm_dot_kernel<<<g2, kColsPerBlock, 0, s>>>(m, kc, M.a_off, M.a_col, M.a_val, w.Pd, w.AP, w.part0, rpb);
            alpha_kernel<<<gc, bc, 0, s>>>(w.nrb, kc, w.part0, w.rz, w.done, w.alpha);
            update_xr_kernel<<<g2, kColsPerBlock, 0, s>>>(m, kc, w.alpha, w.dinv, w.X, w.R, w.Pd, w.AP, w.part0,
                                                          w.part1, rpb);
            cudaMemsetAsync(w.maxres, 0, sizeof(unsigned long long), s);
            beta_kernel<<<gc, bc, 0, s>>>(w.nrb, w.nrb, kc, w.part0, w.part1, w.bnorm, w.rz, w.done, w.beta,
                                          w.maxres, nullptr);
            update_p_kernel<<<g2, kColsPerBlock, 0, s>>>(m, kc, w.beta, w.dinv, w.R, w.Pd, rpb);
            if (it % check_every == 0 || it == max_iter) {
                unsigned long long bits = 0;
                cudaError_t e1 = cudaMemcpyAsync(&bits, w.maxres, sizeof bits, cudaMemcpyDeviceToHost, s);
                cudaError_t e2 = cudaStreamSynchronize(s);
                if (e1 != cudaSuccess || e2 != cudaSuccess) {
                    err = std::string("PCG iteration failed: ") +
                          cudaGetErrorString(e1 != cudaSuccess ? e1 : e2);
                    st = DD_ECUDA;
                    break;
                }
                double r;
                static_assert(sizeof(r) == sizeof(bits), "size");
                std::memcpy(&r, &bits, sizeof r);
                res = r;
                if (res <= rtol) break;
            }
        }
        if (st != DD_OK) break;
        if (it > max_iter) it = max_iter;
        if (it > iters_max) iters_max = it;
        if (res > res_max) res_max = res;
        pack_chunk_kernel<<<dim3((unsigned)w.nrb, (unsigned)((kcur + kColsPerBlock - 1) / kColsPerBlock)),
                            kColsPerBlock, 0, s>>>(m, kcur, kc, c0, M.k_pad, M.interior, w.X, M.P, rpb);
    }
    cudaError_t e = cudaStreamSynchronize(s);
    release();
    if (st != DD_OK) return st;
    if (e != cudaSuccess) {
        err = std::string("PCG failed: ") + cudaGetErrorString(e);
        return DD_ECUDA;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        err = std::string("PCG launch failed: ") + cudaGetErrorString(e);
        return DD_ECUDA;
    }
    M.has_P = true;
    if (iters_out) *iters_out = iters_max;
    if (resid_out) *resid_out = res_max;
    if (!(res_max <= rtol)) {
        char buf[160];
        std::snprintf(buf, sizeof buf, "PCG stopped at %d iterations with relative residual %.3e > %.3e",
                      iters_max, res_max, rtol);
        err = buf;
        return DD_ENOTCONV;
    }
    return DD_OK;
}

dd_status store_poisson(DevMesh &M, const double *P, cudaStream_t s, std::string &err) {
    if (!M.P) {
        DD_CUDA_TRY(cudaMalloc((void **)&M.P, (size_t)M.n_v * M.k_pad * sizeof(float)), err);
        M.owned.push_back(M.P);
        M.bytes += (int64_t)M.n_v * M.k_pad * sizeof(float);
    }
    const size_t n = (size_t)M.n_v * M.k;
    double *d = nullptr;
    if (cudaMalloc((void **)&d, n * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        err = "staging allocation for the Poisson kernel failed";
        return DD_ENOMEM;
    }
    cudaError_t e = cudaMemcpyAsync(d, P, n * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(M.P, 0, (size_t)M.n_v * M.k_pad * sizeof(float), s);
    if (e == cudaSuccess) {
        store_host_p_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(M.n_v, M.k, M.k_pad, d, M.P);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d);
    if (e != cudaSuccess) {
        err = std::string("storing the Poisson kernel failed: ") + cudaGetErrorString(e);
        return DD_ECUDA;
    }
    M.has_P = true;
    return DD_OK;
}
