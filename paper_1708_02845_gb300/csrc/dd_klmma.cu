// FP32-accurate KL fields of many targets on the tensor cores.
//
//   KL_t(x) = e_x - C[x,t],   e_x = sum_b P[x,b] log P[x,b],
//                             C[x,t] = sum_b P[x,b] log P[t,b]      (Eq. 35 with Eq. 17)
//
// C is a contraction, but KL is the small difference of e_x and C (both up to
// about 10), so C is needed to about 2^-28 of its size: more than FP32 products
// with FP32 accumulation give.  Both operands are therefore cut into BF16
// slices on fixed grids, in the manner of Ozaki, Ogita, Oishi and Rump
// ("Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication and its applications", Numerical Algorithms 2012):
// within 64 columns (a chunk) the entries of one row of P are rounded to
// multiples of q = 2^-7 of their largest entry's power of two, the remainder
// to multiples of 2^-9 q, and so on (four slices), and the target's log2 P
// the same way (three slices; entries below -32 keep their own BF16 grid, so
// that one near-empty column does not coarsen its chunk).  The logs are taken
// from a whole number in the middle of their chunk's, c, which counts with the
// chunk's sum of P:  sum_b P l = sum_b P (l - c) + c sum_b P.  Along a boundary
// log2 P varies little, so l - c is several times smaller than l, and so is
// what three slices of it leave.  The second term is summed like the first, by
// columns of their own behind the map's: the chunks' sums of P, exact, on the
// rows' side and c on the targets'.  Slices are integers
// of at most 2^8 times their grid, so a product of two leading slices is an
// integer of at most 2^16 units and a chunk's 64 of them sum exactly in the 24
// bits of an FP32 accumulator.  Nine products are kept,
//   A = p1 l1 (exact),   B = (p4 l1 + p3 l2 + p2 l3) + (p1 l3 + p2 l2 + p3 l1) + (p1 l2 + p2 l1)
// (each bracket 2^-9 of the next, the smallest first), in two accumulators, or
// one a bracket (up to 64 targets); what is dropped is 2^-36 of the chunk's
// largest entry times the logs, and P times what the three slices leave of
// l - c: at most 2^-26 of its largest power of two.  After every chunk
// A is split at multiples of 2^-15: the upper part goes into a total of
// such multiples (exact below 2^9), the rest and B into a second total.
// e_x is summed once per mesh in pairs of floats and kept in the same two parts.
//
// Against 64 bits (KL above 0.07, solved kernels of obstacle grids of 64 to 201
// cells a side) the relative error is 3.5e-8 .. 6.2e-8 in the root mean square
// of every range of KL and at most 3.6e-7, against 6.9e-8 .. 1.7e-7 and 1.4e-6
// for the FP32 sums of the tile kernels and their recompute below 0.25 (slices
// of l itself: up to 1.6e-7 below 0.25).  For target rows of equal entries,
// where what the slices leave does not average out: below 8e-8, against 1.6e-7
// (4.4e-7).  The pairs below kMmaExactBelow are recomputed in the exact form as
// there.  The extra columns cost 0.3 % of a call with a chunk more (grid450,
// 1,024 targets: 54.95 -> 55.13 ms) and up to 1 % of small ones.  Slicing P, once
// a map, takes a quarter longer with the chunks' sums (201 x 201 cells: 131 -> 165
// us, 82 % of the issue slots).
//
// Kernel: persistent, one CTA per SM walks 128-row x N-target output tiles.
// The operands lie in global memory chunk by chunk in the shared-memory image
// of the MMA (K-major, 128-byte swizzle), so a stage is two contiguous bulk
// copies.  Warp 0 copies, warp 1 issues the MMAs (16 or 36 of K = 16 a chunk) into
// one of two accumulator sets in TMEM, warps 2-9 take the finished set of a
// chunk out and add it to the totals in registers while the next chunk's MMAs
// run.  Every wait is bounded and also gives up when another role has.
//
// Measured: grid450, 1,024 targets: 7.8 ms (N = 128; 14.0 TFLOP issued, 1,790
// TFLOP/s = 93 % of the measured burst rate of 1,931), with the TV tile pass
// (45.3 ms) and a recompute of fewer pairs (1.6 against 4.1 ms) in place of
// the 94.5 ms KL+TV tile pass: a call 98.9 -> 55.1 ms.  grid140, 64 targets:
// 34 us (N = 64; the slices' 131 MB from memory bound it), a call 321 -> 181
// us.  KL alone, 201 x 201 cells, 7 targets: a call 228 -> 106 us.
#include <cuda_bf16.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "dd_bulk.cuh"
#include "dd_f32x2.cuh"
#include "dd_internal.h"
#include "dd_logtable.cuh"

namespace {

constexpr int BM = 128, BK = 64;              // rows of a tile, columns of a chunk
constexpr int NSA = 4, NSB = 3;               // slices of P and of log2 P
constexpr int ROW_B = BK * 2;                 // bytes of a slice row in a chunk
constexpr int A_BYTES = NSA * BM * ROW_B;     // 64 KB
constexpr int64_t kMaxColumns = 1 << 17;
constexpr float kLn2 = 0.693147180559945309f;
constexpr float kSplit = 384.0f;              // 1.5 * 2^8: adding it rounds |A| < 128 to multiples of 2^-15

__host__ __device__ constexpr int b_bytes(int N) { return NSB * N * ROW_B; }
__host__ __device__ constexpr int stages(int N) { return N >= 64 ? 2 : 3; }
constexpr int smem_bytes(int N) { return stages(N) * (A_BYTES + b_bytes(N)) + 1024 + 256; }

// byte offset of column c (0 .. 63) of row r in a K-major chunk image, 128-byte swizzle
__device__ __forceinline__ int image_at(int r, int c) {
    return r * ROW_B + ((((c >> 3) ^ (r & 7)) << 4) | ((c & 7) << 1));
}

__device__ __forceinline__ bool wait_or_abort(uint64_t *bar, uint32_t parity, int *err, volatile int *abort) {
    for (uint32_t i = 0; i < kSuspendLimit; ++i) {
        if (mbar_try(bar, parity, 1000u)) return true;
        if (*abort) return false;
    }
    atomicExch(err, 2);
    *abort = 1;
    return false;
}
__device__ __forceinline__ void arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// D = F32, A = B = BF16, both K-major, M = 128
template <int N>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, bool accumulate) {
    constexpr uint32_t idesc =
        (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate ? 1u : 0u)
        : "memory");
}
__device__ __forceinline__ void commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}

// 8 consecutive accumulator columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_ld8(uint32_t (&r)[8], uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
}

struct KlOne {
    const uint8_t *A, *B;    // chunk images of the mesh's rows and of the targets
    const float2 *ex;        // [row tiles * 128]
    float *out;              // [T][n_v]
    int64_t n_v;
    int32_t T, nch;
};

template <int N, bool BATCH>
__global__ void __launch_bounds__(320, 1) kl_mma_kernel(const KlOne one, const BatchProblem *__restrict__ probs,
                                                        const BatchItem *__restrict__ items, int32_t n_items,
                                                        int *__restrict__ err) {
    constexpr int ST = stages(N), SB = A_BYTES + b_bytes(N);
    constexpr int CW = N / 2;            // columns of an epilogue warp
    // An MMA fetches its row operand (128 x 16, 4 KB) from shared memory in some
    // 64 clocks, as long as it takes to multiply 128 columns: with fewer targets
    // the row slices are fetched once each instead of once a product, against
    // the target slices side by side (p1 [l1 l2 l3], p2 [l1 l2 l3], p3 [l1 l2],
    // p4 [l1]), each one accumulator further on, so that the columns of an
    // accumulator hold one bracket of the sum: 16 MMAs a chunk instead of 36
    // (201 x 201 cells, 7 targets: 73 -> 53 us with the quarters above; grid140
    // with 64: 44 -> 34)
    constexpr bool kJoined = N <= 64;
    constexpr int NACC = kJoined ? 4 : 2;
    constexpr uint32_t TCOLS = 2 * NACC * N;    // two sets of N-column accumulators (a power of two)
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + ST * SB);
    uint64_t *empty = full + ST;
    uint64_t *accf = empty + ST;         // [2] accumulators written
    uint64_t *acce = accf + 2;           // [2] accumulators read out
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acce + 2);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accf[b], 1);
            mbar_init(&acce[b], 8);
        }
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    // Few targets: the copies of the rows bound the pass, and a last round of a
    // few tiles takes as long as a full one (201 x 201 cells: 317 tiles on 152
    // SMs, 73 us).  Its tiles are cut into quarters of 32 rows, an item each:
    // only those rows are copied (the MMA's others hold what was there, and
    // their results are not stored).
    constexpr bool kQuarters = !BATCH && N == 16;
    const int rounds = n_items / (int)gridDim.x * (int)gridDim.x;
    const bool cut = kQuarters && rounds > 0 && 2 * (n_items - rounds) <= (int)gridDim.x;
    const int n_whole = cut ? rounds : n_items, n_work = n_whole + 4 * (n_items - n_whole);
    // the quarter of its tile that work item i is, or -1: the whole of it
    auto quarter = [&](int i) { return i < n_whole ? -1 : (i - n_whole) & 3; };

    // item i: its operands and sizes.  One problem: the target tiles vary
    // fastest, so the CTAs that work at one time share their row tiles in L2
    auto problem = [&](int i, int &xt, int &at) {
        if (i > n_whole) i = n_whole + ((i - n_whole) >> 2);
        if (BATCH) {
            const BatchItem w = items[i];
            const BatchProblem &q = probs[w.prob];
            xt = w.x_tile;
            at = w.a_tile;
            return KlOne{q.KA, q.KB, q.kex, q.out_kl, q.n_v, q.T, q.knch};
        }
        const int nat = (one.T + N - 1) / N;
        xt = i / nat;
        at = i - xt * nat;
        return one;
    };

    if (warp == 0) {
        if (lane == 0) {
            int g = 0;
            for (int i = blockIdx.x; i < n_work && !*abort; i += gridDim.x) {
                int xt, at;
                const KlOne q = problem(i, xt, at);
                const int part = quarter(i);
                const uint8_t *a = q.A + (int64_t)xt * q.nch * A_BYTES, *b = q.B + (int64_t)at * q.nch * b_bytes(N);
                for (int c = 0; c < q.nch; ++c, ++g) {
                    const int s = g % ST, round = g / ST;
                    if (round > 0 && !wait_or_abort(&empty[s], (round - 1) & 1, err, abort)) break;
                    uint8_t *st = smem + s * SB;
                    const uint8_t *ac = a + (int64_t)c * A_BYTES;
                    if (part < 0) {
                        mbar_expect_tx(&full[s], SB);
                        bulk_g2s(st, ac, A_BYTES, &full[s]);
                    } else {
                        constexpr int kPart = 32 * ROW_B;      // of each slice
                        mbar_expect_tx(&full[s], NSA * kPart + b_bytes(N));
                        for (int k = 0; k < NSA; ++k)
                            bulk_g2s(st + k * BM * ROW_B + part * kPart, ac + k * BM * ROW_B + part * kPart, kPart,
                                     &full[s]);
                    }
                    bulk_g2s(st + A_BYTES, b + (int64_t)c * b_bytes(N), b_bytes(N), &full[s]);
                }
            }
            // every issued stage must have landed before the CTA may exit
            volatile int never = 0;
            for (int k = g - ST < 0 ? 0 : g - ST; k < g; ++k) wait_or_abort(&full[k % ST], (k / ST) & 1, err, &never);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int g = 0;
            bool ok = true;
            for (int i = blockIdx.x; i < n_work && ok && !*abort; i += gridDim.x) {
                int xt, at;
                const int nch = problem(i, xt, at).nch;
                for (int c = 0; c < nch; ++c, ++g) {
                    const int s = g % ST, buf = g & 1;
                    if ((g >= 2 && !wait_or_abort(&acce[buf], ((g >> 1) - 1) & 1, err, abort)) ||
                        !wait_or_abort(&full[s], (g / ST) & 1, err, abort)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t st = smem_addr(smem + s * SB);
                    const uint64_t a0 = smem_desc(st), b0 = smem_desc(st + A_BYTES);
                    const uint32_t accA = tmem + (uint32_t)(buf * NACC * N), accB = accA + N;
                    constexpr uint64_t SA = (BM * ROW_B) >> 4, SBN = (N * ROW_B) >> 4;   // one slice further
                    if constexpr (kJoined) {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            mma<N>(accA + 3 * N, a0 + 3 * SA + 2 * kk, b0 + 2 * kk, kk > 0);
                            mma<3 * N>(accA, a0 + 2 * kk, b0 + 2 * kk, kk > 0);
                            mma<2 * N>(accA + 2 * N, a0 + 2 * SA + 2 * kk, b0 + 2 * kk, true);
                            mma<3 * N>(accA + N, a0 + SA + 2 * kk, b0 + 2 * kk, true);
                        }
                    } else {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) mma<N>(accA, a0 + 2 * kk, b0 + 2 * kk, kk > 0);
                        constexpr int pi[8] = {3, 2, 1, 0, 1, 2, 0, 1}, li[8] = {0, 1, 2, 2, 1, 0, 1, 0};
#pragma unroll
                        for (int p = 0; p < 8; ++p)
#pragma unroll
                            for (int kk = 0; kk < BK / 16; ++kk)
                                mma<N>(accB, a0 + pi[p] * SA + 2 * kk, b0 + li[p] * SBN + 2 * kk, p > 0 || kk > 0);
                    }
                    commit(&empty[s]);       // the stage is free once these MMAs complete
                    commit(&accf[buf]);
                }
            }
            // every MMA issued here has completed before TMEM may be freed
            volatile int never = 0;
            if (g > 0) wait_or_abort(&accf[(g - 1) & 1], ((g - 1) >> 1) & 1, err, &never);
        }
    } else {
        // warps 2..9: TMEM lanes 32 (warp % 4) .., columns of half (warp - 2) / 4
        const int quad = warp & 3, half = (warp - 2) >> 2;
        const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
        const f2_t split = pk(kSplit, kSplit), nsplit = pk(-kSplit, -kSplit), mone = pk(-1.0f, -1.0f);
        int g = 0;
        bool ok = true;
        for (int i = blockIdx.x; i < n_work && ok; i += gridDim.x) {
            int xt, at;
            const KlOne q = problem(i, xt, at);
            f2_t hi[CW / 2], lo[CW / 2];
#pragma unroll
            for (int j = 0; j < CW / 2; ++j) hi[j] = lo[j] = 0ULL;
            for (int c = 0; c < q.nch; ++c, ++g) {
                const int buf = g & 1;
                ok = __all_sync(0xffffffffu, wait_or_abort(&accf[buf], (g >> 1) & 1, err, abort));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t ta = tmem + lane_base + (uint32_t)(buf * NACC * N + half * CW);
#pragma unroll
                for (int c0 = 0; c0 < CW; c0 += 8) {
                    uint32_t ra[8], rb[8], rc[8], rd[8];
                    tmem_ld8(ra, ta + c0);
                    tmem_ld8(rb, ta + N + c0);
                    if constexpr (kJoined) {
                        tmem_ld8(rc, ta + 2 * N + c0);
                        tmem_ld8(rd, ta + 3 * N + c0);
                    }
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const f2_t a = pk(__uint_as_float(ra[2 * j]), __uint_as_float(ra[2 * j + 1]));
                        f2_t b = pk(__uint_as_float(rb[2 * j]), __uint_as_float(rb[2 * j + 1]));
                        if constexpr (kJoined) {
                            const f2_t c3 = pk(__uint_as_float(rc[2 * j]), __uint_as_float(rc[2 * j + 1]));
                            const f2_t d4 = pk(__uint_as_float(rd[2 * j]), __uint_as_float(rd[2 * j + 1]));
                            b = add2(add2(d4, c3), b);
                        }
                        const f2_t h = add2(add2(a, split), nsplit);
                        f2_t &H = hi[c0 / 2 + j], &L = lo[c0 / 2 + j];
                        H = add2(H, h);
                        L = add2(L, add2(b, fma2(h, mone, a)));
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) arrive(&acce[buf]);
            }
            if (!ok) break;
            const int64_t row = (int64_t)xt * BM + quad * 32 + lane;
            const int part = quarter(i);
            if (row < q.n_v && (part < 0 || part == quad)) {
                const float2 e = q.ex[row];
                const int a0 = at * N + half * CW;
#pragma unroll
                for (int j = 0; j < CW; ++j) {
                    float h[2], l[2];
                    upk(hi[j / 2], h[0], h[1]);
                    upk(lo[j / 2], l[0], l[1]);
                    if (a0 + j < q.T)
                        q.out[(int64_t)(a0 + j) * q.n_v + row] = kLn2 * ((e.x - h[j & 1]) + (e.y - l[j & 1]));
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
}

// ---------------------------------------------------------------- operands
// log2 of a positive normal FP32 number as hi + lo, hi a multiple of 2^-12 (an
// FP32 number exactly), |lo| < 2^-7: Tang's table method (128 midpoints c_j,
// r_j = 1 / c_j rounded) with the Taylor series of log(1 + u), u = m r_j - 1
// rounded once (|u| <= 2^-8, so to 2^-33).  The pair errs by less than 2^-31.
// In FP64, of which this part does one operation for 60 in FP32, the logs of a
// map's slices were most of its first call (201 x 201 cells: 1.0 ms).
constexpr int kTab = 128;
struct Log2Tab {
    float r[kTab], h[kTab], l[kTab];
};
__device__ __forceinline__ void build_log2_table(Log2Tab &t) {
    for (int j = threadIdx.x; j < kTab; j += blockDim.x) {
        t.r[j] = __uint_as_float(kLogTableBits[j]);
        t.h[j] = __uint_as_float(kLogTableBits[2 * kTab + j]);
        t.l[j] = __uint_as_float(kLogTableBits[3 * kTab + j]);
    }
}
__device__ __forceinline__ float2 log2_pair(float p, const Log2Tab &t) {
    const int i = __float_as_int(p);
    const int j = (i >> 16) & (kTab - 1);
    const float u = __fmaf_rn(__int_as_float((i & 0x007FFFFF) | 0x3F800000), t.r[j], -1.0f);
    float s = __fmaf_rn(0.2f, u, -0.25f);
    s = __fmaf_rn(s, u, 1.0f / 3.0f);
    s = __fmaf_rn(s, u, -0.5f);
    const float v = __fmaf_rn(__fmul_rn(s, u), u, u);                       // log(1 + u)
    // times log2 e as the sum of its rounding and the rest
    constexpr float c = 1.44269504f, cl = (float)(1.4426950408889634074 - (double)1.44269504f);
    const float w = __fmaf_rn(v, c, __fmaf_rn(v, cl, t.l[j]));
    return make_float2((float)((i >> 23) - 127) + t.h[j], w);
}
// (s, c) += a: two-sum
__device__ __forceinline__ void pair_add(float &s, float &c, float a) {
    const float t = __fadd_rn(s, a), b = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(a, b)));
    s = t;
}

// Columns: the k_pad of P in chunks of BK, then one for each of those chunks
// (its sum of P; its c), then zeros to whole chunks.
__host__ __device__ constexpr int data_chunks(int64_t k_pad) { return (int)((k_pad + BK - 1) / BK); }
__host__ __device__ constexpr int all_chunks(int64_t k_pad) {
    return (int)((k_pad + data_chunks(k_pad) + BK - 1) / BK);
}

// a + b = s + t
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &t) {
    s = __fadd_rn(a, b);
    const float v = __fsub_rn(s, a);
    t = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
}

// the grid of a chunk of P: 2^-7 of its largest entry's power of two (chunks below 2^-87: of that)
__device__ __forceinline__ int row_grid(float x, float y) {
    // entries are not negative: their bit patterns order as the numbers do
    const unsigned mx = __reduce_max_sync(0xffffffffu, max(__float_as_uint(x), __float_as_uint(y)));
    return min(max((int)(mx >> 23), 40), 200) - 7;
}

constexpr float kMagic = 12582912.0f;       // 1.5 * 2^23
constexpr int kMagicBits = 0x4B400000;

// The slices of P's rows and e_x, one warp per row (rows past n_v: zeros), two
// columns a lane.  Rows that the exactness argument does not cover (an entry
// that is negative, infinite or NaN, or a sum above 1.01) raise *bad.
__global__ void __launch_bounds__(256, 8) kl_rows_kernel(const float *__restrict__ P, int64_t n_v, int64_t n_pad,
                                                      int64_t k_pad, uint8_t *__restrict__ A,
                                                      float2 *__restrict__ ex, int *__restrict__ bad) {
    __shared__ Log2Tab tab;
    extern __shared__ float2 sums[];     // [8][chunks of P]: a row's sums of P, pairs
    build_log2_table(tab);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int nb = data_chunks(k_pad), nch = all_chunks(k_pad), whole = (int)(k_pad / BK);
    float2 *rs = sums + (threadIdx.x >> 5) * nb;
    const int64_t nw = (int64_t)gridDim.x * 8;
    for (int64_t x = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); x < n_pad; x += nw) {
        float es = 0.0f, ec = 0.0f;      // this lane's part of e_x, a pair
        float sum = 0.0f;
        bool wrong = false;
        uint8_t *img = A + (x / BM) * nch * A_BYTES + image_at((int)(x % BM), 2 * lane);
        auto store = [&](int s, float rx, float ry) {
            *reinterpret_cast<__nv_bfloat162 *>(img + s * BM * ROW_B) =
                __nv_bfloat162(__float2bfloat16_rn(rx), __float2bfloat16_rn(ry));
        };
        // (k_pad is a multiple of 4; the next chunk's entries are read ahead of this one's sums)
        auto entries = [&](int c) {
            const int b = c * BK + 2 * lane;
            return x < n_v && b < k_pad ? *reinterpret_cast<const float2 *>(P + x * k_pad + b) : make_float2(0.f, 0.f);
        };
        float2 ahead = entries(0);
        for (int c = 0; c < nb; ++c) {
            float2 p = ahead;
            if (c + 1 < nb) ahead = entries(c + 1);
            wrong |= !(p.x >= 0.f && p.y >= 0.f && p.x <= 2.f && p.y <= 2.f);
            sum += p.x + p.y;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float pv = i ? p.y : p.x;
                if (pv >= FLT_MIN) {
                    const float2 l = log2_pair(pv, tab);
                    const float a = __fmul_rn(pv, l.x);
                    ec = __fadd_rn(ec, __fmaf_rn(pv, l.y, __fmaf_rn(pv, l.x, -a)));
                    pair_add(es, ec, a);
                }
            }
            const int g = row_grid(p.x, p.y);
            float q = __int_as_float(g << 23), iq = __int_as_float((254 - g) << 23);
            int n[NSA];
#pragma unroll
            for (int s = 0; s < NSA; ++s) {
                // to the nearest multiple by adding 1.5 * 2^23, whose last bits then hold it (rintf
                // and conversions to int run at a quarter of the rate)
                const float tx = __fmaf_rn(p.x, iq, kMagic), ty = __fmaf_rn(p.y, iq, kMagic);
                const float rx = (tx - kMagic) * q, ry = (ty - kMagic) * q;
                n[s] = __float_as_int(tx) + __float_as_int(ty) - 2 * kMagicBits;
                if (c < whole) store(s, rx, ry);
                p.x -= rx;
                p.y -= ry;
                q *= 0x1p-9f;
                iq *= 0x1p9f;
            }
            if (c < whole) img += A_BYTES;
            // the slices' sums, up to 2^14 of their grids: two to a word, 2^-9 of a grid apart
            const int n01 = __reduce_add_sync(0xffffffffu, n[0] * 65536 + n[1]),
                      n23 = __reduce_add_sync(0xffffffffu, n[2] * 65536 + n[3]);
            if (lane == 0) {
                auto both = [](int v, int g) {      // exact
                    const int low = (int)(short)(v & 0xffff);
                    return __int_as_float(g << 23) * ((float)((v - low) >> 16) + 0x1p-9f * (float)low);
                };
                rs[c] = make_float2(both(n01, g), both(n23, g - 18));
            }
        }
        __syncwarp();
        // the rest: entries of P behind the whole chunks, then the sums
        for (int c = whole; c < nch; ++c, img += A_BYTES) {
            float h[2], l[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int64_t b = (int64_t)c * BK + 2 * lane + i, j = b - k_pad;
                h[i] = x < n_v && j < 0 ? P[x * k_pad + b] : 0.0f;
                l[i] = 0.0f;
                if (j >= 0 && j < nb) two_sum(rs[j].x, rs[j].y, h[i], l[i]);
            }
            const int g = row_grid(h[0], h[1]);
            float q = __int_as_float(g << 23), iq = __int_as_float((254 - g) << 23);
#pragma unroll
            for (int s = 0; s < NSA; ++s) {
                float r[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    r[i] = rintf(h[i] * iq) * q;
                    two_sum(h[i] - r[i], l[i], h[i], l[i]);
                }
                store(s, r[0], r[1]);
                q *= 0x1p-9f;
                iq *= 0x1p9f;
            }
        }
        double e = (double)es + (double)ec;
        for (int o = 16; o > 0; o >>= 1) {
            e += __shfl_xor_sync(0xffffffffu, e, o);
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
        }
        wrong = __any_sync(0xffffffffu, wrong) || !(sum <= 1.01f);
        if (lane == 0) {
            const float h = (float)(rint(e * 32768.0) / 32768.0);     // a multiple of 2^-15 (|e| < 129)
            ex[x] = make_float2(h, (float)(e - (double)h));
            if (wrong) atomicExch(bad, 1);
        }
        __syncwarp();
    }
}

// The slices of log2 max(P[t,b], FLT_MIN) - c, a CTA per target, a warp per
// chunk; rows past T and columns past the last are zeros.  N targets to a tile.
// cs: c of every chunk of P (shared memory).
__device__ __forceinline__ void kl_target_slices(const float *__restrict__ sP, int32_t T, int64_t k_pad, int N, int a,
                                                 uint8_t *__restrict__ B, int *cs, const Log2Tab &tab) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nb = data_chunks(k_pad), nch = all_chunks(k_pad), whole = (int)(k_pad / BK);
    uint8_t *row = B + (int64_t)(a / N) * nch * b_bytes(N) + image_at(a % N, 2 * lane);
    // log2 of this lane's entry i of chunk c, exponent and table part apart; false past the columns of P
    auto log2_at = [&](int c, int i, float2 &d) {
        const int64_t b = (int64_t)c * BK + 2 * lane + i;
        if (a >= T || b >= k_pad) return false;
        d = log2_pair(fmaxf(sP[(int64_t)a * k_pad + b], FLT_MIN), tab);
        return true;
    };
    // The chunk c with the numbers h + t (|t| within h's rounding; grid: whether an
    // entry counts for the chunk's grid, 2^-7 of the largest magnitude's power of
    // two, at least that of `least`); an entry's own BF16 grid where that is coarser
    auto slices = [&](int c, float (&h)[2], float (&t)[2], const bool (&grid)[2], float least) {
        float mag = least;
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (grid[i]) mag = fmaxf(mag, fabsf(h[i]));
        const unsigned mx = __reduce_max_sync(0xffffffffu, __float_as_uint(mag));
        int qe = max((int)(mx >> 23), 100) - 7;          // biased exponent of the grid
        uint8_t *img = row + (int64_t)c * b_bytes(N);
#pragma unroll
        for (int s = 0; s < NSB; ++s, qe -= 9) {
            __nv_bfloat16 v[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int e = max(qe, ((__float_as_int(h[i]) >> 23) & 255) - 7);
                float r = rintf(h[i] * __int_as_float((254 - e) << 23)) * __int_as_float(e << 23);
                if (s == NSB - 1) r = h[i];              // the last need not lie on a grid
                v[i] = __float2bfloat16_rn(r);
                h[i] = __fadd_rn(__fsub_rn(h[i], r), t[i]);      // h - r is exact
                t[i] = 0.f;
            }
            *reinterpret_cast<__nv_bfloat162 *>(img + s * N * ROW_B) = __nv_bfloat162(v[0], v[1]);
        }
    };
    // entries of P less c: a normalised pair (above its error of 2^-31: the slices reach 2^-18 of the grid)
    auto data = [&](int c, int ci, float (&h)[2], float (&t)[2], bool (&grid)[2]) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float2 d;
            if (log2_at(c, i, d)) {
                grid[i] = d.x >= -32.0f;
                two_sum(d.x - (float)ci, d.y, h[i], t[i]);       // d.x is a multiple of 2^-12: exact
            }
        }
    };
    for (int c = warp; c < nb; c += 8) {
        // the whole number in the middle of the logs down to -32
        int lo = INT_MAX, hi = INT_MIN;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float2 d;
            if (log2_at(c, i, d) && d.x >= -32.0f) {
                const int v = __float2int_rn(d.x);
                lo = min(lo, v);
                hi = max(hi, v);
            }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        const int ci = lo <= hi ? (lo + hi) >> 1 : 0;
        if (lane == 0) cs[c] = ci;
        if (c >= whole) continue;
        float h[2] = {0.f, 0.f}, t[2] = {0.f, 0.f};
        bool grid[2] = {false, false};
        data(c, ci, h, t, grid);
        slices(c, h, t, grid, 0.0f);
    }
    __syncthreads();
    // The rest.  A chunk that also holds c columns keeps a grid of 2^-7 or more, so
    // that their products with sums of P (a row's largest is at least 1 / nb) and
    // those of its entries still sum within 24 bits.
    for (int c = whole + warp; c < nch; c += 8) {
        float h[2] = {0.f, 0.f}, t[2] = {0.f, 0.f};
        bool grid[2] = {false, false};
        if (c < nb) data(c, cs[c], h, t, grid);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int64_t j = (int64_t)c * BK + 2 * lane + i - k_pad;
            if (j >= 0 && j < nb) h[i] = (float)cs[j];
        }
        slices(c, h, t, grid, 1.0f);
    }
}

__global__ void __launch_bounds__(256) kl_targets_kernel(const float *__restrict__ sP, int32_t T, int64_t k_pad, int N,
                                                         uint8_t *__restrict__ B) {
    __shared__ Log2Tab tab;
    extern __shared__ int cs[];
    build_log2_table(tab);
    __syncthreads();
    kl_target_slices(sP, T, k_pad, N, blockIdx.x, B, cs, tab);
}

// blockIdx.y a problem, blockIdx.x one of its targets (tiles of q.ktile)
__global__ void __launch_bounds__(256) kl_batch_targets_kernel(const BatchProblem *__restrict__ probs) {
    __shared__ Log2Tab tab;
    extern __shared__ int cs[];
    const BatchProblem &q = probs[blockIdx.y];
    if ((int)blockIdx.x >= (q.T + q.ktile - 1) / q.ktile * q.ktile) return;
    build_log2_table(tab);
    __syncthreads();
    kl_target_slices(q.sP, q.T, q.k_pad, q.ktile, blockIdx.x, q.KB, cs, tab);
}

int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

}  // namespace

// Maps from 2^20 entries of P on (a grid of about 60 cells a side): below it a
// tile pass takes a few microseconds and the slicing of the targets as much.
// A refined log2 P (dd_log_poisson_kernel) reaches far below log2 FLT_MIN,
// beyond the totals' range: its KL stays in the tile pass.
// (2^17 columns: the sums of a row's chunks, eight rows a CTA, take 128 KB of shared memory.)
bool kl_mma_wanted(const DevMesh &m) {
    return !m.LP && m.n_v * m.k_pad >= (1 << 20) && m.k_pad <= kMaxColumns;
}

int32_t kl_mma_chunks(int64_t k_pad) { return all_chunks(k_pad); }

// Target tile: wider tiles share one read of the row slices among more
// targets and use more of the MMA rate (an MMA's operand reads from shared
// memory bound N = 64 at about two thirds of it, N = 16 at a fifth), narrower
// ones waste less on padding.
int kl_mma_tile(int32_t T) { return T <= 16 ? 16 : T <= 64 ? 64 : 128; }

int kl_mma_batch_tile(int32_t T) { return T <= 64 ? 64 : 128; }

size_t kl_mma_target_bytes(int64_t k_pad, int32_t T, int N) {
    return (size_t)((T + N - 1) / N) * kl_mma_chunks(k_pad) * b_bytes(N);
}

dd_status prepare_kl_mma(DevMesh &m, cudaStream_t s, bool *usable, std::string &err) {
    *usable = m.kl_state == 1;
    if (m.kl_state != 0 || m.kl_no_room == memory_releases()) return DD_OK;
    const int32_t nch = kl_mma_chunks(m.k_pad);
    const int64_t nt = (m.n_v + BM - 1) / BM;
    const size_t abytes = (size_t)nt * nch * A_BYTES, ebytes = (size_t)nt * BM * sizeof(float2);
    uint8_t *a = nullptr, *e = nullptr;
    auto drop = [&]() {
        if (a) cudaFree(a);
        if (e) cudaFree(e);
    };
    if (cudaMalloc((void **)&a, abytes) != cudaSuccess || cudaMalloc((void **)&e, ebytes + sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        drop();
        m.kl_no_room = memory_releases();
        return DD_OK;      // no room: the FP32 tile kernels, which need none, run instead
    }
    int *bad = reinterpret_cast<int *>(e + ebytes);
    int flag = 0;
    cudaError_t ce = cudaMemsetAsync(bad, 0, sizeof(int), s);
    if (ce == cudaSuccess) {
        KMark km_("kl_rows_kernel", s);
        const int64_t blocks = std::min<int64_t>((nt * BM + 7) / 8, 8LL * sm_count());
        const int smem = 8 * data_chunks(m.k_pad) * (int)sizeof(float2);
        cudaFuncSetAttribute(kl_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        kl_rows_kernel<<<(unsigned)blocks, 256, smem, s>>>(m.P, m.n_v, nt * BM, m.k_pad, a, (float2 *)e, bad);
        ce = cudaGetLastError();
    }
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(&flag, bad, sizeof flag, cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) {
        drop();
        err = std::string("slicing P for the tensor-core KL failed: ") + cudaGetErrorString(ce);
        return DD_ECUDA;
    }
    if (flag) {
        drop();
        m.kl_state = -1;
        return DD_OK;
    }
    m.kl_a = a;
    m.kl_ex = (float2 *)e;
    m.kl_state = 1;
    m.owned.push_back(a);
    m.owned.push_back(e);
    m.bytes += (int64_t)(abytes + ebytes);
    *usable = true;
    return DD_OK;
}

size_t kl_mma_row_bytes(const DevMesh &m) {
    return (size_t)((m.n_v + BM - 1) / BM) * kl_mma_chunks(m.k_pad) * A_BYTES;
}
size_t kl_mma_ex_bytes(const DevMesh &m) { return (size_t)((m.n_v + BM - 1) / BM) * BM * sizeof(float2); }

void launch_kl_mma(const KlMmaArgs &ka, const float *sP, int64_t n_v, int64_t k_pad, int32_t T, float *out_kl,
                   int *err, cudaStream_t s) {
    const int N = kl_mma_tile(T);
    const int32_t nch = kl_mma_chunks(k_pad);
    const int nat = (T + N - 1) / N;
    {
        KMark km_("kl_targets_kernel", s);
        kl_targets_kernel<<<(unsigned)(nat * N), 256, data_chunks(k_pad) * sizeof(int), s>>>(sP, T, k_pad, N, ka.B);
    }
    const KlOne one{ka.A, ka.B, ka.ex, out_kl, n_v, T, nch};
    const int64_t n_items = (n_v + BM - 1) / BM * nat;
    const unsigned grid = (unsigned)std::min<int64_t>(n_items, sm_count());
    auto go = [&](auto kern, int smem) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        KMark km_("kl_mma_kernel", s);
        kern<<<grid, 320, smem, s>>>(one, nullptr, nullptr, (int32_t)n_items, err);
    };
    if (N == 16)
        go(kl_mma_kernel<16, false>, smem_bytes(16));
    else if (N == 64)
        go(kl_mma_kernel<64, false>, smem_bytes(64));
    else
        go(kl_mma_kernel<128, false>, smem_bytes(128));
}

void launch_batch_kl_mma(const BatchProblem *d_probs, int32_t n_probs, const BatchKlMma &b, cudaStream_t s) {
    {
        KMark km_("kl_targets_kernel", s);
        kl_batch_targets_kernel<<<dim3((unsigned)((b.max_T + 127) / 128 * 128), (unsigned)n_probs), 256,
                                  data_chunks(b.max_k) * sizeof(int), s>>>(d_probs);
    }
    auto go = [&](auto kern, int smem, const BatchItem *items, int32_t n) {
        if (n <= 0) return;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        KMark km_("kl_mma_kernel", s);
        kern<<<(unsigned)std::min<int64_t>(n, sm_count()), 320, smem, s>>>(KlOne{}, d_probs, items, n, b.err);
    };
    go(kl_mma_kernel<128, true>, smem_bytes(128), b.items, b.n_wide);
    go(kl_mma_kernel<64, true>, smem_bytes(64), b.items + b.n_wide, b.n_items - b.n_wide);
}
