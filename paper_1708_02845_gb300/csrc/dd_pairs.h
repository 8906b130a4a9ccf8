// Numbers of the V-cycle: unevaluated sums of two floats (dd_pcg.cu; the host's
// check of it in dd_amg.cpp).  Host and device.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define DD_BOTH __host__ __device__ __forceinline__
#else
#define DD_BOTH inline
#endif

namespace {

template <typename To, typename From>
DD_BOTH To bits_as(From v) {
    static_assert(sizeof(To) == sizeof(From), "size");
    To r;
    memcpy(&r, &v, sizeof r);
    return r;
}

// The exponents that a column's numbers gain on their way into the V-cycle and
// lose on their way out (df_split, widen).  The residual's norm then lies
// near 2^60: a factor 2^-150 below it is kept and one of 2^58 above it fits,
// whatever the size of the column's right-hand side and however far the column
// has converged.
constexpr int kShiftTop = 60, kShiftMin = -452, kShiftMax = 572;
// from the squared norm (0, subnormal and infinite numbers included)
DD_BOTH int shift_of_square(double rr) {
    return kShiftTop - (((int)(bits_as<uint64_t>(rr) >> 52 & 0x7ff) - 1023) >> 1);
}
// from the largest biased exponent of the entries
DD_BOTH int shift_of_top(int top) {
    const int s = kShiftTop + 1023 - top;
    return s < kShiftMin ? kShiftMin : (s > kShiftMax ? kShiftMax : s);
}

// A double times 2^shift as an unevaluated sum of two floats, by integer
// operations on its bits (this part converts FP64 no faster than it multiplies
// it): the leading 24 bits of the significand, and the 29 that follow as an
// integer scaled.  Magnitudes outside 2^-90 .. 2^120 come out as 0 or as 2^120:
// the column's exponent (shift_of_square) keeps what matters between them.  A
// residual is relative to its own right-hand side, which may be 1e-17 (a
// corner that meets the interior by a right-angled cell's diagonal alone,
// rotated) or far above 1, and falls by 1e-15 and more; without the shift
// such columns stopped at 1e-9 of theirs.
DD_BOTH void df_split(double d, int shift, float &hi, float &lo) {
    const uint64_t u = bits_as<uint64_t>(d);
    const uint32_t sign = (uint32_t)(u >> 32) & 0x80000000u;
    const int e = (int)(u >> 52 & 0x7ff) - 1023 + shift;
    const int ec = e < 120 ? e : 120;
    const uint32_t top = (uint32_t)(u >> 29) & 0x7fffffu;
    const float l = (float)(int)((uint32_t)u & 0x1fffffffu);                   // < 2^29
    const float scale = bits_as<float>((uint32_t)(ec - 29 + 127) << 23);       // 2^(e - 29); times 2^-23 below
    const bool tiny = e < -90;
    hi = tiny ? 0.0f : bits_as<float>(sign | ((uint32_t)(ec + 127) << 23) | top);
    lo = tiny ? 0.0f : bits_as<float>(sign ^ bits_as<uint32_t>(l * scale * 0x1p-23f));
}
// float times 2^-shift to double by its bits (subnormals as 0)
DD_BOTH double widen(float f, int shift) {
    const uint32_t u = bits_as<uint32_t>(f);
    const uint32_t m = u & 0x7fffffffu;
    const uint32_t h = m < 0x00800000u ? 0u : (m >> 3) + ((uint32_t)(896 - shift) << 20);
    return bits_as<double>((uint64_t)((u & 0x80000000u) | h) << 32 | (m < 0x00800000u ? 0u : m << 29));
}

}  // namespace
