// Matrix-vector arithmetic of the Riccati passes.
//
// FP32: plain fused multiply-adds.
//
// FP64: exact integer sums of fixed-point products.  GB300 issues 1.9 FP64
// fused multiply-adds per clock and SM (a 64-cycle slot of its sub-partition
// per warp instruction, 67 cycles of latency) but 56 wide integer ones
// (32 x 32 + 64 bits, 4 cycles), measured.  A factor matrix is stored, in the
// same 8 bytes per entry as a double, as a 57-bit signed integer relative to
// a power of two 2^ea above the largest entry of the same output's sum:
//   a = (a1 2^28 + a0) 2^(ea - 56),  |a1| <= 2^28, |a0| <= 2^27;
// a vector is rounded once to 84 bits relative to a power of two 2^ex above
// its largest entry:
//   x = (x2 2^56 + x1 2^28 + x0) 2^(ex - 83),  |x2|, |x1|, |x0| <= 2^27 (+ 1).
// A product then takes five wide multiply-adds into three 64-bit sums (the
// sixth, a0 x0, is below 2^-78 of the largest term and is left out); sums of
// up to 128 products fit without a check, as |a1 x1 + a0 x2| <= 1.5 * 2^55.
// The sums are exact and do not depend on the order; the result is rounded
// once, to the nearest double.  What is rounded is the stored factor (at most
// 2^-57 of 2^ea, against 2^-54 of the entry itself in a double) and the
// vector (2^-83), so the error of a sum is below that of the same sum in
// FP64 arithmetic unless the terms are far below the largest ones; the
// largest entry is taken per output (matrix) and per vector for that reason.
// Five integer instructions per entry against one in FP64: 6.4 x the rate.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace spock {

constexpr int kFxBits = 28;               // bits per limb
constexpr int kFxNonFinite = 1 << 20;     // exponent of a vector with an infinity or a NaN

template <typename S>
struct Fx;

template <>
struct Fx<float> {
  using Mat = float;    // stored matrix entry
  using Vec = float;    // entry of a vector prepared for products
  struct Acc {
    float v;
  };
  static __device__ __forceinline__ void zero(Acc& a) { a.v = 0.f; }
  static __device__ __forceinline__ void mad(Acc& a, float m, float x) { a.v = fmaf(m, x, a.v); }
  static __device__ __forceinline__ void add(Acc& a, const Acc& b) { a.v += b.v; }
  static __device__ __forceinline__ float value(const Acc& a, int) { return a.v; }
  // bits of the largest entry (see vec_exp) and the prepared entry
  static __device__ __forceinline__ uint32_t key(float) { return 0u; }
  static __device__ __forceinline__ int vec_exp(uint32_t) { return 0; }
  static __device__ __forceinline__ float vec(float x, uint32_t) { return x; }
};

template <>
struct Fx<double> {
  using Mat = int2;     // (a1, a0)
  using Vec = int4;     // (x2, x1, x0, unused)
  struct Acc {
    long long h, m, l;  // sums of a1 x2; a1 x1 + a0 x2; a1 x0 + a0 x1
  };
  static __device__ __forceinline__ void zero(Acc& a) { a.h = a.m = a.l = 0; }
  static __device__ __forceinline__ void madw(long long& s, int a, int b) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s) : "r"(a), "r"(b));
  }
  static __device__ __forceinline__ void mad(Acc& s, int2 a, int4 x) {
    madw(s.h, a.x, x.x);
    madw(s.m, a.x, x.y);
    madw(s.l, a.x, x.z);
    madw(s.m, a.y, x.x);
    madw(s.l, a.y, x.y);
  }
  static __device__ __forceinline__ void add(Acc& a, const Acc& b) {
    a.h += b.h;
    a.m += b.m;
    a.l += b.l;
  }
  // (h 2^56 + m 2^28 + l) 2^(ea + ex - 111), rounded to the nearest double by
  // integer arithmetic; e = ea + ex.
  static __device__ __forceinline__ double value(const Acc& s, int e) {
    const long long m = s.m + (s.l >> kFxBits);
    const long long h = s.h + (m >> kFxBits);
    uint32_t r = (uint32_t)m << (32 - kFxBits);   // fraction of h, top-aligned in 32 bits
    uint64_t H = (uint64_t)h;
    const uint32_t sign = (uint32_t)(H >> 63);
    if (sign) {
      r = 0u - r;
      H = ~H + (r == 0u ? 1u : 0u);
    }
    int k = e - 55;
    if (H == 0) {
      H = (uint64_t)r << 32;
      r = 0;
      k -= 64;
    }
    if (H == 0 && e < kFxNonFinite / 2) return 0.0;
    const int lz = __clzll((long long)H);
    const uint64_t top = (H << lz) | (((uint64_t)r << 32) >> 1 >> (63 - lz));   // lz = 0: r is shifted out
    const uint64_t mant = (top >> 11) + ((top >> 10) & 1u);
    const int be = 1023 + 63 - lz + k;
    if (be >= 1 && be <= 2045) {
      const uint64_t bits = ((uint64_t)(uint32_t)(be - 1) << 52) + mant;
      return __longlong_as_double((long long)(bits | ((uint64_t)sign << 63)));
    }
    if (e >= kFxNonFinite / 2) return __longlong_as_double(0x7ff8000000000000ll);
    const double v = scalbn((double)mant, be - 1075);   // overflow and denormal results
    return sign ? -v : v;
  }
  // Biased exponent (at least 1) of |x|; the largest over the vector's entries
  // is what vec_exp and vec take.
  static __device__ __forceinline__ uint32_t key(double x) {
    const uint32_t e = ((uint32_t)__double2hiint(x) >> 20) & 0x7ffu;
    return e > 1u ? e : 1u;
  }
  static __device__ __forceinline__ int vec_exp(uint32_t kmax) {
    return kmax == 0x7ffu ? kFxNonFinite : (int)kmax - 1022;
  }
  static __device__ __forceinline__ int4 vec(double x, uint32_t kmax) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 0x7ffu;
    const uint32_t mh = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
    const uint32_t d = kmax - (e ? e : 1u);
    // |x| 2^83 / 2^ex = (mantissa << 30) >> d in 96 bits
    uint32_t w0 = lo << 30, w1 = (mh << 30) | (lo >> 2), w2 = mh >> 2;
    if (d & 64u) {
      w0 = w2;
      w1 = w2 = 0;
    }
    if (d & 32u) {
      w0 = w1;
      w1 = w2;
      w2 = 0;
    }
    w0 = __funnelshift_r(w0, w1, d & 31u);
    w1 = __funnelshift_r(w1, w2, d & 31u);
    w2 >>= (d & 31u);
    if (d >= 96u) w0 = w1 = w2 = 0;
    constexpr int kMask = (1 << kFxBits) - 1, kHalf = 1 << (kFxBits - 1);
    int x0 = (int)(w0 & kMask);
    int x1 = (int)(__funnelshift_r(w0, w1, 28) & kMask);
    int x2 = (int)__funnelshift_r(w1, w2, 24);
    if (x0 >= kHalf) {
      x0 -= kMask + 1;
      x1 += 1;
    }
    if (x1 >= kHalf) {
      x1 -= kMask + 1;
      x2 += 1;
    }
    if (hi >> 31) {
      x0 = -x0;
      x1 = -x1;
      x2 = -x2;
    }
    return make_int4(x2, x1, x0, 0);
  }
};

}  // namespace spock
