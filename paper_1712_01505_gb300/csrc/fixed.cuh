// Fixed-point arithmetic of the FP64 hopping stencil (wilson_fx.cu).
//
// GB300 issues 1.7 FP64 instructions per SM and clock, but 32 integer
// multiply-adds 32 x 32 + 64 -> 64 and 128 FP32 multiply-adds (measured), so the
// link products of the FP64 stencil run as integers with an FP32 remainder:
//
//   link element  U  =  (ah + al) 2^-30,            ah integer, al FP32, |al| <= 1/2
//   spinor        x  =  (xh + xl) 2^(e - 1052),     xh integer, xl FP32
//
// where e is the exponent field of the site's largest |component| (which lies in
// [2^(e - 1023), 2^(e - 1022))), so |xh| < 2^30; a double of exponent e splits without
// rounding, and smaller ones to within 1.5 2^-56 of 2^(e - 1022) (the shift drops less than 2^-57,
// the FP32 remainder of 26 bits is rounded by at most 2^-56; what is not zero stays so).
// Half spinors h = u +- B l are formed part by part (|hh| < 2^31), and
//
//   sum a h = HH + C,  HH = sum ah hh (64-bit, exact),  C = sum (ah hl + al hh) (FP32),
//
// one integer multiply-add and two FP32 ones per real product (the sum of six al hl is
// below 6, less than one unit of the last place kept, which is 8).  HH / 8 and C / 8, rounded to nearest,
// are added into 64-bit sums aligned to the largest e of the eight neighbours, E; their unit is 2^(E - 1079).
// Measured against 80-bit arithmetic (tests/test_fixed_point.py), the sum of the
// eight hops is closer to the exact one than FP64 multiply-adds: relative error
// 1.0e-16 against 1.5e-16, the same for fields whose sites differ by orders of
// magnitude.
//
// That is an error of 11 units (rms, nearly all of it the FP32 roundings of C) whatever the component is, 4 with one
// neighbour only, where FP64's is measured by the component's own products.  So a component counts as computed only
// where S = sum |U| |h|, the magnitudes of its products over the eight hops, shows that the error is small beside it:
// S >= 2^(E - 1022) / 16 with one neighbour that outweighs the rest, / 8 with several (kSumMin, sum_min); FP64 computes
// the sites with a component below (wilson_fx.cu).  That leaves at most 5.4 2^-53 S (rms; a chain of FP64 multiply-adds is
// certain to 16 2^-53 S).  Gaussian fields have S = 4.6 2^(E - 1022), and 0.15 2^-53 S here against 0.29 in FP64.
//
// Bounds: with rows of U of 2-norm <= 5/4, |HH| <= 5/4 2^30 sqrt(6) 2^31 < 2^62.7 (with the half that rounds it, at most
// 2^60, below 2^63), |C| <= 5/4 sqrt(6) 2^30 + 6 2^31 / 2 < 2^33.3 (|hl| <= 1, |al| <= 1/2), and the sum of eight hops < 2^62.7.
#pragma once
#include <stdint.h>
#include <string.h>

#include <cmath>

#if defined(__CUDACC__)
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN inline
#endif

namespace qcd {
namespace fx {

// exponent fields (of the largest component) that the fixed-point path takes; sites below kEmin and
// above kEmax (infinities and NaN included) are stored as FP64 with the field kBad; kZero: all components are zero
constexpr int kEmin = 256, kEmax = 1982, kZero = kEmin - 1, kBad = 0x7000;
// HH and C are divided by 2^d, d = E - e + 3; from this d on a neighbour is left out (|HH| / 2^d < 1.6 units)
constexpr int kFar = 62;
// what the magnitudes of a component's products have to add up to, in units of HH where e = E (2^60 is
// 2^(E - 1022)): this times the sum of the neighbours' sizes relative to the largest one's, at most 2
constexpr float kSumMin = 0x1p56f;
// 2-norms of link rows and columns that it takes
constexpr double kNormMax = 1.25, kNormMin = 0.5;

struct Part {
  int h;
  float l;
};

FX_FN uint64_t shr64(uint64_t v, unsigned n) {  // 0 for n >= 64
#if defined(__CUDA_ARCH__)
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return n < 64 ? v >> n : 0;
#endif
}

FX_FN float pow2f(int n) {  // 2^n, -126 <= n <= 127
  const unsigned b = (unsigned)(n + 127) << 23;
  float f;
  memcpy(&f, &b, 4);
  return f;
}

// a link element
FX_FN Part link_part(double v) {
  const double a = v * 0x1p30, r = rint(a);
  return {(int)r, (float)(a - r)};
}

// a double given as its words, aligned to the exponent field e >= its own
FX_FN Part spinor_part(unsigned hi, unsigned lo, int e) {
  const unsigned d = (((unsigned)e << 20 | 0xfffffu) - (hi & 0x7fffffffu)) >> 20;  // e - exponent field
  const unsigned m = (hi & 0xfffffu) | 0x100000u;
  const uint64_t p = shr64(((uint64_t)m << 36) | ((uint64_t)lo << 4), d);  // |v| 2^(1079 - e), 57 bits
  int h = (int)(p >> 27), l = (int)(p & 0x7ffffffu);
  l |= (p == 0) & (((hi << 1) | lo) != 0);  // not zero: the last unit
  const int up = (l >> 26) & (h != 0x3fffffff);  // round h to nearest, but keep it below 2^30
  h += up;
  l -= up << 27;
  const int s = (int)hi >> 31;
  return {(h ^ s) - s, (float)((l ^ s) - s) * 0x1p-27f};
}

// (H + C) / 2^d rounded, 3 <= d < kFar; H holds hop_half besides, sc = 2^-d.  Ties of H (one in eight at d = 3) go up in
// the forward hops and down in the backward ones, so that the eight together have no bias.
FX_FN int64_t hop_half(int d, int back) { return ((int64_t)1 << (d - 1)) - back; }
FX_FN int64_t hop_round(int64_t H, float C, float sc, int d) {
#if defined(__CUDA_ARCH__)
  return (H >> d) + (int64_t)__float2int_rn(C * sc);
#else
  return (H >> d) + (int64_t)lrintf(C * sc);
#endif
}
// the least sum of magnitudes for neighbours whose sizes relative to the largest one's add up to `size` (1 to 8)
FX_FN float sum_min(float size) { return size < 2.f ? kSumMin * size : kSumMin * 2.f; }

// the value of a part as a double; e as in spinor_part
FX_FN double part_value(const Part& p, int e) { return ldexp((double)p.h + (double)p.l, e - 1052); }

// A sum w = (h + l) 2^shift, |w| <= 2^(30 + shift), shift <= 33, as a part with |h| < 2^30
FX_FN Part sum_part(int64_t w, int shift) {
  if (shift <= 0) {
    const int h = (int)((uint64_t)w << -shift);
    return h == -0x40000000 ? Part{h + 1, -1.f} : Part{h, 0.f};
  }
  int h = (int)(w >> shift);
  int64_t rem = w - ((int64_t)h << shift);  // in [0, 2^shift)
  if ((rem > ((int64_t)1 << (shift - 1)) || h == -0x40000000) && h != 0x3fffffff) {
    h += 1;
    rem -= (int64_t)1 << shift;
  }
  const int t = shift > 30 ? shift - 30 : 0;
  const float l = (float)(int)(rem >> t) * pow2f(t - shift);
  return {h, l};
}

}  // namespace fx
}  // namespace qcd
