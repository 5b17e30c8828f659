// Column passes of the site-local domain-wall blocks (see dwf.cu for the
// operators): on one (site, colour, spin) column of Ls values, d + e T and
// (alpha - beta T)^-1 with T the twisted lower (P_+ spins) or upper (P_- spins)
// shift of the fifth dimension (factor -m across the wall); the adjoint
// exchanges the shifts.  Shared by the standalone column kernel (dwf.cu) and
// the epilogue of the fused stencil (dwf_hop.cu).
#pragma once
#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace qcd {
namespace dwcol {

constexpr int kMaxLs = 64;

// A column operator out = post . inv . pre (in) on the (s, spin) columns, every
// factor optional: pre and post are d + e S, inv is (alpha - beta S)^-1.  The
// adjoint applies post^T, inv^T, pre^T in that order.  Coefficients in the
// kernel's arithmetic type (no FP64 in the FP32 kernels).
enum { kPre = 1, kInv = 2, kPost = 4 };

template <typename R>
struct ColCoef {
  int Ls, flags;
  R mf;
  R pre_d, pre_e, post_d, post_e;
  R ainv, ratio;   // 1 / alpha, beta / alpha
  R apow[kMaxLs];  // beta^k alpha^(-1-k) / den
  R row0[kMaxLs];  // alpha times row 0 of the inverse: 1 / den, then -m beta^k alpha^-k / den, k = Ls - t
};

// (d + e T) in place on one column of Ls complex values (stride cs), T = T_lo or T_up
template <typename R>
__device__ __forceinline__ void col_mul(R* re, R* im, int cs, int Ls, bool lower, R d, R e, R mf) {
  const R ew = -mf * e;
  if (lower) {
    const R lr = re[(Ls - 1) * cs], li = im[(Ls - 1) * cs];
    for (int s = Ls - 1; s >= 1; --s) {
      re[s * cs] = fma(e, re[(s - 1) * cs], d * re[s * cs]);
      im[s * cs] = fma(e, im[(s - 1) * cs], d * im[s * cs]);
    }
    re[0] = fma(ew, lr, d * re[0]);
    im[0] = fma(ew, li, d * im[0]);
  } else {
    const R fr = re[0], fi = im[0];
    for (int s = 0; s < Ls - 1; ++s) {
      re[s * cs] = fma(e, re[(s + 1) * cs], d * re[s * cs]);
      im[s * cs] = fma(e, im[(s + 1) * cs], d * im[s * cs]);
    }
    re[(Ls - 1) * cs] = fma(ew, fr, d * re[(Ls - 1) * cs]);
    im[(Ls - 1) * cs] = fma(ew, fi, d * im[(Ls - 1) * cs]);
  }
}

// (alpha - beta T)^-1 in place on one column: the end slice from the closed form,
// the others by substitution psi_s = chi_s / alpha + (beta / alpha) psi_{s-+1}
template <typename R>
__device__ __forceinline__ void col_inv(R* re, R* im, int cs, const ColCoef<R>& c, bool lower) {
  const int Ls = c.Ls;
  if (lower) {
    R pr = c.apow[0] * re[0], pi = c.apow[0] * im[0];
    for (int sp = 1; sp < Ls; ++sp) {
      const R w = -c.mf * c.apow[Ls - sp];
      pr = fma(w, re[sp * cs], pr);
      pi = fma(w, im[sp * cs], pi);
    }
    re[0] = pr;
    im[0] = pi;
    for (int s = 1; s < Ls; ++s) {
      pr = fma(c.ratio, pr, c.ainv * re[s * cs]);
      pi = fma(c.ratio, pi, c.ainv * im[s * cs]);
      re[s * cs] = pr;
      im[s * cs] = pi;
    }
  } else {
    const int l = Ls - 1;
    R pr = c.apow[0] * re[l * cs], pi = c.apow[0] * im[l * cs];
    for (int sp = 0; sp < l; ++sp) {
      const R w = -c.mf * c.apow[sp + 1];
      pr = fma(w, re[sp * cs], pr);
      pi = fma(w, im[sp * cs], pi);
    }
    re[l * cs] = pr;
    im[l * cs] = pi;
    for (int s = l - 1; s >= 0; --s) {
      pr = fma(c.ratio, pr, c.ainv * re[s * cs]);
      pi = fma(c.ratio, pi, c.ainv * im[s * cs]);
      re[s * cs] = pr;
      im[s * cs] = pi;
    }
  }
}

// The same with the column held in registers (Ls <= NR): one read and one write of
// the column instead of two reads and a write (the fused stencil's shared-memory tile)
template <int NR, typename R>
__device__ __forceinline__ void col_inv_reg(R* re, R* im, int cs, const ColCoef<R>& c, bool lower) {
  const int Ls = c.Ls;
  R vr[NR], vi[NR];
#pragma unroll
  for (int s = 0; s < NR; ++s)
    if (s < Ls) {
      vr[s] = re[s * cs];
      vi[s] = im[s * cs];
    }
  if (lower) {
    R pr = c.apow[0] * vr[0], pi = c.apow[0] * vi[0];
#pragma unroll
    for (int sp = 1; sp < NR; ++sp)
      if (sp < Ls) {
        const R w = -c.mf * c.apow[Ls - sp];
        pr = fma(w, vr[sp], pr);
        pi = fma(w, vi[sp], pi);
      }
    re[0] = pr;
    im[0] = pi;
#pragma unroll
    for (int s = 1; s < NR; ++s)
      if (s < Ls) {
        pr = fma(c.ratio, pr, c.ainv * vr[s]);
        pi = fma(c.ratio, pi, c.ainv * vi[s]);
        re[s * cs] = pr;
        im[s * cs] = pi;
      }
  } else {
    const int l = Ls - 1;
    R pr = 0, pi = 0;
#pragma unroll
    for (int sp = 0; sp < NR; ++sp)
      if (sp == l) {
        pr = c.apow[0] * vr[sp];
        pi = c.apow[0] * vi[sp];
      }
#pragma unroll
    for (int sp = 0; sp < NR; ++sp)
      if (sp < l) {
        const R w = -c.mf * c.apow[sp + 1];
        pr = fma(w, vr[sp], pr);
        pi = fma(w, vi[sp], pi);
      }
    // psi_l, then psi_s = chi_s / alpha + (beta / alpha) psi_{s+1} downwards
#pragma unroll
    for (int s = NR - 1; s >= 0; --s) {
      if (s > l) continue;
      if (s < l) {
        pr = fma(c.ratio, pr, c.ainv * vr[s]);
        pi = fma(c.ratio, pi, c.ainv * vi[s]);
      }
      re[s * cs] = pr;
      im[s * cs] = pi;
    }
  }
}

// ----------------------------------------------------------------------------- columns in registers
// The passes of a column operator on several columns of one chirality at once, held in registers from the
// first slice to the last (Ls <= NR): V is a spin pair of FP32 (complex, or its real or imaginary parts
// alone) or a complex FP64.  In the order t = s (lower shift) or Ls - 1 - s (upper) both shifts are the same recurrence:
//   (d + e T): v_t = d x_t + e x_(t-1), x_(-1) = -m x_(Ls-1);
//   (alpha - beta T)^-1: alpha psi_0 = row0 . x, alpha psi_t = x_t + (beta / alpha) (alpha psi_(t-1)),
// two multiply-adds per value; the factor 1 / alpha is left to the caller (unit(), in its own scale factor).
__device__ __forceinline__ P2 vfma(float a, const P2& x, const P2& y) {
  const float2 b = make_float2(a, a);
  return {__ffma2_rn(b, x.re, y.re), __ffma2_rn(b, x.im, y.im)};
}
__device__ __forceinline__ P2 vmul(float a, const P2& x) {
  const float2 b = make_float2(a, a);
  return {__fmul2_rn(b, x.re), __fmul2_rn(b, x.im)};
}
__device__ __forceinline__ float2 vfma(float a, float2 x, float2 y) { return __ffma2_rn(make_float2(a, a), x, y); }
__device__ __forceinline__ float2 vmul(float a, float2 x) { return __fmul2_rn(make_float2(a, a), x); }
__device__ __forceinline__ Cx<double> vfma(double a, const Cx<double>& x, const Cx<double>& y) {
  return {fma(a, x.re, y.re), fma(a, x.im, y.im)};
}
__device__ __forceinline__ Cx<double> vmul(double a, const Cx<double>& x) { return {a * x.re, a * x.im}; }

// v[t], t < Ls, in the order above; last = v[Ls - 1]
template <int NR, typename R, typename V>
__device__ __forceinline__ void col_reg(V (&v)[NR], V last, const ColCoef<R>& c, int dagger) {
  const int Ls = c.Ls;
  const bool first = dagger ? (c.flags & kPost) : (c.flags & kPre);
  const bool then = dagger ? (c.flags & kPre) : (c.flags & kPost);
  if (first) {
    const R d = dagger ? c.post_d : c.pre_d, e = dagger ? c.post_e : c.pre_e;
    V prev = vmul(-c.mf, last);
#pragma unroll
    for (int t = 0; t < NR; ++t)
      if (t < Ls) {
        const V x = v[t];
        last = v[t] = vfma(e, prev, vmul(d, x));
        prev = x;
      }
  }
  if (c.flags & kInv) {
    V p = vmul(c.row0[0], v[0]);
#pragma unroll
    for (int t = 1; t < NR; ++t)
      if (t < Ls) p = vfma(c.row0[t], v[t], p);
    v[0] = p;
#pragma unroll
    for (int t = 1; t < NR; ++t)
      if (t < Ls) {
        p = vfma(c.ratio, p, v[t]);
        v[t] = p;
      }
    last = p;
  }
  if (then) {
    const R d = dagger ? c.pre_d : c.post_d, e = dagger ? c.pre_e : c.post_e;
    V prev = vmul(-c.mf, last);
#pragma unroll
    for (int t = 0; t < NR; ++t)
      if (t < Ls) {
        const V x = v[t];
        v[t] = vfma(e, prev, vmul(d, x));
        prev = x;
      }
  }
}
// the factor that col_reg leaves out
template <typename R>
__device__ __forceinline__ R col_unit(const ColCoef<R>& c) {
  return (c.flags & kInv) ? c.ainv : R(1);
}

// host description of a column operator
struct ColSpec {
  int flags = 0;
  double pre_d = 1, pre_e = 0, post_d = 1, post_e = 0;
  double alpha = 1, beta = 0;  // inverse of alpha - beta S
};

template <typename R>
inline ColCoef<R> make_coef(const DwParams& p, const ColSpec& cs) {
  ColCoef<R> c;
  c.Ls = p.Ls;
  c.flags = cs.flags;
  c.mf = (R)p.mf;
  c.pre_d = (R)cs.pre_d;
  c.pre_e = (R)cs.pre_e;
  c.post_d = (R)cs.post_d;
  c.post_e = (R)cs.post_e;
  const double ratio = cs.beta / cs.alpha;
  const double den = 1.0 + p.mf * std::pow(ratio, p.Ls);
  c.ainv = (R)(1.0 / cs.alpha);
  c.ratio = (R)ratio;
  double w = 1.0 / (cs.alpha * den);
  for (int k = 0; k < p.Ls; ++k) {
    c.apow[k] = (R)w;
    if (k)
      c.row0[p.Ls - k] = (R)(-p.mf * w * cs.alpha);
    else
      c.row0[0] = (R)(w * cs.alpha);
    w *= ratio;
  }
  return c;
}

// W = B A^-1 (A^-1 for Shamir); the adjoint order is handled by the kernels
inline ColSpec w_spec(const DwParams& p) {
  ColSpec cs;
  cs.flags = kInv | (p.mobius() ? kPost : 0);
  cs.alpha = p.alpha();
  cs.beta = p.beta();
  cs.post_d = p.b5;
  cs.post_e = p.c5;
  return cs;
}

// the passes of a column operator (dagger: post^T, inv^T, pre^T) on one complex column;
// NR > 0: the inverse with the column in registers (needs Ls <= NR)
template <typename R, int NR = 0>
__device__ __forceinline__ void col_apply(R* re, R* im, int cs, const ColCoef<R>& c, bool lower, int dagger) {
  const bool first = dagger ? (c.flags & kPost) : (c.flags & kPre);
  const bool last = dagger ? (c.flags & kPre) : (c.flags & kPost);
  if (first) col_mul(re, im, cs, c.Ls, lower, dagger ? c.post_d : c.pre_d, dagger ? c.post_e : c.pre_e, c.mf);
  if (c.flags & kInv) {
    if constexpr (NR > 0)
      col_inv_reg<NR>(re, im, cs, c, lower);
    else
      col_inv(re, im, cs, c, lower);
  }
  if (last) col_mul(re, im, cs, c.Ls, lower, dagger ? c.pre_d : c.post_d, dagger ? c.pre_e : c.post_e, c.mf);
}

}  // namespace dwcol
}  // namespace qcd
