// The FP64 Wilson hopping stencil with its link products in fixed point
// (fixed.cuh): the same operation and storage as the FP64 kernels of wilson.cu,
//
//   out(x) = [x(x) +] a * sum_mu [ (1 - gamma_mu) U_mu(x) in(x+mu)
//                                + (1 + gamma_mu) U_mu(x-mu)^dag in(x-mu) ]
//
// The input is first rewritten as fixed-point parts with one exponent per site (k_to_fx), the links
// are kept that way from the loading of the gauge field, and only the final sum goes through the
// FP64 pipe: 24 conversions and 24 multiply-adds per site instead of 864.  Sites whose components the parts do not
// hold as well as FP64 would are computed in FP64 (fx_sum, fx_careful).  Measured at 32^3 x 64:
// FP64 kernel 1.56 ms (FP64 pipe), here 0.318 ms, 5.3 TB/s = 78% of the copy rate (links 1152 B, input 196 B, x and output
// 192 B each per site; HBM and issue slots), and 0.056 ms for k_to_fx (HBM); 16^3 x 32 x 16 slices 1.56 -> 0.36 ms with
// the conversion (issue slots).  Forms that were slower than 0.315 ms, all without the sums of magnitudes: the conversion
// inside the stencil (8 times per site: 0.555 ms), three integer products per real one instead of one and two FP32
// ones (0.355 ms, the integer multiply pipe), one thread per site (0.333 ms at 168 registers, 12 warps per SM).
#include <cstdio>
#include <vector>

#include "common.cuh"
#include "fixed.cuh"
#include "internal.h"
#include "stencil.cuh"

namespace qcd {

namespace {

using namespace stencil;
using namespace fx;

using HA = HopArgs<P64, 18>;

// Layouts.  Links: the matrices of all eight hops of a site, W[2 mu] = U_mu(x) and
// W[2 mu + 1] = U_mu(x - mu)^dag, as [parity][block of 16 sites][hop][element][16] (each link is stored
// for both of its ends: a half-dslash reads as many bytes as from one copy, contiguously and with
// no transposition).  Spinors: [slice][block of 16 sites][component][16] and one exponent field per
// site.  A unit is int4 (re.h, re.l, im.h, im.l).  A site of exponent field kBad holds its FP64 values.
constexpr int kSB = 16;  // sites per block of the layouts
constexpr int kHopUnits = 9 * kSB, kSiteUnits = 12 * kSB;

struct FxField {
  int4* __restrict__ p;
  int* __restrict__ e;
  long nsb;  // blocks of kSB sites per slice
};

// the exponent field of a site's 12 components (words of doubles); kBad out of range
__device__ __forceinline__ int fx_field_of(unsigned mx, unsigned low) {
  const int e = (int)(mx >> 20);
  if (mx == 0) return low ? kBad : kZero;  // subnormals below 2^-1042 / all zero
  return e < kEmin || e > kEmax ? kBad : e;
}
template <int N>
__device__ __forceinline__ unsigned max_word(const int4 (&w)[N]) {
  unsigned mx = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) mx = max(mx, max((unsigned)w[k].y & 0x7fffffffu, (unsigned)w[k].w & 0x7fffffffu));
  return mx;
}
template <int N>
__device__ __forceinline__ unsigned low_words(const int4 (&w)[N]) {
  unsigned low = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) low |= (unsigned)(w[k].x | w[k].z);
  return low;
}
__device__ __forceinline__ int fx_exponent(const int4 (&w)[12]) { return fx_field_of(max_word(w), low_words(w)); }
// of a site whose components are in the lanes sp = 0, 1 (six each)
__device__ __forceinline__ int fx_exponent_pair(const int4 (&w)[6]) {
  unsigned mx = max_word(w), low = low_words(w);
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, kSB));
  low |= __shfl_xor_sync(0xffffffffu, low, kSB);
  return fx_field_of(mx, low);
}

// store a site's 12 components (words of doubles); blk0: the slice's first block
__device__ __forceinline__ void fx_put(const int4 (&w)[12], int e, const FxField& out, long blk0, int cb) {
  const long blk = blk0 + cb / kSB;
  int4* o = out.p + blk * kSiteUnits + cb % kSB;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    int4 u = w[k];
    if (e != kBad) {
      const Part re = spinor_part(w[k].y, w[k].x, e), im = spinor_part(w[k].w, w[k].z, e);
      u = make_int4(re.h, __float_as_int(re.l), im.h, __float_as_int(im.l));
    }
    o[k * kSB] = u;
  }
  out.e[blk * kSB + cb % kSB] = e;
}

// FP64 -> fixed point: one thread per site, blockIdx.y: (right-hand side, slice)
__global__ void __launch_bounds__(128) k_to_fx(const int4* __restrict__ in, long stride, FxField out, int Vh, int ls,
                                               const int* stop) {
  pdl_enter();
  if (stop && *stop) return;
  const int cb = blockIdx.x * blockDim.x + threadIdx.x;
  if (cb >= Vh) return;
  const int s = blockIdx.y % ls, r = blockIdx.y / ls;
  in += (long)r * 12 * stride + (long)s * Vh + cb;
  int4 w[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) w[k] = __ldg(in + k * stride);
  fx_put(w, fx_exponent(w), out, (long)blockIdx.y * out.nsb, cb);
}

// the same from a canonical field; blockIdx.y: right-hand side, blockIdx.z: parity - parity0
__global__ void __launch_bounds__(128) k_canon_to_fx(Geom g, const double2* __restrict__ canon, FxField even, FxField odd,
                                                     int parity0) {
  __shared__ CanonWarp sm[4];
  pdl_enter();
  const int cb = blockIdx.x * blockDim.x + threadIdx.x, parity = parity0 + blockIdx.z;
  const bool valid = cb < g.Vh;
  double2 v[12];
  canon_load(sm[threadIdx.x >> 5], canon, valid ? ((long)blockIdx.y * g.V + canon_index(g, cb, parity)) * 12 : -1, v);
  if (!valid) return;
  int4 w[12];
#pragma unroll
  for (int k = 0; k < 12; ++k)
    w[k] = make_int4(__double2loint(v[k].x), __double2hiint(v[k].x), __double2loint(v[k].y), __double2hiint(v[k].y));
  const FxField& out = parity ? odd : even;
  fx_put(w, fx_exponent(w), out, (long)blockIdx.y * out.nsb, cb);
}

// A warp owns 16 sites, lane = 16 sp + site: the lane computes the link products of spin sp of the half
// spinors (three colours instead of six: half the registers per thread, twice the warps), sums the upper spin
// sp and, of the lower spins, the one that spin sp of the half spinor feeds: 1 - sp in the x and y hops, sp in the z and
// t hops, so the sums of the lower spins change lanes once, between them.
//
// Shared memory of a block: the links of a warp's sites, one hop per buffer, brought by bulk copies
// (a hop's 9 elements x 16 sites are 2304 contiguous bytes) kBuf hops ahead; and each
// site's eight neighbour indices (the sign bit: the hop carries the antiperiodic factor).
constexpr int kWarps = 4;  // warps per block
constexpr int kBuf = 2;
struct FxShared {
  int4 w[kWarps][kBuf][kHopUnits];
  int nb[8][kWarps * kSB];
  unsigned long long bar[kWarps][kBuf];
};

struct FxWarp {
  FxShared* sm;
  const int4* links;  // of this warp's sites
  int warp, lane;
  bool failed;
  __device__ __forceinline__ void issue(int hop, int buf) {
    if (lane == 0) {
      unsigned long long* bar = &sm->bar[warp][buf];
      fence_proxy_async();  // the lanes' reads of the buffer (ordered by the last __syncwarp) before the copy
      mbar_expect_tx(bar, kHopUnits * 16u);
      bulk_g2s(&sm->w[warp][buf][0], links + hop * kHopUnits, kHopUnits * 16u, bar);
    }
  }
};

// the order of the hops: y, x, z, t (forward, backward)
__device__ __forceinline__ constexpr int fx_order(int i) { return i < 2 ? 2 + i : (i < 4 ? i - 2 : i); }

// barriers and the first copies (the links are constant: before the predecessor kernel is waited for)
__device__ __forceinline__ FxWarp fx_begin(FxShared& sm, const int4* links, long block) {
  FxWarp W{&sm, links + block * (8 * kHopUnits), (int)(threadIdx.x >> 5), (int)(threadIdx.x & 31), false};
  if (W.lane < kBuf) mbar_init(&sm.bar[W.warp][W.lane], 1);
  if (W.lane < kBuf) mbar_init_fence();
  __syncwarp();
#pragma unroll
  for (int b = 0; b < kBuf; ++b) W.issue(fx_order(b), b);
  return W;
}
__device__ __forceinline__ void fx_abandon(FxWarp& W) {  // wait for the copies in flight
#pragma unroll
  for (int b = 0; b < kBuf; ++b) mbar_wait(&W.sm->bar[W.warp][b], 0u);
}

// The half spinor of a hop in direction MU that the lane multiplies (upper spin sp, the lower spin that it meets times
// m): integer and FP32 parts.  nbw: the neighbour's index, negative with the antiperiodic factor.
template <int MU>
__device__ __forceinline__ void fx_half(const FxField& f, int nbw, int sp, int m, int (&hr)[3], int (&hi)[3],
                                        float2 (&y)[3]) {
  const int ncb = nbw & 0x7fffffff;
  const int4* q = f.p + (long)(ncb / kSB) * kSiteUnits + ncb % kSB;
  const int4* qu = q + sp * (3 * kSB);
  const int4* ql = q + 6 * kSB + (MU < 2 ? 1 - sp : sp) * (3 * kSB);  // the lower spin that meets upper spin sp
  const float mf = (float)m;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int4 a = __ldg(qu + c * kSB), b = __ldg(ql + c * kSB);
    const float ar = __int_as_float(a.y), ai = __int_as_float(a.w);
    const float br = __int_as_float(b.y), bi = __int_as_float(b.w);
    if (MU == 0 || MU == 2) {  // -+ i l
      hr[c] = a.x + m * b.z;
      hi[c] = a.z - m * b.x;
      y[c] = make_float2(fmaf(mf, bi, ar), fmaf(-mf, br, ai));
    } else {
      hr[c] = a.x + m * b.x;
      hi[c] = a.z + m * b.z;
      y[c] = make_float2(fmaf(mf, br, ar), fmaf(mf, bi, ai));
    }
  }
  if (nbw < 0) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      hr[c] = -hr[c];
      hi[c] = -hi[c];
      y[c] = make_float2(-y[c].x, -y[c].y);
    }
  }
}

// What the eight hops add up to in a lane: upper spin sp and a lower spin (up to the sign that fx_sum applies), and
// beside each component the sum of |hop| in units of 2^48 (2^(E - 1022) is 2^9 of them), a component's real and
// imaginary part in one word.
struct FxSum {
  int64_t up[6], lo[6];
  unsigned su[3], sl[3];
};

// Hop number I (of fx_order) added to S.  m: the sign of the lower input spin.  Packed FP32 lanes: (re, im).
template <int I>
__device__ __forceinline__ void fx_hop(FxWarp& W, const FxField& f, int E, int sp, int m, FxSum& S) {
  constexpr int HOP = fx_order(I), MU = HOP >> 1;
  constexpr int SG = (HOP & 1) ? 1 : -1;  // (1 - gamma) forward, (1 + gamma) backward
  const int nbw = W.sm->nb[HOP][W.warp * kSB + W.lane % kSB];
  const int d3 = min(E - __ldg(f.e + (nbw & 0x7fffffff)), 100) + 3;
  int hr[3], hi[3];
  float2 y[3];  // the FP32 parts
  fx_half<MU>(f, nbw, sp, m * SG, hr, hi, y);
  if (!mbar_wait(&W.sm->bar[W.warp][I % kBuf], (unsigned)(I / kBuf) & 1u)) W.failed = true;
  if (d3 < kFar) {
    const float sc = __int_as_float((127 - d3) << 23);
    const int4* w = &W.sm->w[W.warp][I % kBuf][W.lane % kSB];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      int64_t Hr = hop_half(d3, HOP & 1), Hi = Hr;
      float2 C = make_float2(0.f, 0.f), D = C;  // (re, im) = (C.x - D.x, C.y + D.y)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const int4 u = w[(a * 3 + b) * kSB];
        const float2 g = make_float2((float)hr[b], (float)hi[b]);  // the integer parts as FP32
        Hr += (int64_t)u.x * hr[b];
        Hr += (int64_t)u.z * -hi[b];
        Hi += (int64_t)u.x * hi[b];
        Hi += (int64_t)u.z * hr[b];
        C = fma2(bc2((float)u.x), y[b], C);
        C = fma2(bc2(__int_as_float(u.y)), g, C);
        D = fma2(bc2((float)u.z), swp(y[b]), D);
        D = fma2(bc2(__int_as_float(u.w)), swp(g), D);
      }
      const int64_t wr = hop_round(Hr, C.x - D.x, sc, d3), wi = hop_round(Hi, C.y + D.y, sc, d3);
      const unsigned size = __byte_perm(abs((int)(wr >> 32)), abs((int)(wi >> 32)), 0x7632);
      S.up[2 * a] += wr;
      S.up[2 * a + 1] += wi;
      S.su[a] += size;
      if (MU == 0 || MU == 2) {  // SG i w
        S.lo[2 * a] -= SG * wi;
        S.lo[2 * a + 1] += SG * wr;
        S.sl[a] += __byte_perm(size, size, 0x1032);
      } else {
        S.lo[2 * a] += SG * wr;
        S.lo[2 * a + 1] += SG * wi;
        S.sl[a] += size;
      }
    }
  }
  __syncwarp();  // every lane has read the buffer
  if (I + kBuf < 8) W.issue(fx_order(I + kBuf < 8 ? I + kBuf : 0), I % kBuf);
}

// The magnitudes of a lane's products, per component (upper spin sp in s, the lower spin in t), the neighbours' sizes relative
// to the largest one's, and bits of nz, nt: a product is not zero.
struct FxMagnitudes {
  float s[6], t[6], size;
  unsigned nz, nt;
};

// Those of hop number I.  links: of the lane's site.
template <int I>
__device__ __forceinline__ void fx_magnitudes(const int* nb, const FxField& f, const int4* links, int E, int sp, int m,
                                              FxMagnitudes& M) {
  constexpr int HOP = fx_order(I), MU = HOP >> 1;
  constexpr int SG = (HOP & 1) ? 1 : -1;  // (1 - gamma) forward, (1 + gamma) backward
  const int nbw = nb[HOP * (kWarps * kSB)];
  const int d = min(E - __ldg(f.e + (nbw & 0x7fffffff)), 100);
  int hr[3], hi[3];
  float2 y[3];
  fx_half<MU>(f, nbw, sp, m * SG, hr, hi, y);
  const float sc = __int_as_float((127 - d) << 23);
  M.size += sc;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float mr = 0.f, mi = 0.f;
    unsigned br = 0, bi = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int4 u = __ldg(links + HOP * kHopUnits + (a * 3 + b) * kSB);
      const float ur = fabsf((float)u.x + __int_as_float(u.y)), ui = fabsf((float)u.z + __int_as_float(u.w));
      const float xr = fabsf((float)hr[b] + y[b].x), xi = fabsf((float)hi[b] + y[b].y);
      mr = fmaf(ur, xr, fmaf(ui, xi, mr));
      mi = fmaf(ur, xi, fmaf(ui, xr, mi));
      br |= (ur != 0.f && xr != 0.f) || (ui != 0.f && xi != 0.f);
      bi |= (ur != 0.f && xi != 0.f) || (ui != 0.f && xr != 0.f);
    }
    constexpr int x = (MU == 0 || MU == 2) ? 1 : 0;  // i w
    M.s[2 * a] = fmaf(mr, sc, M.s[2 * a]);
    M.s[2 * a + 1] = fmaf(mi, sc, M.s[2 * a + 1]);
    M.t[2 * a + x] = fmaf(mr, sc, M.t[2 * a + x]);
    M.t[2 * a + 1 - x] = fmaf(mi, sc, M.t[2 * a + 1 - x]);
    M.nz |= (br | bi << 1) << (2 * a);
    M.nt |= (x ? (bi | br << 1) : (br | bi << 1)) << (2 * a);
  }
}

// Hop number I in FP64, added to the lane's sums as fx_hop does: from the FP64 field that was converted to f where A.in
// names it (src: its slice; of a canonical field if A.in.stride is 1), else from the parts (the first half-dslash of Mhat
// left no other form).
template <int I>
__device__ __forceinline__ void fp64_hop(const HA& A, const FxField& f, const double2* src, const int* nb, int cb, int sp,
                                         int m, Cx<double> (&v)[6]) {
  constexpr int HOP = fx_order(I), MU = HOP >> 1;
  constexpr int SG = (HOP & 1) ? 1 : -1;
  const int nbw = nb[HOP * (kWarps * kSB)], n = nbw & 0x7fffffff;
  const int ku = 3 * sp, kl = 6 + 3 * (MU < 2 ? 1 - sp : sp);  // the first components of the two spins
  Cx<double> u[3], l[3], h[3], U[9];
  if (src) {
    const bool canon = A.in.stride == 1;
    const double2* p = src + (canon ? (long)canon_index(A.g, n, 1 - A.out_parity) * 12 : n);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 x = __ldg(p + (ku + c) * A.in.stride), y = __ldg(p + (kl + c) * A.in.stride);
      u[c] = {x.x, x.y};
      l[c] = {y.x, y.y};
    }
  } else {
    const int e = f.e[n];
    const int4* p = f.p + (long)(n / kSB) * kSiteUnits + n % kSB;
    auto value = [&](int k) {
      const int4 w = p[k * kSB];
      return e == kBad ? Cx<double>{__hiloint2double(w.y, w.x), __hiloint2double(w.w, w.z)}
                       : Cx<double>{part_value({w.x, __int_as_float(w.y)}, e), part_value({w.z, __int_as_float(w.w)}, e)};
    };
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u[c] = value(ku + c);
      l[c] = value(kl + c);
    }
  }
  const double s = m * SG, sign = nbw < 0 ? -1.0 : 1.0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (MU == 0 || MU == 2)
      h[c] = {sign * fma(s, l[c].im, u[c].re), sign * fma(-s, l[c].re, u[c].im)};
    else
      h[c] = {sign * fma(s, l[c].re, u[c].re), sign * fma(s, l[c].im, u[c].im)};
  }
  A.U.load((HOP & 1) ? 1 - A.out_parity : A.out_parity, MU, (HOP & 1) ? n : cb, U);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Cx<double> w = {0.0, 0.0};
#pragma unroll
    for (int b = 0; b < 3; ++b) w = (HOP & 1) ? cjmadd(U[b * 3 + a], h[b], w) : cmadd(U[a * 3 + b], h[b], w);
    v[a] = v[a] + w;
    v[3 + a] = v[3 + a] + ((MU == 0 || MU == 2) ? Cx<double>{-SG * w.im, SG * w.re} : Cx<double>{SG * w.re, SG * w.im});
  }
}

// The hop sums of the lane (upper spin sp, lower spin 2 + sp, the latter times -1 for H^dag) in FP64; the whole warp calls
// it, since a site's two lanes share the work; with keep into the lane's slots, as bits.  Bound by the FP64 pipe.  The full matrix on
// 24^3 x 32 where every site comes here (a point source's solution, links within 1e-4 of 1): 1.15 ms with the two walks
// before; the FP64 kernel, 0.82.
__device__ __noinline__ void fp64_sum(const HA& A, const FxField& f, int q, const int* nb, int cb, int sp, bool keep,
                                      int64_t* slots) {
  const double2* src = A.in.p;
  if (src) {
    const int r = fdiv(q, A.d_ls);
    src += A.in.stride == 1 ? (long)q * A.g.V * 12 : (long)r * 12 * A.in.stride + (long)(q - r * A.ls) * A.g.Vh;
  }
  const int g5 = A.dagger ? -1 : 1, gs = sp ? -g5 : g5;
  Cx<double> v[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) v[k] = {0.0, 0.0};
  auto turn = [&](bool minus) {
#pragma unroll
    for (int k = 3; k < 6; ++k) v[k] = minus ? -v[k] : v[k];
  };
  fp64_hop<0>(A, f, src, nb, cb, sp, -gs, v);  // signs and lanes as in fx_sum
  fp64_hop<1>(A, f, src, nb, cb, sp, -gs, v);
  turn(sp == 0);
  fp64_hop<2>(A, f, src, nb, cb, sp, g5, v);
  fp64_hop<3>(A, f, src, nb, cb, sp, g5, v);
#pragma unroll
  for (int k = 3; k < 6; ++k)
    v[k] = {__shfl_xor_sync(0xffffffffu, v[k].re, kSB), __shfl_xor_sync(0xffffffffu, v[k].im, kSB)};
  turn(sp != 0);
  fp64_hop<4>(A, f, src, nb, cb, sp, gs, v);
  fp64_hop<5>(A, f, src, nb, cb, sp, gs, v);
  turn(sp != 0);
  fp64_hop<6>(A, f, src, nb, cb, sp, g5, v);
  fp64_hop<7>(A, f, src, nb, cb, sp, g5, v);
  if (!keep) return;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    slots[2 * k * 32] = __double_as_longlong(v[k].re);
    slots[(2 * k + 1) * 32] = __double_as_longlong(v[k].im);
  }
}

// The exponent field of the site's largest neighbour (its neighbour indices go to shared memory).
__device__ __forceinline__ int fx_neighbours(const HA& A, FxWarp& W, const FxField& f, int cb) {
  const SiteCoords c = cb_to_site(A.g, cb, A.out_parity);
  int E = kZero;
  const bool back = W.lane >= kSB;  // the site's other lane does the forward hops
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    int wrap;
    const int n = neighbour_index(A.g, c, mu, back ? -1 : +1, &wrap) >> 1;
    W.sm->nb[2 * mu + back][W.warp * kSB + W.lane % kSB] = n | ((wrap && A.g.apbc[mu]) ? 0x80000000 : 0);
    E = max(E, __ldg(f.e + n));
  }
  E = max(E, __shfl_xor_sync(0xffffffffu, E, kSB));
  __syncwarp();
  return E;
}

__device__ __forceinline__ void flip(int64_t (&v)[6], bool minus) {
  const int64_t n = minus ? -1 : 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) v[k] = (v[k] ^ n) - n;
}

__device__ __forceinline__ double fx_unit(int E) { return __hiloint2double((E - 56) << 20, 0); }  // 2^(E - 1079)
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

// S.up, S.lo = the sum of the eight hops for spins sp and 2 + sp, in units of 2^(E - 1079) (lo: times -1 for
// H^dag = g5 H g5); the whole warp calls it.  true (for the whole warp): the sums do not show that they are exact
// enough, or a neighbour is kept in FP64, and fx_careful decides.
//
// The sum of |hop| is a lower bound of the sum of magnitudes that fixed.cuh asks for, and costs 17 instructions per hop: below
// 2^(E - 1022) / 8 in one site of 10^5 of a Gaussian field.  Without it a half-dslash on 32^3 x 64 took 351 us instead of 371,
// a solve on 12x10x14x18 3.53 ms instead of 3.71, and twelve point sources on 24^3 x 48 139 ms instead of 144 to 147 (fx_decide).
__device__ __forceinline__ bool fx_sum(const HA& A, FxWarp& W, const FxField& f, int E, int sp, FxSum& S) {
  const int g5 = A.dagger ? -1 : 1, gs = sp ? -g5 : g5;
#pragma unroll
  for (int k = 0; k < 6; ++k) S.up[k] = S.lo[k] = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) S.su[k] = S.sl[k] = 0;
  fx_hop<0>(W, f, E, sp, -gs, S);  // y: B = (-l1, l0)
  fx_hop<1>(W, f, E, sp, -gs, S);
  flip(S.lo, sp == 0);             // B^dag = (g1, -g0)
  fx_hop<2>(W, f, E, sp, g5, S);   // x: B = -i (l1, l0)
  fx_hop<3>(W, f, E, sp, g5, S);
#pragma unroll
  for (int k = 0; k < 6; ++k) S.lo[k] = __shfl_xor_sync(0xffffffffu, S.lo[k], kSB);
#pragma unroll
  for (int k = 0; k < 3; ++k) S.sl[k] = __shfl_xor_sync(0xffffffffu, S.sl[k], kSB);
  flip(S.lo, sp != 0);
  fx_hop<4>(W, f, E, sp, gs, S);   // z: B = (-i l0, i l1)
  fx_hop<5>(W, f, E, sp, gs, S);
  flip(S.lo, sp != 0);
  fx_hop<6>(W, f, E, sp, g5, S);   // t: B = 1
  fx_hop<7>(W, f, E, sp, g5, S);
  unsigned least = 0xffffffffu;
#pragma unroll
  for (int k = 0; k < 3; ++k) least = __vminu2(least, __vminu2(S.su[k], S.sl[k]));
  const bool weak = (min(least & 0xffffu, least >> 16) < 64u && E > kZero) || E == kBad;  // kZero: all neighbours are zero
  return __any_sync(0xffffffffu, weak);
}

// What fx_sum left open: the magnitudes of the products are formed, and a site with a neighbour that is kept in
// FP64, or with a component that is neither as exact as FP64 would have it (fixed.cuh) nor without a product that is not
// zero, is computed in FP64: true, for both lanes of the site, and the sums in the lane's slots are FP64
// numbers.  It settles all but fields with components far smaller than others that the links hardly mix with them.
__device__ __noinline__ bool fx_decide(const HA& A, const FxField& f, const int4* links, const int* nb, int q, int E, int cb,
                                       int sp, int64_t* slots) {
  const int g5 = A.dagger ? -1 : 1, gs = sp ? -g5 : g5;
  FxMagnitudes M = {};
  fx_magnitudes<0>(nb, f, links, E, sp, -gs, M);  // signs and lanes as in fx_sum
  fx_magnitudes<1>(nb, f, links, E, sp, -gs, M);
  fx_magnitudes<2>(nb, f, links, E, sp, g5, M);
  fx_magnitudes<3>(nb, f, links, E, sp, g5, M);
#pragma unroll
  for (int k = 0; k < 6; ++k) M.t[k] = __shfl_xor_sync(0xffffffffu, M.t[k], kSB);
  M.nt = __shfl_xor_sync(0xffffffffu, M.nt, kSB);
  fx_magnitudes<4>(nb, f, links, E, sp, gs, M);
  fx_magnitudes<5>(nb, f, links, E, sp, gs, M);
  fx_magnitudes<6>(nb, f, links, E, sp, g5, M);
  fx_magnitudes<7>(nb, f, links, E, sp, g5, M);
  const float least = sum_min(M.size);
  bool bad = E == kBad;
#pragma unroll
  for (int k = 0; k < 6; ++k)
    bad = bad || (M.s[k] < least && (M.nz >> k & 1)) || (M.t[k] < least && (M.nt >> k & 1));
  const unsigned all = __ballot_sync(0xffffffffu, bad), site = (all | all >> kSB) & 0xffffu;
  if (!site) return false;
  bad = site >> (threadIdx.x % kSB) & 1;
  fp64_sum(A, f, q, nb, cb, sp, bad, slots);
  return bad;
}

// The sums of fx_sum go through the warp's link buffers, which are free now, so that the kernels' registers hold nothing
// across the calls (with the sums kept in them their spills added 110 MB to the DRAM traffic of a half-dslash on
// 32^3 x 64, and 9 us; with the sums formed again by the second walk the full matrix took 1.34 ms instead of 1.15 where
// every site needs it).
__device__ __forceinline__ bool fx_careful(const HA& A, FxWarp& W, const FxField& f, int q, int E, int cb, int sp, FxSum& S) {
  static_assert(sizeof(W.sm->w[0]) >= 32 * 12 * sizeof(int64_t), "a warp's sums fit its link buffers");
  int64_t* slots = reinterpret_cast<int64_t*>(&W.sm->w[W.warp][0][0]) + W.lane;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    slots[k * 32] = S.up[k];
    slots[(6 + k) * 32] = S.lo[k];
  }
  const bool fp64 = fx_decide(A, f, W.links + W.lane % kSB, &W.sm->nb[0][W.warp * kSB + W.lane % kSB], q, E, cb, sp, slots);
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    S.up[k] = slots[k * 32];
    S.lo[k] = slots[(6 + k) * 32];
  }
  __syncwarp();
  return fp64;
}

// The sums as a fixed-point field of their own (a = 1, no x term: the first half-dslash of Mhat, whose
// result only the second one reads): both lanes of a site find its largest sum.
__device__ __forceinline__ void fx_store(const FxField& out, int cb, int sp, bool valid, int E, bool minus_lo, bool nan,
                                         int64_t (&up)[6], int64_t (&lo)[6]) {
  flip(lo, minus_lo);
  uint64_t mx = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    mx |= (uint64_t)(up[k] ^ (up[k] >> 63));
    mx |= (uint64_t)(lo[k] ^ (lo[k] >> 63));
  }
  mx |= __shfl_xor_sync(0xffffffffu, mx, kSB);
  if (!valid) return;
  const int b = 64 - __clzll((long long)mx);  // -2^b <= every sum < 2^b
  const int e = mx ? b + E - 57 : kZero, shift = b - 30;
  int4* o = out.p + (long)(cb / kSB) * kSiteUnits + sp * (3 * kSB) + cb % kSB;
  const bool wide = nan || (mx && (e < kEmin || e > kEmax));
  const double unit = nan ? fx_nan() : fx_unit(E);
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int c = k % 3;
    const int64_t re = k < 3 ? up[2 * c] : lo[2 * c], im = k < 3 ? up[2 * c + 1] : lo[2 * c + 1];
    int4 w;
    if (wide) {
      const double x = (double)re * unit, y = (double)im * unit;
      w = make_int4(__double2loint(x), __double2hiint(x), __double2loint(y), __double2hiint(y));
    } else {
      const Part pr = sum_part(re, shift), pi = sum_part(im, shift);
      w = make_int4(pr.h, __float_as_int(pr.l), pi.h, __float_as_int(pi.l));
    }
    o[(k < 3 ? c : 6 + c) * kSB] = w;
  }
  if (sp == 0) out.e[cb] = wide ? kBad : e;
}

// FP64 sums of fx_careful as a kBad site of that field
__device__ __forceinline__ void fx_store_fp64(const FxField& out, int cb, int sp, bool minus_lo, const FxSum& S) {
  int4* o = out.p + (long)(cb / kSB) * kSiteUnits + sp * (3 * kSB) + cb % kSB;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int64_t sign = k >= 3 && minus_lo ? INT64_MIN : 0;
    const int64_t x = k < 3 ? S.up[2 * k] : S.lo[2 * k - 6] ^ sign, y = k < 3 ? S.up[2 * k + 1] : S.lo[2 * k - 5] ^ sign;
    o[(k < 3 ? k : 3 + k) * kSB] = make_int4((int)x, (int)(x >> 32), (int)y, (int)(y >> 32));
  }
  if (sp == 0) out.e[cb] = kBad;
}

// the sites and the slice of a lane
struct FxLane {
  int cb0, cb, sp, q, r;
  bool valid, warp_valid;
};
__device__ __forceinline__ FxLane fx_lane(const HA& A) {
  FxLane L;
  const int sblock = fdiv(blockIdx.x, A.d_ntiles);
  L.q = blockIdx.x - sblock * A.ntiles;
  L.r = fdiv(L.q, A.d_ls);
  L.cb0 = (sblock * kWarps + (threadIdx.x >> 5)) * kSB;
  L.cb = L.cb0 + threadIdx.x % kSB;
  L.sp = (threadIdx.x & 31) / kSB;
  L.valid = L.cb < A.g.Vh;
  L.warp_valid = L.cb0 < A.g.Vh;
  return L;
}
__device__ __forceinline__ FxField fx_slice(const FxField& F, int q) {
  return {F.p + (long)q * F.nsb * kSiteUnits, F.e + (long)q * F.nsb * kSB, F.nsb};
}

// a H in for the lane's six components (upper spin sp, lower spin 2 + sp) as a[k / 3] v[k]; the whole warp calls it
__device__ __forceinline__ void fx_values(const HA& A, FxWarp& W, const FxField& f, const FxLane& L, Cx<double> (&v)[6],
                                          double (&a)[2]) {
  const int cb = L.valid ? L.cb : 0;
  const int E = fx_neighbours(A, W, f, cb);
  FxSum S;
  a[0] = A.a * fx_unit(E);
  bool fp64 = false;
  if (fx_sum(A, W, f, E, L.sp, S)) {
    fp64 = fx_careful(A, W, f, L.q, E, cb, L.sp, S);
    if (fp64) a[0] = A.a;
  }
  if (W.failed) a[0] = fx_nan();  // a copy that never arrived
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int64_t re = k < 3 ? S.up[2 * k] : S.lo[2 * k - 6], im = k < 3 ? S.up[2 * k + 1] : S.lo[2 * k - 5];
    v[k] = {fp64 ? __longlong_as_double(re) : (double)re, fp64 ? __longlong_as_double(im) : (double)im};
  }
  a[1] = A.dagger ? -a[0] : a[0];
}

// OUT = 0: [x +] a H in as FP64; OUT = 1: H in as the fixed-point field O
template <int MINB, int OUT>
__global__ void __launch_bounds__(32 * kWarps, MINB) k_hop_fx(const __grid_constant__ HA A,
                                                              const int4* __restrict__ links,
                                                              const __grid_constant__ FxField F,
                                                              const __grid_constant__ FxField O) {
  extern __shared__ __align__(128) unsigned char smraw[];
  FxShared& sm = *reinterpret_cast<FxShared*>(smraw);
  const FxLane L = fx_lane(A);
  if (!L.warp_valid) return;
  FxWarp W = fx_begin(sm, links, (long)A.out_parity * F.nsb + L.cb0 / kSB);
  pdl_enter();
  if (A.stop && *A.stop) {
    fx_abandon(W);
    return;
  }
  const FxField f = fx_slice(F, L.q);
  if constexpr (OUT == 1) {
    const int cb = L.valid ? L.cb : 0;
    const int E = fx_neighbours(A, W, f, cb);
    FxSum S;
    const FxField o = fx_slice(O, L.q);
    bool fp64 = false;
    if (fx_sum(A, W, f, E, L.sp, S)) {
      fp64 = fx_careful(A, W, f, L.q, E, cb, L.sp, S);
      if (fp64 && L.valid) fx_store_fp64(o, L.cb, L.sp, A.dagger != 0, S);
    }
    fx_store(o, L.cb, L.sp, L.valid && !fp64, E, A.dagger != 0, W.failed, S.up, S.lo);
    return;
  }
  Cx<double> v[6];
  double a[2];
  fx_values(A, W, f, L, v, a);
  if (!L.valid) return;
  const long site = (long)(L.q - L.r * A.ls) * A.g.Vh + L.cb;
  const long xstr = A.x.stride, ostr = A.out.stride;
  const double2* x = A.x.offset_rhs(L.r).p + 3 * L.sp * xstr + site;
  double2* o = A.out.offset_rhs(L.r).p + 3 * L.sp * ostr + site;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int n = k < 3 ? k : 3 + k;
    if (A.xpay) {
      const double2 xs = __ldg(x + n * xstr);
      o[n * ostr] = make_double2(fma(a[k / 3], v[k].re, xs.x), fma(a[k / 3], v[k].im, xs.y));
    } else {
      o[n * ostr] = make_double2(a[k / 3] * v[k].re, a[k / 3] * v[k].im);
    }
  }
}

// one right-hand side, the BiCGStab inner products of k_hop_red (wilson.cu) in the epilogue
template <int MINB, int RED>
__global__ void __launch_bounds__(32 * kWarps, MINB) k_hop_fx_red(const __grid_constant__ HA A,
                                                                  const int4* __restrict__ links,
                                                                  const __grid_constant__ FxField F) {
  extern __shared__ __align__(128) unsigned char smraw[];
  FxShared& sm = *reinterpret_cast<FxShared*>(smraw);
  const FxLane L = fx_lane(A);  // one slice
  FxWarp W;
  if (L.warp_valid) W = fx_begin(sm, links, (long)A.out_parity * F.nsb + L.cb0 / kSB);
  pdl_enter();
  if (A.stop && *A.stop) {
    if (L.warp_valid) fx_abandon(W);
    return;
  }
  double red[3] = {0.0, 0.0, 0.0};
  if (L.warp_valid) {
    Cx<double> v[6];
    double a[2];
    fx_values(A, W, F, L, v, a);
    if (L.valid) {
      const double2* x = A.x.p + 3 * L.sp * A.x.stride + L.cb;
      const double2* rt = A.rt.p + 3 * L.sp * A.rt.stride + L.cb;
      double2* out = A.out.p + 3 * L.sp * A.out.stride + L.cb;
      Cx<double> d = {0.0, 0.0};
#pragma unroll
      for (int k = 0; k < 6; ++k) {  // colour k of spin sp, colour k - 3 of spin 2 + sp
        const int n = k < 3 ? k : 3 + k;
        const double2 xs = __ldg(x + n * A.x.stride);
        const Cx<double> o = {fma(a[k / 3], v[k].re, xs.x), fma(a[k / 3], v[k].im, xs.y)};
        out[n * A.out.stride] = make_double2(o.re, o.im);
        if (RED == 1) {  // (rt, out)
          const double2 w = __ldg(rt + n * A.rt.stride);
          d = cjmadd(Cx<double>{w.x, w.y}, o, d);
        } else {  // (out, x), |out|^2
          d = cjmadd(o, Cx<double>{xs.x, xs.y}, d);
          red[2] = fma(o.re, o.re, fma(o.im, o.im, red[2]));
        }
      }
      red[0] = d.re;
      red[1] = d.im;
    }
  }
  red_epilogue<double>(A, red);
}

// ----------------------------------------------------------------------------- outer step
// One outer step of the mixed-precision Wilson solve (true residual of the full system) is three kernels:
// x += xin with the result also in fixed point (k_outer_x); x_o = b_o + kappa H_oe x, in FP64 and in fixed
// point (k_outer_odd); r_e = b_e - x + kappa H_eo x_o, kept only as the inner residual and its norm
// (k_outer_res).  As separate stencils, copies, axpys, norms and conversions the step moved 7.4 KB per site, here
// 4.6, and 14 launches and 3 synchronisations became 6 and 1.  Measured: 24^3 x 48 with FP16 inner vectors (6
// steps) 16.2 -> 14.6 ms, 8^3 x 16 2.77 -> 2.25 ms, 12 right-hand sides 156 -> 150 ms, 32^3 x 64 51.3 -> 49.5 ms.

// a sum over the block (all its warps one slice) into partial[row * 4 + k]
__device__ __forceinline__ void block_partial(double v0, double* partial, long row, int k) {
  double v[1] = {v0};
  block_sum<1>(v);
  if (threadIdx.x == 0) partial[row * 4 + k] = v[0];
}

// x += xin, xin = 0 (xin may be null: x as it is), and x in fixed point; blockIdx.y: right-hand side
__global__ void __launch_bounds__(128) k_outer_x(SpinorView<P64> x, SpinorView<P32> xin, int has_xin, FxField out,
                                                 int Vh) {
  pdl_enter();
  const int cb = blockIdx.x * blockDim.x + threadIdx.x;
  if (cb >= Vh) return;
  x = x.offset_rhs(blockIdx.y);
  Cx<double> v[12];
  if (has_xin) {
    xin = xin.offset_rhs(blockIdx.y);
    float4 d[6];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const double2 w = x.p[k * x.stride + cb];
      v[k] = {w.x, w.y};
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) d[q] = xin.p[q * xin.stride + cb];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int k = q < 3 ? q : q + 3;  // spins a (component k) and b (k + 3) of the pair
      v[k] = {v[k].re + (double)d[q].x, v[k].im + (double)d[q].z};
      v[k + 3] = {v[k + 3].re + (double)d[q].y, v[k + 3].im + (double)d[q].w};
    }
    x.store(cb, v);
#pragma unroll
    for (int q = 0; q < 6; ++q) xin.p[q * xin.stride + cb] = make_float4(0.f, 0.f, 0.f, 0.f);
  } else {
    x.load(cb, v);
  }
  int4 w[12];
#pragma unroll
  for (int k = 0; k < 12; ++k)
    w[k] = make_int4(__double2loint(v[k].re), __double2hiint(v[k].re), __double2loint(v[k].im), __double2hiint(v[k].im));
  const int e = fx_exponent(w);
  fx_put(w, e, out, (long)blockIdx.y * out.nsb, cb);
}

// out = x + a H in, FP64 and as the fixed-point field O; partial k = 1: |x - out + a H in|^2, the rounding of out
__global__ void __launch_bounds__(32 * kWarps, 4) k_outer_odd(const __grid_constant__ HA A,
                                                              const int4* __restrict__ links,
                                                              const __grid_constant__ FxField F,
                                                              const __grid_constant__ FxField O) {
  extern __shared__ __align__(128) unsigned char smraw[];
  FxShared& sm = *reinterpret_cast<FxShared*>(smraw);
  const FxLane L = fx_lane(A);
  FxWarp W;
  if (L.warp_valid) W = fx_begin(sm, links, (long)A.out_parity * F.nsb + L.cb0 / kSB);
  pdl_enter();
  double res = 0.0;
  if (L.warp_valid) {
    const FxField f = fx_slice(F, L.q);
    Cx<double> h[6];
    double a[2];
    fx_values(A, W, f, L, h, a);
    int4 w[6];
    if (L.valid) {
      const double2* x = A.x.offset_rhs(L.r).p + 3 * L.sp * A.x.stride + L.cb;
      double2* o = A.out.offset_rhs(L.r).p + 3 * L.sp * A.out.stride + L.cb;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const int n = k < 3 ? k : 3 + k;
        const double2 xs = __ldg(x + n * A.x.stride);
        const double ak = a[k / 3];
        const Cx<double> v = {fma(ak, h[k].re, xs.x), fma(ak, h[k].im, xs.y)};
        o[n * A.out.stride] = make_double2(v.re, v.im);
        const double dr = fma(ak, h[k].re, xs.x - v.re), di = fma(ak, h[k].im, xs.y - v.im);
        res = fma(dr, dr, fma(di, di, res));
        w[k] = make_int4(__double2loint(v.re), __double2hiint(v.re), __double2loint(v.im), __double2hiint(v.im));
      }
    } else {
#pragma unroll
      for (int k = 0; k < 6; ++k) w[k] = make_int4(0, 0, 0, 0);
    }
    const int e = fx_exponent_pair(w);
    if (L.valid) {
      int4* o = O.p + ((long)L.q * O.nsb + L.cb / kSB) * kSiteUnits + 3 * L.sp * kSB + L.cb % kSB;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        int4 u = w[k];
        if (e != kBad) {
          const Part re = spinor_part(w[k].y, w[k].x, e), im = spinor_part(w[k].w, w[k].z, e);
          u = make_int4(re.h, __float_as_int(re.l), im.h, __float_as_int(im.l));
        }
        o[(k < 3 ? k : 3 + k) * kSB] = u;
      }
      if (L.sp == 0) O.e[(long)L.q * O.nsb * kSB + L.cb] = e;
    }
  }
  const int sblock = fdiv(blockIdx.x, A.d_ntiles);
  block_partial(res, A.partial, (long)L.q * (gridDim.x / A.ntiles) + sblock, 1);
}

// r = b - x + a H in (x only with A.xpay = 2), stored in the inner precision PR; partial k = 0: |b - x + a H in|^2
template <int PR>
__global__ void __launch_bounds__(32 * kWarps, 4) k_outer_res(const __grid_constant__ HA A,
                                                              const int4* __restrict__ links,
                                                              const __grid_constant__ FxField F,
                                                              const __grid_constant__ SpinorView<PR> R) {
  extern __shared__ __align__(128) unsigned char smraw[];
  FxShared& sm = *reinterpret_cast<FxShared*>(smraw);
  const FxLane L = fx_lane(A);
  FxWarp W;
  if (L.warp_valid) W = fx_begin(sm, links, (long)A.out_parity * F.nsb + L.cb0 / kSB);
  pdl_enter();
  double res = 0.0;
  if (L.warp_valid) {
    const FxField f = fx_slice(F, L.q);
    Cx<double> h[6];
    double a[2];
    fx_values(A, W, f, L, h, a);
    const int cb = L.valid ? L.cb : 0;
    const double2* b = A.rt.offset_rhs(L.r).p + 3 * L.sp * A.rt.stride + cb;
    const double2* x = A.x.offset_rhs(L.r).p + 3 * L.sp * A.x.stride + cb;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int n = k < 3 ? k : 3 + k;
      double2 t = __ldg(b + n * A.rt.stride);
      if (A.xpay == 2) {
        const double2 xs = __ldg(x + n * A.x.stride);
        t = make_double2(t.x - xs.x, t.y - xs.y);
      }
      h[k] = {fma(a[k / 3], h[k].re, t.x), fma(a[k / 3], h[k].im, t.y)};
      if (L.valid) res = fma(h[k].re, h[k].re, fma(h[k].im, h[k].im, res));
    }
    const SpinorView<PR> rv = R.offset_rhs(L.r);
    if constexpr (PR == P64) {
      if (L.valid)
#pragma unroll
        for (int k = 0; k < 6; ++k)
          rv.p[(3 * L.sp + (k < 3 ? k : 3 + k)) * rv.stride + cb] = make_double2(h[k].re, h[k].im);
    } else {
      // FP32 / FP16 units hold a spin pair: the lanes of a site exchange halves, lane 0 stores the upper pairs, lane 1
      // the lower ones
      float mine[6], other[6], m = 0.f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const Cx<double> keep = L.sp ? h[3 + c] : h[c], give = L.sp ? h[c] : h[3 + c];
        mine[2 * c] = (float)keep.re;
        mine[2 * c + 1] = (float)keep.im;
        other[2 * c] = __shfl_xor_sync(0xffffffffu, (float)give.re, kSB);
        other[2 * c + 1] = __shfl_xor_sync(0xffffffffu, (float)give.im, kSB);
      }
      float inv = 1.f;
      if constexpr (PR == P16) {
#pragma unroll
        for (int k = 0; k < 6; ++k) m = fmaxf(m, fmaxf(fabsf(mine[k]), fabsf(other[k])));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, kSB));
        inv = (m > 0.f) ? 1.0f / m : 0.f;
      }
      if (L.valid) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int q = 3 * L.sp + c;
          // spins (a, b): lane 0 has spin a of the upper pair, lane 1 spin b of the lower one
          const float ar = L.sp ? other[2 * c] : mine[2 * c], br = L.sp ? mine[2 * c] : other[2 * c];
          const float ai = L.sp ? other[2 * c + 1] : mine[2 * c + 1], bi = L.sp ? mine[2 * c + 1] : other[2 * c + 1];
          if constexpr (PR == P32) {
            rv.p[q * rv.stride + cb] = make_float4(ar, br, ai, bi);
          } else {
            const __half2 re = __floats2half2_rn(ar * inv, br * inv), im = __floats2half2_rn(ai * inv, bi * inv);
            uint2* u = reinterpret_cast<uint2*>(rv.p + (q >> 1) * rv.stride + cb) + (q & 1);
            *u = make_uint2(*reinterpret_cast<const unsigned*>(&re), *reinterpret_cast<const unsigned*>(&im));
          }
        }
        if constexpr (PR == P16)
          if (L.sp == 0) rv.norm[cb] = m;
      }
    }
  }
  const int sblock = fdiv(blockIdx.x, A.d_ntiles);
  block_partial(res, A.partial, (long)L.q * (gridDim.x / A.ntiles) + sblock, 0);
}

// sums[q * stride + k] = sum over the blocks of partial[(q * nb + b) * 4 + k], k < 2 (k = 1 only with both)
__global__ void __launch_bounds__(256) k_outer_sums(const double* __restrict__ partial, int nb, double* __restrict__ sums,
                                                    int stride, int both) {
  pdl_enter();
  const int q = blockIdx.x;
  double v[2] = {0.0, 0.0};
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    v[0] += partial[((long)q * nb + b) * 4];
    if (both) v[1] += partial[((long)q * nb + b) * 4 + 1];
  }
  block_sum<2>(v);
  if (threadIdx.x == 0) {
    sums[(long)q * stride] = v[0];
    sums[(long)q * stride + 1] = v[1];
  }
}

// ----------------------------------------------------------------------------- canonical fields
// out = [x +] a H in on canonical x and out (complex128, both parities): the operators of qcd_dslash on canonical
// FP64 fields without FP64 copies of their halves.  Each warp's 16 sites leave through its link buffers, so that
// whole sites are written in runs; zero: the other site of each pair (the other parity) is zeroed with them.
// Bound by HBM (1732 B per site and half-dslash).  The full matrix at 24^3 x 48: two packings, two conversions, two
// stencils and two unpackings 415 us, one conversion (66 us, at the copy rate) and two of these 307 us
// (96 registers; 327 at 128).  Reading x through shared memory in runs after the hops was slower (368 us): the
// lanes' own loads of 48 bytes are in flight earlier.
__global__ void __launch_bounds__(32 * kWarps, 5) k_hop_fx_canon(const __grid_constant__ HA A,
                                                                    const int4* __restrict__ links,
                                                                    const __grid_constant__ FxField F,
                                                                    const double2* __restrict__ x, double2* out, int zero) {
  extern __shared__ __align__(128) unsigned char smraw[];
  FxShared& sm = *reinterpret_cast<FxShared*>(smraw);
  const FxLane L = fx_lane(A);
  if (!L.warp_valid) return;
  FxWarp W = fx_begin(sm, links, (long)A.out_parity * F.nsb + L.cb0 / kSB);
  pdl_enter();
  const FxField f = fx_slice(F, L.q);
  const long first = (long)L.q * A.g.V * 12;
  const double2* xs = x + first + (long)canon_index(A.g, L.valid ? L.cb : 0, A.out_parity) * 12;
  Cx<double> h[6];
  double a[2];
  fx_values(A, W, f, L, h, a);
  double2* buf = reinterpret_cast<double2*>(&sm.w[W.warp][0][0]);  // [site][12]
  static_assert(sizeof(sm.w[0]) >= kSB * 12 * sizeof(double2), "a warp's sites fit its link buffers");
  __syncwarp();  // every lane has read the last links
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int n = 3 * L.sp + (k < 3 ? k : 3 + k);
    double2 v = make_double2(0.0, 0.0);
    if (A.xpay) v = __ldg(xs + n);
    buf[(L.cb - L.cb0) * 12 + n] = make_double2(fma(a[k / 3], h[k].re, v.x), fma(a[k / 3], h[k].im, v.y));
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < kSB * 12 / 32; ++j) {
    const int u = j * 32 + W.lane, site = u / 12, k = u - 12 * site;
    if (L.cb0 + site < A.g.Vh) {
      double2* o = out + first + k;
      const long c = canon_index(A.g, L.cb0 + site, A.out_parity);
      o[c * 12] = buf[u];
      if (zero) o[(c ^ 1) * 12] = make_double2(0.0, 0.0);
    }
  }
}

// ----------------------------------------------------------------------------- links
// The links of the eight hops as parts, and whether every link has the size the fixed point takes:
// *flag becomes nonzero if a row or column 2-norm lies outside [kNormMin, kNormMax] (or is NaN).
// One thread per (parity, mu, site): both ends of its link.
__global__ void __launch_bounds__(128) k_links_fx(Geom g, const double2* __restrict__ U64, int4* __restrict__ W, long nsb,
                                                  int* flag) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  const long Vh = g.Vh;
  if (i >= 8 * Vh) return;
  const int pm = (int)(i / Vh), cb = (int)(i % Vh), par = pm >> 2, mu = pm & 3;
  const double2* u64 = U64 + (long)pm * 9 * Vh + cb;
  const SiteCoords c = cb_to_site(g, cb, par);
  int wrap, j = 0;
#pragma unroll
  for (int m = 0; m < 4; ++m)
    if (m == mu) j = neighbour_index(g, c, m, +1, &wrap) >> 1;
  int4* wf = W + (((long)par * nsb + cb / kSB) * 8 + 2 * mu) * kHopUnits + cb % kSB;
  int4* wb = W + (((long)(1 - par) * nsb + j / kSB) * 8 + 2 * mu + 1) * kHopUnits + j % kSB;
  float row[3] = {0.f, 0.f, 0.f}, col[3] = {0.f, 0.f, 0.f};
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const double2 u = u64[k * Vh];
    const float x = (float)u.x, y = (float)u.y, n = fmaf(x, x, y * y);
    row[k / 3] += n;
    col[k % 3] += n;
    const Part re = link_part(u.x), im = link_part(u.y);
    ok = ok && (re.h || re.l != 0.f || u.x == 0.0) && (im.h || im.l != 0.f || u.y == 0.0);  // not lost
    wf[k * kSB] = make_int4(re.h, __float_as_int(re.l), im.h, __float_as_int(im.l));
    wb[((k % 3) * 3 + k / 3) * kSB] = make_int4(re.h, __float_as_int(re.l), -im.h, __float_as_int(-im.l));
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    constexpr float lo = (float)(kNormMin * kNormMin), hi = (float)(kNormMax * kNormMax);
    ok = ok && row[k] >= lo && row[k] <= hi && col[k] >= lo && col[k] <= hi;
  }
  if (!ok) *flag = 1;
}

struct FxLaunch {
  HA args;
  const int4* links;
  FxField F, O;
  bool fx_out;
  cudaStream_t st;
};

template <int MINB>
void launch_fx(FxLaunch* L) {
  const HA& A = L->args;
  constexpr int block = 32 * kWarps;
  constexpr size_t smem = sizeof(FxShared);
  const unsigned sblocks = (unsigned)((A.g.Vh + kWarps * kSB - 1) / (kWarps * kSB));
  if (A.red == 1)
    launch_k(k_hop_fx_red<MINB, 1>, sblocks, block, smem, L->st, A, L->links, L->F);
  else if (A.red == 2)
    launch_k(k_hop_fx_red<MINB, 2>, sblocks, block, smem, L->st, A, L->links, L->F);
  else if (L->fx_out)
    launch_k(k_hop_fx<MINB, 1>, sblocks * (unsigned)A.ntiles, block, smem, L->st, A, L->links, L->F, L->O);
  else
    launch_k(k_hop_fx<MINB, 0>, sblocks * (unsigned)A.ntiles, block, smem, L->st, A, L->links, L->F, L->O);
}

// cfg.tile: blocks per SM that the registers are bounded for (5: 96 registers, 20 warps, 52 to 144 bytes of spill
// stores; 4: 128, 16 warps, 40 to 68 bytes; within 2% of each other where HBM bounds them, 4 is 10% faster on a few
// hundred sites.  6 and 7 took 0.345 and 0.376 ms against 0.315 at 32^3 x 64, before the sums of magnitudes)
void run_fx(void* ctx, const LaunchCfg& cfg) {
  auto* L = (FxLaunch*)ctx;
  if (cfg.tile == 4)
    launch_fx<4>(L);
  else
    launch_fx<5>(L);
}

SpinorView<P64> fx_view(const Field& f) {
  SpinorView<P64> v;
  v.p = (double2*)f.data;
  v.norm = nullptr;
  v.stride = f.nsites();
  return v;
}

bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  QCD_CK(cudaStreamIsCapturing(st, &cs));
  return cs != cudaStreamCaptureStatusNone;
}

// A scratch field of the handle; not allocated while the solver captures its iterations, which then run
// without it as the uncaptured first one did.
FxField fx_scratch(qcd_gauge* g, const char* name, const Field& like, cudaStream_t st) {
  const long nsb = (like.Vh + kSB - 1) / kSB, nq = (long)like.ls * like.nrhs;
  const size_t data = (size_t)nq * nsb * kSiteUnits * sizeof(int4), exps = (size_t)nq * nsb * kSB * sizeof(int);
  char* p = (char*)g->ws.find(name, data + exps);
  if (!p) {
    if (capturing(st)) raise(QCD_ERR_OOM, "no scratch for the fixed-point stencil");
    p = (char*)g->ws.get(name, data + exps);
  }
  return {(int4*)p, (int*)(p + data), nsb};
}

void fx_pack(const Field& in, const FxField& out, cudaStream_t st, const int* stop) {
  launch_k(k_to_fx, dim3((unsigned)((in.Vh + 127) / 128), (unsigned)(in.ls * in.nrhs)), 128, 0, st,
           (const int4*)in.data, in.nsites(), out, (int)in.Vh, in.ls, stop);
  QCD_LAUNCH_CK();
}

void fx_args(HA& A, const qcd_gauge* gh, const Field& shape, int out_parity, int dagger, double a) {
  A.g = make_geom(gh->lat.L, gh->lat.bc, gh->lat.V, gh->lat.Vh);
  A.out_parity = out_parity;
  A.ls = shape.ls;
  A.d_ls = make_fastdiv((unsigned)shape.ls);
  A.nslices = A.ntiles = shape.ls * shape.nrhs;
  A.d_ntiles = make_fastdiv((unsigned)A.ntiles);
  A.dagger = dagger;
  A.a = a;
  A.U.p = (const double2*)gh->U64;
  A.U.Vh = gh->lat.Vh;
  A.in = {nullptr, nullptr, 0};  // no FP64 form of the input
}
SpinorView<P64> canon_view(const double2* p) { return {const_cast<double2*>(p), nullptr, 1}; }

// out = [x +] a H in (out FP64), or the fixed-point field fout = H in (a = 1, x null); src: the FP64 form of `in`
void fx_launch(const qcd_gauge* gh, const FxField& in, const SpinorView<P64>* src, const Field& shape, Field* out, const FxField* fout,
               int out_parity, int dagger, double a, const Field* x, cudaStream_t st, const int* stop,
               const RedSpec* red) {
  FxLaunch L;
  HA& A = L.args;
  A.red = 0;
  A.partial = A.gpartial = nullptr;
  A.counters = A.npartial = nullptr;
  if (red && red->mode) {
    if (!x || (red->mode == 1 && !red->rt) || shape.nrhs * shape.ls > 1)
      raise(QCD_ERR_ARG, "fused reductions in FP64 need one slice and an x term");
    A.red = red->mode;
    A.partial = red->partial;
    A.gpartial = red->gpartial;
    A.counters = red->counters;
    A.npartial = red->npartial;
  }
  fx_args(A, gh, shape, out_parity, dagger, a);
  A.xpay = x != nullptr;
  A.out = out ? fx_view(*out) : fx_view(shape);
  if (src) A.in = *src;
  A.x = x ? fx_view(*x) : A.out;
  A.rt = red && red->rt ? fx_view(*red->rt) : A.out;
  A.stop = stop;
  L.links = (const int4*)gh->Ufx;
  L.F = in;
  L.O = fout ? *fout : in;
  L.fx_out = fout != nullptr;
  L.st = st;
  static std::atomic<unsigned long long> attr_mask{0};
  if (first_use_on_device(attr_mask))
    for (const void* k : {(const void*)k_hop_fx<4, 0>, (const void*)k_hop_fx<4, 1>, (const void*)k_hop_fx<5, 0>,
                          (const void*)k_hop_fx<5, 1>, (const void*)k_hop_fx_red<4, 1>, (const void*)k_hop_fx_red<4, 2>,
                          (const void*)k_hop_fx_red<5, 1>, (const void*)k_hop_fx_red<5, 2>})
      QCD_CK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FxShared)));
  const std::vector<LaunchCfg> cands = {{32 * kWarps, 5}, {32 * kWarps, 4}};
  char key[160];
  snprintf(key, sizeof key, "hopfx L%dx%dx%dx%d ns%d xp%d red%d out%d", gh->lat.L[0], gh->lat.L[1], gh->lat.L[2],
           gh->lat.L[3], A.nslices, A.xpay, A.red, (int)L.fx_out);
  LaunchCfg cfg = tune(key, cands, &run_fx, &L, st, true, stop);
  run_fx(&L, cfg);
  QCD_LAUNCH_CK();
}

// The scratch fields belong to the handle, and calls on device buffers are asynchronous on the caller's
// stream.  A stream has a set of its own while there are sets (kFxSets); another stream that takes it over waits for the
// event of its last use.  Streams are told apart by their ids: the address may be that of a stream that was destroyed
// with its work pending, or cudaStreamPerThread, one address for every thread's (which always waits).  The solver's
// own use is recorded when another stream follows.
class FxOrder {
 public:
  FxOrder(qcd_gauge* g, cudaStream_t st) : g_(g), st_(st), set_(g->fx_set[pick(g, st, &same_)]) {
    if (!set_.done) QCD_CK(cudaEventCreateWithFlags(&set_.done, cudaEventDisableTiming));
    if (!set_.used || (set_.on_work ? st == g->work : same_)) return;
    if (set_.on_work) QCD_CK(cudaEventRecord(set_.done, g->work));
    QCD_CK(cudaStreamWaitEvent(st, set_.done, 0));
  }
  ~FxOrder() {
    set_.used = true;
    set_.on_work = st_ == g_->work;
    if (!set_.on_work) cudaEventRecord(set_.done, st_);
  }
  FxOrder(const FxOrder&) = delete;
  FxOrder& operator=(const FxOrder&) = delete;
  // scratch field 'a' or 'b' of the set
  FxField field(char which, const Field& like) const {
    const char name[] = {'o', 'p', 't', '.', 'f', 'x', '.', which, (char)('0' + (&set_ - g_->fx_set)), 0};
    return fx_scratch(g_, name, like, st_);
  }

 private:
  // *same: the set's last use, if not by the solver, was on this very stream
  static int pick(qcd_gauge* g, cudaStream_t st, bool* same) {
    *same = false;
    if (st == g->work) return 0;
    unsigned long long id = 0;
    QCD_CK(cudaStreamGetId(st, &id));
    for (int k = 0; k < qcd_gauge::kFxSets; ++k)
      if (!g->fx_set[k].owned || g->fx_set[k].owner == id) {
        *same = g->fx_set[k].owned && st != cudaStreamPerThread;
        g->fx_set[k].owned = true;
        g->fx_set[k].owner = id;
        return k;
      }
    const int k = g->fx_next++ % qcd_gauge::kFxSets;
    g->fx_set[k].owner = id;
    return k;
  }
  qcd_gauge* g_;
  cudaStream_t st_;
  bool same_ = false;
  qcd_gauge::FxSet& set_;
};

// Whether the fixed-point path may run on `st`: never under a caller's stream capture (a graph that
// outlives the call must not hold the handle's scratch).
bool fx_usable(const qcd_gauge* g, cudaStream_t st) {
  if (!g->fx_ok) return false;
  return st == g->work || !capturing(st);
}

}  // namespace

size_t fx_link_bytes(const Lattice& lat) { return (size_t)2 * ((lat.Vh + kSB - 1) / kSB) * 8 * kHopUnits * sizeof(int4); }

void links_to_fx(qcd_gauge* g, int* flag, cudaStream_t st) {
  const long n = 8 * g->lat.Vh;
  QCD_CK(cudaMemsetAsync(flag, 0, sizeof(int), st));
  k_links_fx<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(make_geom(g->lat.L, g->lat.bc, g->lat.V, g->lat.Vh),
                                                         (const double2*)g->U64, (int4*)g->Ufx, (g->lat.Vh + kSB - 1) / kSB, flag);
  QCD_LAUNCH_CK();
}

bool hop_fx(const qcd_gauge* gh, const Field& in, Field& out, int out_parity, int dagger, double a, const Field* x,
            cudaStream_t st, const int* stop, const RedSpec* red) {
  if (!fx_usable(gh, st)) return false;
  qcd_gauge* g = const_cast<qcd_gauge*>(gh);
  FxOrder order(g, st);
  FxField f;
  try {
    f = order.field('a', in);
  } catch (const Error& e) {
    if (e.status != QCD_ERR_OOM) throw;
    return false;
  }
  fx_pack(in, f, st, stop);
  const SpinorView<P64> src = fx_view(in);
  fx_launch(g, f, &src, in, &out, nullptr, out_parity, dagger, a, x, st, stop, red);
  return true;
}

bool mhat_fx(const qcd_gauge* gh, const Field& in, Field& out, int dagger, double k2, cudaStream_t st, const int* stop,
             const RedSpec* red) {
  if (!fx_usable(gh, st)) return false;
  qcd_gauge* g = const_cast<qcd_gauge*>(gh);
  FxOrder order(g, st);
  FxField f, t;
  try {
    f = order.field('a', in);
    t = order.field('b', in);
  } catch (const Error& e) {
    if (e.status != QCD_ERR_OOM) throw;
    return false;
  }
  fx_pack(in, f, st, stop);
  const SpinorView<P64> src = fx_view(in);
  fx_launch(g, f, &src, in, nullptr, &t, 1, dagger, 1.0, nullptr, st, stop, nullptr);
  fx_launch(g, t, nullptr, in, &out, nullptr, 0, dagger, -k2, &in, st, stop, red);
  return true;
}

bool outer_fx_ready(const qcd_gauge* gh, const Field& shape, cudaStream_t st) {
  if (!fx_usable(gh, st)) return false;
  qcd_gauge* g = const_cast<qcd_gauge*>(gh);
  try {
    FxOrder order(g, st);
    order.field('a', shape);
    order.field('b', shape);
    const size_t nb = (size_t)(shape.Vh + kWarps * kSB - 1) / (kWarps * kSB);
    g->ws.get("opt.fx.sums", sizeof(double) * 4 * nb * shape.nrhs);
  } catch (const Error& e) {
    if (e.status != QCD_ERR_OOM) throw;
    return false;
  }
  return true;
}

void outer_fx(const qcd_gauge* gh, const OuterStep& o, cudaStream_t st) {
  qcd_gauge* g = const_cast<qcd_gauge*>(gh);
  const Field& shape = o.x;
  FxOrder order(g, st);
  const FxField fa = order.field('a', shape), fb = order.field('b', shape);
  const unsigned nb = (unsigned)((shape.Vh + kWarps * kSB - 1) / (kWarps * kSB)), n = (unsigned)shape.nrhs;
  double* partial = (double*)g->ws.get("opt.fx.sums", sizeof(double) * 4 * nb * n);
  const int4* links = (const int4*)g->Ufx;
  static std::atomic<unsigned long long> attr_mask{0};
  if (first_use_on_device(attr_mask))
    for (const void* k : {(const void*)k_outer_odd, (const void*)k_outer_res<P64>, (const void*)k_outer_res<P32>,
                          (const void*)k_outer_res<P16>})
      QCD_CK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FxShared)));
  const dim3 sites((unsigned)((shape.Vh + 127) / 128), n);
  if (o.x_zero) {
    fx_pack(o.b_o, fb, st, nullptr);  // x_o = b_o
  } else {
    SpinorView<P32> xin{};
    if (o.xin) xin = {(float4*)o.xin->data, nullptr, o.xin->nsites()};
    launch_k(k_outer_x, sites, 128, 0, st, fx_view(o.x), xin, (int)(o.xin != nullptr), fa, (int)shape.Vh);
    QCD_LAUNCH_CK();
    HA A;
    fx_args(A, g, shape, 1, o.dagger, o.kappa);
    A.stop = nullptr;
    A.partial = partial;
    A.in = fx_view(o.x);
    A.x = fx_view(o.b_o);
    A.out = fx_view(o.x_o);
    launch_k(k_outer_odd, nb * n, 32 * kWarps, sizeof(FxShared), st, A, links, fa, fb);
    QCD_LAUNCH_CK();
  }
  HA A;
  fx_args(A, g, shape, 0, o.dagger, o.kappa);
  A.stop = nullptr;
  A.partial = partial;
  A.xpay = o.x_zero ? 1 : 2;
  A.in = fx_view(o.x_zero ? o.b_o : o.x_o);
  A.rt = fx_view(o.b_e);
  A.x = fx_view(o.x);
  if (o.r.prec == QCD_F64) {
    launch_k(k_outer_res<P64>, nb * n, 32 * kWarps, sizeof(FxShared), st, A, links, fb, fx_view(o.r));
  } else if (o.r.prec == QCD_F32) {
    const SpinorView<P32> r{(float4*)o.r.data, nullptr, o.r.nsites()};
    launch_k(k_outer_res<P32>, nb * n, 32 * kWarps, sizeof(FxShared), st, A, links, fb, r);
  } else {
    const SpinorView<P16> r{(uint4*)o.r.data, o.r.norm, o.r.nsites()};
    launch_k(k_outer_res<P16>, nb * n, 32 * kWarps, sizeof(FxShared), st, A, links, fb, r);
  }
  QCD_LAUNCH_CK();
  launch_k(k_outer_sums, n, 256, 0, st, partial, (int)nb, o.sums, o.sums_stride, (int)!o.x_zero);
  QCD_LAUNCH_CK();
}

bool canon_fx(const qcd_gauge* gh, const qcd_fermion& f, int op, const double* in, double* out, int nrhs,
              cudaStream_t st) {
  if (!fx_usable(gh, st)) return false;
  qcd_gauge* g = const_cast<qcd_gauge*>(gh);
  Field shape;
  shape.prec = QCD_F64;
  shape.Vh = g->lat.Vh;
  shape.nrhs = nrhs;
  FxOrder order(g, st);
  FxField fa, fb;
  try {
    fa = order.field('a', shape);
    fb = order.field('b', shape);
  } catch (const Error& e) {
    if (e.status != QCD_ERR_OOM) throw;
    return false;
  }
  static std::atomic<unsigned long long> attr_mask{0};
  if (first_use_on_device(attr_mask))
    QCD_CK(cudaFuncSetAttribute(k_hop_fx_canon, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FxShared)));
  const Geom geom = make_geom(g->lat.L, g->lat.bc, g->lat.V, g->lat.Vh);
  const unsigned nb = (unsigned)((shape.Vh + kWarps * kSB - 1) / (kWarps * kSB)), n = (unsigned)nrhs;
  const double2 *src = (const double2*)in;
  const bool full = op == QCD_OP_FULL || op == QCD_OP_FULL_DAG, mhat = op == QCD_OP_MHAT || op == QCD_OP_MHAT_DAG;
  const int dagger = op == QCD_OP_FULL_DAG || op == QCD_OP_MHAT_DAG;
  // fixed-point halves: both for FULL (even in fa, odd in fb), else the one that the operator reads, in fa
  const int p0 = full || mhat || op == QCD_OP_D_OE ? 0 : 1;
  launch_k(k_canon_to_fx, dim3((unsigned)((shape.Vh + 127) / 128), n, full ? 2 : 1), 128, 0, st, geom, src,
           fa, full ? fb : fa, p0);
  QCD_LAUNCH_CK();
  const SpinorView<P64> cv = canon_view(src);
  auto hop = [&](const FxField& from, bool converted, int out_parity, double a, bool xpay, bool zero) {
    HA A;
    fx_args(A, g, shape, out_parity, dagger, a);
    if (converted) A.in = cv;
    A.stop = nullptr;
    A.xpay = xpay;
    launch_k(k_hop_fx_canon, nb * n, 32 * kWarps, sizeof(FxShared), st, A, (const int4*)g->Ufx, from, src,
             (double2*)out, (int)zero);
    QCD_LAUNCH_CK();
  };
  if (full) {
    hop(fb, true, 0, -f.kappa, true, false);
    hop(fa, true, 1, -f.kappa, true, false);
  } else if (mhat) {
    fx_launch(g, fa, &cv, shape, nullptr, &fb, 1, dagger, 1.0, nullptr, st, nullptr, nullptr);
    hop(fb, false, 0, -f.kappa * f.kappa, true, true);
  } else {
    hop(fa, true, op == QCD_OP_D_OE, 1.0, false, true);
  }
  return true;
}

}  // namespace qcd
