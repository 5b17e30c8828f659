// Molecular-dynamics updates of the gauge field and its momenta (the ensemble
// generation that consumes the solver, Sec. II A): momenta P_mu(x) in su(3)
// (traceless anti-Hermitian 3x3), links advanced as U <- exp(eps P) U, momenta as
// P <- P + c F with F the projected force, and the kinetic term sum |P_ab|^2.
// All on canonical complex128 arrays of 3x3 matrices, one thread per matrix.
#include <vector>

#include "common.cuh"
#include "internal.h"

namespace qcd {

namespace {

constexpr int kThreads = 128;

// c = c0 + a b
__device__ __forceinline__ void mat_madd(const Cx<double> a[9], const Cx<double> b[9], const Cx<double> c0[9],
                                         Cx<double> c[9]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      Cx<double> acc = c0[i * 3 + j];
#pragma unroll
      for (int k = 0; k < 3; ++k) acc = cmadd(a[i * 3 + k], b[k * 3 + j], acc);
      c[i * 3 + j] = acc;
    }
}

// exp(A) - 1 for a 3x3 complex matrix: A / 2^s of Frobenius norm <= 1/2, its Taylor series in Horner form
// modulo the characteristic polynomial, A^3 = t A^2 - c A + d (Cayley-Hamilton), then s squarings (1 + F)^2 = 1 + (2 F + F^2).  With
// E = e0 + e1 A + e2 A^2 a Horner step 1 + (A / n) E is three scalar recurrences (18 FP64
// operations instead of the 108 of a matrix product); 16 terms reach (1/2)^17 / 17! < 3e-20, and 11
// reach 0.1^12 / 12! < 3e-21 for the small steps that molecular dynamics takes.  The 1 stays apart so that U + F U
// rounds U once.  Bound by the FP64 pipe: 262144 links 0.88 ms with 13 matrix products, 0.30 ms here.
__constant__ double c_inv[17] = {0.0,       1.0,       1.0 / 2,  1.0 / 3,  1.0 / 4,  1.0 / 5,  1.0 / 6,  1.0 / 7, 1.0 / 8,
                                 1.0 / 9,  1.0 / 10, 1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16};

__device__ void mat_expm1(const Cx<double> a_in[9], Cx<double> e[9]) {
  double n2 = 0.0;
#pragma unroll
  for (int k = 0; k < 9; ++k) n2 = fma(a_in[k].re, a_in[k].re, fma(a_in[k].im, a_in[k].im, n2));
  int s = 0;
  while (n2 > 0.25 && s < 60) {
    n2 *= 0.25;
    ++s;
  }
  Cx<double> a[9], b[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) a[k] = a_in[k];
  if (s) {
    const double sc = ldexp(1.0, -s);
#pragma unroll
    for (int k = 0; k < 9; ++k) a[k] = {a[k].re * sc, a[k].im * sc};
  }
  const Cx<double> zero[9] = {};
  mat_madd(a, a, zero, b);
  // t = tr A, c = (t^2 - tr A^2) / 2, d = det A
  const Cx<double> t = a[0] + a[4] + a[8], t2 = cmul(t, t), tr2 = b[0] + b[4] + b[8];
  const Cx<double> c = {0.5 * (t2.re - tr2.re), 0.5 * (t2.im - tr2.im)};
  auto minor = [&](int p, int q, int r, int u) { return cmadd(a[p], a[u], -cmul(a[q], a[r])); };
  const Cx<double> d = cmadd(a[0], minor(4, 5, 7, 8), cmadd(a[1], minor(5, 3, 8, 6), cmul(a[2], minor(3, 4, 6, 7))));
  Cx<double> e0 = {1.0, 0.0}, e1 = {0.0, 0.0}, e2 = {0.0, 0.0};
  for (int n = n2 > 0.01 ? 16 : 11; n >= 1; --n) {
    const double inv = c_inv[n];
    const Cx<double> f = {inv * e2.re, inv * e2.im};
    const Cx<double> g1 = {inv * e0.re, inv * e0.im}, g2 = {inv * e1.re, inv * e1.im};
    e0 = cmadd(f, d, Cx<double>{n > 1 ? 1.0 : 0.0, 0.0});
    e1 = cmadd(-f, c, g1);
    e2 = cmadd(f, t, g2);
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    e[k] = cmadd(e1, a[k], cmul(e2, b[k]));
    if (k % 4 == 0) e[k] = e[k] + e0;
  }
  for (int i = 0; i < s; ++i) {
#pragma unroll
    for (int k = 0; k < 9; ++k) a[k] = {2.0 * e[k].re, 2.0 * e[k].im};
    mat_madd(e, e, a, b);
#pragma unroll
    for (int k = 0; k < 9; ++k) e[k] = b[k];
  }
}

__global__ void k_link_update(double2* __restrict__ U, const double2* __restrict__ P, double eps, long n) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  Cx<double> a[9], e[9], u[9], o[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const double2 p = P[i * 9 + k], v = U[i * 9 + k];
    a[k] = {eps * p.x, eps * p.y};
    u[k] = {v.x, v.y};
  }
  mat_expm1(a, e);
  const Cx<double> zero[9] = {};
  mat_madd(e, u, zero, o);
#pragma unroll
  for (int k = 0; k < 9; ++k) o[k] = u[k] + o[k];
#pragma unroll
  for (int k = 0; k < 9; ++k) U[i * 9 + k] = make_double2(o[k].re, o[k].im);
}

// P += c F over n complex entries
__global__ void k_mom_update(double2* __restrict__ P, const double2* __restrict__ F, double c, long n) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const double2 p = P[i], f = F[i];
    P[i] = make_double2(fma(c, f.x, p.x), fma(c, f.y, p.y));
  }
}

constexpr int kEnergyBlocks = 512;
__device__ double g_energy_partial[kEnergyBlocks];

// partial sums of |P_ab|^2 (fixed grid and order: the result does not depend on scheduling)
__global__ void k_mom_energy(const double2* __restrict__ P, long n) {
  double acc[1] = {0.0};
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const double2 p = P[i];
    acc[0] = fma(p.x, p.x, fma(p.y, p.y, acc[0]));
  }
  block_sum<1>(acc);
  if (threadIdx.x == 0) g_energy_partial[blockIdx.x] = acc[0];
}

unsigned grid_for(long n) {
  long b = (n + kThreads - 1) / kThreads;
  long cap = 8L * sm_count();
  return (unsigned)(b < cap ? (b > 0 ? b : 1) : cap);
}

}  // namespace

void link_update_device(double* U, const double* P, double eps, long nlinks, cudaStream_t st) {
  if (nlinks == 0) return;
  k_link_update<<<(unsigned)((nlinks + kThreads - 1) / kThreads), kThreads, 0, st>>>((double2*)U,
                                                                                   (const double2*)P, eps, nlinks);
  QCD_LAUNCH_CK();
}

void mom_update_device(double* P, const double* F, double c, long nlinks, cudaStream_t st) {
  const long n = nlinks * 9;
  if (n == 0) return;
  k_mom_update<<<grid_for(n), kThreads, 0, st>>>((double2*)P, (const double2*)F, c, n);
  QCD_LAUNCH_CK();
}

double mom_energy_device(const double* P, long nlinks, cudaStream_t st) {
  const long n = nlinks * 9;
  k_mom_energy<<<kEnergyBlocks, kThreads, 0, st>>>((const double2*)P, n);
  QCD_LAUNCH_CK();
  std::vector<double> h(kEnergyBlocks);
  QCD_CK(cudaMemcpyFromSymbolAsync(h.data(), g_energy_partial, sizeof(double) * kEnergyBlocks, 0,
                                   cudaMemcpyDeviceToHost, st));
  QCD_CK(cudaStreamSynchronize(st));
  double s = 0.0;
  for (double v : h) s += v;
  return s;
}

}  // namespace qcd
