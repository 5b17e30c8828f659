"""The fixed-point arithmetic of the FP64 stencil (csrc/fixed.cuh) on the host: splitting a double into its parts,
and a hop sum formed as the stencil forms it, against extended precision and against FP64 multiply-adds."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1712_01505_gb300", "csrc")

SRC = r"""
#include <math.h>
#include <stdint.h>
#include <string.h>
#include <algorithm>
#include "fixed.cuh"
using namespace qcd::fx;
static unsigned hi_of(double v) { uint64_t b; memcpy(&b, &v, 8); return (unsigned)(b >> 32); }
static unsigned lo_of(double v) { uint64_t b; memcpy(&b, &v, 8); return (unsigned)b; }
static int field(double v) { return (hi_of(v) >> 20) & 0x7ff; }
extern "C" {
// part of v aligned to the exponent field e: h, and the value back
void split(double v, int e, int* h, float* l, double* back) {
  Part p = spinor_part(hi_of(v), lo_of(v), e);
  *h = p.h; *l = p.l; *back = part_value(p, e);
}
// the part of an integer sum, and its value in units of the sum
void sum_split(int64_t w, int shift, int* h, float* l, long double* back) {
  Part p = sum_part(w, shift);
  *h = p.h; *l = p.l;
  *back = ((long double)p.h + (long double)p.l) * powl(2.0L, shift);
}
// n independent sums over 8 hops of row . h (3 complex products), h = u + s l: u, l (n, 8, 3, 2), U (n, 8, 3, 2).
// Errors relative to rms(|sum|): [fixed, FP64] and the largest of each, against long double.
void hop_errors(long n, const double* U, const double* u, const double* l, double* out) {
  long double se = 0, sf = 0, s2 = 0;
  double me = 0, mf = 0;
  for (long i = 0; i < n; ++i) {
    int e[8], E = kEmin;
    for (int k = 0; k < 8; ++k) {
      e[k] = 0;
      for (int c = 0; c < 6; ++c) {
        e[k] = std::max(e[k], field(u[(i * 8 + k) * 6 + c]));
        e[k] = std::max(e[k], field(l[(i * 8 + k) * 6 + c]));
      }
      if (e[k] < kEmin) e[k] = kEmin;
      E = std::max(E, e[k]);
    }
    long double xr = 0, xi = 0;
    double fr = 0, fi = 0;
    int64_t vr = 0, vi = 0;
    for (int k = 0; k < 8; ++k) {
      const double* a = U + (i * 8 + k) * 6;
      const double* p = u + (i * 8 + k) * 6;
      const double* q = l + (i * 8 + k) * 6;
      const int s = k & 1 ? 1 : -1;
      int64_t Hr = 0, Hi = 0;
      float Cr = 0, Cn = 0, Ci = 0;
      double wr = 0, wi = 0;
      for (int c = 0; c < 3; ++c) {
        const double hr = p[2 * c] + s * q[2 * c], hi = p[2 * c + 1] + s * q[2 * c + 1];
        const long double yr = (long double)p[2 * c] + s * (long double)q[2 * c];
        const long double yi = (long double)p[2 * c + 1] + s * (long double)q[2 * c + 1];
        const long double ar = a[2 * c], ai = a[2 * c + 1];
        xr += ar * yr - ai * yi;
        xi += ar * yi + ai * yr;
        wr = fma(a[2 * c], hr, wr); wr = fma(-a[2 * c + 1], hi, wr);
        wi = fma(a[2 * c], hi, wi); wi = fma(a[2 * c + 1], hr, wi);
        const Part ur = link_part(a[2 * c]), ui = link_part(a[2 * c + 1]);
        const Part pr = spinor_part(hi_of(p[2 * c]), lo_of(p[2 * c]), e[k]), pi = spinor_part(hi_of(p[2 * c + 1]), lo_of(p[2 * c + 1]), e[k]);
        const Part qr = spinor_part(hi_of(q[2 * c]), lo_of(q[2 * c]), e[k]), qi = spinor_part(hi_of(q[2 * c + 1]), lo_of(q[2 * c + 1]), e[k]);
        const int gr = pr.h + s * qr.h, gi = pi.h + s * qi.h;
        const float lr = fmaf((float)s, qr.l, pr.l), li = fmaf((float)s, qi.l, pi.l);
        Hr += (int64_t)ur.h * gr; Hr -= (int64_t)ui.h * gi;
        Hi += (int64_t)ur.h * gi; Hi += (int64_t)ui.h * gr;
        Cr = fmaf((float)ur.h, lr, Cr); Cr = fmaf(ur.l, (float)gr, Cr);
        Cn = fmaf((float)ui.h, li, Cn); Cn = fmaf(ui.l, (float)gi, Cn);
        Ci = fmaf((float)ur.h, li, Ci); Ci = fmaf(ur.l, (float)gi, Ci);
        Ci = fmaf((float)ui.h, lr, Ci); Ci = fmaf(ui.l, (float)gr, Ci);
      }
      fr += wr; fi += wi;
      const int d3 = std::min(E - e[k], 100) + 3;
      auto sar = [](int64_t v, int d) { return d > 63 ? (v < 0 ? -1 : 0) : v >> d; };
      vr += sar(Hr, d3) + (int64_t)lrintf((Cr - Cn) * pow2f(-d3));
      vi += sar(Hi, d3) + (int64_t)lrintf(Ci * pow2f(-d3));
    }
    const double rr = ldexp((double)vr, E - 1079), ri = ldexp((double)vi, E - 1079);
    const long double size = sqrtl(xr * xr + xi * xi);
    long double d = hypotl(rr - xr, ri - xi), f = hypotl(fr - xr, fi - xi);
    se += d * d / (size * size); sf += f * f / (size * size); s2 += 1;
    me = std::max(me, (double)(d / size)); mf = std::max(mf, (double)(f / size));
  }
  out[0] = sqrt((double)(se / s2)); out[1] = sqrt((double)(sf / s2)); out[2] = me; out[3] = mf;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src, so = d / "fx.cpp", d / "libfx.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(so)],
                   check=True)
    lib = ctypes.CDLL(str(so))
    lib.split.argtypes = [ctypes.c_double, ctypes.c_int] + [ctypes.c_void_p] * 3
    lib.sum_split.argtypes = [ctypes.c_int64, ctypes.c_int] + [ctypes.c_void_p] * 3
    lib.hop_errors.argtypes = [ctypes.c_long] + [ctypes.c_void_p] * 4
    return lib


def _split(lib, v, e):
    h, l, b = ctypes.c_int(), ctypes.c_float(), ctypes.c_double()
    lib.split(float(v), int(e), ctypes.byref(h), ctypes.byref(l), ctypes.byref(b))
    return h.value, l.value, b.value


def test_parts_of_doubles(lib):
    """Exact for the largest component of a site; for the others the shift drops less than 2^-57 of 2^(e - 1022) and the
    FP32 remainder (26 bits in 24) is rounded by at most 2^-56 of it; |h| < 2^30."""
    rng = np.random.default_rng(3)
    vals = np.concatenate([rng.standard_normal(2000), [1.0, -1.0, 2.0 - 2.0 ** -52, -(2.0 - 2.0 ** -52), 2.0 ** -52, 0.0, -0.0]])
    for v in vals:
        f = int(np.frexp(v)[1]) + 1022 if v else 0
        for e in {max(f, 256), max(f, 256) + 1, max(f, 256) + 7, 1100}:
            if e < f:
                continue
            h, l, back = _split(lib, v, e)
            assert abs(h) < 2 ** 30 and abs(l) <= 1.0
            assert abs(back - v) <= (0.0 if e == f else 1.5 * 2.0 ** (e - 1022 - 56))
    for v in (5e-324, -1e-310):  # subnormal values beside a normal one vanish
        assert abs(_split(lib, v, 256)[0]) == 0


def test_parts_of_sums(lib):
    """|h| < 2^30 for every sum up to +-2^(30 + shift), value kept to 2^-24 of a unit of h."""
    rng = np.random.default_rng(4)
    for shift in (33, 31, 30, 25, 8, 1, 0, -4):
        top = 1 << (30 + shift)
        ws = [0, 1, -1, top - 1, -top, -(top - 1), top // 2, -(top // 2)] + [int(v * top) for v in rng.uniform(-1, 1, 500)]
        for w in ws:
            w = max(-top, min(top - 1, w))
            h, l, b = ctypes.c_int(), ctypes.c_float(), np.zeros(1, np.longdouble)
            lib.sum_split(w, shift, ctypes.byref(h), ctypes.byref(l), b.ctypes.data)
            assert abs(h.value) < 2 ** 30 and abs(l.value) <= 1.0, (w, shift)
            assert abs(b[0] - np.longdouble(w)) <= np.longdouble(2.0) ** (shift - 24), (w, shift)


@pytest.mark.parametrize("spread", [0.0, 0.5, 2.0])
def test_hop_sum_is_no_less_exact_than_fp64(lib, spread):
    """SU(3) rows on Gaussian spinors whose sites differ by factors exp(spread N(0, 1))."""
    rng = np.random.default_rng(5)
    n = 20000
    row = rng.standard_normal((n, 8, 3, 2))
    row /= np.sqrt((row ** 2).sum((2, 3), keepdims=True))
    amp = np.exp(spread * rng.standard_normal((n, 8, 1, 1)))
    u = np.ascontiguousarray(rng.standard_normal((n, 8, 3, 2)) * amp)
    l = np.ascontiguousarray(rng.standard_normal((n, 8, 3, 2)) * amp)
    out = np.zeros(4)
    lib.hop_errors(n, row.ctypes.data, u.ctypes.data, l.ctypes.data, out.ctypes.data)
    assert out[0] <= out[1] and out[2] <= 1.5 * out[3], out
