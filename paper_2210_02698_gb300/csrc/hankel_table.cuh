// hankel_table.cuh - H0^(1)(x) and x H1^(1)(x) of x^2 in FP64 from local
// Taylor expansions, for the kernels that evaluate every matrix entry
// (Eq. termf; the entry is v0 f0 + v1 f1 with tau^2 interpolated, so the
// argument arrives as x^2 = omega^2 tau^2 and no square root is needed
// beyond a single-precision one that picks the expansion).
//
// FP64 is the scarce unit on this part (two FMAs a cycle and SM, 1.25 TFLOP/s):
// Miller's recurrence or the asymptotic series take 250 to 900 FP64
// operations an entry, this takes 28 and one 240-byte row read through L1/L2.
//
// Expansion.  Row k holds the expansion about x0 = k / HT_PER in
// u = (x^2 - x0^2) / (2 x0), |u| <= 1/128 or so:
//   F(u) = H0(x) = sum f_n u^n,   G(u) = x H1(x) = sum g_n u^n,
// and from H0' = -H1, (x H1)' = x H0 (DLMF 10.6.2, 10.6.6), with
// x^2 = x0^2 + 2 x0 u:  G' = x0 F,  (x0 + 2u) F' = -G, hence
//   g_{n+1} = x0 f_n / (n+1),   f_{n+1} = -(g_n + 2 n f_n) / (x0 (n+1)).
// Terms past u^6 are below 4e-19.  Rows cover x in [2, top]; below 2 the
// ascending series (DLMF 10.2.2, 10.8.1) in z = x^2 / 4 <= 1, twelve terms;
// past the table Hankel's expansion (bessel.cuh).
#pragma once
#include "bessel.cuh"

namespace hb {

constexpr int HT_PER = 64;          // rows per unit of x
constexpr int HT_ORDER = 7;         // coefficients per function
constexpr int HT_ROW = 1 + 2 * HT_ORDER;   // double2 per row: (x0^2, 1/(2 x0)), f_0.., g_0..
constexpr double HT_LO = 2.0;
constexpr double HT_CAP = 2048.0;   // largest x tabulated (31 MB)

struct HankelTable {
  const double2* rows;   // row k at (k - HT_LO HT_PER) HT_ROW
  float top;             // x below which rows exist (0: none)
};

// H0 and x H1 at a row's centre, 2 <= x < 25, by Miller's recurrence and
// Neumann's series as in bessel.cuh but in double-double arithmetic
// (Dekker 1971, products by fused multiply-adds): a row's value errs for every
// entry near it alike, so sums do not average it.  Error of the rows' values
// between 8 and 25: 9e-16 by the recurrence in double, 8e-17 by this.
struct DD {
  double h, l;
};
HB_HD DD dd_norm(double a, double b) {   // |a| >= |b|
  const double s = a + b;
  return DD{s, b - (s - a)};
}
HB_HD DD dd_add(DD a, DD b) {
  const double s = a.h + b.h, v = s - a.h;
  return dd_norm(s, ((a.h - (s - v)) + (b.h - v)) + (a.l + b.l));
}
HB_HD DD dd_mul(DD a, DD b) {
  const double p = a.h * b.h;
  return dd_norm(p, fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
HB_HD DD dd_neg(DD a) { return DD{-a.h, -a.l}; }
HB_HD DD dd_div(DD a, DD b) {
  const double q = a.h / b.h;
  const DD r = dd_add(a, dd_neg(dd_mul(DD{q, 0.0}, b)));
  return dd_norm(q, r.h / b.h);
}
HB_HD void hankel_row_near(double x, double* f, double* g) {
  const int M = 2 * (int)(0.8 * x + 22.0);
  const DD two_over_x = dd_div(DD{2.0, 0.0}, DD{x, 0.0});
  DD up{0.0, 0.0}, t{1e-30, 0.0}, norm{0.0, 0.0}, y0{0.0, 0.0}, y1{0.0, 0.0}, j1{0.0, 0.0};
  for (int n = M; n >= 1; --n) {
    const int k = (n + 1) >> 1;
    if ((n & 1) == 0) {
      norm = dd_add(norm, DD{2.0 * t.h, 2.0 * t.l});
      const DD q = dd_div(t, DD{(double)k, 0.0});
      y0 = dd_add(y0, (k & 1) ? dd_neg(q) : q);
    } else if (k >= 2) {
      const DD c = dd_mul(dd_div(DD{(double)(2 * k - 1), 0.0}, DD{(double)(k * (k - 1)), 0.0}), t);
      y1 = dd_add(y1, (k & 1) ? dd_neg(c) : c);
    } else {
      j1 = t;
    }
    const DD dn = dd_add(dd_mul(dd_mul(DD{(double)n, 0.0}, two_over_x), t), dd_neg(up));
    up = t;
    t = dn;
  }
  norm = dd_add(norm, t);
  const DD j0 = dd_div(t, norm);
  j1 = dd_div(j1, norm);
  y0 = dd_div(y0, norm);
  y1 = dd_div(y1, norm);
  const DD lg = dd_add(DD{log(0.5 * x), 0.0}, DD{HB_EULER_GAMMA, -4.942915152430645e-18});
  const DD two_pi{0.63661977236758138243, -3.9357353350364971764e-17};   // 2 / pi
  const DD a = dd_mul(two_pi, dd_add(dd_mul(lg, j0), DD{-2.0 * y0.h, -2.0 * y0.l}));
  const DD b = dd_mul(two_pi, dd_add(dd_add(dd_mul(dd_add(lg, DD{-1.0, 0.0}), j1), dd_neg(dd_div(j0, DD{x, 0.0}))), y1));
  const DD xg0 = dd_mul(DD{x, 0.0}, j1), xg1 = dd_mul(DD{x, 0.0}, b);
  f[0] = j0.h;
  f[1] = a.h;
  g[0] = xg0.h;
  g[1] = xg1.h;
}

#ifdef __CUDACC__
// Row of x0 = (first + blockIdx.x blockDim.x + threadIdx.x) / HT_PER.
static __global__ void hankel_table_kernel(double2* __restrict__ rows, int count) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= count) return;
  const double x0 = (HT_LO * HT_PER + q) / HT_PER;
  double2* r = rows + (size_t)q * HT_ROW;
  r[0] = make_double2(x0 * x0, 0.5 / x0);
  double fr, fi, gr, gi;
  if (x0 < HB_BESSEL_SWITCH) {
    double f[2], g[2];
    hankel_row_near(x0, f, g);
    fr = f[0], fi = f[1], gr = g[0], gi = g[1];
  } else {
    const Bessel01 b = bessel01_asym(x0);
    fr = b.j0, fi = b.y0, gr = x0 * b.j1, gi = x0 * b.y1;
  }
  for (int n = 0; n < HT_ORDER; ++n) {
    r[1 + n] = make_double2(fr, fi);
    r[1 + HT_ORDER + n] = make_double2(gr, gi);
    const double w = 1.0 / (x0 * (n + 1)), v = x0 / (n + 1);
    const double nfr = -(gr + 2.0 * n * fr) * w, nfi = -(gi + 2.0 * n * fi) * w;
    gr = v * fr;
    gi = v * fi;
    fr = nfr;
    fi = nfi;
  }
}

// Coefficients of the ascending series: (-1/4)^k times 1/(k!)^2, H_k/(k!)^2,
// 1/(k! (k+1)!) and (H_k + H_{k+1})/(k! (k+1)!), H_k the harmonic numbers.
constexpr int HS_N = 13;
struct HankelSeries {
  double a[HS_N], b[HS_N], c[HS_N], d[HS_N];
};
constexpr HankelSeries hankel_series_coefs() {
  HankelSeries r{};
  double f = 1.0, h = 0.0;   // (-1/4)^k / (k!)^2, H_k
  for (int k = 0; k < HS_N; ++k) {
    const double h1 = h + 1.0 / (k + 1);
    r.a[k] = f;
    r.b[k] = f * h;
    r.c[k] = f / (k + 1);
    r.d[k] = f / (k + 1) * (h + h1);
    f *= -0.25 / ((k + 1.0) * (k + 1.0));
    h = h1;
  }
  return r;
}

struct HankelFG {
  double2 F, G;   // H0, x H1
};

// Ascending series, 0 < s = x^2 < 4.
static __device__ __forceinline__ HankelFG hankel_series(double s) {
  constexpr HankelSeries S = hankel_series_coefs();
  double a = S.a[HS_N - 1], b = S.b[HS_N - 1], c = S.c[HS_N - 1], d = S.d[HS_N - 1];
#pragma unroll
  for (int k = HS_N - 2; k >= 0; --k) {
    a = fma(s, a, S.a[k]);
    b = fma(s, b, S.b[k]);
    c = fma(s, c, S.c[k]);
    d = fma(s, d, S.d[k]);
  }
  const double lg = 0.5 * log(0.25 * s) + HB_EULER_GAMMA;
  const double g0 = 0.5 * s * c;   // x J1
  HankelFG r;
  r.F = make_double2(a, (2.0 / HB_PI) * fma(lg, a, -b));
  r.G = make_double2(g0, (2.0 / HB_PI) * (fma(lg, g0, -1.0) - 0.25 * s * d));
  return r;
}

// x^2 = xx outside the rows (xx <= 0 as the limit the entries take there:
// x = 1e-12 for H0, a vanishing second term).
static __device__ __noinline__ HankelFG hankel_outside(double xx) {
  const double s = fmax(xx, 1e-24);
  HankelFG r;
  if (s < HT_LO * HT_LO + 0.1) {
    r = hankel_series(s);
    if (!(xx > 1e-24)) {
      const double q = sqrt(fmax(xx, 0.0)) * 1e12;
      r.G.x *= q;
      r.G.y *= q;
    }
    return r;
  }
  const double x = sqrt(s);
  const Bessel01 b = bessel01(x);
  r.F = make_double2(b.j0, b.y0);
  r.G = make_double2(x * b.j1, x * b.y1);
  return r;
}

// H0(x) and x H1(x) of x^2 = (w2 + w2l) t, omega^2 in two parts (rounded to
// one double it would shift the phase of far entries by x 2^-54, as much as
// everything else together).
static __device__ __forceinline__ HankelFG hankel_of_t2(const HankelTable& T, double w2, double w2l, double t) {
  const float xf = sqrtf(fmaxf((float)(w2 * t), 0.0f));
  if (!(xf >= (float)HT_LO && xf < T.top)) return hankel_outside(w2 * t);
  const int k = __float2int_rn(xf * HT_PER);
  const double2* __restrict__ r = T.rows + (size_t)(k - (int)(HT_LO * HT_PER)) * HT_ROW;
  const double2 h = __ldg(r);
  const double u = fma(w2l, t, fma(w2, t, -h.x)) * h.y;
  double2 f = __ldg(r + HT_ORDER), g = __ldg(r + 2 * HT_ORDER);
#pragma unroll
  for (int n = HT_ORDER - 2; n >= 0; --n) {
    const double2 a = __ldg(r + 1 + n), b = __ldg(r + 1 + HT_ORDER + n);
    f.x = fma(u, f.x, a.x);
    f.y = fma(u, f.y, a.y);
    g.x = fma(u, g.x, b.x);
    g.y = fma(u, g.y, b.y);
  }
  return HankelFG{f, g};
}
#endif

}  // namespace hb
