"""The fixed-point arithmetic of the 3D FP64 cell term and faces (fixed_point.cuh,
fixed_tables.cpp), compiled for the host: the cell operator against extended
precision and the conversions at the ends of the exponent range."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2507_17053_gb300", "csrc")

SRC = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <vector>
#include "setup.hpp"
using namespace sbm;
static uint64_t bits(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
static double val(uint64_t b) { double x; std::memcpy(&x, &b, 8); return x; }
static uint64_t rs = 7;
static double rnd() {            // splitmix64, U(-1,1)
  rs += 0x9E3779B97F4A7C15ull;
  uint64_t z = rs;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return 2.0 * (double)(z >> 11) * 0x1p-53 - 1.0;
}

template <int N>
int cell(double h) {
  constexpr int H = N / 2, HE = (N + 1) / 2, L = N * N, ND = L * N;
  constexpr int packed = (HE * (HE + 1) / 2 + H * (H + 1) / 2) | 1;
  Tables1D tb;
  build_tables(N - 1, &tb);
  FixedTables ft;
  if (!build_fixed_tables(tb, h, &ft)) { std::printf("n=%d h=%g: tables\n", N, h); return 1; }
  auto tri = [](int i, int j, int n) { return i * n - i * (i - 1) / 2 + (j - i); };
  auto sym = [&](int i, int j, int n) { return i <= j ? tri(i, j, n) : tri(j, i, n); };
  int bad = 0;
  for (int kind = 0; kind < 4; ++kind) {
    double num = 0, den = 0;
    for (int trial = 0; trial < 8; ++trial) {
      std::vector<double> x(ND);
      for (int c = 0; c < ND; ++c) {
        x[c] = rnd();
        if (kind == 1) x[c] *= std::pow(10.0, 3.0 * rnd() - 3.0);        // graded
        if (kind == 2) x[c] = rnd() > 0 ? 1.0 : -1.0;                    // the bounds
        if (kind == 3) x[c] = std::ldexp(1.0 + 0.01 * x[c], 500);        // near constant
      }
      // reference: sum over axes of M x .. K .. x M in long double
      std::vector<long double> ref(ND, 0), cur(ND), nx(ND);
      const int st[3] = {1, N, L};
      for (int k = 0; k < 3; ++k) {
        for (int c = 0; c < ND; ++c) cur[c] = x[c];
        for (int ax = 0; ax < 3; ++ax) {
          for (int c = 0; c < ND; ++c) {
            const int i = c / st[ax] % N;
            long double s = 0;
            for (int j = 0; j < N; ++j)
              s += (long double)(ax == k ? tb.K[i][j] : tb.M[i][j]) * cur[c + (j - i) * st[ax]];
            nx[c] = s;
          }
          cur = nx;
        }
        for (int c = 0; c < ND; ++c) ref[c] += (long double)h * cur[c];
      }
      uint32_t mx = 0;
      for (double v : x) mx = std::max(mx, fix::mag_hi(bits(v)));
      const int E = (int)(mx >> 20);
      std::vector<int64_t> q(ND);
      for (int c = 0; c < ND; ++c) q[c] = fix::from_double<false>(bits(x[c]), E);
      auto line = [&](int base, int s, auto f) {
        int64_t v[N], w[N];
        for (int j = 0; j < N; ++j) v[j] = q[base + j * s];
        f(v, w);
        for (int j = 0; j < N; ++j) {
          if (std::llabs(w[j]) > (1ll << 60) + 64) { std::printf("n=%d overflow\n", N); bad = 1; }
          q[base + j * s] = w[j];
        }
      };
      for (int l = 0; l < L; ++l)
        line(l, L, [&](auto& v, auto& w) { fix::to_modes<N, 0>(ft.Vt, v, w); });
      for (int l = 0; l < L; ++l)
        line(l % N + l / N * L, N, [&](auto& v, auto& w) { fix::to_modes<N, 0>(ft.Vt, v, w); });
      for (int l = 0; l < L; ++l) {
        const fix::Entry* m = ft.xline.data() + sym(l % N, l / N, N) * packed;
        line(l * N, 1, [&](auto& v, auto& w) {
          fix::apply_line<N, fix::shift_x(N)>(
              [&](int i, int j) { return m[sym(i, j, HE)]; },
              [&](int i, int j) { return m[HE * (HE + 1) / 2 + sym(i, j, H)]; }, v, w);
        });
      }
      for (int l = 0; l < L; ++l)
        line(l % N + l / N * L, N,
             [&](auto& v, auto& w) { fix::from_modes<N, fix::shift_y(N)>(ft.V, v, w); });
      for (int l = 0; l < L; ++l)
        line(l, L, [&](auto& v, auto& w) { fix::from_modes<N, fix::shift_z(N)>(ft.V, v, w); });
      long double big = 0;
      for (int c = 0; c < ND; ++c) big = std::max(big, (long double)std::fabs(x[c]));
      for (int c = 0; c < ND; ++c) {
        const double y = val(fix::to_double<false>(q[c], E + ft.eoff));
        const long double d = ((long double)y - ref[c]) / big;
        num = std::max(num, (double)std::fabs(d));
        den = std::max(den, (double)std::fabs(ref[c] / big));
      }
    }
    // backward-stable bound relative to |A| |x| (|A| by rows ~ 3 h max|K|), with the 1D
    // double tables' own rounding (about n ulps) that the reference shares
    double kmax = 0;
    for (int i = 0; i < N; ++i)
      for (int j = 0; j < N; ++j) kmax = std::max(kmax, std::fabs(tb.K[i][j]));
    const double tol = 8.0 * N * 0x1p-53 * 3.0 * h * kmax;
    if (!(num <= tol)) { std::printf("n=%d kind %d err %g tol %g\n", N, kind, num, tol); bad = 1; }
  }
  return bad;
}

static int conversions() {
  int bad = 0;
  const double inf = std::numeric_limits<double>::infinity();
  const double xs[] = {0.0, -0.0, 1.0, -1.0, 1.9999999999999998, -0x1.8p-7, 0x1.fffffffffffffp-3,
                       0x1.fffffffffffffp+1023, -0x1p-1022, 0x0.0000000000001p-1022,
                       -0x0.8000000000001p-1022, 0x1.23456789abcdep-1000, 0x1p+1000};
  for (double x : xs) {
    const int E = std::max(1, (int)(fix::mag_hi(bits(x)) >> 20));
    for (int d = 0; d < 8 && E + d < 0x7ff; ++d) {       // the cell's largest is 2^d larger
      const int64_t q = fix::from_double<true>(bits(x), E + d);
      const double y = val(fix::to_double<true>(q, E + d - 59));
      if (y != x) { std::printf("round trip %a (+%d): %a\n", x, d, y); bad = 1; }
      if (fix::plain_exp(E + d)) {
        const int64_t p = fix::from_double<false>(bits(x), E + d);
        if (p != q || val(fix::to_double<false>(p, E + d - 59)) != x) {
          std::printf("plain %a (+%d)\n", x, d);
          bad = 1;
        }
      }
    }
  }
  // values far below the largest round down; overflow gives infinity; ties away are nearest
  bad |= fix::from_double<false>(bits(1.0), 1023 + 60) != 0;
  bad |= fix::from_double<false>(bits(-1.0), 1023 + 200) != -1;
  bad |= fix::from_double<false>(bits(1.0), 1023 + 59) != 1;
  bad |= val(fix::to_double<true>(-(1ll << 60), 2046)) != -inf;
  bad |= val(fix::to_double<true>((1ll << 60), 1986)) != 0x1p+1023;
  bad |= val(fix::to_double<true>((1ll << 61) - 1, 1986)) != inf;
  bad |= val(fix::to_double<false>((1ll << 61) - 1, 963)) != 2.0;
  // both conversions of a result agree wherever the plain one is taken
  for (int eb = -2; eb <= 2050; ++eb) {
    if (fix::plain_result(eb) != (eb >= 1 && eb <= 1984)) bad = 1;
    if (!fix::plain_result(eb)) continue;
    for (long long q : {1ll, 3ll, (1ll << 52) - 1, (1ll << 53) + 1, 1ll << 60, (1ll << 61) + 512,
                        (1ll << 62) - 1})
      for (long long v : {q, -q})
        bad |= fix::to_double<false>(v, eb) != fix::to_double<true>(v, eb) ||
               !std::isnormal(val(fix::to_double<false>(v, eb)));
  }
  // the exponents' groups of lanes up to the last of 2^31 - 1 cells
  bad |= fix::group_of(1u << 24, 256, 0, 32) != 1ll << 27;
  bad |= fix::group_of((1u << 28) - 1, 256, 255, 32) != (1ll << 31) - 1;
  bad |= fix::group_of(7, 256, 9, 8) != 225;
  return bad;
}

// Products as entries against 128-bit arithmetic, over the exponents and at the ends.
static int products() {
  int bad = 0;
  auto mant = [](double x, int* e) {
    const double m = std::frexp(x, e);
    return (__int128)std::ldexp(m, 53);
  };
  for (int trial = 0; trial < 20000; ++trial) {
    double a = rnd(), b = rnd();
    if (trial % 3 == 1) a = std::ldexp(a, (int)(1000 * rnd()));
    if (trial % 5 == 1) b = std::ldexp(b, (int)(20 * rnd()));
    if (trial % 7 == 1) a = std::rint(8 * a) / 8;
    if (trial % 11 == 1) a = std::ldexp(a, -1040 - trial % 30);      // subnormal
    int e, ea, eb;
    std::frexp(a * b, &e);
    // a result of up to 61 bits, or far below one unit
    const int t = a == 0 || b == 0 ? 5 : (trial % 13 == 1 ? -20 - trial % 90 : 60) - e;
    const __int128 p = mant(a, &ea) * mant(b, &eb);
    const int sh = 106 - ea - eb - t;                                // a b 2^t = p 2^-sh
    __int128 want = 0;
    const __int128 m = p < 0 ? -p : p;
    if (sh <= 0) want = m << -sh;
    else if (sh < 120) want = (m + ((__int128)1 << (sh - 1))) >> sh;
    if (p < 0) want = -want;
    const fix::Entry q = fix::product(bits(a), bits(b), t);
    if ((__int128)q.h * (1ll << 30) + q.l / 2 != want || q.l % 2) {
      std::printf("product %a %a 2^%d\n", a, b, t);
      bad = 1;
    }
  }
  return bad;
}

// The faces' sums at their bounds (absolute sum of the products 2^61, values of +-2^57;
// overflow stops the program) against 128-bit sums, and the 1D face tables.
template <int N>
int faces() {
  int bad = 0;
  Tables1D tb;
  build_tables(N - 1, &tb);
  FixedTables ft;
  if (!build_fixed_tables(tb, 0.1, &ft)) return 1;
  for (int kind = 0; kind < 4; ++kind) {
    fix::Entry w[N * N];
    fix::Split x[N * N];
    int64_t A[N * N], q[N * N];
    for (int j = 0; j < N * N; ++j) {
      // equal magnitudes with the low part at its largest, or one dominant product
      const double m = std::ldexp(1.0 / (1.0 + 1e-6), 61);
      int64_t a = kind == 3 ? (j ? 1 : (int64_t)m - N * N) : (int64_t)(m / (N * N));
      if (kind < 3) a = ((a >> 30) << 30) - ((int64_t)1 << 29);
      if (kind == 1 && rnd() < 0) a = -a;
      A[j] = a;
      const int64_t h = (a + ((int64_t)1 << 29)) >> 30;
      w[j] = fix::Entry{(int32_t)h, (int32_t)(2 * (a - h * ((int64_t)1 << 30)))};
      const double v = kind == 2 ? -1.9999999999999998 : (A[j] < 0 ? -1.0 : 1.9999999999999998);
      q[j] = fix::from_double<false>(bits(v), 1023) >> 3;
      x[j] = fix::split(q[j]);
    }
    int64_t hi = 0, mid = (int64_t)1 << 27;
    __int128 ref = 0;
    for (int j = 0; j < N * N; ++j) {
      hi = fix::mad_wide(w[j].h, x[j].h, hi);
      mid = fix::mad_wide(w[j].h, x[j].l, mid);
      mid = fix::mad_wide(w[j].l, x[j].h, mid);
      ref += (__int128)A[j] * q[j];
    }
    const int64_t r = fix::shl_add<3>(hi, mid >> 28), e = (int64_t)(ref >> 58);
    // the dropped products l ql: below 2^61 N^2 in units of 2^-59 of r's
    if (std::llabs(r - e) > 2 + 8 * N * N || std::llabs(r) > (1ll << 60)) {
      std::printf("faces n=%d kind %d: %lld %lld\n", N, kind, (long long)r, (long long)e);
      bad = 1;
    }
    fix::Split y[N];
    for (int j = 0; j < N; ++j) y[j] = fix::split(j & 1 ? -(1ll << 60) : (1ll << 60));
    for (int i = 0; i < N; ++i) {
      // columns of S and of M, the row of D0 on 57-bit values
      auto S = [&](int j) { return ft.face[N + N * N + N * j + i]; };
      auto M = [&](int j) { return ft.face[N + N * j + i]; };
      bad |= std::llabs(fix::dot<0, N>(S, y)) > (1ll << 60);
      bad |= std::llabs(fix::dot<0, N>(M, y)) > (1ll << 60);
      for (int j = 0; j < N; ++j) {
        const int tS = 61 - (ft.face_eq - 2) / 2;
        const fix::Entry a = S(j);
        const double s = std::ldexp((double)a.h * 0x1p30 + 0.5 * a.l, -tS);
        // the double table: N - 1 factors of three roundings, |phi| <= 1
        if (std::fabs(s - tb.S[j][i]) > 3 * N * 0x1p-53) { std::printf("S n=%d %d %d\n", N, j, i); bad = 1; }
      }
    }
    fix::Split z[N];
    for (int j = 0; j < N; ++j) z[j] = fix::split(ft.face[j].h < 0 ? -(1ll << 57) : (1ll << 57));
    bad |= std::llabs(fix::dot<3, N>([&](int j) { return ft.face[j]; }, z)) > (1ll << 60);
  }
  return bad;
}

// The DG line operator K u + sum_s Own_s g_s at its bounds (57-bit values, every row's signs;
// overflow stops the program): below 2^59, and right against long double.
template <int N>
int dg_lines(double pen) {
  constexpr int H = N / 2;
  int bad = 0;
  Tables1D tb;
  build_tables(N - 1, &tb);
  FixedTables ft;
  if (!build_fixed_tables(tb, 1.0, &ft, pen)) return 1;
  const fix::DgTab& d = ft.dg;
  if (!ft.dg_pen_in) pen = 0.0;           // added elsewhere, in double
  auto Kf = [&](int i, int j) {           // the row's sign pattern from the folded blocks
    const fix::Entry e = d.K.E[std::min(i, N - 1 - i)][std::min(j, N - 1 - j)];
    if ((N & 1) && (i == H || j == H)) return (double)e.h;
    const fix::Entry o = d.K.O[std::min(i, N - 1 - i)][std::min(j, N - 1 - j)];
    return ((i < N - 1 - i) == (j < N - 1 - j)) ? (double)e.h + o.h : (double)e.h - o.h;
  };
  const int64_t B = (1ll << 57) - 1;
  // eoff = 2 - tR + 2 (61 - tM) (h = 1); tM from an entry of the face tables
  const fix::Entry m = ft.face[N];
  const int tM = (int)std::lround(std::log2(((double)m.h * 0x1p30 + 0.5 * m.l) / tb.M[0][0]));
  const int tR = 2 + 2 * (61 - tM) - d.eoff;
  for (int row = 0; row < N; ++row) {
    int64_t v[N], y[N], g[2][N], nb[2][N];
    for (int j = 0; j < N; ++j) v[j] = Kf(row, j) < 0 ? -B : B;
    for (int s = 0; s < 2; ++s)
      for (int j = 0; j < N; ++j) nb[s][N - 1 - j] = (row + j + s) % 3 == 2 ? v[j] : -v[j];
    fix::apply_line<N, 3>([&](int i, int j) { return d.K.E[i][j]; },
                          [&](int i, int j) { return d.K.O[i][j]; }, v, y);
    for (int s = 0; s < 2; ++s) {
      fix::Split q[N];
      for (int j = 0; j < N; ++j) {
        g[s][j] = v[j] - nb[s][N - 1 - j];
        q[j] = fix::split(g[s][j]);
      }
      y[s ? N - 1 : 0] += fix::dot<3, N>([&](int j) { return d.w[s ? N - 1 - j : j]; }, q);
    }
    const fix::Split e0 = fix::split(g[0][0]), e1 = fix::split(g[1][N - 1]);
    for (int j = 0; j < N; ++j) {
      const fix::Split q1[1] = {j ? e0 : e1}, q2[2] = {e0, e1};
      if (j == 0 || j == N - 1) y[j] += fix::dot<3, 1>([&](int) { return d.w[N - 1]; }, q1);
      else y[j] += fix::dot<3, 2>([&](int i) { return d.w[i ? N - 1 - j : j]; }, q2);
    }
    for (int i = 0; i < N; ++i) {
      long double r = 0;
      for (int j = 0; j < N; ++j) r += (long double)tb.K[i][j] * v[j];
      for (int s = 0; s < 2; ++s) {
        const int e = s ? N - 1 : 0;
        const long double sg = s ? 1 : -1;
        auto D = [&](int j) { return (long double)(s ? tb.D1[j] : tb.D0[j]); };
        long double dg = 0;
        for (int j = 0; j < N; ++j) dg += D(j) * g[s][j];
        if (i == e) r += pen * g[s][e] - 0.5L * sg * dg;
        r -= 0.5L * sg * D(i) * g[s][e];
      }
      // the double tables' rounding (16 N ulps of the terms, whose sum is below 2^59)
      bad |= std::llabs(y[i]) > (1ll << 59);
      if (std::fabs((long double)y[i] - std::ldexp(r, tR - 58)) > 16.0L * N * 0x1p6L) bad = 1;
    }
  }
  if (bad) std::printf("dg n=%d pen %g\n", N, pen);
  return bad;
}

// The 1D tables in long double: stiffness, end derivatives.
template <int N>
struct Exact {
  long double x[N], K[N][N] = {}, D[2][N];
  static void legendre(int m, long double t, long double* P, long double* dP) {
    long double p0 = 1, p1 = t;
    for (int k = 1; k < m; ++k) {
      const long double p2 = ((2 * k + 1) * t * p1 - k * p0) / (k + 1);
      p0 = p1;
      p1 = p2;
    }
    *P = p1;
    *dP = m * (p0 - t * p1) / (1 - t * t);
  }
  void lagrange(long double s, long double* dv) const {
    for (int j = 0; j < N; ++j) {
      long double a = 1, b = 0;
      for (int m = 0; m < N; ++m) {
        if (m == j) continue;
        b = (b * (s - x[m]) + a) / (x[j] - x[m]);
        a = a * (s - x[m]) / (x[j] - x[m]);
      }
      dv[j] = b;
    }
  }
  explicit Exact(const Tables1D& tb) {
    const int p = N - 1;
    for (int j = 0; j < N; ++j) {
      long double s = 2 * (long double)tb.nodes[j] - 1, L, d;
      for (int it = 0; it < 4 && j > 0 && j < p; ++it) {
        legendre(p, s, &L, &d);
        s -= d * (1 - s * s) / (2 * s * d - p * (p + 1) * L);
      }
      x[j] = (s + 1) / 2;
    }
    for (int q = 0; q < N; ++q) {
      long double s = 2 * (long double)tb.gpts[q] - 1, L, d, dv[N];
      for (int it = 0; it < 4; ++it) {
        legendre(N, s, &L, &d);
        s -= L / d;
      }
      legendre(N, s, &L, &d);
      lagrange((s + 1) / 2, dv);
      for (int i = 0; i < N; ++i)
        for (int j = 0; j < N; ++j) K[i][j] += dv[i] * dv[j] / ((1 - s * s) * d * d);
    }
    lagrange(0, D[0]);
    lagrange(1, D[1]);
  }
};

// The DG line operator on smooth lines whose traces match the neighbours': no penalty of
// any size may cost accuracy.  |error| <= 2^-52 B max |u|, B the largest row sum without
// penalty: the operator's is at most 2 B, inputs are cut at 2^-56 of max |u|, at most 8
// roundings at 2^-57 of the row sum follow.
template <int N>
int dg_matching(double pen) {
  int bad = 0;
  Tables1D tb;
  build_tables(N - 1, &tb);
  const Exact<N> T(tb);
  FixedTables ft;
  if (!build_fixed_tables(tb, 1.0, &ft, pen)) return 1;
  const fix::DgTab& d = ft.dg;
  const fix::Entry m = ft.face[N];        // tM as in dg_lines
  const int tM = (int)std::lround(std::log2(((double)m.h * 0x1p30 + 0.5 * m.l) / tb.M[0][0]));
  const int unit = d.eoff - 2 * (61 - tM) - 1023;
  double B = 0;
  for (int i = 0; i < N; ++i) {
    double r = 0, sw = 0;
    for (int j = 0; j < N; ++j) {
      r += std::fabs(tb.K[i][j]);
      sw += std::fabs(tb.D0[j]) * (j ? 0.5 : 1.0);
    }
    r += i == 0 || i == N - 1 ? 2 * sw + std::fabs(tb.D0[N - 1])
                              : std::fabs(tb.D0[i]) + std::fabs(tb.D0[N - 1 - i]);
    B = std::max(B, r);
  }
  for (int trial = 0; trial < 200; ++trial) {
    const double k = 1.0 + 2.0 * std::fabs(rnd()), ph = 3.0 * rnd();
    double v[N], nb[2][N], big = 0;
    for (int j = 0; j < N; ++j) {
      v[j] = std::sin(k * tb.nodes[j] + ph);
      nb[0][j] = std::sin(k * (tb.nodes[j] - 1) + ph);
      nb[1][j] = std::sin(k * (tb.nodes[j] + 1) + ph);
    }
    nb[0][N - 1] = v[0];
    nb[1][0] = v[N - 1];
    for (int j = 0; j < N; ++j)
      big = std::max({big, std::fabs(v[j]), std::fabs(nb[0][j]), std::fabs(nb[1][j])});
    const int E = (int)(fix::mag_hi(bits(big)) >> 20);
    int64_t q[N], y[N], g[2][N];
    for (int j = 0; j < N; ++j) q[j] = fix::from_double<false>(bits(v[j]), E) >> 3;
    fix::apply_line<N, 3>([&](int i, int j) { return d.K.E[i][j]; },
                          [&](int i, int j) { return d.K.O[i][j]; }, q, y);
    for (int s = 0; s < 2; ++s) {
      fix::Split w[N];
      for (int j = 0; j < N; ++j) {
        g[s][j] = q[j] - (fix::from_double<false>(bits(nb[s][N - 1 - j]), E) >> 3);
        w[j] = fix::split(g[s][j]);
      }
      y[s ? N - 1 : 0] += fix::dot<3, N>([&](int j) { return d.w[s ? N - 1 - j : j]; }, w);
    }
    const fix::Split e0 = fix::split(g[0][0]), e1 = fix::split(g[1][N - 1]);
    for (int j = 0; j < N; ++j) {
      const fix::Split q1[1] = {j ? e0 : e1}, q2[2] = {e0, e1};
      if (j == 0 || j == N - 1) y[j] += fix::dot<3, 1>([&](int) { return d.w[N - 1]; }, q1);
      else y[j] += fix::dot<3, 2>([&](int i) { return d.w[i ? N - 1 - j : j]; }, q2);
    }
    for (int i = 0; i < N; ++i) {
      long double r = 0;
      for (int j = 0; j < N; ++j) r += T.K[i][j] * v[j];
      for (int s = 0; s < 2; ++s)
        for (int j = 0; j < N; ++j)
          if (i == (s ? N - 1 : 0))
            r -= (s ? 0.5L : -0.5L) * (T.D[s][j] * v[j] + T.D[!s][j] * nb[s][j]);
      const double err = (double)std::fabs(std::ldexp((long double)y[i], unit + E) - r);
      if (!(err <= 0x1p-52 * B * big)) {
        std::printf("dg traces n=%d pen %g row %d: %g\n", N, pen, i, err);
        return 1;
      }
    }
  }
  return bad;
}

// A penalty that is not finite, or whose row sums overflow, is not in the tables.
template <int N>
int dg_non_finite() {
  Tables1D tb;
  build_tables(N - 1, &tb);
  FixedTables f0;
  if (!build_fixed_tables(tb, 1.0, &f0, 0.0) || !f0.dg_pen_in) return 1;
  for (double pen : {std::numeric_limits<double>::infinity(),
                     std::numeric_limits<double>::quiet_NaN(),
                     std::numeric_limits<double>::max()}) {
    FixedTables ft;
    if (!build_fixed_tables(tb, 1.0, &ft, pen) || ft.dg_pen_in ||
        std::memcmp(&ft.dg, &f0.dg, sizeof(ft.dg))) {
      std::printf("n=%d pen %g: eoff %d\n", N, pen, ft.dg.eoff);
      return 1;
    }
  }
  return 0;
}

int main() {
  int bad = conversions() | products();
  bad |= dg_non_finite<2>() | dg_non_finite<3>() | dg_non_finite<4>() | dg_non_finite<5>() |
         dg_non_finite<6>() | dg_non_finite<7>();
  for (double pen : {4.0, 49.0, 490.0, 4.9e3, 4.9e7, 1e10}) {
    bad |= dg_matching<2>(pen) | dg_matching<3>(pen) | dg_matching<4>(pen) |
           dg_matching<5>(pen) | dg_matching<6>(pen) | dg_matching<7>(pen);
  }
  for (double pen : {1.0, 49.0, 1e6}) {
    bad |= dg_lines<2>(pen) | dg_lines<3>(pen) | dg_lines<4>(pen) | dg_lines<5>(pen) |
           dg_lines<6>(pen) | dg_lines<7>(pen);
  }
  bad |= faces<2>() | faces<3>() | faces<4>() | faces<5>() | faces<6>() | faces<7>();
  for (double h : {2.0, 2.0 / 3, 2.0 / 96, 2.0 / 1000}) {
    bad |= cell<2>(h) | cell<3>(h) | cell<4>(h) | cell<5>(h) | cell<6>(h) | cell<7>(h);
  }
  return bad;
}
"""


def test_fixed_point_cell_term_and_conversions(tmp_path):
    src = tmp_path / "fixed.cpp"
    src.write_text(SRC)
    exe = str(tmp_path / "fixed")
    inc = [f"-I{CSRC}", f"-I{os.path.join(CSRC, '..', '..', 'include')}"]
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off",
                    "-fsanitize=signed-integer-overflow", "-fno-sanitize-recover=all",
                    "-static-libubsan", *inc, str(src),
                    os.path.join(CSRC, "setup.cpp"), os.path.join(CSRC, "fixed_tables.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
