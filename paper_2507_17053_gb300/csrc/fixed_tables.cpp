// Fixed-point tables of the 3D FP64 cell term: the 1D pencil in double-double
// arithmetic (about 2^-104), scaled to the formats of fixed_point.cuh.
#include "fixed_tables.hpp"

#include <algorithm>
#include <cmath>

#include "setup.hpp"

namespace sbm {
namespace {

// ---- double-double arithmetic (Dekker, Knuth: error-free sums and products) ----
struct DD {
  double h = 0.0, l = 0.0;
  DD() {}
  DD(double a) : h(a) {}
  DD(double a, double b) {
    h = a + b;
    const double t = h - a;
    l = (a - (h - t)) + (b - t);
  }
};
DD operator+(const DD& a, const DD& b) {
  const DD s(a.h, b.h);
  return DD(s.h, s.l + (a.l + b.l));
}
DD operator-(const DD& a) {
  DD r;
  r.h = -a.h;
  r.l = -a.l;
  return r;
}
DD operator-(const DD& a, const DD& b) { return a + (-b); }
DD operator*(const DD& a, const DD& b) {
  const double p = a.h * b.h;
  return DD(p, std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
DD operator/(const DD& a, const DD& b) {
  const double q1 = a.h / b.h;
  const DD r = a - DD(q1) * b;
  const double q2 = r.h / b.h;
  const DD r2 = r - DD(q2) * b;
  return DD(q1, q2) + DD(r2.h / b.h);
}
double mag(const DD& a) { return std::fabs(a.h); }

// Legendre P_m and P_m' at t in (-1, 1)
void legendre(int m, const DD& t, DD* P, DD* dP) {
  DD p0 = 1.0, p1 = t;
  for (int k = 1; k < m; ++k) {
    const DD p2 = (DD(2.0 * k + 1.0) * t * p1 - DD((double)k) * p0) / DD(k + 1.0);
    p0 = p1;
    p1 = p2;
  }
  *P = p1;
  *dP = DD((double)m) * (p0 - t * p1) / (DD(1.0) - t * t);
}

struct Pencil {
  int n;
  DD M[kMaxN][kMaxN], K[kMaxN][kMaxN], V[kMaxN][kMaxN], lam[kMaxN];
  DD S[kMaxN][kMaxN], D0[kMaxN];     // phi_j at Gauss point q, phi_j'(0)
};

// 1D mass and stiffness matrices from double-double nodes and Gauss points
// (the double ones polished by Newton steps)
void mass_stiffness(const Tables1D& t, Pencil* P) {
  const int n = t.n, p = n - 1;
  DD x[kMaxN], g[kMaxN], w[kMaxN];
  for (int j = 0; j < n; ++j) {
    if (j == 0 || j == p) {
      x[j] = j ? 1.0 : 0.0;
      continue;
    }
    DD s = DD(2.0) * DD(t.nodes[j]) - DD(1.0);
    for (int it = 0; it < 3; ++it) {      // P_p'(s) = 0; (1-s^2) P'' = 2 s P' - p (p+1) P
      DD L, d;
      legendre(p, s, &L, &d);
      const DD d2 = (DD(2.0) * s * d - DD((double)p * (p + 1)) * L) / (DD(1.0) - s * s);
      s = s - d / d2;
    }
    x[j] = (s + DD(1.0)) * DD(0.5);
  }
  for (int q = 0; q < n; ++q) {
    DD s = DD(2.0) * DD(t.gpts[q]) - DD(1.0), L, d;
    for (int it = 0; it < 3; ++it) {
      legendre(n, s, &L, &d);
      s = s - L / d;
    }
    legendre(n, s, &L, &d);
    g[q] = (s + DD(1.0)) * DD(0.5);
    w[q] = DD(1.0) / ((DD(1.0) - s * s) * d * d);
  }
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) P->M[i][j] = P->K[i][j] = DD();
  auto lagrange = [&](const DD& s, DD* v, DD* dv) {
    for (int j = 0; j < n; ++j) {
      DD a = 1.0, b;
      for (int m = 0; m < n; ++m) {
        if (m == j) continue;
        const DD f = DD(1.0) / (x[j] - x[m]);
        b = (b * (s - x[m]) + a) * f;
        a = a * (s - x[m]) * f;
      }
      v[j] = a;
      dv[j] = b;
    }
  };
  DD ends[kMaxN];
  lagrange(DD(0.0), ends, P->D0);
  for (int q = 0; q < n; ++q) {
    DD v[kMaxN], dv[kMaxN];
    lagrange(g[q], v, dv);
    for (int j = 0; j < n; ++j) P->S[q][j] = v[j];
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        P->M[i][j] = P->M[i][j] + w[q] * v[i] * v[j];
        P->K[i][j] = P->K[i][j] + w[q] * dv[i] * dv[j];
      }
  }
}

// Refine the double eigenbasis V, lam of the tables: with W = V^-1 the
// residuals E1 = W (M - V V^T) W^T and E2 = W (K - V lam V^T) W^T are small;
// V (I + X) with X + X^T = E1 and X lam + lam X^T + D = E2 removes them to
// first order (X_ij = (E2_ij - lam_i E1_ij) / (lam_j - lam_i)).
void refine(const Tables1D& t, Pencil* P) {
  const int n = t.n;
  for (int i = 0; i < n; ++i) {
    P->lam[i] = t.lam[i];
    for (int j = 0; j < n; ++j) P->V[i][j] = t.V[i][j];
  }
  for (int it = 0; it < 3; ++it) {
    DD A[kMaxN][2 * kMaxN];                       // Gauss-Jordan: W = V^-1
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        A[i][j] = P->V[i][j];
        A[i][n + j] = i == j ? 1.0 : 0.0;
      }
    for (int c = 0; c < n; ++c) {
      int pr = c;
      for (int r = c + 1; r < n; ++r)
        if (mag(A[r][c]) > mag(A[pr][c])) pr = r;
      for (int k = 0; k < 2 * n; ++k) std::swap(A[c][k], A[pr][k]);
      const DD f = DD(1.0) / A[c][c];
      for (int k = 0; k < 2 * n; ++k) A[c][k] = A[c][k] * f;
      for (int r = 0; r < n; ++r) {
        if (r == c) continue;
        const DD m = A[r][c];
        for (int k = 0; k < 2 * n; ++k) A[r][k] = A[r][k] - m * A[c][k];
      }
    }
    DD R1[kMaxN][kMaxN], R2[kMaxN][kMaxN], E1[kMaxN][kMaxN], E2[kMaxN][kMaxN];
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        DD a = P->M[i][j], b = P->K[i][j];
        for (int k = 0; k < n; ++k) {
          const DD vv = P->V[i][k] * P->V[j][k];
          a = a - vv;
          b = b - vv * P->lam[k];
        }
        R1[i][j] = a;
        R2[i][j] = b;
      }
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        DD a, b;
        for (int k = 0; k < n; ++k)
          for (int l = 0; l < n; ++l) {
            const DD ww = A[i][n + k] * A[j][n + l];
            a = a + ww * R1[k][l];
            b = b + ww * R2[k][l];
          }
        E1[i][j] = a;
        E2[i][j] = b;
      }
    DD nv[kMaxN][kMaxN];
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        nv[i][j] = P->V[i][j];
        for (int k = 0; k < n; ++k) {
          // modes of opposite parity do not mix
          const int HE = (n + 1) / 2;
          if ((k < HE) != (j < HE)) continue;
          const DD X = k == j ? E1[k][k] * DD(0.5)
                              : (E2[k][j] - P->lam[k] * E1[k][j]) / (P->lam[j] - P->lam[k]);
          nv[i][j] = nv[i][j] + P->V[i][k] * X;
        }
      }
    for (int i = 0; i < n; ++i) {
      if (i > 0) P->lam[i] = P->lam[i] + (E2[i][i] - P->lam[i] * E1[i][i]);   // lam_0 = 0
      for (int j = 0; j < n; ++j) P->V[i][j] = nv[i][j];
    }
  }
}

// A 2^t = h 2^30 + l / 2, |A 2^t| < 2^61
fix::Entry entry(const DD& A, int t) {
  const double s = std::ldexp(A.h, t);
  const int64_t i1 = std::llrint(s);
  const int64_t I = i1 + std::llrint((s - (double)i1) + std::ldexp(A.l, t));
  const int64_t h = (I + ((int64_t)1 << 29)) >> 30;
  return fix::Entry{(int32_t)h, (int32_t)(2 * (I - h * ((int64_t)1 << 30)))};
}

}  // namespace

bool build_fixed_tables(const Tables1D& tb, double scale, FixedTables* out, double pen) {
  const int n = tb.n, H = n / 2, HE = (n + 1) / 2;
  Pencil P;
  P.n = n;
  mass_stiffness(tb, &P);
  refine(tb, &P);
  // scale = hm 2^eh, hm in (1/2, 1]
  int eh;
  double hm = std::frexp(scale, &eh);
  if (hm == 0.5) {
    hm = 1.0;
    --eh;
  }
  auto X = [&](int a, int b, int i, int j) { return P.K[i][j] + (P.lam[a] + P.lam[b]) * P.M[i][j]; };
  // modes scaled by 2^sm: rows of V^T of absolute sum in (1/2, 1]
  double r[kMaxN];
  int sm[kMaxN];
  for (int k = 0; k < n; ++k) {
    r[k] = 0.0;
    for (int j = 0; j < n; ++j) r[k] += mag(P.V[j][k]);
    sm[k] = (int)std::floor(-std::log2(r[k]) + 1e-7);
    if (!(r[k] <= 1.0 + 1e-7)) return false;      // S_1 = S_2 = 0 below
  }
  // largest absolute row sums from the input to the phases' results
  double B3 = 0.0, B4 = 0.0, B5 = 0.0;
  for (int a = 0; a < n; ++a)
    for (int b = 0; b < n; ++b)
      for (int i = 0; i < n; ++i) {
        double s = 0.0;
        for (int j = 0; j < n; ++j) s += mag(X(a, b, i, j));
        B3 = std::max(B3, s * r[a] * r[b]);
      }
  // (mirrored rows have equal sums)
  for (int b = 0; b < n; ++b)
    for (int i = 0; i < HE; ++i)
      for (int y = 0; y < HE; ++y) {
        double s = 0.0;
        for (int j = 0; j < n; ++j)
          for (int yy = 0; yy < n; ++yy) {
            double u = 0.0;
            for (int a = 0; a < n; ++a) u += P.V[y][a].h * P.V[yy][a].h * X(a, b, i, j).h;
            s += std::fabs(u);
          }
        B4 = std::max(B4, s * r[b]);
      }
  for (int i = 0; i < HE; ++i)
    for (int y = i; y < HE; ++y)
      for (int z = y; z < HE; ++z) {   // and the axes can be exchanged
        double s = 0.0;
        for (int j = 0; j < n; ++j)
          for (int yy = 0; yy < n; ++yy)
            for (int zz = 0; zz < n; ++zz)
              s += std::fabs(P.K[i][j].h * P.M[y][yy].h * P.M[z][zz].h +
                             P.M[i][j].h * P.K[y][yy].h * P.M[z][zz].h +
                             P.M[i][j].h * P.M[y][yy].h * P.K[z][zz].h);
        B5 = std::max(B5, s);
      }
  auto scale_of = [](double B) { return -(int)std::ceil(std::log2(B) - 1e-7); };
  const int S3 = scale_of(B3), S4 = scale_of(B4), S5 = scale_of(B5);
  // t = 61 + S_i - S_{i-1} - K per phase, and what a result then sums
  const int t1 = 61, t3 = 61 + S3 - fix::shift_x(n), t4 = 61 + S4 - S3 - fix::shift_y(n),
            t5 = 61 + S5 - S4 - fix::shift_z(n);
  if (t4 != t5) return false;                     // one table serves both
  const double lim = std::ldexp(1.0, 61) * (1.0 - 1e-7);
  out->Vt = out->V = fix::Block{};
  for (int k = 0; k < n; ++k) {
    double s = 0.0;
    const bool odd = k >= HE;
    for (int j = 0; j < (odd ? H : HE); ++j) {
      s += std::ldexp(mag(P.V[j][k]), t1 + sm[k]);
      const fix::Entry e = entry(P.V[j][k], t1 + sm[k]);
      if (odd) out->Vt.O[k - HE][j] = e;
      else out->Vt.E[k][j] = e;
    }
    if (!(s <= lim)) return false;
  }
  for (int j = 0; j < HE; ++j) {
    double se = 0.0, so = 0.0;
    for (int k = 0; k < n; ++k) {
      const bool odd = k >= HE;
      if (odd && j >= H) continue;
      (odd ? so : se) += std::ldexp(mag(P.V[j][k]), t4);
      const fix::Entry e = entry(P.V[j][k], t4);
      if (odd) out->V.O[j][k - HE] = e;
      else out->V.E[j][k] = e;
    }
    if (!(se <= lim && so <= lim)) return false;
  }
  // hm (K + (lam_a + lam_b) M) 2^(-sm_a - sm_b): the upper triangles of the
  // even and the odd block, one slot per unordered pair of modes a <= b
  const int packed = (HE * (HE + 1) / 2 + H * (H + 1) / 2) | 1;
  out->xline.assign((size_t)(n * (n + 1) / 2) * packed, fix::Entry{0, 0});
  size_t slot = 0;
  for (int a = 0; a < n; ++a)
    for (int b = a; b < n; ++b, slot += packed) {
      const int t = t3 - sm[a] - sm[b];
      auto E = [&](int i, int j) {
        const DD v = (n & 1) && j == H ? X(a, b, i, j)
                                       : (X(a, b, i, j) + X(a, b, i, n - 1 - j)) * DD(0.5);
        return v * DD(hm);
      };
      auto O = [&](int i, int j) {
        return (X(a, b, i, j) - X(a, b, i, n - 1 - j)) * DD(0.5) * DD(hm);
      };
      size_t w = slot;
      for (int i = 0; i < HE; ++i) {
        double s = 0.0;
        for (int j = 0; j < HE; ++j) s += std::ldexp(mag(E(i, j)), t);
        if (!(s <= lim)) return false;
        for (int j = i; j < HE; ++j) out->xline[w++] = entry(E(i, j), t);
      }
      for (int i = 0; i < H; ++i) {
        double s = 0.0;
        for (int j = 0; j < H; ++j) s += std::ldexp(mag(O(i, j)), t);
        if (!(s <= lim)) return false;
        for (int j = i; j < H; ++j) out->xline[w++] = entry(O(i, j), t);
      }
    }
  out->eoff = -59 - S5 + eh;
  // faces: t = 61 - ceil(log2) of the largest absolute sum; the trace of D0
  // is taken of 57-bit values and leaves at 60 bits (K = 3)
  double cD = 0.0, cM = 0.0, cS = 0.0;
  for (int j = 0; j < n; ++j) {
    double m = 0.0, s = 0.0;
    for (int i = 0; i < n; ++i) {
      m += mag(P.M[i][j]);
      s += mag(P.S[i][j]);
    }
    cD += mag(P.D0[j]);
    cM = std::max(cM, m);
    cS = std::max(cS, s);
  }
  auto fit = [](double c) { return 61 - (int)std::ceil(std::log2(c * (1.0 + 1e-6))); };
  const int tD = fit(cD), tM = fit(cM), tS = fit(cS);
  out->face.clear();
  for (int j = 0; j < n; ++j) out->face.push_back(entry(P.D0[j], tD));
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) out->face.push_back(entry(P.M[i][j], tM));
  for (int q = 0; q < n; ++q)
    for (int j = 0; j < n; ++j) out->face.push_back(entry(P.S[q][j], tS));
  out->face_eq = 2 + 2 * (61 - tS);
  out->face_etm = 2 - tD + 2 * (61 - tM);
  // DG line operators: row i of K u + sum_s Own_s g_s, |g| <= 2 |u|, scaled to
  // leave 57-bit values at 59 bits (K = 3); hm goes into the entries.  The
  // penalty is part of them while it no more than doubles the largest row sum
  // (dg_apply.cu; a sum that overflows or is NaN does not pass).
  DD w[kMaxN];
  for (int j = 0; j < n; ++j) w[j] = j ? P.D0[j] * DD(0.5) : P.D0[0];
  auto row_sums = [&](double w0) {
    double sw = w0, B = 0.0;
    for (int j = 1; j < n; ++j) sw += mag(w[j]);
    for (int i = 0; i < n; ++i) {
      double r = 0.0;
      for (int j = 0; j < n; ++j) r += mag(P.K[i][j]);
      r += 2.0 * (i == 0 ? sw : mag(w[i]));
      r += 2.0 * (i == n - 1 ? sw : mag(w[n - 1 - i]));
      if (!(r <= B)) B = r;
    }
    return B;
  };
  double B1 = row_sums(mag(w[0]));
  const double B1p = row_sums(std::fabs(pen + w[0].h));
  out->dg_pen_in = B1p <= 2.0 * B1;
  if (out->dg_pen_in) {
    w[0] = DD(pen) + w[0];
    B1 = B1p;
  }
  out->dg = fix::DgTab{};
  const int tR = fit(B1) - 1;
  auto folded = [&](const DD (&A)[kMaxN][kMaxN], int t, double f, fix::Block* o) {
    for (int i = 0; i < HE; ++i)
      for (int j = 0; j < HE; ++j) {
        const bool mid = (n & 1) && j == H;
        const DD e = mid ? A[i][j] : (A[i][j] + A[i][n - 1 - j]) * DD(0.5);
        o->E[i][j] = entry(e * DD(f), t);
        if (i < H && j < H) o->O[i][j] = entry((A[i][j] - A[i][n - 1 - j]) * DD(0.5) * DD(f), t);
      }
  };
  folded(P.K, tR, hm, &out->dg.K);
  folded(P.M, tM, 1.0, &out->dg.M);
  for (int j = 0; j < n; ++j) out->dg.w[j] = entry(w[j] * DD(hm), tR);
  out->dg.eoff = 2 - tR + 2 * (61 - tM) + eh;
  return true;
}

}  // namespace sbm
