// Fixed-point tables of the 3D FP64 cell term: the 1D pencil in double-double
// arithmetic (about 2^-104), scaled to the formats of fixed_point.cuh.
#include "fixed_tables.hpp"

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

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
  DD inv[kMaxN][kMaxN];
  for (int j = 0; j < n; ++j)
    for (int m = 0; m < j; ++m) {
      inv[j][m] = DD(1.0) / (x[j] - x[m]);
      inv[m][j] = -inv[j][m];
    }
  auto lagrange = [&](const DD& s, DD* v, DD* dv) {
    for (int j = 0; j < n; ++j) {
      DD a = 1.0, b;
      for (int m = 0; m < n; ++m) {
        if (m == j) continue;
        const DD f = inv[j][m];
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
    for (int i = 0; i < n; ++i) {
      const DD wv = w[q] * v[i], wd = w[q] * dv[i];
      for (int j = 0; j < n; ++j) {
        P->M[i][j] = P->M[i][j] + wv * v[j];
        P->K[i][j] = P->K[i][j] + wd * dv[j];
      }
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
  for (int it = 0; it < 2; ++it) {
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
    DD T1[kMaxN][kMaxN], T2[kMaxN][kMaxN];
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j)
        for (int k = 0; k < n; ++k) {
          T1[i][j] = T1[i][j] + A[i][n + k] * R1[k][j];
          T2[i][j] = T2[i][j] + A[i][n + k] * R2[k][j];
        }
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j)
        for (int l = 0; l < n; ++l) {
          E1[i][j] = E1[i][j] + T1[i][l] * A[j][n + l];
          E2[i][j] = E2[i][j] + T2[i][l] * A[j][n + l];
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
  return fix::to_entry(i1 + std::llrint((s - (double)i1) + std::ldexp(A.l, t)));
}

// t = 61 - ceil(log2) of the largest absolute sum
int fit(double c) { return 61 - (int)std::ceil(std::log2(c * (1.0 + 1e-6))); }

// What depends on the degree alone, made once per degree and process: the pencil
// and the face tables ...
struct Faces {
  Pencil P;
  std::vector<fix::Entry> face;
  int tM, eq, etm;
};
void make_faces(const Tables1D& tb, Faces* o) {
  const int n = tb.n;
  Pencil& P = o->P;
  P.n = n;
  mass_stiffness(tb, &P);
  // the trace of D0 is taken of 57-bit values and leaves at 60 bits (K = 3)
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
  const int tD = fit(cD), tS = fit(cS);
  o->tM = fit(cM);
  for (int j = 0; j < n; ++j) o->face.push_back(entry(P.D0[j], tD));
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) o->face.push_back(entry(P.M[i][j], o->tM));
  for (int q = 0; q < n; ++q)
    for (int j = 0; j < n; ++j) o->face.push_back(entry(P.S[q][j], tS));
  o->eq = 2 + 2 * (61 - tS);
  o->etm = 2 - tD + 2 * (61 - o->tM);
}

// ... and the eigenbasis and scales of the cell term
struct Cell {
  Pencil P;
  fix::Block Vt = {}, V = {};
  int sm[kMaxN], t3, S5;
  bool ok;
};
bool make_cell(const Tables1D& tb, Cell* o) {
  const int n = tb.n, H = n / 2, HE = (n + 1) / 2;
  Pencil& P = o->P;
  refine(tb, &P);
  // modes scaled by 2^sm: rows of V^T of absolute sum in (1/2, 1]
  double r[kMaxN], lam[kMaxN], M[kMaxN][kMaxN], K[kMaxN][kMaxN];
  int* sm = o->sm;
  for (int k = 0; k < n; ++k) {
    r[k] = 0.0;
    for (int j = 0; j < n; ++j) r[k] += mag(P.V[j][k]);
    sm[k] = (int)std::floor(-std::log2(r[k]) + 1e-7);
    if (!(r[k] <= 1.0 + 1e-7)) return false;      // S_1 = S_2 = 0 below
    lam[k] = P.lam[k].h;
    for (int j = 0; j < n; ++j) {
      M[k][j] = P.M[k][j].h;
      K[k][j] = P.K[k][j].h;
    }
  }
  // largest absolute row sums from the input to the phases' results
  double B3 = 0.0, B4 = 0.0, B5 = 0.0;
  for (int a = 0; a < n; ++a)
    for (int b = a; b < n; ++b)
      for (int i = 0; i < HE; ++i) {               // (mirrored rows have equal sums)
        double s = 0.0;
        for (int j = 0; j < n; ++j) s += std::fabs(K[i][j] + (lam[a] + lam[b]) * M[i][j]);
        B3 = std::max(B3, s * r[a] * r[b]);
      }
  // (summed over the y-modes: V V^T = M, V lam V^T = K)
  for (int b = 0; b < n; ++b)
    for (int i = 0; i < HE; ++i)
      for (int y = 0; y < HE; ++y) {
        double s = 0.0;
        for (int j = 0; j < n; ++j)
          for (int yy = 0; yy < n; ++yy)
            s += std::fabs((K[i][j] + lam[b] * M[i][j]) * M[y][yy] + M[i][j] * K[y][yy]);
        B4 = std::max(B4, s * r[b]);
      }
  for (int i = 0; i < HE; ++i)
    for (int y = i; y < HE; ++y)
      for (int z = y; z < HE; ++z) {   // and the axes can be exchanged
        double s = 0.0;
        for (int j = 0; j < n; ++j)
          for (int yy = 0; yy < n; ++yy) {
            const double km = K[i][j] * M[y][yy] + M[i][j] * K[y][yy], mm = M[i][j] * M[y][yy];
            for (int zz = 0; zz < n; ++zz) s += std::fabs(km * M[z][zz] + mm * K[z][zz]);
          }
        B5 = std::max(B5, s);
      }
  auto scale_of = [](double B) { return -(int)std::ceil(std::log2(B) - 1e-7); };
  const int S3 = scale_of(B3), S4 = scale_of(B4), S5 = scale_of(B5);
  // t = 61 + S_i - S_{i-1} - K per phase, and what a result then sums
  const int t1 = 61, t4 = 61 + S4 - S3 - fix::shift_y(n),
            t5 = 61 + S5 - S4 - fix::shift_z(n);
  if (t4 != t5) return false;                     // one table serves both
  o->t3 = 61 + S3 - fix::shift_x(n);
  o->S5 = S5;
  const double lim = std::ldexp(1.0, 61) * (1.0 - 1e-7);
  for (int k = 0; k < n; ++k) {
    double s = 0.0;
    const bool odd = k >= HE;
    for (int j = 0; j < (odd ? H : HE); ++j) {
      s += std::ldexp(mag(P.V[j][k]), t1 + sm[k]);
      const fix::Entry e = entry(P.V[j][k], t1 + sm[k]);
      if (odd) o->Vt.O[k - HE][j] = e;
      else o->Vt.E[k][j] = e;
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
      if (odd) o->V.O[j][k - HE] = e;
      else o->V.E[j][k] = e;
    }
    if (!(se <= lim && so <= lim)) return false;
  }
  return true;
}

const Faces& faces_of(const Tables1D& tb) {
  static std::once_flag once[kMaxN + 1];
  static Faces made[kMaxN + 1];
  std::call_once(once[tb.n], [&] { make_faces(tb, &made[tb.n]); });
  return made[tb.n];
}
const Cell& cell_of(const Tables1D& tb) {
  static std::once_flag once[kMaxN + 1];
  static Cell made[kMaxN + 1];
  std::call_once(once[tb.n], [&] {
    made[tb.n].P = faces_of(tb).P;
    made[tb.n].ok = make_cell(tb, &made[tb.n]);
  });
  return made[tb.n];
}

// the cell term's part: Vt, V, xline, eoff
bool cell_tables(const Tables1D& tb, double hm, int eh, FixedTables* out) {
  const int n = tb.n, H = n / 2, HE = (n + 1) / 2;
  const Cell& c = cell_of(tb);
  if (!c.ok) return false;
  const Pencil& P = c.P;
  const double lim = std::ldexp(1.0, 61) * (1.0 - 1e-7);
  out->Vt = c.Vt;
  out->V = c.V;
  // hm (K + (lam_a + lam_b) M) 2^(-sm_a - sm_b): the upper triangles of the
  // even and the odd block, one slot per unordered pair of modes a <= b
  const int packed = (HE * (HE + 1) / 2 + H * (H + 1) / 2) | 1;
  out->xline.assign((size_t)(n * (n + 1) / 2) * packed, fix::Entry{0, 0});
  size_t slot = 0;
  for (int a = 0; a < n; ++a)
    for (int b = a; b < n; ++b, slot += packed) {
      const int t = c.t3 - c.sm[a] - c.sm[b];
      const DD mu = P.lam[a] + P.lam[b];
      DD X[fix::kMaxHalf][kMaxN];                 // the upper half of h K + mu M
      for (int i = 0; i < HE; ++i)
        for (int j = 0; j < n; ++j) X[i][j] = P.K[i][j] + mu * P.M[i][j];
      size_t w = slot;
      for (int o = 0; o < 2; ++o)
        for (int i = 0; i < (o ? H : HE); ++i) {
          double s = 0.0;
          for (int j = 0; j < (o ? H : HE); ++j) {
            const DD u = o ? X[i][j] - X[i][n - 1 - j] : X[i][j] + X[i][n - 1 - j];
            const DD v = ((n & 1) && j == H ? X[i][j] : u * DD(0.5)) * DD(hm);
            s += std::ldexp(mag(v), t);
            if (j >= i) out->xline[w++] = entry(v, t);
          }
          if (!(s <= lim)) return false;
        }
    }
  out->eoff = -59 - c.S5 + eh;
  return true;
}

}  // namespace

bool build_fixed_tables(const Tables1D& tb, double scale, FixedTables* out, double pen, int parts) {
  const int n = tb.n, H = n / 2, HE = (n + 1) / 2;
  *out = FixedTables{};
  if (!parts) return true;
  // scale = hm 2^eh, hm in (1/2, 1]
  int eh;
  double hm = std::frexp(scale, &eh);
  if (hm == 0.5) {
    hm = 1.0;
    --eh;
  }
  if ((parts & kFixCell) && !cell_tables(tb, hm, eh, out)) return false;
  const Faces& fa = faces_of(tb);
  const Pencil& P = fa.P;
  const int tM = fa.tM;
  if (parts & kFixFaces) out->face = fa.face;
  out->face_eq = fa.eq;
  out->face_etm = fa.etm;
  if (!(parts & kFixDg)) return true;
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
