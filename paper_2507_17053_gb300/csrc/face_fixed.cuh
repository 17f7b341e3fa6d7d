// Surrogate-boundary faces of the 3D FP64 apply with the exact extension, in
// fixed point (fixed_point.cuh): the method of face_body.cuh on the integer
// units.
//
// Per face: the cell's n^3 values enter as integers with the cell's largest
// exponent (57 bits), then
//   E12[j0] = sum_{j1 j2} P[j1 + n j2] u[j0, j1, j2]   (stored products P)
//   val     = sum_j0 (W phi_j0) E12[j0]                at Gauss point tl
//   Td      = the normal-derivative trace              at tangential node tl
//   q = (S x S)^T val,  tm = (M x M) Td                (two line phases)
// and the two results leave as doubles: rv = sigma q + h^-1 h^(d-1) tm,
// rg = -+ h^-1 q (the end derivatives of the two faces of an axis mirror each
// other, D1[j] = -D0[n-1-j], so Td is taken with D0's mirror image and tm
// enters with one sign for both).
//
// Ranges.  P is scaled per point (2^t, absolute sum below 2^61), W phi per
// point so that all points of a face share one exponent (face_exp); the sums
// of n^2 <= 49 products stay inside 64 bits because the inputs have 57 bits:
//   |sum h ql| <= 2^62 + 2^36, |sum l qh| <= 49 2^30 2^26 < 2^61.7.
// The rounding of a value is 2^-57 of the cell's largest one, 2^-60 in every
// later phase, against 2^-53 of each product in double precision.  All points of
// a face share the exponent of the largest extrapolation among them.
//
// The double form was bound by the double-precision pipe (95 % busy).
// Measured on GB300, face kernel, double -> fixed point: Q4 sphere of 96^3
// cells (21 912 faces) 162 -> 62 us, Q6 ellipsoid of 48^3 cells (4 248 faces)
// 193 -> 54 us; whole FP64 applies 484 -> 381 us and 291 -> 147 us, batch of 9
// problems x 3 right-hand sides 1 130 -> 847 us.
#pragma once

#include "face_body.cuh"

namespace sbm {

template <int N, int FPB>
struct FaceFixSmem {
  static constexpr int L = N * N;
  static constexpr int PL = (L + 1) & ~1;        // z-planes padded to pairs (16-byte reads)
  static constexpr int NDP = N * PL;
  static constexpr int TAB = N + 2 * L;          // D0, M, S
  static constexpr size_t bytes = (size_t)(FPB * (NDP + 4 * L) + TAB) * 8 + FPB * 4;
};

// The 1D tables and cleared exponent words; once per block, before the first
// group.
template <int N, int FPB>
__device__ __forceinline__ void face_fix_begin(const FaceArgs<double>& a,
                                               unsigned char* smem_raw) {
  using FS = FaceFixSmem<N, FPB>;
  int2* tab = reinterpret_cast<int2*>(smem_raw) + FPB * (FS::NDP + 4 * FS::L);
  const int2* src = reinterpret_cast<const int2*>(a.fix.tab);
  for (int i = threadIdx.x; i < FS::TAB; i += blockDim.x) tab[i] = __ldg(src + i);
  uint32_t* slot = reinterpret_cast<uint32_t*>(tab + FS::TAB);
  for (int i = threadIdx.x; i < FPB; i += blockDim.x) slot[i] = 0u;
  __syncthreads();
}

// sum_j a[j] q[j], both read from shared memory
template <int K, int N, typename FA, typename FQ>
__device__ __forceinline__ int64_t face_dot(const FA& A, const FQ& Q) {
  fix::Entry e[N];
  fix::Split q[N];
#pragma unroll
  for (int j = 0; j < N; ++j) {
    e[j] = A(j);
    q[j] = Q(j);
  }
  return fix::dot<K, N>([&](int j) { return e[j]; }, q);
}

__device__ __forceinline__ double face_to_double(int64_t q, int eb) {
  const uint64_t b = fix::plain_result(eb) ? fix::to_double<false>(q, eb)
                                           : fix::to_double<true>(q, eb);
  return __longlong_as_double((long long)b);
}

// Faces [f0, min(f0 + FPB, fend)) of right-hand side rhs, n^2 threads per
// face (threads beyond idle but take part in the barriers); face_fix_begin
// ran before.  ts: the problem's sigma, 1/h and h^(d-1).
template <int N, int FPB>
__device__ __forceinline__ void face_group_fix(const FaceArgs<double>& a, const KTab<double>& ts,
                                               unsigned char* smem_raw, int f0, int fend,
                                               int rhs) {
  using FS = FaceFixSmem<N, FPB>;
  constexpr int L = FS::L, PL = FS::PL;
  const double* __restrict__ xr = a.x + rhs * a.ldx;
  double* __restrict__ outr = a.out + rhs * a.ld_out;
  const int tid = threadIdx.x;
  const int fl = tid / L, tl = tid - fl * L;
  const int nf = min(FPB, fend - f0);
  const bool act = fl < nf;
  const int f = f0 + (act ? fl : 0);
  fix::Split* X = reinterpret_cast<fix::Split*>(smem_raw) + (act ? fl : 0) * FS::NDP;
  fix::Split* val = reinterpret_cast<fix::Split*>(smem_raw) + FPB * FS::NDP + (act ? fl : 0) * 4 * L;
  fix::Split* Td = val + L;
  fix::Split* Va = Td + L;
  fix::Split* Da = Va + L;
  const fix::Entry* D0 = reinterpret_cast<const fix::Entry*>(smem_raw) + FPB * (FS::NDP + 4 * L);
  const fix::Entry* M = D0 + N;
  const fix::Entry* S = M + L;
  uint32_t* slot = reinterpret_cast<uint32_t*>(smem_raw) +
                   2 * (FPB * (FS::NDP + 4 * L) + FS::TAB) + (act ? fl : 0);
  const int2* __restrict__ pp = reinterpret_cast<const int2*>(a.fix.pp) + (size_t)f * L * L + tl;
  const int2* __restrict__ p0 = reinterpret_cast<const int2*>(a.fix.p0) + (size_t)f * N * L + tl;

  // the cell's nodes tl, tl + n^2, ...: in registers until the exponent is known
  uint64_t u[N];
  int2 w[N];                       // the products of plane j2, one plane ahead
  int kind = 0, fe = 0;
  if (act) {
    const int cell = __ldg(a.face_cell + f);
    if (a.dg) {
      const double* xc = xr + (size_t)__ldg(a.cell_rank + cell) * (N * L) + tl;
#pragma unroll
      for (int i = 0; i < N; ++i) u[i] = (uint64_t)__double_as_longlong(__ldg(xc + L * i));
    } else {
      const int32_t* ln = a.lines + (size_t)cell * L + tl / N;
#pragma unroll
      for (int i = 0; i < N; ++i)
        u[i] = (uint64_t)__double_as_longlong(__ldg(xr + (size_t)__ldg(ln + N * i) + tl % N));
    }
#pragma unroll
    for (int j = 0; j < N; ++j) w[j] = __ldg(pp + (size_t)j * L);
    kind = __ldg(a.face_kind + f);
    fe = __ldg(a.fix.exp + f);
    uint32_t mx = 0u;
#pragma unroll
    for (int i = 0; i < N; ++i) mx = max(mx, fix::mag_hi(u[i]));
    cell_max(mx, cell_lanes(fl), slot);
  }
  __syncthreads();
  const int E = max(1, (int)(*slot >> 20));
  if (act) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int64_t v =
          fix::plain_exp(E) ? fix::from_double<false>(u[i], E) : fix::from_double<true>(u[i], E);
      X[PL * i + tl] = fix::split(v >> 3);
    }
  }
  __syncthreads();
  const int k = kind & 3, s = kind >> 2;
  if (act) {
    if (tl == 0) *slot = 0u;       // for the next group (its reads of E are past)
    // the extension at the shifted point of Gauss point tl
    int64_t hi[N], mid[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      hi[j] = 0;
      mid[j] = (int64_t)1 << 27;
    }
#pragma unroll(N <= 2 ? N : 1)
    for (int j2 = 0; j2 < N; ++j2) {
      int2 wn[N];
      if (j2 + 1 < N) {
#pragma unroll
        for (int j = 0; j < N; ++j) wn[j] = __ldg(pp + (size_t)(N * (j2 + 1) + j) * L);
      }
      const int4* xp = reinterpret_cast<const int4*>(X + PL * j2);
#pragma unroll
      for (int m = 0; m < PL / 2; ++m) {
        const int4 v = xp[m];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int i = 2 * m + r;
          if (i >= L) continue;
          const int qh = r ? v.z : v.x, ql = r ? v.w : v.y;
          const int j0 = i % N, j1 = i / N;
          hi[j0] = fix::mad_wide(w[j1].x, qh, hi[j0]);
          mid[j0] = fix::mad_wide(w[j1].x, ql, mid[j0]);
          mid[j0] = fix::mad_wide(w[j1].y, qh, mid[j0]);
        }
      }
      if (j2 + 1 < N) {
#pragma unroll
        for (int j = 0; j < N; ++j) w[j] = wn[j];
      }
    }
    fix::Split e12[N];
#pragma unroll
    for (int j = 0; j < N; ++j) e12[j] = fix::split(fix::shl_add<3>(hi[j], mid[j] >> 28));
    val[tl] = fix::split(fix::dot<0, N>(
        [&](int j) {
          const int2 e = __ldg(p0 + (size_t)j * L);
          return fix::Entry{e.x, e.y};
        },
        e12));
    // the normal-derivative trace at tangential node tl
    const int sk = k == 0 ? 1 : (k == 1 ? N : PL);
    const int bt = (tl % N) * (k == 0 ? N : 1) + (tl / N) * (k == 2 ? N : PL);
    Td[tl] = fix::split(face_dot<3, N>([&](int j) { return D0[s ? N - 1 - j : j]; },
                                       [&](int j) { return X[bt + sk * j]; }));
  }
  __syncthreads();
  const int ia = tl % N, ib = tl / N;
  if (act) {                       // first tangential axis (M is symmetric)
    Va[tl] = fix::split(face_dot<0, N>([&](int j) { return S[N * j + ia]; },
                                       [&](int j) { return val[j + N * ib]; }));
    Da[tl] = fix::split(face_dot<0, N>([&](int j) { return M[N * j + ia]; },
                                       [&](int j) { return Td[j + N * ib]; }));
  }
  __syncthreads();
  if (act) {                       // second tangential axis
    const int64_t qi = face_dot<0, N>([&](int j) { return S[N * j + ib]; },
                                      [&](int j) { return Va[ia + N * j]; });
    const int64_t ti = face_dot<0, N>([&](int j) { return M[N * j + ib]; },
                                      [&](int j) { return Da[ia + N * j]; });
    double q, tm;
    if (E == fix::kExpBad || fe == fix::kFaceExpBad) {
      q = tm = __longlong_as_double(0x7ff8000000000000ll);
    } else {
      q = face_to_double(qi, E + fe + a.fix.eq);
      tm = face_to_double(ti, E + a.fix.etm);
    }
    outr[(size_t)f * 2 * L + tl] = fma(ts.sigma, q, (ts.h_inv * ts.hface) * tm);
    outr[(size_t)f * 2 * L + L + tl] = (s ? -ts.h_inv : ts.h_inv) * q;
  }
}

}  // namespace sbm
