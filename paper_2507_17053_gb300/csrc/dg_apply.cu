// Matrix-free apply (FP64 or FP32) of the SIPG discontinuous Galerkin SBM operator.
//
// Cell-centric: every block owns some cells and writes their DoFs once (a DG
// cell's DoFs belong to it alone), so there is no colouring and there are no
// atomics.  Each interior face is evaluated from both sides (twice the face
// arithmetic, no write conflict), the neighbour's values read straight from
// global memory; surrogate faces (Algorithm 3) are computed beforehand by the
// face kernel and folded in here.
//
// 2D, per cell: the cell term (Algorithm 1), then its faces in the order (k, s):
//  * interior face (neighbour active), Algorithm 2 from this cell's side:
//      [u] = u_K1 - u_K2, {dn u} = (dn u_K1 + dn u_K2)/2 with n = +e_k, K1 the
//      lower cell; the value test gets +T_v (K1) or -T_v (K2),
//      T_v = sigma_F [u] - {dn u}, and the normal-derivative test -[u]/2;
//  * surrogate face: added from the face kernel's scratch.
// 3D: all terms of an axis as one operator per line (below).
#include "chunk_body.cuh"

namespace sbm {

// 2D: lines of n nodes, cells per block
template <int N>
struct Dg2 {
  static constexpr int ND = N * N;
  static constexpr int CPB = 128 / N;
};

template <typename T>
struct DgArgs {
  const T* __restrict__ x;
  T* __restrict__ y;
  const int32_t* __restrict__ cell_rank;   // ordered cell -> active-cell rank
  const int32_t* __restrict__ nbr;         // [rank][2k+s] neighbour rank or -1
  const int32_t* __restrict__ face_start;  // ordered cell -> surrogate-face range
  const int32_t* __restrict__ face_kind;   // 3D
  const T* __restrict__ face_out;          // [F][2L] from the face kernel
  const int32_t* __restrict__ cexp;        // 3D FP64: exponents of the cells
  int ncell;
  T sigma_f;
};

template <typename T, int N>
__global__ void __launch_bounds__(Dg2<N>::CPB * N)
dg_apply_kernel(const DgArgs<T> a, const __grid_constant__ KTab<T> t) {
  constexpr int ND = Dg2<N>::ND, CPB = Dg2<N>::CPB;
  using Pair2 = typename PairOf<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* A = reinterpret_cast<T*>(smem_raw);       // pair tile of the sweeps, then the results
  Pair2* AE = reinterpret_cast<Pair2*>(smem_raw);
  T* X = A + 2 * CPB * ND;                     // CPB input tiles
  T* P1 = X + CPB * ND;                        // face scratch, CPB * N each
  T* P2 = P1 + CPB * N;
  const int tid = threadIdx.x;
  const int first = blockIdx.x * CPB;
  const int ncells = min(CPB, a.ncell - first);
  for (int r = tid; r < ncells * ND; r += blockDim.x) {
    const int c = r / ND;
    X[r] = __ldg(a.x + (size_t)__ldg(a.cell_rank + first + c) * ND + (r - c * ND));
  }
  __syncthreads();
  const int c = tid / N, tl = tid - c * N;
  const bool act = c < ncells;
  const int pos = first + (act ? c : 0);
  const int rank = __ldg(a.cell_rank + pos);
  T* Xc = X + c * ND;
  T* R = A + c * ND;
  {
    // cell term (Algorithm 1), then the x-line result into R once every
    // thread is past the sweeps
    T out[N];
    cell_sweeps_2d<T, N>(t, X, c * ND + tl, N, AE, c, tl, act, out);
    __syncthreads();
    if (act) {
#pragma unroll
      for (int m = 0; m < N; ++m) R[N * tl + m] = out[m];
    }
  }
  __syncthreads();

  int fptr = act ? __ldg(a.face_start + pos) : 0;   // next surrogate face of this cell
  T* p1 = P1 + c * N;
  T* p2 = P2 + c * N;
  for (int k = 0; k < 2; ++k) {
    const int sk = (k == 0) ? 1 : N, bt = tl * ((k == 0) ? N : 1);
    for (int s = 0; s < 2; ++s) {
      const int nb = act ? __ldg(a.nbr + (size_t)rank * 4 + 2 * k + s) : -1;
      const bool interior = nb >= 0;
      const int kend = s ? N - 1 : 0;
      const T sg = s ? T(1) : T(-1);
      const T* fo = nullptr;
      if (act && !interior) fo = a.face_out + (size_t)(fptr++) * 2 * N;
      // A. nodal traces (own side and, for interior faces, the neighbour's),
      // and the two integrands in nodal form: with Gauss quadrature exact on
      // the face, interpolating to the Gauss points, weighting and
      // interpolating back is h M (the exact 1D mass matrix), so
      //   value test:  h M sg (sigma_F [u] - h^-1 {d_k u}),
      //   normal-derivative test:  h M (-[u] / (2 h))
      if (act) {
        T um = Xc[kend * sk + bt], dm = T(0);
#pragma unroll
        for (int j = 0; j < N; ++j) dm = fma(s ? t.D1[j] : t.D0[j], Xc[j * sk + bt], dm);
        T a1 = T(0), a2 = T(0);
        if (interior) {
          const T* xn = a.x + (size_t)nb * ND;
          const int nend = s ? 0 : N - 1;
          T un = __ldg(xn + nend * sk + bt), dnb = T(0);
#pragma unroll
          for (int j = 0; j < N; ++j)
            dnb = fma(s ? t.D0[j] : t.D1[j], __ldg(xn + j * sk + bt), dnb);
          const T jump = s ? (um - un) : (un - um);        // [u] = u_K1 - u_K2
          const T avg = T(0.5) * (dm + dnb);               // {d_k u} (reference)
          a1 = (sg * t.hface) * (a.sigma_f * jump - t.h_inv * avg);
          a2 = (T(-0.5) * t.hface * t.h_inv) * jump;
        }
        p1[tl] = a1;
        p2[tl] = a2;
      }
      __syncthreads();
      // B. M on both integrands
      if (act) {
        T rv = T(0), rg = T(0);
#pragma unroll
        for (int j = 0; j < N; ++j) {
          rv = fma(t.M[tl][j], p1[j], rv);
          rg = fma(t.M[tl][j], p2[j], rg);
        }
        if (!interior) {                // surrogate face: results of the face kernel
          rv = __ldg(fo + tl);
          rg = __ldg(fo + N + tl);
        }
        R[kend * sk + bt] += rv;
#pragma unroll
        for (int j = 0; j < N; ++j)
          R[j * sk + bt] = fma(s ? t.D1[j] : t.D0[j], rg, R[j * sk + bt]);
      }
      __syncthreads();
    }
  }
  for (int r = tid; r < ncells * ND; r += blockDim.x) {
    const int cc = r / ND;
    a.y[(size_t)__ldg(a.cell_rank + first + cc) * ND + (r - cc * ND)] = A[r];
  }
}

// ---- 3D ------------------------------------------------------------------------
//
// With exact quadrature the interior-face terms of axis k have the tensor
// structure of the cell term, a 1D operator along k times the mass matrices
// of the other two axes.  Per line along k, with g_s = u - (the neighbour's
// line, mirrored in the face s):
//   r_k = K u + sum_{s interior} Own_s g_s,
//   Own_s = pen e_s e_s^T - 1/2 sg (e_s D_s^T + D_s e_s^T)
// (the mirrored neighbour has the negative of the end derivative D_s, so jump
// and mean of the normal derivative are both products of g_s), and
//   y = h (M_z (M_y r_x + M_x r_y) + M_y M_x r_z) + surrogate faces.
// Each face costs 2n products per line instead of 7n (its traces, two mass
// products of the two integrands, the test functions); four line phases.
//
// FP64 runs on the integer units (fixed_point.cuh): the exponent of a cell is
// the largest of its own and its neighbours', from dg_exp_kernel (the two sides
// of a face can differ in it, and then round its terms differently); r_k of
// 57-bit values leaves at 59 bits, so that the sum of the last phase stays
// below 2^61.  The penalty is a part of w, and so of that scale, only while it
// no more than doubles the largest row sum (pen_interior = 1 gives 1.1 to 1.7
// times the sum without it).  A larger one would take the low bits of K u and
// of the jump with it, which a conforming u shows: error of a line whose traces
// match, against 128-bit tables, at up to twice the sum without penalty 4.2e-17
// (p = 1) .. 4.9e-14 (p = 6), in double precision 1.3e-15 .. 8.0e-14; at 8 to 14
// times 6.4e-16 .. 2.9e-13 against the same.  There dg_penalty adds it in double
// precision from the exact jumps (whole applies, inside / added: p = 1 of 656 832
// DoFs 29 / 50 us, p = 3 of 1.57 M 60 / 97, p = 6 of 2.05 M 113 / 164).
//
// Measured on GB300, whole applies, before (cell term, then six faces through
// traces, mass products and folds) -> now: FP64 torus of 64^3 cells at p = 3
// (1.57 M DoFs) 254 -> 61.5 us, FP32 35.3 -> 16.8 us.  FP64 is bound by the
// integer pipes, FP32 by launch and load latency at this size.
template <typename T>
struct DgTabs;
template <>
struct DgTabs<double> {
  fix::DgTab x;
};
template <>
struct DgTabs<float> {
  float w[kMaxN];                  // h w
};

template <typename T, int N>
struct Dg3 {
  static constexpr int L = N * N, ND = L * N;
  static constexpr int R = 256 / L;                       // cells per block
  static constexpr int NT = FixMap<N>::threads(R);
  static constexpr int PX = TilePad<T, N>::PX, NDP = TilePad<T, N>::NDP, PL = PX * N;
  static constexpr size_t smem = (size_t)4 * R * NDP * 8 / (8 / sizeof(T));
};

// FP32 lines: plain values
template <typename T, int N>
struct DgLine {
  using V = T;
  const KTab<T>& t;
  const DgTabs<T>& d;
  __device__ __forceinline__ V in(T x, int) const { return x; }
  __device__ __forceinline__ void stiff(const V (&v)[N], V (&y)[N]) const {
    line_apply<T, N>(t.Kh, t.fKh, v, y);
  }
  __device__ __forceinline__ void mass(const V (&v)[N], V (&y)[N]) const {
    line_apply<T, N>(t.M, t.fM, v, y);
  }
  // y_s += w . g, the end value of g
  template <int S>
  __device__ __forceinline__ V side(const V (&v)[N], const V (&nb)[N], V (&y)[N]) const {
    V r = T(0);
#pragma unroll
    for (int j = 0; j < N; ++j) r = fma(d.w[S ? N - 1 - j : j], v[j] - nb[N - 1 - j], r);
    y[S ? N - 1 : 0] += r;
    return S ? v[N - 1] - nb[0] : v[0] - nb[N - 1];
  }
  __device__ __forceinline__ void ends(V g0, V g1, V (&y)[N]) const {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      if (j > 0) y[j] = fma(d.w[j], g0, y[j]);
      if (j < N - 1) y[j] = fma(d.w[N - 1 - j], g1, y[j]);
    }
  }
};

// FP64 lines: fixed point
template <int N>
struct DgLine<double, N> {
  using V = int64_t;
  const KTab<double>& t;
  const DgTabs<double>& d;
  __device__ __forceinline__ V in(double x, int E) const {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    return (fix::plain_exp(E) ? fix::from_double<false>(b, E) : fix::from_double<true>(b, E)) >> 3;
  }
  __device__ __forceinline__ void stiff(const V (&v)[N], V (&y)[N]) const {
    fix::apply_line<N, 3>([&](int i, int j) { return d.x.K.E[i][j]; },
                          [&](int i, int j) { return d.x.K.O[i][j]; }, v, y);
  }
  __device__ __forceinline__ void mass(const V (&v)[N], V (&y)[N]) const {
    fix::apply_line<N, 0>([&](int i, int j) { return d.x.M.E[i][j]; },
                          [&](int i, int j) { return d.x.M.O[i][j]; }, v, y);
  }
  template <int S>
  __device__ __forceinline__ V side(const V (&v)[N], const V (&nb)[N], V (&y)[N]) const {
    fix::Split g[N];
#pragma unroll
    for (int j = 0; j < N; ++j) g[j] = fix::split(v[j] - nb[N - 1 - j]);
    y[S ? N - 1 : 0] += fix::dot<3, N>([&](int j) { return d.x.w[S ? N - 1 - j : j]; }, g);
    return S ? v[N - 1] - nb[0] : v[0] - nb[N - 1];
  }
  __device__ __forceinline__ void ends(V g0, V g1, V (&y)[N]) const {
    const fix::Split s0 = fix::split(g0), s1 = fix::split(g1);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      if (j == 0 || j == N - 1) {
        const fix::Split q[1] = {j ? s0 : s1};
        y[j] += fix::dot<3, 1>([&](int) { return d.x.w[N - 1]; }, q);
      } else {
        const fix::Split q[2] = {s0, s1};
        y[j] += fix::dot<3, 2>([&](int i) { return d.x.w[i ? N - 1 - j : j]; }, q);
      }
    }
  }
};

// r of one line: v the cell's values, nb0 / nb1 the neighbours' ranks (-1:
// none), element j of the same line of a neighbour at its base + off + st j
template <typename T, int N>
__device__ __forceinline__ void dg_line(const DgLine<T, N>& A, const T* __restrict__ x, int nb0,
                                        int nb1, int off, int st, int E,
                                        const typename DgLine<T, N>::V (&v)[N],
                                        typename DgLine<T, N>::V (&y)[N]) {
  using V = typename DgLine<T, N>::V;
  constexpr int ND = N * N * N;
  T f[N];
  V q[N], g0 = 0, g1 = 0;
  if (nb0 >= 0) {
#pragma unroll
    for (int j = 0; j < N; ++j) f[j] = __ldg(x + (size_t)nb0 * ND + off + st * j);
  }
  A.stiff(v, y);
  if (nb0 >= 0) {
#pragma unroll
    for (int j = 0; j < N; ++j) q[j] = A.in(f[j], E);
    g0 = A.template side<0>(v, q, y);
  }
  if (nb1 >= 0) {
#pragma unroll
    for (int j = 0; j < N; ++j) q[j] = A.in(__ldg(x + (size_t)nb1 * ND + off + st * j), E);
    g1 = A.template side<1>(v, q, y);
  }
  A.ends(g0, g1, y);
}

// exponent words (fixed_point.cuh) of the cells: groups of G lanes per cell
template <int N>
__global__ void __launch_bounds__(256)
dg_exp_kernel(const double* __restrict__ x, int32_t* __restrict__ e, int ncell) {
  constexpr int ND = N * N * N, G = ND < 32 ? 8 : 32;
  pdl_trigger();
  const int64_t cell = fix::group_of(blockIdx.x, 256, threadIdx.x, G);
  const int l = threadIdx.x % G;
  uint32_t m = 0u;
  if (cell < ncell)
#pragma unroll
    for (int i = l; i < ND; i += G)
      m = max(m, fix::mag_hi((uint64_t)__double_as_longlong(__ldg(x + (size_t)cell * ND + i))));
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(~0u, m, o));
  if (cell < ncell && l == 0) e[cell] = max(1, (int)(m >> 20));
  pdl_wait();                      // done only after the face kernel: the next one waits for both
}

// The penalty terms of a cell's interior faces, added to the z-line (la, lb) of
// the result: h^2 M x M (sigma_F (own - neighbour)) on the face's nodes.  By the
// whole block, the shared memory free: 6 n^2 doubles per cell, in place.
template <int N>
__device__ __forceinline__ void dg_penalty(const DgArgs<double>& a, const KTab<double>& t,
                                           unsigned char* smem_raw, int rank, const int (&nb)[6],
                                           int c, int tl, bool act, double (&out)[N]) {
  constexpr int L = N * N, ND = L * N;
  const int la = tl % N, lb = tl / N;
  double* P = reinterpret_cast<double*>(smem_raw) + (act ? c : 0) * 6 * L;
  double w[6];
  if (act) {
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const int k = f / 2, sk = k == 0 ? 1 : k == 1 ? N : L;
      const int bt = la * (k == 0 ? N : 1) + lb * (k == 2 ? N : L);
      const int own = bt + (f % 2 ? (N - 1) * sk : 0), other = bt + (f % 2 ? 0 : (N - 1) * sk);
      w[f] = 0.0;
      if (nb[f] >= 0)
        w[f] = t.hface * (a.sigma_f * (__ldg(a.x + (size_t)rank * ND + own) -
                                       __ldg(a.x + (size_t)nb[f] * ND + other)));
    }
  }
#pragma unroll
  for (int ax = 0; ax < 2; ++ax) {            // M along the two axes of the faces
    __syncthreads();
    if (act) {
#pragma unroll
      for (int f = 0; f < 6; ++f) P[f * L + tl] = w[f];
    }
    __syncthreads();
    if (act) {
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        w[f] = 0.0;
#pragma unroll
        for (int j = 0; j < N; ++j)
          w[f] = fma(t.M[ax ? lb : la][j], P[f * L + (ax ? la + N * j : j + N * lb)], w[f]);
      }
    }
  }
  __syncthreads();
  if (act) {
#pragma unroll
    for (int f = 0; f < 4; ++f) P[f * L + tl] = w[f];
  }
  __syncthreads();
  if (!act) return;
#pragma unroll
  for (int m = 0; m < N; ++m) {               // node (la, lb, m): x-faces (lb, m), y-faces (la, m)
    if (la == 0) out[m] += P[lb + N * m];
    if (la == N - 1) out[m] += P[L + lb + N * m];
    if (lb == 0) out[m] += P[2 * L + la + N * m];
    if (lb == N - 1) out[m] += P[3 * L + la + N * m];
  }
  out[0] += w[4];
  out[N - 1] += w[5];
}

// PEN: the penalty is not part of the line operators (FP64)
template <typename T, int N, bool PEN>
__global__ void __launch_bounds__(Dg3<T, N>::NT,
                                  std::is_same<T, double>::value && N > 4 ? (PEN ? 2 : 3) : 4)
dg3_kernel(const DgArgs<T> a, const __grid_constant__ KTab<T> t,
           const __grid_constant__ DgTabs<T> d) {
  using Sh = Dg3<T, N>;
  using Line = DgLine<T, N>;
  using V = typename Line::V;
  constexpr bool FX = std::is_same<T, double>::value;
  constexpr int L = Sh::L, ND = Sh::ND, PX = Sh::PX, PL = Sh::PL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x;
  int c, tl;
  FixMap<N>::of(tid, c, tl);
  const int first = blockIdx.x * Sh::R;
  const bool act = c < min(Sh::R, a.ncell - first);
  V* const U = reinterpret_cast<V*>(smem_raw) + (act ? c : 0) * Sh::NDP;
  V* const X = U + Sh::R * Sh::NDP;
  V* const Y = X + Sh::R * Sh::NDP;
  V* const Z = Y + Sh::R * Sh::NDP;
  const int la = tl % N, lb = tl / N;
  const int zl = la + PX * lb, yl = la + PL * lb, xl = PX * tl;   // first nodes of the lines
  const Line A{t, d};
  int rank = 0, E = 1;
  int nb[6] = {-1, -1, -1, -1, -1, -1};
  V v[N], y[N];
  if (act) {
    rank = __ldg(a.cell_rank + first + c);
    const int2* pn = reinterpret_cast<const int2*>(a.nbr + (size_t)rank * 6);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int2 p = __ldg(pn + k);
      nb[2 * k] = p.x;
      nb[2 * k + 1] = p.y;
    }
    T u[N];
#pragma unroll
    for (int j = 0; j < N; ++j) u[j] = __ldg(a.x + (size_t)rank * ND + tl + L * j);
    if constexpr (FX) {
      pdl_wait();                  // the exponents
      E = __ldcg(a.cexp + rank);
#pragma unroll
      for (int k = 0; k < 6; ++k)
        if (nb[k] >= 0) E = max(E, __ldcg(a.cexp + nb[k]));
    }
#pragma unroll
    for (int j = 0; j < N; ++j) U[zl + PL * j] = v[j] = A.in(u[j], E);
    dg_line<T, N>(A, a.x, nb[4], nb[5], tl, L, E, v, y);
#pragma unroll
    for (int j = 0; j < N; ++j) Z[zl + PL * j] = y[j];
  }
  FixMap<N>::sync(tid);
  if (act) {
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = U[yl + PX * j];
    dg_line<T, N>(A, a.x, nb[2], nb[3], la + L * lb, N, E, v, y);
#pragma unroll
    for (int j = 0; j < N; ++j) Y[yl + PX * j] = y[j];
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = U[xl + j];
    dg_line<T, N>(A, a.x, nb[0], nb[1], N * tl, 1, E, v, y);
#pragma unroll
    for (int j = 0; j < N; ++j) X[xl + j] = y[j];
  }
  FixMap<N>::sync(tid);
  if (act) {                       // y-lines: M_y r_x, M_y r_z
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = X[yl + PX * j];
    A.mass(v, y);
#pragma unroll
    for (int j = 0; j < N; ++j) X[yl + PX * j] = y[j];
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = Z[yl + PX * j];
    A.mass(v, y);
#pragma unroll
    for (int j = 0; j < N; ++j) Z[yl + PX * j] = y[j];
  }
  FixMap<N>::sync(tid);
  if (act) {                       // x-lines: M_y r_x + M_x r_y, M_x M_y r_z
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = Y[xl + j];
    A.mass(v, y);
#pragma unroll
    for (int j = 0; j < N; ++j) X[xl + j] += y[j];
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = Z[xl + j];
    A.mass(v, y);
#pragma unroll
    for (int j = 0; j < N; ++j) Z[xl + j] = y[j];
  }
  FixMap<N>::sync(tid);
  if (!PEN && !act) return;
  T out[N];                        // z-lines, back to the nodes read first
#pragma unroll
  for (int j = 0; j < N; ++j) v[j] = X[zl + PL * j];
  A.mass(v, y);
#pragma unroll
  for (int j = 0; j < N; ++j) y[j] += Z[zl + PL * j];
  if constexpr (FX) {
    const int eb = E + d.x.eoff;
    const bool bad = E == fix::kExpBad, plain = !bad && fix::plain_result(eb);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const uint64_t b = plain ? fix::to_double<false>(y[j], eb)
                               : (bad ? 0x7ff8000000000000ull : fix::to_double<true>(y[j], eb));
      out[j] = __longlong_as_double((long long)b);
    }
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) out[j] = y[j];
  }
  if constexpr (PEN) {
    dg_penalty<N>(a, t, smem_raw, rank, nb, c, tl, act, out);
    if (!act) return;
  }
  const int fs = __ldg(a.face_start + first + c), fe = __ldg(a.face_start + first + c + 1);
  if (!FX && fs < fe) pdl_wait();  // the face kernel's results
  for (int f = fs; f < fe; ++f) {
    const int kind = __ldg(a.face_kind + f);
    fold_face_z<T, N, true>(t, a.face_out + (size_t)f * 2 * L, kind & 3, kind >> 2, la, lb, out);
  }
#pragma unroll
  for (int j = 0; j < N; ++j) a.y[(size_t)rank * ND + tl + L * j] = out[j];
}

static DgTabs<double> dg_tabs(const HostProblem& hp, double) { return DgTabs<double>{hp.fx.dg}; }
static DgTabs<float> dg_tabs(const HostProblem& hp, float) {
  DgTabs<float> d = {};
  for (int j = 0; j < hp.n; ++j)
    d.w[j] = (float)(hp.h * (j ? 0.5 * hp.tab.D0[j] : hp.sigma_f * hp.h + hp.tab.D0[0]));
  return d;
}

template <typename T, int N, bool PEN>
static cudaError_t dg3_t(const HostProblem& hp, const DeviceData& dd, const T* x, T* y,
                         cudaStream_t st, Profiler* prof, int face_mode) {
  using Sh = Dg3<T, N>;
  constexpr bool FX = std::is_same<T, double>::value;
  static cudaError_t attr =
      Sh::smem > 48 * 1024
          ? cudaFuncSetAttribute(dg3_kernel<T, N, PEN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)Sh::smem)
          : cudaSuccess;
  if (attr != cudaSuccess) return attr;
  DgArgs<T> a = {};
  a.x = x;
  a.y = y;
  a.cell_rank = dd.cell_rank;
  a.nbr = dd.nbr;
  a.face_start = dd.face_start;
  a.face_kind = dd.face_kind;
  a.face_out = face_out_of<T>(dd);
  a.cexp = dd.dg_exp;
  a.sigma_f = (T)hp.sigma_f;
  a.ncell = dd.col_start[dd.ncolours];
  if (a.ncell == 0) return cudaSuccess;
  const bool pr = prof && prof->on;
  cudaError_t err;
  if (pr && (err = prof->mark(st)) != cudaSuccess) return err;
  int nlaunch = 1;
  bool pdl = false;
  if (dd.nface > 0) {
    if ((err = launch_faces<T>(hp, dd, x, face_out_of<T>(dd), face_mode, st)) != cudaSuccess)
      return err;
    nlaunch++;
    pdl = !pr;
  }
  if (pr && (err = prof->mark(st)) != cudaSuccess) return err;
  if constexpr (FX) {
    constexpr int G = Sh::ND < 32 ? 8 : 32;
    const unsigned gb = (unsigned)(((int64_t)a.ncell * G + 255) / 256);
    if ((err = launch_maybe_pdl(dg_exp_kernel<N>, dim3(gb), dim3(256), 0, st, pdl, x, dd.dg_exp,
                                a.ncell)) != cudaSuccess)
      return err;
    nlaunch++;
    pdl = !pr;
  }
  const unsigned grid = (unsigned)((a.ncell + Sh::R - 1) / Sh::R);
  if ((err = launch_maybe_pdl(dg3_kernel<T, N, PEN>, dim3(grid), dim3(Sh::NT), Sh::smem, st, pdl, a,
                              make_ktab<T>(hp), dg_tabs(hp, T(0)))) != cudaSuccess)
    return err;
  if (pr) {
    prof->count(nlaunch);
    if ((err = prof->mark(st)) != cudaSuccess) return err;   // cell phase ends
    return prof->mark(st);                                   // no assembly phase
  }
  return cudaSuccess;
}

template <typename T, int N>
static cudaError_t dg2_t(const HostProblem& hp, const DeviceData& dd, const T* x, T* y,
                         cudaStream_t st, Profiler* prof, int face_mode) {
  constexpr int ND = Dg2<N>::ND, CPB = Dg2<N>::CPB;
  constexpr size_t smem = (size_t)(3 * CPB * ND + 2 * CPB * N) * sizeof(T);
  static_assert(smem <= 48 * 1024, "2D DG block");
  cudaError_t err;
  DgArgs<T> a = {};
  a.x = x;
  a.y = y;
  a.cell_rank = dd.cell_rank;
  a.nbr = dd.nbr;
  a.face_start = dd.face_start;
  a.face_out = face_out_of<T>(dd);
  a.ncell = dd.col_start[dd.ncolours];
  a.sigma_f = (T)hp.sigma_f;
  const bool pr = prof && prof->on;
  if (pr && (err = prof->mark(st)) != cudaSuccess) return err;
  int nlaunch = 1;
  if (dd.nface > 0) {
    if ((err = launch_faces<T>(hp, dd, x, face_out_of<T>(dd), face_mode, st)) != cudaSuccess)
      return err;
    nlaunch++;
  }
  if (pr && (err = prof->mark(st)) != cudaSuccess) return err;
  dg_apply_kernel<T, N><<<(a.ncell + CPB - 1) / CPB, CPB * N, smem, st>>>(a, make_ktab<T>(hp));
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  if (pr) {
    prof->count(nlaunch);
    if ((err = prof->mark(st)) != cudaSuccess) return err;   // cell phase ends
    return prof->mark(st);                                   // no assembly phase
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_dg_apply(const HostProblem& hp, const DeviceData& dd, const T* x, T* y,
                            cudaStream_t st, Profiler* prof, int face_mode) {
  constexpr bool FX = std::is_same<T, double>::value;
#define SBM_CASE(NN)                                                                     \
  if (hp.n == NN)                                                                        \
    return hp.d == 2          ? dg2_t<T, NN>(hp, dd, x, y, st, prof, face_mode)          \
           : hp.fx.dg_pen_in || !FX                                                      \
               ? dg3_t<T, NN, false>(hp, dd, x, y, st, prof, face_mode)                  \
               : dg3_t<T, NN, FX>(hp, dd, x, y, st, prof, face_mode);
  SBM_CASE(2) SBM_CASE(3) SBM_CASE(4) SBM_CASE(5) SBM_CASE(6) SBM_CASE(7)
#undef SBM_CASE
  return cudaErrorInvalidValue;
}
template cudaError_t launch_dg_apply<double>(const HostProblem&, const DeviceData&,
                                             const double*, double*, cudaStream_t, Profiler*,
                                             int);
template cudaError_t launch_dg_apply<float>(const HostProblem&, const DeviceData&, const float*,
                                            float*, cudaStream_t, Profiler*, int);

}  // namespace sbm
