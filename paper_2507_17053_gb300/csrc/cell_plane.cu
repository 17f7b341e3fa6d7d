// Cell term of the continuous Galerkin apply with n threads per cell, each
// holding one x-plane of the cell (n^2 nodes) in registers (3D): tile shape 2
// of the single applies.
//
// The chunk kernel (cg_apply.cu) holds one line per thread: every one of the
// five line phases of the eigenbasis cell term (Algorithm 1 in the exact form
// sweeps.cuh describes) passes through shared memory, n reads and n writes
// per line and a barrier.  Here a thread runs the z- and the y-phase of its
// plane on registers with compile-time indices; only the x-phase exchanges
// lines, inside the warp (whole cells per warp).  Per thread:
//  1. load the plane's nodes from x -- the n threads of a cell and the cells
//     of a warp read consecutive addresses;
//  2. z- and y-transforms, the plane to shared memory, the n x-lines of one
//     z-mode through h K + mu_ab M, back, y- and z-transforms back -- the same
//     per-line arithmetic as the chunk kernel;
//  3. fold in the surrogate faces' results, in the chunk kernel's order (only
//     the threads of cells with surrogate faces wait for the face kernel);
//  4. add the x-face values of the previous cell of the chunk (shared memory;
//     a block holds whole chunks), prev + own as the chunk kernel;
//  5. store every node (the last plane of a cell but the chunk's last belongs
//     to the next cell) into y or into the chunk's colour buffer, by the
//     chunk colouring of tile shape 0.
// The results are bitwise those of tile shape 0; the assembly kernel of that
// shape completes the DoFs several colours share.
// @PLANE@
#include <algorithm>

#include "chunk_body.cuh"

namespace sbm {

namespace {

// Warps per block: a block holds whole chunks of R = 256 / n^2 cells, chosen
// so that full chunks fill it.
template <int N>
struct PlaneShape {
  static constexpr int L = N * N;
  static constexpr int CW = 32 / N;                                  // cells per warp
  static constexpr int W = N == 3 ? 3 : N == 6 ? 7 : N <= 4 ? 4 : 5; // warps
  static constexpr int CPB = CW * W, NT = 32 * W;
  static constexpr int PX = N % 2 ? N : N + 1;                       // line stride
  static constexpr int CS = PX * L | 1;                              // cell stride
  static constexpr int MW = (L + 31) / 32;                           // mask words per plane
  static_assert(CPB >= 256 / L, "a block holds a chunk");
};
constexpr int plane_cells(int n) {
  return n == 2 ? PlaneShape<2>::CPB : n == 3 ? PlaneShape<3>::CPB : n == 4 ? PlaneShape<4>::CPB
       : n == 5 ? PlaneShape<5>::CPB : n == 6 ? PlaneShape<6>::CPB : PlaneShape<7>::CPB;
}

// resident warps asked of the compiler
#ifndef SBM_PW32
#define SBM_PW32 (N <= 4 ? 40 : N == 5 ? 30 : 20)
#endif
#ifndef SBM_PW64
#define SBM_PW64 (N <= 3 ? 32 : N == 4 ? 24 : N == 5 ? 20 : N == 6 ? 14 : 10)
#endif
template <typename T, int N>
constexpr int plane_min_blocks() {
  return (std::is_same<T, float>::value ? SBM_PW32 : SBM_PW64) / PlaneShape<N>::W;
}

template <typename T>
struct PlaneArgs {
  const T* __restrict__ x;
  T* __restrict__ y;
  T* __restrict__ ycol;                     // [ncolours][n_dofs]
  const int32_t* __restrict__ lines;        // ordered cells x L
  const int32_t* __restrict__ face_start;
  const int32_t* __restrict__ face_kind;
  const T* face_out;                        // [F][2L]
  const int32_t* __restrict__ chunk_first;  // tile shape 0
  const uint8_t* __restrict__ chunk_col;
  const int32_t* __restrict__ cell_chunk;   // ordered cell -> its chunk
  const uint32_t* __restrict__ mask;        // [Nc][n][MW]: node of the plane shared by several
                                            //   colours
  const int32_t* __restrict__ block_first;  // [nblocks + 1] first chunk of each block
  const fix::Entry* __restrict__ xfix;      // FP64: x-line operators
  int64_t n_dofs;
  int eoff;
};

// one line's phases; FP64 in fixed point
template <typename T, int N>
struct PlaneOps {
  using V = T;
  static __device__ __forceinline__ void to_modes(const KTab<T>& t, const V (&v)[N], V (&w)[N]) {
    line_to_modes<T, N>(t.fVt, v, w);
  }
  static __device__ __forceinline__ void xline(const T* m, const V (&v)[N], V (&y)[N]) {
    XLineShared<T, N>{m}.apply(v, y);
  }
  static __device__ __forceinline__ void back_y(const KTab<T>& t, const V (&w)[N], V (&y)[N]) {
    modes_to_line<T, N>(t.fV, w, y);
  }
  static __device__ __forceinline__ void back_z(const KTab<T>& t, const V (&w)[N], V (&y)[N]) {
    modes_to_line<T, N>(t.fV, w, y);
  }
};
template <int N>
struct PlaneOps<double, N> {
  using V = int64_t;
  static __device__ __forceinline__ void to_modes(const KTab<double>& t, const V (&v)[N],
                                                  V (&w)[N]) {
    fix::to_modes<N, 0>(t.xVt, v, w);
  }
  static __device__ __forceinline__ void xline(const double* md, const V (&v)[N], V (&y)[N]) {
    using Op = XLineOp<double, N>;
    constexpr int HE = (N + 1) / 2;
    const fix::Entry* m = reinterpret_cast<const fix::Entry*>(md);
    fix::apply_line<N, fix::shift_x(N)>(
        [&](int i, int j) { return m[Op::sym(i, j, HE)]; },
        [&](int i, int j) { return m[HE * (HE + 1) / 2 + Op::sym(i, j, N / 2)]; }, v, y);
  }
  static __device__ __forceinline__ void back_y(const KTab<double>& t, const V (&w)[N],
                                                V (&y)[N]) {
    fix::from_modes<N, fix::shift_y(N)>(t.xV, w, y);
  }
  static __device__ __forceinline__ void back_z(const KTab<double>& t, const V (&w)[N],
                                                V (&y)[N]) {
    fix::from_modes<N, fix::shift_z(N)>(t.xV, w, y);
  }
};

// surrogate face (k, s): fold_face_z's operations on the nodes (j0, y, z) of
// the thread's plane x = j0
template <typename T, int N>
__device__ __forceinline__ void fold_plane(const KTab<T>& t, const T* fo, int k, int s, int j0,
                                           T (&u)[N * N]) {
  constexpr int L = N * N;
  const T* rv = fo;
  const T* rg = fo + L;
  const int kend = s ? N - 1 : 0;
  if (k == 0) {
    const T dk = s ? t.D1[j0] : t.D0[j0];
#pragma unroll
    for (int l = 0; l < L; ++l) {
      T add = mul_rn(dk, ld_face<true>(rg + l));
      if (j0 == kend) add = add_rn(add, ld_face<true>(rv + l));
      u[l] = add_rn(u[l], add);
    }
  } else if (k == 1) {
#pragma unroll
    for (int m = 0; m < N; ++m) {
      const T g = ld_face<true>(rg + j0 + N * m), v = ld_face<true>(rv + j0 + N * m);
#pragma unroll
      for (int b = 0; b < N; ++b) {
        T add = mul_rn(s ? t.D1[b] : t.D0[b], g);
        if (b == kend) add = add_rn(add, v);
        u[b + N * m] = add_rn(u[b + N * m], add);
      }
    }
  } else {
#pragma unroll
    for (int b = 0; b < N; ++b) {
      const T g = ld_face<true>(rg + j0 + N * b), v = ld_face<true>(rv + j0 + N * b);
#pragma unroll
      for (int m = 0; m < N; ++m) {
        T& o = u[b + N * m];
        o = fma(s ? t.D1[m] : t.D0[m], g, o);
        if (m == kend) o = add_rn(o, v);
      }
    }
  }
}

template <typename T, int N>
__global__ void __launch_bounds__(PlaneShape<N>::NT, (plane_min_blocks<T, N>()))
cg_plane_kernel(const PlaneArgs<T> a, const __grid_constant__ KTab<T> t) {
  using Sh = PlaneShape<N>;
  using Op = PlaneOps<T, N>;
  using V = typename Op::V;
  using XO = XLineOp<T, N>;
  constexpr bool FX = std::is_same<T, double>::value;
  constexpr int L = Sh::L, P = N - 1, PX = Sh::PX, MW = Sh::MW;
  __shared__ V S[Sh::CPB * Sh::CS];
  __shared__ T xface[Sh::CPB][L | 1];           // j0 = P plane of each cell
  __shared__ T xops[XO::kSlots * XO::kPacked];
  const int tid = threadIdx.x, lane = tid & 31;
  const int cell = (tid >> 5) * Sh::CW + lane / N, j0 = lane % N;
  const int b0 = __ldg(a.block_first + blockIdx.x), b1 = __ldg(a.block_first + blockIdx.x + 1);
  const int c0 = __ldg(a.chunk_first + b0), c1 = __ldg(a.chunk_first + b1);
  const int pos = c0 + cell;
  const bool act = lane < Sh::CW * N && pos < c1;
  int c = 0, nc = 0, ch = 0, off = 0;
  const int32_t* ln = a.lines;
  T u[L];
  if (act) {
    ch = __ldg(a.cell_chunk + pos);
    const int f = __ldg(a.chunk_first + ch);
    c = pos - f;
    nc = __ldg(a.chunk_first + ch + 1) - f;
    ln += (size_t)f * L;                        // a chunk's lines continue from cell to cell
    off = P * c + j0;
#pragma unroll
    for (int l = 0; l < L; ++l) u[l] = __ldg(a.x + (__ldg(ln + l) + off));
  } else {
#pragma unroll
    for (int l = 0; l < L; ++l) u[l] = T(0);
  }
  if constexpr (FX) {
    xline_copy<N>(reinterpret_cast<fix::Entry*>(xops), a.xfix, tid);
  } else {
    if (tid < L && tid % N <= tid / N)
      XO(t, tid % N, tid / N).store(xops + XO::slot(tid % N, tid / N) * XO::kPacked);
  }
  V v[L], p[N], q[N];
  int E = 1;
  if constexpr (FX) {                           // the cell's exponent
    uint32_t mx = 0u;
#pragma unroll
    for (int l = 0; l < L; ++l) mx = max(mx, fix::mag_hi((uint64_t)__double_as_longlong(u[l])));
    uint32_t m = mx;
#pragma unroll
    for (int k = 1; k < N; ++k) {
      const int from = lane - j0 + (j0 + k < N ? j0 + k : j0 + k - N);
      m = max(m, __shfl_sync(0xffffffffu, mx, from & 31));
    }
    E = max(1, (int)(m >> 20));
    if (fix::plain_exp(E)) {
#pragma unroll
      for (int l = 0; l < L; ++l)
        v[l] = fix::from_double<false>((uint64_t)__double_as_longlong(u[l]), E);
    } else {
#pragma unroll
      for (int l = 0; l < L; ++l)
        v[l] = fix::from_double<true>((uint64_t)__double_as_longlong(u[l]), E);
    }
  } else {
#pragma unroll
    for (int l = 0; l < L; ++l) v[l] = u[l];
  }
#pragma unroll
  for (int a1 = 0; a1 < N; ++a1) {              // z-lines -> z-modes
#pragma unroll
    for (int k = 0; k < N; ++k) p[k] = v[a1 + N * k];
    Op::to_modes(t, p, q);
#pragma unroll
    for (int k = 0; k < N; ++k) v[a1 + N * k] = q[k];
  }
#pragma unroll
  for (int b = 0; b < N; ++b) {                 // y-lines -> y-modes
#pragma unroll
    for (int k = 0; k < N; ++k) p[k] = v[k + N * b];
    Op::to_modes(t, p, q);
#pragma unroll
    for (int k = 0; k < N; ++k) v[k + N * b] = q[k];
  }
  V* const Sc = S + (lane < Sh::CW * N ? cell : 0) * Sh::CS;
  if (act) {
#pragma unroll
    for (int l = 0; l < L; ++l) Sc[PX * l + j0] = v[l];
  }
  __syncthreads();                              // xops; the planes
  if (act) {                                    // x-lines of z-mode j0
#pragma unroll
    for (int a1 = 0; a1 < N; ++a1) {
      V* line = Sc + PX * (a1 + N * j0);
#pragma unroll
      for (int k = 0; k < N; ++k) p[k] = line[k];
      Op::xline(xops + XO::slot(a1, j0) * XO::kPacked, p, q);
#pragma unroll
      for (int k = 0; k < N; ++k) line[k] = q[k];
    }
  }
  __syncwarp();
  if (act) {
#pragma unroll
    for (int l = 0; l < L; ++l) v[l] = Sc[PX * l + j0];
  }
#pragma unroll
  for (int b = 0; b < N; ++b) {                 // y-modes back
#pragma unroll
    for (int k = 0; k < N; ++k) p[k] = v[k + N * b];
    Op::back_y(t, p, q);
#pragma unroll
    for (int k = 0; k < N; ++k) v[k + N * b] = q[k];
  }
#pragma unroll
  for (int a1 = 0; a1 < N; ++a1) {              // z-modes back
#pragma unroll
    for (int k = 0; k < N; ++k) p[k] = v[a1 + N * k];
    Op::back_z(t, p, q);
#pragma unroll
    for (int k = 0; k < N; ++k) v[a1 + N * k] = q[k];
  }
  if constexpr (FX) {
    if (fix::plain_exp(E)) {
#pragma unroll
      for (int l = 0; l < L; ++l)
        u[l] = __longlong_as_double((long long)fix::to_double<false>(v[l], E + a.eoff));
    } else {
#pragma unroll
      for (int l = 0; l < L; ++l)
        u[l] = E == fix::kExpBad
                   ? __longlong_as_double(0x7ff8000000000000ll)
                   : __longlong_as_double((long long)fix::to_double<true>(v[l], E + a.eoff));
    }
  } else {
#pragma unroll
    for (int l = 0; l < L; ++l) u[l] = v[l];
  }
  if (act) {
    const int fs = __ldg(a.face_start + pos), fe = __ldg(a.face_start + pos + 1);
    if (fs < fe) pdl_wait();
    for (int f2 = fs; f2 < fe; ++f2) {
      const int kind = __ldg(a.face_kind + f2);
      fold_plane<T, N>(t, a.face_out + (size_t)f2 * 2 * L, kind & 3, kind >> 2, j0, u);
    }
    if (j0 == P && c < nc - 1) {
#pragma unroll
      for (int l = 0; l < L; ++l) xface[cell][l] = u[l];
    }
  }
  __syncthreads();
  if (!act || (j0 == P && c < nc - 1)) return;
  // the x-face plane shared with the previous cell of the chunk: prev + own
  if (j0 == 0 && c > 0) {
#pragma unroll
    for (int l = 0; l < L; ++l) u[l] = add_rn(xface[cell - 1][l], u[l]);
  }
  uint32_t mk[MW];
#pragma unroll
  for (int i = 0; i < MW; ++i) mk[i] = __ldg(a.mask + ((size_t)pos * N + j0) * MW + i);
  T* yc = a.ycol + (size_t)__ldg(a.chunk_col + ch) * a.n_dofs;
#pragma unroll
  for (int l = 0; l < L; ++l) {
    T* dst = ((mk[l >> 5] >> (l & 31)) & 1u) ? yc : a.y;
    dst[__ldg(ln + l) + off] = u[l];
  }
}

// per-plane multi-colour bits from the chunk run bits (tile shape 0): node
// (j0, line l) of cell c of chunk ch is element l S + P c + j0 of the
// chunk's runs, S = P nc + 1; one thread per plane
__global__ void k_plane_mask(const int32_t* __restrict__ cell_chunk,
                             const int32_t* __restrict__ chunk_first,
                             const uint32_t* __restrict__ run_bits, int bit_words, int n,
                             int nc_all, int words, uint32_t* __restrict__ mask) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)nc_all * n) return;
  const int pos = (int)(i / n), j0 = (int)(i - (int64_t)pos * n);
  const int P = n - 1, L = n * n;
  const int ch = cell_chunk[pos];
  const int f = chunk_first[ch], nc = chunk_first[ch + 1] - f, c = pos - f;
  const int S = P * nc + 1;
  const uint32_t* bits = run_bits + (size_t)ch * bit_words;
  for (int w = 0; w < words; ++w) {
    uint32_t m = 0u;
    for (int l = 32 * w; l < min(L, 32 * w + 32); ++l) {
      const int e = l * S + P * c + j0;
      if ((bits[e >> 5] >> (e & 31)) & 1u) m |= 1u << (l & 31);
    }
    mask[i * words + w] = m;
  }
}

template <typename T, int N>
cudaError_t launch_plane(const HostProblem& hp, const DeviceData& dd, const T* x, T* y,
                         const T* fo, T* ycol, cudaStream_t st, bool pdl) {
  PlaneArgs<T> a;
  a.x = x;
  a.y = y;
  a.ycol = ycol;
  a.lines = dd.lines;
  a.face_start = dd.face_start;
  a.face_kind = dd.face_kind;
  a.face_out = fo;
  a.chunk_first = dd.chunks[0].first;
  a.chunk_col = dd.chunks[0].colour;
  a.cell_chunk = dd.plane_cell_chunk;
  a.mask = dd.plane_mask;
  a.block_first = dd.plane_block_first;
  a.xfix = dd.xfix;
  a.n_dofs = hp.n_dofs;
  a.eoff = hp.fx.eoff;
  // pdl: a programmatic dependent of the face kernel; a thread waits for it
  // only when its cell has surrogate faces and reads the results with
  // coherent loads.  The kernel does not trigger its own dependents early
  // (the assembly starts as its blocks finish).
  return launch_maybe_pdl(cg_plane_kernel<T, N>, dim3(dd.plane_nblocks), dim3(PlaneShape<N>::NT),
                          0, st, pdl, a, make_ktab<T>(hp));
}

}  // namespace

bool cell_plane_available(const HostProblem& hp, bool fp32) {
  return hp.d == 3 && !hp.desc.dg && hp.n >= 2 && hp.n <= (fp32 ? 7 : 7);
}

// The tables of tile shape 2 (3D continuous Galerkin): the chunk of every
// ordered cell, blocks of whole chunks (at most plane_cells(n) cells), and the
// per-plane multi-colour bits (from the device run bits of tile shape 0).
cudaError_t build_cell_plane_tables(const HostProblem& hp, const std::vector<int32_t>& ch_first,
                                    DeviceData* dd) {
  if (hp.d != 3 || hp.desc.dg) return cudaSuccess;
  const int nch = (int)ch_first.size() - 1;
  const int nc_all = ch_first.back();
  const int cells = plane_cells(hp.n);
  std::vector<int32_t> cell_chunk(nc_all), block_first;
  for (int q = 0; q < nch; ++q) {
    if (ch_first[q + 1] - ch_first[q] > cells) return cudaErrorInvalidValue;
    for (int i = ch_first[q]; i < ch_first[q + 1]; ++i) cell_chunk[i] = q;
  }
  for (int q = 0; q < nch;) {
    block_first.push_back(q);
    int q1 = q;
    while (q1 < nch && ch_first[q1 + 1] - ch_first[q] <= cells) ++q1;
    q = std::max(q1, q + 1);
  }
  block_first.push_back(nch);
  const int words = (hp.L + 31) / 32;
  cudaError_t e = cudaMalloc((void**)&dd->plane_cell_chunk, cell_chunk.size() * sizeof(int32_t));
  if (e == cudaSuccess)
    e = cudaMemcpy(dd->plane_cell_chunk, cell_chunk.data(), cell_chunk.size() * sizeof(int32_t),
                   cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMalloc((void**)&dd->plane_block_first, block_first.size() * sizeof(int32_t));
  if (e == cudaSuccess)
    e = cudaMemcpy(dd->plane_block_first, block_first.data(),
                   block_first.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMalloc((void**)&dd->plane_mask, (size_t)nc_all * hp.n * words * sizeof(uint32_t));
  if (e == cudaSuccess && nc_all > 0) {
    k_plane_mask<<<(unsigned)(((int64_t)nc_all * hp.n + 255) / 256), 256>>>(
        dd->plane_cell_chunk, dd->chunks[0].first, dd->chunks[0].run_bits,
        dd->chunks[0].bit_words, hp.n, nc_all, words, dd->plane_mask);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
  }
  dd->plane_nblocks = (int)block_first.size() - 1;
  return e;
}

template <typename T>
cudaError_t launch_cell_plane(const HostProblem& hp, const DeviceData& dd, const T* x, T* y,
                              const T* fo, T* ycol, cudaStream_t st, bool pdl) {
  if (!dd.plane_mask) return cudaErrorInvalidValue;
  switch (hp.n) {
    case 2: return launch_plane<T, 2>(hp, dd, x, y, fo, ycol, st, pdl);
    case 3: return launch_plane<T, 3>(hp, dd, x, y, fo, ycol, st, pdl);
    case 4: return launch_plane<T, 4>(hp, dd, x, y, fo, ycol, st, pdl);
    case 5: return launch_plane<T, 5>(hp, dd, x, y, fo, ycol, st, pdl);
    case 6: return launch_plane<T, 6>(hp, dd, x, y, fo, ycol, st, pdl);
    case 7: return launch_plane<T, 7>(hp, dd, x, y, fo, ycol, st, pdl);
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_cell_plane<float>(const HostProblem&, const DeviceData&, const float*,
                                              float*, const float*, float*, cudaStream_t, bool);
template cudaError_t launch_cell_plane<double>(const HostProblem&, const DeviceData&,
                                               const double*, double*, const double*, double*,
                                               cudaStream_t, bool);

}  // namespace sbm
