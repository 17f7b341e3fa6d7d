// Cell term of the continuous Galerkin FP32 apply with n threads per cell, each
// holding one x-plane of the cell (n^2 nodes) in registers (3D, p >= 3; at p = 1
// and 2 one thread holds the whole cell, cell_reg.cu).
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
// Measured on GB300, FP32 applies with the best other tile shape -> this:
// Q4 sphere of 96^3 cells 132 (one thread per cell, 168 registers and 12 warps
// per SM) -> 116 us (few cells: f32_few_cells in cg_apply.cu), Q3 57.7 -> 55.7, Q5 of 64^3 88.6 (chunks
// without staged runs) -> 77, Q6 ellipsoid of 48^3 48.9 -> 46.1 us.  The cell
// term of the Q4 sphere takes 71 us for 133 MB: load latency (6 of 13 stall
// cycles per instruction) and 1 180 instructions per warp of six cells.  In
// FP64 the fixed-point plane (50 registers and more of 64-bit values) is
// slower than the chunks (p = 4 535 against 372 us).
#include <algorithm>
#include <cmath>
#include <vector>

#include "chunk_body.cuh"

namespace sbm {

namespace {

// Warps per block: a block holds whole chunks of R = 256 / n^2 cells, chosen
// so that full chunks fill it.
template <int N>
struct PlaneShape {
  static constexpr int L = N * N;
  static constexpr int CW = 32 / N;                                  // cells per warp
  static constexpr int W = N == 4 ? 4 : N == 6 ? 7 : 5;              // warps
  static constexpr int CPB = CW * W, NT = 32 * W;
  static constexpr int PX = N % 2 ? N : N + 1;                       // line stride
  static constexpr int CS = PX * L | 1;                              // cell stride
  static constexpr int MW = (L + 31) / 32;                           // mask words per plane
  static_assert(CPB >= 256 / L, "a block holds a chunk");
};
constexpr int plane_cells(int n) {
  return n == 4 ? PlaneShape<4>::CPB : n == 5 ? PlaneShape<5>::CPB
       : n == 6 ? PlaneShape<6>::CPB : PlaneShape<7>::CPB;
}

// Resident warps asked of the compiler (FP32 applies, spheres of 96^3 cells at
// p = 3, 4, 64^3 at p = 5, ellipsoid of 48^3 at p = 6; 28 / 36 / 44 warps):
// p = 3 59.7 / 55.7 / 60.1 us, p = 4 119.1 / 115.3 / 121.4, p = 5 77.0 / 87.9 /
// 123.0 (spills), p = 6 46.1 with 20, 47.4 / 67.2 / 76.6.
constexpr int plane_warps(int n) { return n == 4 ? 36 : n == 5 ? 36 : n == 6 ? 28 : 20; }
template <int N>
constexpr int plane_min_blocks() { return plane_warps(N) / PlaneShape<N>::W; }

struct PlaneArgs {
  const float* __restrict__ x;
  float* __restrict__ y;
  float* __restrict__ ycol;                 // [ncolours][n_dofs]
  const int32_t* __restrict__ lines;        // ordered cells x L
  const int32_t* __restrict__ face_start;
  const int32_t* __restrict__ face_kind;
  const float* face_out;                    // [F][2L]
  const int32_t* __restrict__ chunk_first;  // tile shape 0
  const uint8_t* __restrict__ chunk_col;
  const int32_t* __restrict__ cell_chunk;   // ordered cell -> its chunk
  const uint32_t* __restrict__ mask;        // [Nc][n][MW]: node of the plane shared by several
                                            //   colours
  const int32_t* __restrict__ block_first;  // [nblocks + 1] first chunk of each block
  const float* __restrict__ xops;           // x-line operators, slot by slot (XLineOp)
  int64_t n_dofs;
};

// surrogate face (k, s): fold_face_z's operations on the nodes (j0, y, z) of
// the thread's plane x = j0
template <int N>
__device__ __forceinline__ void fold_plane(const KTab<float>& t, const float* fo, int k, int s, int j0,
                                           float (&u)[N * N]) {
  constexpr int L = N * N;
  const float* rv = fo;
  const float* rg = fo + L;
  const int kend = s ? N - 1 : 0;
  if (k == 0) {
    const float dk = s ? t.D1[j0] : t.D0[j0];
#pragma unroll
    for (int l = 0; l < L; ++l) {
      float add = mul_rn(dk, ld_face<true>(rg + l));
      if (j0 == kend) add = add_rn(add, ld_face<true>(rv + l));
      u[l] = add_rn(u[l], add);
    }
  } else if (k == 1) {
#pragma unroll
    for (int m = 0; m < N; ++m) {
      const float g = ld_face<true>(rg + j0 + N * m), v = ld_face<true>(rv + j0 + N * m);
#pragma unroll
      for (int b = 0; b < N; ++b) {
        float add = mul_rn(s ? t.D1[b] : t.D0[b], g);
        if (b == kend) add = add_rn(add, v);
        u[b + N * m] = add_rn(u[b + N * m], add);
      }
    }
  } else {
#pragma unroll
    for (int b = 0; b < N; ++b) {
      const float g = ld_face<true>(rg + j0 + N * b), v = ld_face<true>(rv + j0 + N * b);
#pragma unroll
      for (int m = 0; m < N; ++m) {
        float& o = u[b + N * m];
        o = fma(s ? t.D1[m] : t.D0[m], g, o);
        if (m == kend) o = add_rn(o, v);
      }
    }
  }
}

// h K + mu_ab M of modes (a, b) in XLineOp's packed form, as XLineShared
template <int N>
__device__ __forceinline__ void plane_xline(const float* m, const float (&v)[N],
                                            float (&y)[N]) {
  using Op = XLineOp<float, N>;
  constexpr int H = N / 2, HE = (N + 1) / 2;
  const LineFold<float, N> f(v);
  LineAcc<float, N> acc;
  const float* e = m;
  const float* o = m + HE * (HE + 1) / 2;
#pragma unroll
  for (int i = 0; i < HE; ++i)
#pragma unroll
    for (int j = 0; j < HE; ++j) acc.s[i] = fma(e[Op::sym(i, j, HE)], f.e[j], acc.s[i]);
#pragma unroll
  for (int i = 0; i < H; ++i)
#pragma unroll
    for (int j = 0; j < H; ++j) acc.d[i] = fma(o[Op::sym(i, j, H)], f.o[j], acc.d[i]);
  acc.unfold(y);
}

// barrier id of two warps; immediate ids, as a register one reserves all 16
template <int ID, int W>
__device__ __forceinline__ void pair_arrive(int id) {
  if constexpr (ID < W) {
    if (id == ID) asm volatile("bar.arrive %0, 64;" ::"n"(ID) : "memory");
    else pair_arrive<ID + 1, W>(id);
  }
}
template <int ID, int W>
__device__ __forceinline__ void pair_wait(int id) {
  if constexpr (ID < W) {
    if (id == ID) asm volatile("bar.sync %0, 64;" ::"n"(ID) : "memory");
    else pair_wait<ID + 1, W>(id);
  }
}

// Warps run independently but for the x-face of two cells of a chunk in
// neighbouring warps: the first one arrives at a barrier of the two when its
// plane is stored, the second one waits there.
template <int N>
__global__ void __launch_bounds__(PlaneShape<N>::NT, (plane_min_blocks<N>()))
cg_plane_kernel(const PlaneArgs a, const __grid_constant__ KTab<float> t) {
  using Sh = PlaneShape<N>;
  using XO = XLineOp<float, N>;
  constexpr int L = Sh::L, P = N - 1, PX = Sh::PX, MW = Sh::MW, LAST = Sh::CW * N - 1;
  __shared__ float S[Sh::CPB * Sh::CS];
  __shared__ float xops[XO::kSlots * XO::kPacked];
  for (int i = threadIdx.x; i < XO::kSlots * XO::kPacked; i += Sh::NT) xops[i] = __ldg(a.xops + i);
  __shared__ float xface[Sh::W][L];             // j0 = P plane of a warp's last cell
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int cell = w * Sh::CW + lane / N, j0 = lane % N;
  const int b0 = __ldg(a.block_first + blockIdx.x), b1 = __ldg(a.block_first + blockIdx.x + 1);
  const int c0 = __ldg(a.chunk_first + b0), c1 = __ldg(a.chunk_first + b1);
  const int pos = c0 + cell;
  const bool act = lane <= LAST && pos < c1;
  int c = 0, nc = 0, ch = 0, off = 0;
  const int32_t* ln = a.lines;
  float u[L], p[N], q[N];
  if (act) {
    ch = __ldg(a.cell_chunk + pos);
    const int f = __ldg(a.chunk_first + ch);
    c = pos - f;
    nc = __ldg(a.chunk_first + ch + 1) - f;
    ln += (size_t)f * L;                        // a chunk's lines continue from cell to cell
    off = P * c + j0;
#pragma unroll
    for (int l = 0; l < L; ++l) u[l] = __ldg(a.x + (__ldg(ln + l) + off));
#pragma unroll
    for (int a1 = 0; a1 < N; ++a1) {            // z-lines -> z-modes
#pragma unroll
      for (int k = 0; k < N; ++k) p[k] = u[a1 + N * k];
      line_to_modes<float, N>(t.fVt, p, q);
#pragma unroll
      for (int k = 0; k < N; ++k) u[a1 + N * k] = q[k];
    }
    float* Sc = S + cell * Sh::CS;
#pragma unroll
    for (int b = 0; b < N; ++b) {               // y-lines -> y-modes
#pragma unroll
      for (int k = 0; k < N; ++k) p[k] = u[k + N * b];
      line_to_modes<float, N>(t.fVt, p, q);
#pragma unroll
      for (int k = 0; k < N; ++k) Sc[PX * (k + N * b) + j0] = q[k];
    }
  }
  __syncthreads();                              // xops; the planes
  if (act) {                                    // x-lines of z-mode j0
#pragma unroll
    for (int a1 = 0; a1 < N; ++a1) {
      float* line = S + cell * Sh::CS + PX * (a1 + N * j0);
#pragma unroll
      for (int k = 0; k < N; ++k) p[k] = line[k];
      plane_xline<N>(xops + XO::slot(a1, j0) * XO::kPacked, p, q);
#pragma unroll
      for (int k = 0; k < N; ++k) line[k] = q[k];
    }
  }
  __syncwarp();
  if (act) {
    const float* Sc = S + cell * Sh::CS;
#pragma unroll
    for (int b = 0; b < N; ++b) {               // y-modes back
#pragma unroll
      for (int k = 0; k < N; ++k) p[k] = Sc[PX * (k + N * b) + j0];
      modes_to_line<float, N>(t.fV, p, q);
#pragma unroll
      for (int k = 0; k < N; ++k) u[k + N * b] = q[k];
    }
#pragma unroll
    for (int a1 = 0; a1 < N; ++a1) {            // z-modes back
#pragma unroll
      for (int k = 0; k < N; ++k) p[k] = u[a1 + N * k];
      modes_to_line<float, N>(t.fV, p, q);
#pragma unroll
      for (int k = 0; k < N; ++k) u[a1 + N * k] = q[k];
    }
    const int fs = __ldg(a.face_start + pos), fe = __ldg(a.face_start + pos + 1);
    if (fs < fe) pdl_wait();
    for (int f2 = fs; f2 < fe; ++f2) {
      const int kind = __ldg(a.face_kind + f2);
      fold_plane<N>(t, a.face_out + (size_t)f2 * 2 * L, kind & 3, kind >> 2, j0, u);
    }
  }
  __syncwarp();
  // the x-face plane shared with the previous cell of the chunk: prev + own
  if (w + 1 < Sh::W) {
    if (lane == LAST) {
#pragma unroll
      for (int l = 0; l < L; ++l) xface[w][l] = u[l];
    }
    __syncwarp();                 // the whole warp arrives, the plane stored
    pair_arrive<1, Sh::W>(w + 1);
  }
  __syncwarp();
  if (w > 0) pair_wait<1, Sh::W>(w);
  const bool add = act && j0 == 0 && c > 0;
#pragma unroll
  for (int l = 0; l < L; ++l) {
    float prev = __shfl_up_sync(0xffffffffu, u[l], 1);
    if (lane == 0 && add) prev = xface[w - 1][l];
    if (add) u[l] = add_rn(prev, u[l]);
  }
  if (!act || (j0 == P && c < nc - 1)) return;
  uint32_t mk[MW];
#pragma unroll
  for (int i = 0; i < MW; ++i) mk[i] = __ldg(a.mask + ((size_t)pos * N + j0) * MW + i);
  float* yc = a.ycol + (size_t)__ldg(a.chunk_col + ch) * a.n_dofs;
#pragma unroll
  for (int l = 0; l < L; ++l) {
    float* dst = ((mk[l >> 5] >> (l & 31)) & 1u) ? yc : a.y;
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

// the x-line operators, with the device's arithmetic (fused multiply-adds)
template <int N>
std::vector<float> make_xops(const KTab<float>& t) {
  using XO = XLineOp<float, N>;
  constexpr int H = N / 2, HE = (N + 1) / 2;
  std::vector<float> o((size_t)XO::kSlots * XO::kPacked, 0.f);
  for (int b = 0; b < N; ++b)
    for (int a = 0; a <= b; ++a) {
      float* m = o.data() + XO::sym(a, b, N) * XO::kPacked;
      const float mu = t.hlam[a] + t.hlam[b];
      for (int i = 0; i < HE; ++i)
        for (int j = i; j < HE; ++j) m[XO::tri(i, j, HE)] = std::fma(mu, t.fM.E[i][j], t.fKh.E[i][j]);
      for (int i = 0; i < H; ++i)
        for (int j = i; j < H; ++j)
          m[HE * (HE + 1) / 2 + XO::tri(i, j, H)] = std::fma(mu, t.fM.O[i][j], t.fKh.O[i][j]);
    }
  return o;
}

template <int N>
cudaError_t launch_plane(const HostProblem& hp, const DeviceData& dd, const float* x, float* y,
                         const float* fo, float* ycol, cudaStream_t st, bool pdl) {
  PlaneArgs a;
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
  a.xops = dd.plane_xops;
  a.n_dofs = hp.n_dofs;
  // pdl: a programmatic dependent of the face kernel; a thread waits for it
  // only when its cell has surrogate faces and reads the results with
  // coherent loads.  The kernel does not trigger its own dependents early
  // (the assembly starts as its blocks finish).
  return launch_maybe_pdl(cg_plane_kernel<N>, dim3(dd.plane_nblocks), dim3(PlaneShape<N>::NT), 0,
                          st, pdl, a, make_ktab<float>(hp));
}

std::vector<float> xops_of(const HostProblem& hp) {
  const KTab<float> t = make_ktab<float>(hp);
  switch (hp.n) {
    case 4: return make_xops<4>(t);
    case 5: return make_xops<5>(t);
    case 6: return make_xops<6>(t);
    default: return make_xops<7>(t);
  }
}

}  // namespace

bool cell_plane_used(const HostProblem& hp) { return hp.d == 3 && !hp.desc.dg && hp.n >= 4; }

// The tables of the plane kernel: the chunk of every
// ordered cell, blocks of whole chunks (at most plane_cells(n) cells), and the
// per-plane multi-colour bits (from the device run bits of tile shape 0).
cudaError_t build_cell_plane_tables(const HostProblem& hp, const std::vector<int32_t>& ch_first,
                                    DeviceData* dd) {
  if (!cell_plane_used(hp)) return cudaSuccess;
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
  const std::vector<float> xo = xops_of(hp);
  if (e == cudaSuccess) e = cudaMalloc((void**)&dd->plane_xops, xo.size() * sizeof(float));
  if (e == cudaSuccess)
    e = cudaMemcpy(dd->plane_xops, xo.data(), xo.size() * sizeof(float), cudaMemcpyHostToDevice);
  dd->plane_nblocks = (int)block_first.size() - 1;
  return e;
}

cudaError_t launch_cell_plane(const HostProblem& hp, const DeviceData& dd, const float* x,
                              float* y, const float* fo, float* ycol, cudaStream_t st, bool pdl) {
  if (!dd.plane_mask) return cudaErrorInvalidValue;
  switch (hp.n) {
    case 4: return launch_plane<4>(hp, dd, x, y, fo, ycol, st, pdl);
    case 5: return launch_plane<5>(hp, dd, x, y, fo, ycol, st, pdl);
    case 6: return launch_plane<6>(hp, dd, x, y, fo, ycol, st, pdl);
    case 7: return launch_plane<7>(hp, dd, x, y, fo, ycol, st, pdl);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sbm
