// Matrix-free apply (FP64 or FP32) of the continuous Galerkin SBM operator.
//
// One apply = three launches:
//  1. the surrogate-face kernel (face_kernel.cu, or tc_face.cu on the tensor
//     cores): every face into per-face scratch;
//  2. the chunk kernel.  Active cells are cut into chunks: up to R
//     consecutive active cells of one x-row of the mesh.  In the compact DoF
//     numbering the x-lines of consecutive active cells continue each other,
//     so the chunk's line (j1, j2) is one contiguous run of p*nc + 1 values:
//     the block gathers those runs coalesced, runs the cell sweeps
//     (Algorithm 1) for each cell, folds in the cells' surrogate faces, sums
//     the values of the x-face nodes its consecutive cells share in shared
//     memory, and writes each run once, coalesced: a DoF that no other chunk
//     touches goes straight to y, any other into the accumulation buffer of
//     the chunk's colour.  A chunk's colour is (its parity within its row
//     run, cy mod 2[, cz mod 2]); chunks of one colour share no DoF, so every
//     element of y and of the buffers has a single writer;
//  3. the assembly kernel, over the DoFs that two colours or more touch:
//     y_i = sum over those colours (a per-DoF bit mask) of buffer_c[i], in
//     fixed colour order.
// No atomics, no read-modify-write, no y = 0 fill; repeated applies are
// bitwise equal.
#include <algorithm>
#include <type_traits>

#include "chunk_body.cuh"

namespace sbm {

template <int D, int N>
struct ChunkShape {
  static constexpr int L = Shape<D, N>::L;
  static constexpr int R = (256 / L) > 0 ? (256 / L) : 1;     // cells per chunk
};

int chunk_cells(int d, int n) {
  const int L = (d == 3) ? n * n : n;
  return (256 / L) > 0 ? (256 / L) : 1;
}

CellLaunch cell_launch_shape(int d, int n) {
  const int r = chunk_cells(d, n);
  return CellLaunch{d, n, r, r * ((d == 3) ? n * n : n)};
}


// Resident blocks asked of the compiler.  FP64 3D (fixed-point cell term),
// blocks of about 250 threads: 6 up to p = 3 (40 registers), 4 above (64; two
// blocks fewer per SM cost 10 % at p = 4 and 20 % at p = 5, 6); half-size
// blocks (shape 1) twice as many.  The others: none asked (0) gives 32 to 40
// registers, 1 gives 40 to 72.  Measured with 0 / 1 (us, disks of 400^2 and
// 900^2 cells): FP64 2D p = 3 56.1, 201 / 55.3, 202, p = 5 116, 500 / 114, 508, p
// = 6 159, 729 / 156, 719; FP32 2D p = 2 13.8, 25.0 / 14.5, 26.8, p = 6 29.2, 100 /
// 27.3, 105, half-size blocks p = 6 29.8, 103 / 27.1, 98.8; FP32 3D half-size
// blocks (balls of 20^3 and 48^3 cells) p = 2 14.0, 15.6 / 13.8, 17.4, p = 5 23.1,
// 54.1 / 15.4, 51.7.
template <typename T, int D, int N, int R>
constexpr int chunk_min_blocks() {
  constexpr bool half = R < ChunkShape<D, N>::R;
  if (kFixed<T, D>) return (N <= 4 ? 6 : 4) * (R * N * N <= 128 ? 2 : 1);
  if (std::is_same<T, double>::value) return N == 6 ? 0 : 1;
  return half && N >= (D == 2 ? 6 : 4) ? 1 : 0;
}

template <typename T, int D, int N, int R>
__global__ void __launch_bounds__(block_threads<T, D, N>(R), (chunk_min_blocks<T, D, N, R>()))
cg_chunk_kernel(const ChunkArgs<T> a, const __grid_constant__ KTab<T> t) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // launched as a programmatic dependent of the face kernel (coherent face
  // loads, a wait before the first chunk's cells)
  pdl_trigger();
  chunk_xline_build<T, D, N, R>(smem_raw, t, a.xfix, threadIdx.x);
  chunk_loop<T, D, N, R, true, block_threads<T, D, N>(R), true>(a, t, smem_raw, blockIdx.y,
                                                         a.q0 + blockIdx.x, a.q1, gridDim.x);
}

// The same chunks with colour-ordered stores (chunk_loop, ORD): a
// persistent grid taking chunks from the ticket counter, no assembly pass.
template <typename T, int D, int N, int R>
__global__ void __launch_bounds__(block_threads<T, D, N>(R))
cg_chunk_ord_kernel(const ChunkArgs<T> a, const __grid_constant__ KTab<T> t,
                    const __grid_constant__ OrdArgs o) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  chunk_xline_build<T, D, N, R>(smem_raw, t, a.xfix, threadIdx.x);
  chunk_loop_ord<T, D, N, R>(a, t, smem_raw, o);
}

// Tile shape 3 (3D): the chunks of shape 0 without staged runs.  Resident
// blocks asked of the compiler: FP32 6 (40 registers, no spills); FP64 5 up
// to p = 4 (48 registers), 4 above (64 registers; 5 would spill).
template <typename T, int N>
constexpr int direct_min_blocks() {
  return std::is_same<T, float>::value ? 6 : (N <= 5 ? 5 : 4);
}

template <typename T, int N, int R>
__global__ void __launch_bounds__(block_threads<T, 3, N>(R), (direct_min_blocks<T, N>()))
cg_direct_kernel(const ChunkArgs<T> a, const __grid_constant__ KTab<T> t) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_trigger();                                           // as cg_chunk_kernel
  chunk_loop_direct<T, N, R, true, false, true>(a, t, t, smem_raw, blockIdx.y,
                                                a.q0 + blockIdx.x, a.q1, gridDim.x);
}

template <typename T, int N, int R>
__global__ void __launch_bounds__(block_threads<T, 3, N>(R), (direct_min_blocks<T, N>()))
cg_direct_ord_kernel(const ChunkArgs<T> a, const __grid_constant__ KTab<T> t,
                     const __grid_constant__ OrdArgs o) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // waits before its folds: it may run as a dependent of the face kernel
  chunk_loop_direct<T, N, R, true, true, true>(a, t, t, smem_raw, 0, 0, 0, 0, &o);
}

// Resident blocks per SM x SMs of a kernel (the persistent grid of the
// colour-ordered launches), once per kernel.
template <typename K>
static cudaError_t resident_grid(K kernel, int threads, size_t smem, int* cache, int* grid) {
  if (*cache == 0) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && smem > 48 * 1024)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    if (e != cudaSuccess) return e;
    *cache = std::max(1, per_sm) * sms;
  }
  *grid = *cache;
  return cudaSuccess;
}

template <typename T, int N, int R>
static cudaError_t direct_prepare(int* grid_cap) {
  static int per_sm = 0, sms = 0;
  static cudaError_t attr = cudaSuccess;
  constexpr size_t smem = DirectSmem<T, N, R>::bytes;
  if (per_sm == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (smem > 48 * 1024)
      attr = cudaFuncSetAttribute(cg_direct_kernel<T, N, R>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cg_direct_kernel<T, N, R>,
                                                      block_threads<T, 3, N>(R), smem) != cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
  }
  *grid_cap = 4 * per_sm * sms;
  return attr;
}

// The DoFs that several colours touch (assemble_warp), one per thread;
// grid.y = right-hand side.
template <typename T>
__global__ void assemble_kernel(const T* __restrict__ ycol, const int32_t* __restrict__ multi,
                                const uint8_t* __restrict__ multi_mask, T* __restrict__ y,
                                int64_t n, int64_t nmulti, int ncol, int64_t ld_ycol = 0,
                                int64_t ldy = 0) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  assemble_warp<T, false>(ycol + blockIdx.y * ld_ycol, multi, multi_mask, y + blockIdx.y * ldy, n,
                          nmulti, ncol, t);
}

// Single right-hand side: two shared DoFs per thread (entries b + tid and
// b + 256 + tid of a 512-entry tile; assemble_pair).  FP32: Q4 sphere 41 ->
// 37.5 us, p = 3 20.6 -> 16.7 us against one per thread (four: 41 / 20.6).
// The tiles go in reverse list order (block 0 takes the last tile), so that
// the first blocks read the colour values the cell kernel stored last (the
// list ascends in DoF number, as its stores do).  Every DoF's sum is
// independent of the order.  Measured: Q4 sphere FP32 35.6 -> 33.1 us, FP64
// 50.0 -> 46.3 us in a loop of applies, and also faster with cold caches
// (ncu, FP64 39.0 -> 34.7 us), so L2 reuse is not the whole reason.
template <typename T>
__global__ void __launch_bounds__(256)
assemble_set_kernel(const T* __restrict__ ycol, const int32_t* __restrict__ multi,
                    const uint8_t* __restrict__ multi_mask, T* __restrict__ y, int64_t n,
                    int64_t nmulti, int ncol) {
  const int64_t tile = (int64_t)(gridDim.x - 1u - blockIdx.x);
  assemble_pair<T, false, true>(ycol, multi, multi_mask, y, n, nmulti,
                                                         ncol, tile * 512 + threadIdx.x, 256);
}

// Blocks of the chunk kernel: 4 x (resident blocks per SM) x SMs at most
// (each block walks over several chunks), capped by the number of chunks.
template <typename T, int D, int N, int R>
static cudaError_t chunk_prepare(int* grid_cap) {
  static int per_sm = 0, sms = 0;
  static cudaError_t attr = cudaSuccess;
  constexpr size_t smem = ChunkSmem<T, D, N, R>::bytes;
  if (per_sm == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (smem > 48 * 1024)
      attr = cudaFuncSetAttribute(cg_chunk_kernel<T, D, N, R>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cg_chunk_kernel<T, D, N, R>,
                                                      block_threads<T, D, N>(R), smem) != cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
  }
  *grid_cap = 4 * per_sm * sms;
  return attr;
}

static int sm_count() {
  static const int sms = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v;
  }();
  return sms;
}

// Which part of the operator one apply_r call runs: surrogate faces
// [f0, f1), chunks [q0, q1), shared DoFs [m0, m1) of the assembly list (all:
// f1 = q1 = m1 = -1).
struct Part {
  int f0 = 0, f1 = -1, q0 = 0, q1 = -1;
  int64_t m0 = 0, m1 = -1;
};

// face stage + chunk kernel + assembly, with explicit scratch and nrhs
// right-hand sides (x, y: nrhs vectors ld apart).
template <typename T, int D, int N, int R>
static cudaError_t apply_r(const HostProblem& hp, const DeviceData& dd, const ChunkTable& ct,
                           const T* x, T* y, int64_t ld, int nrhs, T* fo, T* ycol, int face_mode,
                           cudaStream_t st, Profiler* prof, Part part, bool reg,
                           bool direct, bool ord, bool allow_pdl) {
  constexpr int L = Shape<D, N>::L, NT = block_threads<T, D, N>(R);
  const KTab<T> t = make_ktab<T>(hp);
  constexpr size_t smem = ChunkSmem<T, D, N, R>::bytes;
  if (part.f1 < 0) part.f1 = dd.nface;
  if (part.q1 < 0) part.q1 = ct.n;
  if (part.m1 < 0) part.m1 = ct.nmulti;
  cudaError_t err;
  const bool pr = prof && prof->on;
  int nlaunch = 0;
  if (pr && (err = prof->mark(st)) != cudaSuccess) return err;
  // programmatic dependent launches (whole applies, no profiling marks
  // between the kernels): the cell kernels (shapes 0, 2, 3) after the
  // CUDA-core face kernel (which x's producers precede in the stream), the
  // assembly after the cell kernel.  Measured (unprofiled applies, GB300):
  // FP32 p = 6 ellipsoid (shape 3) 62.7 -> 57.4 us, p = 3 / 4 spheres
  // (shapes 0, 3) 1-5 % faster, shape 2 1-8 % faster (cell_plane.cu); FP64 (with
  // the fixed-point faces) disk of 1 801 DoFs 18.0 -> 14.1 us, p = 3 box of
  // 24^3 cells 29.2 -> 22.7, p = 6 ellipsoid 148 -> 137, p = 4 sphere 381 ->
  // 372 us.
  bool pdl_cell = false;
  if (part.f1 > part.f0) {
    err = face_mode != 0 ? launch_faces<T>(hp, dd, x, fo, face_mode, st)
                         : launch_face_kernel<T>(hp, dd, x, fo, st, part.f0, part.f1);
    if (err != cudaSuccess) return err;
    nlaunch++;
    pdl_cell = allow_pdl && !pr;
  }
  if (pr && (err = prof->mark(st)) != cudaSuccess) return err;
  ChunkArgs<T> a;
  a.x = x;
  a.y = y;
  a.ycol = ycol;
  a.run_bits = ct.run_bits;
  a.bit_words = ct.bit_words;
  a.lines = dd.lines;
  a.face_start = dd.face_start;
  a.face_kind = dd.face_kind;
  a.face_out = fo;
  a.chunk_first = ct.first;
  a.chunk_col = ct.colour;
  a.n_dofs = hp.n_dofs;
  a.q0 = part.q0;
  a.q1 = part.q1;
  a.xfix = dd.xfix;
  a.eoff = hp.fx.eoff;
  a.ldx = ld;
  a.ld_ycol = (int64_t)dd.ncolours * hp.n_dofs;
  a.ld_face = (int64_t)dd.nface * 2 * L;
  OrdArgs oa{ct.ord, ct.add_bits, ct.deps, ct.ndeps, ct.done, ct.tickets, dd.err_flag, ct.n,
             ct.dep_cap};
  const int nl0 = nlaunch;
  if (reg) {                 // one or n threads per cell (cell_reg.cu, cell_plane.cu)
    if constexpr (std::is_same<T, float>::value) {
      err = cell_reg_used(hp) ? launch_cell_reg(hp, dd, x, y, fo, ycol, st, pdl_cell)
                              : launch_cell_plane(hp, dd, x, y, fo, ycol, st, pdl_cell);
      if (err != cudaSuccess) return err;
      nlaunch++;
    }
  } else if (ord && part.q1 > part.q0) {      // colour-ordered stores, no assembly
    if constexpr (R == ChunkShape<D, N>::R) {
      static int cache = 0;
      int grid = 0;
      if (direct) {
        if constexpr (D == 3) {
          if ((err = resident_grid(cg_direct_ord_kernel<T, N, R>, NT,
                                   DirectSmem<T, N, R>::bytes, &cache, &grid)) != cudaSuccess)
            return err;
          if ((err = launch_maybe_pdl(cg_direct_ord_kernel<T, N, R>, dim3(std::min(grid, ct.n)),
                                      dim3(NT), DirectSmem<T, N, R>::bytes, st, pdl_cell, a,
                                      t, oa)) != cudaSuccess)
            return err;
        }
      } else {
        static int cache0 = 0;
        if ((err = resident_grid(cg_chunk_ord_kernel<T, D, N, R>, NT, smem, &cache0, &grid)) !=
            cudaSuccess)
          return err;
        // 2D FP64 p = 6 starts after the faces: its blocks, spread over the SMs that
        // the face kernel leaves, took 40.4 / 146 / 214 / 276 us as a dependent
        // against 37.5 / 126 / 188 / 266 (disks of 100^2 / 300^2 / 400^2 / 500^2
        // cells); p <= 5 gains 0 .. 25 %
        const bool pdl = pdl_cell && !(D == 2 && N == 7 && std::is_same<T, double>::value);
        if ((err = launch_maybe_pdl(cg_chunk_ord_kernel<T, D, N, R>, dim3(std::min(grid, ct.n)),
                                    dim3(NT), smem, st, pdl, a, t, oa)) != cudaSuccess)
          return err;
      }
      nlaunch++;
    }
  } else if (direct && part.q1 > part.q0) {   // tile shape 3: no staged runs (3D)
    if constexpr (D == 3 && R == ChunkShape<D, N>::R) {
      int dcap = 0;
      if ((err = direct_prepare<T, N, R>(&dcap)) != cudaSuccess) return err;
      const int grid = std::min(part.q1 - part.q0, dcap);
      if ((err = launch_maybe_pdl(cg_direct_kernel<T, N, R>, dim3(grid, nrhs), dim3(NT),
                                  DirectSmem<T, N, R>::bytes, st, pdl_cell, a, t)) !=
          cudaSuccess)
        return err;
      nlaunch++;
    }
  } else if (part.q1 > part.q0) {
    // (FP32 in 3D: whole applies on chunks of R cells are the register kernels')
    if constexpr (std::is_same<T, float>::value && D == 3 && R == ChunkShape<D, N>::R) {
      return cudaErrorInvalidValue;
    } else {
      int cap = 0;
      if ((err = chunk_prepare<T, D, N, R>(&cap)) != cudaSuccess) return err;
      const int grid = std::min(part.q1 - part.q0, cap);
      // 2D FP64 p = 6 with 3/4 to 3 full-size blocks per SM starts after the faces:
      // as a dependent its blocks fall unevenly on the SMs around the face kernel's,
      // one more on some, 37.6 against 29.3 us (disk of 100^2 cells, 149 blocks) and
      // 49.7 / 39.6 (148^2, 290); other counts and degrees gain 0 .. 20 %
      const int64_t quarters = (int64_t)grid * NT / (64 * (int64_t)sm_count());
      const bool pdl = pdl_cell && !(D == 2 && N == 7 && std::is_same<T, double>::value &&
                                     quarters >= 3 && quarters < 12);
      if ((err = launch_maybe_pdl(cg_chunk_kernel<T, D, N, R>, dim3(grid, nrhs), dim3(NT), smem,
                                  st, pdl, a, t)) != cudaSuccess)
        return err;
      nlaunch++;
    }
  }
  const bool pdl_asm = allow_pdl && !pr && nlaunch > nl0;
  if (pr && (err = prof->mark(st)) != cudaSuccess) return err;
  const int64_t n = hp.n_dofs, nm = ord ? 0 : part.m1 - part.m0;
  if (nm > 0 && nrhs == 1) {
    if ((err = launch_maybe_pdl(assemble_set_kernel<T>, dim3((unsigned)((nm + 511) / 512)),
                                dim3(256), 0, st, pdl_asm, (const T*)ycol,
                                (const int32_t*)(ct.multi + part.m0),
                                (const uint8_t*)(ct.multi_mask + part.m0), y, n, nm,
                                dd.ncolours)) != cudaSuccess)
      return err;
    nlaunch++;
  } else if (nm > 0) {
    assemble_kernel<T><<<dim3((unsigned)((nm + 255) / 256), nrhs), 256, 0, st>>>(
        ycol, ct.multi + part.m0, ct.multi_mask + part.m0, y, n, nm, dd.ncolours,
        (int64_t)dd.ncolours * n, ld);
    nlaunch++;
  }
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  if (pr) {
    prof->count(nlaunch);
    return prof->mark(st);
  }
  return cudaSuccess;
}

// FP32 applies of shape 0 too small for the plane kernel, whose threads each run
// n^2 lines: the time of one thread is a floor that more cells have to fill.
// Measured on balls (us, chunk kernel / plane kernel / shape 3): p = 4 1 502
// cells 15.5 / 15.8 / 14.3, 6 151 20.3 / 17.8 / 16.0, 11 956 27.2 / 20.4 / 23.0;
// p = 5 519 21.0 / 23.6 / 14.3, 6 151 27.2 / 29.1 / 21.9, 11 956 37.9 / 31.9 /
// 29.7, 20 719 52.8 / 39.3 / 41.8.  At p = 3 and 6 the plane kernel was never
// behind the chunk kernel.
bool f32_few_cells(const HostProblem& hp, const DeviceData& dd) {
  const int cells = dd.col_start[dd.ncolours];
  return hp.n == 5 ? cells < 9000 : hp.n == 6 && cells < 16000;
}

// variant 0: R cells per chunk; variant 1: R/2 (a second tile shape for the
// autotuner); variant 2: the cells of variant 0's chunks one thread or n
// threads each (FP32, whole applies; FP64 runs variant 0, which gives the same
// bits); variant 3 (3D): variant 0's chunks
// without staged runs (chunk_loop_direct; slabs too).  Both chunkings are built at set-up
// with the same colouring rule, so the variants give bitwise-equal results.
template <typename T, int D, int N>
static cudaError_t apply_t(const HostProblem& hp, const DeviceData& dd, const T* x, T* y,
                           int64_t ld, int nrhs, T* fo, T* ycol, int face_mode, int variant,
                           bool ordered, cudaStream_t st, Profiler* prof, int slab, int stages) {
  constexpr int R = ChunkShape<D, N>::R;
  constexpr int RH = (R / 2) > 0 ? R / 2 : 1;
  const int v = (variant == 1 && RH < R) ? 1 : 0;
  // FP32 whole applies of shapes 0 and 2 run the register kernels, which give
  // the same bits and were faster than the chunk kernel (us, chunk kernel / shape
  // 3 / register kernels: p = 1 128^3 47.5 / 35.1 / 24.8, p = 2 96^3 55.6 / 42.3 /
  // 24.4, p = 3 105 / 78.9 / 55.4, p = 4 195 / 153 / 114, p = 5 64^3 109 / 88.6 /
  // 77, p = 6 48^3 60 / 48.9 / 46.1), but for few cells at p = 4, 5: there shape 0
  // is shape 3 (f32_few_cells)
  const bool single32 = std::is_same<T, float>::value && D == 3 && slab < 0 && nrhs == 1;
  const bool few = single32 && variant == 0 && f32_few_cells(hp, dd);
  const bool reg = single32 && (variant == 2 || (variant == 0 && !ordered && !few));
  const bool direct = D == 3 && (variant == 3 || (few && !ordered));
  const ChunkTable& ct = dd.chunks[v];
  // colour-ordered stores: whole single applies of chunking 0 by the chunk
  // kernels (shapes 0 and 3; shape 2 keeps the colour buffers)
  const bool ord = ordered && v == 0 && !reg && slab < 0 && nrhs == 1 && ct.ordered;
  Part part;
  if (slab >= 0) {
    const bool faces = stages & 1, cells = stages & 2;
    part.f0 = dd.slab_face[slab];
    part.f1 = faces ? dd.slab_face[slab + 1] : part.f0;
    part.q0 = ct.slab_chunk[slab];
    part.q1 = cells ? ct.slab_chunk[slab + 1] : part.q0;
    part.m0 = ct.slab_multi[slab];
    part.m1 = cells ? ct.slab_multi[slab + 1] : part.m0;
  }
  if (v == 1)
    return apply_r<T, D, N, RH>(hp, dd, ct, x, y, ld, nrhs, fo, ycol, face_mode, st, prof, part,
                                false, false, false, slab < 0);
  return apply_r<T, D, N, R>(hp, dd, ct, x, y, ld, nrhs, fo, ycol, face_mode, st, prof, part,
                             reg, direct, ord, slab < 0);
}

template <typename T>
static cudaError_t dispatch(const HostProblem& hp, const DeviceData& dd, const T* x, T* y,
                            int64_t ld, int nrhs, T* fo, T* ycol, int face_mode, int variant,
                            bool ordered, cudaStream_t st, Profiler* prof, int slab = -1,
                            int stages = 3) {
#define SBM_CASE(DD, NN)                                                                   \
  if (hp.d == DD && hp.n == NN)                                                            \
    return apply_t<T, DD, NN>(hp, dd, x, y, ld, nrhs, fo, ycol, face_mode, variant, ordered, \
                              st, prof, slab, stages);
  SBM_CASE(2, 2) SBM_CASE(2, 3) SBM_CASE(2, 4) SBM_CASE(2, 5) SBM_CASE(2, 6) SBM_CASE(2, 7)
  SBM_CASE(3, 2) SBM_CASE(3, 3) SBM_CASE(3, 4) SBM_CASE(3, 5) SBM_CASE(3, 6) SBM_CASE(3, 7)
#undef SBM_CASE
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_cg_apply(const HostProblem& hp, const DeviceData& dd, const T* x, T* y,
                            cudaStream_t st, Profiler* prof, int face_mode) {
  const int pi = std::is_same<T, float>::value ? 1 : 0;
  return dispatch<T>(hp, dd, x, y, 0, 1, face_out_of<T>(dd), ycol_of<T>(dd), face_mode,
                     dd.variant[pi], dd.ordered[pi], st, prof);
}
template cudaError_t launch_cg_apply<double>(const HostProblem&, const DeviceData&,
                                             const double*, double*, cudaStream_t, Profiler*,
                                             int);
template cudaError_t launch_cg_apply<float>(const HostProblem&, const DeviceData&, const float*,
                                            float*, cudaStream_t, Profiler*, int);

// Slab s of the FP64 apply (the pipelined host-buffer apply): stages 1 =
// the surrogate faces of the cells of slab s, 2 = their chunks and the shared
// DoFs the slab completes; after both, y is final on the DoFs [slab_y[s],
// slab_y[s+1]) given x on [0, slab_x[s]).
cudaError_t launch_cg_apply_slab(const HostProblem& hp, const DeviceData& dd, const double* x,
                                 double* y, int slab, int stages, cudaStream_t st) {
  return dispatch<double>(hp, dd, x, y, 0, 1, dd.face_out, dd.ycol, 0, dd.variant[0], false, st,
                          nullptr, slab, stages);
}

// The same launches with caller-provided scratch: per-face results
// ([F][2L]) and colour buffers ([ncolours][n_dofs]).
template <typename T>
cudaError_t launch_cg_apply_scratch(const HostProblem& hp, const DeviceData& dd, const T* x, T* y,
                                    T* face_scratch, T* colour_scratch, int variant,
                                    cudaStream_t st) {
  return dispatch<T>(hp, dd, x, y, 0, 1, face_scratch, colour_scratch, 0, variant, false, st,
                     nullptr);
}
template cudaError_t launch_cg_apply_scratch<double>(const HostProblem&, const DeviceData&,
                                                     const double*, double*, double*, double*,
                                                     int, cudaStream_t);

}  // namespace sbm
