// Krylov drivers on the matrix-free operator: conjugate gradients, restarted
// GMRES, BiCGStab, and FP64 iterative refinement around an FP32 inner solve.
//
// The paper gives no solver; it states that the mat-vec dominates iterative
// solvers (Section 4.2).  These drivers keep every vector on the device:
//  * reductions are deterministic (fixed grid, fixed tree order, FP64
//    accumulation), so a solve is bitwise reproducible;
//  * CG keeps its scalars on the device; the host enqueues iterations
//    CG_AHEAD ahead of the outcome it reads, and a converged/failed flag turns
//    those after the last one into no-ops;
//  * GMRES(m) orthogonalises with classical Gram-Schmidt applied twice
//    (CGS2), three kernels per Arnoldi step; each writes its column of the
//    Hessenberg matrix to page-locked memory, and the host (Givens rotations)
//    follows one step behind, so the device never waits for it.
#include <algorithm>
#include <cmath>
#include <functional>
#include <vector>

#include "internal.hpp"
#include "krylov.hpp"

namespace sbm {

constexpr int RED_BLOCKS = 1216;   // 8 x 152 SMs
constexpr int RED_THREADS = 256;
constexpr int CG_AHEAD = 2;

// ---- deterministic reductions ---------------------------------------------

// The BiCGStab chunk's vector and scalar kernels are launched as
// programmatic dependents of the kernel before them (their launch overlaps
// its end); each waits for it before touching memory, so the order is that
// of the stream.  A no-op when a kernel is launched without the attribute.
__device__ __forceinline__ void pdl_wait_all() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Sums over the block in fixed order, in thread 0 (sh: 16 values).  The
// double-precision pipe does 2 operations per SM and clock, so additions are
// what a small reduction costs: warp shuffles, the two sums of block_sum2
// sharing theirs (half of the lanes carry on with each after the first step),
// then one warp over the warps' sums.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int tid = threadIdx.x;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(~0u, v, o);
  if ((tid & 31) == 0) sh[tid >> 5] = v;
  __syncthreads();
  double r = 0.0;
  if (tid < 32) {
    r = tid < RED_THREADS / 32 ? sh[tid] : 0.0;
    for (int o = RED_THREADS / 64; o > 0; o >>= 1) r += __shfl_xor_sync(~0u, r, o);
  }
  __syncthreads();
  return r;
}
__device__ __forceinline__ void block_sum2(double& a, double& b, double* sh) {
  const int tid = threadIdx.x;
  const bool h = tid & 16;
  double v = (h ? b : a) + __shfl_xor_sync(~0u, h ? a : b, 16);
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(~0u, v, o);
  if ((tid & 15) == 0) sh[(tid >> 5) + (h ? 8 : 0)] = v;
  __syncthreads();
  if (tid < 32) {
    double r = tid < RED_THREADS / 16 ? sh[tid] : 0.0;
    for (int o = RED_THREADS / 64; o > 0; o >>= 1) r += __shfl_xor_sync(~0u, r, o);
    a = r;
    b = __shfl_sync(~0u, r, 8);
  }
  __syncthreads();
}

// Blocks of a reduction over n values: 512 values per block (two per thread)
// up to two blocks per SM, so that a small vector's time is not that of its
// blocks' sums; 2 048 per block up to eight per SM, which a vector larger than
// the L2 cache needs to keep enough loads in flight.
static inline int red_blocks(int64_t n) {
  const int64_t b = std::min<int64_t>((n + 511) / 512, RED_BLOCKS / 4);
  return (int)std::max<int64_t>(1, std::max(b, std::min<int64_t>(n / 2048, RED_BLOCKS)));
}

// True in every thread of the grid's last block to get here, whose reads
// after it see what the other blocks wrote before theirs; *cnt counts the
// blocks and is left at zero.
__device__ __forceinline__ bool last_block(unsigned* cnt) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(cnt, 1u) == gridDim.x - 1u;
    if (s_last) *cnt = 0u;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

// sum of part[0 .. nb-1] (in thread 0), nb partials of other blocks
__device__ __forceinline__ double part_sum(const double* part, int nb, double* sh) {
  double s = 0.0;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) s += __ldcg(part + i);
  return block_sum(s, sh);
}

__device__ __forceinline__ void part_sum2(const double* part, int nb, double* sh, double (&v)[2]) {
  v[0] = v[1] = 0.0;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    v[0] += __ldcg(part + i);
    v[1] += __ldcg(part + RED_BLOCKS + i);
  }
  block_sum2(v[0], v[1], sh);
}

// part[j * RED_BLOCKS + block] = partial sum of a_j . b over this block's rows,
// a_j = a + j * lda (blockIdx.y = j).
template <typename T>
__global__ void k_multi_dot(const T* __restrict__ a, int64_t lda, const T* __restrict__ b,
                            int64_t n, double* __restrict__ part) {
  pdl_wait_all();
  __shared__ double sh[RED_THREADS / 16];
  const T* aj = a + (int64_t)blockIdx.y * lda;
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    s = fma((double)aj[i], (double)b[i], s);
  s = block_sum(s, sh);
  if (threadIdx.x == 0) part[blockIdx.y * RED_BLOCKS + blockIdx.x] = s;
}

// out[j] = sum of part[j * RED_BLOCKS + 0 .. nb-1] (blockIdx.x = j)
__global__ void k_finalize(const double* __restrict__ part, int nb, double* __restrict__ out) {
  __shared__ double sh[RED_THREADS / 16];
  const double s = part_sum(part + blockIdx.x * RED_BLOCKS, nb, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// ---- CG -----------------------------------------------------------------

struct CgState {
  double rz, pq, alpha, beta, rr, bb, tol2;
  int done;     // 0 running, 1 converged (recursive residual), 2 breakdown/divergence, 3 maxit
  int iters;
  int maxit;
  unsigned cnt[2];   // finished blocks of k_cg_dot and k_cg_update
};

// The vector work of an iteration is three kernels: the last block of a
// reduction also updates the scalars (five kernels before, box of 226 981
// DoFs, 372 iterations: 20.7 -> 18.1 ms).

// r = b - q; z = dinv * r (no preconditioner: z is r, not stored); p = z; partials of r.z, r.r, b.b
__global__ void k_cg_init(const double* __restrict__ b, const double* __restrict__ q,
                          double* __restrict__ r, double* z, double* __restrict__ p,
                          const double* __restrict__ dinv, int64_t n, double* __restrict__ part) {
  __shared__ double sh[RED_THREADS / 16];
  double srz = 0.0, srr = 0.0, sbb = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double ri = b[i] - q[i];
    const double zi = dinv ? ri * dinv[i] : ri;
    r[i] = ri;
    if (dinv) z[i] = zi;
    p[i] = zi;
    srz = fma(ri, zi, srz);
    srr = fma(ri, ri, srr);
    sbb = fma(b[i], b[i], sbb);
  }
  srz = block_sum(srz, sh);
  block_sum2(srr, sbb, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = srz;
    part[RED_BLOCKS + blockIdx.x] = srr;
    part[2 * RED_BLOCKS + blockIdx.x] = sbb;
  }
}

__global__ void k_cg_init_fin(const double* __restrict__ part, int nb, CgState* st) {
  __shared__ double sh[RED_THREADS / 16];
  double v[3];
  for (int j = 0; j < 3; ++j) {
    v[j] = part_sum(part + j * RED_BLOCKS, nb, sh);
  }
  if (threadIdx.x == 0) {
    st->rz = v[0];
    st->rr = v[1];
    st->bb = v[2];
    st->done = (v[1] <= st->tol2 * v[2]) ? 1 : 0;
    if (!(v[0] == v[0]) || v[2] == 0.0) st->done = (v[2] == 0.0) ? 1 : 2;
  }
}

// alpha = rz / (p, q): partials per block, the last block's sum
__global__ void k_cg_dot(const double* p, const double* q, int64_t n, double* part, CgState* st) {
  __shared__ double sh[RED_THREADS / 16];
  pdl_wait_all();
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    s = fma(p[i], q[i], s);
  s = block_sum(s, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
  if (!last_block(&st->cnt[0])) return;
  s = part_sum(part, gridDim.x, sh);
  if (threadIdx.x == 0) {
    st->pq = s;
    if (st->done) {
      st->alpha = 0.0;
    } else if (!(s != 0.0) || !isfinite(s)) {
      st->alpha = 0.0;
      st->done = 2;
    } else {
      st->alpha = st->rz / s;
    }
  }
}

// x += alpha p; r -= alpha q; z = dinv r; beta from r.z, r.r (the last block)
__global__ void k_cg_update(double* x, double* r, double* z, const double* p, const double* q,
                            const double* __restrict__ dinv, int64_t n, CgState* st,
                            double* part, int* host_done) {
  __shared__ double sh[RED_THREADS / 16];
  pdl_wait_all();
  const double al = st->alpha;
  double srz = 0.0, srr = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double pi = p[i], qi = q[i], xi = x[i], r0 = r[i];   // loads before the stores
    x[i] = fma(al, pi, xi);
    const double ri = fma(-al, qi, r0);
    r[i] = ri;
    srr = fma(ri, ri, srr);
    if (dinv) {
      const double zi = ri * dinv[i];
      z[i] = zi;
      srz = fma(ri, zi, srz);
    }
  }
  if (dinv) block_sum2(srz, srr, sh);
  else srz = srr = block_sum(srr, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = srz;
    part[RED_BLOCKS + blockIdx.x] = srr;
  }
  if (!last_block(&st->cnt[1])) return;
  double v[2];
  part_sum2(part, gridDim.x, sh, v);
  if (threadIdx.x == 0) {
    if (st->done) {
      st->beta = 0.0;
    } else {
      st->iters += 1;
      st->rr = v[1];
      if (v[1] <= st->tol2 * st->bb) st->done = 1;
      else if (!isfinite(v[1]) || v[1] > 1e24 * st->bb || !(v[0] != 0.0)) st->done = 2;
      else if (st->iters >= st->maxit) st->done = 3;
      st->beta = v[0] / st->rz;
      st->rz = v[0];
      if (st->done) st->beta = 0.0;
    }
    *host_done = st->done;
  }
}

__global__ void k_cg_p(double* p, const double* z, int64_t n, const CgState* st) {
  pdl_wait_all();
  if (st->done) return;
  const double be = st->beta;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    p[i] = fma(be, p[i], z[i]);
}

// dinv = 1 / diag
__global__ void k_reciprocal(const double* __restrict__ d, double* __restrict__ o, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    o[i] = 1.0 / d[i];
}

// ---- generic vector kernels (GMRES, IR) ------------------------------------

// y = b - y (y holds A x on entry)
template <typename T>
__global__ void k_residual(const T* __restrict__ b, T* __restrict__ y, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = b[i] - y[i];
}

// x += sum_j y[j] V_j, accumulated in double (x may be T or double)
template <typename TX, typename T>
__global__ void k_update_x(TX* __restrict__ x, const T* __restrict__ V, int64_t ldv,
                           const double* __restrict__ y, int m, double scale, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int j = 0; j < m; ++j) acc = fma(y[j], (double)V[j * ldv + i], acc);
    x[i] = (TX)((double)x[i] + scale * acc);
  }
}

template <typename TO, typename TI>
__global__ void k_convert_scaled(TO* __restrict__ o, const TI* __restrict__ in, double scale,
                                 int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    o[i] = (TO)((double)in[i] * scale);
}

// x += s * c (FP64)
__global__ void k_axpy_d(double* __restrict__ x, const double* __restrict__ c, double s,
                         int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    x[i] = fma(s, c[i], x[i]);
}

// x += s * c (c in FP32, x in FP64)
__global__ void k_add_scaled(double* __restrict__ x, const float* __restrict__ c, double s,
                             int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    x[i] = fma(s, (double)c[i], x[i]);
}

static inline int vec_grid(int64_t n) {
  int64_t g = (n + 255) / 256;
  return (int)(g < 4864 ? (g < 1 ? 1 : g) : 4864);
}

// ---- workspace ---------------------------------------------------------------

void Workspace::release() {
  for (void* p : bufs) cudaFree(p);
  bufs.clear();
}

cudaError_t Workspace::alloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaSuccess) bufs.push_back(*p);
  return e;
}

// dot products into dev scalars out[0..m-1] = a_j . b
template <typename T>
static cudaError_t multi_dot(const T* a, int64_t lda, const T* b, int64_t n, int m, double* part,
                             double* out, cudaStream_t st) {
  k_multi_dot<T><<<dim3(red_blocks(n), m), RED_THREADS, 0, st>>>(a, lda, b, n, part);
  k_finalize<<<m, RED_THREADS, 0, st>>>(part, red_blocks(n), out);
  return cudaGetLastError();
}

#define CK(x)                                   \
  do {                                          \
    cudaError_t e_ = (x);                       \
    if (e_ != cudaSuccess) return {SBM_ERR_CUDA, e_}; \
  } while (0)

// ---- CG --------------------------------------------------------------------

// Page-locked copy of the state, the iterations' outcomes and their events.
struct CgHost : HostRing {
  static constexpr int kRing = CG_AHEAD + 1;
  using HostRing::HostRing;
  CgState* state() { return (CgState*)mem; }
  int* done(int i) { return (int*)((char*)mem + 256) + i; }
  cudaError_t init() {
    static_assert(sizeof(CgState) <= 256, "CgHost layout");
    return HostRing::init(256 + kRing * sizeof(int), kRing);
  }
};

SolveStatus solve_cg(const ApplyFn<double>& apply, int64_t n, const double* b, double* x,
                     const double* diag, double rtol, int maxit, cudaStream_t st, Workspace& ws,
                     SolveInfo* info) {
  // one allocation: r, p, q [, z, 1 / diag], the partials and the state
  const int nb = red_blocks(n);
  const size_t vec = ((size_t)n * 8 + 255) / 256 * 256;
  char* base;
  CK(ws.alloc((void**)&base, vec * (diag ? 5 : 3) + 3 * RED_BLOCKS * 8 + sizeof(CgState)));
  double* r = (double*)base;
  double* p = (double*)(base + vec);
  double* q = (double*)(base + 2 * vec);
  double* z = diag ? (double*)(base + 3 * vec) : r;
  double* dinv = diag ? (double*)(base + 4 * vec) : nullptr;
  double* part = (double*)(base + vec * (diag ? 5 : 3));
  CgState* dst = (CgState*)(part + 3 * RED_BLOCKS);
  if (diag) {
    k_reciprocal<<<vec_grid(n), 256, 0, st>>>(diag, dinv, n);
    CK(cudaGetLastError());
  }
  CgHost ch(st);
  CK(ch.init());
  CgState* hs = ch.state();

  int total = 0, restarts = 0, status = SBM_NOT_DONE;
  double relres = INFINITY;
  SolveStatus ret{SBM_OK, cudaSuccess};
  while (true) {
    // (re)start from the current x: r = b - A x
    CgState init{};
    init.tol2 = rtol * rtol;
    init.maxit = maxit - total;
    CK(cudaMemcpyAsync(dst, &init, sizeof(CgState), cudaMemcpyHostToDevice, st));
    CK(apply(x, q, st));
    k_cg_init<<<nb, RED_THREADS, 0, st>>>(b, q, r, z, p, dinv, n, part);
    k_cg_init_fin<<<1, RED_THREADS, 0, st>>>(part, nb, dst);
    CK(cudaGetLastError());
    // the iterations, CG_AHEAD enqueued beyond the one whose outcome is read
    // (those after the last one change nothing)
    CK(cudaMemcpyAsync(hs, dst, sizeof(CgState), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    const double *cp = p, *cq = q, *cz = z, *cd = dinv;
    const int lim = hs->done ? 0 : init.maxit;
    for (int it = 0, enq = 0; it < lim; ++it) {
      for (; enq < lim && enq <= it + CG_AHEAD; ++enq) {
        const int slot = enq % CgHost::kRing;
        CK(apply(p, q, st));
        CK(launch_maybe_pdl(k_cg_dot, dim3(nb), dim3(RED_THREADS), 0, st, true, cp, cq, n, part,
                            dst));
        CK(launch_maybe_pdl(k_cg_update, dim3(nb), dim3(RED_THREADS), 0, st, true, x, r, z, cp,
                            cq, cd, n, dst, part, ch.done(slot)));
        CK(cudaEventRecord(ch.ev[slot], st));
        CK(launch_maybe_pdl(k_cg_p, dim3(vec_grid(n)), dim3(256), 0, st, true, p, cz, n,
                            (const CgState*)dst));
      }
      CK(cudaEventSynchronize(ch.ev[it % CgHost::kRing]));
      if (*ch.done(it % CgHost::kRing)) break;
    }
    CK(cudaMemcpyAsync(hs, dst, sizeof(CgState), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    const int done = hs->done;
    total += hs->iters;
    // true residual
    CK(apply(x, q, st));
    k_residual<double><<<vec_grid(n), 256, 0, st>>>(b, q, n);
    CK(multi_dot<double>(q, 0, q, n, 1, part, part + 2 * RED_BLOCKS, st));
    double rr;
    CK(cudaMemcpyAsync(&rr, part + 2 * RED_BLOCKS, 8, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    const double bb = hs->bb;
    relres = (bb > 0) ? std::sqrt(rr / bb) : 0.0;
    if (relres <= rtol) { status = SBM_OK; break; }
    if (done == 2 || done == 3 || total >= maxit || ++restarts > 5 || !std::isfinite(relres)) {
      status = SBM_ERR_NOT_CONVERGED;
      break;
    }
  }
  info->iters = total;
  info->relres = relres;
  info->restarts = restarts;
  ret.status = status;
  return ret;
}

// ---- Arnoldi step (GMRES) ----------------------------------------------------
//
// Basis vectors are kept unnormalised, v_i = s_i U_i (s_i = 1 / |U_i|), so no
// kernel only scales.  q = A U_j; one step is
//   kDot1   h1_i = s_j s_i (U_i, q)
//   kDot2   U_{j+1} = s_j q - sum_i h1_i s_i U_i,  h2_i = s_i (U_i, U_{j+1})
//   kNorm   U_{j+1} -= sum_i h2_i s_i U_i,  column h1 + h2, |U_{j+1}|
// A block owns gm_rows rows and walks them in tiles of tr rows: 256 / tr
// threads share a row's sum over i, a warp takes four dot products over the
// tile at a time.  The last block to finish sums the blocks' partials in
// block order, so results do not depend on the schedule.  Few rows: tiles of
// 64 rows and up to 8 blocks (gridDim.y) that split the dot products of the
// same rows (each repeats the rows' axpy; the double-precision pipe of one SM
// would bind, 2 operations per clock).
// Residual norm: with phi the left null vector of the (k+1) x k Hessenberg
// matrix, phi_0 = 1, it is beta / |phi|; one dot product per step ends the
// cycle on the device (ctl->done), where Givens rotations would be a chain of
// j dependent operations.
// Measured, disk of 1 801 DoFs, restart 100, 625 steps: whole solve 341 -> 26.6
// ms with the apply at 18 us (1 216 blocks per dot product, eleven stream
// operations and a host round trip per step before), 22.1 ms with it at 14.
constexpr int GM_MAXB = 304;       // row blocks at most, 2 per SM
constexpr int GM_SLICES = 8;       // blocks sharing the dot products of the same rows, at most
constexpr int GM_RING = 4;         // columns in flight to the host
constexpr int GM_AHEAD = 2;        // steps enqueued ahead of the host's test
enum { kDot1 = 0, kDot2 = 1, kNorm = 2 };

struct GmCtl {
  double sumphi2, beta, tol;       // |phi|^2, |r_0|, absolute residual to stop at
  int done;
  unsigned cnt[3][GM_SLICES];      // finished blocks (reset by the last one)
};

// scales, h1, h2, phi: [m + 1] each
struct GmVecs {
  double *s, *h1, *h2, *phi, *part;   // part [(m + 1)][GM_MAXB]
};

__global__ void k_gm_begin(GmCtl* ctl, GmVecs g, double beta, double tol) {
  ctl->sumphi2 = 1.0;
  ctl->beta = beta;
  ctl->tol = tol;
  ctl->done = 0;
  for (int i = 0; i < 3 * GM_SLICES; ++i) (&ctl->cnt[0][0])[i] = 0u;
  g.s[0] = 1.0;
  g.phi[0] = 1.0;
}

template <typename T, int MODE>
__global__ void __launch_bounds__(256)
k_gm_step(const T* q, T* V, int64_t n, int j, int rows, int tr,
          const GmVecs g, GmCtl* ctl, double* __restrict__ col) {
  extern __shared__ double gm_smem[];
  __shared__ double wt[256], red[256];
  __shared__ int s_last;
  pdl_wait_all();
  if (ctl->done) return;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nj = j + 1, per = (nj + gridDim.y - 1) / gridDim.y;
  const int i0 = min(nj, (int)blockIdx.y * per), i1 = min(nj, i0 + per);
  double* coef = gm_smem;            // [nj]
  double* dacc = gm_smem + nj;       // [per] dot products of the block's rows
  if (MODE != kDot1)
    for (int i = tid; i < nj; i += 256) coef[i] = (MODE == kDot2 ? g.h1[i] : g.h2[i]) * g.s[i];
  if (MODE != kNorm)
    for (int i = tid; i < per; i += 256) dacc[i] = 0.0;
  const double sj = g.s[j];
  T* u = V + (int64_t)nj * n;
  const int64_t r_end = min(n, ((int64_t)blockIdx.x + 1) * rows);
  const int r = tid % tr, js = tid / tr, split = 256 / tr;
  double nrm = 0.0;
  for (int64_t base = (int64_t)blockIdx.x * rows; base < r_end; base += tr) {
    const int nr = (int)min((int64_t)tr, r_end - base);
    __syncthreads();                 // coef; wt and red are reused
    if (MODE == kDot1) {
      if (tid < nr) wt[tid] = (double)q[base + tid];
    } else {
      double acc = 0.0;
      if (r < nr) {
        const T* vr = V + base + r;
#pragma unroll 4
        for (int i = js; i < nj; i += split) acc = fma(-coef[i], (double)vr[(int64_t)i * n], acc);
      }
      red[tid] = acc;
      __syncthreads();
      if (tid < nr) {
        double w = MODE == kDot2 ? sj * (double)q[base + tid] : (double)u[base + tid];
        for (int k = 0; k < split; ++k) w += red[tid + k * tr];
        const T wr = (T)w;
        wt[tid] = (double)wr;
        if (blockIdx.y == 0) u[base + tid] = wr;
        if (MODE == kNorm) nrm = fma((double)wr, (double)wr, nrm);
      }
    }
    if (MODE == kNorm) continue;
    __syncthreads();
    for (int ib = i0 + 4 * wid; ib < i1; ib += 32) {
      double a[4] = {0.0, 0.0, 0.0, 0.0};
      for (int rr = lane; rr < nr; rr += 32) {
        const double w = wt[rr];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          a[k] = fma((double)V[(int64_t)min(ib + k, i1 - 1) * n + base + rr], w, a[k]);
      }
      // four sums over the warp in six additions: lanes >= 16 keep a[2..3],
      // then every other eight lanes one of the two
      const bool h16 = lane & 16, h8 = lane & 8;
      const double s0 = __shfl_xor_sync(~0u, h16 ? a[0] : a[2], 16);
      const double s1 = __shfl_xor_sync(~0u, h16 ? a[1] : a[3], 16);
      const double b0 = (h16 ? a[2] : a[0]) + s0, b1 = (h16 ? a[3] : a[1]) + s1;
      double c = (h8 ? b1 : b0) + __shfl_xor_sync(~0u, h8 ? b0 : b1, 8);
      for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(~0u, c, o);
      const int i = ib + (h16 ? 2 : 0) + (h8 ? 1 : 0);
      if ((lane & 7) == 0 && i < i1) dacc[i - i0] += c;
    }
  }
  __syncthreads();
  const int nb = gridDim.x;
  if (MODE == kNorm) {
    for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(~0u, nrm, o);
    if (lane == 0) red[wid] = nrm;
    __syncthreads();
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < 8; ++w) s += red[w];
      g.part[blockIdx.x] = s;
    }
  } else {
    for (int i = i0 + tid; i < i1; i += 256) g.part[(int64_t)i * GM_MAXB + blockIdx.x] = dacc[i - i0];
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    unsigned* c = &ctl->cnt[MODE][blockIdx.y];
    s_last = atomicAdd(c, 1u) == (unsigned)nb - 1u;
    if (s_last) *c = 0u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (MODE != kNorm) {               // eight lanes per dot product
    for (int ib = i0; ib < i1; ib += 32) {
      const int i = ib + (tid >> 3);
      double s = 0.0;
      if (i < i1)
        for (int b = tid & 7; b < nb; b += 8) s += __ldcg(g.part + (int64_t)i * GM_MAXB + b);
      for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(~0u, s, o);
      if (i < i1 && (tid & 7) == 0) {
        if (MODE == kDot1) g.h1[i] = s * sj * g.s[i];
        else g.h2[i] = s * g.s[i];
      }
    }
    return;
  }
  // the column, its norm and the residual
  double ph = 0.0, s = 0.0;
  for (int i = tid; i < nj; i += 256) {
    const double c = g.h1[i] + g.h2[i];
    col[1 + i] = c;
    ph = fma(g.phi[i], c, ph);
  }
  for (int b = tid; b < nb; b += 256) s += __ldcg(g.part + b);
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(~0u, s, o);
    ph += __shfl_xor_sync(~0u, ph, o);
  }
  __syncthreads();
  if (lane == 0) {
    red[wid] = s;
    red[8 + wid] = ph;
  }
  __syncthreads();
  if (tid == 0) {
    s = ph = 0.0;
    for (int w = 0; w < 8; ++w) {
      s += red[w];
      ph += red[8 + w];
    }
    const double nr = sqrt(s);
    col[1 + nj] = nr;
    g.s[nj] = 1.0 / nr;
    const double f = -ph / nr;
    g.phi[nj] = f;
    const double sum = fma(f, f, ctl->sumphi2);
    ctl->sumphi2 = sum;
    const double res = ctl->beta / sqrt(sum);
    const bool done = !(res > ctl->tol) || !(s > 0.0);
    if (done) ctl->done = 1;
    col[0] = done ? 1.0 : 0.0;
  }
}

// rows per block and tile of the Arnoldi kernels
static inline int gm_tile(int64_t n) { return n <= 64 * GM_MAXB ? 64 : 256; }
static inline int gm_rows(int64_t n) {
  const int tr = gm_tile(n);
  const int64_t r = (n + GM_MAXB - 1) / GM_MAXB;
  return (int)((r + tr - 1) / tr * tr);
}

template <typename T>
static cudaError_t gm_step(const T* q, T* V, int64_t n, int j, const GmVecs& g, GmCtl* ctl,
                           double* col, cudaStream_t st) {
  const int rows = gm_rows(n), tr = gm_tile(n);
  const int nb = (int)((n + rows - 1) / rows);
  const int ny = std::max(1, std::min({GM_SLICES, GM_MAXB / nb, (j + 8) / 8}));
  const size_t sm = (size_t)2 * (j + 1) * 8;
  cudaError_t e;
  if ((e = launch_maybe_pdl(k_gm_step<T, kDot1>, dim3(nb, ny), dim3(256), sm, st, true, q, V, n, j,
                            rows, tr, g, ctl, col)) != cudaSuccess ||
      (e = launch_maybe_pdl(k_gm_step<T, kDot2>, dim3(nb, ny), dim3(256), sm, st, true, q, V, n, j,
                            rows, tr, g, ctl, col)) != cudaSuccess)
    return e;
  return launch_maybe_pdl(k_gm_step<T, kNorm>, dim3(nb, 1), dim3(256), sm, st, true, q, V, n, j,
                          rows, tr, g, ctl, col);
}

// page-locked ring of Hessenberg columns (each: last step of the cycle or
// not, then the column) and the events of the steps
struct GmHost : HostRing {
  using HostRing::HostRing;
  int m = 0;
  double* slot(int step) { return (double*)mem + (size_t)(step % GM_RING) * (m + 3); }
  cudaError_t init(int restart) {
    m = restart;
    return HostRing::init((size_t)GM_RING * (m + 3) * 8, GM_RING);
  }
};

// ---- GMRES(m) --------------------------------------------------------------

// Givens-based least squares of the Arnoldi relation, host side
struct Hess {
  int m;
  std::vector<double> H, cs, sn, g;
  explicit Hess(int m_) : m(m_), H((m_ + 1) * m_, 0.0), cs(m_), sn(m_), g(m_ + 1) {}
  double& h(int i, int j) { return H[j * (m + 1) + i]; }
  // apply the previous rotations to column j, create rotation j; return |g[j+1]|
  double add_column(int j, const double* col) {
    for (int i = 0; i <= j + 1; ++i) h(i, j) = col[i];
    for (int i = 0; i < j; ++i) {
      const double a = cs[i] * h(i, j) + sn[i] * h(i + 1, j);
      const double bb = -sn[i] * h(i, j) + cs[i] * h(i + 1, j);
      h(i, j) = a;
      h(i + 1, j) = bb;
    }
    const double a = h(j, j), bb = h(j + 1, j);
    const double rr = std::hypot(a, bb);
    cs[j] = (rr == 0.0) ? 1.0 : a / rr;
    sn[j] = (rr == 0.0) ? 0.0 : bb / rr;
    h(j, j) = rr;
    h(j + 1, j) = 0.0;
    g[j + 1] = -sn[j] * g[j];
    g[j] = cs[j] * g[j];
    return std::fabs(g[j + 1]);
  }
  void solve(int k, double* y) {   // back substitution on the k x k triangle
    for (int i = k - 1; i >= 0; --i) {
      double s = g[i];
      for (int j = i + 1; j < k; ++j) s -= h(i, j) * y[j];
      y[i] = s / h(i, i);
    }
  }
};

template <typename T, typename TX>
SolveStatus solve_gmres(const ApplyFn<T>& apply, int64_t n, const TX* b, TX* x, double rtol,
                        int maxit, int restart, cudaStream_t st, Workspace& ws, SolveInfo* info,
                        const ApplyFn<TX>* apply_x) {
  static_assert(std::is_same<T, TX>::value, "rx is also the Arnoldi step's A U_j");
  // apply_x: operator in the precision of x/b for the outer residual (T == TX: same as apply)
  const int m = restart;
  // one allocation: the basis, A U_j / the outer residual, scalars, partials
  GmVecs g;
  const auto up = [](size_t v) { return (v + 255) / 256 * 256; };
  const size_t bV = up((size_t)(m + 1) * n * sizeof(T)), br = up((size_t)n * sizeof(TX)),
               bs = up((size_t)5 * (m + 4) * 8), bp = up((size_t)(m + 1) * GM_MAXB * 8),
               bq = up((size_t)RED_BLOCKS * 8);
  char* base;
  CK(ws.alloc((void**)&base, bV + br + bs + bp + bq + sizeof(GmCtl)));
  T* V = (T*)base;
  TX* rx = (TX*)(base + bV);
  double* dsc = (double*)(base + bV + br);
  g.s = dsc + (m + 4);
  g.h1 = g.s + (m + 4);
  g.h2 = g.h1 + (m + 4);
  g.phi = g.h2 + (m + 4);
  g.part = (double*)(base + bV + br + bs);
  double* part = (double*)(base + bV + br + bs + bp);
  GmCtl* ctl = (GmCtl*)(base + bV + br + bs + bp + bq);
  GmHost gh(st);
  CK(gh.init(m));
  std::vector<double> y(m + 1), scale(m + 2);
  int total = 0, cycles = 0;
  double relres = INFINITY, bnorm = 0.0;
  {
    CK(multi_dot<TX>(b, 0, b, n, 1, part, dsc, st));
    CK(cudaMemcpyAsync(&bnorm, dsc, 8, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    bnorm = std::sqrt(bnorm);
  }
  if (bnorm == 0.0) {
    CK(cudaMemsetAsync(x, 0, n * sizeof(TX), st));
    info->iters = 0;
    info->relres = 0.0;
    return {SBM_OK, cudaSuccess};
  }
  const ApplyFn<TX>& ax = *apply_x;
  int status = SBM_ERR_NOT_CONVERGED;
  while (total < maxit) {
    // r = b - A x, v0 = r / |r|
    CK(ax(x, rx, st));
    k_residual<TX><<<vec_grid(n), 256, 0, st>>>(b, rx, n);
    CK(multi_dot<TX>(rx, 0, rx, n, 1, part, dsc, st));
    double rr;
    CK(cudaMemcpyAsync(&rr, dsc, 8, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    relres = std::sqrt(rr) / bnorm;
    if (relres <= rtol) { status = SBM_OK; break; }
    if (!std::isfinite(relres)) break;
    k_convert_scaled<T, TX><<<vec_grid(n), 256, 0, st>>>(V, rx, 1.0 / std::sqrt(rr), n);
    k_gm_begin<<<1, 1, 0, st>>>(ctl, g, std::sqrt(rr), 0.5 * rtol * bnorm);
    CK(cudaGetLastError());
    Hess H(m);
    H.g[0] = std::sqrt(rr);
    scale[0] = 1.0;
    const int lim = std::min(m, maxit - total);
    int k = 0, enq = 0;
    while (k < lim) {
      for (; enq < lim && enq < k + GM_AHEAD; ++enq) {
        CK(apply(V + (size_t)enq * n, rx, st));
        CK(gm_step<T>(rx, V, n, enq, g, ctl, gh.slot(enq), st));
        CK(cudaEventRecord(gh.ev[enq % GM_RING], st));
      }
      CK(cudaEventSynchronize(gh.ev[k % GM_RING]));
      const double* slot = gh.slot(k);
      const bool last = slot[0] != 0.0;   // the device ended the cycle with this step
      const double* col = slot + 1;
      const double hn = col[k + 1];
      scale[k + 1] = 1.0 / hn;
      const double res = H.add_column(k, col);
      ++total;
      ++k;
      if (last || res / bnorm <= rtol * 0.5 || !(hn > 0.0) || !std::isfinite(res)) break;
    }
    H.solve(k, y.data());
    for (int i = 0; i < k; ++i) y[i] *= scale[i];
    CK(cudaMemcpyAsync(dsc, y.data(), k * 8, cudaMemcpyHostToDevice, st));
    k_update_x<TX, T><<<vec_grid(n), 256, 0, st>>>(x, V, n, dsc, k, 1.0, n);
    CK(cudaGetLastError());
    ++cycles;
  }
  if (status != SBM_OK) {
    // final true residual
    CK(ax(x, rx, st));
    k_residual<TX><<<vec_grid(n), 256, 0, st>>>(b, rx, n);
    CK(multi_dot<TX>(rx, 0, rx, n, 1, part, dsc, st));
    double rr;
    CK(cudaMemcpyAsync(&rr, dsc, 8, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    relres = std::sqrt(rr) / bnorm;
    if (relres <= rtol) status = SBM_OK;
  }
  info->iters = total;
  info->relres = relres;
  info->restarts = cycles;
  return {status, cudaSuccess};
}

template SolveStatus solve_gmres<double, double>(const ApplyFn<double>&, int64_t, const double*,
                                                 double*, double, int, int, cudaStream_t,
                                                 Workspace&, SolveInfo*, const ApplyFn<double>*);
template SolveStatus solve_gmres<float, float>(const ApplyFn<float>&, int64_t, const float*,
                                               float*, double, int, int, cudaStream_t, Workspace&,
                                               SolveInfo*, const ApplyFn<float>*);

// ---- BiCGStab ----------------------------------------------------------------
//
// van der Vorst's stabilised bi-conjugate gradients, two operator
// applications and three reductions per iteration.  Vectors are in T
// (FP64 or FP32); every scalar is FP64 and stays on the device, so a chunk of
// BI_CHUNK iterations is one CUDA-graph launch with no host round trip.  A
// breakdown (rho or (r^, v) vanishing, omega = 0) or a recursive residual that
// disagrees with the true one restarts from the current iterate with a fresh
// shadow residual r^ = r.

constexpr int BI_CHUNK = 8;
constexpr int kIrFinishMaxit = 20000;   // FP64 BiCGStab finish of the refinement, at most

struct BiState {
  double rho, alpha, omega, beta, rr, bb, tol2;
  int done;     // 0 running, 1 converged (recursive residual), 2 breakdown/divergence, 3 maxit
  int iters;
  int maxit;
};

// r = b - q (q = A x; q == nullptr for x = 0); r^ = r; p = r; partials r.r, b.b
template <typename T>
__global__ void k_bi_init(const T* __restrict__ b, const T* __restrict__ q, T* __restrict__ r,
                          T* __restrict__ rh, T* __restrict__ p, int64_t n,
                          double* __restrict__ part) {
  __shared__ double sh[RED_THREADS / 16];
  double srr = 0.0, sbb = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const T ri = q ? (T)(b[i] - q[i]) : b[i];
    r[i] = ri;
    rh[i] = ri;
    p[i] = ri;
    srr = fma((double)ri, (double)ri, srr);
    sbb = fma((double)b[i], (double)b[i], sbb);
  }
  block_sum2(srr, sbb, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = srr;
    part[RED_BLOCKS + blockIdx.x] = sbb;
  }
}

__global__ void k_bi_init_fin(const double* __restrict__ part, int nb, BiState* st) {
  __shared__ double sh[RED_THREADS / 16];
  double v[2];
  part_sum2(part, nb, sh, v);
  if (threadIdx.x == 0) {
    st->rr = v[0];
    st->bb = v[1];
    st->rho = v[0];              // (r^, r) with r^ = r
    st->alpha = st->omega = 1.0;
    st->beta = 0.0;
    st->done = (v[0] <= st->tol2 * v[1]) ? 1 : 0;
    if (!isfinite(v[0])) st->done = 2;
    if (st->maxit <= 0 && !st->done) st->done = 3;
  }
}

// alpha = rho / (r^, v)
__global__ void k_bi_alpha(const double* __restrict__ part, int nb, BiState* st) {
  pdl_wait_all();
  __shared__ double sh[RED_THREADS / 16];
  if (st->done) return;
  const double s = part_sum(part, nb, sh);
  if (threadIdx.x == 0) {
    if (!(s != 0.0) || !isfinite(s)) st->done = 2;
    else st->alpha = st->rho / s;
  }
}

// s = r - alpha v
template <typename T>
__global__ void k_bi_s(const T* __restrict__ r, const T* __restrict__ v, T* __restrict__ s,
                       int64_t n, const BiState* st) {
  pdl_wait_all();
  if (st->done) return;
  const double al = st->alpha;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    s[i] = (T)fma(-al, (double)v[i], (double)r[i]);
}

// partials of (t, s) and (t, t)
template <typename T>
__global__ void k_bi_dot2(const T* __restrict__ t, const T* __restrict__ s, int64_t n,
                          const BiState* st, double* __restrict__ part) {
  pdl_wait_all();
  __shared__ double sh[RED_THREADS / 16];
  if (st->done) return;
  double sts = 0.0, stt = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double ti = (double)t[i];
    sts = fma(ti, (double)s[i], sts);
    stt = fma(ti, ti, stt);
  }
  block_sum2(sts, stt, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = sts;
    part[RED_BLOCKS + blockIdx.x] = stt;
  }
}

// omega = (t, s) / (t, t)  (0 when t = 0: the update then keeps r = s)
__global__ void k_bi_omega(const double* __restrict__ part, int nb, BiState* st) {
  pdl_wait_all();
  __shared__ double sh[RED_THREADS / 16];
  if (st->done) return;
  double v[2];
  part_sum2(part, nb, sh, v);
  if (threadIdx.x == 0) {
    st->omega = (v[1] > 0.0) ? v[0] / v[1] : 0.0;
    if (!isfinite(st->omega)) st->done = 2;
  }
}

// x += alpha p + omega s; r = s - omega t; partials of (r^, r), (r, r)
template <typename T>
__global__ void k_bi_update(T* __restrict__ x, T* __restrict__ r, const T* __restrict__ p,
                            const T* __restrict__ s, const T* __restrict__ t,
                            const T* __restrict__ rh, int64_t n, const BiState* st,
                            double* __restrict__ part) {
  pdl_wait_all();
  __shared__ double sh[RED_THREADS / 16];
  if (st->done) return;
  const double al = st->alpha, om = st->omega;
  double srh = 0.0, srr = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double si = (double)s[i];
    x[i] = (T)fma(om, si, fma(al, (double)p[i], (double)x[i]));
    const T ri = (T)fma(-om, (double)t[i], si);
    r[i] = ri;
    srh = fma((double)rh[i], (double)ri, srh);
    srr = fma((double)ri, (double)ri, srr);
  }
  block_sum2(srh, srr, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = srh;
    part[RED_BLOCKS + blockIdx.x] = srr;
  }
}

// rho' = (r^, r); convergence / breakdown tests; beta = (rho'/rho)(alpha/omega)
__global__ void k_bi_beta(const double* __restrict__ part, int nb, BiState* st) {
  pdl_wait_all();
  __shared__ double sh[RED_THREADS / 16];
  if (st->done) return;
  double v[2];
  part_sum2(part, nb, sh, v);
  if (threadIdx.x == 0) {
    st->iters += 1;
    st->rr = v[1];
    if (v[1] <= st->tol2 * st->bb) st->done = 1;
    else if (!isfinite(v[1]) || v[1] > 1e24 * st->bb) st->done = 2;
    else if (!(v[0] != 0.0) || !(st->omega != 0.0)) st->done = 2;
    else if (st->iters >= st->maxit) st->done = 3;
    if (!st->done) {
      st->beta = (v[0] / st->rho) * (st->alpha / st->omega);
      st->rho = v[0];
    }
  }
}

// reliable update: r = b - q (q = A x with the accurate operator); partials
// of (r^, r), (r, r)
template <typename T>
__global__ void k_bi_replace(const T* __restrict__ b, const T* __restrict__ q,
                             T* __restrict__ r, const T* __restrict__ rh, int64_t n,
                             double* __restrict__ part) {
  __shared__ double sh[RED_THREADS / 16];
  double srh = 0.0, srr = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const T ri = (T)((double)b[i] - (double)q[i]);
    r[i] = ri;
    srh = fma((double)rh[i], (double)ri, srh);
    srr = fma((double)ri, (double)ri, srr);
  }
  block_sum2(srh, srr, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = srh;
    part[RED_BLOCKS + blockIdx.x] = srr;
  }
}

// rho = (r^, r) and rr = (r, r) of the replaced residual; convergence test
__global__ void k_bi_replace_fin(const double* __restrict__ part, int nb, BiState* st) {
  __shared__ double sh[RED_THREADS / 16];
  if (st->done) return;
  double v[2];
  part_sum2(part, nb, sh, v);
  if (threadIdx.x == 0) {
    st->rr = v[1];
    st->rho = v[0];
    if (v[1] <= st->tol2 * st->bb) st->done = 1;
    else if (!isfinite(v[1]) || !(v[0] != 0.0)) st->done = 2;
  }
}

// p = r + beta (p - omega v)
template <typename T>
__global__ void k_bi_p(T* __restrict__ p, const T* __restrict__ r, const T* __restrict__ v,
                       int64_t n, const BiState* st) {
  pdl_wait_all();
  if (st->done) return;
  const double be = st->beta, om = st->omega;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    p[i] = (T)fma(be, fma(-om, (double)v[i], (double)p[i]), (double)r[i]);
}

template <typename T>
cudaError_t Bicgstab<T>::setup(const ApplyFn<T>& apply_, int64_t n_, const T* b_, T* x_,
                               Workspace& ws) {
  apply = apply_;
  n = n_;
  b = b_;
  x = x_;
  cudaError_t e;
  T** vecs[7] = {&r, &rh, &p, &v, &s, &t, &xb};
  for (T** pv : vecs)
    if ((e = ws.alloc((void**)pv, (size_t)n * sizeof(T))) != cudaSuccess) return e;
  if ((e = ws.alloc((void**)&part, 2 * RED_BLOCKS * 8)) != cudaSuccess) return e;
  if ((e = ws.alloc(&dstate, sizeof(BiState))) != cudaSuccess) return e;
  if ((e = cudaMallocHost(&hstate, sizeof(BiState))) != cudaSuccess) return e;
  if ((e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking)) != cudaSuccess) return e;
  BiState* dst = (BiState*)dstate;
  const int nb = red_blocks(n);
  cudaGraph_t graph;
  if ((e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal)) != cudaSuccess)
    return e;
  cudaError_t ae = cudaSuccess;
  for (int it = 0; it < BI_CHUNK && ae == cudaSuccess; ++it) {
    ae = apply(p, v, cap);
    if (ae != cudaSuccess) break;
    const T* crh = rh;
    const T* cv = v;
    const T* cr = r;
    const T* cs = s;
    const T* ct = t;
    const T* cp = p;
    if ((ae = launch_maybe_pdl(k_multi_dot<T>, dim3(nb, 1), dim3(RED_THREADS), 0, cap,
                               true, crh, (int64_t)0, cv, n, part)) != cudaSuccess ||
        (ae = launch_maybe_pdl(k_bi_alpha, dim3(1), dim3(RED_THREADS), 0, cap, true,
                               (const double*)part, nb, dst)) != cudaSuccess ||
        (ae = launch_maybe_pdl(k_bi_s<T>, dim3(vec_grid(n)), dim3(256), 0, cap, true, cr, cv, s,
                               n, (const BiState*)dst)) != cudaSuccess)
      break;
    ae = apply(s, t, cap);
    if (ae != cudaSuccess) break;
    if ((ae = launch_maybe_pdl(k_bi_dot2<T>, dim3(nb), dim3(RED_THREADS), 0, cap, true,
                               ct, cs, n, (const BiState*)dst, part)) != cudaSuccess ||
        (ae = launch_maybe_pdl(k_bi_omega, dim3(1), dim3(RED_THREADS), 0, cap, true,
                               (const double*)part, nb, dst)) != cudaSuccess ||
        (ae = launch_maybe_pdl(k_bi_update<T>, dim3(nb), dim3(RED_THREADS), 0, cap,
                               true, x, r, cp, cs, ct, crh, n, (const BiState*)dst, part)) !=
            cudaSuccess ||
        (ae = launch_maybe_pdl(k_bi_beta, dim3(1), dim3(RED_THREADS), 0, cap, true,
                               (const double*)part, nb, dst)) != cudaSuccess ||
        (ae = launch_maybe_pdl(k_bi_p<T>, dim3(vec_grid(n)), dim3(256), 0, cap, true, p, cr, cv,
                               n, (const BiState*)dst)) != cudaSuccess)
      break;
  }
  e = cudaStreamEndCapture(cap, &graph);
  if (ae != cudaSuccess) {
    if (e == cudaSuccess) cudaGraphDestroy(graph);
    return ae;
  }
  if (e != cudaSuccess) return e;
  e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  return e;
}

template <typename T>
void Bicgstab<T>::destroy() {
  if (exec) cudaGraphExecDestroy(exec);
  exec = nullptr;
  if (hstate) cudaFreeHost(hstate);
  hstate = nullptr;
  if (cap) cudaStreamDestroy(cap);
  cap = nullptr;
}

template <typename T>
SolveStatus Bicgstab<T>::solve(bool x_zero, double rtol, int maxit, cudaStream_t st,
                               SolveInfo* info) {
  BiState* dst = (BiState*)dstate;
  BiState* hs = (BiState*)hstate;
  const int nb = red_blocks(n);
  int total = 0, restarts = 0, status = SBM_NOT_DONE;
  double relres = INFINITY, best = INFINITY;
  bool zero = x_zero;
  const bool reliable = (bool)apply_hi;
  const ApplyFn<T>& ap_true = reliable ? apply_hi : apply;   // first and final residuals
  while (true) {
    BiState init{};
    init.tol2 = rtol * rtol;
    init.maxit = maxit - total;
    CK(cudaMemcpyAsync(dst, &init, sizeof(BiState), cudaMemcpyHostToDevice, st));
    if (!zero) CK(ap_true(x, v, st));
    k_bi_init<T><<<nb, RED_THREADS, 0, st>>>(b, zero ? nullptr : v, r, rh, p, n, part);
    k_bi_init_fin<<<1, RED_THREADS, 0, st>>>(part, nb, dst);
    CK(cudaGetLastError());
    zero = false;
    int done = 0;
    double rr_ref = -1.0;        // recursive residual at the last reliable update
    double rr_true = INFINITY;   // true residual at the last reliable update
    bool replaced = false, stalled = false;
    while (true) {
      CK(cudaMemcpyAsync(hs, dst, sizeof(BiState), cudaMemcpyDeviceToHost, st));
      CK(cudaStreamSynchronize(st));
      done = hs->done;
      if (rr_ref < 0.0) {
        // a true residual (the first one, or just replaced)
        rr_ref = hs->rr;
        // one that no longer halves between updates: the reduced-precision
        // iteration has stalled (the caller finishes)
        if (replaced) stalled = !done && hs->rr > 0.25 * rr_true;
        rr_true = hs->rr;
        replaced = false;
        // with reliable updates: keep the iterate of least true residual
        if (reliable && std::isfinite(hs->rr) && hs->rr < best) {
          best = hs->rr;
          CK(cudaMemcpyAsync(xb, x, (size_t)n * sizeof(T), cudaMemcpyDeviceToDevice, st));
        }
      }
      if (stalled) {
        done = 3;
        break;
      }
      // reliable update: the true residual replaces the recursive one
      if (reliable && !done && std::isfinite(hs->rr) &&
          hs->rr < reliable_factor * reliable_factor * rr_ref) {
        CK(apply_hi(x, t, st));
        k_bi_replace<T><<<nb, RED_THREADS, 0, st>>>(b, t, r, rh, n, part);
        k_bi_replace_fin<<<1, RED_THREADS, 0, st>>>(part, nb, dst);
        CK(cudaGetLastError());
        ++replacements;
        rr_ref = -1.0;           // re-read: the reference is the replaced residual
        replaced = true;
        continue;
      }
      // keep the iterate of least (recursive) residual seen at a chunk end
      if (!reliable && std::isfinite(hs->rr) && hs->rr < best) {
        best = hs->rr;
        CK(cudaMemcpyAsync(xb, x, (size_t)n * sizeof(T), cudaMemcpyDeviceToDevice, st));
      }
      if (done) break;
      CK(cudaGraphLaunch(exec, st));
    }
    total += hs->iters;
    // after a breakdown, divergence, a stall or the iteration cap, continue
    // from the best iterate rather than the last one (reliable updates: the
    // best true residual; otherwise the best recursive one)
    if (done != 1 && (reliable || !(hs->rr <= best)))
      CK(cudaMemcpyAsync(x, xb, (size_t)n * sizeof(T), cudaMemcpyDeviceToDevice, st));
    if (hs->bb == 0.0) {
      relres = 0.0;
      status = SBM_OK;
      break;
    }
    // true residual of the current iterate
    CK(ap_true(x, v, st));
    k_residual<T><<<vec_grid(n), 256, 0, st>>>(b, v, n);
    CK(multi_dot<T>(v, 0, v, n, 1, part, part + RED_BLOCKS, st));
    double rr;
    CK(cudaMemcpyAsync(&rr, part + RED_BLOCKS, 8, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    relres = std::sqrt(rr / hs->bb);
    if (relres <= rtol) { status = SBM_OK; break; }
    if (done == 3 || total >= maxit || ++restarts > 50 || !std::isfinite(relres)) {
      status = SBM_ERR_NOT_CONVERGED;
      break;
    }
  }
  info->iters = total;
  info->relres = relres;
  info->restarts = restarts;
  return {status, cudaSuccess};
}

template struct Bicgstab<double>;
template struct Bicgstab<float>;

// ---- BiCGStab on the FP32 apply with FP64 reliable updates -------------------

SolveStatus solve_bicgstab_reliable(const ApplyFn<double>& apply64,
                                    const ApplyFn<float>& apply32, int64_t n, const double* b,
                                    double* x, double rtol, int maxit, cudaStream_t st,
                                    Workspace& ws, SolveInfo* info, int* replacements) {
  float *xa = nullptr, *ya = nullptr;
  CK(ws.alloc((void**)&xa, n * 4));
  CK(ws.alloc((void**)&ya, n * 4));
  ApplyFn<double> apply_mixed = [&](const double* xin, double* yout, cudaStream_t s) {
    k_convert_scaled<float, double><<<vec_grid(n), 256, 0, s>>>(xa, xin, 1.0, n);
    cudaError_t e = apply32(xa, ya, s);
    if (e != cudaSuccess) return e;
    k_convert_scaled<double, float><<<vec_grid(n), 256, 0, s>>>(yout, ya, 1.0, n);
    return cudaGetLastError();
  };
  Bicgstab<double> bi;
  bi.apply_hi = apply64;
  cudaError_t e = bi.setup(apply_mixed, n, b, x, ws);
  SolveStatus s{SBM_ERR_CUDA, e};
  if (e == cudaSuccess) s = bi.solve(false, rtol, maxit, st, info);
  if (replacements) *replacements = bi.replacements;
  bi.destroy();
  // FP64 finish when the reduced-precision iteration stalled (the FP32
  // operator's rounding, about kappa * 6e-8 of |b|, limits its corrections)
  if (s.status == SBM_ERR_NOT_CONVERGED && std::isfinite(info->relres) &&
      info->iters < maxit) {
    Bicgstab<double> bf;
    SolveInfo fi{};
    e = bf.setup(apply64, n, b, x, ws);
    SolveStatus f{SBM_ERR_CUDA, e};
    if (e == cudaSuccess) f = bf.solve(false, rtol, maxit - info->iters, st, &fi);
    bf.destroy();
    if (f.status == SBM_ERR_CUDA) return f;
    info->iters += fi.iters;
    info->relres = fi.relres;
    info->restarts += 1;
    s = f;
  }
  return s;
}

// ---- FP64 iterative refinement around an FP32 inner solve --------------------

SolveStatus solve_ir(const ApplyFn<double>& apply64, const ApplyFn<float>& apply32, int64_t n,
                     const double* b, double* x, double rtol, int maxit, int restart,
                     double inner_rtol, int inner_maxit, int inner, cudaStream_t st,
                     Workspace& ws, SolveInfo* info) {
  double *r, *part, *dsc;
  float *r32, *c32;
  CK(ws.alloc((void**)&r, n * 8));
  CK(ws.alloc((void**)&r32, n * 4));
  CK(ws.alloc((void**)&c32, n * 4));
  CK(ws.alloc((void**)&part, RED_BLOCKS * 8));
  CK(ws.alloc((void**)&dsc, 8));
  double bb;
  CK(multi_dot<double>(b, 0, b, n, 1, part, dsc, st));
  CK(cudaMemcpyAsync(&bb, dsc, 8, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  const double bnorm = std::sqrt(bb);
  int outer = 0, inner_total = 0;
  double relres = INFINITY;
  int status = SBM_ERR_NOT_CONVERGED;
  Workspace inner_ws;
  Bicgstab<float> bi;
  if (inner == SBM_INNER_BICGSTAB) {
    cudaError_t e = bi.setup(apply32, n, r32, c32, ws);
    if (e != cudaSuccess) {
      bi.destroy();
      return {SBM_ERR_CUDA, e};
    }
  }
  // mixed inner solver: FP64 vectors and scalars, the FP32 apply (converted
  // in and out around every application)
  Bicgstab<double> bm;
  double *r64 = nullptr, *c64 = nullptr;
  float *xa = nullptr, *ya = nullptr;
  ApplyFn<double> apply_mixed = [&](const double* xin, double* yout, cudaStream_t s) {
    k_convert_scaled<float, double><<<vec_grid(n), 256, 0, s>>>(xa, xin, 1.0, n);
    cudaError_t e = apply32(xa, ya, s);
    if (e != cudaSuccess) return e;
    k_convert_scaled<double, float><<<vec_grid(n), 256, 0, s>>>(yout, ya, 1.0, n);
    return cudaGetLastError();
  };
  if (inner == SBM_INNER_BICGSTAB_MIXED) {
    cudaError_t e;
    if ((e = ws.alloc((void**)&r64, n * 8)) != cudaSuccess ||
        (e = ws.alloc((void**)&c64, n * 8)) != cudaSuccess ||
        (e = ws.alloc((void**)&xa, n * 4)) != cudaSuccess ||
        (e = ws.alloc((void**)&ya, n * 4)) != cudaSuccess ||
        (e = bm.setup(apply_mixed, n, r64, c64, ws)) != cudaSuccess) {
      bm.destroy();
      return {SBM_ERR_CUDA, e};
    }
  }
  while (outer <= maxit) {
    CK(apply64(x, r, st));
    k_residual<double><<<vec_grid(n), 256, 0, st>>>(b, r, n);
    CK(multi_dot<double>(r, 0, r, n, 1, part, dsc, st));
    double rr;
    CK(cudaMemcpyAsync(&rr, dsc, 8, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    relres = bnorm > 0 ? std::sqrt(rr) / bnorm : 0.0;
    if (relres <= rtol) { status = SBM_OK; break; }
    if (!std::isfinite(relres) || outer == maxit) break;
    // inner: A32 c = r / |r| to inner_rtol, c starts at 0
    const double rn = std::sqrt(rr);
    SolveInfo ii{};
    SolveStatus s;
    if (inner == SBM_INNER_BICGSTAB_MIXED) {
      k_convert_scaled<double, double><<<vec_grid(n), 256, 0, st>>>(r64, r, 1.0 / rn, n);
      CK(cudaMemsetAsync(c64, 0, n * 8, st));
      s = bm.solve(true, inner_rtol, inner_maxit, st, &ii);
      if (s.status == SBM_ERR_CUDA) {
        bm.destroy();
        bi.destroy();
        info->iters = inner_total;
        return s;
      }
      inner_total += ii.iters;
      if (s.status != SBM_OK && !(ii.relres < 1.0)) break;
      k_axpy_d<<<vec_grid(n), 256, 0, st>>>(x, c64, rn, n);       // x += |r| c
      CK(cudaGetLastError());
      ++outer;
      continue;
    }
    k_convert_scaled<float, double><<<vec_grid(n), 256, 0, st>>>(r32, r, 1.0 / rn, n);
    CK(cudaMemsetAsync(c32, 0, n * 4, st));
    if (inner == SBM_INNER_BICGSTAB) {
      s = bi.solve(true, inner_rtol, inner_maxit, st, &ii);
    } else {
      s = solve_gmres<float, float>(apply32, n, r32, c32, inner_rtol, inner_maxit, restart, st,
                                    inner_ws, &ii, &apply32);
      inner_ws.release();
    }
    if (s.status == SBM_ERR_CUDA) {
      bi.destroy();
      info->iters = inner_total;
      return s;
    }
    inner_total += ii.iters;
    // an inner solve that made no progress would only spoil x
    if (s.status != SBM_OK && !(ii.relres < 1.0)) break;
    // x += |r| c
    k_add_scaled<<<vec_grid(n), 256, 0, st>>>(x, c32, rn, n);
    CK(cudaGetLastError());
    ++outer;
  }
  bi.destroy();
  bm.destroy();
  // FP64 finish: when the reduced-precision corrections stall (an ill-conditioned
  // operator whose FP32 rounding, about kappa * 6e-8 of |b|, floors what an
  // inner solve can reach), BiCGStab on the FP64 operator continues from x
  if (status != SBM_OK && std::isfinite(relres) && bnorm > 0) {
    Bicgstab<double> bf;
    cudaError_t e = bf.setup(apply64, n, b, x, ws);
    SolveInfo fi{};
    SolveStatus s{SBM_ERR_CUDA, e};
    const int cap = (int)std::min<int64_t>(kIrFinishMaxit, (int64_t)maxit * inner_maxit);
    if (e == cudaSuccess) s = bf.solve(false, rtol, cap, st, &fi);
    bf.destroy();
    if (s.status == SBM_ERR_CUDA) {
      info->iters = inner_total;
      return s;
    }
    inner_total += fi.iters;
    relres = fi.relres;
    status = s.status;
    ++outer;
  }
  info->iters = inner_total;
  info->relres = relres;
  info->restarts = outer;
  return {status, cudaSuccess};
}

}  // namespace sbm
