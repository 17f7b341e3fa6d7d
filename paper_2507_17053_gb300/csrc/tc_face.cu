// Surrogate-boundary faces with the shifted point evaluation on the 5th-
// generation tensor cores (tcgen05), for the FP32 apply in TF32 or BF16 mode.
//
// The O((p+1)^(2d-1)) step of Algorithm 3 is, per face, the contraction
//   T[q][l] = sum_{j0} phi_{j0}(xi_{q,0}) u[j0][l]       (q: face point, l: x-line)
// followed by per-point weighted sums over the remaining axes.  The first
// contraction is a dense (points x n) . (n x lines) product: one
//   tcgen05.mma.cta_group::1.kind::{tf32, f16}  M = 128, N = 128, K = 8 | 16
// for a group of 2 to 32 faces, their points stacked in the rows and their
// x-lines in the columns (the products between different faces are computed
// and not read: the tensor cores are idle otherwise, and the kernel's time is
// the latency of a group's steps).  Both operands lie in shared memory in the
// canonical K-major, no-swizzle core-matrix layout (8 rows x 16 bytes per core
// matrix; core matrices adjacent in K 128 bytes apart, 8-row groups 256 bytes
// apart), the FP32 accumulator in tensor memory, read back with tcgen05.ld by
// the warps that own its rows.  Everything else (normal-derivative trace, the
// remaining two contractions, the integrands, the transposed interpolation)
// runs on the CUDA cores in FP32, as in face_body.cuh, and the output has the
// same format.
//
// Measured on GB300, one face per block and group -> this (four faces and more
// in flight per block, the next group's loads behind the current one's work):
// 19 704 faces (torus of 96^3) at p = 1 43 -> 8.5 us, 8 776 (64^3) at p = 3 27
// -> 11.8, 4 912 (48^3) at p = 6 35 -> 26.7 us; FP32 apply with TF32 faces of
// the Q6 ellipsoid of 48^3 cells 83.8 -> 60.3 us, with BF16 faces of the p = 3
// DG torus 41.0 -> 20.5 us (the cell kernel its dependent in both).
//
// Waits on the MMA's mbarrier are bounded: on expiry the kernel records
// SBM_ERR_TIMEOUT in the problem's device error word, stops, frees its tensor
// memory and returns.
#include <algorithm>

#include "sweeps.cuh"
#include "tc_common.cuh"

namespace sbm {

template <typename T>
struct TcArgs {
  const float* __restrict__ x;
  const int32_t* __restrict__ lines;       // CG gather (null for DG)
  const int32_t* __restrict__ cell_rank;   // DG gather
  const int32_t* __restrict__ face_cell;
  const int32_t* __restrict__ face_kind;
  const float* __restrict__ face_phi;      // [F][L][3][N] FP32
  float* __restrict__ out;                 // [F][2L]
  const float* __restrict__ tab;           // M, S [n][n], W [n^2]
  int* __restrict__ err;                   // device error word
  int nface;
  int dg;
};

// Points of a group's faces in the MMA's 128 rows (and their x-lines in its
// 128 columns, same numbering): n^2 > 32, two warps per face; n^2 <= 32,
// floor(32 / n^2) faces per warp.  A thread owns the row of its id.
template <int N>
struct TcShape {
  static constexpr int L = N * N, ND = L * N;
  static constexpr int FW = L <= 32 ? 32 / L : 0;         // faces per warp
  static constexpr int F = FW ? 4 * FW : 2;               // faces per group
  static constexpr int COLS = FW || L > 48 ? (FW ? 32 : 64) : 48;   // columns a warp reads
  static constexpr int kTmem = 128;
  __host__ __device__ static constexpr int row(int f, int i) {
    return FW ? 32 * (f / (FW ? FW : 1)) + (f % (FW ? FW : 1)) * L + i : 64 * f + i;
  }
  static constexpr int NX = (F * ND + 127) / 128;         // tile values per thread
  static constexpr int NA = (F * L * N + 127) / 128;      // 1D values per thread and axis
};

// KIND: 0 = TF32 (K = 8), 1 = BF16 (K = 16).  Persistent blocks over groups of
// F faces; the next group's values travel from global memory to registers
// (line starts first, then the values) while the current one is computed.
template <int KIND, int N>
__global__ void __launch_bounds__(tc::kThreads, 4)
tc_face_kernel(const TcArgs<float> a, const __grid_constant__ KTab<float> t) {
  using Sh = TcShape<N>;
  constexpr int D = 3, L = Sh::L, ND = Sh::ND, F = Sh::F, NX = Sh::NX, NA = Sh::NA;
  constexpr int ES = KIND == 0 ? 4 : 2;
  constexpr int FWd = Sh::FW ? Sh::FW : 1;
  __shared__ __align__(1024) unsigned char opA[tc::kM / 8 * tc::kGroupBytes];   // 4 KB
  __shared__ __align__(1024) unsigned char opB[tc::kM / 8 * tc::kGroupBytes];   // 4 KB
  __shared__ float X[F * ND];
  __shared__ float P12[2][N][tc::kM];      // phi of axes 1, 2 by row
  __shared__ float Td[F * L], Da[F * L], val[F * L], Va[F * L];
  __shared__ float tM[3 * L];              // M, S, W (face_body.cuh)
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  pdl_trigger();                           // the cell kernel may start (it waits before its folds)

  // zero both operands and the 1D values once (padding rows stay zero), set
  // up the mbarrier, allocate tensor memory (warp 0)
  for (int i = tid; i < (int)sizeof(opA) / 4; i += tc::kThreads) {
    ((uint32_t*)opA)[i] = 0u;
    ((uint32_t*)opB)[i] = 0u;
  }
  for (int i = tid; i < 2 * N * tc::kM; i += tc::kThreads) (&P12[0][0][0])[i] = 0.f;
  for (int i = tid; i < 3 * L; i += tc::kThreads) tM[i] = __ldg(a.tab + i);
  const float* tS = tM + L;
  if (tid == 0) {
    abort_flag = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base)),
                 "r"(Sh::kTmem));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const uint32_t idesc = tc_instr_desc(KIND == 0 ? 2 : 1, tc::kM, tc::kM);
  const uint64_t adesc = tc_smem_desc(smem_u32(opA), tc::kLBO, tc::kSBO);
  const uint64_t bdesc = tc_smem_desc(smem_u32(opB), tc::kLBO, tc::kSBO);
  uint32_t phase = 0;
  // the thread's face of the group and point
  const int fl = Sh::FW ? warp * FWd + lane / L : warp / 2;
  const int q = Sh::FW ? lane % L : tid % 64;
  const bool row_used = Sh::FW ? lane < FWd * L : q < L;
  const uint32_t tcol = tmem + ((uint32_t)(warp * 32) << 16) +
                        (uint32_t)(Sh::FW ? 32 * warp : 64 * (warp / 2));

  // prefetch registers
  int64_t gx[NX];                          // global index of each tile value
  float xv[NX], pv[3][NA];
  auto load_index = [&](int f0) {
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      const int r = tid + 128 * i, f = r / ND, loc = r - f * ND;
      gx[i] = -1;
      if (f < F && f0 + f < a.nface) {
        const int cell = __ldg(a.face_cell + f0 + f);
        gx[i] = a.dg ? (int64_t)__ldg(a.cell_rank + cell) * ND + loc
                     : (int64_t)__ldg(a.lines + (size_t)cell * L + loc / N) + loc % N;
      }
    }
  };
  auto load_values = [&]() {
#pragma unroll
    for (int i = 0; i < NX; ++i) xv[i] = gx[i] >= 0 ? __ldg(a.x + gx[i]) : 0.f;
  };
  auto load_phi = [&](int f0) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int r = tid + 128 * i, f = r / (L * N), e = r - f * (L * N);
      const bool in = f < F && f0 + f < a.nface;
      const float* p = a.face_phi + ((size_t)(f0 + f) * L + e / N) * D * N + e % N;
#pragma unroll
      for (int k = 0; k < 3; ++k) pv[k][i] = in ? __ldg(p + N * k) : 0.f;
    }
  };

  int f0 = blockIdx.x * F;
  if (f0 < a.nface) {
    load_index(f0);
    load_phi(f0);
    load_values();
  }
  for (; f0 < a.nface; f0 += gridDim.x * F) {
    const int nf = min(F, a.nface - f0);
    const bool act = row_used && fl < nf;
    // tiles and MMA operands: B[line l][j0] = u[j0][l], A[point q][j0] = phi_{j0}(xi_{q,0})
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      const int r = tid + 128 * i, f = r / ND, loc = r - f * ND;
      if (f < F) {
        X[r] = xv[i];
        const uint32_t o = tc::opnd_offset(Sh::row(f, loc / N), loc % N, ES);
        if (KIND == 0) *(uint32_t*)(opB + o) = to_tf32(xv[i]);
        else *(uint16_t*)(opB + o) = to_bf16(xv[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int r = tid + 128 * i, f = r / (L * N), e = r - f * (L * N);
      if (f < F) {
        const int rw = Sh::row(f, e / N), j = e % N;
        const uint32_t o = tc::opnd_offset(rw, j, ES);
        if (KIND == 0) *(uint32_t*)(opA + o) = to_tf32(pv[0][i]);
        else *(uint16_t*)(opA + o) = to_bf16(pv[0][i]);
        P12[0][j][rw] = pv[1][i];
        P12[1][j][rw] = pv[2][i];
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid == 0) {
      // D = A . B (enable-input-d false: no accumulation into old contents);
      // the products of one face's points with another's lines are not read
      if constexpr (KIND == 0)
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(0));
      else
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(0));
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              smem_u32(&mbar))
          : "memory");
    }
    // meanwhile: the next group's line starts and 1D values, and this one's
    // normal-derivative trace at the tangential nodes
    const int fn = f0 + gridDim.x * F;
    if (fn < a.nface) {
      load_index(fn);
      load_phi(fn);
    }
    int kind = 0;
    if (act) {
      kind = __ldg(a.face_kind + f0 + fl);
      const int k = kind & 3;
      const int sk = (k == 0) ? 1 : (k == 1 ? N : N * N);
      const int bt = (q % N) * ((k == 0) ? N : 1) + (q / N) * ((k == 2) ? N : N * N);
      float dsum = 0.f;
#pragma unroll
      for (int j = 0; j < N; ++j)
        dsum = fmaf((kind >> 2) ? t.D1[j] : t.D0[j], X[fl * ND + j * sk + bt], dsum);
      Td[fl * L + q] = dsum;
    }
    // wait for the MMA (bounded)
    uint32_t ok = 0;
    for (long long it = 0; it < tc::kWaitLimit && !ok; ++it) {
      asm volatile(
          "{\n\t.reg .pred P1;\n\tmbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
          "selp.b32 %0, 1, 0, P1;\n\t}\n"
          : "=r"(ok)
          : "r"(smem_u32(&mbar)), "r"(phase)
          : "memory");
    }
    phase ^= 1u;
    if (!ok) {
      abort_flag = 1;
      if (tid == 0) atomicExch(a.err, SBM_ERR_TIMEOUT);
    }
    if (__all_sync(0xffffffffu, ok != 0)) {
      // every warp reads its rows of T and finishes their points
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float Tq[Sh::COLS];
#pragma unroll
      for (int c0 = 0; c0 < Sh::COLS; c0 += 16) {
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
            "%10, %11, %12, %13, %14, %15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
              "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
              "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(tcol + (uint32_t)c0));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 16; ++i) Tq[c0 + i] = __uint_as_float(r[i]);
      }
      // several faces per warp: the columns of the thread's own one
#pragma unroll
      for (int g = 1; g < FWd; ++g) {
        const bool own = lane / L == g;
#pragma unroll
        for (int i = 0; i < L; ++i) Tq[i] = own ? Tq[g * L + i] : Tq[i];
      }
      float e = 0.f;
#pragma unroll
      for (int j2 = 0; j2 < N; ++j2) {
        float s1 = 0.f;
#pragma unroll
        for (int j1 = 0; j1 < N; ++j1) s1 = fmaf(P12[0][j1][tid], Tq[j1 + N * j2], s1);
        e = fmaf(P12[1][j2][tid], s1, e);
      }
      if (act) val[fl * L + q] = tS[L + q] * e;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (abort_flag) break;
    if (fn < a.nface) load_values();
    // q = (S x S)^T (W E) and (M x M) Td as in face_body.cuh
    const int ia = q % N, ib = q / N;
    if (act) {
      float v1 = 0.f, v2 = 0.f;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        v1 = fmaf(tS[N * j + ia], val[fl * L + j + N * ib], v1);
        v2 = fmaf(tM[N * j + ia], Td[fl * L + j + N * ib], v2);
      }
      Va[fl * L + q] = v1;
      Da[fl * L + q] = v2;
    }
    __syncthreads();
    if (act) {
      float qv = 0.f, tm = 0.f;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        qv = fmaf(tS[N * j + ib], Va[fl * L + ia + N * j], qv);
        tm = fmaf(tM[N * j + ib], Da[fl * L + ia + N * j], tm);
      }
      const float sg = (kind >> 2) ? 1.f : -1.f;
      float* o = a.out + (size_t)(f0 + fl) * 2 * L + q;
      o[0] = fmaf(t.sigma, qv, -(sg * t.h_inv * t.hface) * tm);
      o[L] = -(sg * t.h_inv) * qv;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(Sh::kTmem));
}

// Diagnostic: wait (bounded, `limit` polls) on an mbarrier that nothing ever
// arrives on, so the wait expires and the device error word gets
// SBM_ERR_TIMEOUT -- the same path the tensor-core kernel takes when an MMA
// never completes.  Exercises failure detection without faulting the GPU.
__global__ void timeout_selftest_kernel(int* err, long long limit) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar)));
    uint32_t ok = 0;
    for (long long it = 0; it < limit && !ok; ++it)
      asm volatile(
          "{\n\t.reg .pred P1;\n\tmbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
          "selp.b32 %0, 1, 0, P1;\n\t}\n"
          : "=r"(ok)
          : "r"(smem_u32(&bar)), "r"(0u)
          : "memory");
    if (!ok) atomicExch(err, SBM_ERR_TIMEOUT);
  }
}

cudaError_t launch_timeout_selftest(int* err, cudaStream_t st) {
  timeout_selftest_kernel<<<1, 32, 0, st>>>(err, 1ll << 14);
  return cudaGetLastError();
}

template <int KIND, int N>
static cudaError_t tc_t(const HostProblem& hp, const DeviceData& dd, const float* x, float* out,
                        cudaStream_t st) {
  if (dd.nface == 0) return cudaSuccess;
  const KTab<float> t = make_ktab<float>(hp);
  TcArgs<float> a;
  a.x = x;
  a.lines = dd.lines;
  a.cell_rank = dd.cell_rank;
  a.face_cell = dd.face_cell;
  a.face_kind = dd.face_kind;
  a.face_phi = dd.face_phi32;
  a.out = out;
  a.tab = dd.face_tab32;
  a.err = dd.err_flag;
  a.nface = dd.nface;
  a.dg = hp.desc.dg;
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // at most 4 x 128 of 512 TMEM columns per SM
  const int grid = std::min((dd.nface + TcShape<N>::F - 1) / TcShape<N>::F, 4 * sms);
  tc_face_kernel<KIND, N><<<grid, tc::kThreads, 0, st>>>(a, t);
  return cudaGetLastError();
}

cudaError_t launch_tc_face_kernel(const HostProblem& hp, const DeviceData& dd, const float* x,
                                  float* out, int face_mode, cudaStream_t st) {
  if (hp.d != 3) return cudaErrorInvalidValue;
  const int kind = (face_mode == SBM_FACE_TF32) ? 0 : 1;
#define SBM_CASE(NN)                                                  \
  if (hp.n == NN)                                                     \
    return kind == 0 ? tc_t<0, NN>(hp, dd, x, out, st) : tc_t<1, NN>(hp, dd, x, out, st);
  SBM_CASE(2) SBM_CASE(3) SBM_CASE(4) SBM_CASE(5) SBM_CASE(6) SBM_CASE(7)
#undef SBM_CASE
  return cudaErrorInvalidValue;
}

}  // namespace sbm
