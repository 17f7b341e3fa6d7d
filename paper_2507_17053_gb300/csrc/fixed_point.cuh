// Fixed-point line arithmetic of the FP64 cell term.
//
// GB300 executes 2 double-precision operations per SM and clock but 64
// multiply-adds of 32-bit integers into a 64-bit sum (mad.wide; measured 17.9
// T/s against 0.63 T/s).  A 3D cell's values therefore enter the cell term as
// 61-bit fixed-point numbers with one exponent per cell, every 1D product of
// Algorithm 1 runs on the integer units, and the results are rounded to double
// once at the end.
//
// Formats.  A value is q 2^(E - 1022 - 60), E the cell's largest biased
// exponent, |q| <= 2^60.  A matrix entry is the integer A 2^t = h 2^30 + l / 2
// (|h| < 2^31, |l| <= 2^30), t such that the entries a result sums add up to
// less than 2^61; then with q = qh 2^31 + ql (0 <= ql < 2^31), |q| <= 2^61
//   sum A q 2^(t - 61 + K) = 2^K sum h qh + 2^(K - 31) sum (h ql + l qh)
//                            + (l ql terms, below 2^(K + 1) units)
// -- three mad.wide per product and every sum inside 64 bits.
//
// Scales.  Phase i of the cell term leaves its values at 2^S_i of the input's
// scale, S_i the largest with |q| <= 2^60 for every input: from the largest
// absolute row sum of the operator from the input to that phase (not of the
// phases' product, which would cost up to 7 bits), the modes' rows scaled by
// powers of two to nearly equal sums first.  No phase can overflow, and the
// rounding of a phase is 2^-60 of its largest possible value: the error of
// the cell term, measured against quadruple precision over random, smooth,
// graded and single-spike data, is 5e-17 .. 1.3e-15 of the result's norm,
// against 8e-16 .. 2.6e-15 in double precision.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define SBM_FIX __host__ __device__ __forceinline__
#else
#define SBM_FIX inline
#endif

namespace sbm {
namespace fix {

constexpr int kMaxHalf = 4;          // ceil(7 / 2)
constexpr int kFaceExpBad = -0x40000000;   // exponent of a face with non-finite tables

// the output shifts K of the phases for n nodes: x-lines, y-modes back,
// z-modes back (the transforms to the modes need none)
SBM_FIX constexpr int shift_x(int n) {
  return n == 2 ? 1 : n == 3 ? 2 : n == 4 ? 1 : n == 5 ? 2 : 0;
}
SBM_FIX constexpr int shift_y(int n) { return n == 3 ? 0 : n == 7 ? 2 : 1; }
SBM_FIX constexpr int shift_z(int n) { return n <= 3 ? 1 : n == 4 ? 2 : 3; }

struct alignas(8) Entry {
  int32_t h, l;                      // A 2^t = h 2^30 + l / 2
};

SBM_FIX Entry to_entry(int64_t I) {
  const int64_t h = (I + ((int64_t)1 << 29)) >> 30;
  return Entry{(int32_t)h, (int32_t)(2 * (I - h * ((int64_t)1 << 30)))};
}

// a b 2^t as an entry, rounded to nearest, of two finite doubles' bits;
// |a b 2^t| < 2^61.  (In integers: in double precision the product, its error and
// their conversions took nine operations of the slow pipe.)
SBM_FIX Entry product(uint64_t a, uint64_t b, int t) {
  const uint64_t frac = ((uint64_t)1 << 52) - 1;
  const int ea = (int)(a >> 52) & 0x7ff, eb = (int)(b >> 52) & 0x7ff;
  const uint64_t ma = (a & frac) | (ea ? frac + 1 : 0), mb = (b & frac) | (eb ? frac + 1 : 0);
  const int sh = 2150 - (ea ? ea : 1) - (eb ? eb : 1) - t;
  const uint64_t lo = ma * mb;
#ifdef __CUDA_ARCH__
  const uint64_t hi = __umul64hi(ma, mb);
#else
  const uint64_t hi = (uint64_t)(((unsigned __int128)ma * mb) >> 64);
#endif
  uint64_t r = 0;                              // the product is below 2^106
  if (sh <= 0) r = sh > -64 ? lo << -sh : 0;
  else if (sh < 64) r = ((hi << (64 - sh)) | (lo >> sh)) + ((lo >> (sh - 1)) & 1u);
  else if (sh == 64) r = hi + (lo >> 63);
  else if (sh < 107) r = (hi >> (sh - 64)) + ((hi >> (sh - 65)) & 1u);
  return to_entry((int64_t)((a ^ b) >> 63 ? 0 - r : r));
}

// even and odd block of a centrosymmetric or (anti)symmetric-column matrix
struct Block {
  Entry E[kMaxHalf][kMaxHalf];
  Entry O[kMaxHalf][kMaxHalf];
};

// Line operators of the 3D DG apply (dg_apply.cu): K and M folded, and the
// interior-face vector w (w[0] = pen + D0[0], without pen where the apply adds
// the penalty in double; w[j] = D0[j] / 2); the result's exponent word is
// E + eoff.
struct DgTab {
  Block K, M;
  Entry w[2 * kMaxHalf];
  int eoff;
};

// a value split for the products
struct alignas(8) Split {
  int32_t h, l;                      // q = h 2^31 + l, 0 <= l < 2^31
};
SBM_FIX Split split(int64_t q) { return Split{(int32_t)(q >> 31), (int32_t)(q & 0x7fffffff)}; }

// c + a b; one instruction on the device (left to the compiler, the products
// with ql, known to be non-negative, become mixed-sign 64-bit multiplications)
SBM_FIX int64_t mad_wide(int32_t a, int32_t b, int64_t c) {
#ifdef __CUDA_ARCH__
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"((long long)c));
  return d;
#else
  return c + (int64_t)a * b;
#endif
}

// (a << K) + b
template <int K>
SBM_FIX int64_t shl_add(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
  // on the multiply-add pipe (the adds and shifts of the rest fill the other)
  int lo, hi, blo, bhi;
  long long d;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"((long long)a));
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(lo), "n"(1 << K), "l"((long long)b));
  asm("mov.b64 {%0, %1}, %2;" : "=r"(blo), "=r"(bhi) : "l"(d));
  asm("mad.lo.s32 %0, %1, %2, %0;" : "+r"(bhi) : "r"(hi), "n"(1 << K));
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(blo), "r"(bhi));
  return d;
#else
  return (int64_t)((uint64_t)a << K) + b;
#endif
}

// sum_j A[j] q[j] 2^(t - 61 + K); A(j), the entries
template <int K, int M, typename At>
SBM_FIX int64_t dot(const At& A, const Split (&q)[M]) {
  int64_t mid = (int64_t)1 << (30 - K);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int j = 0; j < M; ++j) {
    const Entry a = A(j);
    mid = mad_wide(a.h, q[j].l, mid);
    mid = mad_wide(a.l, q[j].h, mid);
  }
  if (K == 0) {
    int64_t r = mid >> 31;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = 0; j < M; ++j) r = mad_wide(A(j).h, q[j].h, r);
    return r;
  }
  int64_t r = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int j = 0; j < M; ++j) r = mad_wide(A(j).h, q[j].h, r);
  return shl_add<K>(r, mid >> (31 - K));
}

// even and odd parts of a line
template <int N>
struct Fold {
  static constexpr int H = N / 2, HE = (N + 1) / 2;
  Split e[HE];
  Split o[H];
  SBM_FIX explicit Fold(const int64_t (&v)[N]) {
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = 0; j < H; ++j) {
      e[j] = split(v[j] + v[N - 1 - j]);
      o[j] = split(v[j] - v[N - 1 - j]);
    }
    if (N & 1) e[H] = split(v[H]);
  }
  SBM_FIX Fold() {}
  // modes: even ones first, already apart
  SBM_FIX static Fold of_modes(const int64_t (&w)[N]) {
    Fold f;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int i = 0; i < HE; ++i) f.e[i] = split(w[i]);
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int i = 0; i < H; ++i) f.o[i] = split(w[HE + i]);
    return f;
  }
};

// w = V^T v (even modes first)
template <int N, int K>
SBM_FIX void to_modes(const Block& Vt, const int64_t (&v)[N], int64_t (&w)[N]) {
  constexpr int H = N / 2, HE = (N + 1) / 2;
  const Fold<N> f(v);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int i = 0; i < HE; ++i) w[i] = dot<K, HE>([&](int j) { return Vt.E[i][j]; }, f.e);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int i = 0; i < H; ++i) w[HE + i] = dot<K, H>([&](int j) { return Vt.O[i][j]; }, f.o);
}

// y = V w
template <int N, int K>
SBM_FIX void from_modes(const Block& V, const int64_t (&w)[N], int64_t (&y)[N]) {
  constexpr int H = N / 2, HE = (N + 1) / 2;
  const Fold<N> f = Fold<N>::of_modes(w);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int i = 0; i < H; ++i) {
    const int64_t s = dot<K, HE>([&](int j) { return V.E[i][j]; }, f.e);
    const int64_t d = dot<K, H>([&](int j) { return V.O[i][j]; }, f.o);
    y[i] = s + d;
    y[N - 1 - i] = s - d;
  }
  if (N & 1) y[H] = dot<K, HE>([&](int j) { return V.E[H][j]; }, f.e);
}

// y = A v for a centrosymmetric A whose blocks are read by E(i, j), O(i, j)
template <int N, int K, typename FE, typename FO>
SBM_FIX void apply_line(const FE& E, const FO& O, const int64_t (&v)[N], int64_t (&y)[N]) {
  constexpr int H = N / 2, HE = (N + 1) / 2;
  const Fold<N> f(v);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int i = 0; i < H; ++i) {
    const int64_t s = dot<K, HE>([&](int j) { return E(i, j); }, f.e);
    const int64_t d = dot<K, H>([&](int j) { return O(i, j); }, f.o);
    y[i] = s + d;
    y[N - 1 - i] = s - d;
  }
  if (N & 1) y[H] = dot<K, HE>([&](int j) { return E(H, j); }, f.e);
}

// ---- conversion ------------------------------------------------------------
//
// E is the largest biased exponent of the cell (1 if all are subnormal).
// Cells with E outside [kExpMin, kExpMax] (zeros, subnormals, near overflow)
// take the careful conversions (the apply of a zero vector, p = 1 .. 6, takes as long
// as another in CG, up to 4 % longer in DG); kExpBad marks infinities and NaN
// (the cell's results are NaN).
constexpr int kExpMin = 128, kExpMax = 1900, kExpBad = 0x7ff;

SBM_FIX bool plain_exp(int E) { return E >= kExpMin && E <= kExpMax; }

// index of a thread's group of lanes (2^27 cells of 32 lanes are 2^32 threads)
SBM_FIX int64_t group_of(unsigned block, int threads, unsigned thread, int lanes) {
  return ((int64_t)block * threads + thread) / lanes;
}

// a value's magnitude by its high word; the cell's largest >> 20 is E
SBM_FIX uint32_t mag_hi(uint64_t bits) { return (uint32_t)(bits >> 32) & 0x7fffffffu; }

// double -> q (rounded down)
template <bool Careful>
SBM_FIX int64_t from_double(uint64_t bits, int E) {
  const uint32_t hi = (uint32_t)(bits >> 32), lo = (uint32_t)bits;
  int e = (int)((hi >> 20) & 0x7ffu);
  uint32_t mh = (hi & 0xfffffu) | 0x100000u;
  if (Careful && e == 0) {
    mh = hi & 0xfffffu;
    e = 1;
  }
  uint64_t m = (((uint64_t)mh << 32) | lo) << 7;
  const int sh = E - e;
  const int64_t s = (int64_t)((int32_t)hi >> 31);
  return (((int64_t)m ^ s) - s) >> (sh < 63 ? sh : 63);
}

// to_double<false> serves results that can be neither subnormal nor infinite:
// biased exponents eb + 63 - lz, 2 <= lz <= 63
SBM_FIX bool plain_result(int eb) { return eb >= 1 && eb <= 1984; }

// q 2^(eb - 1023) -> double, rounded to nearest; |q| < 2^62
template <bool Careful>
SBM_FIX uint64_t to_double(int64_t q, int eb) {
  const int64_t s = q >> 63;
  const uint64_t mag = (uint64_t)((q ^ s) - s);
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)mag);
#else
  const int lz = mag ? __builtin_clzll(mag) : 64;
#endif
  if (mag == 0) return 0;
  const uint64_t sign = (uint64_t)s & 0x8000000000000000ull;
  const uint64_t m = ((mag << (lz - 1)) + 0x200u) >> 10;   // leading bit 52 (53 after a carry)
  const int ex = eb + 62 - lz;                             // biased exponent - 1
  if (Careful) {
    if (ex >= 2046 || (ex == 2045 && (m >> 53))) return sign | 0x7ff0000000000000ull;
    if (ex < 0) return sign | (ex < -53 ? 0 : m >> (-ex));
  }
  return sign | (((uint64_t)(uint32_t)ex << 52) + m);
}

}  // namespace fix
}  // namespace sbm
