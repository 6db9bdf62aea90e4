// Internal helpers shared by the library's translation units.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>

#include "class_sum.cuh"
#include "lno_ot.h"

namespace lno {

// Spin-case kinds of one triplet group.
enum CaseKind { SAME = 0, MIXED = 1 };

// One K-segment of a per-triplet contraction in float64:
//   XT[n][m] += sign * sum_k A[m][k] * B[n][k],  k < K.
struct SegF64 {
  const double* A;  // row m at A + m * lda
  const double* B;  // row n at B + n * ldb
  int K;
  int lda, ldb;
  double sign;
};

constexpr int kMaxSeg = 3;

// Problem of a grouped float64 contraction: output XT [N][ldo] (column m < M).
struct ProbF64 {
  SegF64 seg[kMaxSeg];
  int nseg;
  double* XT;
};

// Triplet descriptor for the energy kernels.
struct Trip {
  int i, j, k;   // same spin: i<j<k; mixed: i<j (spin s), k = K (spin t)
};

// Energy-kernel arguments of one triplet group.
struct EnergyArgs {
  int kind;            // SAME or MIXED
  int nvs, nvt;        // virtual counts (same spin: nvt == nvs)
  int nos, not_;       // occupied counts
  const double* eps_s; // [nbas] orbital energies of spin s (occ then vir)
  const double* eps_t; // [nbas] spin t
  const double* t1s;   // [nos][nvs]
  const double* t1t;   // [not][nvt]
  // V-term integral blocks, stored only for the occupied orbitals the computed
  // triplets use (occupied index -> slot through oslot_s / oslot_t, -1 = absent):
  // (ia|jb) spin s-s as [slot i][a][slot j][b], i.e. [ns_c][nvs][ns_c][nvs]
  const double* ovov_ss;
  // mixed: (jb|KC) as [slot K][C][slot j][b], i.e. [nt_c][nvt][ns_c][nvs]
  const double* ovov_ts;
  const int* oslot_s;  // [nos]
  const int* oslot_t;  // [not] (same spin: equal to oslot_s)
  int ns_c, nt_c;      // number of slots
  // Source of V.  vmode 0: coefficients t1s/t1t, planes from the integral
  // blocks above, the kernels sum W (W + V) / D.  vmode 1 (the restricted
  // open-shell f_ov term): t1s/t1t point at the f_ov blocks, the planes are
  // the doubles amplitudes of the same indices, and the kernels sum W V / D.
  int vmode;
  const double* t2ss;  // [nos][nos][nvs][nvs] t^{xy}_{pr} (vmode 1)
  const double* t2st;  // [nos][not][nvs][nvt] t^{xC}_{pK} (vmode 1, mixed)
  const double* fs;    // [nos][nvs] f_ov of spin s (fused mixed pass only)
  const double* ft;    // [not][nvt] f_ov of spin t (fused mixed pass only)
  const int3* blocks;  // cube tiles (A,B,C) of 16-blocks
  int nblocks;
  int pitch_x;         // row pitch (elements) of XT / YT (same: a; mixed: a)
  int pitch_z;         // row pitch of ZT (mixed: C)
  int64_t x_stride;    // elements between consecutive triplets' XT (or YT)
  int64_t z_stride;    // between consecutive ZT
  const Trip* trips;   // [ntrip]
  double* partial;     // float64 path: [ntrip][gridDim.x]; float32 path: [ntrip][nchunk][8]
  // float32 path: the tiles of a triplet are split into nchunk items
  // (chunk c: tiles c, c + nchunk, ...); nitems = ntrip * nchunk items run on a
  // persistent grid of at most (resident CTAs per SM) * nsm CTAs
  int nchunk, nitems, nsm;
  int* flag;           // device error flag (bounded waits of the TMA-staged variant)
  // bounded-wait test hook of the TMA-staged variant: stage waits give up after
  // wait_cycles (0: the normal 4e9); starve = 1 issues no copy at all
  long long wait_cycles;
  int starve;
  // mixed spin: Y and Z' stored as 16^3 tiles (kOutYTile / kOutZTile, strides
  // in floats per triplet above); selects the TMA-staged kernel
  int tiled;
  // Laplace form (Sec. 3.7, eq laplace_transform): with lap_w != 0 the
  // kernels weight each element by -lap_w exp(lap_s D) instead of 1/D (one
  // quadrature point of 1/D = -sum_q w_q exp(s_q D), D < 0)
  double lap_s, lap_w;
};

// (px|ry) of spin s in the slot-compacted [ns][nvs][ns][nvs] block
__device__ __forceinline__ int64_t ovss_idx(const EnergyArgs& a, int p, int x, int r, int y) {
  return (((int64_t)a.oslot_s[p] * a.nvs + x) * a.ns_c + a.oslot_s[r]) * a.nvs + y;
}
// (px|KC) with p of spin s, K of spin t: [nt][nvt][ns][nvs]
__device__ __forceinline__ int64_t ovts_idx(const EnergyArgs& a, int K, int C, int p, int x) {
  return (((int64_t)a.oslot_t[K] * a.nvt + C) * a.ns_c + a.oslot_s[p]) * a.nvs + x;
}

// Case sums of one call (case_sums in energy.cu): out[c] = sum of e[c][0..n[c]), copied
// to copy[c] where given.
struct CaseSums {
  const double* e[4];
  int64_t n[4];
  double* copy[4];
  double* out;
};

// Arrays measured by one launch of absmax: *out[q] = max |x[q]| (bits of a double).
struct AbsmaxList {
  static constexpr int kMax = 5;
  const double* x[kMax];
  int64_t n[kMax];
  unsigned long long* out[kMax];
  int count;
};

// The DF factor blocks of one spin in one layout launch (transpose_blocks).
template <class St>
struct BlockList {
  static constexpr int kMax = 3;
  int p0[kMax], np[kMax], q0[kMax], nq[kMax], Qp[kMax];
  St st[kMax];
};

// Inputs of the orbital partition: per-case triplets and contributions.
struct OrbPartArgs {
  const double* e[4];   // per-triplet contributions of cases aaa, aab, abb, bbb
  const Trip* trips[4];
  int64_t n[4];
  int na, nb;
  double* out[2];       // [na], [nb] (either may be NULL)
  // 0: the prefactors of eq cim_pt_energy (mixed triplet 1/4, 1/4, 1/2);
  // 1: eq local_pt's 1/3 of every triplet to each of its orbitals
  int thirds;
};

// V plane on two spin-s virtuals: vmode 0 <pr||xy> = (px|ry) - (py|rx),
// vmode 1 t^{xy}_{pr}
__device__ __forceinline__ double vplane_ss(const EnergyArgs& a, int p, int x, int r, int y) {
  if (a.vmode) return a.t2ss[(((int64_t)p * a.nos + r) * a.nvs + x) * a.nvs + y];
  return a.ovov_ss[ovss_idx(a, p, x, r, y)] - a.ovov_ss[ovss_idx(a, p, y, r, x)];
}
// V plane on a spin-s and a spin-t virtual: vmode 0 (px|KC), vmode 1 t^{xC}_{pK}
__device__ __forceinline__ double vplane_ts(const EnergyArgs& a, int K, int C, int p, int x) {
  if (a.vmode) return a.t2st[(((int64_t)p * a.not_ + K) * a.nvs + x) * a.nvt + C];
  return a.ovov_ts[ovts_idx(a, K, C, p, x)];
}

// Tensor-core contraction problem: up to kMaxSeg K-segments, each a row block
// of a sliced operand tensor addressed through a TMA map (index 0 or 1).
struct TcSeg {
  int amap, bmap;   // tensor map index (0/1) for A and B
  int a_row, b_row; // first row of the A / B operand block in its tensor
  int K;            // contraction length (k < K is real data)
  int neg;          // 1: subtract this segment
  int k0;           // first k (multiple of 32), tc_pair.cu only
};

// TcProb.flags: kTcAccum adds the result to out instead of storing it;
// kTcFloatRest forms the float64 result as HI + the float32 sum of the lower
// weight classes instead of the sum of all in integers (the adjoint's products)
// kTcAtomic (tc_pair.cu) adds with atomics: problems of one launch share an output
constexpr int kTcAccum = 1, kTcFloatRest = 2, kTcAtomic = 4;

struct TcProb {
  TcSeg seg[kMaxSeg];
  int nseg;
  int flags;        // float64 transposed output only: kTcAccum, kTcFloatRest, kTcAtomic
  void* out;        // output of this problem: [N][ldo] (transposed) or [M][ldo] (row-major)
  // float64 output of tc_pair.cu: exponents of the operands' scales on the
  // device (scale 2^(*ea + *eb - 14)); NULL: the launch's scale
  const int *ea, *eb;
};

// Output layout of a row-major float32 contraction launch (tc_pair.cu).
//   kOutRows:  out[m][n], pitch ldo.
//   kOutYTile: mixed-spin Y, rows m = b nvt + C, columns a, stored as 16^3
//              tiles (b/16, C/16, a/16), tile index (B nbt + C') nbs + A; in a
//              tile, row r = (b%16) 16 + C%16 holds 16 floats of a with its four
//              16-byte chunks permuted (chunk ^ ((r >> 1) & 3)).
//   kOutZTile: mixed-spin Z', rows m = pair(a, b) (a < b), columns C, stored as
//              tiles (a/16 <= b/16, C/16), tile index (B(B+1)/2 + A) nbt + C';
//              row r = (a%16) 16 + b%16 sits at row r ^ ((r >> 1) & 1) of the
//              tile.
// The energy kernel reads each 16^3 sub-cube of the tiled layouts with one
// 16 KB bulk copy, in the shared-memory layout its element loops index.
// Float64 output (tc_pair.cu): kOutRows out[n][m], kOutF64Rows out[m][n].
constexpr int kOutRows = 0, kOutYTile = 1, kOutZTile = 2, kOutF64Rows = 3;
struct TcOut {
  int mode;
  int nvt;    // kOutYTile: C count per b
  int nbs;    // 16-blocks of a (and b)
  int nbt;    // 16-blocks of C
};
constexpr int kTile = 4096;   // floats of one 16^3 tile

// Bounded-wait settings of one contraction launch: wait_cycles limits every
// wait for work; starve = 1 is the timeout test hook (no copy is issued, so
// the first wait for data runs out).  Library calls use tc_normal().
struct TcDiag {
  long long wait_cycles;
  int starve;
};

// tc_gemm.cu
long long tc_default_wait_cycles();
inline TcDiag tc_normal() { return TcDiag{tc_default_wait_cycles(), 0}; }
int make_operand_map(CUtensorMap* map, const void* base, int64_t Kp, int64_t rows, int S,
                     int64_t slice_stride, int box_rows, int esz = 2, int box_slices = 1);

// tc_pair.cu: the W contractions on CTA pairs, float32 row-major output
// out[m][n] in the layout `lay`.  Slice formats (the instruction descriptor's
// codes); tile of a launch (pair_tile).
// BF16 and TF32 slices carry their weights 2^(-8q), 2^(-11q); FP16 slices are
// the integer digits (weights 2^(-11q) applied to the class sums).
constexpr int kFmtF16 = 0, kFmtBF16 = 1, kFmtTF32 = 2;
struct PairTile {
  int w;        // columns of one n-tile (multiple of 16)
  int nN;       // n-tiles
  int nbuf;     // accumulator sets in TMEM (2 when 2 S w <= 512)
  int stages;   // k blocks in flight in shared memory
};
PairTile pair_tile(int S, int N, int cap);
PairTile pair_tile_f64(int S, int nprob, int M, int N);
template <int S, int FMT>
cudaError_t launch_tc_pair(const CUtensorMap* mA, const CUtensorMap* mB, const TcProb* probs_dev,
                           int nprob, int M, int N, int ldo, double scale, int* flag, int nsm,
                           cudaStream_t st, TcDiag diag, TcOut lay, PairTile tile);
template <int S, int FMT>
cudaError_t launch_tc_pair_f64(const CUtensorMap* mA, const CUtensorMap* mB, const TcProb& p,
                               int M, int N, int ldo, double scale, int* flag,
                               unsigned long long* amax, int nsm, cudaStream_t st, PairTile tile);
template <int S, int FMT>
cudaError_t launch_tc_pair_f64_group(const CUtensorMap* mA, const CUtensorMap* mB,
                                     const TcProb* probs_dev, int nprob, int M, int N, int ldo,
                                     double scale, int* flag, int nsm, cudaStream_t st,
                                     int mode, PairTile tile, TcDiag diag = tc_normal());
int sliced_product_bn(int S);
cudaError_t launch_sliced_product(int S, const CUtensorMap* mA, const CUtensorMap* mB,
                                  const TcProb* dp, int M, int N, double scale, int* flag,
                                  int nsm, cudaStream_t st, TcDiag dg);

// Augmented domain of the central-LMO pass (central.cu): P pseudo-orbitals
// appended after the occupied orbitals of spin `spin`, for quadrature point s.
struct AugmentArgs {
  int spin, P, nbas, naux, nocc[2];
  double s;
  const double* U;        // [P][nocc[spin]] LMO coefficients
  const double* B_in;     // [naux][nbas][nbas] of `spin`
  const double* eps_in;   // [nbas]
  const double* t1_in;    // [nocc][nvir]
  const double* fov_in;   // [nocc][nvir] or NULL
  const double* t2ss_in;  // same-spin doubles of `spin`
  const double* t2ab_in;  // [na][nb][va][vb]
  double* coef;           // [P][nocc[spin]]
  double *B_out, *eps_out, *t1_out, *fov_out, *t2ss_out, *t2ab_out;
};
cudaError_t launch_lmo_augment(const AugmentArgs& A, cudaStream_t st);
int laplace_quadrature(double xmin, double xmax, double tol, int nmax, double* s, double* w,
                       int* nq);

// Operand stores used by the layout kernels.  `part` says whether the value
// is an amplitude (0) or an integral (1): the two have separate scales.
// store16 writes 16 consecutive elements (idx a multiple of 16, rows starting
// on 32-byte boundaries); bit j of `parts` is the part of element j.
struct StoreF64 {
  double* p;
  __device__ __forceinline__ void operator()(int64_t idx, double v, int) const { p[idx] = v; }
  __device__ __forceinline__ void store16(int64_t idx, const double (&v)[16], uint32_t) const {
#pragma unroll
    for (int j = 0; j < 16; ++j) p[idx + j] = v[j];
  }
};

// round(v 2^e2) to nearest (ties to even) from the bits of v, in integer
// arithmetic (this GPU's float64 rate is 1/64 of its float32 rate); |v 2^e2|
// must stay below 2^62, v finite.
__device__ __forceinline__ int64_t round_scaled(double v, int e2) {
  const uint64_t b = (uint64_t)__double_as_longlong(v);
  const int ex = (int)((b >> 52) & 0x7ff);
  uint64_t m = b & ((1ull << 52) - 1);
  if (ex != 0) m |= 1ull << 52;
  const int sh = (ex == 0 ? 1 : ex) - 1075 + e2;   // |v| 2^e2 = m 2^sh
  uint64_t q;
  if (m == 0) {
    q = 0;
  } else if (sh >= 0) {
    q = m << sh;
  } else if (-sh > 54) {
    q = 0;                                        // m 2^sh < 1/2
  } else {
    const int r = -sh;
    const uint64_t rem = m & ((1ull << r) - 1), half = 1ull << (r - 1);
    q = m >> r;
    if (rem > half || (rem == half && (q & 1))) ++q;
  }
  return (b >> 63) ? -(int64_t)q : (int64_t)q;
}

// Exact slices of S digits of BITS bits: value = 2^-e (s_0 + ... + s_{S-1}),
// s_q an integer multiple of 2^(-BITS q), |s_0| <= 2^(BITS - 1) (2^BITS / 2, the
// scale's choice), |s_q| 2^(BITS q) <= 2^(BITS - 1) below it, each digit the
// nearest one to what is left.  Integer arithmetic throughout: the value is
// rounded once, to 54 - BITS bits after the point (beyond what a float64 near the
// scale holds, so the digits are those of the value itself), and cut from the top
// (float64 rounding steps of every digit made the layout kernels 10-20x slower
// than their memory traffic).  A value that is not finite, or too large for the
// scale, becomes NaN.
template <int S, int BITS, bool INTS = false>   // INTS: f[q] = s_q 2^(BITS q)
__device__ __forceinline__ void slice_digits(double v, int e, float (&f)[S]) {
  constexpr int kX = 54 - BITS * S;   // bits kept below the last digit
  const int ex = (int)(((uint64_t)__double_as_longlong(v) >> 52) & 0x7ff);
  if (ex == 0x7ff || ex - 1023 + e > 60 - (BITS * (S - 1) + kX)) {
    f[0] = __int_as_float(0x7fc00000);
#pragma unroll
    for (int q = 1; q < S; ++q) f[q] = 0.f;
    return;
  }
  int64_t R = round_scaled(v, e + BITS * (S - 1) + kX);
  float w = 1.0f;
#pragma unroll
  for (int q = 0; q < S; ++q) {
    const int sh = BITS * (S - 1 - q) + kX;
    // nearest, ties to even (integrals lie on a grid of their own, so ties are common)
    const int64_t d = (R + ((1ll << (sh - 1)) - 1) + ((R >> sh) & 1)) >> sh;
    R -= d << sh;
    f[q] = (float)(int)d * w;   // exact
    if (!INTS) w *= 1.0f / (float)(1 << BITS);
  }
}

// 16-bit slices.  BF16: value = scale 2^-7 (s_0 + ... + s_{S-1}), s_0 an integer
// in [-128,128], s_q a multiple of 2^(-8q).  FP16: value = scale 2^-10 (d_0 +
// 2^-11 d_1 + 2^-22 d_2), integers of [-1024, 1024] (11 bits, exact in FP16).
template <typename T>
struct SliceFmt;
template <>
struct SliceFmt<__nv_bfloat16> {
  static constexpr int bits = 8;
  static constexpr bool ints = false;
  static __device__ __forceinline__ __nv_bfloat16 one(float x) { return __float2bfloat16_rn(x); }
  static __device__ __forceinline__ uint32_t two(float a, float b) {
    const __nv_bfloat162 x = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&x);
  }
};
template <>
struct SliceFmt<__half> {
  static constexpr int bits = 11;
  static constexpr bool ints = true;
  static __device__ __forceinline__ __half one(float x) { return __float2half_rn(x); }
  static __device__ __forceinline__ uint32_t two(float a, float b) {
    const __half2 x = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&x);
  }
};

template <int S, typename T = __nv_bfloat16>
struct StoreSlices {
  using F = SliceFmt<T>;
  T* p;
  int64_t slice_stride;  // elements between slices
  int e_t, e_i;          // log2(2^7 or 2^10 / scale) of amplitudes and of integrals
  __device__ __forceinline__ void operator()(int64_t idx, double v, int part) const {
    float f[S];
    slice_digits<S, F::bits, F::ints>(v, part ? e_i : e_t, f);
#pragma unroll
    for (int s = 0; s < S; ++s) p[s * slice_stride + idx] = F::one(f[s]);
  }
  __device__ __forceinline__ void store16(int64_t idx, const double (&v)[16],
                                          uint32_t parts) const {
    uint32_t w[S][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float a[S], b[S];
      slice_digits<S, F::bits, F::ints>(v[2 * j], (parts >> (2 * j)) & 1 ? e_i : e_t, a);
      slice_digits<S, F::bits, F::ints>(v[2 * j + 1], (parts >> (2 * j + 1)) & 1 ? e_i : e_t, b);
#pragma unroll
      for (int s = 0; s < S; ++s) w[s][j] = F::two(a[s], b[s]);
    }
#pragma unroll
    for (int s = 0; s < S; ++s) {
      uint4* d = reinterpret_cast<uint4*>(p + s * slice_stride + idx);
      d[0] = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
      d[1] = make_uint4(w[s][4], w[s][5], w[s][6], w[s][7]);
    }
  }
};

// TF32 slices (stored as float): value = scale 2^-10 (s_0 + ... + s_{S-1}), s_0
// an integer in [-1024, 1024], s_q a multiple of 2^(-11q): 11 significant bits
// each, what one TF32 operand holds.
template <int S>
struct StoreTF32 {
  float* p;
  int64_t slice_stride;
  int e_t, e_i;          // log2(2^10 / scale) of amplitudes and of integrals
  __device__ __forceinline__ void operator()(int64_t idx, double v, int part) const {
    float f[S];
    slice_digits<S, 11>(v, part ? e_i : e_t, f);
#pragma unroll
    for (int s = 0; s < S; ++s) p[s * slice_stride + idx] = f[s];
  }
  __device__ __forceinline__ void store16(int64_t idx, const double (&v)[16],
                                          uint32_t parts) const {
#pragma unroll
    for (int j = 0; j < 16; ++j) (*this)(idx + j, v[j], (parts >> j) & 1);
  }
};

__host__ __device__ inline int64_t pair_index(int p, int q) {  // p < q
  return (int64_t)q * (q - 1) / 2 + p;
}
__host__ __device__ inline int64_t npairs(int n) { return (int64_t)n * (n - 1) / 2; }

inline int ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }
inline int64_t round_up(int64_t a, int64_t b) { return (a + b - 1) / b * b; }

}  // namespace lno

#define LNO_CUDA_TRY(expr)                                                   \
  do {                                                                       \
    cudaError_t e__ = (expr);                                                \
    if (e__ != cudaSuccess) {                                                \
      lno_set_last_error(#expr, e__, __FILE__, __LINE__);                    \
      return LNO_OT_ECUDA;                                                   \
    }                                                                        \
  } while (0)

void lno_set_last_error(const char* what, cudaError_t e, const char* file, int line);
