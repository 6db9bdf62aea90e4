// W / V assembly and denominator-weighted energy reduction of one triplet
// group (eq cim_pt_energy: sum over restricted abc of W (W + V) / D).
//
// The contraction kernels leave, per triplet, the P(i/jk)-antisymmetrised
// intermediate X (same spin) or Y and Z' (mixed spin) in HBM.  This kernel
// applies the virtual antisymmetriser on the fly:
//   same spin  W_abc = X[a,(bc)] - X[b,(ac)] + X[c,(ab)]            a<b<c
//   mixed      W_abC = Y[a,(bC)] - Y[b,(aC)] + Z'[C,(ab)]           a<b
// adds the T1 term V, and sums W (W + V) / D over the restricted elements.
//
// Work split: a CTA owns a list of 16x16x16 cube tiles (A<=B<=C blocks for
// same spin, A<=B plus any C for mixed) of one triplet, stages the three X
// sub-cubes it needs in shared memory (each X element is read once), and
// writes one float64 partial.  Partials are reduced per triplet in a fixed
// order afterwards, so results are bitwise reproducible.
//
// Precision: with float64 X everything is float64.  With float32 X (tensor
// core path) W, V and W (W+V) are float32, the denominator is formed from
// float64 orbital energies as a double-float and rounded once to float32,
// the quotient is correctly rounded, 16 elements are summed in float32 and
// every such partial is added in float64 (all roundings to nearest, so no
// systematic bias builds up over the ~1e12 elements of a large domain).
#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"

namespace lno {

namespace {

constexpr int TB = 16;          // cube tile edge
constexpr int TP = TB + 1;      // padded row pitch in shared memory

struct TwoF { float hi, lo; };

__device__ __forceinline__ TwoF split_df(double x) {
  float h = __double2float_rn(x);
  float l = __double2float_rn(x - (double)h);
  return {h, l};
}

// Double-float a - b rounded once to float (Knuth two-sum on the high words).
__device__ __forceinline__ float df_sub_round(TwoF a, TwoF b) {
  float s = __fsub_rn(a.hi, b.hi);
  float bb = __fsub_rn(s, a.hi);
  float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(-b.hi, bb));
  float lo = __fadd_rn(err, __fsub_rn(a.lo, b.lo));
  return __fadd_rn(s, lo);
}

template <typename T>
__device__ __forceinline__ void load_row16(T* dst, const T* src) {
#pragma unroll
  for (int q = 0; q < TB; ++q) dst[q] = src[q];
}

template <>
__device__ __forceinline__ void load_row16<float>(float* dst, const float* src) {
  const float4* s4 = reinterpret_cast<const float4*>(src);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float4 v = __ldg(s4 + q);
    dst[4 * q + 0] = v.x; dst[4 * q + 1] = v.y; dst[4 * q + 2] = v.z; dst[4 * q + 3] = v.w;
  }
}

template <>
__device__ __forceinline__ void load_row16<double>(double* dst, const double* src) {
  const double2* s2 = reinterpret_cast<const double2*>(src);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    double2 v = __ldg(s2 + q);
    dst[2 * q + 0] = v.x; dst[2 * q + 1] = v.y;
  }
}

template <typename T, bool MIXED, bool FM>
__global__ void __launch_bounds__(256)
energy_group(EnergyArgs a, const T* __restrict__ X, const T* __restrict__ Z) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* T1 = reinterpret_cast<T*>(smem_raw);
  T* T2 = T1 + TB * TB * TP;
  T* T3 = T2 + TB * TB * TP;
  // V tables: 9 planes of 16x16 (same: K^{jk},K^{ki},K^{ij} on BC, AC, AB;
  // mixed: (jb|KC),(ib|KC) on BC; (ja|KC),(ia|KC) on AC; <ij||ab> on AB)
  __shared__ T vt[9][TB][TP];
  __shared__ T t1s[9][TB];        // t1 of the triplet's occupied on A, B, C
  __shared__ double ev[3][TB];    // virtual energies of the A, B, C blocks
  __shared__ double red[8];

  const int g = blockIdx.y;
  const Trip tr = a.trips[g];
  const T* Xg = X + (int64_t)g * a.x_stride;
  const T* Zg = MIXED ? Z + (int64_t)g * a.z_stride : nullptr;
  const int tid = threadIdx.x;
  const int r1 = tid / TB, r2 = tid % TB;
  const int nvs = a.nvs, nvt = a.nvt;
  const double eocc = MIXED
      ? a.eps_s[tr.i] + a.eps_s[tr.j] + a.eps_t[tr.k]
      : a.eps_s[tr.i] + a.eps_s[tr.j] + a.eps_s[tr.k];

  double acc = 0.0;
  for (int q = blockIdx.x; q < a.nblocks; q += gridDim.x) {
    const int3 blk = a.blocks[q];
    const int a0 = blk.x * TB, b0 = blk.y * TB, c0 = blk.z * TB;
    // ---- stage X sub-cubes: thread owns row (r1, r2) of each tile --------
    if (!MIXED) {
      {  // T1[b][c][a] = X[a,(bc)]
        int b = b0 + r1, c = c0 + r2;
        if (b < c && c < nvs)
          load_row16(T1 + (r1 * TB + r2) * TP, Xg + pair_index(b, c) * a.pitch_x + a0);
      }
      {  // T2[a][c][b] = X[b,(ac)]
        int aa = a0 + r1, c = c0 + r2;
        if (aa < c && c < nvs)
          load_row16(T2 + (r1 * TB + r2) * TP, Xg + pair_index(aa, c) * a.pitch_x + b0);
      }
      {  // T3[a][b][c] = X[c,(ab)]
        int aa = a0 + r1, b = b0 + r2;
        if (aa < b && b < nvs)
          load_row16(T3 + (r1 * TB + r2) * TP, Xg + pair_index(aa, b) * a.pitch_x + c0);
      }
    } else {
      {  // T1[b][C][a] = Y[a,(bC)]
        int b = b0 + r1, c = c0 + r2;
        if (b < nvs && c < nvt)
          load_row16(T1 + (r1 * TB + r2) * TP, Xg + ((int64_t)b * nvt + c) * a.pitch_x + a0);
      }
      {  // T2[a][C][b] = Y[b,(aC)]
        int aa = a0 + r1, c = c0 + r2;
        if (aa < nvs && c < nvt)
          load_row16(T2 + (r1 * TB + r2) * TP, Xg + ((int64_t)aa * nvt + c) * a.pitch_x + b0);
      }
      {  // T3[a][b][C] = Z'[C,(ab)]
        int aa = a0 + r1, b = b0 + r2;
        if (aa < b && b < nvs)
          load_row16(T3 + (r1 * TB + r2) * TP, Zg + pair_index(aa, b) * a.pitch_z + c0);
      }
    }
    // ---- V tables -----------------------------------------------------------
    {
      if (!MIXED) {
        const int occ3[3][2] = {{tr.j, tr.k}, {tr.k, tr.i}, {tr.i, tr.j}};
        const int offs[3][2] = {{b0, c0}, {a0, c0}, {a0, b0}};
#pragma unroll
        for (int pl = 0; pl < 3; ++pl) {          // index plane (BC, AC, AB)
          const int x = offs[pl][0] + r1, y = offs[pl][1] + r2;
#pragma unroll
          for (int o = 0; o < 3; ++o) {
            T v = 0;
            if (x < nvs && y < nvs) {
              const int p = occ3[o][0], r = occ3[o][1];
              v = (T)vplane_ss(a, p, x, r, y);   // K^{pr}_{xy} (or t^{xy}_{pr})
            }
            vt[pl * 3 + o][r1][r2] = v;
          }
        }
      } else {
        const int nt = a.not_;
        const int K = tr.k;
        // planes 0,1: (jb|KC),(ib|KC) on (B,C); 2,3: (ja|KC),(ia|KC) on (A,C)
        const int offs[2] = {b0, a0};
#pragma unroll
        for (int pl = 0; pl < 2; ++pl) {
          const int x = offs[pl] + r1, y = c0 + r2;
#pragma unroll
          for (int o = 0; o < 2; ++o) {
            T v = 0;
            if (x < nvs && y < nvt) {
              const int p = o == 0 ? tr.j : tr.i;
              v = (T)vplane_ts(a, K, y, p, x);
            }
            vt[pl * 2 + o][r1][r2] = v;
          }
        }
        {  // plane 4: (ia|jb) - (ib|ja) on (A,B)
          const int x = a0 + r1, y = b0 + r2;
          T v = 0;
          if (x < nvs && y < nvs) v = (T)vplane_ss(a, tr.i, x, tr.j, y);
          vt[4][r1][r2] = v;
        }
        (void)nt;
      }
      if (tid < 3 * TB) {
        const int bl = tid / TB, l = tid % TB;
        const int base = bl == 0 ? a0 : (bl == 1 ? b0 : c0);
        const int x = base + l;
        const bool tblock = MIXED && bl == 2;
        const int nv = tblock ? nvt : nvs;
        if (!MIXED) {
          const int occ[3] = {tr.i, tr.j, tr.k};
#pragma unroll
          for (int o = 0; o < 3; ++o)
            t1s[bl * 3 + o][l] = x < nvs ? (T)a.t1s[(int64_t)occ[o] * nvs + x] : (T)0;
        } else if (!tblock) {
          t1s[bl * 3 + 0][l] = x < nvs ? (T)a.t1s[(int64_t)tr.i * nvs + x] : (T)0;
          t1s[bl * 3 + 1][l] = x < nvs ? (T)a.t1s[(int64_t)tr.j * nvs + x] : (T)0;
        } else {
          t1s[bl * 3 + 0][l] = x < nvt ? (T)a.t1t[(int64_t)tr.k * nvt + x] : (T)0;
        }
        const double* e = tblock ? a.eps_t : a.eps_s;
        const int no = tblock ? a.not_ : a.nos;
        ev[bl][l] = x < nv ? e[no + x] : 0.0;
      }
    }
    __syncthreads();
    // ---- elements: thread (b = r1, c = r2), loop over a ---------------------
    {
      const int bl = r1, cl = r2;
      const int b = b0 + bl, c = c0 + cl;
      const bool rowok = MIXED ? (b < nvs && c < nvt) : (b < c && c < nvs);
      if (rowok) {
        const double dbc = eocc - ev[1][bl] - ev[2][cl];
        int amax = MIXED ? min(b, a0 + TB) : min(b, a0 + TB);  // a < b
        const int na = amax - a0;
        if constexpr (sizeof(T) == 8) {
          for (int al = 0; al < na; ++al) {
            const double x1 = T1[(bl * TB + cl) * TP + al];
            const double x2 = T2[(al * TB + cl) * TP + bl];
            const double x3 = T3[(al * TB + bl) * TP + cl];
            const double w = x1 - x2 + x3;
            double v;
            if (!MIXED) {
              const double ya = t1s[0][al] * vt[0][bl][cl] + t1s[1][al] * vt[1][bl][cl] +
                                t1s[2][al] * vt[2][bl][cl];
              const double yb = t1s[3][bl] * vt[3][al][cl] + t1s[4][bl] * vt[4][al][cl] +
                                t1s[5][bl] * vt[5][al][cl];
              const double yc = t1s[6][cl] * vt[6][al][bl] + t1s[7][cl] * vt[7][al][bl] +
                                t1s[8][cl] * vt[8][al][bl];
              v = ya - yb + yc;
            } else {
              v = t1s[0][al] * vt[0][bl][cl] - t1s[1][al] * vt[1][bl][cl] -
                  t1s[3][bl] * vt[2][al][cl] + t1s[4][bl] * vt[3][al][cl] +
                  t1s[6][cl] * vt[4][al][bl];
            }
            const double D = dbc - ev[0][al];
            const double num = FM ? w * v : w * (w + v);
            acc += a.lap_w != 0.0 ? num * (-a.lap_w * exp(a.lap_s * D)) : num / D;
          }
        } else {
          const TwoF dd = split_df(dbc);
          float part = 0.f;
          for (int al = 0; al < na; ++al) {
            const float x1 = T1[(bl * TB + cl) * TP + al];
            const float x2 = T2[(al * TB + cl) * TP + bl];
            const float x3 = T3[(al * TB + bl) * TP + cl];
            const float w = x1 - x2 + x3;
            float v;
            if (!MIXED) {
              const float ya = t1s[0][al] * vt[0][bl][cl] + t1s[1][al] * vt[1][bl][cl] +
                               t1s[2][al] * vt[2][bl][cl];
              const float yb = t1s[3][bl] * vt[3][al][cl] + t1s[4][bl] * vt[4][al][cl] +
                               t1s[5][bl] * vt[5][al][cl];
              const float yc = t1s[6][cl] * vt[6][al][bl] + t1s[7][cl] * vt[7][al][bl] +
                               t1s[8][cl] * vt[8][al][bl];
              v = ya - yb + yc;
            } else {
              v = t1s[0][al] * vt[0][bl][cl] - t1s[1][al] * vt[1][bl][cl] -
                  t1s[3][bl] * vt[2][al][cl] + t1s[4][bl] * vt[3][al][cl] +
                  t1s[6][cl] * vt[4][al][bl];
            }
            const float num = FM ? __fmul_rn(w, v) : __fmul_rn(w, __fadd_rn(w, v));
            const float D = df_sub_round(dd, split_df(ev[0][al]));
            part = __fadd_rn(part, a.lap_w != 0.0
                                       ? num * (float)(-a.lap_w * exp(a.lap_s * (double)D))
                                       : __fdiv_rn(num, D));
          }
          acc += (double)part;
        }
      }
    }
    __syncthreads();
  }
  // ---- CTA reduction (fixed order) ---------------------------------------------
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
  if ((tid & 31) == 0) red[tid >> 5] = acc;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w];
    a.partial[(int64_t)g * gridDim.x + blockIdx.x] = s;
  }
}

// ---------------------------------------------------------------------------
// Tensor-core path (float32 X): per-triplet V tables, then the energy.
//
// energy_prep writes, per triplet of the group, the float32 integral tables
// the T1 term needs (full square, rows padded to a multiple of 16):
//   same spin: plane o = K^{pr}_{xy} = (px|ry) - (py|rx) for
//              (p,r) = (j,k), (k,i), (i,j)                  [3][nv][pv]
//   mixed:     plane 0 (jx|KC), plane 1 (ix|KC)             [nvs][pvt] each
//              plane 2 (ia|jb) - (ib|ja)                    [nvs][pvs]
__global__ void energy_prep(EnergyArgs a, float* __restrict__ vt_out, int64_t vt_stride, int pv,
                            int pvt) {
  const int g = blockIdx.y;
  const Trip tr = a.trips[g];
  float* out = vt_out + (int64_t)g * vt_stride;
  const int nvs = a.nvs, nvt = a.nvt;
  if (a.kind == SAME) {
    const int occ3[3][2] = {{tr.j, tr.k}, {tr.k, tr.i}, {tr.i, tr.j}};
    const int64_t n = 3LL * nvs * nvs;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
         idx += (int64_t)gridDim.x * blockDim.x) {
      const int y = (int)(idx % nvs);
      const int64_t r = idx / nvs;
      const int x = (int)(r % nvs);
      const int o = (int)(r / nvs);
      const int p = occ3[o][0], q = occ3[o][1];
      out[((int64_t)o * nvs + x) * pv + y] = (float)vplane_ss(a, p, x, q, y);
    }
  } else {
    const int64_t n1 = 2LL * nvs * nvt, n2 = (int64_t)nvs * nvs;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n1 + n2;
         idx += (int64_t)gridDim.x * blockDim.x) {
      if (idx < n1) {
        const int C = (int)(idx % nvt);
        const int64_t r = idx / nvt;
        const int x = (int)(r % nvs);
        const int o = (int)(r / nvs);   // 0: j, 1: i
        const int p = o == 0 ? tr.j : tr.i;
        out[((int64_t)o * nvs + x) * pvt + C] = (float)vplane_ts(a, tr.k, C, p, x);
      } else {
        const int64_t q = idx - n1;
        const int y = (int)(q % nvs), x = (int)(q / nvs);
        out[2LL * nvs * pvt + (int64_t)x * pv + y] = (float)vplane_ss(a, tr.i, x, tr.j, y);
      }
    }
  }
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// double-float a - b (both hi+lo), renormalised
__device__ __forceinline__ TwoF df_sub(TwoF a, TwoF b) {
  float s, e;
  two_sum(a.hi, -b.hi, s, e);
  e = __fadd_rn(e, __fsub_rn(a.lo, b.lo));
  const float h = __fadd_rn(s, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s))};
}

// q ~ num / D: hardware reciprocal refined by one Newton step (its error is
// then ~2^-46, i.e. the bias of the approximation is gone), times num with
// one round-to-nearest.  |D| >= 0.8 Eh here (occupied < 0 < virtual).
__device__ __forceinline__ float div_nr(float num, float D) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(D));
  const float e = __fmaf_rn(-D, r, 1.0f);
  r = __fmaf_rn(r, e, r);
  return __fmul_rn(num, r);
}

// exp(x) in float for x <= 0: Cody-Waite reduction x = k ln2 + r, |r| <= ln2/2
// (ln2 split into a 16-bit head and its tail), a degree-7 Taylor polynomial of
// exp(r) by Horner (truncation < 6e-9 relative), and 2^k by the exponent
// field.  Every step rounds to nearest, so the result carries no systematic
// bias (a library exp with an average bias of a fraction of an ulp would
// shift every Laplace factor, and the energy, by that fraction).
__device__ __forceinline__ float exp_neg(float x) {
  if (x < -87.0f) return 0.0f;
  const float k = rintf(__fmul_rn(x, 1.44269504088896341f));      // x / ln2
  const float r = __fmaf_rn(-k, 1.42860682030941723e-6f, __fmaf_rn(-k, 0.693145751953125f, x));
  float p = 1.0f / 5040.0f;
  p = __fmaf_rn(p, r, 1.0f / 720.0f);
  p = __fmaf_rn(p, r, 1.0f / 120.0f);
  p = __fmaf_rn(p, r, 1.0f / 24.0f);
  p = __fmaf_rn(p, r, 1.0f / 6.0f);
  p = __fmaf_rn(p, r, 0.5f);
  p = __fmaf_rn(p, r, 1.0f);
  p = __fmaf_rn(p, r, 1.0f);
  return __fmul_rn(p, __int_as_float(((int)k + 127) << 23));
}

// Laplace factor exp(s D) of one element (D < 0, so the argument is <= 0),
// with s carried as a float pair (s_hi + s_lo): rounding s to one float would
// shift every factor by the same relative amount, a bias; the quadrature
// weight -w is applied to the float64 partial sums instead, for the same
// reason.
__device__ __forceinline__ float lap_factor(float shi, float slo, float D) {
  return exp_neg(__fmaf_rn(shi, D, __fmul_rn(slo, D)));
}

// Energy of float32 X with register prefetch of the next cube tile.
// Work split inside a 16^3 tile: thread (c, b-pair, a-half) computes the 16
// elements a in [8h, 8h+8), b in {2p, 2p+1}, c; values that depend on a only
// (T1 amplitudes, orbital energy, V planes on (a,c)) are loaded once for both
// b.  Shared layout (pitches chosen for conflict-free vector reads):
//   T1[b][c][a] pitch 20 (float4 along a)   X[a,(bc)] / Y[a,(bC)]
//   T2[a][c][b] pitch 18 (float2 along b)   X[b,(ac)] / Y[b,(aC)]
//   T3[a][b][c] pitch 24                    X[c,(ab)] / Z'[C,(ab)]
// FU (mixed spin only): V = V(T1) + V(f_ov) in one pass; the f_ov planes sit
// vt_half floats after the T1 planes of each triplet's table and the f_ov
// coefficients come from a.fs / a.ft.
// TM (mixed spin only): Y and Z' are stored as 16^3 tiles (kOutYTile /
// kOutZTile), and the three sub-cubes come by bulk copies (16 KB each) into a
// two-stage ring in dynamic shared memory (tile i in stage i & 1, issued two
// tiles ahead by thread 0, completion on one mbarrier per stage) instead of
// through registers:
//   T1[b][c][a]  Y tile (B, C, A), 64-byte rows, 16-byte chunk q of row r at
//                chunk q ^ ((r >> 1) & 3)
//   T2[a][c][b]  Y tile (A, C, B), the same row layout
//   T3[a][b][C]  Z' tile (A, B, C), row r = a 16 + b at row r ^ ((r >> 1) & 1)
template <bool MIXED, bool FM, bool FU, bool LAP, bool TM>
__global__ void __launch_bounds__(256, 2)
energy_f32(EnergyArgs a, const float* __restrict__ X, const float* __restrict__ Z,
           const float* __restrict__ VT, int64_t vt_stride, int pv, int pvt, int64_t vt_half) {
  static_assert(!FU || (MIXED && !FM), "the fused f_ov pass is the mixed-spin W (W + V) sum");
  static_assert(!TM || (MIXED && !FU), "TMA staging: mixed spin without the fused f_ov pass");
  constexpr int P1 = 20, P2 = 18, P3 = 24;
  constexpr int FT = FU ? TB : 1, FP = FU ? TP : 1;   // f_ov table sizes (1 when absent)
  constexpr int CUBE = TB * TB * TB;                   // floats of one sub-cube
  __shared__ __align__(16) float T1[TM ? 4 : TB * TB * P1];
  __shared__ __align__(16) float T2[TM ? 4 : TB * TB * P2];
  __shared__ __align__(16) float T3[TM ? 4 : TB * TB * P3];
  extern __shared__ unsigned char dsm_raw[];
  // TM ring: stage s at ring + 3 CUBE s (T1, T2, T3), then two mbarriers
  float* const ring = reinterpret_cast<float*>(
      (reinterpret_cast<uintptr_t>(dsm_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* const fullb = reinterpret_cast<uint64_t*>(ring + 6 * CUBE);
  __shared__ __align__(16) float4 kac[TB][TB];
  __shared__ __align__(16) float4 kab[TB][TB];
  __shared__ float kbc[3][TB][TP];
  __shared__ __align__(16) float4 ad[TB];
  __shared__ float ael[TB];
  __shared__ float tb_s[3][TB], tc_s[3][TB];
  __shared__ float ebh[2][TB], ebl[2][TB];
  // f_ov planes (b,C): t^{bC}_{jK}, t^{bC}_{iK}; (a,C): t^{aC}_{jK}, t^{aC}_{iK};
  // (a,b): t^{ab}_{ij}; coefficients f_ia, f_ja / f_ib, f_jb / f_KC
  __shared__ float kbcf[2][FT][FP];
  __shared__ __align__(8) float2 kacf[FT][FT];
  __shared__ float kabf[FT][FT];
  __shared__ __align__(8) float2 adf[FT];
  __shared__ float tbf_s[2][FT], tcf_s[FT];

  // Persistent item loop: item w = g * P + chunk (P = a.nchunk) covers the
  // tiles chunk, chunk + P, ... of triplet g; CTA b takes items b, b + grid,
  // ...  Each item's sum is formed in a fixed order and written as one
  // float64 partial per warp, so results do not depend on the grid size.
  const int P = a.nchunk;
  int w = blockIdx.x;
  if (w >= a.nitems) return;
  int g = w / P;
  const int tid = threadIdx.x;
  const int r1 = tid / TB, r2 = tid % TB;           // row owned in the fetch phase
  const int lane = tid & 31, wid = tid >> 5;
  const int cl = lane & 15;                          // compute phase: c
  const int bl0 = 2 * (((wid & 3) << 1) | (lane >> 4));   // first of the b pair
  const int al0 = 8 * (wid >> 2);                    // a half
  const int nvs = a.nvs, nvt = a.nvt;
  auto occ_sum = [&](int gg) {
    const Trip t = a.trips[gg];
    return split_df(MIXED ? a.eps_s[t.i] + a.eps_s[t.j] + a.eps_t[t.k]
                          : a.eps_s[t.i] + a.eps_s[t.j] + a.eps_s[t.k]);
  };
  TwoF eocc = occ_sum(g);
  const float lshi = (float)a.lap_s;                          // Laplace s (LAP only)
  const float lslo = (float)(a.lap_s - (double)lshi);

  float4 xr[3][4];
  uint32_t okm = 0;
  float vr[9];
  float t1r[3];
  float vrf[FU ? 5 : 1];
  float f1r[2];
  TwoF er;

  // Fetch of a tile's three X sub-cubes, coalesced: in round u thread t loads
  // the 16-byte chunk (t & 3) of sub-cube row R = 64 u + (t >> 2), so four
  // neighbouring lanes read one 64-byte row and a warp reads 8 whole rows per
  // load instruction.  okm bit (3 u + cube) marks the valid rows.
  int3 blkf;   // cube tile of the last fetch (prefetched with its data)
  auto fetch = [&](int gq, int q) {
    const Trip tr = a.trips[gq];
    const float* Xg = X + (int64_t)gq * a.x_stride;
    const float* Zg = MIXED ? Z + (int64_t)gq * a.z_stride : nullptr;
    const float* Vg = VT + (int64_t)gq * vt_stride;
    const float* Vf = Vg + vt_half;
    (void)Zg;
    (void)Vf;
    const int3 blk = a.blocks[q];
    blkf = blk;
    const int a0 = blk.x * TB, b0 = blk.y * TB, c0 = blk.z * TB;
    const int ch = (tid & 3) * 4;
    okm = 0;
#pragma unroll
    for (int u = 0; u < (TM ? 0 : 4); ++u) {
      const int R = 64 * u + (tid >> 2);
      const int s1 = R >> 4, s2 = R & 15;
      const float4* p1 = nullptr;
      const float4* p2 = nullptr;
      const float4* p3 = nullptr;
      bool k1, k2, k3;
      if (!MIXED) {
        int b = b0 + s1, c = c0 + s2;
        k1 = b < c && c < nvs;
        if (k1) p1 = reinterpret_cast<const float4*>(Xg + pair_index(b, c) * a.pitch_x + a0 + ch);
        int aa = a0 + s1;
        k2 = aa < c && c < nvs;
        if (k2) p2 = reinterpret_cast<const float4*>(Xg + pair_index(aa, c) * a.pitch_x + b0 + ch);
        b = b0 + s2;
        k3 = aa < b && b < nvs;
        if (k3) p3 = reinterpret_cast<const float4*>(Xg + pair_index(aa, b) * a.pitch_x + c0 + ch);
      } else {
        int b = b0 + s1, c = c0 + s2;
        k1 = b < nvs && c < nvt;
        if (k1)
          p1 = reinterpret_cast<const float4*>(Xg + ((int64_t)b * nvt + c) * a.pitch_x + a0 + ch);
        int aa = a0 + s1;
        k2 = aa < nvs && c < nvt;
        if (k2)
          p2 = reinterpret_cast<const float4*>(Xg + ((int64_t)aa * nvt + c) * a.pitch_x + b0 + ch);
        b = b0 + s2;
        k3 = aa < b && b < nvs;
        if (k3) p3 = reinterpret_cast<const float4*>(Zg + pair_index(aa, b) * a.pitch_z + c0 + ch);
      }
      if (k1) xr[0][u] = __ldg(p1);
      if (k2) xr[1][u] = __ldg(p2);
      if (k3) xr[2][u] = __ldg(p3);
      okm |= (k1 ? 1u : 0u) << (3 * u) | (k2 ? 2u : 0u) << (3 * u) | (k3 ? 4u : 0u) << (3 * u);
    }
    if (!MIXED) {
      const int rows[3] = {b0, a0, a0}, cols[3] = {c0, c0, b0};
#pragma unroll
      for (int pl = 0; pl < 3; ++pl) {
        const int x = rows[pl] + r1, y = cols[pl] + r2;
        const bool in = x < nvs && y < nvs;
#pragma unroll
        for (int o = 0; o < 3; ++o)
          vr[pl * 3 + o] = in ? __ldg(Vg + ((int64_t)o * nvs + x) * pv + y) : 0.f;
      }
    } else {
      const int rows[2] = {b0, a0};
#pragma unroll
      for (int pl = 0; pl < 2; ++pl) {
        const int x = rows[pl] + r1, y = c0 + r2;
        const bool in = x < nvs && y < nvt;
#pragma unroll
        for (int o = 0; o < 2; ++o)
          vr[pl * 2 + o] = in ? __ldg(Vg + ((int64_t)o * nvs + x) * pvt + y) : 0.f;
      }
      const int x = a0 + r1, y = b0 + r2;
      vr[4] = (x < nvs && y < nvs) ? __ldg(Vg + 2LL * nvs * pvt + (int64_t)x * pv + y) : 0.f;
      if constexpr (FU) {   // the same positions of the f_ov planes
#pragma unroll
        for (int pl = 0; pl < 2; ++pl) {
          const int xx = rows[pl] + r1, yy = c0 + r2;
          const bool in = xx < nvs && yy < nvt;
#pragma unroll
          for (int o = 0; o < 2; ++o)
            vrf[pl * 2 + o] = in ? __ldg(Vf + ((int64_t)o * nvs + xx) * pvt + yy) : 0.f;
        }
        vrf[4] = (x < nvs && y < nvs) ? __ldg(Vf + 2LL * nvs * pvt + (int64_t)x * pv + y) : 0.f;
      }
    }
    if (tid < 3 * TB) {
      const int bl = tid / TB, l = tid % TB;
      const int base = bl == 0 ? a0 : (bl == 1 ? b0 : c0);
      const int x = base + l;
      const bool tblock = MIXED && bl == 2;
      const int nv = tblock ? nvt : nvs;
      if (!MIXED) {
        const int occ[3] = {tr.i, tr.j, tr.k};
#pragma unroll
        for (int o = 0; o < 3; ++o) t1r[o] = x < nvs ? (float)a.t1s[(int64_t)occ[o] * nvs + x] : 0.f;
      } else if (!tblock) {
        t1r[0] = x < nvs ? (float)a.t1s[(int64_t)tr.i * nvs + x] : 0.f;
        t1r[1] = x < nvs ? (float)a.t1s[(int64_t)tr.j * nvs + x] : 0.f;
        t1r[2] = 0.f;
        if constexpr (FU) {
          f1r[0] = x < nvs ? (float)a.fs[(int64_t)tr.i * nvs + x] : 0.f;
          f1r[1] = x < nvs ? (float)a.fs[(int64_t)tr.j * nvs + x] : 0.f;
        }
      } else {
        t1r[0] = x < nvt ? (float)a.t1t[(int64_t)tr.k * nvt + x] : 0.f;
        t1r[1] = t1r[2] = 0.f;
        if constexpr (FU) {
          f1r[0] = x < nvt ? (float)a.ft[(int64_t)tr.k * nvt + x] : 0.f;
          f1r[1] = 0.f;
        }
      }
      const double* e = tblock ? a.eps_t : a.eps_s;
      const int no = tblock ? a.not_ : a.nos;
      er = split_df(x < nv ? e[no + x] : 0.0);
    }
  };

  TwoF acc = {0.f, 0.f};
  int q = w - g * P;
  // TM: the producer cursor (pw, pg, pq) runs two tiles ahead of (w, g, q)
  auto advance = [&](int& cw, int& cg, int& cq) {
    cq += P;
    if (cq >= a.nblocks) {
      cw += (int)gridDim.x;
      cg = cw / P;
      cq = cw - cg * P;
    }
  };
  auto issue = [&](int cg, int cq, int st) {
    if (a.starve) return;   // test hook: nothing will complete the stage barrier
    const int3 bk = a.blocks[cq];
    const int nbs = (nvs + TB - 1) / TB, nbt = (nvt + TB - 1) / TB;
    const float* Yg = X + (int64_t)cg * a.x_stride;
    const float* Zt = Z + (int64_t)cg * a.z_stride;
    const uint32_t bar = smem_u32(fullb + st);
    float* base = ring + 3 * CUBE * st;
    mbar_expect_tx(bar, 3u * CUBE * 4u);
    bulk_load(smem_u32(base), Yg + ((int64_t)(bk.y * nbt + bk.z) * nbs + bk.x) * CUBE,
              CUBE * 4u, bar);
    bulk_load(smem_u32(base + CUBE), Yg + ((int64_t)(bk.x * nbt + bk.z) * nbs + bk.y) * CUBE,
              CUBE * 4u, bar);
    bulk_load(smem_u32(base + 2 * CUBE),
              Zt + ((int64_t)(bk.y * (bk.y + 1) / 2 + bk.x) * nbt + bk.z) * CUBE, CUBE * 4u, bar);
  };
  int pw = w, pg = g, pq = q, issued = 0;
  uint32_t it = 0;   // tiles of this CTA so far
  const float* cur = ring;
  if constexpr (TM) {
    if (tid == 0) {
      mbar_init(smem_u32(fullb), 1);
      mbar_init(smem_u32(fullb + 1), 1);
      mbar_init_fence();
    }
    __syncthreads();
#pragma unroll 1
    for (int st = 0; st < 2 && pw < a.nitems; ++st) {
      if (tid == 0) issue(pg, pq, st);
      issued += a.starve ? 0 : 1;
      advance(pw, pg, pq);
    }
  }
  fetch(g, q);
  for (;;) {
    const int3 blk = blkf;
    const int a0 = blk.x * TB, b0 = blk.y * TB, c0 = blk.z * TB;
    if constexpr (TM) {   // this tile's sub-cubes
      const int st = (int)(it & 1u);
      const bool ok = mbar_wait_bounded(smem_u32(fullb + st), (it >> 1) & 1u,
                                        a.wait_cycles > 0 ? a.wait_cycles : 4000000000LL);
      if (__syncthreads_or(!ok)) {
        // give up: record the error, let the copies in flight land, leave
        if (tid == 0) {
          atomicCAS(a.flag, 0, 7);
          for (uint32_t j = it; j < (uint32_t)issued; ++j)
            mbar_wait_bounded(smem_u32(fullb + (j & 1u)), (j >> 1) & 1u, 4000000000LL);
        }
        __syncthreads();
        return;
      }
      cur = ring + 3 * CUBE * st;
    }
    // ---- registers -> shared ----
    {
      const int ch = (tid & 3) * 4;
#pragma unroll
      for (int u = 0; u < (TM ? 0 : 4); ++u) {
        const int R = 64 * u + (tid >> 2);
        if (okm & (1u << (3 * u))) *reinterpret_cast<float4*>(T1 + R * P1 + ch) = xr[0][u];
        if (okm & (2u << (3 * u))) {
          float2* d2 = reinterpret_cast<float2*>(T2 + R * P2 + ch);
          d2[0] = make_float2(xr[1][u].x, xr[1][u].y);
          d2[1] = make_float2(xr[1][u].z, xr[1][u].w);
        }
        if (okm & (4u << (3 * u))) *reinterpret_cast<float4*>(T3 + R * P3 + ch) = xr[2][u];
      }
      if (!MIXED) {
        kbc[0][r1][r2] = vr[0]; kbc[1][r1][r2] = vr[1]; kbc[2][r1][r2] = vr[2];
        kac[r1][r2] = make_float4(vr[3], vr[4], vr[5], 0.f);
        kab[r1][r2] = make_float4(vr[6], vr[7], vr[8], 0.f);
      } else {
        kbc[0][r1][r2] = vr[0]; kbc[1][r1][r2] = vr[1];
        kac[r1][r2] = make_float4(vr[2], vr[3], 0.f, 0.f);
        kab[r1][r2] = make_float4(vr[4], 0.f, 0.f, 0.f);
        if constexpr (FU) {
          kbcf[0][r1][r2] = vrf[0]; kbcf[1][r1][r2] = vrf[1];
          kacf[r1][r2] = make_float2(vrf[2], vrf[3]);
          kabf[r1][r2] = vrf[4];
        }
      }
      if (tid < 3 * TB) {
        const int bl = tid / TB, l = tid % TB;
        if (bl == 0) {
          ad[l] = make_float4(t1r[0], t1r[1], t1r[2], er.hi);
          ael[l] = er.lo;
          if constexpr (FU) adf[l] = make_float2(f1r[0], f1r[1]);
        } else {
          float* tt = bl == 1 ? &tb_s[0][0] : &tc_s[0][0];
          tt[l] = t1r[0]; tt[TB + l] = t1r[1]; tt[2 * TB + l] = t1r[2];
          ebh[bl - 1][l] = er.hi;
          ebl[bl - 1][l] = er.lo;
          if constexpr (FU) {
            if (bl == 1) {
              tbf_s[0][l] = f1r[0]; tbf_s[1][l] = f1r[1];
            } else {
              tcf_s[l] = f1r[0];
            }
          }
        }
      }
    }
    __syncthreads();
    // next tile (of this item, else the first of the CTA's next item) in flight
    int wn = w, gn = g, qn = q + P;
    if (qn >= a.nblocks) {
      wn = w + (int)gridDim.x;
      gn = wn / P;
      qn = wn - gn * P;
    }
    const bool more = wn < a.nitems;
    if (more) fetch(gn, qn);
    // ---- elements: (a in half, b pair, c) ----------------------------------
    {
      const int c = c0 + cl;
      float part = 0.f;
      bool rowok[2];
      TwoF dbc[2];
      float k0[2], k1[2], k2[2], tb0[2], tb1[2], tb2[2];
      float kf0[2] = {0.f, 0.f}, kf1[2] = {0.f, 0.f}, tbf0[2] = {0.f, 0.f}, tbf1[2] = {0.f, 0.f};
#pragma unroll
      for (int sb = 0; sb < 2; ++sb) {
        const int bl = bl0 + sb, b = b0 + bl;
        rowok[sb] = MIXED ? (b < nvs && c < nvt) : (b < c && c < nvs);
        dbc[sb] = df_sub(df_sub(eocc, TwoF{ebh[0][bl], ebl[0][bl]}), TwoF{ebh[1][cl], ebl[1][cl]});
        k0[sb] = kbc[0][bl][cl]; k1[sb] = kbc[1][bl][cl]; k2[sb] = kbc[2][bl][cl];
        tb0[sb] = tb_s[0][bl]; tb1[sb] = tb_s[1][bl]; tb2[sb] = tb_s[2][bl];
        if constexpr (FU) {
          kf0[sb] = kbcf[0][bl][cl]; kf1[sb] = kbcf[1][bl][cl];
          tbf0[sb] = tbf_s[0][bl]; tbf1[sb] = tbf_s[1][bl];
        }
      }
      const float tc0 = tc_s[0][cl], tc1 = tc_s[1][cl], tc2 = tc_s[2][cl];
      const float tcf0 = FU ? tcf_s[cl] : 0.f;
      // last a (exclusive) any element of this thread can use: a < b <= b0+bl0+1
      const int aend = min(al0 + 8, b0 + bl0 + 1 - a0);
      if ((rowok[0] || rowok[1]) && aend > al0) {
        const float* x1r0 = T1 + ((bl0 + 0) * TB + cl) * P1;
        const float* x1r1 = T1 + ((bl0 + 1) * TB + cl) * P1;
        if constexpr (MIXED) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          // mixed spin: all 8 x 2 elements are evaluated and masked with a
          // select (a < b also bounds a by aend), so the independent element
          // chains interleave; the same-spin tiles keep the branches (more of
          // their elements are masked on the diagonal blocks)
          const int a4 = al0 + 4 * h;
          float4 q0, q1;
          if constexpr (TM) {   // swizzled 64-byte rows (b, c) of T1
            const int ra = bl0 * TB + cl, rb = ra + TB;
            q0 = *reinterpret_cast<const float4*>(cur + ra * TB + (((a4 >> 2) ^ ((ra >> 1) & 3)) << 2));
            q1 = *reinterpret_cast<const float4*>(cur + rb * TB + (((a4 >> 2) ^ ((rb >> 1) & 3)) << 2));
          } else {
            q0 = *reinterpret_cast<const float4*>(x1r0 + a4);
            q1 = *reinterpret_cast<const float4*>(x1r1 + a4);
          }
          const float x1a[2][4] = {{q0.x, q0.y, q0.z, q0.w}, {q1.x, q1.y, q1.z, q1.w}};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int al = a4 + u;
            const float4 da = ad[al];
            const float del = ael[al];
            float2 x2;
            if constexpr (TM) {   // swizzled 64-byte rows (a, c) of T2
              const int r = al * TB + cl;
              x2 = *reinterpret_cast<const float2*>(
                  cur + CUBE + r * TB + ((((bl0 >> 2) ^ ((r >> 1) & 3)) << 2) | (bl0 & 3)));
            } else {
              x2 = *reinterpret_cast<const float2*>(T2 + (al * TB + cl) * P2 + bl0);
            }
            const float4 vac = kac[al][cl];
            const float x2a[2] = {x2.x, x2.y};
            float2 daf = make_float2(0.f, 0.f), vacf = make_float2(0.f, 0.f);
            if constexpr (FU) {
              daf = adf[al];
              vacf = kacf[al][cl];
            }
#pragma unroll
            for (int sb = 0; sb < 2; ++sb) {
              const int bl = bl0 + sb;
              const bool valid = rowok[sb] && a0 + al < b0 + bl;
              const int r3 = al * TB + bl;
              const float x3 = TM ? cur[2 * CUBE + (r3 ^ ((r3 >> 1) & 1)) * TB + cl]
                                  : T3[(al * TB + bl) * P3 + cl];
              const float vab = kab[al][bl].x;
              const float w = x1a[sb][u] - x2a[sb] + x3;
              float v = da.x * k0[sb] - da.y * k1[sb] - tb0[sb] * vac.x +
                        tb1[sb] * vac.y + tc0 * vab;
              if constexpr (FU)   // the f_ov term: f for t1, the doubles for the integrals
                v += daf.x * kf0[sb] - daf.y * kf1[sb] - tbf0[sb] * vacf.x +
                     tbf1[sb] * vacf.y + tcf0 * kabf[al][bl];
              const float num = FM ? __fmul_rn(w, v) : __fmul_rn(w, __fadd_rn(w, v));
              float s, e;
              two_sum(dbc[sb].hi, -da.w, s, e);
              const float D = __fadd_rn(s, __fadd_rn(e, __fsub_rn(dbc[sb].lo, del)));
              const float qv = LAP ? __fmul_rn(num, lap_factor(lshi, lslo, D)) : div_nr(num, D);
              part = __fadd_rn(part, valid ? qv : 0.f);
            }
          }
        }
        } else {
        for (int a4 = al0; a4 < aend; a4 += 4) {
          const float4 q0 = *reinterpret_cast<const float4*>(x1r0 + a4);
          const float4 q1 = *reinterpret_cast<const float4*>(x1r1 + a4);
          const float x1a[2][4] = {{q0.x, q0.y, q0.z, q0.w}, {q1.x, q1.y, q1.z, q1.w}};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int al = a4 + u;
            if (al < aend) {
              const float4 da = ad[al];
              const float del = ael[al];
              const float2 x2 = *reinterpret_cast<const float2*>(T2 + (al * TB + cl) * P2 + bl0);
              const float4 vac = kac[al][cl];
              const float x2a[2] = {x2.x, x2.y};
#pragma unroll
              for (int sb = 0; sb < 2; ++sb) {
                const int bl = bl0 + sb;
                if (rowok[sb] && a0 + al < b0 + bl) {
                  const float x3 = T3[(al * TB + bl) * P3 + cl];
                  const float4 vab = kab[al][bl];
                  const float w = x1a[sb][u] - x2a[sb] + x3;
                  float v;
                  if (!MIXED) {
                    const float ya = da.x * k0[sb] + da.y * k1[sb] + da.z * k2[sb];
                    const float yb = tb0[sb] * vac.x + tb1[sb] * vac.y + tb2[sb] * vac.z;
                    const float yc = tc0 * vab.x + tc1 * vab.y + tc2 * vab.z;
                    v = ya - yb + yc;
                  } else {
                    v = da.x * k0[sb] - da.y * k1[sb] - tb0[sb] * vac.x + tb1[sb] * vac.y +
                        tc0 * vab.x;
                  }
                  const float num = FM ? __fmul_rn(w, v) : __fmul_rn(w, __fadd_rn(w, v));
                  float s, e;
                  two_sum(dbc[sb].hi, -da.w, s, e);
                  const float D = __fadd_rn(s, __fadd_rn(e, __fsub_rn(dbc[sb].lo, del)));
                  part = __fadd_rn(part, LAP ? __fmul_rn(num, lap_factor(lshi, lslo, D))
                                             : div_nr(num, D));
                }
              }
            }
          }
        }
        }
        float s, e;
        two_sum(acc.hi, part, s, e);
        acc = {s, __fadd_rn(acc.lo, e)};
      }
      (void)tc1;
      (void)tc2;
    }
    __syncthreads();
    if constexpr (TM) {   // stage it & 1 is free: the tile two ahead goes there
      if (pw < a.nitems) {
        if (tid == 0) issue(pg, pq, (int)(it & 1u));
        issued += a.starve ? 0 : 1;
        advance(pw, pg, pq);
      }
      ++it;
    }
    if (wn != w) {   // item (g, w - g P) complete: one float64 partial per warp
      double dacc = (double)acc.hi + (double)acc.lo;
      for (int off = 16; off > 0; off >>= 1) dacc += __shfl_down_sync(0xffffffffu, dacc, off);
      if (lane == 0) a.partial[((int64_t)w * 8) + wid] = LAP ? -a.lap_w * dacc : dacc;
      acc = {0.f, 0.f};
      if (!more) break;
      w = wn;
      if (gn != g) eocc = occ_sum(gn);
      g = gn;
    }
    q = qn;
  }
}

// A Neumaier pair (sum, compensation).
struct Nsum {
  double s, c;
  __device__ __forceinline__ void add(double x) {
    const double t = s + x;
    c += fabs(s) >= fabs(x) ? (s - t) + x : (x - t) + s;
    s = t;
  }
  __device__ __forceinline__ void add(const Nsum& o) {
    add(o.s);
    c += o.c;
  }
};

// Sum of the block's pairs (256 threads), in a fixed order: a shuffle tree per warp,
// then the eight warps in turn; valid in thread 0.
__device__ __forceinline__ Nsum block_sum(Nsum v) {
  __shared__ double ws[8], wc[8];
  for (int off = 16; off > 0; off >>= 1) {
    Nsum o;
    o.s = __shfl_down_sync(0xffffffffu, v.s, off);
    o.c = __shfl_down_sync(0xffffffffu, v.c, off);
    v.add(o);
  }
  __syncthreads();   // the shared arrays may hold an earlier sum
  if ((threadIdx.x & 31) == 0) {
    ws[threadIdx.x >> 5] = v.s;
    wc[threadIdx.x >> 5] = v.c;
  }
  __syncthreads();
  Nsum t{0.0, 0.0};
  if (threadIdx.x == 0)
    for (int w = 0; w < 8; ++w) t.add(Nsum{ws[w], wc[w]});
  return t;
}

// e_trip[g] = sum_p partial[g][p] (+ sum_p partial2[g][p] when given): one CTA per
// triplet, thread t sums p = t, t + 256, ... (Neumaier), combined in a fixed
// order, so the result does not depend on timing.  (One warp per triplet took
// 22 us for 64 triplets of 1200 partials, this 4.)
__global__ void __launch_bounds__(256)
reduce_partials(const double* __restrict__ partial, int np, const double* __restrict__ partial2,
                double* __restrict__ e_trip) {
  const int g = blockIdx.x;
  Nsum v{0.0, 0.0};
  for (int half = 0; half < (partial2 ? 2 : 1); ++half) {
    const double* src = (half ? partial2 : partial) + (int64_t)g * np;
    for (int p = threadIdx.x; p < np; p += 256) v.add(src[p]);
  }
  v = block_sum(v);
  if (threadIdx.x == 0) e_trip[g] = v.s + v.c;
}

// Orbital contributions of eq cim_pt_energy from per-triplet contributions:
// same-spin triplet 1/3 to each of its orbitals; mixed triplet 1/4 to each of
// its two same-spin orbitals and 1/2 to the third (A.thirds: 1/3 each, the
// partition of eq local_pt).  One CTA per occupied
// orbital (spin up first), fixed-order Neumaier sums: bitwise reproducible.
__global__ void __launch_bounds__(256) orbital_partition(OrbPartArgs A) {
  const int b = blockIdx.x;
  const int s = b < A.na ? 0 : 1;
  const int p = s == 0 ? b : b - A.na;
  Nsum v{0.0, 0.0};
  auto add = [&](double x) { v.add(x); };
  for (int c = 0; c < 4; ++c) {
    const Trip* tr = A.trips[c];
    const double* e = A.e[c];
    // case c: 0 aaa, 1 aab (i,j up; K down), 2 abb (I,J down; k up), 3 bbb
    const int pair_spin = (c == 0 || c == 1) ? 0 : 1;
    const bool same = c == 0 || c == 3;
    for (int64_t q = threadIdx.x; q < A.n[c]; q += blockDim.x) {
      const Trip t = tr[q];
      if (same) {
        if (s == pair_spin && (t.i == p || t.j == p || t.k == p)) add(e[q] / 3.0);
      } else if (s == pair_spin) {
        if (t.i == p || t.j == p) add(A.thirds ? e[q] / 3.0 : e[q] * 0.25);
      } else if (t.k == p) {
        add(A.thirds ? e[q] / 3.0 : e[q] * 0.5);
      }
    }
  }
  v = block_sum(v);
  double* out = s == 0 ? A.out[0] : A.out[1];
  if (threadIdx.x == 0 && out) out[p] = v.s + v.c;
}

// Per-case Neumaier sums (fixed order) and the caller's copies of the per-triplet
// values: one CTA per case, one launch per call.  (Adding the 256 threads' pairs
// one after the other took 73 us a case, this 7 for all.)
__global__ void __launch_bounds__(256) case_sums(CaseSums A) {
  const int c = blockIdx.x;
  const double* e = A.e[c];
  Nsum v{0.0, 0.0};
  for (int64_t q = threadIdx.x; q < A.n[c]; q += 256) {
    const double x = e[q];
    v.add(x);
    if (A.copy[c]) A.copy[c][q] = x;
  }
  v = block_sum(v);
  if (threadIdx.x == 0) A.out[c] = v.s + v.c;
}

}  // namespace

size_t energy_smem_bytes(bool f64) { return 3 * TB * TB * TP * (f64 ? 8 : 4); }

// Dynamic shared memory of the TMA-staged variant: two stages of three
// sub-cubes, two mbarriers, 1024 bytes of alignment slack.
constexpr int kRingBytes = 6 * TB * TB * TB * 4 + 16 + 1024;

// Resident CTAs per SM of one energy_f32 variant (queried once).
template <bool M, bool F, bool U, bool L, bool T>
int ef32_resident() {
  static int occ = 0;
  if (occ == 0) {
    int n = 0;
    auto k = energy_f32<M, F, U, L, T>;
    if (T) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, 256, T ? kRingBytes : 0) !=
        cudaSuccess)
      n = 1;
    occ = n > 0 ? n : 1;
  }
  return occ;
}

template <bool M, bool F, bool U, bool L, bool T>
void launch_ef32(EnergyArgs a, const float* X, const float* Z, const float* vtab,
                 int64_t vt_stride, int pv, int pvt, int64_t vt_half, int ntrip, int nchunks,
                 cudaStream_t st) {
  a.nchunk = nchunks;
  a.nitems = ntrip * nchunks;
  const int grid = std::max(1, std::min(a.nitems, ef32_resident<M, F, U, L, T>() * a.nsm));
  energy_f32<M, F, U, L, T><<<grid, 256, T ? kRingBytes : 0, st>>>(a, X, Z, vtab, vt_stride, pv,
                                                                   pvt, vt_half);
}

// float32-X path: V-table prep + energy (nchunks items per triplet on a
// persistent grid; partial holds 8 values per item).
cudaError_t launch_energy_f32(const EnergyArgs& a, const float* X, const float* Z, float* vtab,
                              int64_t vt_stride, int pv, int pvt, int ntrip, int nchunks,
                              cudaStream_t st) {
  if (ntrip <= 0) return cudaSuccess;
  if (nchunks < 1 || nchunks > a.nblocks || a.nsm < 1) return cudaErrorInvalidValue;
  dim3 gp(64, ntrip);
  energy_prep<<<gp, 256, 0, st>>>(a, vtab, vt_stride, pv, pvt);
#define LNO_EF32(M, F, L) \
  launch_ef32<M, F, false, L, false>(a, X, Z, vtab, vt_stride, pv, pvt, 0, ntrip, nchunks, st)
  const bool lap = a.lap_w != 0.0;
  if (a.kind == SAME) {
    if (a.vmode) {
      if (lap) LNO_EF32(false, true, true); else LNO_EF32(false, true, false);
    } else {
      if (lap) LNO_EF32(false, false, true); else LNO_EF32(false, false, false);
    }
  } else if (a.vmode) {
    if (lap) LNO_EF32(true, true, true); else LNO_EF32(true, true, false);
  } else if (!a.tiled) {
    if (lap) LNO_EF32(true, false, true); else LNO_EF32(true, false, false);
  } else {
    // mixed spin, tiled Y / Z': sub-cubes staged by bulk copies
    if (a.flag == nullptr || (reinterpret_cast<uintptr_t>(X) & 15) ||
        (reinterpret_cast<uintptr_t>(Z) & 15))
      return cudaErrorInvalidValue;
    if (lap)
      launch_ef32<true, false, false, true, true>(a, X, Z, vtab, vt_stride, pv, pvt, 0, ntrip,
                                                  nchunks, st);
    else
      launch_ef32<true, false, false, false, true>(a, X, Z, vtab, vt_stride, pv, pvt, 0, ntrip,
                                                   nchunks, st);
  }
#undef LNO_EF32
  return cudaGetLastError();
}

template <typename T, bool MIXED, bool FM>
cudaError_t launch_group(const EnergyArgs& a, const void* X, const void* Z, dim3 grid, size_t sm,
                         cudaStream_t st) {
  auto k = energy_group<T, MIXED, FM>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k<<<grid, 256, sm, st>>>(a, (const T*)X, (const T*)Z);
  return cudaGetLastError();
}

// Mixed spin with the f_ov term in one pass: T1 planes in [0, vt_half) and
// f_ov planes in [vt_half, 2 vt_half) of each triplet's table (stride
// 2 vt_half); a.t1s/t1t and a.fs/ft the two coefficient sets.
cudaError_t launch_energy_f32_fused(const EnergyArgs& a, const float* X, const float* Z,
                                   float* vtab, int64_t vt_half, int pv, int pvt, int ntrip,
                                   int nchunks, cudaStream_t st) {
  if (ntrip <= 0) return cudaSuccess;
  if (a.kind == SAME) return cudaErrorInvalidValue;
  if (nchunks < 1 || nchunks > a.nblocks || a.nsm < 1) return cudaErrorInvalidValue;
  dim3 gp(64, ntrip);
  EnergyArgs a0 = a, a1 = a;
  a0.vmode = 0;
  a1.vmode = 1;
  energy_prep<<<gp, 256, 0, st>>>(a0, vtab, 2 * vt_half, pv, pvt);
  energy_prep<<<gp, 256, 0, st>>>(a1, vtab + vt_half, 2 * vt_half, pv, pvt);
  if (a.tiled) return cudaErrorInvalidValue;   // the fused f_ov pass reads [pair][a] rows
  if (a.lap_w != 0.0)
    launch_ef32<true, false, true, true, false>(a0, X, Z, vtab, 2 * vt_half, pv, pvt, vt_half,
                                                ntrip, nchunks, st);
  else
    launch_ef32<true, false, true, false, false>(a0, X, Z, vtab, 2 * vt_half, pv, pvt, vt_half,
                                                 ntrip, nchunks, st);
  return cudaGetLastError();
}

cudaError_t launch_energy(const EnergyArgs& a, const void* X, const void* Z, bool f64,
                          int ntrip, int nchunks, cudaStream_t st) {
  if (ntrip <= 0) return cudaSuccess;
  dim3 grid(nchunks, ntrip);
  const size_t sm = energy_smem_bytes(f64);
  const bool mixed = a.kind != SAME, fm = a.vmode != 0;
  if (f64) {
    if (!mixed) return fm ? launch_group<double, false, true>(a, X, Z, grid, sm, st)
                          : launch_group<double, false, false>(a, X, Z, grid, sm, st);
    return fm ? launch_group<double, true, true>(a, X, Z, grid, sm, st)
              : launch_group<double, true, false>(a, X, Z, grid, sm, st);
  }
  if (!mixed) return fm ? launch_group<float, false, true>(a, X, Z, grid, sm, st)
                        : launch_group<float, false, false>(a, X, Z, grid, sm, st);
  return fm ? launch_group<float, true, true>(a, X, Z, grid, sm, st)
            : launch_group<float, true, false>(a, X, Z, grid, sm, st);
}

cudaError_t launch_reduce_partials(const double* partial, int np, const double* partial2,
                                   int ntrip, double* e_trip, cudaStream_t st) {
  if (ntrip <= 0) return cudaSuccess;
  reduce_partials<<<ntrip, 256, 0, st>>>(partial, np, partial2, e_trip);
  return cudaGetLastError();
}

cudaError_t launch_orbital_partition(const OrbPartArgs& A, cudaStream_t st) {
  if (A.na + A.nb <= 0) return cudaSuccess;
  orbital_partition<<<A.na + A.nb, 256, 0, st>>>(A);
  return cudaGetLastError();
}

// Bounded-wait check of the TMA-staged energy kernel: one mixed-spin 16^3
// tile of zeros (two occupied, 16 virtual orbitals per spin) with the test hook
// that issues no copy, so the first stage wait can only end by its limit.
// *code gets the kernel's flag (7 when the wait gave up).
cudaError_t energy_timeout_selftest(long long wait_cycles, int nsm, int* code, cudaStream_t st) {
  constexpr int nv = 16, no = 2, pitch = 16;
  const int64_t xs = kTile, zs = kTile;   // one Y tile and one Z' tile
  const int64_t vts = 2LL * nv * pitch + (int64_t)nv * pitch;
  const size_t bytes = (size_t)(xs + zs + vts) * 4 + 4 * (no + nv) * 8 + 2 * no * nv * 8 +
                       8 * 8 + 64 + 4 * 256;
  unsigned char* buf = nullptr;
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&buf), bytes, st);
  if (e != cudaSuccess) return e;
  auto finish = [&](cudaError_t r) {
    cudaFreeAsync(buf, st);
    return r;
  };
  if ((e = cudaMemsetAsync(buf, 0, bytes, st)) != cudaSuccess) return finish(e);
  unsigned char* p = buf;
  auto take = [&](size_t n) {
    unsigned char* q = p;
    p += (n + 255) / 256 * 256;
    return q;
  };
  float* X = reinterpret_cast<float*>(take(xs * 4));
  float* Z = reinterpret_cast<float*>(take(zs * 4));
  float* VT = reinterpret_cast<float*>(take(vts * 4));
  double* eps = reinterpret_cast<double*>(take(2 * (no + nv) * 8));
  double* t1 = reinterpret_cast<double*>(take(2 * no * nv * 8));
  double* part = reinterpret_cast<double*>(take(8 * 8));
  int* flag = reinterpret_cast<int*>(take(64));
  int3* blk = reinterpret_cast<int3*>(take(16));
  Trip* trip = reinterpret_cast<Trip*>(take(16));
  const int3 hb = make_int3(0, 0, 0);
  const Trip ht{0, 1, 0};
  if ((e = cudaMemcpyAsync(blk, &hb, sizeof hb, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
      (e = cudaMemcpyAsync(trip, &ht, sizeof ht, cudaMemcpyHostToDevice, st)) != cudaSuccess)
    return finish(e);
  EnergyArgs a{};
  a.kind = MIXED;
  a.nvs = a.nvt = nv;
  a.nos = a.not_ = no;
  a.eps_s = eps;
  a.eps_t = eps + no + nv;
  a.t1s = t1;
  a.t1t = t1 + no * nv;
  a.blocks = blk;
  a.nblocks = 1;
  a.pitch_x = a.pitch_z = pitch;
  a.x_stride = xs;
  a.z_stride = zs;
  a.trips = trip;
  a.partial = part;
  a.nsm = nsm;
  a.flag = flag;
  a.wait_cycles = wait_cycles;
  a.starve = 1;
  a.tiled = 1;
  launch_ef32<true, false, false, false, true>(a, X, Z, VT, vts, pitch, pitch, 0, 1, 1, st);
  if ((e = cudaGetLastError()) != cudaSuccess) return finish(e);
  int h = 0;
  if ((e = cudaMemcpyAsync(&h, flag, sizeof h, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
    return finish(e);
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return finish(e);
  *code = h;
  return finish(cudaSuccess);
}

cudaError_t launch_case_sums(const CaseSums& A, cudaStream_t st) {
  case_sums<<<4, 256, 0, st>>>(A);
  return cudaGetLastError();
}

}  // namespace lno
