// Layout kernels: DF factor blocks and the K-concatenated operands of the
// per-triplet W contractions (eq cim_pt_energy, connected triples).
//
// Same spin s (o occupied, v virtual, Kx = v + o):
//   AT[p][q][a][kk] = t^{ae}_{pq}            (kk = e < v)
//                   = <ma||qp> = H_qp[m][a]  (kk = v + m), H_xy[m][a] = (mx|ay)-(my|ax)
//   BT[x][(b<c)][kk] = <ex||bc> = (eb|xc)-(ec|xb)   (kk = e)
//                    = t^{bc}_{xm}                   (kk = v + m)
//   X_{ijk}[a,(bc)] = AT[j][k].BT[i] + AT[k][i].BT[j] + AT[i][j].BT[k]
//   (= P(i/jk) of the particle and hole terms; the signs are absorbed by
//   t^{ae}_{pq} = -t^{ae}_{qp} and H_qp = -H_pq).
// Mixed (i<j spin s, K spin t):
//   A1[p][K][a][kk]  = -t^{aE}_{pK} (kk=E<vt),  (pa|MK) (kk = vt+M)
//   BG[x][(b,C)][kk] = (xb|EC)      (kk=E),     t^{bC}_{xM} (kk = vt+M)
//   BF[K][(b,C)][kk] = (be|KC)      (kk=e<vs),  -t^{bC}_{mK} (kk = vs+m)
//   AT2[p][K][C][kk] = t^{eC}_{pK}  (kk=e),     (mp|CK) (kk = vs+m)
//   Y[a,(bC)]   = A1[j][K].BG[i] - A1[i][K].BG[j] + AT[i][j].BF[K]
//   Z'[C,(a<b)] = -AT2[j][K].BT[i] + AT2[i][K].BT[j]
// Rows are padded with zeros to a pitch Kp (a multiple of 32 elements on 16-bit
// slices, of 16 otherwise; of 8 for the DF blocks where a memory bound asks for it).
// Occupied indices come in two ranges: the summed (internal) m, M run over the
// first oi (oti) orbitals, the external ones over all o (ot) the arrays hold.
// The two differ only when pseudo-orbitals (the central LMOs of the Laplace
// form, Sec. 3.7) are appended after the real occupied orbitals; the DF
// blocks with one internal occupied index are laid out [internal][external].
//
// Every pack kernel is templated on its store: float64, or the slices of the
// tensor-core path (BF16: value = scale 2^-7 (s1 + s2 + s3), s1 an integer in
// [-128, 128], s2 a multiple of 2^-8 in [-1/2, 1/2], ..., each digit the nearest;
// FP16 and TF32 in common.cuh).
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace lno {

namespace {

// B[s] [naux][nbas][nbas] -> out[p'][q'][Q] = B[Q][p0+p'][q0+q'] (p' < np, q' < nq),
// for the blocks of a list: blockIdx.x runs over the 32-row tiles of all of them
template <class St>
__global__ void transpose_blocks(const double* __restrict__ B, int naux, int nbas,
                                 BlockList<St> L) {
  __shared__ double tile[32][33];
  int k = 0;
  int64_t t = blockIdx.x;
  for (; k < BlockList<St>::kMax - 1; ++k) {
    const int64_t nt = ((int64_t)L.np[k] * L.nq[k] + 31) / 32;
    if (t < nt) break;
    t -= nt;
  }
  const int p0 = L.p0[k], np = L.np[k], q0 = L.q0[k], nq = L.nq[k], Qp = L.Qp[k];
  const int64_t nrows = (int64_t)np * nq;
  const int64_t r0 = t * 32;
  const int Q0 = blockIdx.y * 32;
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int Q = Q0 + yy;
    const int64_t r = r0 + threadIdx.x;
    double v = 0.0;
    if (Q < naux && r < nrows) {
      const int p = (int)(r / nq), q = (int)(r % nq);
      v = B[((int64_t)Q * nbas + p0 + p) * nbas + q0 + q];
    }
    tile[yy][threadIdx.x] = v;
  }
  __syncthreads();
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int64_t r = r0 + yy;
    const int Q = Q0 + threadIdx.x;
    if (r < nrows && Q < Qp) L.st[k](r * Qp + Q, Q < naux ? tile[threadIdx.x][yy] : 0.0, 1);
  }
}

// AT[slot][a][kk] for same-spin pair (p,q) = pairs[slot]
template <class St>
__global__ void pack_at_same(const int2* __restrict__ pairs, int nslot, int o, int oi, int v,
                             int Kp, const double* __restrict__ t2ss,
                             const double* __restrict__ oovoT, St st) {
  const int64_t total = (int64_t)nslot * v * Kp;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int kk = (int)(idx % Kp);
    const int64_t r = idx / Kp;
    const int a = (int)(r % v);
    const int slot = (int)(r / v);
    const int2 pq = pairs[slot];
    double val = 0.0;
    if (kk < v) {
      val = t2ss[(((int64_t)pq.x * o + pq.y) * v + a) * v + kk];
    } else if (kk < v + oi) {
      const int m = kk - v;
      const int64_t oo = (int64_t)oi * o;
      // H_qp[m][a] = (mq|ap) - (mp|aq);  oovoT[(y*v+a)][(m*o+x)] = (mx|ya)
      val = oovoT[((int64_t)pq.x * v + a) * oo + m * o + pq.y] -
            oovoT[((int64_t)pq.y * v + a) * oo + m * o + pq.x];
    }
    st(idx, val, kk >= v);
  }
}

// The large operands BT, BG, BF are written in runs of 16 consecutive k per
// thread (32 bytes per slice: whole sectors), read so that a warp's loads run
// along the DF block's contiguous index; blockIdx.z is the occupied orbital x0 +
// z, slot slot0 + z, whose DF block follows the previous one.  Bound by the
// float64 reads and the slice writes plus ~50 integer operations per element.

// BT[slot][pair(b<c)][kk] for occupied x; vvovT[c][(e*v+b)] = (eb|xc).
// A CTA owns a 16 x 16 block of (b, c), b-block <= c-block, and 16 k: thread
// (c, b) keeps (eb|xc) of its row (read along b) and takes (ec|xb), read along c
// by the transposed thread, from shared memory.
template <class St>
__global__ void __launch_bounds__(256)
pack_bt_same(int slot0, int x0, int o, int oi, int v, int Kp, const double* __restrict__ vvovT,
             const double* __restrict__ t2ss, St st) {
  __shared__ double tr[16][16][17];
  const int slot = slot0 + (int)blockIdx.z, x = x0 + (int)blockIdx.z;
  // block pair (B <= C): index C (C + 1) / 2 + B
  int C = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
  while (C * (C + 1) / 2 > (int)blockIdx.x) --C;
  while ((C + 1) * (C + 2) / 2 <= (int)blockIdx.x) ++C;
  const int B = (int)blockIdx.x - C * (C + 1) / 2;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int k0 = blockIdx.y * 16;
  const int64_t vv = (int64_t)v * v;
  const double* src = vvovT + (int64_t)blockIdx.z * v * vv;
  const int b = B * 16 + tx, c = C * 16 + ty;      // this thread's row
  const int b2 = B * 16 + ty, c2 = C * 16 + tx;    // what it fetches for the others
  double val[16];
  uint32_t parts = 0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int kk = k0 + j;
    double own = 0.0, other = 0.0;
    if (kk < v) {
      if (b < v && c < v) own = src[(int64_t)c * vv + (int64_t)kk * v + b];
      if (b2 < v && c2 < v) other = src[(int64_t)b2 * vv + (int64_t)kk * v + c2];
      parts |= 1u << j;
    } else if (kk < v + oi && b2 < v && c2 < v) {
      other = -t2ss[(((int64_t)x * o + (kk - v)) * v + b2) * v + c2];
    }
    val[j] = own;
    tr[j][ty][tx] = other;
  }
  __syncthreads();
  if (b < c && c < v) {
#pragma unroll
    for (int j = 0; j < 16; ++j) val[j] -= tr[j][tx][ty];
    st.store16(((int64_t)slot * npairs(v) + pair_index(b, c)) * Kp + k0, val, parts);
  }
}

// A1[slot][a][kk] for mixed pair (p,K) = pk[slot]; jT[(M*ot+K)][(p*vs+a)] = (pa|MK)
template <class St>
__global__ void pack_a1(const int2* __restrict__ pk, int nslot, int os, int vs, int ot, int oti,
                        int vt, int Kp, const double* __restrict__ t2st,
                        const double* __restrict__ jT, St st) {
  const int64_t total = (int64_t)nslot * vs * Kp;
  const int64_t ld = (int64_t)os * vs;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int kk = (int)(idx % Kp);
    const int64_t r = idx / Kp;
    const int a = (int)(r % vs);
    const int2 p = pk[r / vs];
    double val = 0.0;
    if (kk < vt) {
      val = -t2st[(((int64_t)p.x * ot + p.y) * vs + a) * vt + kk];
    } else if (kk < vt + oti) {
      const int M = kk - vt;
      val = jT[((int64_t)M * ot + p.y) * ld + (int64_t)p.x * vs + a];
    }
    st(idx, val, kk >= vt);
  }
}

// BG[slot][(b*vt+C)][kk] for occupied x (spin s); gT[b][(E*vt+C)] = (xb|EC):
// thread = row, reads along C
template <class St>
__global__ void __launch_bounds__(256)
pack_bg(int slot0, int x0, int os, int vs, int ot, int oti, int vt, int Kp,
        const double* __restrict__ gT, const double* __restrict__ t2st, St st) {
  const int slot = slot0 + (int)blockIdx.z, x = x0 + (int)blockIdx.z;
  const int64_t rows = (int64_t)vs * vt, vv = (int64_t)vt * vt;
  const int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (r >= rows) return;
  const int k0 = blockIdx.y * 16;
  const int b = (int)(r / vt), C = (int)(r - (int64_t)b * vt);
  const double* src = gT + ((int64_t)blockIdx.z * vs + b) * vv + C;
  double val[16];
  uint32_t parts = 0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int kk = k0 + j;
    val[j] = 0.0;
    if (kk < vt) {
      val[j] = src[(int64_t)kk * vt];
      parts |= 1u << j;
    } else if (kk < vt + oti) {
      val[j] = t2st[(((int64_t)x * ot + (kk - vt)) * vs + b) * vt + C];
    }
  }
  st.store16(((int64_t)slot * rows + r) * Kp + k0, val, parts);
}

// BF[slot][(b*vt+C)][kk] for occupied K (spin t); fT[C][(b*vs+e)] = (be|KC):
// thread = row, reads its 16 e (one 128-byte line)
template <class St>
__global__ void __launch_bounds__(256)
pack_bf(int slot0, int K0, int os, int osi, int vs, int ot, int vt, int Kp,
        const double* __restrict__ fT, const double* __restrict__ t2st, St st) {
  const int slot = slot0 + (int)blockIdx.z, K = K0 + (int)blockIdx.z;
  const int64_t rows = (int64_t)vs * vt, vv = (int64_t)vs * vs;
  const int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (r >= rows) return;
  const int k0 = blockIdx.y * 16;
  const int b = (int)(r / vt), C = (int)(r - (int64_t)b * vt);
  const double* src = fT + ((int64_t)blockIdx.z * vt + C) * vv + (int64_t)b * vs;
  double val[16];
  uint32_t parts = 0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int kk = k0 + j;
    val[j] = 0.0;
    if (kk < vs) {
      val[j] = src[kk];
      parts |= 1u << j;
    } else if (kk < vs + osi) {
      val[j] = -t2st[(((int64_t)(kk - vs) * ot + K) * vs + b) * vt + C];
    }
  }
  st.store16(((int64_t)slot * rows + r) * Kp + k0, val, parts);
}

// AT2[slot][C][kk] for (p,K) = pk[slot]; lT[(K*vt+C)][(m*os+p)] = (mp|KC)
template <class St>
__global__ void pack_at2(const int2* __restrict__ pk, int nslot, int os, int osi, int vs, int ot,
                         int vt, int Kp, const double* __restrict__ t2st,
                         const double* __restrict__ lT, St st) {
  const int64_t total = (int64_t)nslot * vt * Kp;
  const int64_t ld = (int64_t)osi * os;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int kk = (int)(idx % Kp);
    const int64_t r = idx / Kp;
    const int C = (int)(r % vt);
    const int2 p = pk[r / vt];
    double val = 0.0;
    if (kk < vs) {
      val = t2st[(((int64_t)p.x * ot + p.y) * vs + kk) * vt + C];
    } else if (kk < vs + osi) {
      const int m = kk - vs;
      val = lT[((int64_t)p.y * vt + C) * ld + (int64_t)m * os + p.x];
    }
    st(idx, val, kk >= vs);
  }
}

// t2ba[I][k][A][c] = t2ab[k][I][c][A]
__global__ void transpose_t2ab(const double* __restrict__ t2ab, int na, int nb, int va, int vb,
                               double* __restrict__ out) {
  const int64_t total = (int64_t)na * nb * va * vb;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    // out index (I, k, A, c)
    int c = (int)(idx % va);
    int64_t r = idx / va;
    int A = (int)(r % vb);
    r /= vb;
    int k = (int)(r % na);
    int I = (int)(r / na);
    out[idx] = t2ab[(((int64_t)k * nb + I) * va + c) * vb + A];
  }
}

// Strided float64 views for the tensor-core adjoint: element (r, k) of a
// rows x K view sits at in[r rs + k ks].  Work goes in 32 x 32 tiles whose
// loads run along the view's unit-stride index (k when ks == 1, else r), so
// they coalesce either way.
__device__ __forceinline__ double view_at(const double* in, int64_t rs, int64_t ks, int rows,
                                          int K, int r, int k) {
  return (r < rows && k < K) ? in[(int64_t)r * rs + (int64_t)k * ks] : 0.0;
}

// max |x| over the view (bits of a non-negative double, atomicMax into *out)
__global__ void view_absmax(const double* __restrict__ in, int64_t rs, int64_t ks, int rows,
                            int K, unsigned long long* __restrict__ out) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  const bool rfast = ks != 1 && rs == 1;
  double m = 0.0;
  for (int r0 = blockIdx.y * 32; r0 < rows; r0 += gridDim.y * 32) {
    const int k0 = blockIdx.x * 32;
    for (int i = ty; i < 32; i += 8) {
      const double x = rfast ? view_at(in, rs, ks, rows, K, r0 + tx, k0 + i)
                             : view_at(in, rs, ks, rows, K, r0 + i, k0 + tx);
      m = fmax(m, fabs(x));
    }
  }
  for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, off));
  if ((tx & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// The same exact slices as StoreSlices, from one rounding of the scaled value
// to S * 8 - 1 fractional bits followed by integer digit extraction (base 256,
// each digit rounded half up, so |s_0| <= 128 and |s_q 2^(8q)| <= 128):
// value = 2^-e7 (s_0 + ... + s_{S-1}), e7 = e2 - 8 (S - 1), e2 passed in.
template <int S>
struct StoreSlicesInt {
  __nv_bfloat16* p;
  int64_t slice_stride;
  int e2;   // log2(2^7 / scale) + 8 (S - 1)
  __device__ __forceinline__ void operator()(int64_t idx, double v) const {
    if (isnan(v)) {   // NaN in the leading slice reaches the product
      p[idx] = __float2bfloat16_rn(__int_as_float(0x7fc00000));
#pragma unroll
      for (int q = 1; q < S; ++q) p[q * slice_stride + idx] = __float2bfloat16_rn(0.f);
      return;
    }
    int64_t R = round_scaled(v, e2);
#pragma unroll
    for (int q = 0; q < S; ++q) {
      const int sh = 8 * (S - 1 - q);
      const int64_t d = sh ? (R + (1ll << (sh - 1))) >> sh : R;
      R -= d << sh;
      p[q * slice_stride + idx] = __float2bfloat16_rn(ldexpf((float)d, -8 * q));
    }
  }
};

// Matrices of a batch, each rows x cols float64 at src + z src_stride (row pitch
// ld), sliced in both layouts for the adjoint's grouped products: n [z][r][Kd] (k
// = column) and t [z][c][Nd] (k = row), Kd and Nd multiples of 32, zero in the
// pads.  Each matrix has its own scale 2^e[z] (slice_exponents).
__global__ void batch_absmax(const double* __restrict__ src, int64_t src_stride, int count,
                             int rows, int cols, int ld, unsigned long long* __restrict__ amax) {
  const int64_t n = (int64_t)rows * cols;
  for (int z = blockIdx.y; z < count; z += gridDim.y) {
    const double* p = src + (int64_t)z * src_stride;
    double m = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
      const int64_t r = i / cols;
      m = fmax(m, fabs(p[r * ld + (i - r * cols)]));
    }
    for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0 && m > 0.0)
      atomicMax(amax + z, (unsigned long long)__double_as_longlong(m));
  }
}

// e = smallest exponent with 2^e >= max (0 for a zero matrix); an infinite
// maximum raises the error flag (code 9: invalid input).
__global__ void slice_exponents(const unsigned long long* __restrict__ amax, int n,
                                int* __restrict__ e, int* __restrict__ flag) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double m = __longlong_as_double((long long)amax[i]);
    int ex = 0;
    if (isinf(m)) {
      atomicCAS(flag, 0, 9);
    } else if (m > 0.0) {
      const double f = frexp(m, &ex);
      if (f == 0.5) --ex;
    }
    e[i] = ex;
  }
}

// Row tiles and matrices beyond the grid's limits (65535 each) are taken in strides.
template <int S>
__global__ void batch_slices(const double* __restrict__ src, int64_t src_stride, int count,
                             int rows, int cols, int ld, const int* __restrict__ e,
                             __nv_bfloat16* __restrict__ dn, int Kd, int64_t stride_n,
                             __nv_bfloat16* __restrict__ dt, int Nd, int64_t stride_t) {
  __shared__ double t[32][33];   // [r][c]
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int c0 = blockIdx.x * 32;
  for (int z = blockIdx.z; z < count; z += gridDim.z) {
    const double* p = src + (int64_t)z * src_stride;
    const int e2 = 7 - e[z] + 8 * (S - 1);
    for (int64_t r0 = (int64_t)blockIdx.y * 32; r0 < Nd; r0 += (int64_t)gridDim.y * 32) {
      for (int i = ty; i < 32; i += 8) {
        const int64_t r = r0 + i;
        const int c = c0 + tx;
        t[i][tx] = r < rows && c < cols ? p[r * ld + c] : 0.0;
      }
      __syncthreads();
      if (dn != nullptr) {
        const StoreSlicesInt<S> st{dn, stride_n, e2};
        for (int i = ty; i < 32; i += 8)
          if (r0 + i < rows) st(((int64_t)z * rows + r0 + i) * Kd + c0 + tx, t[i][tx]);
      }
      if (dt != nullptr) {
        const StoreSlicesInt<S> st{dt, stride_t, e2};
        for (int i = ty; i < 32; i += 8)
          if (c0 + i < cols) st(((int64_t)z * cols + c0 + i) * Nd + r0 + tx, t[tx][i]);
      }
      __syncthreads();
    }
  }
}

// view -> S BF16 slices [s][r][Kp] (k-contiguous rows, zero for k >= K)
template <int S>
__global__ void view_slices(const double* __restrict__ in, int64_t rs, int64_t ks, int rows,
                            int K, int Kp, StoreSlicesInt<S> st) {
  __shared__ double t[32][33];   // [k][r]
  const int tx = threadIdx.x, ty = threadIdx.y;
  const bool rfast = ks != 1 && rs == 1;
  const int k0 = blockIdx.x * 32;
  for (int r0 = blockIdx.y * 32; r0 < rows; r0 += gridDim.y * 32) {
    for (int i = ty; i < 32; i += 8) {
      if (rfast)
        t[i][tx] = view_at(in, rs, ks, rows, K, r0 + tx, k0 + i);
      else
        t[tx][i] = view_at(in, rs, ks, rows, K, r0 + i, k0 + tx);
    }
    __syncthreads();
    for (int i = ty; i < 32; i += 8) {
      const int r = r0 + i, k = k0 + tx;
      if (r < rows && k < Kp) st((int64_t)r * Kp + k, t[tx][i]);
    }
    __syncthreads();
  }
}

// C[m ldc + n] = (accum ? C : 0) + sum over c of part[c][m][n], in chunk order.
__global__ void sum_partials(const double* __restrict__ part, int nsp, int M, int N,
                             double* __restrict__ C, int64_t ldc, int accum) {
  const int64_t n_all = (int64_t)M * N;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_all;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t m = i / N, n = i - m * N;
    double v = 0.0;
    for (int c = 0; c < nsp; ++c) v += part[(int64_t)c * n_all + i];
    double* o = C + m * ldc + n;
    *o = accum ? *o + v : v;
  }
}

// max |x| over the arrays of a list, as the bits of a non-negative double in their
// *out (atomicMax); blockIdx.y is the array.
__global__ void absmax_kernel(AbsmaxList L) {
  const double* __restrict__ x = L.x[blockIdx.y];
  const int64_t n = L.n[blockIdx.y];
  double m = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    m = fmax(m, fabs(x[i]));
  for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0 && m > 0.0)
    atomicMax(L.out[blockIdx.y], (unsigned long long)__double_as_longlong(m));
}

// Row-block gather: dst slot q <- src slot list[q], each slot `row16` 16-byte
// words, repeated over `nslice` slices (bf16 slices of one operand, or one
// float64 plane).  Used to keep only the occupied orbitals a triplet set uses.
__global__ void gather_rows_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst,
                                   const int* __restrict__ list, int nlist, int64_t row16,
                                   int nslice, int64_t src_slice16, int64_t dst_slice16) {
  const int64_t per = (int64_t)nlist * row16, n = per * nslice;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t sl = e / per, r = e - sl * per;
    const int64_t q = r / row16, w = r - q * row16;
    dst[sl * dst_slice16 + r] = src[sl * src_slice16 + (int64_t)list[q] * row16 + w];
  }
}

// dst slot list[q] += src slot q (float64; slots of `row` elements, list
// entries distinct, so no two threads touch one element).
__global__ void scatter_add_rows_kernel(const double* __restrict__ src, double* __restrict__ dst,
                                        const int* __restrict__ list, int nlist, int64_t row) {
  const int64_t n = (int64_t)nlist * row;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q = e / row, w = e - q * row;
    dst[(int64_t)list[q] * row + w] += src[e];
  }
}

// Largest sum of squares of one row of an operand's leading FP16 slice (the
// integers d_0), as the bits of a double in *out (atomicMax): a warp per row.
__global__ void __launch_bounds__(256)
row_norm2(const uint4* __restrict__ p, int64_t rows, int row16, unsigned long long* out) {
  const int lane = threadIdx.x & 31;
  float best = 0.f;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < rows;
       r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    float ss = 0.f;
    for (int w = lane; w < row16; w += 32) {
      const uint4 u = p[r * row16 + w];
      const uint32_t h[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h[q]));
        ss += f.x * f.x + f.y * f.y;
      }
    }
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    best = isnan(ss) ? INFINITY : fmaxf(best, ss);
  }
  if (lane == 0 && best > 0.f)
    atomicMax(out, (unsigned long long)__double_as_longlong((double)best));
}

// Number of elements with |t2ab[i][J][a][B] - t2ab[J][i][B][a]| > tol (n
// occupied and v virtual of each spin); zero means the mixed amplitudes are
// spin-flip symmetric to within tol.
__global__ void t2ab_flip_mismatch(const double* __restrict__ t2ab, int n, int v, double tol,
                                   unsigned int* __restrict__ count) {
  const int64_t total = (int64_t)n * n * v * v;
  unsigned int bad = 0;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int B = (int)(idx % v);
    int64_t r = idx / v;
    const int a = (int)(r % v);
    r /= v;
    const int J = (int)(r % n), i = (int)(r / n);
    if (!(fabs(t2ab[idx] - t2ab[(((int64_t)J * n + i) * v + B) * v + a]) <= tol)) ++bad;
  }
  if (bad) atomicAdd(count, bad);
}

inline int grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)(b < 152 * 32 ? (b < 1 ? 1 : b) : 152 * 32);
}

}  // namespace

// ---------------------------------------------------------------------------
// Host launchers (templated store: F64 or slices)
// ---------------------------------------------------------------------------
template <class St>
cudaError_t launch_transpose_blocks(const double* B, int naux, int nbas, const BlockList<St>& L,
                                    cudaStream_t s) {
  int64_t tiles = 0;
  int Qp = 0;
  for (int k = 0; k < BlockList<St>::kMax; ++k) {
    tiles += ((int64_t)L.np[k] * L.nq[k] + 31) / 32;
    Qp = std::max(Qp, L.Qp[k]);
  }
  if (tiles == 0) return cudaSuccess;
  transpose_blocks<<<dim3((unsigned)tiles, ceil_div(Qp, 32)), dim3(32, 8), 0, s>>>(B, naux, nbas,
                                                                                 L);
  return cudaGetLastError();
}

template <class St>
cudaError_t launch_pack_at_same(const int2* pairs, int nslot, int o, int oi, int v, int Kp,
                                const double* t2ss, const double* oovoT, St st, cudaStream_t s) {
  int64_t n = (int64_t)nslot * v * Kp;
  if (n == 0) return cudaSuccess;
  pack_at_same<<<grid_for(n), 256, 0, s>>>(pairs, nslot, o, oi, v, Kp, t2ss, oovoT, st);
  return cudaGetLastError();
}

template <class St>
cudaError_t launch_pack_bt_same(int slot0, int x0, int nx, int o, int oi, int v, int Kp,
                                const double* vvovT, const double* t2ss, St st, cudaStream_t s) {
  if (npairs(v) * Kp * nx == 0) return cudaSuccess;
  const int nb = (v + 15) / 16;
  pack_bt_same<<<dim3(nb * (nb + 1) / 2, (Kp + 15) / 16, nx), 256, 0, s>>>(slot0, x0, o, oi, v, Kp,
                                                                         vvovT, t2ss, st);
  return cudaGetLastError();
}

template <class St>
cudaError_t launch_pack_a1(const int2* pk, int nslot, int os, int vs, int ot, int oti, int vt,
                           int Kp, const double* t2st, const double* jT, St st, cudaStream_t s) {
  int64_t n = (int64_t)nslot * vs * Kp;
  if (n == 0) return cudaSuccess;
  pack_a1<<<grid_for(n), 256, 0, s>>>(pk, nslot, os, vs, ot, oti, vt, Kp, t2st, jT, st);
  return cudaGetLastError();
}

template <class St>
cudaError_t launch_pack_bg(int slot0, int x0, int nx, int os, int vs, int ot, int oti, int vt,
                           int Kp, const double* gT, const double* t2st, St st, cudaStream_t s) {
  if ((int64_t)vs * vt * Kp * nx == 0) return cudaSuccess;
  const dim3 grid(ceil_div((int64_t)vs * vt, 256), (Kp + 15) / 16, nx);
  pack_bg<<<grid, 256, 0, s>>>(slot0, x0, os, vs, ot, oti, vt, Kp, gT, t2st, st);
  return cudaGetLastError();
}

template <class St>
cudaError_t launch_pack_bf(int slot0, int K0, int nx, int os, int osi, int vs, int ot, int vt,
                           int Kp, const double* fT, const double* t2st, St st, cudaStream_t s) {
  if ((int64_t)vs * vt * Kp * nx == 0) return cudaSuccess;
  const dim3 grid(ceil_div((int64_t)vs * vt, 256), (Kp + 15) / 16, nx);
  pack_bf<<<grid, 256, 0, s>>>(slot0, K0, os, osi, vs, ot, vt, Kp, fT, t2st, st);
  return cudaGetLastError();
}

template <class St>
cudaError_t launch_pack_at2(const int2* pk, int nslot, int os, int osi, int vs, int ot, int vt,
                            int Kp, const double* t2st, const double* lT, St st,
                            cudaStream_t s) {
  int64_t n = (int64_t)nslot * vt * Kp;
  if (n == 0) return cudaSuccess;
  pack_at2<<<grid_for(n), 256, 0, s>>>(pk, nslot, os, osi, vs, ot, vt, Kp, t2st, lT, st);
  return cudaGetLastError();
}

cudaError_t launch_transpose_t2ab(const double* t2ab, int na, int nb, int va, int vb, double* out,
                                  cudaStream_t s) {
  int64_t n = (int64_t)na * nb * va * vb;
  if (n == 0) return cudaSuccess;
  transpose_t2ab<<<grid_for(n), 256, 0, s>>>(t2ab, na, nb, va, vb, out);
  return cudaGetLastError();
}

cudaError_t launch_gather_rows(const void* src, void* dst, const int* list, int nlist,
                               int64_t row_bytes, int nslice, int64_t src_slice_bytes,
                               int64_t dst_slice_bytes, cudaStream_t s) {
  if (nlist == 0 || row_bytes == 0 || nslice == 0) return cudaSuccess;
  if (row_bytes % 16 || src_slice_bytes % 16 || dst_slice_bytes % 16 ||
      reinterpret_cast<uintptr_t>(src) % 16 || reinterpret_cast<uintptr_t>(dst) % 16)
    return cudaErrorInvalidValue;
  const int64_t n = (int64_t)nlist * (row_bytes / 16) * nslice;
  gather_rows_kernel<<<grid_for(n), 256, 0, s>>>(
      static_cast<const uint4*>(src), static_cast<uint4*>(dst), list, nlist, row_bytes / 16,
      nslice, src_slice_bytes / 16, dst_slice_bytes / 16);
  return cudaGetLastError();
}

cudaError_t launch_scatter_add_rows(const double* src, double* dst, const int* list, int nlist,
                                    int64_t row, cudaStream_t s) {
  const int64_t n = (int64_t)nlist * row;
  if (n == 0) return cudaSuccess;
  scatter_add_rows_kernel<<<grid_for(n), 256, 0, s>>>(src, dst, list, nlist, row);
  return cudaGetLastError();
}

cudaError_t launch_t2ab_flip_mismatch(const double* t2ab, int n, int v, double tol,
                                     unsigned int* count, cudaStream_t s) {
  const int64_t total = (int64_t)n * n * v * v;
  if (total == 0) return cudaSuccess;
  t2ab_flip_mismatch<<<grid_for(total), 256, 0, s>>>(t2ab, n, v, tol, count);
  return cudaGetLastError();
}

cudaError_t launch_row_norm2(const void* p, int64_t rows, int Kp, unsigned long long* out,
                             cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  if (Kp % 8 || reinterpret_cast<uintptr_t>(p) % 16) return cudaErrorInvalidValue;
  row_norm2<<<grid_for(rows * 32), 256, 0, s>>>(static_cast<const uint4*>(p), rows, Kp / 8, out);
  return cudaGetLastError();
}

cudaError_t launch_absmax_list(const AbsmaxList& L, cudaStream_t s) {
  int64_t n = 0;
  for (int q = 0; q < L.count; ++q) n = std::max(n, L.n[q]);
  if (n == 0) return cudaSuccess;
  absmax_kernel<<<dim3(std::min(grid_for(n), 152 * 8), L.count), 256, 0, s>>>(L);
  return cudaGetLastError();
}

cudaError_t launch_absmax(const double* x, int64_t n, unsigned long long* out, cudaStream_t s) {
  AbsmaxList L{};
  L.x[0] = x;
  L.n[0] = n;
  L.out[0] = out;
  L.count = 1;
  return launch_absmax_list(L, s);
}

cudaError_t launch_sum_partials(const double* part, int nsp, int M, int N, double* C,
                                int64_t ldc, bool accum, cudaStream_t s) {
  const int64_t n = (int64_t)M * N;
  if (n <= 0) return cudaSuccess;
  sum_partials<<<grid_for(n), 256, 0, s>>>(part, nsp, M, N, C, ldc, accum ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_view_absmax(const double* in, int64_t rs, int64_t ks, int rows, int K,
                               unsigned long long* out, cudaStream_t s) {
  if (rows <= 0 || K <= 0) return cudaSuccess;
  const dim3 grid((unsigned)((K + 31) / 32), (unsigned)std::min((rows + 31) / 32, 4096));
  view_absmax<<<grid, dim3(32, 8), 0, s>>>(in, rs, ks, rows, K, out);
  return cudaGetLastError();
}

cudaError_t launch_batch_slices(const double* src, int64_t src_stride, int count, int rows,
                                int cols, int ld, unsigned long long* amax, int* e, int* flag,
                                __nv_bfloat16* dn, int Kd, int64_t stride_n, __nv_bfloat16* dt,
                                int Nd, int64_t stride_t, cudaStream_t s) {
  if (count <= 0 || rows <= 0 || cols <= 0) return cudaSuccess;
  if (Kd % 32 || Nd % 32) return cudaErrorInvalidValue;
  cudaError_t rc = cudaMemsetAsync(amax, 0, (size_t)count * sizeof(unsigned long long), s);
  if (rc != cudaSuccess) return rc;
  constexpr int kMaxGrid = 65535;   // y and z
  const int bx = (int)std::min<int64_t>(((int64_t)rows * cols + 1023) / 1024, 512);
  batch_absmax<<<dim3(bx, std::min(count, kMaxGrid)), 256, 0, s>>>(src, src_stride, count, rows,
                                                                  cols, ld, amax);
  slice_exponents<<<ceil_div(count, 256), 256, 0, s>>>(amax, count, e, flag);
  const dim3 grid(Kd / 32, std::min(Nd / 32, kMaxGrid), std::min(count, kMaxGrid));
  batch_slices<4><<<grid, dim3(32, 8), 0, s>>>(src, src_stride, count, rows, cols, ld, e, dn, Kd,
                                               stride_n, dt, Nd, stride_t);
  return cudaGetLastError();
}

// inv = 2^7 / scale, a power of two
template <int S>
cudaError_t launch_view_slices(const double* in, int64_t rs, int64_t ks, int rows, int K,
                               int Kp, __nv_bfloat16* out, int64_t slice_stride, double inv,
                               cudaStream_t s) {
  if (rows <= 0 || Kp <= 0) return cudaSuccess;
  int e;
  if (!(inv > 0) || std::frexp(inv, &e) != 0.5) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)((Kp + 31) / 32), (unsigned)std::min((rows + 31) / 32, 4096));
  view_slices<S><<<grid, dim3(32, 8), 0, s>>>(
      in, rs, ks, rows, K, Kp, StoreSlicesInt<S>{out, slice_stride, (e - 1) + 8 * (S - 1)});
  return cudaGetLastError();
}
template cudaError_t launch_view_slices<4>(const double*, int64_t, int64_t, int, int, int,
                                           __nv_bfloat16*, int64_t, double, cudaStream_t);

#define LNO_INST(St)                                                                           \
  template cudaError_t launch_transpose_blocks<St>(const double*, int, int,                      \
                                                   const BlockList<St>&, cudaStream_t);         \
  template cudaError_t launch_pack_at_same<St>(const int2*, int, int, int, int, int,           \
                                               const double*, const double*, St, cudaStream_t); \
  template cudaError_t launch_pack_bt_same<St>(int, int, int, int, int, int, int,               \
                                               const double*, const double*, St, cudaStream_t); \
  template cudaError_t launch_pack_a1<St>(const int2*, int, int, int, int, int, int, int,      \
                                          const double*, const double*, St, cudaStream_t);     \
  template cudaError_t launch_pack_bg<St>(int, int, int, int, int, int, int, int, int,          \
                                          const double*, const double*, St, cudaStream_t);     \
  template cudaError_t launch_pack_bf<St>(int, int, int, int, int, int, int, int, int,          \
                                          const double*, const double*, St, cudaStream_t);     \
  template cudaError_t launch_pack_at2<St>(const int2*, int, int, int, int, int, int, int,     \
                                           const double*, const double*, St, cudaStream_t);

LNO_INST(StoreF64)
LNO_INST(StoreSlices<2>)
LNO_INST(StoreSlices<3>)
LNO_INST(StoreSlices<4>)
LNO_INST(StoreSlices<5>)
LNO_INST(StoreTF32<2>)
using StoreF16x3 = StoreSlices<3, __half>;
LNO_INST(StoreF16x3)
#undef LNO_INST

}  // namespace lno
