// Natural auxiliary functions of a domain (arXiv 2311.10048, Sec. 3.6, eq
// naf_w), in float64 on the CUDA cores:
//   1. J^s[X][(p<=q)] = B^X_pq (pair-packed factors of each spin);
//   2. W = (J^up J^up^T + J^down J^down^T) / 2, one symmetric contraction;
//   3. eigenvectors of W by cyclic Jacobi rotations in the round-robin order
//      (n/2 disjoint rotations per round, n - 1 rounds per sweep, one launch per
//      round, until the off-diagonal norm is below 1e-14 of the Frobenius norm);
//   4. the eigenvectors with eigenvalues above eps_naf, in descending order;
//   5. B'^s[X'][pq] = sum_X V[X][X'] B^s[X][pq] (one contraction per spin, over
//      the packed pairs p <= q when the factors are symmetric to the bit).
// The eigen-decomposition runs on the device; only the n eigenvalues and the
// convergence measure come back to the host (to sort and to stop).
#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

#include "common.cuh"

namespace lno {

namespace {

inline int grid_n(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)(b < 152 * 32 ? (b < 1 ? 1 : b) : 152 * 32);
}

// J[X][pair] = B[X][p][q] for p <= q (pair = q (q + 1) / 2 + p)
__global__ void pack_pairs(const double* __restrict__ B, int naux, int n,
                           double* __restrict__ J) {
  const int64_t np = (int64_t)n * (n + 1) / 2;
  const int64_t total = (int64_t)naux * np;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t pr = idx % np;
    const int X = (int)(idx / np);
    int q = (int)((sqrt(8.0 * (double)pr + 1.0) - 1.0) * 0.5);
    while ((int64_t)q * (q + 1) / 2 > pr) --q;
    while ((int64_t)(q + 1) * (q + 2) / 2 <= pr) ++q;
    const int p = (int)(pr - (int64_t)q * (q + 1) / 2);
    J[idx] = B[((int64_t)X * n + p) * n + q];
  }
}

// Bt[pq][X] = B[X][pq]
__global__ void transpose_x(const double* __restrict__ B, int naux, int64_t n2,
                            double* __restrict__ Bt) {
  __shared__ double tile[32][33];
  const int64_t r0 = (int64_t)blockIdx.x * 32;
  const int X0 = blockIdx.y * 32;
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int X = X0 + yy;
    const int64_t r = r0 + threadIdx.x;
    tile[yy][threadIdx.x] = (X < naux && r < n2) ? B[(int64_t)X * n2 + r] : 0.0;
  }
  __syncthreads();
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int64_t r = r0 + yy;
    const int X = X0 + threadIdx.x;
    if (r < n2 && X < naux) Bt[r * naux + X] = tile[threadIdx.x][yy];
  }
}

// Round-robin pair k of round r over m = np / 2 pairs of np (even) indices:
// pair 0 is (r, np - 1), pair k > 0 is ((r + k) mod (np-1), (r - k) mod (np-1)).
__device__ __forceinline__ void rr_pair(int r, int k, int np, int& p, int& q) {
  const int L = np - 1;
  if (k == 0) {
    p = r;
    q = L;
  } else {
    p = (r + k) % L;
    q = (r - k + L) % L;
  }
  if (p > q) {
    const int t = p;
    p = q;
    q = t;
  }
}

// rotation (c, s) that zeroes A[p][q]; indices >= n are padding (no rotation)
__device__ __forceinline__ double2 jac_angle(const double* A, int n, int p, int q) {
  double c = 1.0, s = 0.0;
  if (q < n) {
    const double apq = A[(int64_t)p * n + q];
    if (apq != 0.0) {
      const double app = A[(int64_t)p * n + p], aqq = A[(int64_t)q * n + q];
      const double tau = (aqq - app) / (2.0 * apq);
      const double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
      c = 1.0 / sqrt(1.0 + t * t);
      s = t * c;
    }
  }
  return make_double2(c, s);
}

// One round: A <- J^T A J for the round's disjoint rotations J, V^T <- J^T V^T.
// Blocks (x, y < m16) own the 2 x 2 element blocks of 16 x 16 pairs: one read of
// the old matrix and one write of the new one (two buffers: every block takes its
// 32 angles from the old), so a round is one launch.  Blocks y >= m16 rotate 16
// pairs of rows of V^T (128 columns each) in place.  Bound by the round's latency
// (angles: two square roots and three divisions, then one pass over the matrix in
// L2).  600 x 600: 21 us a round with three launches (angles, rows, and strided
// columns of A and V), 3.5 us so.
constexpr int JT = 16, JC = 128;
__global__ void __launch_bounds__(256)
jac_round(const double* __restrict__ Ain, double* __restrict__ Aout, double* __restrict__ VT,
          int n, int np, int r) {
  __shared__ double2 cs[2][JT];
  __shared__ int pp[2][JT], qq[2][JT];
  const int m = np / 2, m16 = (m + JT - 1) / JT;
  const bool vec = (int)blockIdx.y >= m16;
  const int tid = threadIdx.x;
  if (tid < 2 * JT) {
    const int w = tid / JT, l = tid % JT;
    const int k = (w == 0 || !vec ? (w == 0 ? (int)blockIdx.x : (int)blockIdx.y) : 0) * JT + l;
    int p = n, q = n;
    if (k < m) rr_pair(r, k, np, p, q);
    pp[w][l] = p;
    qq[w][l] = q;
    cs[w][l] = k < m ? jac_angle(Ain, n, p, q) : make_double2(1.0, 0.0);
  }
  __syncthreads();
  if (vec) {
    const int c0 = ((int)blockIdx.y - m16) * JC;
    for (int e = tid; e < JT * JC; e += 256) {
      const int l = e / JC, i = c0 + e % JC;
      const int p = pp[0][l], q = qq[0][l];
      if (i >= n || q >= n) continue;
      const double2 g = cs[0][l];
      const double ap = VT[(int64_t)p * n + i], aq = VT[(int64_t)q * n + i];
      VT[(int64_t)p * n + i] = g.x * ap - g.y * aq;
      VT[(int64_t)q * n + i] = g.y * ap + g.x * aq;
    }
    return;
  }
  // rows: pair a of blockIdx.x; columns: pair b of blockIdx.y
  const int a = tid / JT, b = tid % JT;
  const int p = pp[0][a], q = qq[0][a], u = pp[1][b], w = qq[1][b];
  if (p >= n || u >= n) return;
  const bool q_in = q < n, w_in = w < n;
  const double2 g = cs[0][a], h = cs[1][b];
  const double pu = Ain[(int64_t)p * n + u], pw = w_in ? Ain[(int64_t)p * n + w] : 0.0;
  const double qu = q_in ? Ain[(int64_t)q * n + u] : 0.0,
               qw = q_in && w_in ? Ain[(int64_t)q * n + w] : 0.0;
  // rows first, then columns
  const double tpu = g.x * pu - g.y * qu, tqu = g.y * pu + g.x * qu;
  const double tpw = g.x * pw - g.y * qw, tqw = g.y * pw + g.x * qw;
  Aout[(int64_t)p * n + u] = h.x * tpu - h.y * tpw;
  if (w_in) Aout[(int64_t)p * n + w] = h.y * tpu + h.x * tpw;
  if (q_in) Aout[(int64_t)q * n + u] = h.x * tqu - h.y * tqw;
  if (q_in && w_in) Aout[(int64_t)q * n + w] = h.y * tqu + h.x * tqw;
}

// part[2 b], part[2 b + 1] = block b's sums of squares of the off-diagonal elements
// and of all; jac_norms_sum adds them in block order.
constexpr int kNormBlocks = 128;
__global__ void __launch_bounds__(256)
jac_norms(const double* __restrict__ A, int n, double* __restrict__ part) {
  __shared__ double so[256], sa[256];
  double o = 0.0, a = 0.0;
  for (int64_t idx = blockIdx.x * 256LL + threadIdx.x; idx < (int64_t)n * n;
       idx += kNormBlocks * 256LL) {
    const double x = A[idx];
    a += x * x;
    if (idx / n != idx % n) o += x * x;
  }
  so[threadIdx.x] = o;
  sa[threadIdx.x] = a;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      so[threadIdx.x] += so[threadIdx.x + w];
      sa[threadIdx.x] += sa[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = so[0];
    part[2 * blockIdx.x + 1] = sa[0];
  }
}
__global__ void jac_norms_sum(const double* __restrict__ part, double* __restrict__ out) {
  if (threadIdx.x < 2) {
    double t = 0.0;
    for (int b = 0; b < kNormBlocks; ++b) t += part[2 * b + threadIdx.x];
    out[threadIdx.x] = t;
  }
}

__global__ void set_identity(double* __restrict__ V, int n) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)n * n;
       idx += (int64_t)gridDim.x * blockDim.x)
    V[idx] = (idx / n == idx % n) ? 1.0 : 0.0;
}

__global__ void get_diag(const double* __restrict__ A, int n, double* __restrict__ d) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    d[i] = A[(int64_t)i * n + i];
}

// out[c][X] = VT[rows[c]][X]  (kept eigenvectors)
__global__ void gather_rows(const double* __restrict__ VT, int n, const int* __restrict__ rows,
                            int nk, double* __restrict__ out) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)nk * n;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int X = (int)(idx % n), c = (int)(idx / n);
    out[idx] = VT[(int64_t)rows[c] * n + X];
  }
}

// Jt[pair][X] = J[X][pair]: transpose_x on the packed pairs.  unpack_pairs: B[X][p][q]
// and B[X][q][p] from the pairs.
__global__ void unpack_pairs(const double* __restrict__ J, int nx, int n,
                             double* __restrict__ B) {
  const int64_t np = (int64_t)n * (n + 1) / 2, n2 = (int64_t)n * n, total = (int64_t)nx * n2;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t X = idx / n2, e = idx - X * n2;
    const int p = (int)(e / n), q = (int)(e - (int64_t)p * n);
    const int lo = min(p, q), hi = max(p, q);
    B[idx] = J[X * np + (int64_t)hi * (hi + 1) / 2 + lo];
  }
}

// *count += elements with B[X][p][q] != B[X][q][p] (p < q)
__global__ void asym_count(const double* __restrict__ B, int naux, int n,
                           unsigned int* __restrict__ count) {
  __shared__ double t[32][33];
  const int bx = blockIdx.x, by = blockIdx.y;
  if (bx < by) return;   // tile (by, bx) against tile (bx, by)
  unsigned int bad = 0;
  for (int X = blockIdx.z; X < naux; X += gridDim.z) {
    const double* M = B + (int64_t)X * n * n;
    for (int i = threadIdx.y; i < 32; i += 8) {
      const int p = bx * 32 + i, q = by * 32 + threadIdx.x;
      t[i][threadIdx.x] = p < n && q < n ? M[(int64_t)p * n + q] : 0.0;
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += 8) {
      const int p = by * 32 + i, q = bx * 32 + threadIdx.x;
      if (p < n && q < n && !(M[(int64_t)p * n + q] == t[threadIdx.x][i])) ++bad;
    }
    __syncthreads();
  }
  if (bad) atomicAdd(count, bad);
}

}  // namespace

// Symmetric eigen-decomposition of A (n x n, device, destroyed: its diagonal
// ends up holding the eigenvalues) with eigenvectors in the rows of VT.  A2 is a
// second n x n buffer, norms holds 2 (1 + kNormBlocks) doubles.
// Returns the number of sweeps, or a negative lno_ot_status.
int jacobi_eigh(double* A, double* A2, double* VT, int n, double* norms, cudaStream_t st,
                int max_sweeps) {
  if (n <= 0) return 0;
  set_identity<<<grid_n((int64_t)n * n), 256, 0, st>>>(VT, n);
  if (n == 1) return 0;
  const int np = n + (n & 1);
  const int m16 = (np / 2 + JT - 1) / JT;
  const dim3 grid(m16, m16 + (n + JC - 1) / JC);
  double *cur = A, *other = A2;
  int sweeps = 0;
  cudaError_t e = cudaSuccess;
  for (; sweeps < max_sweeps && e == cudaSuccess; ++sweeps) {
    double h[2];
    jac_norms<<<kNormBlocks, 256, 0, st>>>(cur, n, norms + 2);
    jac_norms_sum<<<1, 32, 0, st>>>(norms + 2, norms);
    e = cudaMemcpyAsync(h, norms, sizeof h, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess || !(h[0] > 1e-28 * h[1])) break;   // off-diagonal norm < 1e-14
    for (int r = 0; r < np - 1; ++r) {
      jac_round<<<grid, 256, 0, st>>>(cur, other, VT, n, np, r);
      std::swap(cur, other);
    }
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && cur != A)
    e = cudaMemcpyAsync(A, cur, (size_t)n * n * sizeof(double), cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return LNO_OT_ECUDA;
  }
  return sweeps;
}

size_t jacobi_norm_doubles() { return 2 * (1 + kNormBlocks); }

cudaError_t launch_pack_pairs(const double* B, int naux, int n, double* J, cudaStream_t st) {
  pack_pairs<<<grid_n((int64_t)naux * n * (n + 1) / 2), 256, 0, st>>>(B, naux, n, J);
  return cudaGetLastError();
}

cudaError_t launch_transpose_x(const double* B, int naux, int64_t n2, double* Bt,
                               cudaStream_t st) {
  dim3 grid((unsigned)((n2 + 31) / 32), (unsigned)((naux + 31) / 32));
  transpose_x<<<grid, dim3(32, 8), 0, st>>>(B, naux, n2, Bt);
  return cudaGetLastError();
}

cudaError_t launch_get_diag(const double* A, int n, double* d, cudaStream_t st) {
  get_diag<<<grid_n(n), 256, 0, st>>>(A, n, d);
  return cudaGetLastError();
}

cudaError_t launch_gather_rows_f64(const double* VT, int n, const int* rows, int nk, double* out,
                                   cudaStream_t st) {
  if (nk <= 0) return cudaSuccess;
  gather_rows<<<grid_n((int64_t)nk * n), 256, 0, st>>>(VT, n, rows, nk, out);
  return cudaGetLastError();
}

cudaError_t launch_unpack_pairs(const double* J, int nx, int n, double* B, cudaStream_t st) {
  if (nx <= 0) return cudaSuccess;
  unpack_pairs<<<grid_n((int64_t)nx * n * n), 256, 0, st>>>(J, nx, n, B);
  return cudaGetLastError();
}

cudaError_t launch_asym_count(const double* B, int naux, int n, unsigned int* count,
                              cudaStream_t st) {
  const int t = (n + 31) / 32;
  asym_count<<<dim3(t, t, std::min(naux, 64)), dim3(32, 8), 0, st>>>(B, naux, n, count);
  return cudaGetLastError();
}

}  // namespace lno
