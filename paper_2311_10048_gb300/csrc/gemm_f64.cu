// Plain float64 contractions on the CUDA cores (the FP64 comparator path).
//
// One launch evaluates a group of independent problems, each
//   XT[n][m] = sum_seg sign_seg * sum_{k < K_seg} A_seg[m][k] * B_seg[n][k]
// (both operands K-contiguous, output stored transposed so that the m index
// is contiguous).  This is the per-triplet W contraction of eq cim_pt_energy
// with the particle and hole sums of one occupied permutation concatenated
// along k, and also the DF assembly (pq|rs) = sum_Q B^Q_pq B^Q_rs.
// Bound by the float64 pipe: 2 multiply-adds per clock and SM, so one 64 x 64 x
// 120 tile keeps an SM for 128 us and the launch lasts as long as the SM with the
// most of them.  The tile edge T (64, 32 or 16; 16 x 16 threads with T / 16 rows
// and columns each) is the one that leaves the fullest SM least (launch_gemm_f64).
// 40/6/4 domain: contractions 8.5 ms with 64 x 64 tiles only.
#include <algorithm>

#include "common.cuh"

namespace lno {

namespace {

constexpr int BK = 16;

// SYM: both operands are the same and only tiles on or below the diagonal run;
// each value is also stored at its mirrored place.
template <int T, bool SYM>
__global__ void __launch_bounds__(256)
gemm_f64_grouped(const ProbF64* __restrict__ probs, int M, int N, int ldo) {
  constexpr int R = T / 16;
  if (SYM && blockIdx.x > blockIdx.y) return;
  __shared__ double As[BK][T + 1];
  __shared__ double Bs[BK][T + 1];
  const ProbF64& P = probs[blockIdx.z];
  const int m0 = blockIdx.y * T, n0 = blockIdx.x * T;
  const int tid = threadIdx.x;
  const int tm = tid % 16, tn = tid / 16;
  double acc[R][R];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) acc[a][b] = 0.0;

  for (int s = 0; s < P.nseg; ++s) {
    const SegF64 sg = P.seg[s];
    for (int k0 = 0; k0 < sg.K; k0 += BK) {
      const int k = k0 + tm;   // loader: 16 consecutive k of a row per 16 threads
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int row = r * 16 + tn;
        const int m = m0 + row, n = n0 + row;
        As[tm][row] = m < M && k < sg.K ? sg.sign * sg.A[(int64_t)m * sg.lda + k] : 0.0;
        Bs[tm][row] = n < N && k < sg.K ? sg.B[(int64_t)n * sg.ldb + k] : 0.0;
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        double av[R], bv[R];
#pragma unroll
        for (int a = 0; a < R; ++a) av[a] = As[kk][tm * R + a];
#pragma unroll
        for (int b = 0; b < R; ++b) bv[b] = Bs[kk][tn * R + b];
#pragma unroll
        for (int a = 0; a < R; ++a)
#pragma unroll
          for (int b = 0; b < R; ++b) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int b = 0; b < R; ++b) {
    const int n = n0 + tn * R + b;
    if (n >= N) continue;
#pragma unroll
    for (int a = 0; a < R; ++a) {
      const int m = m0 + tm * R + a;
      if (m >= M) continue;
      P.XT[(int64_t)n * ldo + m] = acc[a][b];
      if (SYM && blockIdx.x < blockIdx.y) P.XT[(int64_t)m * ldo + n] = acc[a][b];
    }
  }
}

constexpr int kSMs = 152;

// Multiply-adds (in units of one k) of the SM that gets the most tiles, weighted
// by what the smaller tiles lose to loads and barriers.
double fullest_sm(int T, int nprob, int M, int N, bool sym, double weight) {
  int64_t tiles = (int64_t)ceil_div(M, T) * ceil_div(N, T);
  if (sym) tiles = (tiles + ceil_div(M, T)) / 2;
  return (double)((tiles * nprob + kSMs - 1) / kSMs) * T * T * weight;
}

template <bool SYM>
cudaError_t launch(const ProbF64* probs_dev, int nprob, int M, int N, int ldo, cudaStream_t st) {
  if (nprob <= 0 || M <= 0 || N <= 0) return cudaSuccess;
  const double c64 = fullest_sm(64, nprob, M, N, SYM, 1.0),
               c32 = fullest_sm(32, nprob, M, N, SYM, 1.04),
               c16 = fullest_sm(16, nprob, M, N, SYM, 1.2);
  int T = c64 <= std::min(c32, c16) ? 64 : c32 <= c16 ? 32 : 16;
  while (T < 64 && ceil_div(M, T) > 65535) T *= 2;
  const dim3 grid(ceil_div(N, T), ceil_div(M, T), nprob);
  if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
  if (T == 64)
    gemm_f64_grouped<64, SYM><<<grid, 256, 0, st>>>(probs_dev, M, N, ldo);
  else if (T == 32)
    gemm_f64_grouped<32, SYM><<<grid, 256, 0, st>>>(probs_dev, M, N, ldo);
  else
    gemm_f64_grouped<16, SYM><<<grid, 256, 0, st>>>(probs_dev, M, N, ldo);
  return cudaGetLastError();
}

}  // namespace

// probs: device array of nprob problems sharing M, N and the output pitch.
cudaError_t launch_gemm_f64(const ProbF64* probs_dev, int nprob, int M, int N,
                            int ldo, cudaStream_t st) {
  return launch<false>(probs_dev, nprob, M, N, ldo, st);
}

// One problem whose A and B segments are the same rows: half of the tiles.
cudaError_t launch_gemm_f64_sym(const ProbF64* prob_dev, int N, int ldo, cudaStream_t st) {
  return launch<true>(prob_dev, 1, N, N, ldo, st);
}

}  // namespace lno
