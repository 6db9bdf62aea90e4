// Host driver of the C ABI declared in include/lno_ot.h.
//
// One domain (eq cim_pt_energy, spin cases aaa, aab, abb, bbb):
//  1. stage: validate, lay the DF factors out as K-contiguous blocks
//     (occ-occ, occ-vir, vir-vir rows, Q fastest), assemble (ia|jb);
//  2. per spin s: assemble the DF integrals and build the K-concatenated
//     contraction operands AT, BT (same spin) and A1, BG, BF, AT2 (mixed,
//     spin s twice and the other spin once), see pack.cu;
//  3. per group of triplets: one grouped contraction launch writes X (same
//     spin) or Y and Z' (mixed) per triplet, one energy launch assembles W,
//     V and sums W (W + V) / D per triplet (energy.cu);
//  4. per-triplet sums -> per-case compensated sums -> host.
// Precision FP64 runs every contraction on the CUDA cores in float64; the others
// run them on the tensor cores on 16-bit or TF32 slices of the float64 operands
// (tc_pair.cu), with float64 kept for orbital energies and sums.
#include <algorithm>
#include <cstdlib>
#include <chrono>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <numeric>
#include <string>
#include <vector>

#include "common.cuh"

namespace lno {
// gemm_f64.cu
cudaError_t launch_gemm_f64(const ProbF64* probs_dev, int nprob, int M, int N, int ldo,
                            cudaStream_t st);
// energy.cu
cudaError_t launch_energy(const EnergyArgs& a, const void* X, const void* Z, bool f64, int ntrip,
                          int nchunks, cudaStream_t st);
cudaError_t launch_energy_f32(const EnergyArgs& a, const float* X, const float* Z, float* vtab,
                              int64_t vt_stride, int pv, int pvt, int ntrip, int nchunks,
                              cudaStream_t st);
cudaError_t launch_energy_f32_fused(const EnergyArgs& a, const float* X, const float* Z,
                                   float* vtab, int64_t vt_half, int pv, int pvt, int ntrip,
                                   int nchunks, cudaStream_t st);
cudaError_t launch_reduce_partials(const double* partial, int np, const double* partial2,
                                   int ntrip, double* e_trip, cudaStream_t st);
cudaError_t launch_orbital_partition(const OrbPartArgs& A, cudaStream_t st);
cudaError_t launch_case_sums(const CaseSums& A, cudaStream_t st);
cudaError_t energy_timeout_selftest(long long wait_cycles, int nsm, int* code, cudaStream_t st);
// pack.cu
template <class St>
cudaError_t launch_transpose_blocks(const double*, int, int, const BlockList<St>&, cudaStream_t);
template <class St>
cudaError_t launch_pack_at_same(const int2*, int, int, int, int, int, const double*, const double*,
                                St, cudaStream_t);
template <class St>
cudaError_t launch_pack_bt_same(int, int, int, int, int, int, int, const double*, const double*,
                                St, cudaStream_t);
template <class St>
cudaError_t launch_pack_a1(const int2*, int, int, int, int, int, int, int, const double*,
                           const double*, St, cudaStream_t);
template <class St>
cudaError_t launch_pack_bg(int, int, int, int, int, int, int, int, int, const double*,
                           const double*, St, cudaStream_t);
template <class St>
cudaError_t launch_pack_bf(int, int, int, int, int, int, int, int, int, const double*,
                           const double*, St, cudaStream_t);
template <class St>
cudaError_t launch_pack_at2(const int2*, int, int, int, int, int, int, int, const double*,
                            const double*, St, cudaStream_t);
cudaError_t launch_transpose_t2ab(const double*, int, int, int, int, double*, cudaStream_t);
cudaError_t launch_absmax(const double*, int64_t, unsigned long long*, cudaStream_t);
cudaError_t launch_absmax_list(const AbsmaxList& L, cudaStream_t s);
cudaError_t launch_row_norm2(const void* p, int64_t rows, int Kp, unsigned long long* out,
                             cudaStream_t s);
cudaError_t launch_view_absmax(const double* in, int64_t rs, int64_t ks, int rows, int K,
                               unsigned long long* out, cudaStream_t s);
cudaError_t launch_sum_partials(const double* part, int nsp, int M, int N, double* C,
                                int64_t ldc, bool accum, cudaStream_t s);
template <int S>
cudaError_t launch_view_slices(const double* in, int64_t rs, int64_t ks, int rows, int K,
                               int Kp, __nv_bfloat16* out, int64_t slice_stride, double inv,
                               cudaStream_t s);
cudaError_t launch_batch_slices(const double* src, int64_t src_stride, int count, int rows,
                                int cols, int ld, unsigned long long* amax, int* e, int* flag,
                                __nv_bfloat16* dn, int Kd, int64_t stride_n, __nv_bfloat16* dt,
                                int Nd, int64_t stride_t, cudaStream_t s);
cudaError_t launch_t2ab_flip_mismatch(const double* t2ab, int n, int v, double tol,
                                     unsigned int* count, cudaStream_t s);
cudaError_t launch_gather_rows(const void* src, void* dst, const int* list, int nlist,
                               int64_t row_bytes, int nslice, int64_t src_slice_bytes,
                               int64_t dst_slice_bytes, cudaStream_t s);
cudaError_t launch_scatter_add_rows(const double* src, double* dst, const int* list, int nlist,
                                    int64_t row, cudaStream_t s);
// naf.cu
int jacobi_eigh(double* A, double* A2, double* VT, int n, double* norms, cudaStream_t st,
                int max_sweeps);
size_t jacobi_norm_doubles();
cudaError_t launch_unpack_pairs(const double* J, int nx, int n, double* B, cudaStream_t st);
cudaError_t launch_asym_count(const double* B, int naux, int n, unsigned int* count,
                              cudaStream_t st);
cudaError_t launch_gemm_f64_sym(const ProbF64* prob_dev, int N, int ldo, cudaStream_t st);
cudaError_t launch_pack_pairs(const double* B, int naux, int n, double* J, cudaStream_t st);
cudaError_t launch_transpose_x(const double* B, int naux, int64_t n2, double* Bt,
                               cudaStream_t st);
cudaError_t launch_get_diag(const double* A, int n, double* d, cudaStream_t st);
cudaError_t launch_gather_rows_f64(const double* VT, int n, const int* rows, int nk, double* out,
                                   cudaStream_t st);
// backward.cu
struct GemmS {
  const double* A;
  const double* B;
  double* C;
  int M, N, K;
  int atomic;
  int64_t sam, sak, sbk, sbn, scm, scn;
  double alpha;
};
cudaError_t launch_gemm_strided(const GemmS* probs_dev, int nprob, int maxM, int maxN,
                                cudaStream_t st);
cudaError_t launch_energy_backward(const EnergyArgs& a, const double* X, const double* Z,
                                   double* dX, double* dZ, double* dt1s, double* dt1t,
                                   double* dov_ss, double* dov_ts, double* deps_s,
                                   double* deps_t, double gscale, int ntrip, int nchunks,
                                   cudaStream_t st);
cudaError_t launch_adj_at_same(const int2*, int, int, int, int, const double*, double*, double*,
                               cudaStream_t);
cudaError_t launch_adj_bt_same(int, int, int, int, int, const double*, double*, double*,
                               cudaStream_t);
cudaError_t launch_adj_a1(const int2*, int, int, int, int, int, int, const double*, double*,
                          double*, cudaStream_t);
cudaError_t launch_adj_bg(int, int, int, int, int, int, int, const double*, double*, double*,
                          cudaStream_t);
cudaError_t launch_adj_bf(int, int, int, int, int, int, int, const double*, double*, double*,
                          cudaStream_t);
cudaError_t launch_adj_at2(const int2*, int, int, int, int, int, int, const double*, double*,
                           double*, cudaStream_t);
cudaError_t launch_adj_transpose_block(const double*, int, int, int, int, int, int, int, double*,
                                       cudaStream_t);
cudaError_t launch_sym_project(const double*, int, int, double, double*, cudaStream_t);
cudaError_t launch_antisym_project(const double*, int, int, double, double*, cudaStream_t);
cudaError_t launch_adj_transpose_t2ab(const double*, int, int, int, int, double*, cudaStream_t);
cudaError_t launch_scale_copy(const double*, int64_t, double, double*, cudaStream_t);
cudaError_t launch_sym_inplace(double*, int, int, cudaStream_t);
cudaError_t launch_antisym_inplace(double*, int, int, cudaStream_t);
}  // namespace lno

using namespace lno;

// ----------------------------------------------------------------------------
static thread_local std::string g_last_error;

void lno_set_last_error(const char* what, cudaError_t e, const char* file, int line) {
  char buf[512];
  snprintf(buf, sizeof buf, "%s failed: %s (%s:%d)", what, cudaGetErrorString(e), file, line);
  g_last_error = buf;
}

struct lno_ot_ctx {
  int device = 0;
  int prec = LNO_OT_FP64;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  size_t ws_limit = 0;
  int nsm = 152;
  // tuning table: per virtual-space size bucket (rows of the contraction,
  // ascending vmax) a cap on the contraction tile's width (0 = none) and the
  // triplet-group cap
  struct TuneRow {
    int vmax, bn, group_cap;
  };
  std::vector<TuneRow> tune;
  const TuneRow* tune_for(int v) const {
    for (const TuneRow& r : tune)
      if (v <= r.vmax) return &r;
    return tune.empty() ? nullptr : &tune.back();
  }
  // one device block (CallState), read back in one copy at the end of a call
  double* d_sums = nullptr;                 // [4] per-case sums
  unsigned long long* d_amax = nullptr;     // magnitudes (bits of doubles)
  int* d_flag = nullptr;                    // error flag (bounded waits)
  lno_ot_stats stats{};
  std::vector<cudaEvent_t> ev_pool;
  size_t ev_used = 0;
  // Host-to-device copy of descriptors and lists, from pageable memory: the driver
  // carries small ones with the command stream (measured 5% of a small call faster
  // than a pinned source, whose copies wait for the copy engine one by one).
  cudaError_t h2d(void* dst, const void* src, size_t n) {
    return n ? cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, stream) : cudaSuccess;
  }
  bool exact_measure = false;          // integral scale from every slice (measure_sigI)
  bool no_f16 = false;                 // BF16X10 on its BF16 slices only (kNoF16)
  bool frugal = false;                 // the call runs again after the device ran out of memory
  bool small_pieces = false;           // every call does (lno_ot_selftest_small_pieces)
  // prepared operands of the last domain (options.keep_operands)
  bool keep = false;
  struct DomainCache* cache = nullptr;
};

void destroy_cache(DomainCache* c);

namespace {

// Device state of a call: per-case sums, magnitudes (0, 1 scratch, 2 the largest
// DF integral assembled with the current scale; squared row norms of FP16
// operands: of the DF blocks per spin, of AT, BT, A1, BG, BF, AT2), error flag.
constexpr int kNormB = 4, kNormW = 8, kAmaxSlots = 16;
struct CallState {
  double sums[4];
  unsigned long long amax[kAmaxSlots];
  int flag;
};

// Internal codes, the call has to run again: with the integral scale measured in
// full (scale_too_small), or without FP16 slices (class 0 of the DF products not
// provably exact; known before any contraction).
constexpr int kRescale = 1, kNoF16 = 2;

// Precision BF16X10 runs on three FP16 slices of 11 bits (6 slice products
// instead of 10) for domains of at least
// kF16MinVirtuals virtual orbitals per spin and kF16MinOccupied occupied ones, or
// of kF16WideVirtuals virtuals whatever they occupy.  200/20/18 domain: whole
// call 600 -> 436 ms, error against float64 slightly smaller.  Where the line
// lies: the two slicings' triplet energies differ by the coarser one's error,
// ~1e-9 (100 / v)^1.5 of a triplet's energy (measured 1.0e-9 at 100 virtuals,
// 4.2e-10 at 180, 1.6e-10 at 360), and a precision keeps its results: the rule
// holds that to half of 1e-9 for cases of many triplets and to a quarter for
// single ones.  Smaller domains spend little of a call in the contraction.
// Amplitudes use 10 bits of their leading slice: 32 bits of each operand's
// largest magnitude for them and 33 for integrals (BF16: 32 and 32), dropped slice
// products of at most 2 x 2^-32 of the largest product (BF16: 3 x 2^-32), and
// leading sums half as large (kExactSum).
constexpr int kF16MinVirtuals = 160, kF16MinOccupied = 8, kF16WideVirtuals = 256;
bool f16_sizes(const int* nvir, const int* nocc) {
  const int v = std::min(nvir[0], nvir[1]);
  return v >= kF16WideVirtuals ||
         (v >= kF16MinVirtuals && std::min(nocc[0], nocc[1]) >= kF16MinOccupied);
}
// FP32 sums of integers are exact while no partial sum exceeds 2^24: by
// Cauchy-Schwarz the product of the leading slices' row norms bounds every sum of
// class 0 (on the BF16 slices class g is exact for any data to K = 1024 / (g + 1)).
// Classes 1 and 2 are not checked: their digits run over +-1024 whatever the data,
// so a sum may pass 2^24 and lose its last bits there, 2^-11 or 2^-22 of class 0's
// unit each.  By estimate that is 1/20 of what the dropped products leave for K =
// 1200 factors of mixed signs, and about as much as those for factors of one sign
// and size throughout; per-triplet errors against float64 are those of the BF16
// slices (sd 4e-11 to 9e-11 Eh at 160 to 290 virtuals, worst 2e-10 to 5e-10 up to 360).
// 0.999: the norms' own rounding.
constexpr double kExactSum = 16777216.0 * 0.999;

#define TRY(expr)                       \
  do {                                  \
    int rc__ = (expr);                  \
    if (rc__ != LNO_OT_OK) return rc__; \
  } while (0)

// Stream-ordered device allocations released at scope exit.
struct Arena {
  cudaStream_t st;
  size_t limit, used = 0;
  struct Block {
    void* p;
    size_t bytes;
  };
  std::vector<Block> ptrs;
  Arena(cudaStream_t s, size_t lim) : st(s), limit(lim) {}
  ~Arena() { release(); }
  void release() {
    for (const Block& b : ptrs) cudaFreeAsync(b.p, st);
    ptrs.clear();
    used = 0;
  }
  template <typename T>
  static size_t bytes_of(size_t n) {
    return (std::max<size_t>(n * sizeof(T), 256) + 255) / 256 * 256;
  }
  template <typename T>
  int get(T** out, size_t n) {
    const size_t bytes = bytes_of<T>(n);
    if (limit && used + bytes > limit) return LNO_OT_ENOMEM;
    void* p = nullptr;
    if (cudaMallocAsync(&p, bytes, st) != cudaSuccess) {
      cudaGetLastError();
      return LNO_OT_ENOMEM;
    }
    ptrs.push_back({p, bytes});
    used += bytes;
    *out = static_cast<T*>(p);
    return LNO_OT_OK;
  }
  void drop(void* p) {
    for (auto& q : ptrs)
      if (q.p == p) {
        cudaFreeAsync(p, st);
        used -= q.bytes;
        q = ptrs.back();
        ptrs.pop_back();
        return;
      }
  }
};

int cuda_rc(cudaError_t e, const char* what) {
  if (e == cudaSuccess) return LNO_OT_OK;
  lno_set_last_error(what, e, __FILE__, __LINE__);
  cudaGetLastError();
  return LNO_OT_ECUDA;
}
#define CU(...) TRY(cuda_rc((__VA_ARGS__), #__VA_ARGS__))

int64_t pow2ceil_exp(double x) {  // smallest e with 2^e >= x (x > 0)
  int e;
  double m = std::frexp(x, &e);    // x = m 2^e, m in [0.5, 1)
  return (m == 0.5) ? e - 1 : e;
}

double pow2_scale(double amax) {
  if (!(amax > 0.0) || !std::isfinite(amax)) return 1.0;
  return std::ldexp(1.0, (int)pow2ceil_exp(amax));
}

// K-concatenated operand tensor: nslot slots of `rows` rows, pitch Kp.
struct Operand {
  int nslot = 0;
  int64_t rows = 0;  // rows per slot
  int K = 0, Kp = 0;
  double* f64 = nullptr;
  __nv_bfloat16* bf = nullptr;   // BF16 slices
  float* f32 = nullptr;          // TF32 slices (stored as float)
  int esz = 2;                   // bytes per slice element
  int S = 0;
  int64_t slice_stride = 0;
  int64_t total_rows() const { return (int64_t)nslot * rows; }
  // TMA map of the pair kernel: boxes of box_rows rows x the first ns slices
  // (0: all)
  int pair_map(CUtensorMap* m, int box_rows, int ns = 0) const {
    return make_operand_map(m, esz == 4 ? (const void*)f32 : (const void*)bf, Kp,
                            std::max<int64_t>(total_rows(), 1), S, slice_stride, box_rows, esz,
                            ns > 0 ? ns : S);
  }
};

// One grouped W-contraction launch with float32 output XT[n][m] (pitch ldo)
// = sum_seg A_seg[m] . B_seg[n], m < M the virtual index of the A operands, n
// < N the (pair) rows of the B operands.  The kernel runs it row-major with
// the roles exchanged: its row tiles run over the N rows (a long dimension, so
// they are full) and its n-tiles over the M rows.  seg_tc stores the segments
// with the roles already exchanged.  bn > 0 caps the tile width.
cudaError_t launch_contract(int S, int fmt, int bn, const Operand& A0, const Operand& A1,
                            const Operand& B0, const Operand& B1, const TcProb* dpt, int nprob,
                            int M, int N, int ldo, double scale, int* flag, int nsm,
                            cudaStream_t st, TcOut lay) {
  std::swap(M, N);
  const PairTile t = pair_tile(S, N, bn);
  CUtensorMap mA[2], mB[2];
  if (B0.pair_map(&mA[0], 128) || B1.pair_map(&mA[1], 128) || A0.pair_map(&mB[0], t.w / 2) ||
      A1.pair_map(&mB[1], t.w / 2))
    return cudaErrorInvalidValue;
#define LNO_CALL(SS, FF) \
  launch_tc_pair<SS, FF>(mA, mB, dpt, nprob, M, N, ldo, scale, flag, nsm, st, tc_normal(), lay, t)
  if (fmt == kFmtTF32) return LNO_CALL(2, kFmtTF32);
  if (fmt == kFmtF16) return LNO_CALL(3, kFmtF16);
  switch (S) {
    case 2: return LNO_CALL(2, kFmtBF16);
    case 3: return LNO_CALL(3, kFmtBF16);
    case 4: return LNO_CALL(4, kFmtBF16);
    default: return LNO_CALL(5, kFmtBF16);
  }
#undef LNO_CALL
}

// Strided float64 view: element (r, k) at p[r rs + k ks].
struct View {
  const double* p;
  int64_t rs, ks;
};
constexpr int64_t kMaxSplit = 64;   // K chunks of one tc_matmul
struct Run;
int tc_matmul(Run& R, Arena& A, int M, int N, int K, View a, View b, double* C, int64_t ldc,
              double alpha, bool accum, bool b_const = false);

// Slices of a read-only view kept by tc_matmul for the rest of a Run (the DF
// factor blocks that every slot's DF adjoint multiplies).
struct SliceCacheEntry {
  const double* p;
  int64_t rs, ks;
  int rows, K, Kc, nsp;
  __nv_bfloat16* q;
  double sigma;
};

struct Run {
  lno_ot_ctx* ctx;
  const lno_ot_domain* dom;
  cudaStream_t st;
  Arena arena;
  size_t held_back = 0;   // bytes that a bounded call takes of the arena after stage()
  bool f64;
  bool tf32 = false;  // W contraction operands as TF32 slices (precision TF32)
  bool f16 = false;   // precision BF16X10 on three FP16 slices (set_precision)
  bool tc_adjoint = false;  // adjoint: its contractions on the tensor cores (tc_matmul)
  int S = 0;          // slices of the W contraction operands
  int Sdf = 4;        // slices of the DF factors
  double sigT = 1, sigI = 1, sigB = 1;
  bool amax_pass = false;  // true while measuring integral magnitudes
  bool amax_exact = false; // ... with every slice of the factors
  bool track_amax = false; // while building the operands: their largest integral
  int nbas, naux, no[2], nv[2];
  // orbitals per spin: nbas, or nbas + P for a spin that carries P central
  // pseudo-orbitals (set before stage(); 0 = nbas)
  int nbs[2] = {0, 0};
  // occupied orbitals the internal (summed) indices run over: no[s] unless
  // pseudo-orbitals (central LMOs, Sec. 3.7) follow the real ones
  int noi[2] = {-1, -1};
  // Laplace quadrature point of the central-LMO pass (lap_w = 0: 1/D)
  double lap_s = 0.0, lap_w = 0.0;
  // DF factor blocks per spin (rows, K = naux); Boo rows are [internal][external]
  Operand Boo[2], Bov[2], Bvv[2];
  const double* fov[2] = {nullptr, nullptr};  // f_ov blocks (both or none)
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> contract_ev, energy_ev;
  std::vector<SliceCacheEntry> slice_cache;   // tc_matmul, read-only B views
  lno_ot_stats* stats;

  Run(lno_ot_ctx* c, const lno_ot_domain* d)
      : ctx(c), dom(d), st(c->stream), arena(c->stream, c->ws_limit), stats(&c->stats) {}

  cudaEvent_t event() {
    if (ctx->ev_used == ctx->ev_pool.size()) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
      ctx->ev_pool.push_back(e);
    }
    return ctx->ev_pool[ctx->ev_used++];
  }

  // ---- operand allocation -------------------------------------------------
  // tf: TF32 slices (the W operands of precision TF32); DF blocks are BF16.
  // pitch: multiple of the row pitch in elements (0: the widest useful one).
  int alloc_operand(Arena& ar, Operand& op, int nslot, int64_t rows, int K, int S_,
                    bool tf = false, int pitch = 0) {
    op.nslot = nslot;
    op.rows = rows;
    op.K = K;
    // sliced rows start on 64-byte boundaries: the contractions' 64-byte box
    // rows then are two sectors of L2 (1.3x fewer bytes than at 16-byte pitches)
    if (pitch == 0) pitch = f64 || tf ? 16 : 32;
    op.Kp = (int)round_up(std::max(K, 1), pitch);
    op.S = f64 ? 0 : S_;
    const int64_t n = std::max<int64_t>((int64_t)nslot * rows * op.Kp, 8);
    if (f64) {
      TRY(ar.get(&op.f64, (size_t)n));
    } else {
      op.slice_stride = round_up(n, 8);
      if (tf) {
        op.esz = 4;
        TRY(ar.get(&op.f32, (size_t)(op.slice_stride * op.S)));
      } else {
        op.esz = 2;
        TRY(ar.get(&op.bf, (size_t)(op.slice_stride * op.S)));
      }
    }
    return LNO_OT_OK;
  }

  // Store functor for an operand (amplitude scale sigT, integral scale sigI).
  template <int SS>
  StoreSlices<SS> slices(const Operand& op) const {
    return StoreSlices<SS>{op.bf, op.slice_stride, 7 - std::ilogb(sigT), 7 - std::ilogb(sigI)};
  }
  StoreTF32<2> tf32_slices(const Operand& op) const {
    return StoreTF32<2>{op.f32, op.slice_stride, 10 - std::ilogb(sigT), 10 - std::ilogb(sigI)};
  }
  StoreSlices<3, __half> f16_slices(const Operand& op) const {
    return StoreSlices<3, __half>{reinterpret_cast<__half*>(op.bf), op.slice_stride,
                                  9 - std::ilogb(sigT), 10 - std::ilogb(sigI)};
  }

  // Largest squared row norm of the leading (integer) slice of an FP16 operand.
  int row_norm2(const Operand& op, int slot) {
    stats->other_launches++;
    CU(launch_row_norm2(op.bf, op.total_rows(), op.Kp, ctx->d_amax + slot, st));
    return LNO_OT_OK;
  }

  // ---- DF integrals: out[n][m] = sum_Q L[m][Q] R[n][Q] (float64) ------------
  // L rows [l0, l0+M) of operand Lo, R rows [r0, r0+N) of Ro.
  int df(const Operand& Lo, int64_t l0, int M, const Operand& Ro, int64_t r0, int N, double* out,
         int ldo) {
    if (M <= 0 || N <= 0) return LNO_OT_OK;
    stats->other_launches++;
    if (f64 && tc_adjoint)   // adjoint of a tensor-core precision: float64 blocks, TC product
      return tc_matmul(*this, arena, N, M, naux, View{Ro.f64 + r0 * Ro.Kp, Ro.Kp, 1},
                       View{Lo.f64 + l0 * Lo.Kp, Lo.Kp, 1}, out, ldo, 1.0, false);
    if (f64) {
      ProbF64 p{};
      p.nseg = 1;
      p.seg[0] = SegF64{Lo.f64 + l0 * Lo.Kp, Ro.f64 + r0 * Ro.Kp, naux, Lo.Kp, Ro.Kp, 1.0};
      p.XT = out;
      ProbF64* dp;
      TRY(arena.get(&dp, 1));
      CU(ctx->h2d(dp, &p, sizeof p));
      CU(launch_gemm_f64(dp, 1, M, N, ldo, st));
      return LNO_OT_OK;
    }
    TcProb p{};
    p.nseg = 1;
    p.seg[0] = TcSeg{0, 0, (int)l0, (int)r0, naux, 0};
    p.out = amax_pass ? nullptr : out;
    const double scale = sigB * sigB * std::ldexp(1.0, f16 ? -20 : -14);
    // the measuring pass takes the two leading slices of each factor (3 of the 10
    // products) unless that leaves the scale open (measure_sigI)
    const int ns = amax_pass && !amax_exact ? 2 : Sdf;
    unsigned long long* am = amax_pass ? ctx->d_amax : track_amax ? ctx->d_amax + 2 : nullptr;
    const PairTile t = pair_tile_f64(ns, 1, M, N);
    CUtensorMap mA[2], mB[2];
    TRY(Lo.pair_map(&mA[0], 128, ns));
    TRY(Ro.pair_map(&mB[0], t.w / 2, ns));
    mA[1] = mA[0];
    mB[1] = mB[0];
#define LNO_DF(SS, FF)                                                                        \
  CU((launch_tc_pair_f64<SS, FF>(mA, mB, p, M, N, ldo, scale, ctx->d_flag, am, ctx->nsm, st, t)))
    if (f16) {
      if (ns == 2) LNO_DF(2, kFmtF16);
      else LNO_DF(3, kFmtF16);
    } else if (ns == 2) {
      LNO_DF(2, kFmtBF16);
    } else if (ns == 5) {
      LNO_DF(5, kFmtBF16);
    } else {
      LNO_DF(4, kFmtBF16);
    }
#undef LNO_DF
    return LNO_OT_OK;
  }

  // ---- stage ----------------------------------------------------------------
  int stage() {
    nbas = dom->nbas;
    naux = dom->naux;
    for (int s = 0; s < 2; ++s) {
      if (nbs[s] <= 0) nbs[s] = nbas;
      no[s] = dom->nocc[s];
      nv[s] = nbs[s] - no[s];
      if (noi[s] < 0 || noi[s] > no[s]) noi[s] = no[s];
    }
    if (!f64) {  // global scales of B and T2
      CU(cudaMemsetAsync(ctx->d_amax, 0, 2 * sizeof(unsigned long long), st));
      AbsmaxList L{};
      auto measure = [&](const double* x, int64_t n, int slot) {
        if (n == 0) return;
        L.x[L.count] = x;
        L.n[L.count] = n;
        L.out[L.count++] = ctx->d_amax + slot;
      };
      for (int s = 0; s < 2; ++s) measure(dom->B[s], (int64_t)naux * nbs[s] * nbs[s], 0);
      measure(dom->t2aa, (int64_t)no[0] * no[0] * nv[0] * nv[0], 1);
      measure(dom->t2bb, (int64_t)no[1] * no[1] * nv[1] * nv[1], 1);
      measure(dom->t2ab, (int64_t)no[0] * no[1] * nv[0] * nv[1], 1);
      CU(launch_absmax_list(L, st));
      double h[2];
      CU(cudaMemcpyAsync(h, ctx->d_amax, sizeof h, cudaMemcpyDeviceToHost, st));
      CU(cudaStreamSynchronize(st));
      sigB = pow2_scale(h[0]);
      sigT = pow2_scale(h[1]);
      stats->other_launches++;
    }
    if (dom->fov[0] || dom->fov[1]) {  // a missing spin block is zero
      for (int s = 0; s < 2; ++s) {
        if (dom->fov[s]) {
          fov[s] = dom->fov[s];
        } else {
          double* z;
          const size_t n = std::max<size_t>((size_t)no[s] * nv[s], 1);
          TRY(arena.get(&z, n));
          CU(cudaMemsetAsync(z, 0, n * sizeof(double), st));
          fov[s] = z;
        }
      }
    }
    return stage_blocks();
  }

  // the DF factor blocks in the present slice format
  int stage_blocks() {
    // Under a bound (workspace_bytes) rows have the 8-element pitch that the loads need
    // unless everything fits with the wide one, so that the bound admits as large a
    // domain as it can (366/8/6, naux 1000: whole call 245 ms wide, 263 ms at 8).
    int pitch = 0;
    if (arena.limit) {
      size_t wide = arena.used + held_back;
      for (int s = 0; s < 2; ++s)
        for (int64_t rows : {(int64_t)noi[s] * no[s], (int64_t)no[s] * nv[s],
                             (int64_t)nv[s] * nv[s]})
          wide += round_up(std::max<int64_t>(rows * round_up(naux, 32), 8) * Sdf * 2, 256);
      pitch = f64 || wide > arena.limit ? 8 : 0;
    }
    for (int s = 0; s < 2; ++s) {
      const int o = no[s], oi = noi[s], v = nv[s];
      TRY(alloc_operand(arena, Boo[s], 1, (int64_t)oi * o, naux, Sdf, false, pitch));
      TRY(alloc_operand(arena, Bov[s], 1, (int64_t)o * v, naux, Sdf, false, pitch));
      TRY(alloc_operand(arena, Bvv[s], 1, (int64_t)v * v, naux, Sdf, false, pitch));
      Operand* ops[3] = {&Boo[s], &Bov[s], &Bvv[s]};
      const int p0[3] = {0, 0, o}, np[3] = {oi, o, v}, q0[3] = {0, o, o}, nq[3] = {o, v, v};
      const int eB = 7 - std::ilogb(sigB);
      auto layout = [&](auto&& store) {
        BlockList<std::decay_t<decltype(store(Boo[s]))>> L{};
        for (int k = 0; k < 3; ++k) {
          L.p0[k] = p0[k];
          L.np[k] = np[k];
          L.q0[k] = q0[k];
          L.nq[k] = nq[k];
          L.Qp[k] = ops[k]->Kp;
          L.st[k] = store(*ops[k]);
        }
        return launch_transpose_blocks(dom->B[s], naux, nbs[s], L, st);
      };
      stats->other_launches++;
      if (f64)
        CU(layout([&](const Operand& op) { return StoreF64{op.f64}; }));
      else if (f16)
        CU(layout([&](const Operand& op) {
          return StoreSlices<3, __half>{reinterpret_cast<__half*>(op.bf), op.slice_stride, eB + 3,
                                        eB + 3};
        }));
      else if (Sdf == 5)
        CU(layout([&](const Operand& op) {
          return StoreSlices<5>{op.bf, op.slice_stride, eB, eB};
        }));
      else
        CU(layout([&](const Operand& op) {
          return StoreSlices<4>{op.bf, op.slice_stride, eB, eB};
        }));
      if (f16) {
        CU(cudaMemsetAsync(ctx->d_amax + kNormB + s, 0, sizeof(unsigned long long), st));
        for (const Operand* op : {&Boo[s], &Bov[s], &Bvv[s]}) TRY(row_norm2(*op, kNormB + s));
      }
    }
    return LNO_OT_OK;
  }

  // From here on without FP16 slices: the DF blocks are laid out again.
  int leave_f16() {
    f16 = false;
    S = Sdf = 4;
    for (int s = 0; s < 2; ++s)
      for (Operand* op : {&Boo[s], &Bov[s], &Bvv[s]}) arena.drop(op->bf);
    return stage_blocks();
  }

  // dst slot q = src rows [dlist[q] * rows, (dlist[q] + 1) * rows): a DF block
  // restricted to some occupied orbitals (same slicing and scales as src)
  int gather_operand(Arena& ar, const Operand& src, const int* dlist, int nlist, int64_t rows,
                     Operand& dst) {
    TRY(alloc_operand(ar, dst, nlist, rows, src.K, Sdf, false, src.Kp));
    if (nlist == 0 || rows == 0) return LNO_OT_OK;
    stats->other_launches++;
    if (f64)
      CU(launch_gather_rows(src.f64, dst.f64, dlist, nlist, rows * src.Kp * 8, 1, 0, 0, st));
    else
      CU(launch_gather_rows(src.bf, dst.bf, dlist, nlist, rows * src.Kp * 2, src.S,
                            src.slice_stride * 2, dst.slice_stride * 2, st));
    return LNO_OT_OK;
  }
};

// ---- grouped products of the adjoint -----------------------------------------
// A batch of float64 matrices [rows][cols] as 4 BF16 slices in one or both
// layouts (launch_batch_slices), each matrix with its own power-of-two scale kept
// on the device: nothing waits for the host.
struct SlicedBatch {
  int count = 0, rows = 0, cols = 0, Kd = 0, Nd = 0;
  __nv_bfloat16 *n = nullptr, *t = nullptr;
  int64_t sn = 0, st = 0;
  int* e = nullptr;
  unsigned long long* amax = nullptr;
  static int64_t bytes(int64_t count, int64_t rows, int64_t cols, bool both) {
    return 8 * count * ((both ? rows * round_up(cols, 32) : 0) + cols * round_up(rows, 32));
  }
  int alloc(Arena& A, int count_, int rows_, int cols_, bool want_n, bool want_t) {
    count = count_;
    rows = rows_;
    cols = cols_;
    Kd = (int)round_up(cols, 32);
    Nd = (int)round_up(rows, 32);
    sn = (int64_t)count * rows * Kd;
    st = (int64_t)count * cols * Nd;
    if (want_n) TRY(A.get(&n, (size_t)(4 * sn)));
    if (want_t) TRY(A.get(&t, (size_t)(4 * st)));
    TRY(A.get(&e, (size_t)std::max(count, 1)));
    TRY(A.get(&amax, (size_t)std::max(count, 1)));
    return LNO_OT_OK;
  }
  int fill(Run& R, const double* src, int64_t stride, int ld, int ncount) {
    R.stats->other_launches += 3;
    CU(launch_batch_slices(src, stride, ncount, rows, cols, ld, amax, e, R.ctx->d_flag, n, Kd, sn,
                           t, Nd, st, R.st));
    return LNO_OT_OK;
  }
  int map(CUtensorMap* m, bool tr, int box) const {
    return tr ? make_operand_map(m, t, Nd, std::max<int64_t>((int64_t)count * cols, 1), 4, st, box,
                                 2, 4)
              : make_operand_map(m, n, Kd, std::max<int64_t>((int64_t)count * rows, 1), 4, sn, box,
                                 2, 4);
  }
};

// One launch of products 2^(ea + eb - 14) sum_k a[m][k] b[n][k], m < M, n < N, into
// out[n][m] (mode kOutRows) or out[m][n] (kOutF64Rows), over slices of two batches
// (ta, tb: their transposed layouts).  a takes the longer side: row tiles are 256.
int grouped_products(Run& R, Arena& A, const std::vector<TcProb>& pr, const SlicedBatch& a,
                     bool ta, const SlicedBatch& b, bool tb, int M, int N, int ldo, int mode) {
  if (pr.empty() || M <= 0 || N <= 0) return LNO_OT_OK;
  const PairTile t = pair_tile_f64(4, (int)pr.size(), M, N);
  CUtensorMap mA[2], mB[2];
  TRY(a.map(&mA[0], ta, 128));
  TRY(b.map(&mB[0], tb, t.w / 2));
  mA[1] = mA[0];
  mB[1] = mB[0];
  TcProb* dp;
  TRY(A.get(&dp, pr.size()));
  cudaEvent_t e0 = R.event(), e1 = R.event();
  if (e0) cudaEventRecord(e0, R.st);
  CU(R.ctx->h2d(dp, pr.data(), pr.size() * sizeof(TcProb)));
  CU((launch_tc_pair_f64_group<4, kFmtBF16>(mA, mB, dp, (int)pr.size(), M, N, ldo, 1.0,
                                            R.ctx->d_flag, R.ctx->nsm, R.st, mode, t)));
  if (e1) cudaEventRecord(e1, R.st);
  if (e0 && e1) R.contract_ev.push_back({e0, e1});
  R.stats->contract_launches++;
  A.drop(dp);
  return LNO_OT_OK;
}

// Problems of one product, its k range in chunks of at most `chunk`: enough
// problems for the device.  (Class 0 of a chunk is exact for any data to K = 1024
// and for random signs far beyond; a longer sum of one sign rounds at 2^-24 of
// itself, as the single products of tc_matmul do.)
void add_chunks(std::vector<TcProb>& out, int a_row, int b_row, int K, bool neg, double* dst,
                int flags, const int* ea, const int* eb, int chunk = 4096) {
  for (int k = 0; k < K; k += chunk) {
    TcProb p{};
    p.nseg = 1;
    p.seg[0] = TcSeg{0, 0, a_row, b_row, std::min(chunk, K - k), neg ? 1 : 0, k};
    p.flags = flags | kTcFloatRest;
    p.out = dst;
    p.ea = ea;
    p.eb = eb;
    out.push_back(p);
  }
}

// Several host arrays in one device buffer and one copy.
struct Upload {
  std::vector<char> blob;
  std::vector<std::pair<const void**, size_t>> dst;
  char* base = nullptr;   // the device buffer
  template <typename T>
  void add(const std::vector<T>& h, const T** d) {
    *d = nullptr;
    const size_t off = (blob.size() + 63) / 64 * 64;
    if (h.empty()) return;
    blob.resize(off + h.size() * sizeof(T));
    std::memcpy(blob.data() + off, h.data(), h.size() * sizeof(T));
    dst.push_back({reinterpret_cast<const void**>(d), off});
  }
  int send(Run& R, Arena& A) {
    if (blob.empty()) return LNO_OT_OK;
    TRY(A.get(&base, blob.size()));
    CU(R.ctx->h2d(base, blob.data(), blob.size()));
    for (auto& d : dst) *d.first = base + d.second;
    return LNO_OT_OK;
  }
};

// Spin-case triplet selection.
struct CaseSel {
  std::vector<Trip> trips;   // triplets to compute, in output order
  int64_t ntot = 0;          // all restricted triplets of the case
};

int64_t c2(int64_t n) { return n * (n - 1) / 2; }
int64_t c3(int64_t n) { return n * (n - 1) * (n - 2) / 6; }

Trip decode_triplet(int c, int64_t q, int na, int nb) {
  // lexicographic enumeration as in the header
  auto same = [](int64_t q, int n) {
    for (int i = 0; i < n; ++i)
      for (int j = i + 1; j < n; ++j) {
        int64_t cnt = n - j - 1;
        if (q < cnt) return Trip{i, j, (int)(j + 1 + q)};
        q -= cnt;
      }
    return Trip{-1, -1, -1};
  };
  auto mixed = [](int64_t q, int n2, int n1) {
    int64_t pairi = q / n1;
    int k = (int)(q % n1);
    for (int i = 0; i < n2; ++i) {
      int64_t cnt = n2 - i - 1;
      if (pairi < cnt) return Trip{i, (int)(i + 1 + pairi), k};
      pairi -= cnt;
    }
    return Trip{-1, -1, -1};
  };
  switch (c) {
    case 0: return same(q, na);
    case 3: return same(q, nb);
    case 1: return mixed(q, na, nb);
    default: return mixed(q, nb, na);
  }
}

int select_case(const lno_ot_domain* d, int c, CaseSel& cs) {
  const int na = d->nocc[0], nb = d->nocc[1];
  cs.ntot = c == 0 ? c3(na) : c == 3 ? c3(nb) : c == 1 ? c2(na) * nb : c2(nb) * na;
  cs.trips.clear();
  if (d->trip_sel[c]) {
    if (d->n_sel[c] < 0) return LNO_OT_EINVAL;
    cs.trips.reserve((size_t)d->n_sel[c]);
    for (int64_t q = 0; q < d->n_sel[c]; ++q) {
      int64_t id = d->trip_sel[c][q];
      if (id < 0 || id >= cs.ntot) return LNO_OT_EINVAL;
      cs.trips.push_back(decode_triplet(c, id, na, nb));
    }
  } else {
    // enumerate directly (fast path)
    if (c == 0 || c == 3) {
      const int n = c == 0 ? na : nb;
      for (int i = 0; i < n; ++i)
        for (int j = i + 1; j < n; ++j)
          for (int k = j + 1; k < n; ++k) cs.trips.push_back(Trip{i, j, k});
    } else {
      const int n2 = c == 1 ? na : nb, n1 = c == 1 ? nb : na;
      for (int i = 0; i < n2; ++i)
        for (int j = i + 1; j < n2; ++j)
          for (int k = 0; k < n1; ++k) cs.trips.push_back(Trip{i, j, k});
    }
  }
  return LNO_OT_OK;
}

double flops_alg_same(double v, double o) { return 3.0 * (2 * v * v * v * v + 2 * v * v * v * o); }
double flops_alg_mixed(double vs, double vt, double os, double ot) {
  return 4 * vs * vs * vt * vt + 6 * vs * vs * vs * vt + 4 * vs * vs * vt * ot + 6 * os * vs * vs * vt;
}
double kpad16(double k) { return std::ceil(k / 16.0) * 16.0; }

// Triplets per group where the tuning table says nothing: virtual spaces of ~100
// then reach the group's memory budget or have a case in a few launches.  At 64,
// launch gaps, each launch's last round of tiles and the energy kernel's items of
// one or two tiles (their number per triplet falls as the group grows) cost 20%:
// 121/14/11 domain 28.8 ms at 64, 24.6 at 256, 23.4 at 1024.
constexpr int kGroupCap = 1024;
// After an allocation failed (the device is shared, or nearly full) a call runs
// again in small pieces: groups of at most 64 triplets, DF blocks of one orbital,
// the adjoint's recompute and adjoint products one by one.  (Its DF assembly keeps
// the slices of a whole factor block: a single product would need them as well.)
constexpr int kFrugalGroup = 64;
// Triplets whose contraction problems are on the device at once (17 MB).
constexpr int kWindow = 65536;

// ----------------------------------------------------------------------------
// Per spin s: same-spin case (sss) and the mixed case with two s orbitals.
struct SpinPass {
  Run& R;
  int s, t;
  int o, v, ot, vt;
  int oi, oti;  // internal occupied ranges (== o, ot without pseudo-orbitals)
  CaseSel& same;   // case s==0 ? aaa : bbb
  CaseSel& mixed;  // case s==0 ? aab : abb
  double* e_same;  // per-triplet outputs (device)
  double* e_mixed;

  bool f16;                  // W operands as FP16 slices (prepare may refuse them)
  int S;                     // slices of the W operands
  Operand AT, BT, A1, BG, BF, AT2;
  std::vector<int> slotAT, slotBT, slotA1, slotBG, slotBF, slotAT2;  // -1 = unused
  std::vector<int2> listAT, listA1, listAT2;
  std::vector<int> listBT, listBG, listBF;
  int bn = 0;                // widest contraction tile of the current case (0 = default)
  int group_cap = kGroupCap; // triplets per group (upper bound)
  double* t2st = nullptr;    // [os][ot][vs][vt]
  const double* t2ss = nullptr;
  // V-term integrals over the occupied orbitals in use: spin-s slots are those
  // of listBT (every i, j, k of a computed triplet), spin-t slots those of
  // listBF (every K of a mixed triplet)
  Operand BsS, BsT;          // Bov rows of the slots, [slot][vir] x naux
  double* ovss = nullptr;    // (ia|jb) as [nS][vs][nS][vs]
  double* ovts = nullptr;    // (jb|KC) as [nT][vt][nS][vs]
  const int* d_slot_s = nullptr;   // occupied index -> slot (-1 absent), spin s [os]
  const int* d_slot_t = nullptr;   // spin t [ot]
  const int* d_list_s = nullptr;   // slot -> occupied index
  const int* d_list_t = nullptr;
  const int2 *d_AT = nullptr, *d_A1 = nullptr, *d_AT2 = nullptr;   // pair lists

  Arena own;  // operands and temporaries of this spin pass

  SpinPass(Run& r, int s_, CaseSel& sm, CaseSel& mx, double* es, double* em)
      : R(r), s(s_), t(1 - s_), same(sm), mixed(mx), e_same(es), e_mixed(em), f16(r.f16),
        S(r.S), own(r.st, 0) {
    o = R.no[s];
    v = R.nv[s];
    ot = R.no[t];
    vt = R.nv[t];
    oi = R.noi[s];
    oti = R.noi[t];
  }

  void plan() {
    listAT.clear();
    listA1.clear();
    listAT2.clear();
    listBT.clear();
    listBG.clear();
    listBF.clear();
    slotAT.assign((size_t)o * o, -1);
    slotBT.assign(o, -1);
    slotA1.assign((size_t)o * ot, -1);
    slotBG.assign(o, -1);
    slotBF.assign(ot, -1);
    slotAT2.assign((size_t)o * ot, -1);
    auto need_pair = [&](std::vector<int>& slot, std::vector<int2>& list, int p, int q, int w) {
      int& sl = slot[(size_t)p * w + q];
      if (sl < 0) {
        sl = (int)list.size();
        list.push_back(make_int2(p, q));
      }
    };
    auto need_one = [&](std::vector<int>& slot, std::vector<int>& list, int x) {
      if (slot[x] < 0) {
        slot[x] = (int)list.size();
        list.push_back(x);
      }
    };
    for (const Trip& tr : same.trips) {
      need_pair(slotAT, listAT, tr.j, tr.k, o);
      need_pair(slotAT, listAT, tr.k, tr.i, o);
      need_pair(slotAT, listAT, tr.i, tr.j, o);
      need_one(slotBT, listBT, tr.i);
      need_one(slotBT, listBT, tr.j);
      need_one(slotBT, listBT, tr.k);
    }
    for (const Trip& tr : mixed.trips) {
      need_pair(slotA1, listA1, tr.j, tr.k, ot);
      need_pair(slotA1, listA1, tr.i, tr.k, ot);
      need_one(slotBG, listBG, tr.i);
      need_one(slotBG, listBG, tr.j);
      need_pair(slotAT, listAT, tr.i, tr.j, o);
      need_one(slotBF, listBF, tr.k);
      need_pair(slotAT2, listAT2, tr.j, tr.k, ot);
      need_pair(slotAT2, listAT2, tr.i, tr.k, ot);
      need_one(slotBT, listBT, tr.i);
      need_one(slotBT, listBT, tr.j);
    }
  }

  // Runs of consecutive orbitals in a slot list: slots [q, q + n) hold orbitals
  // x, x + 1, ...; the DF blocks of a run come from one launch (their rows are
  // consecutive) and are laid out by one.  A run's float64 blocks stay within
  // kRunBytes, except a single block that is larger.
  struct OrbRun {
    int q, x, n;
  };
  static constexpr int64_t kRunBytes = (int64_t)512 << 20;
  static std::vector<OrbRun> orb_runs(const std::vector<int>& list, int64_t block_elems,
                                      bool frugal) {
    const int cap =
        frugal ? 1
               : (int)std::max<int64_t>(1, std::min<int64_t>(65535, kRunBytes / 8 /
                                                  std::max<int64_t>(block_elems, 1)));
    std::vector<OrbRun> runs;
    for (size_t q = 0; q < list.size(); ++q) {
      if (!runs.empty() && runs.back().n < cap && runs.back().x + runs.back().n == list[q])
        runs.back().n++;
      else
        runs.push_back({(int)q, list[q], 1});
    }
    return runs;
  }
  static int longest(const std::vector<OrbRun>& runs) {
    int n = 0;
    for (const OrbRun& r : runs) n = std::max(n, r.n);
    return n;
  }

  template <class St>
  int pack_all(St stAT, St stBT, St stA1, St stBG, St stBF, St stAT2) {
    Arena& A = own;
    cudaStream_t st = R.st;
    const bool meas = R.amax_pass;   // magnitudes only: no blocks, no layout
    R.track_amax = !meas;
    auto block = [&](double** p, int64_t n) -> int {
      *p = nullptr;
      return meas ? LNO_OT_OK : A.get(p, (size_t)n);
    };
    auto drop = [&](double* p) {
      if (p) A.drop(p);
    };
    // pair operands: one DF block, one layout launch
    // per-orbital operands: the blocks (L rows x [x][r_rows]) of a run at a time
    auto per_orbital = [&](const std::vector<int>& list, const Operand& L, int64_t l_rows,
                           const Operand& Ro, int r_rows, auto&& pack) -> int {
      const auto runs = orb_runs(list, l_rows * r_rows, R.ctx->frugal);
      double* buf;
      TRY(block(&buf, l_rows * r_rows * longest(runs)));
      // adjoint on the tensor cores: one launch per run as well, each orbital's rows
      // with their own scale
      SlicedBatch sL, sR;
      const bool sliced = R.tc_adjoint && R.naux <= kWideBF16 && !runs.empty() && l_rows > 0 &&
                          r_rows > 0;
      if (sliced) {
        const int norb = (int)(Ro.total_rows() / r_rows);
        TRY(sL.alloc(A, 1, (int)l_rows, R.naux, true, false));
        TRY(sL.fill(R, L.f64, 0, L.Kp, 1));
        TRY(sR.alloc(A, norb, r_rows, R.naux, true, false));
        TRY(sR.fill(R, Ro.f64, (int64_t)r_rows * Ro.Kp, Ro.Kp, norb));
      }
      for (const OrbRun& r : runs) {
        if (sliced) {
          std::vector<TcProb> pr;
          for (int i = 0; i < r.n; ++i)
            add_chunks(pr, 0, (r.x + i) * r_rows, R.naux, false, buf + i * l_rows * r_rows, 0,
                       sL.e, sR.e + r.x + i, R.naux);
          TRY(grouped_products(R, A, pr, sL, false, sR, false, (int)l_rows, r_rows, (int)l_rows,
                               kOutRows));
        } else {
          TRY(R.df(L, 0, (int)l_rows, Ro, (int64_t)r.x * r_rows, r.n * r_rows, buf, (int)l_rows));
        }
        if (!meas) {
          R.stats->other_launches++;
          CU(pack(r, buf));
        }
      }
      drop(buf);
      if (sliced)
        for (void* q : {(void*)sL.n, (void*)sL.e, (void*)sL.amax, (void*)sR.n, (void*)sR.e,
                        (void*)sR.amax})
          A.drop(q);
      return LNO_OT_OK;
    };
    // ---- same-spin operands -------------------------------------------------
    if (!listAT.empty()) {
      double* oovoT;
      TRY(block(&oovoT, (int64_t)o * v * oi * o));
      TRY(R.df(R.Boo[s], 0, oi * o, R.Bov[s], 0, o * v, oovoT, oi * o));
      if (!meas) {
        R.stats->other_launches++;
        CU(launch_pack_at_same(d_AT, (int)listAT.size(), o, oi, v, AT.Kp, t2ss, oovoT, stAT, st));
      }
      drop(oovoT);
    }
    TRY(per_orbital(listBT, R.Bvv[s], (int64_t)v * v, R.Bov[s], v,
                    [&](const OrbRun& r, const double* b) {
                      return launch_pack_bt_same(r.q, r.x, r.n, o, oi, v, BT.Kp, b, t2ss, stBT,
                                                 st);
                    }));
    // ---- mixed operands -----------------------------------------------------
    if (!listA1.empty()) {
      double* jT;
      TRY(block(&jT, (int64_t)o * v * oti * ot));
      TRY(R.df(R.Bov[s], 0, o * v, R.Boo[t], 0, oti * ot, jT, o * v));
      if (!meas) {
        R.stats->other_launches++;
        CU(launch_pack_a1(d_A1, (int)listA1.size(), o, v, ot, oti, vt, A1.Kp, t2st, jT, stA1, st));
      }
      drop(jT);
    }
    TRY(per_orbital(listBG, R.Bvv[t], (int64_t)vt * vt, R.Bov[s], v,
                    [&](const OrbRun& r, const double* b) {
                      return launch_pack_bg(r.q, r.x, r.n, o, v, ot, oti, vt, BG.Kp, b, t2st,
                                            stBG, st);
                    }));
    TRY(per_orbital(listBF, R.Bvv[s], (int64_t)v * v, R.Bov[t], vt,
                    [&](const OrbRun& r, const double* b) {
                      return launch_pack_bf(r.q, r.x, r.n, o, oi, v, ot, vt, BF.Kp, b, t2st, stBF,
                                            st);
                    }));
    if (!listAT2.empty()) {
      double* lT;
      TRY(block(&lT, (int64_t)ot * vt * oi * o));
      TRY(R.df(R.Boo[s], 0, oi * o, R.Bov[t], 0, ot * vt, lT, oi * o));
      if (!meas) {
        R.stats->other_launches++;
        CU(launch_pack_at2(d_AT2, (int)listAT2.size(), o, oi, v, ot, vt, AT2.Kp, t2st, lT, stAT2,
                           st));
      }
      drop(lT);
    }
    R.track_amax = false;
    return LNO_OT_OK;
  }

  int build_v_blocks() {
    const int nS = (int)listBT.size(), nT = (int)listBF.size();
    Upload up;
    up.add(slotBT, &d_slot_s);
    up.add(slotBF, &d_slot_t);
    up.add(listBT, &d_list_s);
    up.add(listBF, &d_list_t);
    up.add(listAT, &d_AT);
    up.add(listA1, &d_A1);
    up.add(listAT2, &d_AT2);
    TRY(up.send(R, own));
    const int64_t ns = (int64_t)nS * v;
    TRY(R.gather_operand(own, R.Bov[s], d_list_s, nS, v, BsS));
    TRY(own.get(&ovss, (size_t)std::max<int64_t>(ns * ns, 1)));
    TRY(R.df(BsS, 0, (int)ns, BsS, 0, (int)ns, ovss, (int)ns));
    if (!mixed.trips.empty()) {
      const int64_t nt = (int64_t)nT * vt;
      TRY(R.gather_operand(own, R.Bov[t], d_list_t, nT, vt, BsT));
      TRY(own.get(&ovts, (size_t)std::max<int64_t>(nt * ns, 1)));
      TRY(R.df(BsS, 0, (int)ns, BsT, 0, (int)nt, ovts, (int)ns));
    }
    return LNO_OT_OK;
  }

  void set_v_args(EnergyArgs& ea, bool is_mixed) const {
    ea.ovov_ss = ovss;
    ea.ovov_ts = ovts;
    ea.oslot_s = d_slot_s;
    ea.oslot_t = is_mixed ? d_slot_t : d_slot_s;
    ea.ns_c = (int)listBT.size();
    ea.nt_c = is_mixed ? (int)listBF.size() : ea.ns_c;
  }

  int prepare_inputs() {
    t2ss = s == 0 ? R.dom->t2aa : R.dom->t2bb;
    if (!mixed.trips.empty() && t2st == nullptr) {
      if (s == 0) {
        t2st = const_cast<double*>(R.dom->t2ab);
      } else {
        TRY(own.get(&t2st, (size_t)std::max<int64_t>((int64_t)o * ot * v * vt, 1)));
        R.stats->other_launches++;
        CU(launch_transpose_t2ab(R.dom->t2ab, ot, o, vt, v, t2st, R.st));
      }
    }
    return LNO_OT_OK;
  }

  // measure integral magnitudes (sliced path, first pass)
  int measure() {
    if (listAT.empty() && listBT.empty() && listA1.empty() && listBG.empty() && listBF.empty() &&
        listAT2.empty())
      return LNO_OT_OK;
    R.amax_pass = true;
    StoreF64 dummy{nullptr};
    int rc = pack_all(dummy, dummy, dummy, dummy, dummy, dummy);
    R.amax_pass = false;
    return rc;
  }

  int build() {
    const bool tf = R.tf32;
    TRY(R.alloc_operand(own, AT, (int)listAT.size(), v, v + oi, S, tf));
    TRY(R.alloc_operand(own, BT, (int)listBT.size(), npairs(v), v + oi, S, tf));
    TRY(R.alloc_operand(own, A1, (int)listA1.size(), v, vt + oti, S, tf));
    TRY(R.alloc_operand(own, BG, (int)listBG.size(), (int64_t)v * vt, vt + oti, S, tf));
    TRY(R.alloc_operand(own, BF, (int)listBF.size(), (int64_t)v * vt, v + oi, S, tf));
    TRY(R.alloc_operand(own, AT2, (int)listAT2.size(), vt, v + oi, S, tf));
    if (R.f64) return pack_all(StoreF64{AT.f64}, StoreF64{BT.f64}, StoreF64{A1.f64},
                               StoreF64{BG.f64}, StoreF64{BF.f64}, StoreF64{AT2.f64});
    if (tf)
      return pack_all(R.tf32_slices(AT), R.tf32_slices(BT), R.tf32_slices(A1),
                      R.tf32_slices(BG), R.tf32_slices(BF), R.tf32_slices(AT2));
    if (f16)
      return pack_all(R.f16_slices(AT), R.f16_slices(BT), R.f16_slices(A1), R.f16_slices(BG),
                      R.f16_slices(BF), R.f16_slices(AT2));
    if (S == 2)
      return pack_all(R.slices<2>(AT), R.slices<2>(BT), R.slices<2>(A1), R.slices<2>(BG),
                      R.slices<2>(BF), R.slices<2>(AT2));
    if (S == 4)
      return pack_all(R.slices<4>(AT), R.slices<4>(BT), R.slices<4>(A1), R.slices<4>(BG),
                      R.slices<4>(BF), R.slices<4>(AT2));
    if (S == 5)
      return pack_all(R.slices<5>(AT), R.slices<5>(BT), R.slices<5>(A1), R.slices<5>(BG),
                      R.slices<5>(BF), R.slices<5>(AT2));
    return pack_all(R.slices<3>(AT), R.slices<3>(BT), R.slices<3>(A1), R.slices<3>(BG),
                    R.slices<3>(BF), R.slices<3>(AT2));
  }

  // ---- contraction launches -------------------------------------------------
  int contract(int nprob, int M, int N, int ldo, const Operand& opA0, const Operand& opA1,
               const Operand& opB0, const Operand& opB1, const ProbF64* dpf, const TcProb* dpt,
               TcOut lay) {
    cudaEvent_t e0 = R.event(), e1 = R.event();
    if (e0) cudaEventRecord(e0, R.st);
    if (R.f64) {
      CU(launch_gemm_f64(dpf, nprob, M, N, ldo, R.st));
    } else {
      const double scale = R.sigT * R.sigI * std::ldexp(1.0, f16 ? -19 : R.tf32 ? -20 : -14);
      const int fmt = R.tf32 ? kFmtTF32 : f16 ? kFmtF16 : kFmtBF16;
      CU(launch_contract(S, fmt, bn, opA0, opA1, opB0, opB1, dpt, nprob, M, N, ldo, scale,
                         R.ctx->d_flag, R.ctx->nsm, R.st, lay));
    }
    if (e1) cudaEventRecord(e1, R.st);
    if (e0 && e1) R.contract_ev.push_back({e0, e1});
    R.stats->contract_launches++;
    return LNO_OT_OK;
  }

  void seg_f64(SegF64& sg, const Operand& A, int64_t arow, const Operand& B, int64_t brow,
               double sign) {
    sg = SegF64{A.f64 + arow * A.Kp, B.f64 + brow * B.Kp, A.K, A.Kp, B.Kp, sign};
  }
  // roles exchanged for the row-major launch (launch_contract): the kernel's
  // A is the pair operand B, its B the virtual operand A
  void seg_tc(TcSeg& sg, int amap, const Operand& A, int64_t arow, int bmap, const Operand& B,
              int64_t brow, int neg) {
    sg = TcSeg{bmap, amap, (int)brow, (int)arow, A.K, neg};
  }

  int run_case(bool is_mixed) {
    CaseSel& cs = is_mixed ? mixed : same;
    const int ntrip = (int)cs.trips.size();
    if (ntrip == 0) return LNO_OT_OK;
    Arena A(R.st, 0);  // per-case buffers
    const bool f64 = R.f64;
    const size_t esz = f64 ? 8 : 4;
    // output layouts
    const int M1 = v;                                       // rows a
    const int64_t N1 = is_mixed ? (int64_t)v * vt : npairs(v);
    const int P1 = (int)round_up(std::max(M1, 1), 16);
    const int M2 = vt;                                      // mixed Z': rows C
    const int64_t N2 = is_mixed ? npairs(v) : 0;
    const int P2 = (int)round_up(std::max(M2, 1), 16);
    const int nbs = (v + 15) / 16, nbt = (vt + 15) / 16;
    // mixed spin on the tensor cores without f_ov: Y and Z' as 16^3 tiles (the
    // TMA-staged energy kernel reads each sub-cube with one bulk copy);
    // otherwise rows [pair][a] of pitch P1 (P2)
    const bool fov = R.fov[0] != nullptr;   // restricted open-shell f_ov term
    const bool tiled = !f64 && is_mixed && !fov;
    const int64_t xs = tiled ? (int64_t)nbs * nbt * nbs * kTile : N1 * P1;   // per triplet
    const int64_t zs = tiled ? (int64_t)nbs * (nbs + 1) / 2 * nbt * kTile : N2 * P2;
    const TcOut lay1 = tiled ? TcOut{kOutYTile, vt, nbs, nbt} : TcOut{kOutRows, 0, 0, 0};
    const TcOut lay2 = tiled ? TcOut{kOutZTile, 0, nbs, nbt} : TcOut{kOutRows, 0, 0, 0};
    const int64_t per_trip = (xs + zs) * (int64_t)esz;
    const int64_t budget = (int64_t)6 << 30;
    bn = 0;
    group_cap = kGroupCap;
    if (const auto* row = R.ctx->tune_for(v)) {
      bn = row->bn;
      group_cap = std::max(1, row->group_cap);
    }
    int G = (int)std::max<int64_t>(
        1, std::min<int64_t>(group_cap, budget / std::max<int64_t>(per_trip, 1)));
    // energy chunks per triplet from the domain's shape only (a full group of all
    // the case's triplets), so that a triplet's partial sums (and its e_t, bit for
    // bit) do not depend on which other triplets the call selects, nor on whether
    // it has to run in small pieces
    const int Gshape = cs.ntot > 0 ? (int)std::min<int64_t>(G, cs.ntot) : std::min(G, ntrip);
    if (R.ctx->frugal) G = std::min(G, kFrugalGroup);
    G = std::min(G, ntrip);
    char *X = nullptr, *Z = nullptr;
    TRY(A.get(&X, (size_t)(G * xs * esz) + 64));
    if (is_mixed) TRY(A.get(&Z, (size_t)(G * zs * esz) + 64));
    // (the pads of rows and tiles stay unwritten: the energy kernels select the
    // restricted elements, so no pad reaches a sum)
    // cube tiles
    std::vector<int3> blocks;
    if (!is_mixed) {
      for (int a = 0; a < nbs; ++a)
        for (int b = a; b < nbs; ++b)
          for (int c = b; c < nbs; ++c) blocks.push_back(make_int3(a, b, c));
    } else {
      for (int a = 0; a < nbs; ++a)
        for (int b = a; b < nbs; ++b)
          for (int c = 0; c < nbt; ++c) blocks.push_back(make_int3(a, b, c));
    }
    if (blocks.empty()) {  // no virtual orbitals in this case: every W is empty
      CU(cudaMemsetAsync(is_mixed ? e_mixed : e_same, 0, (size_t)ntrip * sizeof(double), R.st));
      return LNO_OT_OK;
    }
    // float64 path: P chunks per triplet, one CTA each.  Float32 path: P
    // items per triplet on a persistent grid, about 32 items per resident CTA
    // in a full group (so the last round of items is a small fraction), one
    // partial per warp and item.
    const int P = f64 ? std::max(1, std::min((int)blocks.size(), R.ctx->nsm * 6 / Gshape + 1))
                      : std::max(1, std::min((int)blocks.size(),
                                             (64 * R.ctx->nsm + Gshape - 1) / Gshape));
    const int npart = f64 ? P : 8 * P;   // partials per triplet
    double* partial;
    TRY(A.get(&partial, (size_t)G * npart * (fov ? 2 : 1)));
    // float32 V tables of the tensor-core path, per triplet
    const int pv = (int)round_up(std::max(v, 1), 16), pvt = (int)round_up(std::max(vt, 1), 16);
    const int64_t vt_stride = is_mixed ? round_up(2LL * v * pvt + (int64_t)v * pv, 16)
                                       : 3LL * v * pv;
    // mixed spin on the tensor-core path takes the f_ov term in the same pass
    // (T1 and f_ov planes side by side in the V table); elsewhere a second pass
    const bool fuse = fov && !f64 && is_mixed;
    float* vtab = nullptr;
    if (!f64) TRY(A.get(&vtab, (size_t)(G * vt_stride * (fuse ? 2 : 1))));
    double* eout = is_mixed ? e_mixed : e_same;

    EnergyArgs ea{};
    ea.kind = is_mixed ? MIXED : SAME;
    ea.nvs = v;
    ea.nvt = is_mixed ? vt : v;
    ea.nos = o;
    ea.not_ = is_mixed ? ot : o;
    ea.eps_s = R.dom->eps[s];
    ea.eps_t = R.dom->eps[is_mixed ? t : s];
    ea.t1s = R.dom->t1[s];
    ea.t1t = R.dom->t1[is_mixed ? t : s];
    set_v_args(ea, is_mixed);
    ea.nblocks = (int)blocks.size();
    ea.pitch_x = P1;
    ea.pitch_z = P2;
    ea.x_stride = xs;
    ea.z_stride = zs;
    ea.tiled = tiled ? 1 : 0;
    ea.lap_s = R.lap_s;
    ea.lap_w = R.lap_w;
    ea.nsm = R.ctx->nsm;
    ea.flag = R.ctx->d_flag;

    // stats
    const double dv = v, dvt = vt;
    const double alg = is_mixed ? flops_alg_mixed(dv, dvt, (double)oi, (double)oti)
                                : flops_alg_same(dv, (double)oi);
    const double doi = oi, doti = oti;   // K of the hole parts: the internal ranges
    const double exe = is_mixed ? 2.0 * dv * (dv * dvt) * (2 * (dvt + doti) + dv + doi) +
                                      2.0 * dvt * (double)npairs(v) * 2 * (dv + doi)
                                : 2.0 * dv * (double)npairs(v) * 3 * (dv + doi);
    const double tens = is_mixed ? 2.0 * dv * (dv * dvt) * (2 * kpad16(dvt + doti) + kpad16(dv + doi)) +
                                       2.0 * dvt * (double)npairs(v) * 2 * kpad16(dv + doi)
                                 : 2.0 * dv * (double)npairs(v) * 3 * kpad16(dv + doi);
    R.stats->flops_algorithmic += alg * ntrip;
    R.stats->flops_executed += exe * ntrip;
    if (!f64) R.stats->tensor_flops += tens * ntrip * (S * (S + 1) / 2);
    R.stats->triplets += ntrip;
    R.stats->elements += (int64_t)ntrip *
                         (is_mixed ? npairs(v) * vt : (int64_t)v * (v - 1) * (v - 2) / 6);

    // Contraction problems, uploaded kWindow triplets at a time: a copy from pageable
    // memory waits for the stream, so one per group kept the launches from running
    // ahead of the device, and one for all triplets took 250 bytes of each.
    const int W = std::max(G, kWindow / G * G);
    const int3* dblocks = nullptr;
    const Trip* dtrips = nullptr;
    for (int w0 = 0; w0 < ntrip; w0 += W) {
      const int nw = std::min(W, ntrip - w0);
      std::vector<ProbF64> pf(f64 ? nw : 0), pf2(f64 && is_mixed ? nw : 0);
      std::vector<TcProb> pt(f64 ? 0 : nw), pt2(!f64 && is_mixed ? nw : 0);
      for (int q = 0; q < nw; ++q) {
        const Trip tr = cs.trips[w0 + q];
        const int g = q % G;   // its place in its group
        const int i = tr.i, j = tr.j, k = tr.k;
        char* Xg = X + (size_t)g * xs * esz;
        if (!is_mixed) {
          const int64_t r_jk = (int64_t)slotAT[(size_t)j * o + k] * v;
          const int64_t r_ki = (int64_t)slotAT[(size_t)k * o + i] * v;
          const int64_t r_ij = (int64_t)slotAT[(size_t)i * o + j] * v;
          const int64_t b_i = slotBT[i] * npairs(v), b_j = slotBT[j] * npairs(v),
                        b_k = slotBT[k] * npairs(v);
          if (f64) {
            ProbF64& p = pf[q];
            p.nseg = 3;
            seg_f64(p.seg[0], AT, r_jk, BT, b_i, 1.0);
            seg_f64(p.seg[1], AT, r_ki, BT, b_j, 1.0);
            seg_f64(p.seg[2], AT, r_ij, BT, b_k, 1.0);
            p.XT = reinterpret_cast<double*>(Xg);
          } else {
            TcProb& p = pt[q];
            p.nseg = 3;
            seg_tc(p.seg[0], 0, AT, r_jk, 0, BT, b_i, 0);
            seg_tc(p.seg[1], 0, AT, r_ki, 0, BT, b_j, 0);
            seg_tc(p.seg[2], 0, AT, r_ij, 0, BT, b_k, 0);
            p.out = Xg;
          }
        } else {
          const int K = k;
          const int64_t a1_jK = (int64_t)slotA1[(size_t)j * ot + K] * v;
          const int64_t a1_iK = (int64_t)slotA1[(size_t)i * ot + K] * v;
          const int64_t at_ij = (int64_t)slotAT[(size_t)i * o + j] * v;
          const int64_t bg_i = (int64_t)slotBG[i] * v * vt, bg_j = (int64_t)slotBG[j] * v * vt;
          const int64_t bf_K = (int64_t)slotBF[K] * v * vt;
          const int64_t a2_jK = (int64_t)slotAT2[(size_t)j * ot + K] * vt;
          const int64_t a2_iK = (int64_t)slotAT2[(size_t)i * ot + K] * vt;
          const int64_t bt_i = slotBT[i] * npairs(v), bt_j = slotBT[j] * npairs(v);
          char* Zg = Z + (size_t)g * zs * esz;
          if (f64) {
            ProbF64& p = pf[q];
            p.nseg = 3;
            seg_f64(p.seg[0], A1, a1_jK, BG, bg_i, 1.0);
            seg_f64(p.seg[1], A1, a1_iK, BG, bg_j, -1.0);
            seg_f64(p.seg[2], AT, at_ij, BF, bf_K, 1.0);
            p.XT = reinterpret_cast<double*>(Xg);
            ProbF64& p2 = pf2[q];
            p2.nseg = 2;
            seg_f64(p2.seg[0], AT2, a2_jK, BT, bt_i, -1.0);
            seg_f64(p2.seg[1], AT2, a2_iK, BT, bt_j, 1.0);
            p2.XT = reinterpret_cast<double*>(Zg);
          } else {
            TcProb& p = pt[q];
            p.nseg = 3;
            seg_tc(p.seg[0], 0, A1, a1_jK, 0, BG, bg_i, 0);
            seg_tc(p.seg[1], 0, A1, a1_iK, 0, BG, bg_j, 1);
            seg_tc(p.seg[2], 1, AT, at_ij, 1, BF, bf_K, 0);
            p.out = Xg;
            TcProb& p2 = pt2[q];
            p2.nseg = 2;
            seg_tc(p2.seg[0], 0, AT2, a2_jK, 0, BT, bt_i, 1);
            seg_tc(p2.seg[1], 0, AT2, a2_iK, 0, BT, bt_j, 0);
            p2.out = Zg;
          }
        }
      }
      const ProbF64 *dpf = nullptr, *dpf2 = nullptr;
      const TcProb *dpt = nullptr, *dpt2 = nullptr;
      Upload up;
      if (w0 == 0) {
        up.add(blocks, &dblocks);
        up.add(cs.trips, &dtrips);
      }
      up.add(pf, &dpf);
      up.add(pf2, &dpf2);
      up.add(pt, &dpt);
      up.add(pt2, &dpt2);
      TRY(up.send(R, A));
      ea.blocks = dblocks;

      for (int g0 = w0; g0 < w0 + nw; g0 += G) {
        const int ng = std::min(G, w0 + nw - g0), gw = g0 - w0;
        TRY(contract(ng, M1, (int)N1, P1, is_mixed ? A1 : AT, AT, is_mixed ? BG : BT,
                     is_mixed ? BF : BT, f64 ? dpf + gw : nullptr, f64 ? nullptr : dpt + gw, lay1));
        if (is_mixed)
          TRY(contract(ng, M2, (int)N2, P2, AT2, AT2, BT, BT, f64 ? dpf2 + gw : nullptr,
                       f64 ? nullptr : dpt2 + gw, lay2));
        // energy
        ea.trips = dtrips + g0;
        ea.partial = partial;
        cudaEvent_t e0 = R.event(), e1 = R.event();
        if (e0) cudaEventRecord(e0, R.st);
        if (f64) {
          CU(launch_energy(ea, X, Z, f64, ng, P, R.st));
        } else if (fuse) {
          EnergyArgs ef = ea;
          ef.fs = R.fov[s];
          ef.ft = R.fov[t];
          ef.t2ss = t2ss;
          ef.t2st = t2st;
          CU(launch_energy_f32_fused(ef, reinterpret_cast<const float*>(X),
                                     reinterpret_cast<const float*>(Z), vtab, vt_stride, pv, pvt,
                                     ng, P, R.st));
          R.stats->energy_launches += 1;
        } else {
          CU(launch_energy_f32(ea, reinterpret_cast<const float*>(X),
                               reinterpret_cast<const float*>(Z), vtab, vt_stride, pv, pvt, ng, P,
                               R.st));
        }
        double* partial2 = nullptr;
        if (fov && !fuse) {
          // the f_ov part of V in a second pass over the same X (and Z'):
          // sum W V_f / D with V_f built like the T1 term from f_ov and T2
          EnergyArgs ef = ea;
          ef.vmode = 1;
          ef.t1s = R.fov[s];
          ef.t1t = R.fov[is_mixed ? t : s];
          ef.t2ss = t2ss;
          ef.t2st = t2st;
          ef.partial = partial2 = partial + (size_t)G * npart;
          if (f64)
            CU(launch_energy(ef, X, Z, f64, ng, P, R.st));
          else
            CU(launch_energy_f32(ef, reinterpret_cast<const float*>(X),
                                 reinterpret_cast<const float*>(Z), vtab, vt_stride, pv, pvt, ng,
                                 P, R.st));
          R.stats->energy_launches += 2;
        }
        CU(launch_reduce_partials(partial, npart, partial2, ng, eout + g0, R.st));
        if (e1) cudaEventRecord(e1, R.st);
        if (e0 && e1) R.energy_ev.push_back({e0, e1});
        R.stats->energy_launches += 2;
      }
      if (w0 > 0) A.drop(up.base);
    }
    return LNO_OT_OK;
  }

  // operands for the current selections (the whole domain when cached)
  int prepare() {
    f16 = R.f16;
    S = R.S;
    plan();
    TRY(prepare_inputs());
    TRY(build_v_blocks());
    TRY(build());
    if (!f16) return LNO_OT_OK;
    bool exact;
    TRY(check_exact(&exact));
    if (exact) return LNO_OT_OK;
    // Not provably exact: this spin again, DF blocks and operands on the BF16 slices
    // (as a whole call on them computes it).  What the other spin has computed on FP16
    // slices stands.
    own.release();
    t2st = nullptr;
    TRY(R.leave_f16());
    return prepare();
  }
  // FP16 slices: whether the class-0 sums of every contraction are exact (kExactSum)
  int check_exact(bool* exact) {
    unsigned long long* slot = R.ctx->d_amax + kNormW;
    CU(cudaMemsetAsync(slot, 0, 6 * sizeof(unsigned long long), R.st));
    const Operand* ops[6] = {&AT, &BT, &A1, &BG, &BF, &AT2};
    for (int q = 0; q < 6; ++q) TRY(R.row_norm2(*ops[q], kNormW + q));
    unsigned long long h[6];
    CU(cudaMemcpyAsync(h, slot, sizeof h, cudaMemcpyDeviceToHost, R.st));
    CU(cudaStreamSynchronize(R.st));
    double n[6];
    std::memcpy(n, h, sizeof h);
    for (double& x : n) x = std::sqrt(x);
    const double x = 3 * n[0] * n[1], y = 2 * n[2] * n[3] + n[0] * n[4], z = 2 * n[5] * n[1];
    *exact = std::max({x, y, z}) <= kExactSum;
    return LNO_OT_OK;
  }
  int compute() {
    TRY(run_case(false));
    TRY(run_case(true));
    return LNO_OT_OK;
  }
  int run() {
    if (same.trips.empty() && mixed.trips.empty()) return LNO_OT_OK;
    TRY(prepare());
    return compute();
  }
};

int check_ptr(const lno_ot_ctx* ctx, const void* p, bool required) {
  if (!p) return required ? LNO_OT_EINVAL : LNO_OT_OK;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return LNO_OT_EDEVICE;
  }
  if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged) return LNO_OT_EDEVICE;
  if (at.device != ctx->device) return LNO_OT_EDEVICE;
  return LNO_OT_OK;
}

int validate(const lno_ot_ctx* ctx, const lno_ot_domain* d) {
  if (!d) return LNO_OT_EINVAL;
  if (d->nbas <= 0 || d->naux <= 0) return LNO_OT_EINVAL;
  if (d->nocc[1] < 0 || d->nocc[1] > d->nocc[0] || d->nocc[0] > d->nbas) return LNO_OT_EINVAL;
  if ((int64_t)d->nbas * d->nbas * d->naux > ((int64_t)1 << 40)) return LNO_OT_EINVAL;
  for (int s = 0; s < 2; ++s) {
    TRY(check_ptr(ctx, d->B[s], true));
    TRY(check_ptr(ctx, d->eps[s], true));
    const bool need_t1 = d->nocc[s] > 0 && d->nocc[s] < d->nbas;
    TRY(check_ptr(ctx, d->t1[s], need_t1));
  }
  const bool va = d->nocc[0] < d->nbas, vb = d->nocc[1] < d->nbas;
  TRY(check_ptr(ctx, d->t2aa, d->nocc[0] > 0 && va));
  TRY(check_ptr(ctx, d->t2bb, d->nocc[1] > 0 && vb));
  TRY(check_ptr(ctx, d->t2ab, d->nocc[0] > 0 && d->nocc[1] > 0 && va && vb));
  for (int c = 0; c < 4; ++c) TRY(check_ptr(ctx, d->e_trip[c], false));
  for (int s = 0; s < 2; ++s) {
    const bool has = d->nocc[s] > 0 && d->nocc[s] < d->nbas;
    TRY(check_ptr(ctx, d->fov[s], false));
    if (d->fov[s] && !has) return LNO_OT_EINVAL;   // nothing to hold
    TRY(check_ptr(ctx, d->e_orb[s], false));
  }
  return LNO_OT_OK;
}

// Whether the blocks built with this scale hold larger integrals than it
// allows (d_amax[2], collected by the assembly; its rounding to float32 is the
// measuring pass's).
bool scale_too_small(const Run& R, unsigned long long built) {
  if (R.f64) return false;
  double m;
  std::memcpy(&m, &built, 8);
  return std::isfinite(m) && 2.0 * m > R.sigI;
}

// Per-case sums, per-triplet and orbital outputs, results and stats of one
// call (after the spin passes have filled e_int).
int finish_call(lno_ot_ctx* ctx, Run& R, Arena& A, const lno_ot_domain* dom, const CaseSel* cs,
                double* const* e_int, bool thirds, bool kept, cudaEvent_t t0, cudaEvent_t t1,
                cudaEvent_t t2, lno_ot_result* out) {
  // per-case sums and the caller's per-triplet values
  CaseSums sums{};
  for (int c = 0; c < 4; ++c) {
    sums.e[c] = e_int[c];
    sums.n[c] = (int64_t)cs[c].trips.size();
    sums.copy[c] = dom->e_trip[c];
  }
  sums.out = ctx->d_sums;
  CU(launch_case_sums(sums, R.st));
  R.stats->other_launches++;
  // orbital contributions (eq cim_pt_energy) of the computed triplets
  if (dom->e_orb[0] || dom->e_orb[1]) {
    OrbPartArgs oa{};
    oa.na = dom->nocc[0];
    oa.nb = dom->nocc[1];
    oa.thirds = thirds;
    oa.out[0] = dom->e_orb[0];
    oa.out[1] = dom->e_orb[1];
    for (int c = 0; c < 4; ++c) {
      oa.e[c] = e_int[c];
      oa.n[c] = (int64_t)cs[c].trips.size();
      Trip* dt;
      TRY(A.get(&dt, std::max<size_t>(cs[c].trips.size(), 1)));
      if (!cs[c].trips.empty())
        CU(ctx->h2d(dt, cs[c].trips.data(), cs[c].trips.size() * sizeof(Trip)));
      oa.trips[c] = dt;
    }
    CU(launch_orbital_partition(oa, R.st));
    R.stats->other_launches++;
  }
  CallState h;
  CU(cudaMemcpyAsync(&h, ctx->d_sums, sizeof h, cudaMemcpyDeviceToHost, R.st));
  if (t2) cudaEventRecord(t2, R.st);
  CU(cudaStreamSynchronize(R.st));
  if (h.flag) return LNO_OT_ETIMEOUT;
  if (!kept && scale_too_small(R, h.amax[2])) return kRescale;
  const double* hs = h.sums;
  // stats
  float ms = 0;
  if (t0 && t2 && cudaEventElapsedTime(&ms, t0, t2) == cudaSuccess) ctx->stats.ms_total = ms;
  if (t0 && t1 && cudaEventElapsedTime(&ms, t0, t1) == cudaSuccess) ctx->stats.ms_stage = ms;
  double acc = 0;
  for (auto& p : R.contract_ev)
    if (cudaEventElapsedTime(&ms, p.first, p.second) == cudaSuccess) acc += ms;
  ctx->stats.ms_contract = acc;
  acc = 0;
  for (auto& p : R.energy_ev)
    if (cudaEventElapsedTime(&ms, p.first, p.second) == cudaSuccess) acc += ms;
  ctx->stats.ms_energy = acc;
  // order: aaa, aab, abb, bbb, total (Neumaier on the host for the last 4)
  double S = 0, Cc = 0;
  for (int c = 0; c < 4; ++c) {
    out->e[c] = hs[c];
    double x = hs[c], tt = S + x;
    Cc += std::fabs(S) >= std::fabs(x) ? (S - tt) + x : (x - tt) + S;
    S = tt;
  }
  out->e[4] = S + Cc;
  return LNO_OT_OK;
}

}  // namespace

// Whole-domain operands kept between calls (options.keep_operands): the DF
// blocks and scales of the Run and the operand tensors of both spin passes,
// built for every triplet of the domain.  A later call on the same arrays
// (another triplet selection) only runs the contractions and energy kernels.
struct DomainCache {
  lno_ot_domain key{};      // arrays and sizes the operands were built from
  int prec = 0;
  std::unique_ptr<Run> R;
  CaseSel cs[4];            // full selections at build time, the call's afterwards
  std::unique_ptr<SpinPass> pa, pb;
  bool has_a = false, has_b = false;

  bool matches(const lno_ot_domain* d, int p) const {
    if (p != prec || d->nbas != key.nbas || d->naux != key.naux) return false;
    for (int s = 0; s < 2; ++s)
      if (d->nocc[s] != key.nocc[s] || d->B[s] != key.B[s] || d->eps[s] != key.eps[s] ||
          d->t1[s] != key.t1[s] || d->fov[s] != key.fov[s])
        return false;
    return d->t2aa == key.t2aa && d->t2bb == key.t2bb && d->t2ab == key.t2ab;
  }
};

void destroy_cache(DomainCache* c) {
  if (!c) return;
  c->pa.reset();  // spin-pass operands first, then the Run's DF blocks
  c->pb.reset();
  c->R.reset();
  delete c;
}

namespace {

// Settings of an internal energy pass over an augmented domain (the central
// LMOs of the Laplace form): explicit triplet lists, per-spin orbital counts,
// internal occupied ranges, one quadrature point and eq local_pt's partition.
struct PassSpec {
  const CaseSel* cs;   // [4]
  int nbs[2];
  int noi[2];
  double lap_s, lap_w;
};

void set_precision(Run& R, int prec, const int* nvir, const int* nocc, bool no_f16) {
  R.f16 = prec == LNO_OT_BF16X10 && !no_f16 && f16_sizes(nvir, nocc);
  R.f64 = prec == LNO_OT_FP64;
  R.tf32 = prec == LNO_OT_TF32;
  R.S = prec == LNO_OT_BF16X6 || R.f16 ? 3
        : prec == LNO_OT_BF16X10 ? 4
        : prec == LNO_OT_BF16X15 ? 5
                                 : 2;
  R.Sdf = prec == LNO_OT_BF16X15 ? 5 : R.f16 ? 3 : 4;
}

// Integral scale of the sliced path: one pass over every DF block the two
// spin passes need (their current selections).
int measure_sigI(lno_ot_ctx* ctx, Run& R, SpinPass* pa, SpinPass* pb) {
  if (R.f64) return LNO_OT_OK;
  if (pa) pa->plan();
  if (pb) pb->plan();
  if (pa) TRY(pa->prepare_inputs());
  if (pb) TRY(pb->prepare_inputs());
  // Two of the four or five slices of each factor (3 products instead of 10 or
  // 15) give the largest integral to ~1e-4, and the scale is a power of two: it
  // is settled unless the maximum lies within 1% of one.  Then, or when the
  // blocks as built turn out larger than this measure said (finish_call), every
  // slice is taken.
  for (int pass = ctx->exact_measure ? 1 : 0; pass < 2; ++pass) {
    CU(cudaMemsetAsync(ctx->d_amax, 0, 4 * sizeof(unsigned long long), R.st));
    R.amax_exact = pass == 1;
    if (pa) TRY(pa->measure());
    if (pb) TRY(pb->measure());
    unsigned long long h[kNormB + 2];
    CU(cudaMemcpyAsync(h, ctx->d_amax, sizeof h, cudaMemcpyDeviceToHost, R.st));
    CU(cudaStreamSynchronize(R.st));
    double m, nB[2];
    std::memcpy(&m, &h, 8);
    std::memcpy(nB, h + kNormB, sizeof nB);
    if (R.f16 && !(std::max(nB[0], nB[1]) <= kExactSum)) return kNoF16;
    R.sigI = pow2_scale(2.0 * m);  // antisymmetrised combinations are <= 2 max
    int ex;
    const double f = std::frexp(2.0 * m, &ex);
    if (f > 0.505 && f < 0.99) break;
  }
  return LNO_OT_OK;
}

// Builds ctx->cache for dom (every triplet of the domain).
int build_cache(lno_ot_ctx* ctx, const lno_ot_domain* dom) {
  destroy_cache(ctx->cache);
  ctx->cache = nullptr;
  std::unique_ptr<DomainCache> C(new DomainCache());
  C->key = *dom;
  for (int c = 0; c < 4; ++c) {
    C->key.e_trip[c] = nullptr;
    C->key.trip_sel[c] = nullptr;
    C->key.n_sel[c] = 0;
  }
  C->key.e_orb[0] = C->key.e_orb[1] = nullptr;
  C->prec = ctx->prec;
  C->R.reset(new Run(ctx, &C->key));
  Run& R = *C->R;
  const int nvir[2] = {dom->nbas - dom->nocc[0], dom->nbas - dom->nocc[1]};
  set_precision(R, ctx->prec, nvir, dom->nocc, ctx->no_f16);
  for (int c = 0; c < 4; ++c) TRY(select_case(&C->key, c, C->cs[c]));
  TRY(R.stage());
  C->has_a = !C->cs[0].trips.empty() || !C->cs[1].trips.empty();
  C->has_b = !C->cs[3].trips.empty() || !C->cs[2].trips.empty();
  C->pa.reset(new SpinPass(R, 0, C->cs[0], C->cs[1], nullptr, nullptr));
  C->pb.reset(new SpinPass(R, 1, C->cs[3], C->cs[2], nullptr, nullptr));
  TRY(measure_sigI(ctx, R, C->has_a ? C->pa.get() : nullptr, C->has_b ? C->pb.get() : nullptr));
  if (C->has_a) TRY(C->pa->prepare());
  if (C->has_b) TRY(C->pb->prepare());
  unsigned long long built;
  CU(cudaMemcpyAsync(&built, ctx->d_amax + 2, sizeof built, cudaMemcpyDeviceToHost, R.st));
  CU(cudaStreamSynchronize(R.st));
  if (scale_too_small(R, built) && !ctx->exact_measure) return kRescale;
  ctx->cache = C.release();
  return LNO_OT_OK;
}

// One call through the cache (built on a miss).  Returns LNO_OT_ENOMEM when
// the whole-domain operands do not fit; the caller then runs uncached.
int cached_energy(lno_ot_ctx* ctx, const lno_ot_domain* dom, lno_ot_result* out) {
  ctx->stats = lno_ot_stats{};
  ctx->ev_used = 0;
  CU(cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), ctx->stream));
  cudaEvent_t t0 = nullptr, t1 = nullptr, t2 = nullptr;
  const bool hit = ctx->cache && ctx->cache->matches(dom, ctx->prec);
  {
    // events from the pool (the Run may not exist yet)
    for (cudaEvent_t* e : {&t0, &t1, &t2}) {
      if (ctx->ev_used == ctx->ev_pool.size()) {
        cudaEvent_t ev;
        if (cudaEventCreate(&ev) != cudaSuccess) {
          cudaGetLastError();
          break;
        }
        ctx->ev_pool.push_back(ev);
      }
      *e = ctx->ev_pool[ctx->ev_used++];
    }
  }
  if (t0) cudaEventRecord(t0, ctx->stream);
  if (!hit) {
    const int rc = build_cache(ctx, dom);
    if (rc != LNO_OT_OK) {
      destroy_cache(ctx->cache);
      ctx->cache = nullptr;
      cudaGetLastError();
      return rc;
    }
  }
  DomainCache* C = ctx->cache;
  Run& R = *C->R;
  R.dom = dom;
  R.contract_ev.clear();
  R.energy_ev.clear();
  if (t1) cudaEventRecord(t1, R.st);
  CaseSel sel[4];
  for (int c = 0; c < 4; ++c) {
    TRY(select_case(dom, c, sel[c]));
    C->cs[c].trips.swap(sel[c].trips);
    C->cs[c].ntot = sel[c].ntot;
  }
  Arena A(R.st, ctx->ws_limit);
  double* e_int[4];
  for (int c = 0; c < 4; ++c)
    TRY(A.get(&e_int[c], std::max<size_t>(C->cs[c].trips.size(), 1)));
  C->pa->e_same = e_int[0];
  C->pa->e_mixed = e_int[1];
  C->pb->e_same = e_int[3];
  C->pb->e_mixed = e_int[2];
  if (C->has_a) TRY(C->pa->compute());
  if (C->has_b) TRY(C->pb->compute());
  return finish_call(ctx, R, A, dom, C->cs, e_int, false, true, t0, t1, t2, out);
}

bool flip_candidate(const lno_ot_domain* dom) {
  bool flip = dom->nocc[0] == dom->nocc[1] && dom->B[0] == dom->B[1] &&
              dom->eps[0] == dom->eps[1] && dom->t1[0] == dom->t1[1] &&
              dom->t2aa == dom->t2bb && dom->fov[0] == dom->fov[1];
  for (int c = 0; c < 4; ++c) flip = flip && dom->trip_sel[c] == nullptr;
  return flip;
}

int energy_once(lno_ot_ctx* ctx, const lno_ot_domain* dom, lno_ot_result* out,
                const PassSpec* spec) {
  if (!spec) TRY(validate(ctx, dom));
  CU(cudaSetDevice(ctx->device));
  if (!spec && ctx->keep && !flip_candidate(dom)) {
    const int rc = cached_energy(ctx, dom, out);
    if (rc != LNO_OT_ENOMEM) return rc;   // the whole domain did not fit: run uncached
  }
  if (!spec) ctx->stats = lno_ot_stats{};
  ctx->ev_used = 0;
  Run R(ctx, dom);
  if (spec) {
    for (int s = 0; s < 2; ++s) {
      R.nbs[s] = spec->nbs[s];
      R.noi[s] = spec->noi[s];
    }
    R.lap_s = spec->lap_s;
    R.lap_w = spec->lap_w;
  }
  const int nvir[2] = {(spec ? spec->nbs[0] : dom->nbas) - dom->nocc[0],
                       (spec ? spec->nbs[1] : dom->nbas) - dom->nocc[1]};
  set_precision(R, ctx->prec, nvir, dom->nocc, ctx->no_f16);
  CU(cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), ctx->stream));
  cudaEvent_t t0 = R.event(), t1 = R.event(), t2 = R.event();
  if (t0) cudaEventRecord(t0, R.st);

  CaseSel cs[4];
  for (int c = 0; c < 4; ++c) {
    if (spec)
      cs[c] = spec->cs[c];
    else
      TRY(select_case(dom, c, cs[c]));
  }
  double* e_int[4];
  for (int c = 0; c < 4; ++c)
    TRY(R.arena.get(&e_int[c], std::max<size_t>(cs[c].trips.size(), 1)));
  if (dom->e_orb[0] || dom->e_orb[1])   // the triplet lists of finish_call
    for (int c = 0; c < 4; ++c)
      R.held_back += Arena::bytes_of<Trip>(std::max<size_t>(cs[c].trips.size(), 1));
  // Closed-shell domain (both spins given by the same arrays, spin-flip
  // symmetric mixed amplitudes): bbb and abb are the spin-flip images of aaa
  // and aab, with identical values, so only the spin-up pass runs.
  bool flip = flip_candidate(dom) && spec == nullptr;
  if (flip && dom->nocc[0] > 0 && dom->nocc[0] < dom->nbas) {
    // symmetric to within 1e-12 of the largest amplitude: amplitudes from a
    // closed-shell calculation agree with their spin-flip images to rounding
    const int n = dom->nocc[0], v = dom->nbas - dom->nocc[0];
    CU(cudaMemsetAsync(ctx->d_amax, 0, sizeof(unsigned long long), R.st));
    CU(launch_absmax(dom->t2ab, (int64_t)n * n * v * v, ctx->d_amax, R.st));
    unsigned long long hm = 0;
    CU(cudaMemcpyAsync(&hm, ctx->d_amax, sizeof hm, cudaMemcpyDeviceToHost, R.st));
    CU(cudaStreamSynchronize(R.st));
    double amax;
    std::memcpy(&amax, &hm, 8);
    unsigned int* cnt;
    TRY(R.arena.get(&cnt, 1));
    CU(cudaMemsetAsync(cnt, 0, sizeof(unsigned int), R.st));
    CU(launch_t2ab_flip_mismatch(dom->t2ab, n, v, 1e-12 * amax, cnt, R.st));
    unsigned int h = 1;
    CU(cudaMemcpyAsync(&h, cnt, sizeof h, cudaMemcpyDeviceToHost, R.st));
    CU(cudaStreamSynchronize(R.st));
    R.stats->other_launches += 2;
    flip = h == 0;
  }
  TRY(R.stage());
  {
    SpinPass pa(R, 0, cs[0], cs[1], e_int[0], e_int[1]);
    SpinPass pb(R, 1, cs[3], cs[2], e_int[3], e_int[2]);
    // integral scale: first pass over every DF block both spins need
    TRY(measure_sigI(ctx, R, &pa, flip ? nullptr : &pb));
    if (t1) cudaEventRecord(t1, R.st);
    TRY(pa.run());
    pa.own.release();
    if (!flip) {
      TRY(pb.run());
    } else {  // spin-flip images: bbb = aaa, abb = aab, triplet for triplet
      if (!cs[3].trips.empty())
        CU(cudaMemcpyAsync(e_int[3], e_int[0], cs[3].trips.size() * sizeof(double),
                           cudaMemcpyDeviceToDevice, R.st));
      if (!cs[2].trips.empty())
        CU(cudaMemcpyAsync(e_int[2], e_int[1], cs[2].trips.size() * sizeof(double),
                           cudaMemcpyDeviceToDevice, R.st));
    }
  }
  return finish_call(ctx, R, R.arena, dom, cs, e_int, spec != nullptr, false, t0, t1, t2, out);
}

int energy_impl(lno_ot_ctx* ctx, const lno_ot_domain* dom, lno_ot_result* out,
                const PassSpec* spec = nullptr) {
  ctx->frugal = ctx->small_pieces;
  int rc = energy_once(ctx, dom, out, spec);
  for (int tries = 0; tries < 4; ++tries) {
    if (rc == kRescale && ctx->exact_measure) ctx->no_f16 = true;   // measured and built alike
    else if (rc == kRescale) ctx->exact_measure = true;
    else if (rc == kNoF16) ctx->no_f16 = true;
    else if (rc == LNO_OT_ENOMEM && !ctx->frugal) ctx->frugal = true;
    else break;
    rc = energy_once(ctx, dom, out, spec);
  }
  ctx->exact_measure = ctx->no_f16 = ctx->frugal = false;
  return rc > 0 ? LNO_OT_EINVAL : rc;   // not reached: none comes again
}

// ---------------------------------------------------------------------------
// Natural auxiliary functions (Sec. 3.6, eq naf_w), float64 (naf.cu).
int naf_impl(lno_ot_ctx* ctx, const lno_ot_domain* dom, double eps, double* const* Bout,
             int* naux_out, double* lam_host) {
  if (!dom || !Bout || !naux_out || !(eps >= 0.0) || !std::isfinite(eps)) return LNO_OT_EINVAL;
  if (dom->nbas <= 0 || dom->naux <= 0) return LNO_OT_EINVAL;
  if ((int64_t)dom->nbas * dom->nbas * dom->naux > ((int64_t)1 << 40)) return LNO_OT_EINVAL;
  for (int s = 0; s < 2; ++s) {
    TRY(check_ptr(ctx, dom->B[s], true));
    TRY(check_ptr(ctx, Bout[s], true));
  }
  CU(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  const int n = dom->naux, nb = dom->nbas;
  const int64_t npair = (int64_t)nb * (nb + 1) / 2, n2 = (int64_t)nb * nb;
  Arena A(st, ctx->ws_limit);
  double *J[2], *W, *W2, *V, *d, *norms;
  ProbF64* dp;
  unsigned int* asym;
  TRY(A.get(&asym, 1));
  CU(cudaMemsetAsync(asym, 0, sizeof(unsigned int), st));
  for (int s = 0; s < 2; ++s) {
    TRY(A.get(&J[s], (size_t)(n * npair)));
    CU(launch_pack_pairs(dom->B[s], n, nb, J[s], st));
    CU(launch_asym_count(dom->B[s], n, nb, asym, st));
  }
  TRY(A.get(&W, (size_t)n * n));
  TRY(A.get(&W2, (size_t)n * n));
  TRY(A.get(&dp, 2));
  ProbF64 pw{};   // W = (J^up J^up^T + J^down J^down^T) / 2
  pw.nseg = 2;
  pw.seg[0] = SegF64{J[0], J[0], (int)npair, (int)npair, (int)npair, 0.5};
  pw.seg[1] = SegF64{J[1], J[1], (int)npair, (int)npair, (int)npair, 0.5};
  pw.XT = W;
  CU(ctx->h2d(dp, &pw, sizeof pw));
  CU(launch_gemm_f64_sym(dp, n, n, st));
  TRY(A.get(&V, (size_t)n * n));
  TRY(A.get(&norms, jacobi_norm_doubles()));
  TRY(A.get(&d, (size_t)n));
  const int sweeps = jacobi_eigh(W, W2, V, n, norms, st, 40);
  if (sweeps < 0) return sweeps;
  CU(launch_get_diag(W, n, d, st));
  std::vector<double> lam(n);
  unsigned int hasym = 1;
  for (double* q : {W, W2, norms}) A.drop(q);   // before the factors' copies
  CU(cudaMemcpyAsync(lam.data(), d, (size_t)n * sizeof(double), cudaMemcpyDeviceToHost, st));
  CU(cudaMemcpyAsync(&hasym, asym, sizeof hasym, cudaMemcpyDeviceToHost, st));
  CU(cudaStreamSynchronize(st));
  std::vector<int> order(n);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return lam[a] > lam[b]; });
  int nk = 0;
  while (nk < n && lam[order[nk]] > eps) ++nk;
  if (lam_host)
    for (int i = 0; i < n; ++i) lam_host[i] = lam[order[i]];
  *naux_out = nk;
  if (nk > 0) {
    int* cols;
    double *Vt, *Bt;
    TRY(A.get(&cols, (size_t)nk));
    CU(ctx->h2d(cols, order.data(), (size_t)nk * sizeof(int)));
    TRY(A.get(&Vt, (size_t)nk * n));
    CU(launch_gather_rows_f64(V, n, cols, nk, Vt, st));
    // B'[X'][pq] = sum_X V[X][X'] B[X][pq]: symmetric factors (as the header asks)
    // over the pairs p <= q, half of the products and the same values; factors
    // that differ in any bit from their transpose element by element
    const bool sym = hasym == 0;
    const int64_t rows = sym ? npair : n2;
    if (!sym) {
      A.drop(J[0]);
      A.drop(J[1]);
    }
    TRY(A.get(&Bt, (size_t)(rows * n)));
    ProbF64 p[2] = {};
    for (int s = 0; s < 2; ++s) {
      CU(launch_transpose_x(sym ? J[s] : dom->B[s], n, rows, Bt, st));
      p[s].nseg = 1;
      p[s].seg[0] = SegF64{Bt, Vt, n, n, n, 1.0};
      p[s].XT = sym ? J[s] : Bout[s];   // the pairs' input is in Bt by then
      CU(ctx->h2d(dp + s, &p[s], sizeof p[s]));
      CU(launch_gemm_f64(dp + s, 1, (int)rows, nk, (int)rows, st));
      if (sym) CU(launch_unpack_pairs(J[s], nk, nb, Bout[s], st));
    }
  }
  CU(cudaStreamSynchronize(st));
  return LNO_OT_OK;
}

// ---------------------------------------------------------------------------
// Central-LMO share in the Laplace form (Sec. 3.7, eqs laplace_transform and
// local_pt): per quadrature point, an augmented domain with one pseudo-orbital
// per central orbital (central.cu), the triplets that hold exactly one of
// them, the element weight -w_q exp(s_q D), and eq local_pt's 1/3 of each
// triplet to the pseudo-orbital; the quadrature points are summed on the host.
int central_impl(lno_ot_ctx* ctx, const lno_ot_domain* dom, const lno_ot_central* c) {
  if (!c) return LNO_OT_EINVAL;
  TRY(validate(ctx, dom));
  if (c->nq < 1 || c->nq > 256 || !c->s || !c->w || c->spin < 0 || c->spin > 1 || c->nlmo < 0)
    return LNO_OT_EINVAL;
  if (c->nlmo > 0 && !c->dE) return LNO_OT_EINVAL;
  for (int q = 0; q < c->nq; ++q)
    if (!(c->s[q] > 0.0) || !std::isfinite(c->s[q]) || !std::isfinite(c->w[q]))
      return LNO_OT_EINVAL;
  const int sg = c->spin, tg = 1 - sg, P = c->nlmo;
  const int nbas = dom->nbas, naux = dom->naux;
  const int na = dom->nocc[0], nb = dom->nocc[1], o = dom->nocc[sg];
  const int v = nbas - o;
  for (int l = 0; l < P; ++l) c->dE[l] = 0.0;
  if (P == 0) return LNO_OT_OK;
  if (o == 0) return LNO_OT_EINVAL;
  TRY(check_ptr(ctx, c->U, true));
  CU(cudaSetDevice(ctx->device));
  ctx->stats = lno_ot_stats{};
  cudaStream_t st = ctx->stream;
  Arena A(st, ctx->ws_limit);
  // augmented arrays of spin sg
  const int nb2 = nbas + P, o2 = o + P;
  AugmentArgs ag{};
  ag.spin = sg;
  ag.P = P;
  ag.nbas = nbas;
  ag.naux = naux;
  ag.nocc[0] = na;
  ag.nocc[1] = nb;
  ag.U = c->U;
  ag.B_in = dom->B[sg];
  ag.eps_in = dom->eps[sg];
  ag.t1_in = dom->t1[sg];
  ag.fov_in = dom->fov[sg];
  ag.t2ss_in = sg == 0 ? dom->t2aa : dom->t2bb;
  ag.t2ab_in = dom->t2ab;
  const int va = nbas - na, vb = nbas - nb;
  TRY(A.get(&ag.coef, (size_t)P * o));
  TRY(A.get(&ag.B_out, (size_t)naux * nb2 * nb2));
  TRY(A.get(&ag.eps_out, (size_t)nb2));
  TRY(A.get(&ag.t1_out, (size_t)std::max(o2 * v, 1)));
  if (ag.fov_in) TRY(A.get(&ag.fov_out, (size_t)std::max(o2 * v, 1)));
  TRY(A.get(&ag.t2ss_out, (size_t)std::max<int64_t>((int64_t)o2 * o2 * v * v, 1)));
  TRY(A.get(&ag.t2ab_out, (size_t)std::max<int64_t>(
                              (int64_t)(sg == 0 ? o2 : na) * (sg == 0 ? nb : o2) * va * vb, 1)));
  double* eorb;
  TRY(A.get(&eorb, (size_t)o2));
  // triplets holding exactly one pseudo-orbital (augmented indices o + p)
  CaseSel cs[4];
  const int ot = dom->nocc[tg];
  for (int p = 0; p < P; ++p) {
    const int u = o + p;
    for (int j = 0; j < o; ++j)      // same spin: (j, k, u), j < k < u
      for (int k = j + 1; k < o; ++k) cs[sg == 0 ? 0 : 3].trips.push_back(Trip{j, k, u});
    for (int j = 0; j < o; ++j)      // u and j of spin sg, K of the other: (j, u; K)
      for (int K = 0; K < ot; ++K) cs[sg == 0 ? 1 : 2].trips.push_back(Trip{j, u, K});
    for (int J = 0; J < ot; ++J)     // J < K of the other spin, u the single: (J, K; u)
      for (int K = J + 1; K < ot; ++K) cs[sg == 0 ? 2 : 1].trips.push_back(Trip{J, K, u});
  }
  lno_ot_domain ad = *dom;
  ad.nocc[sg] = o2;
  ad.B[sg] = ag.B_out;
  ad.eps[sg] = ag.eps_out;
  ad.t1[sg] = ag.t1_out;
  if (ag.fov_in) ad.fov[sg] = ag.fov_out;
  if (sg == 0)
    ad.t2aa = ag.t2ss_out;
  else
    ad.t2bb = ag.t2ss_out;
  ad.t2ab = ag.t2ab_out;
  for (int k = 0; k < 4; ++k) {
    ad.e_trip[k] = nullptr;
    ad.trip_sel[k] = nullptr;
    ad.n_sel[k] = 0;
  }
  ad.e_orb[sg] = eorb;
  ad.e_orb[tg] = nullptr;
  PassSpec spec{};
  spec.cs = cs;
  spec.nbs[sg] = nb2;
  spec.nbs[tg] = nbas;
  spec.noi[0] = na;
  spec.noi[1] = nb;
  std::vector<double> acc(P, 0.0), comp(P, 0.0), part(P);
  double ms[4] = {0, 0, 0, 0};
  for (int q = 0; q < c->nq; ++q) {
    ag.s = c->s[q];
    CU(launch_lmo_augment(ag, st));
    ctx->stats.other_launches += 7;
    spec.lap_s = c->s[q];
    spec.lap_w = c->w[q];
    lno_ot_result r;
    TRY(energy_impl(ctx, &ad, &r, &spec));
    ms[0] += ctx->stats.ms_total;
    ms[1] += ctx->stats.ms_stage;
    ms[2] += ctx->stats.ms_contract;
    ms[3] += ctx->stats.ms_energy;
    CU(cudaMemcpyAsync(part.data(), eorb + o, (size_t)P * sizeof(double), cudaMemcpyDeviceToHost,
                       st));
    CU(cudaStreamSynchronize(st));
    for (int l = 0; l < P; ++l) {   // Neumaier over the quadrature points, in order
      const double x = part[l], t = acc[l] + x;
      comp[l] += std::fabs(acc[l]) >= std::fabs(x) ? (acc[l] - t) + x : (x - t) + acc[l];
      acc[l] = t;
    }
  }
  for (int l = 0; l < P; ++l) c->dE[l] = acc[l] + comp[l];
  ctx->stats.ms_total = ms[0];
  ctx->stats.ms_stage = ms[1];
  ctx->stats.ms_contract = ms[2];
  ctx->stats.ms_energy = ms[3];
  return LNO_OT_OK;
}

// ---------------------------------------------------------------------------
// Adjoint (float64).  Gradient accumulators of one domain (raw, unprojected).
struct GradAcc {
  Operand dBoo[2], dBov[2], dBvv[2];  // same layout as the DF blocks
  double* dt1[2];
  double* deps[2];
  double* dfov[2];                    // f_ov gradients (when the domain has f_ov)
  double* dt2aa;
  double* dt2bb;
  double* dt2ab;
};

int zeros(Arena& A, double** p, int64_t n, cudaStream_t st) {
  TRY(A.get(p, (size_t)std::max<int64_t>(n, 1)));
  CU(cudaMemsetAsync(*p, 0, (size_t)std::max<int64_t>(n, 1) * sizeof(double), st));
  return LNO_OT_OK;
}

int zero_operand_like(Arena& A, const Operand& src, Operand& d, cudaStream_t st) {
  d = src;
  const int64_t n = std::max<int64_t>((int64_t)src.nslot * src.rows * src.Kp, 8);
  return zeros(A, &d.f64, n, st);
}

// C[m ldc + n] (+)= alpha sum_k a(m, k) b(n, k) on the tensor cores: both views
// are cut into 4 BF16 slices with power-of-two scales (the DF assembly's
// representation, 10 slice products, float64 output: class 0 plus the float32 sum of
// the others).
// Used by the adjoint of the tensor-core precisions.
int tc_matmul(Run& R, Arena& A, int M, int N, int K, View a, View b, double* C, int64_t ldc,
              double alpha, bool accum, bool b_const) {
  if (M <= 0 || N <= 0 || K <= 0) return LNO_OT_OK;
  constexpr int S = 4;
  cudaStream_t st = R.st;
  cudaEvent_t e0 = R.event(), e1 = R.event();
  if (e0) cudaEventRecord(e0, st);
  // Split K when the output has few 128 x 128 tiles (a long contraction onto a
  // short output: the contraction adjoints over the pair rows, the DF adjoints
  // over v^2 rows): chunk c is problem c of one launch, writing its own float64
  // partial; the partials are added into C in chunk order.
  const int64_t tiles = (int64_t)ceil_div(N, 128) * ceil_div(M, 128);
  int nsp = 1;
  if (tiles < 2 * R.ctx->nsm && K >= 4096)
    nsp = (int)std::max<int64_t>(1, std::min<int64_t>({ceil_div(4 * R.ctx->nsm, tiles),
                                                       K / 2048, kMaxSplit}));
  nsp = std::max(nsp, ceil_div(K, kWideBF16));   // class sums within class_sum's range
  const int Kc = (int)round_up(ceil_div(K, nsp), 32);
  nsp = ceil_div(K, Kc);
  const int64_t Kp = round_up(Kc, 32);
  // a read-only B view sliced before with the same chunking
  const SliceCacheEntry* hit = nullptr;
  if (b_const)
    for (const auto& e : R.slice_cache)
      if (e.p == b.p && e.rs == b.rs && e.ks == b.ks && e.rows == N && e.K == K && e.Kc == Kc &&
          e.nsp == nsp)
        hit = &e;
  unsigned long long* am = R.ctx->d_amax;
  CU(cudaMemsetAsync(am, 0, 2 * sizeof(unsigned long long), st));
  CU(launch_view_absmax(a.p, a.rs, a.ks, M, K, am, st));
  if (!hit) CU(launch_view_absmax(b.p, b.rs, b.ks, N, K, am + 1, st));
  unsigned long long hb[2];
  CU(cudaMemcpyAsync(hb, am, sizeof hb, cudaMemcpyDeviceToHost, st));
  CU(cudaStreamSynchronize(st));
  double amax[2];
  std::memcpy(amax, hb, sizeof amax);
  if (hit) amax[1] = hit->sigma;
  if (!std::isfinite(amax[0]) || !std::isfinite(amax[1])) return LNO_OT_EINVAL;
  if (amax[0] == 0.0 || amax[1] == 0.0) {   // a zero operand: nothing to add
    if (!accum)
      for (int m = 0; m < M; ++m)
        CU(cudaMemsetAsync(C + (int64_t)m * ldc, 0, (size_t)N * sizeof(double), st));
    return LNO_OT_OK;
  }
  auto pow2_at_least = [](double x) {
    int e;
    const double f = std::frexp(x, &e);
    return std::ldexp(1.0, f == 0.5 ? e - 1 : e);
  };
  const double sa = pow2_at_least(amax[0]), sb = hit ? hit->sigma : pow2_at_least(amax[1]);
  __nv_bfloat16 *qa, *qb = hit ? hit->q : nullptr;
  TRY(A.get(&qa, (size_t)(S * nsp * M * Kp)));
  if (!qb) {
    if (b_const)
      TRY(R.arena.get(&qb, (size_t)(S * nsp * N * Kp)));
    else
      TRY(A.get(&qb, (size_t)(S * nsp * N * Kp)));
  }
  for (int c = 0; c < nsp; ++c) {
    const int k0 = c * Kc, kc = std::min(Kc, K - k0);
    CU(launch_view_slices<S>(a.p + k0 * a.ks, a.rs, a.ks, M, kc, (int)Kp, qa + c * M * Kp,
                             (int64_t)nsp * M * Kp, 128.0 / sa, st));
    if (!hit)
      CU(launch_view_slices<S>(b.p + k0 * b.ks, b.rs, b.ks, N, kc, (int)Kp, qb + c * N * Kp,
                               (int64_t)nsp * N * Kp, 128.0 / sb, st));
  }
  if (b_const && !hit) R.slice_cache.push_back({b.p, b.rs, b.ks, N, K, Kc, nsp, qb, sb});
  // the kernel writes its output transposed: its rows (A role) are n, its
  // columns (B role) m, so out[m ldc + n]
  CUtensorMap mA[2], mB[2];
  const PairTile tile = pair_tile_f64(S, nsp, N, M);
  TRY(make_operand_map(&mA[0], qb, Kp, (int64_t)nsp * N, S, (int64_t)nsp * N * Kp, 128, 2, S));
  TRY(make_operand_map(&mB[0], qa, Kp, (int64_t)nsp * M, S, (int64_t)nsp * M * Kp, tile.w / 2, 2,
                       S));
  mA[1] = mA[0];
  mB[1] = mB[0];
  double* part = nullptr;
  if (nsp > 1) TRY(A.get(&part, (size_t)nsp * M * N));
  // the output is formed with a power-of-two scale: |alpha| must be one (the
  // adjoint's products use +-1)
  int ex;
  if (std::frexp(std::fabs(alpha), &ex) != 0.5) return LNO_OT_EINVAL;
  const double scale = sa * sb * std::ldexp(1.0, -14) * std::fabs(alpha);
  std::vector<TcProb> pv(nsp);
  for (int c = 0; c < nsp; ++c) {
    TcProb& p = pv[c];
    p.nseg = 1;
    p.seg[0] = TcSeg{0, 0, c * N, c * M, std::min(Kc, K - c * Kc), alpha < 0 ? 1 : 0};
    p.flags = kTcFloatRest | (nsp == 1 && accum ? kTcAccum : 0);
    p.out = nsp == 1 ? C : part + (int64_t)c * M * N;
  }
  TcProb* dp;
  TRY(A.get(&dp, (size_t)nsp));
  CU(R.ctx->h2d(dp, pv.data(), nsp * sizeof(TcProb)));
  CU((launch_tc_pair_f64_group<S, kFmtBF16>(mA, mB, dp, nsp, N, M, nsp == 1 ? (int)ldc : N, scale,
                                            R.ctx->d_flag, R.ctx->nsm, st, kOutRows, tile)));
  if (nsp > 1) CU(launch_sum_partials(part, nsp, M, N, C, ldc, accum, st));
  if (e1) cudaEventRecord(e1, st);
  if (e0 && e1) R.contract_ev.push_back({e0, e1});
  R.stats->contract_launches++;
  R.stats->other_launches += 3 + 2 * nsp;
  A.drop(qa);
  if (!b_const) A.drop(qb);
  A.drop(dp);
  if (part) A.drop(part);
  return LNO_OT_OK;
}

// DF adjoint: out[n][m] = sum_Q L[l0+m][Q] R[r0+n][Q]  ->  dL, dR (+=)
int df_adjoint(Run& R, Arena& A, const Operand& Lo, Operand& dL, int64_t l0, int M,
               const Operand& Ro, Operand& dR, int64_t r0, int N, const double* dout, int ldo) {
  if (M <= 0 || N <= 0) return LNO_OT_OK;
  const int64_t Qp = Lo.Kp;
  if (R.tc_adjoint) {
    // dL[l0+m][Q] += sum_n dout[n][m] R[r0+n][Q];  dR[r0+n][Q] += sum_m dout[n][m] L[l0+m][Q]
    TRY(tc_matmul(R, A, M, R.naux, N, View{dout, 1, ldo}, View{Ro.f64 + r0 * Qp, 1, Qp},
                  dL.f64 + l0 * Qp, Qp, 1.0, true, true));
    TRY(tc_matmul(R, A, N, R.naux, M, View{dout, ldo, 1}, View{Lo.f64 + l0 * Qp, 1, Qp},
                  dR.f64 + r0 * Qp, Qp, 1.0, true, true));
    return LNO_OT_OK;
  }
  GemmS g[2];
  g[0] = GemmS{dout, Ro.f64 + r0 * Qp, dL.f64 + l0 * Qp, M, R.naux, N, 0,
               1, ldo, Qp, 1, Qp, 1, 1.0};
  g[1] = GemmS{dout, Lo.f64 + l0 * Qp, dR.f64 + r0 * Qp, N, R.naux, M, 0,
               ldo, 1, Qp, 1, Qp, 1, 1.0};
  GemmS* dg;
  TRY(A.get(&dg, 2));
  CU(R.ctx->h2d(dg, g, sizeof g));
  CU(launch_gemm_strided(dg, 1, M, R.naux, R.st));
  CU(launch_gemm_strided(dg + 1, 1, N, R.naux, R.st));
  R.stats->other_launches += 2;
  CU(cudaStreamSynchronize(R.st));  // g lives on the host stack
  A.drop(dg);
  return LNO_OT_OK;
}

// Operands of the adjoint in the batched form: slices of every slot in both
// layouts, kept while they are within kBatchBytes; otherwise the products run one
// by one (tc_matmul), slicing what they need.
constexpr int64_t kBatchBytes = (int64_t)8 << 30;

int backward_spin(SpinPass& P, GradAcc& G, double gE) {
  Run& R = P.R;
  cudaStream_t st = R.st;
  Arena A(st, 0);
  const int o = P.o, v = P.v, ot = P.ot, vt = P.vt, s = P.s, t = P.t;
  Operand dAT, dBT, dA1, dBG, dBF, dAT2;
  TRY(zero_operand_like(A, P.AT, dAT, st));
  TRY(zero_operand_like(A, P.BT, dBT, st));
  TRY(zero_operand_like(A, P.A1, dA1, st));
  TRY(zero_operand_like(A, P.BG, dBG, st));
  TRY(zero_operand_like(A, P.BF, dBF, st));
  TRY(zero_operand_like(A, P.AT2, dAT2, st));
  // gradients of the slot-compacted V-term blocks
  const int nS = (int)P.listBT.size(), nT = (int)P.listBF.size();
  const int64_t ns = (int64_t)nS * v, nt = (int64_t)nT * vt;
  double* dovss = nullptr;
  double* dovts = nullptr;
  TRY(zeros(A, &dovss, ns * ns, st));
  if (!P.mixed.trips.empty()) TRY(zeros(A, &dovts, nt * ns, st));
  double* dt2ss = s == 0 ? G.dt2aa : G.dt2bb;
  double* dt2st = G.dt2ab;
  if (s == 1 && !P.mixed.trips.empty()) TRY(zeros(A, &dt2st, (int64_t)o * ot * v * vt, st));

  // slices of all operand slots (batched form)
  const Operand* ops[6] = {&P.AT, &P.BT, &P.A1, &P.BG, &P.BF, &P.AT2};
  SlicedBatch sl[6];
  bool batched = R.tc_adjoint && !R.ctx->frugal;
  if (batched) {
    int64_t bytes = 0;
    for (const Operand* op : ops) {
      if (op->nslot * op->rows == 0) continue;
      bytes += SlicedBatch::bytes(op->nslot, op->rows, op->K, true);
      batched = batched && op->nslot <= 65535 && op->rows <= (1 << 20);
    }
    batched = batched && bytes <= kBatchBytes;
  }
  if (batched)
    for (int q = 0; q < 6; ++q) {
      if (ops[q]->nslot * ops[q]->rows == 0) continue;
      TRY(sl[q].alloc(A, ops[q]->nslot, (int)ops[q]->rows, ops[q]->K, true, true));
      TRY(sl[q].fill(R, ops[q]->f64, ops[q]->rows * ops[q]->Kp, ops[q]->Kp, ops[q]->nslot));
    }
  auto sliced = [&](const Operand* op) -> const SlicedBatch& {
    for (int q = 0; q < 6; ++q)
      if (ops[q] == op) return sl[q];
    return sl[0];
  };

  // ---- per case: recompute, energy adjoint, contraction adjoint ------------
  for (int im = 0; im < 2; ++im) {
    const bool is_mixed = im == 1;
    CaseSel& cs = is_mixed ? P.mixed : P.same;
    const int ntrip = (int)cs.trips.size();
    if (ntrip == 0) continue;
    if (v == 0 || (is_mixed && vt == 0)) continue;
    const int M1 = v;
    const int64_t N1 = is_mixed ? (int64_t)v * vt : npairs(v);
    const int P1 = (int)round_up(std::max(M1, 1), 16);
    const int M2 = vt;
    const int64_t N2 = is_mixed ? npairs(v) : 0;
    const int P2 = (int)round_up(std::max(M2, 1), 16);
    // X, dX and, in the batched form, the slices of dX in two layouts; there a group
    // is one launch per product, so it is as large as the budget allows
    const int64_t per = (N1 * P1 + N2 * P2) * 8 * (batched ? 4 : 2);
    int Gn = (int)std::max<int64_t>(
        1, std::min<int64_t>(batched ? 1024 : 32, ((int64_t)4 << 30) / std::max<int64_t>(per, 1)));
    Gn = std::min(Gn, ntrip);
    double *X, *Z = nullptr, *dX, *dZ = nullptr;
    TRY(A.get(&X, (size_t)(Gn * N1 * P1) + 8));
    TRY(A.get(&dX, (size_t)(Gn * N1 * P1) + 8));
    if (is_mixed) {
      TRY(A.get(&Z, (size_t)(Gn * N2 * P2) + 8));
      TRY(A.get(&dZ, (size_t)(Gn * N2 * P2) + 8));
    }
    std::vector<int3> blocks;
    const int nbs = (v + 15) / 16, nbt = (vt + 15) / 16;
    for (int a = 0; a < nbs; ++a)
      for (int b = a; b < nbs; ++b)
        if (!is_mixed) {
          for (int c = b; c < nbs; ++c) blocks.push_back(make_int3(a, b, c));
        } else {
          for (int c = 0; c < nbt; ++c) blocks.push_back(make_int3(a, b, c));
        }
    int3* dblocks;
    TRY(A.get(&dblocks, blocks.size()));
    CU(R.ctx->h2d(dblocks, blocks.data(), blocks.size() * sizeof(int3)));
    Trip* dtrips;
    TRY(A.get(&dtrips, (size_t)ntrip));
    CU(R.ctx->h2d(dtrips, cs.trips.data(), ntrip * sizeof(Trip)));
    const int Pch = std::max(1, std::min((int)blocks.size(), R.ctx->nsm * 4 / Gn + 1));
    SlicedBatch sx, sz;   // slices of a group's dX and dZ'
    if (batched) {
      TRY(sx.alloc(A, Gn, (int)N1, M1, true, true));
      if (is_mixed) TRY(sz.alloc(A, Gn, (int)N2, M2, true, true));
    }
    EnergyArgs ea{};
    ea.kind = is_mixed ? MIXED : SAME;
    ea.nvs = v;
    ea.nvt = is_mixed ? vt : v;
    ea.nos = o;
    ea.not_ = is_mixed ? ot : o;
    ea.eps_s = R.dom->eps[s];
    ea.eps_t = R.dom->eps[is_mixed ? t : s];
    ea.t1s = R.dom->t1[s];
    ea.t1t = R.dom->t1[is_mixed ? t : s];
    P.set_v_args(ea, is_mixed);
    ea.blocks = dblocks;
    ea.nblocks = (int)blocks.size();
    ea.pitch_x = P1;
    ea.pitch_z = P2;
    ea.x_stride = N1 * P1;
    ea.z_stride = N2 * P2;
    ProbF64* dpf;
    ProbF64* dpf2;
    GemmS* dgs;
    TRY(A.get(&dpf, (size_t)Gn));
    TRY(A.get(&dpf2, (size_t)Gn));
    TRY(A.get(&dgs, (size_t)Gn * 6));
    std::vector<ProbF64> pf(Gn), pf2(Gn);
    struct SegRef {
      const Operand* A;
      Operand* dA;
      int64_t arow;
      const Operand* B;
      Operand* dB;
      int64_t brow;
      double sign;
    };
    for (int g0 = 0; g0 < ntrip; g0 += Gn) {
      const int ng = std::min(Gn, ntrip - g0);
      std::vector<std::vector<SegRef>> segs1(ng), segs2(ng);
      for (int g = 0; g < ng; ++g) {
        const Trip tr = cs.trips[g0 + g];
        const int i = tr.i, j = tr.j, k = tr.k;
        if (!is_mixed) {
          const int64_t bp = npairs(v);
          segs1[g] = {{&P.AT, &dAT, (int64_t)P.slotAT[(size_t)j * o + k] * v, &P.BT, &dBT, P.slotBT[i] * bp, 1.0},
                      {&P.AT, &dAT, (int64_t)P.slotAT[(size_t)k * o + i] * v, &P.BT, &dBT, P.slotBT[j] * bp, 1.0},
                      {&P.AT, &dAT, (int64_t)P.slotAT[(size_t)i * o + j] * v, &P.BT, &dBT, P.slotBT[k] * bp, 1.0}};
        } else {
          const int K = k;
          const int64_t bp = npairs(v), bgr = (int64_t)v * vt;
          segs1[g] = {{&P.A1, &dA1, (int64_t)P.slotA1[(size_t)j * ot + K] * v, &P.BG, &dBG, P.slotBG[i] * bgr, 1.0},
                      {&P.A1, &dA1, (int64_t)P.slotA1[(size_t)i * ot + K] * v, &P.BG, &dBG, P.slotBG[j] * bgr, -1.0},
                      {&P.AT, &dAT, (int64_t)P.slotAT[(size_t)i * o + j] * v, &P.BF, &dBF, P.slotBF[K] * bgr, 1.0}};
          segs2[g] = {{&P.AT2, &dAT2, (int64_t)P.slotAT2[(size_t)j * ot + K] * vt, &P.BT, &dBT, P.slotBT[i] * bp, -1.0},
                      {&P.AT2, &dAT2, (int64_t)P.slotAT2[(size_t)i * ot + K] * vt, &P.BT, &dBT, P.slotBT[j] * bp, 1.0}};
        }
        auto fill = [&](ProbF64& pr, const std::vector<SegRef>& sg, double* out) {
          pr.nseg = (int)sg.size();
          for (size_t q = 0; q < sg.size(); ++q)
            pr.seg[q] = SegF64{sg[q].A->f64 + sg[q].arow * sg[q].A->Kp,
                               sg[q].B->f64 + sg[q].brow * sg[q].B->Kp, sg[q].A->K, sg[q].A->Kp,
                               sg[q].B->Kp, sg[q].sign};
          pr.XT = out;
        };
        fill(pf[g], segs1[g], X + (size_t)g * N1 * P1);
        if (is_mixed) fill(pf2[g], segs2[g], Z + (size_t)g * N2 * P2);
      }
      // recompute X (and Z')
      if (batched) {
        // XT[n][m] = sum_seg sign A[arow+m][:] . B[brow+n][:]: segment q of all the
        // group's triplets in one launch, the later ones added
        auto recompute = [&](const std::vector<std::vector<SegRef>>& segs, double* Xb, int64_t Nn,
                             int Mm, int ldo) -> int {
          for (size_t q = 0; q < segs[0].size(); ++q) {
            std::vector<TcProb> pr;
            const SegRef& r0 = segs[0][q];
            const SlicedBatch &a = sliced(r0.A), &b = sliced(r0.B);
            for (int g = 0; g < ng; ++g) {
              const SegRef& r = segs[g][q];
              const int ia = (int)(r.arow / a.rows), ib = (int)(r.brow / b.rows);
              TcProb p{};
              p.nseg = 1;
              p.seg[0] = TcSeg{0, 0, (int)r.brow, (int)r.arow, r.A->K, r.sign < 0 ? 1 : 0, 0};
              p.flags = kTcFloatRest | (q > 0 ? kTcAccum : 0);
              p.out = Xb + (size_t)g * Nn * ldo;
              p.ea = b.e + ib;
              p.eb = a.e + ia;
              pr.push_back(p);
            }
            TRY(grouped_products(R, A, pr, b, false, a, false, (int)Nn, Mm, ldo, kOutF64Rows));
          }
          return LNO_OT_OK;
        };
        TRY(recompute(segs1, X, N1, M1, P1));
        if (is_mixed) TRY(recompute(segs2, Z, N2, M2, P2));
      } else if (R.tc_adjoint) {
        // XT[n][m] = sum_seg sign A[arow+m][:] . B[brow+n][:], one tensor-core
        // product per segment, the later ones added
        auto recompute = [&](const std::vector<std::vector<SegRef>>& segs, double* Xb, int64_t Nn,
                             int Mm, int ldo) -> int {
          for (int g = 0; g < ng; ++g)
            for (size_t q = 0; q < segs[g].size(); ++q) {
              const SegRef& r = segs[g][q];
              TRY(tc_matmul(R, A, (int)Nn, Mm, r.A->K,
                            View{r.B->f64 + r.brow * r.B->Kp, r.B->Kp, 1},
                            View{r.A->f64 + r.arow * r.A->Kp, r.A->Kp, 1},
                            Xb + (size_t)g * Nn * ldo, ldo, r.sign, q > 0));
            }
          return LNO_OT_OK;
        };
        TRY(recompute(segs1, X, N1, M1, P1));
        if (is_mixed) TRY(recompute(segs2, Z, N2, M2, P2));
      } else {
        CU(R.ctx->h2d(dpf, pf.data(), ng * sizeof(ProbF64)));
        CU(launch_gemm_f64(dpf, ng, M1, (int)N1, P1, st));
        if (is_mixed) {
          CU(R.ctx->h2d(dpf2, pf2.data(), ng * sizeof(ProbF64)));
          CU(launch_gemm_f64(dpf2, ng, M2, (int)N2, P2, st));
        }
      }
      // energy adjoint -> dX, dT1, deps, V-integral gradients
      CU(cudaMemsetAsync(dX, 0, (size_t)ng * N1 * P1 * sizeof(double), st));
      if (is_mixed) CU(cudaMemsetAsync(dZ, 0, (size_t)ng * N2 * P2 * sizeof(double), st));
      ea.trips = dtrips + g0;
      cudaEvent_t ee0 = R.event(), ee1 = R.event();
      if (ee0) cudaEventRecord(ee0, st);
      CU(launch_energy_backward(ea, X, Z, dX, dZ, G.dt1[s], G.dt1[is_mixed ? t : s], dovss,
                                dovts, G.deps[s], G.deps[is_mixed ? t : s], gE, ng, Pch, st));
      if (ee1) cudaEventRecord(ee1, st);
      if (ee0 && ee1) R.energy_ev.push_back({ee0, ee1});
      if (R.fov[0]) {  // the f_ov part: planes are T2 amplitudes, coefficients f_ov
        EnergyArgs ef = ea;
        ef.vmode = 1;
        ef.t1s = R.fov[s];
        ef.t1t = R.fov[is_mixed ? t : s];
        ef.t2ss = P.t2ss;
        ef.t2st = P.t2st;
        CU(launch_energy_backward(ef, X, Z, dX, dZ, G.dfov[s], G.dfov[is_mixed ? t : s], dt2ss,
                                  dt2st, G.deps[s], G.deps[is_mixed ? t : s], gE, ng, Pch, st));
        R.stats->energy_launches += 1;
      }
      // contraction adjoint, batched: per operand pair (A, B) one launch of
      // dA[arow+m][k] += s sum_n dX[n][m] B[brow+n][k] over all triplets and
      // segments, one of dB[brow+n][k] += s sum_m dX[n][m] A[arow+m][k]
      auto adj_batched = [&](const std::vector<std::vector<SegRef>>& segs, const SlicedBatch& dx,
                             int64_t Nn, int Mm) -> int {
        std::vector<bool> done(segs[0].size(), false);
        for (size_t q0 = 0; q0 < segs[0].size(); ++q0) {
          if (done[q0]) continue;
          const SegRef& r0 = segs[0][q0];
          const SlicedBatch &a = sliced(r0.A), &b = sliced(r0.B);
          std::vector<TcProb> pa, pb;
          for (size_t q = q0; q < segs[0].size(); ++q) {
            if (segs[0][q].A != r0.A || segs[0][q].B != r0.B) continue;
            done[q] = true;
            for (int g = 0; g < ng; ++g) {
              const SegRef& r = segs[g][q];
              const int ia = (int)(r.arow / a.rows), ib = (int)(r.brow / b.rows);
              add_chunks(pa, ib * b.cols, g * Mm, (int)Nn, r.sign < 0,
                         r.dA->f64 + r.arow * r.A->Kp, kTcAtomic, b.e + ib, dx.e + g);
              add_chunks(pb, (int)(g * Nn), ia * a.cols, Mm, r.sign < 0,
                         r.dB->f64 + r.brow * r.B->Kp, kTcAtomic, dx.e + g, a.e + ia);
            }
          }
          TRY(grouped_products(R, A, pa, b, true, dx, true, r0.A->K, Mm, r0.A->Kp, kOutRows));
          TRY(grouped_products(R, A, pb, dx, false, a, true, (int)Nn, r0.A->K, r0.B->Kp,
                               kOutF64Rows));
        }
        return LNO_OT_OK;
      };
      if (batched) {
        TRY(sx.fill(R, dX, N1 * P1, P1, ng));
        TRY(adj_batched(segs1, sx, N1, M1));
        if (is_mixed) {
          TRY(sz.fill(R, dZ, N2 * P2, P2, ng));
          TRY(adj_batched(segs2, sz, N2, M2));
        }
        R.stats->energy_launches += 1;
        continue;
      }
      // contraction adjoint: dA += sign dX.B, dB += sign dX^T.A
      auto adj = [&](const std::vector<std::vector<SegRef>>& segs, const double* dXb, int64_t Nn,
                     int Mm, int ldo) -> int {
        if (R.tc_adjoint) {
          // dA[arow+m][k] += s sum_n dX[n][m] B[brow+n][k]
          // dB[brow+n][k] += s sum_m dX[n][m] A[arow+m][k]
          for (int g = 0; g < ng; ++g)
            for (const SegRef& r : segs[g]) {
              const double* dxg = dXb + (size_t)g * Nn * ldo;
              const int K = r.A->K;
              TRY(tc_matmul(R, A, Mm, K, (int)Nn, View{dxg, 1, ldo},
                            View{r.B->f64 + r.brow * r.B->Kp, 1, r.B->Kp},
                            r.dA->f64 + r.arow * r.A->Kp, r.A->Kp, r.sign, true));
              TRY(tc_matmul(R, A, (int)Nn, K, Mm, View{dxg, ldo, 1},
                            View{r.A->f64 + r.arow * r.A->Kp, 1, r.A->Kp},
                            r.dB->f64 + r.brow * r.B->Kp, r.B->Kp, r.sign, true));
            }
          return LNO_OT_OK;
        }
        for (int q = 0; q < 3; ++q) {  // one launch per segment position
          std::vector<GemmS> ga, gb;
          int maxKa = 0;
          for (int g = 0; g < ng; ++g) {
            if ((int)segs[g].size() <= q) continue;
            const SegRef& r = segs[g][q];
            const double* dxg = dXb + (size_t)g * Nn * ldo;
            const int K = r.A->K;
            maxKa = std::max(maxKa, K);
            ga.push_back(GemmS{dxg, r.B->f64 + r.brow * r.B->Kp, r.dA->f64 + r.arow * r.A->Kp,
                               Mm, K, (int)Nn, 1, 1, ldo, r.B->Kp, 1, r.A->Kp, 1, r.sign});
            gb.push_back(GemmS{dxg, r.A->f64 + r.arow * r.A->Kp, r.dB->f64 + r.brow * r.B->Kp,
                               (int)Nn, K, Mm, 1, ldo, 1, r.A->Kp, 1, r.B->Kp, 1, r.sign});
          }
          if (ga.empty()) continue;
          const int n = (int)ga.size();
          CU(R.ctx->h2d(dgs, ga.data(), n * sizeof(GemmS)));
          CU(launch_gemm_strided(dgs, n, Mm, maxKa, st));
          CU(R.ctx->h2d(dgs + Gn * 3, gb.data(), n * sizeof(GemmS)));
          CU(launch_gemm_strided(dgs + Gn * 3, n, (int)Nn, maxKa, st));
          CU(cudaStreamSynchronize(st));
        }
        return LNO_OT_OK;
      };
      TRY(adj(segs1, dX, N1, M1, P1));
      if (is_mixed) TRY(adj(segs2, dZ, N2, M2, P2));
      CU(cudaStreamSynchronize(st));
      R.stats->contract_launches += is_mixed ? 2 : 1;
      R.stats->energy_launches += 1;
    }
  }

  // ---- layout adjoints and DF adjoints ---------------------------------------
  auto upload_pairs = [&](const std::vector<int2>& l, int2** d) -> int {
    TRY(A.get(d, std::max<size_t>(l.size(), 1)));
    if (!l.empty())
      CU(R.ctx->h2d(*d, l.data(), l.size() * sizeof(int2)));
    return LNO_OT_OK;
  };
  if (!P.listAT.empty()) {
    double* doovoT;
    TRY(zeros(A, &doovoT, (int64_t)o * v * o * o, st));
    int2* dl;
    TRY(upload_pairs(P.listAT, &dl));
    CU(launch_adj_at_same(dl, (int)P.listAT.size(), o, v, dAT.Kp, dAT.f64, dt2ss, doovoT, st));
    TRY(df_adjoint(R, A, R.Boo[s], G.dBoo[s], 0, o * o, R.Bov[s], G.dBov[s], 0, o * v, doovoT,
                   o * o));
    A.drop(doovoT);
  }
  // Per-orbital DF blocks, batched: a run of orbitals x, x + 1, ... at a time,
  // dout[x][n][m] (n < r_rows, m < l_rows): dL[m][Q] += sum_n dout R[x r_rows + n][Q],
  // dR[x r_rows + n][Q] += sum_m dout L[m][Q].
  auto per_orbital = [&](const std::vector<int>& list, const Operand& L, Operand& dL,
                         int64_t l_rows, const Operand& Ro, Operand& dR, int r_rows,
                         auto&& layout) -> int {
    const auto runs = SpinPass::orb_runs(list, l_rows * r_rows, R.ctx->frugal);
    const int nmax = SpinPass::longest(runs);
    if (nmax == 0 || l_rows == 0 || r_rows == 0) return LNO_OT_OK;
    const int64_t blk = l_rows * r_rows;
    const int norb = (int)(Ro.total_rows() / r_rows);
    double* dout;
    TRY(A.get(&dout, (size_t)(blk * nmax)));
    SlicedBatch sL, sR, sd;
    TRY(sL.alloc(A, 1, (int)l_rows, R.naux, false, true));
    TRY(sL.fill(R, L.f64, 0, L.Kp, 1));
    TRY(sR.alloc(A, norb, r_rows, R.naux, false, true));
    TRY(sR.fill(R, Ro.f64, (int64_t)r_rows * Ro.Kp, Ro.Kp, norb));
    TRY(sd.alloc(A, nmax, r_rows, (int)l_rows, true, true));
    for (const auto& r : runs) {
      CU(cudaMemsetAsync(dout, 0, (size_t)(blk * r.n) * sizeof(double), st));
      for (int i = 0; i < r.n; ++i) CU(layout(r.q + i, r.x + i, dout + i * blk));
      TRY(sd.fill(R, dout, blk, (int)l_rows, r.n));
      std::vector<TcProb> pl, pr;
      for (int i = 0; i < r.n; ++i) {
        const int x = r.x + i;
        add_chunks(pl, (int)(i * l_rows), x * R.naux, r_rows, false, dL.f64, kTcAtomic, sd.e + i,
                   sR.e + x);
        add_chunks(pr, 0, i * r_rows, (int)l_rows, false, dR.f64 + (int64_t)x * r_rows * dR.Kp,
                   kTcAtomic, sL.e, sd.e + i);
      }
      TRY(grouped_products(R, A, pl, sd, true, sR, true, (int)l_rows, R.naux, dL.Kp,
                           kOutF64Rows));
      TRY(grouped_products(R, A, pr, sL, true, sd, false, R.naux, r_rows, dR.Kp, kOutRows));
    }
    A.drop(dout);
    for (SlicedBatch* b : {&sL, &sR, &sd}) {
      if (b->n) A.drop(b->n);
      A.drop(b->t);
      A.drop(b->e);
      A.drop(b->amax);
    }
    return LNO_OT_OK;
  };
  // within the run and slice budgets (one orbital's block may not be)
  const bool batched_df = batched && 24 * (int64_t)v * v * std::max(v, vt) <= kBatchBytes &&
                          24 * (int64_t)vt * vt * v <= kBatchBytes &&
                          SlicedBatch::bytes(1, (int64_t)std::max(v, vt) * std::max(v, vt), R.naux,
                                             false) <= kBatchBytes;
  if (batched_df) {
    TRY(per_orbital(P.listBT, R.Bvv[s], G.dBvv[s], (int64_t)v * v, R.Bov[s], G.dBov[s], v,
                    [&](int q, int x, double* d) {
                      return launch_adj_bt_same(q, x, o, v, dBT.Kp, dBT.f64, d, dt2ss, st);
                    }));
    TRY(per_orbital(P.listBG, R.Bvv[t], G.dBvv[t], (int64_t)vt * vt, R.Bov[s], G.dBov[s], v,
                    [&](int q, int x, double* d) {
                      return launch_adj_bg(q, x, o, v, ot, vt, dBG.Kp, dBG.f64, d, dt2st, st);
                    }));
    TRY(per_orbital(P.listBF, R.Bvv[s], G.dBvv[s], (int64_t)v * v, R.Bov[t], G.dBov[t], vt,
                    [&](int q, int x, double* d) {
                      return launch_adj_bf(q, x, o, v, ot, vt, dBF.Kp, dBF.f64, d, dt2st, st);
                    }));
  }
  if (!batched_df && !P.listBT.empty()) {
    double* dvv;
    TRY(A.get(&dvv, (size_t)v * v * v));
    for (size_t q = 0; q < P.listBT.size(); ++q) {
      const int x = P.listBT[q];
      CU(cudaMemsetAsync(dvv, 0, (size_t)v * v * v * sizeof(double), st));
      CU(launch_adj_bt_same((int)q, x, o, v, dBT.Kp, dBT.f64, dvv, dt2ss, st));
      TRY(df_adjoint(R, A, R.Bvv[s], G.dBvv[s], 0, v * v, R.Bov[s], G.dBov[s], (int64_t)x * v, v,
                     dvv, v * v));
    }
    A.drop(dvv);
  }
  if (!P.listA1.empty()) {
    double* djT;
    TRY(zeros(A, &djT, (int64_t)o * v * ot * ot, st));
    int2* dl;
    TRY(upload_pairs(P.listA1, &dl));
    CU(launch_adj_a1(dl, (int)P.listA1.size(), o, v, ot, vt, dA1.Kp, dA1.f64, dt2st, djT, st));
    TRY(df_adjoint(R, A, R.Bov[s], G.dBov[s], 0, o * v, R.Boo[t], G.dBoo[t], 0, ot * ot, djT,
                   o * v));
    A.drop(djT);
  }
  if (!batched_df && !P.listBG.empty()) {
    double* dgT;
    TRY(A.get(&dgT, (size_t)v * vt * vt));
    for (size_t q = 0; q < P.listBG.size(); ++q) {
      const int x = P.listBG[q];
      CU(cudaMemsetAsync(dgT, 0, (size_t)v * vt * vt * sizeof(double), st));
      CU(launch_adj_bg((int)q, x, o, v, ot, vt, dBG.Kp, dBG.f64, dgT, dt2st, st));
      TRY(df_adjoint(R, A, R.Bvv[t], G.dBvv[t], 0, vt * vt, R.Bov[s], G.dBov[s], (int64_t)x * v, v,
                     dgT, vt * vt));
    }
    A.drop(dgT);
  }
  if (!batched_df && !P.listBF.empty()) {
    double* dfT;
    TRY(A.get(&dfT, (size_t)vt * v * v));
    for (size_t q = 0; q < P.listBF.size(); ++q) {
      const int K = P.listBF[q];
      CU(cudaMemsetAsync(dfT, 0, (size_t)vt * v * v * sizeof(double), st));
      CU(launch_adj_bf((int)q, K, o, v, ot, vt, dBF.Kp, dBF.f64, dfT, dt2st, st));
      TRY(df_adjoint(R, A, R.Bvv[s], G.dBvv[s], 0, v * v, R.Bov[t], G.dBov[t], (int64_t)K * vt, vt,
                     dfT, v * v));
    }
    A.drop(dfT);
  }
  if (!P.listAT2.empty()) {
    double* dlT;
    TRY(zeros(A, &dlT, (int64_t)ot * vt * o * o, st));
    int2* dl;
    TRY(upload_pairs(P.listAT2, &dl));
    CU(launch_adj_at2(dl, (int)P.listAT2.size(), o, v, ot, vt, dAT2.Kp, dAT2.f64, dt2st, dlT, st));
    TRY(df_adjoint(R, A, R.Boo[s], G.dBoo[s], 0, o * o, R.Bov[t], G.dBov[t], 0, ot * vt, dlT,
                   o * o));
    A.drop(dlT);
  }
  // V-term blocks over the gathered rows, then added back into the Bov rows:
  // (ia|jb): L = R = BsS; (jb|KC): L = BsS rows (j,b), R = BsT rows (K,C)
  if (nS > 0) {
    Operand dBsS;
    TRY(zero_operand_like(A, P.BsS, dBsS, st));
    TRY(df_adjoint(R, A, P.BsS, dBsS, 0, (int)ns, P.BsS, dBsS, 0, (int)ns, dovss, (int)ns));
    if (dovts && nT > 0) {
      Operand dBsT;
      TRY(zero_operand_like(A, P.BsT, dBsT, st));
      TRY(df_adjoint(R, A, P.BsS, dBsS, 0, (int)ns, P.BsT, dBsT, 0, (int)nt, dovts, (int)ns));
      CU(launch_scatter_add_rows(dBsT.f64, G.dBov[t].f64, P.d_list_t, nT, (int64_t)vt * dBsT.Kp,
                                 st));
      R.stats->other_launches++;
    }
    CU(launch_scatter_add_rows(dBsS.f64, G.dBov[s].f64, P.d_list_s, nS, (int64_t)v * dBsS.Kp, st));
    R.stats->other_launches++;
  }
  if (s == 1 && !P.mixed.trips.empty())
    CU(launch_adj_transpose_t2ab(dt2st, ot, o, vt, v, G.dt2ab, st));
  CU(cudaStreamSynchronize(st));
  return LNO_OT_OK;
}

int backward_once(lno_ot_ctx* ctx, const lno_ot_domain* dom, double gE, lno_ot_grad* g) {
  TRY(validate(ctx, dom));
  const int nbas = dom->nbas, naux = dom->naux;
  const int na = dom->nocc[0], nb = dom->nocc[1];
  const int va = nbas - na, vb = nbas - nb;
  const int64_t nB = (int64_t)naux * nbas * nbas;
  const int64_t n1[2] = {(int64_t)na * va, (int64_t)nb * vb};
  const int64_t naa = (int64_t)na * na * va * va, nbb = (int64_t)nb * nb * vb * vb,
                nab = (int64_t)na * nb * va * vb;
  for (int s = 0; s < 2; ++s) {
    TRY(check_ptr(ctx, g->dB[s], false));
    TRY(check_ptr(ctx, g->deps[s], false));
    TRY(check_ptr(ctx, g->dt1[s], false));
    TRY(check_ptr(ctx, g->dfov[s], false));
  }
  TRY(check_ptr(ctx, g->dt2aa, false));
  TRY(check_ptr(ctx, g->dt2bb, false));
  TRY(check_ptr(ctx, g->dt2ab, false));
  CU(cudaSetDevice(ctx->device));
  ctx->stats = lno_ot_stats{};
  ctx->ev_used = 0;
  Run R(ctx, dom);
  R.f64 = true;
  R.S = 0;
  // float64 operands and energy adjoint; with a tensor-core precision the
  // contractions (X recompute, contraction and DF adjoints) run on the tensor
  // cores through tc_matmul
  R.tc_adjoint = ctx->prec != LNO_OT_FP64;
  CU(cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), ctx->stream));
  // wall-clock phases (the stream is synchronised at each boundary)
  using clk = std::chrono::steady_clock;
  const auto w0 = clk::now();
  double wbuild = 0.0;
  CaseSel cs[4];
  for (int c = 0; c < 4; ++c) TRY(select_case(dom, c, cs[c]));
  TRY(R.stage());
  CU(cudaStreamSynchronize(R.st));
  const double wstage = std::chrono::duration<double, std::milli>(clk::now() - w0).count();
  if (!R.fov[0] && (g->dfov[0] || g->dfov[1])) {
    // dE/df_ov at f_ov = 0 (E is affine in f_ov): run the f_ov pass on zeros
    for (int s = 0; s < 2; ++s) {
      double* z;
      TRY(zeros(R.arena, &z, n1[s], R.st));
      R.fov[s] = z;
    }
  }
  Arena GA(R.st, 0);
  GradAcc G{};
  for (int s = 0; s < 2; ++s) {
    TRY(zero_operand_like(GA, R.Boo[s], G.dBoo[s], R.st));
    TRY(zero_operand_like(GA, R.Bov[s], G.dBov[s], R.st));
    TRY(zero_operand_like(GA, R.Bvv[s], G.dBvv[s], R.st));
    TRY(zeros(GA, &G.dt1[s], n1[s], R.st));
    G.dfov[s] = nullptr;
    if (R.fov[0]) TRY(zeros(GA, &G.dfov[s], n1[s], R.st));
    TRY(zeros(GA, &G.deps[s], nbas, R.st));
  }
  // T2 gradients accumulate in the caller's buffers when given (projected in
  // place at the end), else in scratch
  auto acc_buf = [&](double* user, int64_t n, double** out) -> int {
    if (user) {
      CU(cudaMemsetAsync(user, 0, (size_t)std::max<int64_t>(n, 1) * sizeof(double), R.st));
      *out = user;
      return LNO_OT_OK;
    }
    return zeros(GA, out, n, R.st);
  };
  TRY(acc_buf(g->dt2aa, naa, &G.dt2aa));
  TRY(acc_buf(g->dt2bb, nbb, &G.dt2bb));
  TRY(acc_buf(g->dt2ab, nab, &G.dt2ab));
  double* e_dummy[4];
  for (int c = 0; c < 4; ++c)
    TRY(GA.get(&e_dummy[c], std::max<size_t>(cs[c].trips.size(), 1)));
  for (int s = 0; s < 2; ++s) {
    SpinPass P(R, s, s == 0 ? cs[0] : cs[3], s == 0 ? cs[1] : cs[2], e_dummy[s == 0 ? 0 : 3],
               e_dummy[s == 0 ? 1 : 2]);
    if (P.same.trips.empty() && P.mixed.trips.empty()) continue;
    const auto b0 = clk::now();
    P.plan();
    TRY(P.prepare_inputs());
    TRY(P.build_v_blocks());
    TRY(P.build());
    CU(cudaStreamSynchronize(R.st));
    wbuild += std::chrono::duration<double, std::milli>(clk::now() - b0).count();
    TRY(backward_spin(P, G, gE));
    CU(cudaStreamSynchronize(R.st));
  }
  // outputs: dB (symmetrised), deps, dt1, dt2 (antisymmetrised same-spin)
  for (int s = 0; s < 2; ++s) {
    const int o = dom->nocc[s], v = nbas - o;
    if (g->dB[s]) {  // raw gradient into the caller's buffer, symmetrised in place
      double* raw = g->dB[s];
      CU(cudaMemsetAsync(raw, 0, (size_t)nB * sizeof(double), R.st));
      CU(launch_adj_transpose_block(G.dBoo[s].f64, naux, nbas, 0, o, 0, o, G.dBoo[s].Kp, raw, R.st));
      CU(launch_adj_transpose_block(G.dBov[s].f64, naux, nbas, 0, o, o, v, G.dBov[s].Kp, raw, R.st));
      CU(launch_adj_transpose_block(G.dBvv[s].f64, naux, nbas, o, v, o, v, G.dBvv[s].Kp, raw, R.st));
      CU(launch_sym_inplace(raw, naux, nbas, R.st));
    }
    if (g->deps[s]) CU(launch_scale_copy(G.deps[s], nbas, 1.0, g->deps[s], R.st));
    if (g->dt1[s]) CU(launch_scale_copy(G.dt1[s], n1[s], 1.0, g->dt1[s], R.st));
    if (g->dfov[s]) CU(launch_scale_copy(G.dfov[s], n1[s], 1.0, g->dfov[s], R.st));
  }
  if (g->dt2aa) CU(launch_antisym_inplace(g->dt2aa, na, va, R.st));
  if (g->dt2bb) CU(launch_antisym_inplace(g->dt2bb, nb, vb, R.st));
  CU(cudaStreamSynchronize(R.st));
  int flag = 0;
  CU(cudaMemcpy(&flag, ctx->d_flag, sizeof flag, cudaMemcpyDeviceToHost));
  if (flag == 9) return LNO_OT_EINVAL;   // an infinite operand (slice_exponents)
  if (flag) return LNO_OT_ETIMEOUT;
  // stats of the adjoint: ms_total wall clock, ms_stage the staging plus the
  // operand and V-block builds (their DF assembly), ms_contract the event time
  // of its contractions (tensor-core products or float64 GEMMs), ms_energy the
  // energy adjoint kernels
  ctx->stats.ms_total = std::chrono::duration<double, std::milli>(clk::now() - w0).count();
  ctx->stats.ms_stage = wstage + wbuild;
  float ms = 0;
  double acc = 0;
  for (auto& p : R.contract_ev)
    if (cudaEventElapsedTime(&ms, p.first, p.second) == cudaSuccess) acc += ms;
  ctx->stats.ms_contract = acc;
  acc = 0;
  for (auto& p : R.energy_ev)
    if (cudaEventElapsedTime(&ms, p.first, p.second) == cudaSuccess) acc += ms;
  ctx->stats.ms_energy = acc;
  return LNO_OT_OK;
}

// Every gradient buffer is cleared or written by the call itself, so a second run
// leaves what a first one would.
int backward_impl(lno_ot_ctx* ctx, const lno_ot_domain* dom, double gE, lno_ot_grad* g) {
  ctx->frugal = ctx->small_pieces;
  int rc = backward_once(ctx, dom, gE, g);
  if (rc == LNO_OT_ENOMEM && !ctx->frugal) {
    ctx->frugal = true;
    rc = backward_once(ctx, dom, gE, g);
  }
  ctx->frugal = false;
  return rc;
}

}  // namespace

// ============================================================================
extern "C" {

int lno_ot_init(lno_ot_ctx** ctx, const lno_ot_options* opt) {
  if (!ctx || !opt) return LNO_OT_EINVAL;
  if (opt->precision < 0 || opt->precision > LNO_OT_BF16X15) return LNO_OT_EINVAL;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
    cudaGetLastError();
    return LNO_OT_ECUDA;
  }
  if (opt->device < 0 || opt->device >= ndev) return LNO_OT_EDEVICE;
  CU(cudaSetDevice(opt->device));
  cudaDeviceProp prop;
  CU(cudaGetDeviceProperties(&prop, opt->device));
  if (opt->precision != LNO_OT_FP64 && !(prop.major == 10 && prop.minor == 3))
    return LNO_OT_EUNSUPPORTED;  // the tensor-core path is built for sm_103a only
  lno_ot_ctx* c = new lno_ot_ctx();
  c->device = opt->device;
  c->prec = opt->precision;
  c->ws_limit = opt->workspace_bytes;
  c->nsm = prop.multiProcessorCount;
  if (opt->tune_cache && opt->tune_cache[0]) {  // "vmax bn group_cap" per line
    FILE* f = fopen(opt->tune_cache, "r");
    if (!f) {
      lno_ot_destroy(c);
      return LNO_OT_EINVAL;
    }
    char line[256];
    while (fgets(line, sizeof line, f)) {
      if (line[0] == '#') continue;
      lno_ot_ctx::TuneRow r;
      if (sscanf(line, "%d %d %d", &r.vmax, &r.bn, &r.group_cap) == 3 && r.vmax > 0)
        c->tune.push_back(r);
    }
    fclose(f);
    std::sort(c->tune.begin(), c->tune.end(),
              [](const lno_ot_ctx::TuneRow& a, const lno_ot_ctx::TuneRow& b) { return a.vmax < b.vmax; });
  }
  c->keep = opt->keep_operands != 0;
  // NULL = the legacy default stream (ordered with every blocking stream)
  c->stream = static_cast<cudaStream_t>(opt->stream);
  c->own_stream = false;
  // keep freed stream-ordered memory in the pool between calls
  cudaMemPool_t pool;
  if (cudaDeviceGetDefaultMemPool(&pool, c->device) == cudaSuccess) {
    uint64_t thr = UINT64_MAX;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
  }
  if (cudaMalloc(&c->d_sums, sizeof(CallState)) != cudaSuccess) {
    c->d_sums = nullptr;
    cudaGetLastError();
    lno_ot_destroy(c);
    return LNO_OT_ENOMEM;
  }
  c->d_amax = reinterpret_cast<unsigned long long*>(c->d_sums + 4);
  c->d_flag = reinterpret_cast<int*>(c->d_amax + kAmaxSlots);
  *ctx = c;
  return LNO_OT_OK;
}

void lno_ot_destroy(lno_ot_ctx* c) {
  if (!c) return;
  cudaSetDevice(c->device);
  if (c->stream) cudaStreamSynchronize(c->stream);
  destroy_cache(c->cache);
  c->cache = nullptr;
  if (c->stream) cudaStreamSynchronize(c->stream);
  for (auto e : c->ev_pool) cudaEventDestroy(e);
  cudaFree(c->d_sums);
  if (c->own_stream) cudaStreamDestroy(c->stream);
  delete c;
}

int lno_ot_energy(lno_ot_ctx* ctx, const lno_ot_domain* dom, lno_ot_result* out) {
  if (!ctx || !out) return LNO_OT_EINVAL;
  int rc = energy_impl(ctx, dom, out);
  out->status = rc;
  if (rc != LNO_OT_OK)
    for (double& e : out->e) e = 0.0;
  return rc;
}

int lno_ot_energy_batched(lno_ot_ctx* ctx, int ndom, const lno_ot_domain* doms,
                          lno_ot_result* out) {
  if (!ctx || ndom < 0 || (ndom > 0 && (!doms || !out))) return LNO_OT_EINVAL;
  int first = LNO_OT_OK;
  lno_ot_stats tot{};
  for (int d = 0; d < ndom; ++d) {
    int rc = lno_ot_energy(ctx, doms + d, out + d);
    if (rc != LNO_OT_OK && first == LNO_OT_OK) first = rc;
    const lno_ot_stats& s = ctx->stats;
    tot.ms_total += s.ms_total;
    tot.ms_stage += s.ms_stage;
    tot.ms_contract += s.ms_contract;
    tot.ms_energy += s.ms_energy;
    tot.flops_algorithmic += s.flops_algorithmic;
    tot.flops_executed += s.flops_executed;
    tot.tensor_flops += s.tensor_flops;
    tot.contract_launches += s.contract_launches;
    tot.energy_launches += s.energy_launches;
    tot.other_launches += s.other_launches;
    tot.triplets += s.triplets;
    tot.elements += s.elements;
  }
  ctx->stats = tot;
  return first;
}

int lno_ot_backward(lno_ot_ctx* ctx, const lno_ot_domain* dom, double gE, lno_ot_grad* g) {
  if (!ctx || !dom || !g) return LNO_OT_EINVAL;
  if (!std::isfinite(gE)) return LNO_OT_EINVAL;
  return backward_impl(ctx, dom, gE, g);
}

int lno_ot_energy_central(lno_ot_ctx* ctx, const lno_ot_domain* dom, const lno_ot_central* c) {
  if (!ctx) return LNO_OT_EINVAL;
  return central_impl(ctx, dom, c);
}

int lno_ot_naf(lno_ot_ctx* ctx, const lno_ot_domain* dom, double eps_naf, double* B_out[2],
               int* naux_out, double* eigenvalues) {
  if (!ctx) return LNO_OT_EINVAL;
  return naf_impl(ctx, dom, eps_naf, B_out, naux_out, eigenvalues);
}

int lno_ot_laplace_quadrature(double xmin, double xmax, double tol, int nmax, double* s,
                              double* w, int* nq) {
  return laplace_quadrature(xmin, xmax, tol, nmax, s, w, nq);
}

int lno_ot_release(lno_ot_ctx* ctx) {
  if (!ctx) return LNO_OT_EINVAL;
  if (cudaSetDevice(ctx->device) != cudaSuccess) {
    cudaGetLastError();
    return LNO_OT_ECUDA;
  }
  destroy_cache(ctx->cache);
  ctx->cache = nullptr;
  CU(cudaStreamSynchronize(ctx->stream));
  return LNO_OT_OK;
}

int lno_ot_last_stats(const lno_ot_ctx* ctx, lno_ot_stats* st) {
  if (!ctx || !st) return LNO_OT_EINVAL;
  *st = ctx->stats;
  return LNO_OT_OK;
}

const char* lno_ot_strerror(int code) {
  switch (code) {
    case LNO_OT_OK: return "ok";
    case LNO_OT_EINVAL: return "invalid argument (sizes, null pointer, nocc[1] > nocc[0])";
    case LNO_OT_EDEVICE: return "pointer is not device memory of the context's device";
    case LNO_OT_ENOMEM: return "device workspace allocation failed";
    case LNO_OT_ECUDA: return "CUDA call failed";
    case LNO_OT_ETIMEOUT: return "bounded device wait gave up";
    case LNO_OT_EUNSUPPORTED: return "unsupported option or input";
    default: return "unknown status";
  }
}

const char* lno_ot_version(void) { return "lno_ot 0.1 sm_103a"; }

int lno_ot_selftest_gemm(int device, int S, int M, int N, int K, const double* A, const double* B,
                         double* Cout, void* stream) {
  if (S < 1 || S > 5 || M <= 0 || N <= 0 || K <= 0 || !A || !B || !Cout) return LNO_OT_EINVAL;
  CU(cudaSetDevice(device));
  cudaDeviceProp prop;
  CU(cudaGetDeviceProperties(&prop, device));
  if (!(prop.major == 10 && prop.minor == 3)) return LNO_OT_EUNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Arena ar(st, 0);
  unsigned long long* amax;
  int* flag;
  TRY(ar.get(&amax, 2));
  TRY(ar.get(&flag, 1));
  CU(cudaMemsetAsync(amax, 0, 16, st));
  CU(cudaMemsetAsync(flag, 0, 4, st));
  CU(launch_absmax(A, (int64_t)M * K, amax, st));
  CU(launch_absmax(B, (int64_t)N * K, amax + 1, st));
  unsigned long long h[2];
  CU(cudaMemcpyAsync(h, amax, 16, cudaMemcpyDeviceToHost, st));
  CU(cudaStreamSynchronize(st));
  double ma, mb;
  std::memcpy(&ma, &h[0], 8);
  std::memcpy(&mb, &h[1], 8);
  const double sa = pow2_scale(ma), sb = pow2_scale(mb);
  const int Kp = (int)round_up(K, 8);
  const int64_t na = round_up((int64_t)M * Kp, 8), nb = round_up((int64_t)N * Kp, 8);
  __nv_bfloat16 *a16, *b16;
  TRY(ar.get(&a16, (size_t)(na * S)));
  TRY(ar.get(&b16, (size_t)(nb * S)));
  // slice on the host (diagnostic path only; the product path slices on the GPU)
  std::vector<double> ha((size_t)M * K), hb((size_t)N * K);
  CU(cudaMemcpyAsync(ha.data(), A, ha.size() * 8, cudaMemcpyDeviceToHost, st));
  CU(cudaMemcpyAsync(hb.data(), B, hb.size() * 8, cudaMemcpyDeviceToHost, st));
  CU(cudaStreamSynchronize(st));
  std::vector<uint16_t> sa16((size_t)na * S, 0), sb16((size_t)nb * S, 0);
  auto host_slices = [&](const std::vector<double>& src, int rows, std::vector<uint16_t>& dst,
                         int64_t stride, double sc) {
    for (int r = 0; r < rows; ++r)
      for (int k = 0; k < K; ++k) {
        double x = src[(size_t)r * K + k] * (128.0 / sc), w = 1.0;
        for (int q = 0; q < S; ++q) {
          double v = std::nearbyint(x * w) / w;
          x -= v;
          float f = (float)v;  // exact: at most 8 significant bits
          uint32_t u;
          std::memcpy(&u, &f, 4);
          dst[(size_t)q * stride + (size_t)r * Kp + k] = (uint16_t)(u >> 16);
          w *= 256.0;
        }
      }
  };
  host_slices(ha, M, sa16, na, sa);
  host_slices(hb, N, sb16, nb, sb);
  CU(cudaMemcpyAsync(a16, sa16.data(), sa16.size() * 2, cudaMemcpyHostToDevice, st));
  CU(cudaMemcpyAsync(b16, sb16.data(), sb16.size() * 2, cudaMemcpyHostToDevice, st));
  CUtensorMap mA[2], mB[2];
  TRY(make_operand_map(&mA[0], a16, Kp, M, S, na, 128));
  TRY(make_operand_map(&mB[0], b16, Kp, N, S, nb, sliced_product_bn(S)));
  mA[1] = mA[0];
  mB[1] = mB[0];
  TcProb p{};
  p.nseg = 1;
  p.seg[0] = TcSeg{0, 0, 0, 0, K, 0};
  p.out = Cout;
  TcProb* dp;
  TRY(ar.get(&dp, 1));
  CU(cudaMemcpyAsync(dp, &p, sizeof p, cudaMemcpyHostToDevice, st));
  const double scale = sa * sb * std::ldexp(1.0, -14);
  CU(launch_sliced_product(S, mA, mB, dp, M, N, scale, flag, prop.multiProcessorCount, st,
                           tc_normal()));
  int hflag = 0;
  CU(cudaMemcpyAsync(&hflag, flag, 4, cudaMemcpyDeviceToHost, st));
  CU(cudaStreamSynchronize(st));
  return hflag ? LNO_OT_ETIMEOUT : LNO_OT_OK;
}

int lno_ot_selftest_timeout(int device, long long wait_cycles, int* code, void* stream) {
  if (wait_cycles < 1000 || wait_cycles > tc_default_wait_cycles()) return LNO_OT_EINVAL;
  if (code) *code = 0;
  CU(cudaSetDevice(device));
  cudaDeviceProp prop;
  CU(cudaGetDeviceProperties(&prop, device));
  if (!(prop.major == 10 && prop.minor == 3)) return LNO_OT_EUNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // one 128 x 256 tile of a 2-slice product, K = 64: grid of one CTA
  constexpr int S = 2, SD = 4, M = 128, N = 256, K = 64;
  Arena ar(st, 0);
  int* flag;
  __nv_bfloat16 *a16, *b16;
  double* out;
  TcProb* dp;
  TRY(ar.get(&flag, 1));
  TRY(ar.get(&a16, (size_t)SD * M * K));
  TRY(ar.get(&b16, (size_t)SD * N * K));
  TRY(ar.get(&out, (size_t)M * N));
  TRY(ar.get(&dp, 1));
  CU(cudaMemsetAsync(flag, 0, 4, st));
  CU(cudaMemsetAsync(a16, 0, (size_t)SD * M * K * 2, st));
  CU(cudaMemsetAsync(b16, 0, (size_t)SD * N * K * 2, st));
  CUtensorMap mA[2], mB[2];
  TRY(make_operand_map(&mA[0], a16, K, M, S, (int64_t)M * K, 128));
  TRY(make_operand_map(&mB[0], b16, K, N, S, (int64_t)N * K, sliced_product_bn(S)));
  mA[1] = mA[0];
  mB[1] = mB[0];
  TcProb p{};
  p.nseg = 1;
  p.seg[0] = TcSeg{0, 0, 0, 0, K, 0};
  p.out = out;
  CU(cudaMemcpyAsync(dp, &p, sizeof p, cudaMemcpyHostToDevice, st));
  CU(launch_sliced_product(S, mA, mB, dp, M, N, 1.0, flag, 1, st, TcDiag{wait_cycles, 1}));
  int hflag = 0;
  CU(cudaMemcpyAsync(&hflag, flag, 4, cudaMemcpyDeviceToHost, st));
  CU(cudaStreamSynchronize(st));
  if (hflag) {   // the same of the pair kernel: one tile, one pair
    const PairTile t = pair_tile(S, N, 0);
    TRY(make_operand_map(&mA[0], a16, K, M, S, (int64_t)M * K, 128, 2, S));
    TRY(make_operand_map(&mB[0], b16, K, N, S, (int64_t)N * K, t.w / 2, 2, S));
    mA[1] = mA[0];
    mB[1] = mB[0];
    CU(cudaMemsetAsync(flag, 0, 4, st));
    CU((launch_tc_pair<S, kFmtBF16>(mA, mB, dp, 1, M, N, N, 1.0, flag, 2, st,
                                    TcDiag{wait_cycles, 1}, TcOut{kOutRows, 0, 0, 0}, t)));
    CU(cudaMemcpyAsync(&hflag, flag, 4, cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
  }
  for (int mode : {kOutRows, kOutF64Rows}) {   // and of its float64 outputs
    if (!hflag) break;
    const PairTile t = pair_tile_f64(SD, 1, M, N);
    TRY(make_operand_map(&mA[0], a16, K, M, SD, (int64_t)M * K, 128, 2, SD));
    TRY(make_operand_map(&mB[0], b16, K, N, SD, (int64_t)N * K, t.w / 2, 2, SD));
    mA[1] = mA[0];
    mB[1] = mB[0];
    CU(cudaMemsetAsync(flag, 0, 4, st));
    CU((launch_tc_pair_f64_group<SD, kFmtBF16>(mA, mB, dp, 1, M, N, mode == kOutRows ? M : N, 1.0,
                                               flag, 2, st, mode, t, TcDiag{wait_cycles, 1})));
    CU(cudaMemcpyAsync(&hflag, flag, 4, cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
  }
  if (code) *code = hflag;
  return hflag ? LNO_OT_ETIMEOUT : LNO_OT_OK;
}

int lno_ot_selftest_small_pieces(lno_ot_ctx* ctx, int on) {
  if (!ctx) return LNO_OT_EINVAL;
  ctx->small_pieces = on != 0;
  return LNO_OT_OK;
}

int lno_ot_selftest_energy_timeout(int device, long long wait_cycles, int* code, void* stream) {
  if (wait_cycles < 1000 || wait_cycles > tc_default_wait_cycles()) return LNO_OT_EINVAL;
  if (code) *code = 0;
  CU(cudaSetDevice(device));
  cudaDeviceProp prop;
  CU(cudaGetDeviceProperties(&prop, device));
  if (!(prop.major == 10 && prop.minor == 3)) return LNO_OT_EUNSUPPORTED;
  int h = 0;
  CU(energy_timeout_selftest(wait_cycles, prop.multiProcessorCount, &h,
                             static_cast<cudaStream_t>(stream)));
  if (code) *code = h;
  return h ? LNO_OT_ETIMEOUT : LNO_OT_OK;
}

const char* lno_ot_last_error(void) { return g_last_error.c_str(); }

}  // extern "C"
