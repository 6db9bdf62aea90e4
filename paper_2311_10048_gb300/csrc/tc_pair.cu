// Tensor-core contraction on CTA pairs for sm_103a: tcgen05.mma.cta_group::2
// (256 x w tiles, FP32 accumulators in TMEM) fed by TMA, on sliced float64
// operands.  Runs the W contractions (float32 row-major output), the DF assembly
// (float64 output out[n][m], or only its largest magnitude) and the adjoint's
// products.  One TMEM accumulator per weight class g = p + q of the slice products,
// so that none is rounded at the magnitude of a larger one; the classes are added
// smallest first (float32 output) or as integers (class_sum.cuh).  A class is exact
// while it stays below 2^24 of its unit: on BF16 slices for any data to K = 1024 / (g +
// 1) and for random signs far beyond; on FP16 slices class 0 is shown to be (row norms,
// lno_ot.cu), classes 1 and 2 may round at 2^-24 of themselves; TF32 rounds.
//
// What bounds it: the feed from L2 into shared memory.  A tile that one CTA
// computes alone loads S (128 + w) 64-byte rows per k block; measured on five
// shapes every launch of that form moved 8.0-9.2 TB/s of operand rows whatever its
// tensor rate (21-60%); this form moves 11.4 TB/s at 182 virtuals (tensor pipe 63%
// active) and at 360 (87%).  So
//  * the two CTAs of a pair share one 256 x w tile: each loads its 128 rows of
//    the long (pair) operand and half of the w rows of the short one, and the
//    tensor cores of both read both halves: S (128 + w / 2) rows per k block;
//  * w is not a constant: the n-tiles of a problem are as equal as multiples
//    of 16 allow, up to what S accumulators leave of TMEM (S w <= 512, at most
//    256), and the box of the short operand has w / 2 rows, so no n-tile loads
//    rows that it does not use;
//  * operand rows start on 64-byte boundaries, so a 64-byte box row is two
//    sectors (pitches that were multiples of 16 bytes moved 1.3x the payload).
//
// Kernel structure (one CTA per SM, pairs persistent over tiles):
//   warp 0   TMA producer of its CTA (one elected lane); completion of both
//            CTAs' copies on the leader's full barriers
//   warp 1   leader: MMA issuer (the warp waits, one elected lane issues),
//            commits to both CTAs' barriers
//   warps 2-9  epilogue, two warps per 32-lane quarter (even and odd 16-column
//            chunks): TMEM -> registers, TMEM released, then global stores.
//            Two accumulator sets where 2 S w <= 512, so the next tile's MMAs
//            run during the whole epilogue.
// Every wait is bounded; on a timeout the kernel records an error code, lets
// its copies and MMAs finish, frees TMEM and returns.
#include <algorithm>
#include <cmath>

#include "class_sum.cuh"
#include "common.cuh"
#include "ptx.cuh"

namespace lno {

namespace {

constexpr int BM = 128;                    // rows of one CTA (256 per pair)
constexpr int BK = 32;                     // 16-bit elements per 64-byte row, SWIZZLE_64B
constexpr long long kWaitCycles = 4000000000LL;
constexpr int kSmemBytes = 227 * 1024;
constexpr int kMaxStages = 16;
constexpr int kF64Width = 64;              // widest tile of a float64-output launch
constexpr int kBarBytes = 512;
// Epilogue warps: float32 output 8 (up to 80 columns of results a thread);
// float64 output 16, for its integer conversions
template <typename OutT>
constexpr int epi_warps() {
  return sizeof(OutT) == 4 ? 8 : 16;
}
template <typename OutT>
constexpr int pair_threads() {
  return 64 + 32 * epi_warps<OutT>();
}

__device__ __noinline__ bool pair_wait(uint32_t bar, uint32_t parity, int* flag, int code,
                                       bool abortable, long long limit = kWaitCycles) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255u) == 0) {
      if (abortable && *(volatile int*)flag != 0) return false;
      if (clock64() - t0 > limit) {
        atomicCAS(flag, 0, code);
        return false;
      }
    }
  }
}

// The same for a whole warp: all lanes return the same, so that none runs a
// warp-wide instruction (tcgen05.ld, shuffles) without the others after an abort.
__device__ __noinline__ bool pair_wait_warp_slow(uint32_t bar, uint32_t parity, int* flag,
                                                 int code, long long limit) {
  const long long t0 = clock64();
  for (uint32_t it = 1;; ++it) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if ((it & 255u) == 0) {
      if (__any_sync(0xffffffffu, *(volatile int*)flag != 0)) return false;
      if (__any_sync(0xffffffffu, clock64() - t0 > limit)) {
        if ((threadIdx.x & 31) == 0) atomicCAS(flag, 0, code);
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool pair_wait_warp(uint32_t bar, uint32_t parity, int* flag, int code,
                                               long long limit) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  return pair_wait_warp_slow(bar, parity, flag, code, limit);
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// shared::cluster address of `addr` in the CTA of rank `rank`
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar)
               : "memory");
}
// Tiled load into this CTA's shared memory that completes on a barrier of
// either CTA of the pair.
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map,
                                                 uint32_t bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}

// One pair MMA with a collector-buffer usage for A (consecutive MMAs that
// share slice pa of A read it from shared memory once).
#define LNO_PAIR_MMA(NAME, KIND, COLL)                                                     \
  __device__ __forceinline__ void NAME(uint32_t d, uint64_t a, uint64_t b, uint32_t id,    \
                                       uint32_t acc) {                                     \
    asm volatile("{\n\t.reg .pred p;\n\t"                                                  \
                 "setp.ne.b32 p, %4, 0;\n\t"                                               \
                 "tcgen05.mma.cta_group::2.kind::" KIND COLL " [%0], %1, %2, %3, p;\n\t}" ::"r"( \
                     d),                                                                   \
                 "l"(a), "l"(b), "r"(id), "r"(acc)                                         \
                 : "memory");                                                              \
  }
LNO_PAIR_MMA(pmma_f16, "f16", "")
LNO_PAIR_MMA(pmma_f16_fill, "f16", ".collector::a::fill")
LNO_PAIR_MMA(pmma_f16_use, "f16", ".collector::a::use")
LNO_PAIR_MMA(pmma_f16_last, "f16", ".collector::a::lastuse")
LNO_PAIR_MMA(pmma_tf32, "tf32", "")
LNO_PAIR_MMA(pmma_tf32_fill, "tf32", ".collector::a::fill")
LNO_PAIR_MMA(pmma_tf32_use, "tf32", ".collector::a::use")
LNO_PAIR_MMA(pmma_tf32_last, "tf32", ".collector::a::lastuse")
#undef LNO_PAIR_MMA

// mode 0: no collector, 1: fill, 2: use, 3: last use
template <int FMT>
__device__ __forceinline__ void pair_mma(int mode, uint32_t d, uint64_t a, uint64_t b,
                                         uint32_t id, uint32_t acc) {
  if constexpr (FMT == kFmtTF32) {
    if (mode == 1) pmma_tf32_fill(d, a, b, id, acc);
    else if (mode == 2) pmma_tf32_use(d, a, b, id, acc);
    else if (mode == 3) pmma_tf32_last(d, a, b, id, acc);
    else pmma_tf32(d, a, b, id, acc);
  } else {
    if (mode == 1) pmma_f16_fill(d, a, b, id, acc);
    else if (mode == 2) pmma_f16_use(d, a, b, id, acc);
    else if (mode == 3) pmma_f16_last(d, a, b, id, acc);
    else pmma_f16(d, a, b, id, acc);
  }
}

// Arrive on the barrier at this offset in every CTA of `mask` when the MMAs
// issued so far are complete.
__device__ __forceinline__ void pair_commit(uint32_t bar, uint16_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32"
      " {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Shared-memory matrix descriptor: K-major, 64-byte swizzle, rows of 64 B in
// groups of 8 (stride 512 B between groups).
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;            // leading byte offset (unused when swizzled)
  d |= (uint64_t)(512 >> 4) << 32;   // stride byte offset
  d |= (uint64_t)1 << 46;            // descriptor version for tcgen05
  d |= (uint64_t)4 << 61;            // SWIZZLE_64B
  return d;
}

// Instruction descriptor: D FP32, A/B K-major of format FMT (0 FP16, 1 BF16,
// 2 TF32), M = 256 over the pair, N = n (a multiple of 16, 16..256).
template <int FMT>
__device__ __forceinline__ uint32_t idesc_pair(int neg, int n) {
  constexpr uint32_t fmt = (uint32_t)FMT;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)neg << 13) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(2 * BM >> 4) << 24);
}

// Where one output row goes: 16-column chunk c (columns 16 c .. 16 c + 15) at
// p + c * step, its four 16-byte pieces permuted by q ^ sw.
struct RowOut {
  float* p;
  int64_t step;
  int sw;
};

__device__ __forceinline__ RowOut row_out(float* out, const TcOut& lay, int ldo, int m) {
  if (lay.mode == kOutYTile) {
    const int b = m / lay.nvt, c = m - b * lay.nvt;
    const int r = ((b & 15) << 4) | (c & 15);
    return {out + (int64_t)((b >> 4) * lay.nbt + (c >> 4)) * lay.nbs * kTile + r * 16, kTile,
            (r >> 1) & 3};
  }
  if (lay.mode == kOutZTile) {   // m = pair(a, b) = b (b - 1) / 2 + a
    int b = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)m)) * 0.5f);
    while ((int64_t)b * (b - 1) / 2 > m) --b;
    while ((int64_t)(b + 1) * b / 2 <= m) ++b;
    const int a = m - (int)((int64_t)b * (b - 1) / 2);
    const int A = a >> 4, B = b >> 4;
    const int r = ((a & 15) << 4) | (b & 15), slot = r ^ ((r >> 1) & 1);
    return {out + (int64_t)(B * (B + 1) / 2 + A) * lay.nbt * kTile + slot * 16, kTile, 0};
  }
  return {out + (int64_t)m * ldo, 16, 0};
}

// 32 bytes, 32-byte aligned: one full L2 sector (16-byte stores leave it two
// masked half-sector writes).
__device__ __forceinline__ void store32(float* d, const float* lo, const float* hi, bool swap) {
  float x[8];
#pragma unroll
  for (int j = 0; j < 4; ++j) {   // selects: lanes of one warp differ in `swap`
    x[j] = swap ? hi[j] : lo[j];
    x[4 + j] = swap ? lo[j] : hi[j];
  }
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(d), "f"(x[0]),
               "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(x[4]), "f"(x[5]), "f"(x[6]), "f"(x[7])
               : "memory");
}

// One chunk of a row; `left` = columns that remain in the row (only those are
// written).
__device__ __forceinline__ void store_chunk(const RowOut& ro, int chunk, const float* v,
                                            int left) {
  float* p = ro.p + chunk * ro.step;
  if (left >= 16) {
#pragma unroll
    for (int h = 0; h < 2; ++h)   // pieces 2 h, 2 h + 1 land in one 32-byte sector
      store32(p + ((h ^ (ro.sw >> 1)) << 3), v + 8 * h, v + 8 * h + 4, ro.sw & 1);
    return;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float* d = p + ((q ^ ro.sw) << 2);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (4 * q + j < left) d[j] = v[4 * q + j];
  }
}

// Columns of one tile: S accumulators in TMEM, N <= 256.  Float64 output: 64, and
// two accumulator sets (2 S w <= 512), so its long epilogue (~100 instructions an
// element) runs beside the next tile's MMAs, converting and storing 8 columns at a
// time (holding a 128-column tile's results to free TMEM first spilled, and a K =
// 60 product of 2809 x 53 outputs took 5.5 us an output tile instead of 1.5).
template <int S, typename OutT>
constexpr int pair_max_width() {
  return sizeof(OutT) == 4 ? std::min(256, 512 / S / 16 * 16)
                           : std::min(kF64Width, 256 / S / 16 * 16);
}

// TF32: 32-bit elements, 16 per 64-byte row, K 8 per MMA; the 16-bit formats
// have 32 per row, K 16.  ROWS: float64 output as out[m][n]; WIDE: its
// K may pass what class_sum needs no checks for.  diag is the bounded-wait test hook (TcDiag).
template <int S, int FMT, typename OutT, bool ROWS, bool WIDE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(pair_threads<OutT>(), 1)
tc_pair_gemm(const __grid_constant__ CUtensorMap mapA0, const __grid_constant__ CUtensorMap mapA1,
             const __grid_constant__ CUtensorMap mapB0, const __grid_constant__ CUtensorMap mapB1,
             const TcProb* __restrict__ probs, const __grid_constant__ TcProb one, int nprob, int M,
             int N, int ldo, float scale, int escale, int* __restrict__ flag,
             unsigned long long* __restrict__ amax, TcDiag diag, TcOut lay, PairTile tile) {
  constexpr int BKE = FMT == kFmtTF32 ? BK / 2 : BK;   // elements per 64-byte row
  constexpr int KM = FMT == kFmtTF32 ? 8 : 16;         // K of one MMA
  constexpr int kABytes = BM * 64;                     // one slice of this CTA's A rows
  constexpr int kEpiWarps = epi_warps<OutT>();
  constexpr float kW = 1.0f / 2048.0f;                 // weight step of FP16 classes
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int bbytes = tile.w * 32;                      // one slice of its half of the B rows
  const int stage_bytes = S * (kABytes + bbytes);
  const int nst = tile.stages, nbuf = tile.nbuf;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + kSmemBytes - kBarBytes);
  // bars: full[16], empty[16], tfull[2], tempty[2], drain; then the TMEM address
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 5);
  auto full_bar = [&](int s) { return smem_u32(bars + s); };
  auto empty_bar = [&](int s) { return smem_u32(bars + kMaxStages + s); };
  auto tfull = [&](int b) { return smem_u32(bars + 2 * kMaxStages + b); };
  auto tempty = [&](int b) { return smem_u32(bars + 2 * kMaxStages + 2 + b); };
  const uint32_t drain = smem_u32(bars + 2 * kMaxStages + 4);
  const uint32_t base = smem_u32(smem);

  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nM = (M + 2 * BM - 1) / (2 * BM), nN = tile.nN;
  const long long nunits = (long long)nprob * nM * nN;
  const long long u0 = blockIdx.x >> 1, ustep = gridDim.x >> 1;
  const long long wlim = diag.wait_cycles;
  // unit -> (problem, m-tile, n-tile), n fastest: the pairs that run together
  // share m-tiles of the long operand (read from HBM once) and the short
  // operand of a problem (resident in L2)
  auto decode = [&](long long u, int& mt, int& nt, long long& pr) {
    nt = (int)(u % nN);
    const long long r = u / nN;
    mt = (int)(r % nM);
    pr = r / nM;
  };
  auto ntile_w = [&](int nt) { return min(tile.w, (N - nt * tile.w + 15) & ~15); };

  if (warp == 0 && lane == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull(b), 1);
      mbar_init(tempty(b), 2 * kEpiWarps);
    }
    mbar_init(drain, 1);
    mbar_init_fence();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // both CTAs' barriers are initialised
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // ------------------------------ producer -------------------------------
      int stage = 0;
      uint32_t phase = 0, used = 0, last_phase = 0;
      bool ok = diag.starve == 0;
      for (long long u = u0; u < nunits && ok; u += ustep) {
        int mt, nt;
        long long pr;
        decode(u, mt, nt, pr);
        const TcProb& P = probs ? probs[pr] : one;
        const int ar = mt * 2 * BM + (int)rank * BM;
        const int br = nt * tile.w + (int)rank * (ntile_w(nt) >> 1);
        for (int sg = 0; sg < P.nseg && ok; ++sg) {
          const TcSeg seg = P.seg[sg];
          const CUtensorMap* ma = seg.amap ? &mapA1 : &mapA0;
          const CUtensorMap* mb = seg.bmap ? &mapB1 : &mapB0;
          for (int k0 = 0; k0 < seg.K; k0 += BKE) {
            if (!pair_wait(empty_bar(stage), phase ^ 1u, flag, 1, true, wlim)) {
              ok = false;
              break;
            }
            // the leader's full barrier takes the bytes of both CTAs
            if (rank == 0) mbar_expect_tx(full_bar(stage), 2u * (uint32_t)stage_bytes);
            const uint32_t bar = map_rank(full_bar(stage), 0);
            const uint32_t dst = base + (uint32_t)(stage * stage_bytes);
            tma_load_3d_pair(dst, ma, bar, seg.k0 + k0, seg.a_row + ar, 0);
            tma_load_3d_pair(dst + S * kABytes, mb, bar, seg.k0 + k0, seg.b_row + br, 0);
            used |= 1u << stage;
            last_phase = (last_phase & ~(1u << stage)) | (phase << stage);
            if (++stage == nst) {
              stage = 0;
              phase ^= 1u;
            }
          }
        }
      }
      // Every stage that this thread filled must have been read (so the copies
      // have landed and no arrival on this CTA's barriers is pending) before
      // the CTA leaves.  After an abort nobody reads them: the leader waits for
      // the copies that both sides issued, and both give the rest time to land.
      for (int s = 0; s < nst; ++s)
        if (used & (1u << s)) {
          if (ok && pair_wait(empty_bar(s), (last_phase >> s) & 1u, flag, 4, true)) continue;
          ok = false;
          if (rank == 0) pair_wait(full_bar(s), (last_phase >> s) & 1u, flag, 4, false, 20000000);
        }
      if (!ok && used) {
        const long long t0 = clock64();
        while (clock64() - t0 < 20000000) {
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // -------------------------------- MMA ----------------------------------
      // The whole warp runs the loop and one elected lane issues: descriptors
      // and addresses are then warp-uniform values.  (Issued from a loop that
      // one lane ran alone, an MMA cost ~76 cycles of issue and the tensor pipe
      // idled 40-60% whatever the loads did.)
      const bool el = elect_one();
      const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
      int stage = 0;
      uint32_t phase = 0, it = 0;
      bool ok = true, any = false;
      for (long long u = u0; u < nunits && ok; u += ustep, ++it) {
        int mt, nt;
        long long pr;
        decode(u, mt, nt, pr);
        const TcProb& P = probs ? probs[pr] : one;
        const int buf = nbuf == 2 ? (int)(it & 1u) : 0;
        const uint32_t use = nbuf == 2 ? it >> 1 : it;   // how often this buffer was used
        const int nseg = P.nseg, nw = ntile_w(nt);
        TcSeg seg = P.seg[0];
        if (use > 0 && !pair_wait_warp(tempty(buf), (use - 1) & 1u, flag, 2, wlim)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t dt = tm + (uint32_t)(buf * S * tile.w);
        uint32_t acc0 = 0;   // 0 until every class accumulator has been written
        for (int sg = 0; sg < nseg && ok; ++sg) {
          const uint32_t idesc = idesc_pair<FMT>(seg.neg, nw);
          const int K = seg.K;
          if (sg + 1 < nseg) seg = P.seg[sg + 1];
          for (int k0 = 0; k0 < K; k0 += BKE) {
            if (!pair_wait_warp(full_bar(stage), phase, flag, 3, wlim)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sa = base + (uint32_t)(stage * stage_bytes);
            const uint64_t a0 = sdesc_sw64(sa), b0 = sdesc_sw64(sa + S * kABytes);
            if (el) {
#pragma unroll
              for (int ks = 0; ks < 2; ++ks) {   // two 32-byte MMA steps per 64-byte row
                if (k0 + ks * KM < K) {
#pragma unroll
                  for (int pa = 0; pa < S; ++pa) {
#pragma unroll
                    for (int pb = 0; pb + pa < S; ++pb) {
                      const int last = S - 1 - pa;
                      const int mode = last == 0 ? 0 : pb == 0 ? 1 : pb == last ? 3 : 2;
                      // shared addresses stay below 2^18: no carry out of the address field
                      pair_mma<FMT>(mode, dt + (uint32_t)((pa + pb) * tile.w),
                                    a0 + (uint64_t)((pa * kABytes + ks * 32) >> 4),
                                    b0 + (uint64_t)((pb * bbytes + ks * 32) >> 4), idesc,
                                    pa == 0 ? acc0 : 1u);
                    }
                  }
                  acc0 = 1;
                }
              }
              pair_commit(empty_bar(stage), 3);
            }
            acc0 = 1;
            any = true;
            if (++stage == nst) {
              stage = 0;
              phase ^= 1u;
            }
          }
        }
        if (ok && el) pair_commit(tfull(buf), 3);
      }
      if (!ok && any) {  // this warp's MMAs end before TMEM is released
        if (el) pair_commit(drain, 1);
        pair_wait(drain, 0, flag, 5, false);
      }
    }
  } else {
    // ------------------------------- epilogue ---------------------------------
    const int q = warp & 3, part = (warp - 2) >> 2;   // TMEM quarter, column share
    const int row = (int)rank * BM + q * 32 + lane;
    uint32_t it = 0;
    float lmax = 0.f;
    for (long long u = u0; u < nunits; u += ustep, ++it) {
      int mt, nt;
      long long pr;
      decode(u, mt, nt, pr);
      const int buf = nbuf == 2 ? (int)(it & 1u) : 0;
      const uint32_t use = nbuf == 2 ? it >> 1 : it;
      const int m = mt * 2 * BM + row;
      const TcProb& P = probs ? probs[pr] : one;
      void* outp = P.out;
      const bool mok = m < M;
      const int n0 = nt * tile.w;
      const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * S * tile.w);
      if constexpr (sizeof(OutT) == 4) {
        constexpr int CH = (pair_max_width<S, OutT>() / 16 + 1) / 2;   // chunks of one warp
        const RowOut ro = mok ? row_out(reinterpret_cast<float*>(outp), lay, ldo, m)
                              : RowOut{nullptr, 0, 0};
        if (!pair_wait_warp(tfull(buf), use & 1u, flag, 6, wlim)) break;
        tc_fence_after();
        const int nch = ntile_w(nt) / 16;
        float v[CH * 16];
#pragma unroll
        for (int c = 0; c < CH; ++c) {
          const int chunk = 2 * c + part;
          if (chunk < nch) {
            uint32_t acc[S][16];
#pragma unroll
            for (int g = 0; g < S; ++g) tmem_ld16(tb + g * tile.w + chunk * 16, acc[g]);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              // lower classes first, then one rounding against class 0
              float lo = 0.f;
#pragma unroll
              for (int g = S - 1; g >= 1; --g)
                lo = FMT == kFmtF16 ? __fmaf_rn(lo, kW, __uint_as_float(acc[g][j]))
                                    : __fadd_rn(lo, __uint_as_float(acc[g][j]));
              v[c * 16 + j] =
                  __fmul_rn(FMT == kFmtF16 ? __fmaf_rn(lo, kW, __uint_as_float(acc[0][j]))
                                           : __fadd_rn(__uint_as_float(acc[0][j]), lo),
                            scale);
            }
          }
        }
        // TMEM is read: the leader may start the next tile in this buffer
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_cluster(map_rank(tempty(buf), 0));
        if (mok) {
#pragma unroll
          for (int c = 0; c < CH; ++c) {
            const int chunk = 2 * c + part;
            if (chunk < nch) store_chunk(ro, (n0 >> 4) + chunk, v + c * 16, N - n0 - chunk * 16);
          }
        }
      } else {
        constexpr int BITS = FMT == kFmtBF16 ? 8 : 11;
        const int es = P.ea ? *P.ea + *P.eb - 14 : escale, fl = P.flags;
        // out[n][m]: this lane's row m of column n + j in turn.  out[m][n] (ROWS): the
        // 8 x 8 blocks of 8 lanes are transposed, so that 8 lanes write 8 columns of
        // one row (64 bytes, whole sectors; one lane per row made four times the L2
        // operations, and atomics run at the rate of those: 105 products of 2809 x
        // 53 added in 385 us, now 146)
        double* const out = reinterpret_cast<double*>(outp);
        const int b8 = lane & 7, m8 = m - b8;   // first row of the lane's 8 x 8 block
        if (!pair_wait_warp(tfull(buf), use & 1u, flag, 6, wlim)) break;
        tc_fence_after();
        const int nch = ntile_w(nt) / 8;   // 8-column chunks, dealt over the four warps
#pragma unroll 1
        for (int chunk = part; chunk < nch; chunk += 4) {
          const int n = n0 + chunk * 8;
          double* const rp = out + (int64_t)m8 * ldo + n + b8;   // ROWS: this lane's column
          const bool cok = n + b8 < N;
          double old[ROWS ? 8 : 1];   // what is added to, asked for before the conversions
          if constexpr (ROWS) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              old[j] = (fl & kTcAccum) && cok && m8 + j < M ? rp[(int64_t)j * ldo] : 0.0;
          }
          uint32_t acc[S][8];
#pragma unroll
          for (int g = 0; g < S; ++g) tmem_ld8(tb + g * tile.w + chunk * 8, acc[g]);
          tmem_ld_wait();
          double v[ROWS ? 8 : 1];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float x[S], lo = 0.f;
#pragma unroll
            for (int g = S - 1; g >= 0; --g) {
              x[g] = __uint_as_float(acc[g][j]);
              lo = FMT == kFmtF16 ? __fmaf_rn(lo, kW, x[g]) : __fadd_rn(lo, x[g]);
            }
            if constexpr (ROWS) {
              v[j] = class_sum<S, BITS, FMT == kFmtF16, WIDE>(x, es, fl & kTcFloatRest);
            } else {
              if (!mok || n + j >= N) continue;
              if (amax != nullptr) lmax = fmaxf(lmax, fabsf(__fmul_rn(lo, scale)));
              if (outp != nullptr) {
                const double y = class_sum<S, BITS, FMT == kFmtF16, WIDE>(x, es, fl & kTcFloatRest);
                double* o = out + (int64_t)(n + j) * ldo + m;
                if (fl & kTcAtomic)
                  atomicAdd(o, y);
                else
                  *o = fl & kTcAccum ? *o + y : y;
              }
            }
          }
          if constexpr (ROWS) {
#pragma unroll
            for (int sft = 1; sft < 8; sft <<= 1)
#pragma unroll
              for (int j = 0; j < 8; ++j)
                if (!(j & sft)) {
                  const bool up = b8 & sft;
                  const double y = __shfl_xor_sync(0xffffffffu, up ? v[j] : v[j | sft], sft);
                  if (up)
                    v[j] = y;
                  else
                    v[j | sft] = y;
                }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if (!cok || m8 + j >= M) continue;
              double* o = rp + (int64_t)j * ldo;
              if (fl & kTcAtomic)
                atomicAdd(o, v[j]);
              else
                *o = fl & kTcAccum ? old[j] + v[j] : v[j];
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_cluster(map_rank(tempty(buf), 0));
      }
    }
    if (sizeof(OutT) == 8 && amax != nullptr) {
      for (int off = 16; off > 0; off >>= 1)
        lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, off));
      if (lane == 0) atomicMax(amax, (unsigned long long)__double_as_longlong((double)lmax));
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();   // no CTA leaves while its peer may still reach its memory
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// Pairs that fit the device at once (queried once; the persistent loop deals
// its tiles over them, so none may wait for a slot).
template <int S, int FMT, typename OutT, bool ROWS, bool WIDE>
int pair_clusters(int nsm) {
  static const int n = [] {
    auto k = tc_pair_gemm<S, FMT, OutT, ROWS, WIDE>;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(pair_threads<OutT>());
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int c = 0;
    if (cudaOccupancyMaxActiveClusters(&c, k, &cfg) != cudaSuccess) {
      cudaGetLastError();
      c = 0;
    }
    return c;
  }();
  return std::max(1, n > 0 ? std::min(n, nsm / 2) : nsm / 2);
}

template <int S, int FMT, typename OutT, bool ROWS = false, bool WIDE = false>
cudaError_t launch_pair(const CUtensorMap* mA, const CUtensorMap* mB, const TcProb* probs,
                        const TcProb& one, int nprob, int M, int N, int ldo, double scale,
                        int* flag, unsigned long long* amax, int nsm, cudaStream_t st,
                        TcDiag diag, TcOut lay, PairTile tile) {
  if (nprob <= 0 || M <= 0 || N <= 0) return cudaSuccess;
  if (tile.w < 16 || tile.w % 16 || tile.w > pair_max_width<S, OutT>() || tile.stages < 2 ||
      tile.stages > kMaxStages || (tile.nbuf == 2 && 2 * S * tile.w > 512) ||
      (int64_t)tile.nN * tile.w < N || (int64_t)(tile.nN - 1) * tile.w >= N)
    return cudaErrorInvalidValue;
  if (sizeof(OutT) == 8 && tile.nbuf != 2) return cudaErrorInvalidValue;
  int ex;
  if (std::frexp(scale, &ex) != 0.5) return cudaErrorInvalidValue;   // scale = 2^(ex - 1)
  auto k = tc_pair_gemm<S, FMT, OutT, ROWS, WIDE>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e != cudaSuccess) return e;
  const long long units = (long long)nprob * ((M + 2 * BM - 1) / (2 * BM)) * tile.nN;
  const int pairs = (int)std::min<long long>(units, pair_clusters<S, FMT, OutT, ROWS, WIDE>(nsm));
  k<<<2 * pairs, pair_threads<OutT>(), kSmemBytes, st>>>(mA[0], mA[1], mB[0], mB[1], probs, one,
                                                         nprob, M, N, ldo, (float)scale, ex - 1,
                                                         flag, amax, diag, lay, tile);
  return cudaGetLastError();
}

}  // namespace

// Tile of a pair launch with N columns: the fewest n-tiles the widest tile
// allows (cap > 0: no wider than cap), equal up to 16 columns; two accumulator
// sets where they fit; as many stages as shared memory holds.
PairTile pair_tile(int S, int N, int cap) {
  const int wmax = std::min(256, 512 / S / 16 * 16);
  const int lim = cap > 0 ? std::max(16, std::min(wmax, cap / 16 * 16)) : wmax;
  PairTile t;
  const int n16 = (N + 15) / 16;
  t.nN = std::max(1, (n16 + lim / 16 - 1) / (lim / 16));
  t.w = std::max(1, (n16 + t.nN - 1) / t.nN) * 16;
  t.nN = std::max(1, (n16 * 16 + t.w - 1) / t.w);
  t.nbuf = 2 * S * t.w <= 512 ? 2 : 1;
  t.stages = std::min(kMaxStages, (kSmemBytes - kBarBytes - 1024) / (S * (BM * 64 + t.w * 32)));
  return t;
}

// Tile of a float64-output launch: 64 columns at most, fewer (32, 16) while the
// launch has fewer tiles than the device has pairs.
PairTile pair_tile_f64(int S, int nprob, int M, int N) {
  const int wide = std::min(kF64Width, 256 / S / 16 * 16);
  int cap = wide;
  const long long mt = (long long)nprob * ((M + 2 * BM - 1) / (2 * BM));
  while (cap > 16 && mt * ((N + cap - 1) / cap) < 76) cap = cap > 32 ? 32 : 16;
  return pair_tile(S, N, cap);
}

// mA: maps with boxes of 128 rows x S slices, mB: of tile.w / 2 rows x S slices.
template <int S, int FMT>
cudaError_t launch_tc_pair(const CUtensorMap* mA, const CUtensorMap* mB, const TcProb* probs_dev,
                           int nprob, int M, int N, int ldo, double scale, int* flag, int nsm,
                           cudaStream_t st, TcDiag diag, TcOut lay, PairTile tile) {
  if (lay.mode == kOutRows ? (ldo % 4 != 0 || ldo < ((N + 15) & ~15))
                           : (lay.nbs < 1 || lay.nbt < 1 || (lay.mode == kOutYTile && lay.nvt < 1)))
    return cudaErrorInvalidValue;
  if (probs_dev == nullptr) return cudaErrorInvalidValue;
  return launch_pair<S, FMT, float>(mA, mB, probs_dev, TcProb{}, nprob, M, N, ldo, scale, flag,
                                    nullptr, nsm, st, diag, lay, tile);
}

// One product with float64 output: p.out[n][m] (pitch ldo) = scale 2^14 units of
// the class sums of segment p.seg[0], and / or its largest magnitude in *amax
// (p.out NULL: only that).  Tile from pair_tile_f64.
template <int S, int FMT>
cudaError_t launch_tc_pair_f64(const CUtensorMap* mA, const CUtensorMap* mB, const TcProb& p,
                               int M, int N, int ldo, double scale, int* flag,
                               unsigned long long* amax, int nsm, cudaStream_t st, PairTile tile) {
  auto launch = launch_pair<S, FMT, double>;
  if constexpr (S > 2)   // two slices: the measuring pass only
    if (p.seg[0].K > (FMT == kFmtF16 ? kWideFP16 : kWideBF16))
      launch = launch_pair<S, FMT, double, false, true>;
  return launch(mA, mB, nullptr, p, 1, M, N, ldo, scale, flag, amax, nsm, st, tc_normal(),
                TcOut{kOutRows, 0, 0, 0}, tile);
}

// A group of such products, each with its own flags and, where TcProb.ea and eb
// are given, its own scale; K at most kWideBF16.
template <int S, int FMT>
cudaError_t launch_tc_pair_f64_group(const CUtensorMap* mA, const CUtensorMap* mB,
                                     const TcProb* probs_dev, int nprob, int M, int N, int ldo,
                                     double scale, int* flag, int nsm, cudaStream_t st,
                                     int mode, PairTile tile, TcDiag diag) {
  if (nprob > 0 && probs_dev == nullptr) return cudaErrorInvalidValue;
  auto launch = mode == kOutF64Rows ? launch_pair<S, FMT, double, true>
                                    : launch_pair<S, FMT, double, false>;
  return launch(mA, mB, probs_dev, TcProb{}, nprob, M, N, ldo, scale, flag, nullptr, nsm, st,
                diag, TcOut{mode, 0, 0, 0}, tile);
}
template cudaError_t launch_tc_pair_f64_group<4, kFmtBF16>(const CUtensorMap*, const CUtensorMap*,
                                                           const TcProb*, int, int, int, int,
                                                           double, int*, int, cudaStream_t, int,
                                                           PairTile, TcDiag);

#define LNO_PAIR_INST(S, F)                                                                   \
  template cudaError_t launch_tc_pair<S, F>(const CUtensorMap*, const CUtensorMap*,            \
                                            const TcProb*, int, int, int, int, double, int*,  \
                                            int, cudaStream_t, TcDiag, TcOut, PairTile);
LNO_PAIR_INST(2, kFmtBF16)
LNO_PAIR_INST(3, kFmtBF16)
LNO_PAIR_INST(4, kFmtBF16)
LNO_PAIR_INST(5, kFmtBF16)
LNO_PAIR_INST(2, kFmtTF32)
LNO_PAIR_INST(3, kFmtF16)
#undef LNO_PAIR_INST
#define LNO_PAIR_F64(S, F)                                                                      \
  template cudaError_t launch_tc_pair_f64<S, F>(const CUtensorMap*, const CUtensorMap*,          \
                                                const TcProb&, int, int, int, double, int*,     \
                                                unsigned long long*, int, cudaStream_t, PairTile);
LNO_PAIR_F64(2, kFmtBF16)
LNO_PAIR_F64(4, kFmtBF16)
LNO_PAIR_F64(5, kFmtBF16)
LNO_PAIR_F64(2, kFmtF16)
LNO_PAIR_F64(3, kFmtF16)
#undef LNO_PAIR_F64

}  // namespace lno
