// The library's own dense contractions: the n^3 squarings and sums of the
// re-evaluation strategy (Section 4.2.2, "Re-evaluation"; Table 1), the
// products of the reverse pass (the adjoint chain through the squarings, the
// G_i = A^T G_{i+1} products and dA = [G_1 .. G_k][T_0 .. T_{k-1}]^T), the
// iteration's n x n x p products (T_i = A T_{i-1} + B, the hybrid strategy's
// D_i = A D_{i-1}) and the small factor products of the general form.
//
//  * tc_gemm_kernel<BN> (FP32): D = A B^T (+ beta C) on tcgen05 from operands
//    split into two 11-bit halves, x = hi + lo, and three products,
//    A B^T ~= lo(A) hi(B)^T + hi(A) lo(B)^T + hi(A) hi(B)^T (the dropped lo lo^T
//    term is ~2^-22 relative): near-FP32 accuracy, where one TF32 product alone
//    gives ~5e-4.  The halves are FP16 by default (tcgen05 kind::f16, twice the
//    rate and half the bytes of TF32): each run of 64 values of an operand row is
//    scaled by a power of two that takes its largest entry to [2^14, 2^15), so
//    that every entry down to 2^-17 of the run's largest keeps the 22 bits of a
//    TF32 pair and a smaller one is off by at most 2^-40 of the largest; a run is
//    one K chunk of the MMAs, whose result the epilogue scales back exactly as it
//    adds it up.  Operands for which that is not enough (entries that lose bits
//    beside runs of mostly small or zero entries, see needs_tf32), whose scale is out of
//    the exponent's comfortable range, or that hold infinities or NaN are found
//    while they are split, and such a product runs on TF32 halves instead (same
//    kernel, kind::tf32; hi = x rounded to nearest
//    TF32, lo = x - hi rounded in turn).  Operands are stored in blocks of 128 rows x
//    one K chunk, [hi | lo] of 16 KB each, rows of 128 bytes (the split also transposes
//    where the product needs the other layout): a chunk of a CTA's A is one copy of
//    32 contiguous KB (as rows [hi | lo] of length K every box line was 128 bytes 32 KB
//    apart, and 8192 x 64 x 8192, which streams A from memory, took 57 us, 53 now).
//    CTA pairs (cta_group::2) compute tiles of 256 x BN outputs (BN = 256, 128 or
//    64), each CTA holding 128 rows of A and half of B's rows, in K chunks of
//    one 128-byte swizzle atom (64 FP16 or 32 TF32 values); a persistent grid
//    walks the tiles in groups of 8 row blocks (the A and B chunks a wave reads
//    stay in L2).  Per CTA: warp 0 streams its A and B chunks with TMA into an
//    S-stage ring, one thread of the pair's first CTA issues 12 MMAs per chunk
//    (3 products x 4 K steps of 32 bytes) into one of 512 / BN BN-column FP32
//    accumulators in tensor memory, and the epilogue warps read the ones before
//    it back (tcgen05.ld).  The tensor
//    cores accumulate with round-toward-zero, a bias that grows with the number
//    of accumulation steps (measured 7.9e-6 relative at K = 1000, ~6e-5 at
//    K = 8192 if the whole K were accumulated in tensor memory), so the MMAs
//    accumulate only one chunk into a fresh accumulator
//    (its two small correction products first, while the accumulator
//    is small), and the epilogue warps add each chunk's result into FP32
//    registers (round to nearest), 128 columns per thread (8 epilogue warps
//    for 256-column tiles, 4 otherwise); after the tile's last chunk they
//    scale back, add beta C and store D.  Single CTAs on 128 x 256 tiles would
//    read 96 bytes of shared memory per clock for the FP16 products and twice
//    the operand bytes from L2; the pair halves B's share of both.
//    Every wait is bounded; an expired wait latches LINVIEW_ETIMEOUT and the
//    pair drains its copies and MMAs and frees its tensor memory.
//  * gemm_simt_kernel<T>: C = alpha op(A) op(B) + beta C with arbitrary
//    strides on the CUDA cores (64 x 64 tiles, 4 x 4 outputs per thread), with
//    a deterministic split of long inner dimensions (partials summed in a
//    fixed order by a second kernel): the FP64 programs' products (GB300 has
//    no fast FP64 tensor path) and the small FP32 factor products.
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "lv_device.cuh"
#include "lv_internal.h"

namespace lv {

namespace {

constexpr int kGBM = 256;       // tile rows (MMA M, 128 per CTA of the pair)
constexpr int kGroupM = 8;      // row blocks per raster group

template <int BN>
struct GShape {
  static constexpr uint32_t AHalf = 128 * 128;            // one half (hi or lo) of a CTA's A chunk
  static constexpr uint32_t BHalf = BN / 2 * 128;         // ... of its B chunk
  static constexpr uint32_t StageBytes = 2 * AHalf + 2 * BHalf;  // 64, 48, 40 KB
  static constexpr int S = BN == 256 ? 3 : (BN == 128 ? 4 : 5);
  static constexpr uint32_t OffBar = S * StageBytes;
  static constexpr int NB = 512 / BN;                         // accumulators (all of tensor memory)
  static constexpr uint32_t TmemCols = 512;
  static constexpr int CW = BN < 128 ? BN : 128;              // columns per epilogue thread
  static constexpr int NE = 4 * (BN / CW);                    // epilogue warps
  // 4 KB per epilogue warp: the CW column factors of a chunk; after a tile's last
  // chunk 32 rows x 32 columns on their way to D
  static constexpr uint32_t OffStage = OffBar + 512;
  static constexpr uint32_t SmemBytes = OffStage + NE * 4096 + 1024;  // + alignment slack
  // warps 0-3: copies, MMAs, two idle; then the epilogue
  static constexpr int Threads = 128 + 32 * NE;
  // With eight epilogue warps (BN = 256) a thread has 168 registers, too few for
  // 128 sums and the 64 accumulator columns in flight: the first four warps hand
  // theirs over (40 x 128 + 224 x 256 <= 168 x 384).
  static constexpr bool Rebalance = NE == 8;
  // instruction descriptor: D F32, A and B K-major, N = BN, M = 256; the operand
  // type fields are 0 (F16) or 2 (TF32)
  static constexpr uint32_t Idesc16 =
      (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(kGBM >> 4) << 24);
  static constexpr uint32_t Idesc32 = Idesc16 | (2u << 7) | (2u << 10);
};
static_assert(GShape<256>::SmemBytes <= 232448 && GShape<128>::SmemBytes <= 232448 &&
                  GShape<64>::SmemBytes <= 232448,
              "shared memory per CTA");

struct GBars {
  uint64_t full[5], empty[5];
  uint64_t acc_full[8], acc_empty[8];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(GBars) <= 512, "barrier block");

// shared-memory descriptor of a K-major operand in 128-byte swizzled rows,
// 8-row groups 1024 bytes apart (the layout TMA writes with SWIZZLE_128B)
__device__ __forceinline__ uint64_t g_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);  // start address
  d |= (uint64_t)1u << 16;                   // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024u >> 4) << 32;         // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1u << 46;                   // descriptor version
  d |= (uint64_t)2u << 61;                   // 128-byte swizzle
  return d;
}

template <bool F16>
__device__ __forceinline__ void g_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                      uint32_t accumulate) {
  if constexpr (F16)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

// arrive on ``bar`` of both CTAs of the pair once every MMA issued so far is done
__device__ __forceinline__ void g_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 "
      "[%0], %1;" ::"r"(smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}

__device__ __forceinline__ void g_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void g_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// cluster-window address of a barrier of the pair's first CTA
__device__ __forceinline__ uint32_t lead_bar(uint64_t* bar) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(smem_u32(bar)));
  return a;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// TMA box into this CTA's shared memory, completing bytes on a barrier of the pair
__device__ __forceinline__ void g_tma(void* dst, const void* tmap, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void g_arrive_lead(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar)
               : "memory");
}

// 32 columns of this warp's 32 lanes (complete after g_tmem_wait_ld)
__device__ __forceinline__ void g_tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}

__device__ __forceinline__ void g_tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ bool g_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                       unsigned* status) {
  if (mbar_try_wait(bar, parity)) return true;
  if (*abort_flag) return false;
  if (mbar_wait_bounded(bar, parity, status)) return true;
  *abort_flag = 1;
  return false;
}
// tile t of the raster: groups of kGroupM row blocks, column blocks within
__device__ __forceinline__ void g_tile(long long t, int mt, int nt, int& mb, int& nb) {
  const long long per_group = (long long)kGroupM * nt;
  const int group = (int)(t / per_group);
  const int first = group * kGroupM;
  const int gm = (mt - first < kGroupM) ? (mt - first) : kGroupM;
  const int rem = (int)(t - (long long)group * per_group);
  mb = first + rem % gm;
  nb = rem / gm;
}

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }  // |e| <= 126

// Work of one CTA pair: whole tiles pair, pair + npairs, .. < dp, then its range of
// the chunk sequence of the tiles left over, which would leave most pairs idle as
// whole tiles (their last wave).  A tile's pieces are numbered range + cut tile
// (both grow along the sequence, so the numbers are distinct) and go to that
// slot of the work buffer, unless one range covers the tile.
struct GWork {
  long long t, pos, end;
  int npairs, dp, nk, pair;
  int tile, kb, ke, slot;  // current piece; slot < 0: a whole tile
  bool rev;                // the pair's range of the cut tiles from its end
  __device__ GWork(int pair_, int npairs_, int dp_, int cut, int tiles, int nk_, bool rev_)
      : t(pair_), pos(0), end(0), npairs(npairs_), dp(dp_), nk(nk_), pair(pair_), rev(rev_) {
    if (pair < cut) {
      const long long W = (long long)(tiles - dp) * nk;
      pos = W * pair / cut;
      end = W * (pair + 1) / cut;
    }
  }
  __device__ bool next() {
    if (t < dp) {
      tile = (int)t;
      kb = 0;
      ke = nk;
      slot = -1;
      t += npairs;
      return true;
    }
    if (pos >= end) return false;
    const int r = (int)((rev ? end - 1 : pos) / nk);
    const long long first = (long long)r * nk;
    tile = dp + r;
    kb = (int)(pos > first ? pos - first : 0);
    ke = (int)(end - first < nk ? end - first : nk);
    slot = kb == 0 && ke == nk ? -1 : pair + r;
    if (rev)
      end = first + kb;
    else
      pos = first + ke;
    return true;
  }
};

struct GMaps {
  CUtensorMap a16, b16, a32, b32;
};
struct GArgs {
  int M, N, kp16, kp32;
  float* D;
  int64_t ldd;
  const float* C;
  int64_t ldc;
  float alpha, beta;
  int vec_ok;
  int reverse;    // visit a pair's K chunks last to first
  int dp;         // tiles computed whole; the others are cut into ``cut`` equal ranges
  int cut;        // of K chunks, one per CTA pair
  float* work;    // [range + cut tile][256][BN] partial sums of the tiles cut
  const float* sa;      // factors of A's and B's runs of 64: [chunk][row], strides pa, pb
  const float* sb;
  int64_t pa, pb;
  unsigned* fmta;       // format of each split buffer, written here for later products
  unsigned* fmtb;
  const unsigned* flag;
  unsigned* status;
};

// The flag word of a product: three bits per operand, A's from bit 0, B's from bit 4.  kLossy:
// entries that keep fewer than 22 bits.  kSparse, kSparser: runs of which more than 3/8 lie
// below 512 and below 7, where the largest is 2^14 to 2^15 (below 256 and 8 in runs of fewer
// than 48), zeros among them, runs of zeros aside.  Entries that lose bits do no harm where
// dense runs meet: where no run of one operand is kSparse and none of the other kSparser, a
// quarter of a run of length L meets with products of 3584 and more, a sum of |a||b| of at
// least L/4 3584, while the at most 2 + 8 entries that lose bits add 2^-25 2^15 each: 2^-22.5
// of the sum at L = 64 (2^-20 in a last run of 16, with at most 4 + 4), about what the halves of
// the other entries leave.  Else such an entry may meet zeros and small entries only, and a
// product is as good as that entry.  (Runs with more of them, zeros counted where there is one,
// are kSparser.)  Dense data has entries that lose bits (2e-5 of normal ones) and no sparse
// runs; a matrix with a diagonal or a few rows some hundred times the rest is kSparse along one
// of its sides and not kSparser.
constexpr unsigned kLossy = 1u, kSparse = 2u, kSparser = 4u, kFlagAll = 7u;
__device__ __forceinline__ bool needs_tf32(unsigned flag) {
  const unsigned a = flag & kFlagAll, b = flag >> 4;
  return ((a | b) & kLossy) && ((a & b & kSparse) || ((a | b) & kSparser));
}

// D (M x N, row-major, ldd) = alpha A B^T + beta C over the split blocks of K = kp16
// (FP16) or kp32 (TF32) values.
// HALVES: every other chunk (FP16) goes to two accumulators.
template <int BN, bool HALVES>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GShape<BN>::Threads, 1)
    tc_gemm_kernel(const __grid_constant__ GMaps maps, const GArgs a) {
  using Sh = GShape<BN>;
  constexpr int S = Sh::S, CW = Sh::CW, NE = Sh::NE, NB = Sh::NB;
  extern __shared__ __align__(1024) unsigned char g_smem_raw[];
  const uint32_t raw = smem_u32(g_smem_raw);
  unsigned char* base = g_smem_raw + (((raw + 1023u) & ~1023u) - raw);
  GBars* bars = reinterpret_cast<GBars*>(base + Sh::OffBar);
  volatile int* abort_flag = &bars->abort;
  unsigned* status = a.status;
  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  const uint32_t rank = cta_rank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;

  if (tid == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(&bars->full[i], 1);
      mbar_init(&bars->empty[i], 1);
    }
    for (int i = 0; i < NB; ++i) {
      mbar_init(&bars->acc_full[i], 1);
      mbar_init(&bars->acc_empty[i], 2 * NE);  // one arrival per epilogue warp of the pair
    }
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&bars->tmem_base)),
                 "r"(Sh::TmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  g_fence_before();
  __syncthreads();
  cluster_sync();
  g_fence_after();
  const uint32_t tmem = bars->tmem_base;
  griddep_wait();  // the splits
  griddep_launch_dependents();
  const bool f16 = !needs_tf32(*a.flag);
  const int kc_len = f16 ? 64 : 32;
  const int kp = f16 ? a.kp16 : a.kp32;
  const int nk = kp / kc_len;
  const int mt = (a.M + kGBM - 1) / kGBM;
  const int nt = (a.N + BN - 1) / BN;
  GWork work(pair, npairs, a.dp, a.cut, mt * nt, nk, a.reverse != 0);
  // Reversed, a pair walks its own range backwards, so it starts on the blocks of A it read
  // last in the product before.  Mirrored over the whole of K it met blocks that another
  // pair had read at another time: adjoint of 16 rounds at 8192 x 64 1313 -> 1238 us, at
  // 5000 x 30 582 -> 535, 8 rounds at 7000 x 120 733 -> 715.
  auto chunk = [&](int kc) { return a.reverse ? work.kb + work.ke - 1 - kc : kc; };
  // accumulators that chunk kc takes
  auto halves = [&](int kc) { return HALVES && f16 && !((kc - work.kb) & 1) ? 2 : 1; };
  if (blockIdx.x == 0 && tid == 0) {  // the buffers' format, for later products on the same split
    *a.fmta = f16 ? 0u : 1u;
    *a.fmtb = f16 ? 0u : 1u;
  }

  if (warp < 4) {
    if constexpr (Sh::Rebalance) asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 0 && lane == 0) {
      // ---------------- producer (each CTA its own half) ----------------
      const CUtensorMap* ma = f16 ? &maps.a16 : &maps.a32;
      const CUtensorMap* mb_ = f16 ? &maps.b16 : &maps.b32;
      prefetch_tmap(ma);
      prefetch_tmap(mb_);
      const uint32_t lead_full = lead_bar(&bars->full[0]);
      int st = 0;
      uint32_t phase = 0;      // of the ring's current round
      long long loaded = 0;    // chunks requested
      while (!*abort_flag && work.next()) {
        int mb, nb;
        g_tile(work.tile, mt, nt, mb, nb);
        // 256 lines of 128 bytes per block: hi of 128 rows, then lo
        const int aline = (mb * 2 + (int)rank) * nk * 256;
        const int brow = nb * BN + (int)rank * (BN / 2);
        const int bline = (brow >> 7) * nk * 256 + (brow & 127);
        for (int kc = work.kb; kc < work.ke; ++kc, ++loaded) {
          if (loaded >= S && !g_wait(&bars->empty[st], phase ^ 1u, abort_flag, status)) break;
          const int line = chunk(kc) * 256;
          unsigned char* sb = base + st * Sh::StageBytes;
          // the first CTA's barrier counts both CTAs' bytes
          const uint32_t fb = lead_full + st * 8;
          if (rank == 0) mbar_arrive_expect_tx(&bars->full[st], 2 * Sh::StageBytes);
          g_tma(sb, ma, 0, aline + line, fb);
          g_tma(sb + 2 * Sh::AHalf, mb_, 0, bline + line, fb);
          if (BN < 256) g_tma(sb + 2 * Sh::AHalf + Sh::BHalf, mb_, 0, bline + line + 128, fb);
          if (++st == S) {
            st = 0;
            phase ^= 1u;
          }
        }
      }
      if (*abort_flag && rank == 0) {
        // the stages loaded last may still be in flight: wait (bounded) for them
        const long long first = loaded > S ? loaded - S : 0;
        for (long long j = first; j < loaded; ++j)
          mbar_wait_bounded(&bars->full[j % S], (uint32_t)((j / S) & 1), nullptr);
      }
    }
    if (warp == 1 && rank == 0) {
      // ---------------- MMA issuer (first CTA of the pair) ----------------
      // The whole warp walks the chunks and one elected lane issues, so that the
      // descriptors and counters are warp-uniform: with the loop inside a
      // lane-0 branch every MMA took about 35 ns to issue and a chunk at least
      // 0.70 us whatever its width (4096^3 in 64-column tiles 626 us, now 449).
      int st = 0, buf = 0;
      uint32_t phase = 0, aphase = 0;
      bool first_round = true;  // the accumulators have not been used yet
      const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
      const uint64_t d0 = g_desc(smem_u32(base));
      bool ok = true;
      while (ok && !*abort_flag && work.next()) {
        for (int kc = work.kb; kc < work.ke && ok; ++kc) {
          const uint64_t a_hi = d0 + (uint32_t)st * (Sh::StageBytes >> 4);
          const uint64_t a_lo = a_hi + (Sh::AHalf >> 4);
          const uint64_t b_hi = a_hi + (2 * Sh::AHalf >> 4);
          const uint64_t b_lo = b_hi + (Sh::BHalf >> 4);
          // lo(A) hi(B), hi(A) lo(B), then hi(A) hi(B)
          const uint64_t pa[3] = {a_lo, a_hi, a_hi};
          const uint64_t pb[3] = {b_hi, b_lo, b_hi};
          ok = g_wait(&bars->full[st], phase, abort_flag, status);
          const int nh = halves(kc);
          for (int h = 0; h < nh; ++h) {
            if (ok && !first_round) ok = g_wait(&bars->acc_empty[buf], aphase ^ 1u, abort_flag, status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            g_fence_after();
            if (elect_one()) {
              const uint32_t d = tm + buf * BN;
              auto issue = [&](auto kind, auto k0, auto k1) {  // K steps of 32 bytes of a row
                constexpr bool F16 = decltype(kind)::value;
#pragma unroll
                for (int pr = 0; pr < 3; ++pr)
#pragma unroll
                  for (int kk = k0.value; kk < k1.value; ++kk)
                    g_mma<F16>(d, pa[pr] + kk * 2, pb[pr] + kk * 2, F16 ? Sh::Idesc16 : Sh::Idesc32,
                               (pr != 0 || kk != k0.value) ? 1u : 0u);
              };
              const std::integral_constant<int, 0> k0;
              const std::integral_constant<int, 2> k2;
              const std::integral_constant<int, 4> k4;
              if (!f16)
                issue(std::false_type{}, k0, k4);
              else if (nh == 1)
                issue(std::true_type{}, k0, k4);
              else if (h == 0)
                issue(std::true_type{}, k0, k2);
              else
                issue(std::true_type{}, k2, k4);
              if (h == nh - 1) g_commit(&bars->empty[st]);
              g_commit(&bars->acc_full[buf]);
            }
            __syncwarp();
            if (++buf == NB) {
              buf = 0;
              aphase ^= 1u;
              first_round = false;
            }
          }
          if (++st == S) {
            st = 0;
            phase ^= 1u;
          }
        }
      }
      // every MMA issued has completed before the tensor memory is freed
      if (elect_one()) g_commit(&bars->drain);
      __syncwarp();
    }
    // both CTAs: the MMAs' arrivals have reached this CTA's barriers
    if (warp == 1 && lane == 0) mbar_wait_bounded(&bars->drain, 0, status);
  } else {
    // ---------------- epilogue (warps 4 .. 4 + NE - 1) ----------------
    if constexpr (Sh::Rebalance) asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    const int ew = warp - 4;
    const int quarter = warp & 3;     // tensor-memory lanes 32*quarter .. +31
    const int cpart = ew >> 2;        // column part: columns cpart*CW .. +CW-1
    const int row = quarter * 32 + lane;
    float* cs = reinterpret_cast<float*>(base + Sh::OffStage + ew * 4096);
    const uint32_t ae = lead_bar(&bars->acc_empty[0]);
    int buf = 0;
    uint32_t aphase = 0;
    bool ok = true;
    while (ok && work.next()) {
      int mb, nb;
      g_tile(work.tile, mt, nt, mb, nb);
      const int grow = mb * kGBM + (int)rank * 128 + row;
      const int gc0 = nb * BN + cpart * CW;
      // the chunk's factors, loaded one chunk ahead: this thread's row, and four
      // columns a lane to be shared with the warp
      const bool has_row = f16 && grow < a.M, has_col = f16 && 4 * lane < CW && gc0 + 4 * lane < a.pb;
      const float* sa = a.sa + grow;
      const float* sb = a.sb + gc0 + 4 * lane;
      auto row_factor = [&](int kc) { return has_row ? __ldg(sa + chunk(kc) * a.pa) : 1.f; };
      auto col_factors = [&](int kc) {
        return has_col ? __ldg(reinterpret_cast<const float4*>(sb + chunk(kc) * a.pb))
                       : make_float4(1.f, 1.f, 1.f, 1.f);
      };
      float fr_next = row_factor(work.kb);
      float4 fc_next = col_factors(work.kb);
      float2 acc[CW / 2];
#pragma unroll
      for (int c = 0; c < CW / 2; ++c) acc[c] = make_float2(0.f, 0.f);
      for (int kc = work.kb; kc < work.ke; ++kc) {
        const float2 fr2 = make_float2(fr_next, fr_next);
        __syncwarp();
        if (4 * lane < CW) reinterpret_cast<float4*>(cs)[lane] = fc_next;
        if (kc + 1 < work.ke) {
          fr_next = row_factor(kc + 1);
          fc_next = col_factors(kc + 1);
        }
        const int nh = halves(kc);
#pragma unroll 1
        for (int h = 0; h < nh; ++h) {
          const bool w = g_wait(&bars->acc_full[buf], aphase, abort_flag, status);
          if (!__all_sync(0xffffffffu, w)) {  // tcgen05.ld is warp-collective
            ok = false;
            break;
          }
          g_fence_after();
          const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + buf * BN + cpart * CW;
#pragma unroll
          for (int q = 0; q < CW / 64; ++q) {  // 64 columns in flight
            uint32_t v[2][32];
            g_tmem_ld32(ta + q * 64, v[0]);
            g_tmem_ld32(ta + q * 64 + 32, v[1]);
            g_tmem_wait_ld();
            if (q == CW / 64 - 1) {  // all read: the accumulator is free
              g_fence_before();
              __syncwarp();
              if (lane == 0) g_arrive_lead(ae + buf * 8);
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              // the factors are powers of two: one rounding, in the addition
              const float4 f = reinterpret_cast<const float4*>(cs)[q * 16 + e];
              const uint32_t* x = &v[e / 8][e % 8 * 4];
              float2& a0 = acc[q * 32 + 2 * e];
              float2& a1 = acc[q * 32 + 2 * e + 1];
              a0 = __ffma2_rn(__fmul2_rn(make_float2(__uint_as_float(x[0]), __uint_as_float(x[1])),
                                         make_float2(f.x, f.y)), fr2, a0);
              a1 = __ffma2_rn(__fmul2_rn(make_float2(__uint_as_float(x[2]), __uint_as_float(x[3])),
                                         make_float2(f.z, f.w)), fr2, a1);
            }
          }
          if (++buf == NB) {
            buf = 0;
            aphase ^= 1u;
          }
        }
        if (!ok) break;
      }
      if (!ok) break;
      // A thread holds a row, memory wants lines: blocks of 32 x 32 go through shared
      // memory (16-byte unit u of row r at u ^ (r & 7)), so that a store writes four
      // whole lines, not 16 bytes of 32 (or, for D whose rows are not on 16-byte units,
      // 4): 8192 x 8192 x 1024 313 -> 264 us.
      if (gc0 < a.N) {
        float4* stg = reinterpret_cast<float4*>(cs);
        const int wrow0 = (int)rank * 128 + quarter * 32;
        const int r0 = mb * kGBM + wrow0;
        const bool add_c = a.C && a.beta != 0.f;
#pragma unroll
        for (int q = 0; q < CW / 32; ++q) {
          __syncwarp();
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const float2 x = acc[q * 16 + 2 * u], y = acc[q * 16 + 2 * u + 1];
            stg[lane * 8 + (u ^ (lane & 7))] = make_float4(x.x, x.y, y.x, y.y);
          }
          __syncwarp();
          const int col = gc0 + q * 32;
          if (work.slot >= 0 || (a.vec_ok && col + 32 <= a.N)) {
#pragma unroll 2
            for (int it = 0; it < 8; ++it) {
              const int r = it * 4 + (lane >> 3);
              float4 o = stg[r * 8 + ((lane & 7) ^ (r & 7))];
              if (r0 + r >= a.M) continue;
              if (work.slot >= 0) {  // a piece of a tile, to be summed by gemm_parts_kernel
                *reinterpret_cast<float4*>(
                    a.work + ((int64_t)work.slot * kGBM + wrow0 + r) * BN + cpart * CW + q * 32 +
                    4 * (lane & 7)) = o;
                continue;
              }
              o.x *= a.alpha;
              o.y *= a.alpha;
              o.z *= a.alpha;
              o.w *= a.alpha;
              if (add_c) {
                const float4 c = *reinterpret_cast<const float4*>(
                    a.C + (int64_t)(r0 + r) * a.ldc + col + 4 * (lane & 7));
                o.x += a.beta * c.x;
                o.y += a.beta * c.y;
                o.z += a.beta * c.z;
                o.w += a.beta * c.w;
              }
              *reinterpret_cast<float4*>(a.D + (int64_t)(r0 + r) * a.ldd + col + 4 * (lane & 7)) = o;
            }
          } else {
#pragma unroll 4
            for (int r = 0; r < 32; ++r) {
              if (r0 + r >= a.M || col + lane >= a.N) continue;
              float o = a.alpha * reinterpret_cast<const float*>(
                                      stg)[r * 32 + (((lane >> 2) ^ (r & 7)) << 2) + (lane & 3)];
              if (add_c) o += a.beta * a.C[(int64_t)(r0 + r) * a.ldc + col + lane];
              a.D[(int64_t)(r0 + r) * a.ldd + col + lane] = o;
            }
          }
        }
      }
      __syncwarp();
    }
  }
  g_fence_before();
  __syncthreads();
  cluster_sync();  // neither CTA leaves while the other's MMAs or copies use its memory
  if (warp == 1) {
    g_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(Sh::TmemCols)
                 : "memory");
  }
}

// ---------------------------------------------------------------- operand split
// Element (i, k) of op(X) is X[i * rs + k * cs] with rs or cs == 1.
struct SplitOp {
  const float* X;
  int64_t rs, cs;
  int rows, K;
  unsigned char* dst;
  float* sc;        // factors of the runs of 64, [run][row] with stride ``pitch``
  int64_t pitch;
  unsigned* fmt;    // 0: FP16 rows, 1: TF32 rows
  int vec;          // rows of X start on 16-byte units
  int blocks;       // CTAs of this operand in the launch at hand
  int bit;          // first of this operand's bits in the flag word: 0 (A) or 4 (B)
};
struct SplitPair {
  SplitOp o[2];
  unsigned* flag;
};

// line (of 128 bytes) of row i in the block of chunk kc of nk: its hi half; lo lies 128
// lines on
__device__ __forceinline__ int64_t block_line(int i, int kc, int nk) {
  return ((int64_t)(i >> 7) * nk + kc) * 256 + (i & 127);
}

// FP16 rows put K's values in slots 0 .. kp - 1 (kp = rup(K, 64)), zeros in the rest.  A last
// run of 1 to 15 values is too short to say whether it is sparse, so the 16 values before it
// move over to it: the run before ends in 16 zeros.
__host__ __device__ __forceinline__ int slot_gap(int K) {
  return K > 64 && K % 64 >= 1 && K % 64 < 16 ? 16 : 0;
}
// first slot behind the moved ones, kp for none
__device__ __forceinline__ int slot_last(int K) {
  return slot_gap(K) ? K / 64 * 64 : (K + 63) / 64 * 64;
}
// value of a slot that is a multiple of 8 (and of the seven behind it); K or more: zeros
__device__ __forceinline__ int slot_value(int slot, int K) {
  const int last = slot_last(K);
  return slot >= last ? slot - slot_gap(K) : (slot_gap(K) && slot >= last - 16 ? K : slot);
}
// values of the run of 64 slots at ``slot``
__device__ __forceinline__ int run_length(int slot, int K) {
  const int run = slot / 64 * 64, last = slot_last(K);
  if (!slot_gap(K)) return min(64, max(0, K - run));
  return run >= last ? K - last + 16 : (run == last - 64 ? 48 : 64);
}

// Slots k .. k + 7 of row i (a run of 64 belongs to eight neighbouring lanes; all lanes
// of the warp take part): scale, split, store (``in``: inside the operand).  Returns the run's
// bits of the flag, all where its scale is out of range or an entry is not finite.
__device__ __forceinline__ unsigned split_run(const float (&x)[8], const SplitOp& o, int i, int k,
                                              bool in, int kp) {
  unsigned mx = 0, mn = 0xffffffffu;  // mn: the least entry that is not zero, less one
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const unsigned m = __float_as_uint(x[e]) & 0x7fffffffu;
    mx = max(mx, m);
    mn = min(mn, m - 1u);
  }
#pragma unroll
  for (int d = 1; d < 8; d <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, d));
  int sh = mx ? 14 - ((int)(mx >> 23) - 127) : 0;
  unsigned bits = sh > 60 || sh < -60 ? kFlagAll : 0u;  // (non-finite: sh = -114)
  sh = min(60, max(-60, sh));
  const float sc = pow2f(sh);
  const bool lossy = mn < ((unsigned)(125 - sh) << 23) - 1u;  // 2^sh x below 2^-2
  // pairs: one instruction per two values
  __align__(16) __half2 hi[4], lo[4];
  __half2 lows = __float2half2_rn(0.f);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float y0 = x[2 * e] * sc, y1 = x[2 * e + 1] * sc;
    hi[e] = __floats2half2_rn(y0, y1);
    const float2 h = __half22float2(hi[e]);
    lo[e] = __floats2half2_rn(y0 - h.x, y1 - h.y);
    lows = __hadd2(lows, __hlt2(__habs2(hi[e]), __float2half2_rn(512.f)));
  }
  // rare in dense data (a sparse run has four such entries in one lane)
  const bool few = __low2float(lows) + __high2float(lows) >= 4.f;
  if (__any_sync(0xffffffffu, few || lossy)) {
    const int len = run_length(k, o.K), most = mx ? len * 3 / 8 : 64;
    auto below = [&](float bound) {  // entries of the run, from what its lanes hold
      __half2 c = __float2half2_rn(0.f);
#pragma unroll
      for (int e = 0; e < 4; ++e) c = __hadd2(c, __hlt2(__habs2(hi[e]), __float2half2_rn(bound)));
      int m = (int)(__low2float(c) + __high2float(c));
#pragma unroll
      for (int d = 1; d < 8; d <<= 1) m += __shfl_xor_sync(0xffffffffu, m, d);
      return m - (64 - len);
    };
    if (below(len < 48 ? 256.f : 512.f) > most) bits |= kSparse;
    if (below(len < 48 ? 8.f : 7.f) > most) bits |= kSparser;
    const int lost = below(0.25f);
    if (lossy) bits |= lost > (len < 48 ? 4 : bits & kSparse ? 8 : 2) ? kFlagAll : kLossy;
  }
  if (in) {
    unsigned char* d = o.dst + block_line(i, k / 64, kp / 64) * 128 + k % 64 * 2;
    *reinterpret_cast<uint4*>(d) = *reinterpret_cast<const uint4*>(hi);
    *reinterpret_cast<uint4*>(d + 16384) = *reinterpret_cast<const uint4*>(lo);
    if (k % 64 == 0) o.sc[(int64_t)(k / 64) * o.pitch + i] = pow2f(-sh);
  }
  return bits;
}

// what the runs of a warp raise (all lanes take part)
__device__ __forceinline__ void raise_bits(unsigned* flag, unsigned bits, const SplitOp& o) {
  bits = __reduce_or_sync(0xffffffffu, bits) << o.bit;
  if (bits && (threadIdx.x & 31) == 0 && bits & ~*const_cast<volatile unsigned*>(flag))
    atomicOr(flag, bits);
}

// FP16 halves: tiles of 64 rows x 128 k (two runs), zero past K (kp = rup(K, 64)), one
// pass over the operand: eight lanes hold a run and find its largest entry by shuffles.
// An entry y = 2^sh x with 0 < |y| < 2^-2 may have fewer than 22 bits.
// 8192 x 8192: 101 us transposed, 93 us not, 4 bytes read and 4 written per entry
// (floor 79); TF32 halves (8 written) took 196 us.  Conversions in pairs and a thread's loads
// issued at once take 3 us off a split inside the adjoint (8192 x 64, 16 rounds: 1310.3 ->
// 1303.9 us, 1313.8 -> 1310.5 in a second run).  Five CTAs per SM (48 registers): with the 62
// of a free choice 3001 and 1025 rows of 5003, read by scalars, took 47 us instead of 42.
constexpr int kSpR = 64, kSpK = 128;
__global__ void __launch_bounds__(256, 5) split_f16_kernel(const __grid_constant__ SplitPair sp) {
  __shared__ float tile[kSpK][kSpR + 1];
  const bool second = (int)blockIdx.x >= sp.o[0].blocks;
  const SplitOp& o = sp.o[second];
  const int b = blockIdx.x - (second ? sp.o[0].blocks : 0);
  const int kp = (o.K + 63) / 64 * 64;
  const int kb = (kp + kSpK - 1) / kSpK, ib = (o.rows + kSpR - 1) / kSpR;
  // neighbouring CTAs read neighbouring memory
  const int i0 = (o.cs == 1 ? b / kb : b % ib) * kSpR, k0 = (o.cs == 1 ? b % kb : b / ib) * kSpK;
  const int tid = threadIdx.x;
  griddep_wait();
  griddep_launch_dependents();
  if (b == 0 && tid == 0) *o.fmt = 0u;
  // one thread's reading for the CTA, which leaves as a whole
  const unsigned flag = tid == 0 ? *const_cast<volatile unsigned*>(sp.flag) : 0u;
  if (o.cs != 1) {  // transpose: 16 lanes read 64 rows of one k
    const int il = 4 * (tid & 15);
#pragma unroll
    for (int u = 0; u < kSpK / 16; ++u) {
      const int kl = u * 16 + (tid >> 4), i = i0 + il;
      const int k = slot_value(k0 + u * 16, o.K) + (tid >> 4);
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (k < o.K) {
        const float* col = o.X + (int64_t)k * o.cs + i;
        if (o.vec && i + 4 <= o.rows) {
          const float4 x = *reinterpret_cast<const float4*>(col);
          v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (i + e < o.rows) v[e] = col[e];
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) tile[kl][il + e] = v[e];
    }
  }
  constexpr int NU = kSpR * kSpK / (8 * 256);
  float x[NU][8];
  if (o.cs == 1) {  // all loads of a thread in flight at once
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const int idx = u * 256 + tid;
      const int i = i0 + idx / (kSpK / 8), slot = k0 + idx % (kSpK / 8) * 8;
      const int k = slot_value(slot, o.K);
      const bool in = i < o.rows && slot < kp;
      const float* row = o.X + (int64_t)i * o.rs + k;
      if (in && o.vec && k + 8 <= o.K) {
        const float4 p = reinterpret_cast<const float4*>(row)[0];
        const float4 q = reinterpret_cast<const float4*>(row)[1];
        x[u][0] = p.x; x[u][1] = p.y; x[u][2] = p.z; x[u][3] = p.w;
        x[u][4] = q.x; x[u][5] = q.y; x[u][6] = q.z; x[u][7] = q.w;
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) x[u][e] = in && k + e < o.K ? row[e] : 0.f;
      }
    }
  }
  if (__syncthreads_or(needs_tf32(flag))) return;
  unsigned bits = 0;
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    const int idx = u * 256 + tid;
    const int il = idx / (kSpK / 8), kl = idx % (kSpK / 8) * 8;
    const int i = i0 + il, k = k0 + kl;
    const bool in = i < o.rows && k < kp;
    if (o.cs != 1) {
#pragma unroll
      for (int e = 0; e < 8; ++e) x[u][e] = tile[kl + e][il];  // zeros past the operand
    }
    bits |= split_run(x[u], o, i, k, in, kp);
  }
  raise_bits(sp.flag, bits, o);
}

// TF32 halves, only when the flag is set (else the kernel returns at once) and
// the buffer does not hold them already (kp = rup(K, 32), zero past K): tiles of 32 rows x 32 k,
// two at a time for their loads, read along whichever index has unit stride.  With one tile and
// half the CTAs, after an FP16 split that ran to its end, a product on TF32 halves took 881 us
// at 8192 x 64 x 8192 and 186 at 2048^3; 326 and 136 so.
constexpr int kSt = 2;
__global__ void __launch_bounds__(256, 4) split_tf32_kernel(const __grid_constant__ SplitPair sp) {
  griddep_wait();
  griddep_launch_dependents();
  if (!needs_tf32(*sp.flag)) return;
  __shared__ float tile[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 1
  for (int w = 0; w < 2; ++w) {
    const SplitOp& o = sp.o[w];
    if (*o.fmt != 0u) continue;
    const int kp = (o.K + 31) / 32 * 32;
    const int kb = kp / 32, ib = (o.rows + 31) / 32;
    const long long tiles = (long long)kb * ib;
    const bool k_fast = o.cs == 1;
    // this thread's four values of a tile: row il, k kl .. kl + 3
    const int il = warp * 4 + (lane >> 3), kl = (lane & 7) * 4;
    for (long long t0 = (long long)blockIdx.x * kSt; t0 < tiles; t0 += (long long)gridDim.x * kSt) {
      float x[kSt][4];
#pragma unroll
      for (int u = 0; u < kSt; ++u) {
        const long long t = t0 + u;
        const int i0 = (int)(k_fast ? t / kb : t % ib) * 32, k0 = (int)(k_fast ? t % kb : t / ib) * 32;
        if (k_fast) {
          const int i = i0 + il, k = k0 + kl;
          const float* row = o.X + (int64_t)i * o.rs + k;
          const bool in = t < tiles && i < o.rows;
          if (in && o.vec && k + 4 <= o.K) {
            const float4 v = *reinterpret_cast<const float4*>(row);
            x[u][0] = v.x; x[u][1] = v.y; x[u][2] = v.z; x[u][3] = v.w;
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) x[u][e] = in && k + e < o.K ? row[e] : 0.f;
          }
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {  // k warp + 8 e, row lane
            const int i = i0 + lane, k = k0 + warp + 8 * e;
            x[u][e] = t < tiles && i < o.rows && k < o.K ? o.X[(int64_t)k * o.cs + i] : 0.f;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kSt; ++u) {
        const long long t = t0 + u;
        if (t >= tiles) break;
        if (!k_fast) {
          __syncthreads();
#pragma unroll
          for (int e = 0; e < 4; ++e) tile[warp + 8 * e][lane] = x[u][e];
          __syncthreads();
#pragma unroll
          for (int e = 0; e < 4; ++e) x[u][e] = tile[kl + e][il];
        }
        const int i = (int)(k_fast ? t / kb : t % ib) * 32 + il, kc = (int)(k_fast ? t % kb : t / ib);
        if (i >= o.rows) continue;
        float hi[4], lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          // round to nearest TF32 (ties away from zero): add half of the dropped
          // 13-bit field, then clear it; x - hi is exact
          hi[e] = __uint_as_float((__float_as_uint(x[u][e]) + 0x1000u) & 0xFFFFE000u);
          const float r = x[u][e] - hi[e];
          lo[e] = __uint_as_float((__float_as_uint(r) + 0x1000u) & 0xFFFFE000u);
        }
        float4* d = reinterpret_cast<float4*>(o.dst + block_line(i, kc, kb) * 128) + kl / 4;
        d[0] = make_float4(hi[0], hi[1], hi[2], hi[3]);
        d[1024] = make_float4(lo[0], lo[1], lo[2], lo[3]);
      }
    }
  }
}

// ---------------------------------------------------------------- CUDA-core GEMM
constexpr int kSB = 64;   // tile
constexpr int kSK = 16;   // inner chunk

// One tile of C (or of a split's partial): acc = sum over k in [k0, k1) of
// A(m, k) B(k, n) with A(m, k) = A[m * a_rs + k * a_cs], B(k, n) = B[k * b_rs +
// n * b_cs].  One split: C(m, n) = alpha acc + beta C(m, n) (C(m, n) at
// C[m * c_rs + n * c_cs]); else the partial goes to work[split][m][n].
template <typename T>
__global__ void __launch_bounds__(256)
    gemm_simt_kernel(int M, int N, int K, int kchunk, T alpha, const T* __restrict__ A,
                     int64_t a_rs, int64_t a_cs, const T* __restrict__ B, int64_t b_rs,
                     int64_t b_cs, T beta, T* C, int64_t c_rs, int64_t c_cs, T* work) {
  __shared__ T As[kSK][kSB + 1];
  __shared__ T Bs[kSK][kSB + 1];
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * kSB, n0 = blockIdx.x * kSB;
  const int kbeg = blockIdx.z * kchunk;
  const int kend = (kbeg + kchunk < K) ? kbeg + kchunk : K;
  T acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
  const bool a_kfast = a_cs == 1;
  const bool b_nfast = b_cs == 1;
  for (int k0 = kbeg; k0 < kend; k0 += kSK) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int e = tid + 256 * l;  // 0 .. 1023 = 64 x 16
      int mm, kk;
      if (a_kfast) {
        kk = e & 15;
        mm = e >> 4;
      } else {
        mm = e & 63;
        kk = e >> 6;
      }
      const int gm = m0 + mm, gk = k0 + kk;
      As[kk][mm] = (gm < M && gk < kend) ? A[(int64_t)gm * a_rs + (int64_t)gk * a_cs] : T(0);
      int nn, kb;
      if (b_nfast) {
        nn = e & 63;
        kb = e >> 6;
      } else {
        kb = e & 15;
        nn = e >> 4;
      }
      const int gn = n0 + nn, gkb = k0 + kb;
      Bs[kb][nn] = (gn < N && gkb < kend) ? B[(int64_t)gkb * b_rs + (int64_t)gn * b_cs] : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kSK; ++kk) {
      T a[4], b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a[q] = As[kk][ty + 16 * q];
        b[q] = Bs[kk][tx + 16 * q];
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = fma(a[x], b[y], acc[x][y]);
    }
    __syncthreads();
  }
  T* wb = work ? work + (int64_t)blockIdx.z * M * N : nullptr;
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const int m = m0 + ty + 16 * x;
    if (m >= M) continue;
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int n = n0 + tx + 16 * y;
      if (n >= N) continue;
      if (wb) {
        wb[(int64_t)m * N + n] = acc[x][y];
      } else {
        T* c = C + (int64_t)m * c_rs + (int64_t)n * c_cs;
        *c = beta == T(0) ? alpha * acc[x][y] : alpha * acc[x][y] + beta * *c;
      }
    }
  }
}

// C(m, n) = alpha sum_s work[s][m][n] + beta C(m, n): one warp per output, lanes over
// the splits, then a fixed shuffle tree (deterministic).
template <typename T>
__global__ void gemm_reduce_kernel(int M, int N, int splits, T alpha, const T* __restrict__ work,
                                   T beta, T* C, int64_t c_rs, int64_t c_cs) {
  const int lane = threadIdx.x & 31;
  const int64_t mn = (int64_t)M * N;
  const int64_t wpb = blockDim.x / 32;
  for (int64_t o = blockIdx.x * wpb + (threadIdx.x >> 5); o < mn; o += (int64_t)gridDim.x * wpb) {
    T s = T(0);
    for (int q = lane; q < splits; q += 32) s += work[(int64_t)q * mn + o];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) {
      const int m = (int)(o / N), n = (int)(o - (int64_t)m * N);
      T* c = C + (int64_t)m * c_rs + (int64_t)n * c_cs;
      *c = beta == T(0) ? alpha * s : alpha * s + beta * *c;
    }
  }
}

// D = alpha (pieces) + beta C for the tiles cut along K: a CTA adds ROWS rows of one
// tile, the pieces in their order along K.  SPLIT (ROWS = 64 = BN, every tile cut): D's
// columns also go to the split operand ``nx``, a run of 64 slots per CTA and column.
// Bound by the latency of its few CTAs (128 at 8192 rows x 64 columns: 2 MB of D, 8 MB of
// pieces from L2), so a thread has four values and every piece's load in flight (four
// times the rows per thread: 10.1 us against 7.8); the split inside it saves the launches
// of a split of its own: the adjoint of 16 rounds at 8192 x 64 1445 -> 1394 us.
template <int BN, int ROWS, bool SPLIT>
__global__ void __launch_bounds__(ROWS * BN / 4)
    gemm_parts_kernel(const GArgs a, int tiles, const __grid_constant__ SplitOp nx,
                      unsigned* nx_flag) {
  __shared__ float tile[SPLIT ? ROWS : 1][SPLIT ? BN + 1 : 1];
  griddep_wait();
  griddep_launch_dependents();
  const unsigned flag = *a.flag;
  const bool f16 = !needs_tf32(flag);
  const int nk = f16 ? a.kp16 / 64 : a.kp32 / 32;
  const int row0 = blockIdx.y * ROWS;
  const int e = threadIdx.x, lrow = e / (BN / 4), col = e % (BN / 4) * 4;
  int r = blockIdx.x, mb, nb;
  g_tile(a.dp + r, (a.M + kGBM - 1) / kGBM, (a.N + BN - 1) / BN, mb, nb);
  int m = mb * kGBM + row0 + lrow;
  const int n = nb * BN + col;
  if constexpr (SPLIT) {  // slots; a moved row may lie in the tile before (one column: mb == r)
    m = slot_value(m & ~15, nx.K) + (m & 15);
    if (m < r * kGBM) r = --mb;
  }
  const long long W = (long long)(tiles - a.dp) * nk, lo = (long long)r * nk, hi = lo + nk;
  // ranges that meet the tile: W c / cut < hi and W (c + 1) / cut > lo (both rounded down;
  // multiplied out: 64-bit divisions in every warp took 1 us of 9)
  int c0 = r * a.cut / (tiles - a.dp), c1;
  while (c0 > 0 && W * c0 >= (lo + 1) * a.cut) --c0;
  while (W * (c0 + 1) < (lo + 1) * a.cut) ++c0;
  c1 = c0;
  while (W * (c1 + 1) < hi * a.cut) ++c1;
  const bool whole = c0 == c1;  // computed by one range: D is complete
  if (whole && !SPLIT) return;
  float v[4] = {0.f, 0.f, 0.f, 0.f};
  if (m < a.M && n < a.N) {
    float* d = a.D + (int64_t)m * a.ldd + n;
    const bool vec = a.vec_ok && n + 4 <= a.N;
    if (!whole) {
      const float* w = a.work + ((int64_t)(c0 + r) * kGBM + m - mb * kGBM) * BN + col;
      float4 s = *reinterpret_cast<const float4*>(w);
#pragma unroll 8
      for (int c = c0 + 1; c <= c1; ++c) {
        const float4 x = *reinterpret_cast<const float4*>(w + (int64_t)(c - c0) * kGBM * BN);
        s.x += x.x;
        s.y += x.y;
        s.z += x.z;
        s.w += x.w;
      }
      v[0] = a.alpha * s.x; v[1] = a.alpha * s.y; v[2] = a.alpha * s.z; v[3] = a.alpha * s.w;
      if (a.C && a.beta != 0.f) {
        const float* cp = a.C + (int64_t)m * a.ldc + n;
        for (int j = 0; j < 4 && n + j < a.N; ++j) v[j] += a.beta * cp[j];
      }
      if (vec)
        *reinterpret_cast<float4*>(d) = make_float4(v[0], v[1], v[2], v[3]);
      else
        for (int j = 0; j < 4 && n + j < a.N; ++j) d[j] = v[j];
    } else {
      for (int j = 0; j < 4 && n + j < a.N; ++j) v[j] = d[j];
    }
  }
  if constexpr (SPLIT) {
#pragma unroll
    for (int j = 0; j < 4; ++j) tile[lrow][col + j] = n + j < a.N ? v[j] : 0.f;
  }
  if constexpr (SPLIT) {
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *nx.fmt = 0u;
    __syncthreads();
    const int kp = (nx.K + 63) / 64 * 64, k0 = blockIdx.x * kGBM + row0;
    unsigned bits = 0;
    if (e < BN * ROWS / 8) {  // whole warps
      const int i = e / (ROWS / 8), kl = e % (ROWS / 8) * 8, k = k0 + kl;
      float x[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = tile[kl + j][i];  // zeros past D
      bits = split_run(x, nx, i, k, i < nx.rows && k < kp, kp);
    }
    raise_bits(nx_flag, bits, nx);
    // A goes on as it is; once on TF32 halves, the chain stays there
    if (blockIdx.x == 0 && blockIdx.y == 0 && e == 0) atomicOr(nx_flag, f16 ? flag & kFlagAll : flag);
  }
}

template <int BN, bool HALVES>
cudaError_t launch_tc_gemm_t(const GMaps& maps, const GArgs& a, const SplitOp* next, bool* did,
                             unsigned* next_flag, int num_sms, cudaStream_t s) {
  using Sh = GShape<BN>;
  static const cudaError_t configured = [] {
    cudaFuncAttributes at;
    cudaError_t e = cudaFuncGetAttributes(&at, tc_gemm_kernel<BN, HALVES>);
    // the registers handed over must be there, or setmaxnreg would wait forever
    if (e == cudaSuccess && Sh::Rebalance && at.numRegs * Sh::Threads < 40 * 128 + 224 * 256)
      e = cudaErrorInvalidConfiguration;
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(tc_gemm_kernel<BN, HALVES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Sh::SmemBytes);
  }();
  if (configured != cudaSuccess) return configured;
  const int tiles = ((a.M + kGBM - 1) / kGBM) * ((a.N + BN - 1) / BN);
  const int busy = a.dp > a.cut ? a.dp : a.cut;
  const int pairs = busy < num_sms / 2 ? busy : num_sms / 2;
  const cudaError_t e =
      launch_pdl(tc_gemm_kernel<BN, HALVES>, 2 * pairs, Sh::Threads, Sh::SmemBytes, s, maps, a);
  if (e != cudaSuccess || tiles == a.dp) return e;
  if constexpr (BN == 64) {
    if (next && a.dp == 0 && a.N <= BN) {
      *did = true;
      return launch_pdl(gemm_parts_kernel<BN, 64, true>, dim3(tiles, kGBM / 64), 1024, 0, s,
                        a, tiles, *next, next_flag);
    }
  }
  constexpr int kRows = 1024 / BN;  // four values per thread
  return launch_pdl(gemm_parts_kernel<BN, kRows, false>, dim3(tiles - a.dp, kGBM / kRows), 256, 0,
                    s, a, tiles, SplitOp{}, nullptr);
}

// A split operand as lines of 128 bytes (64 FP16 or 32 TF32 values), boxes of
// box_lines contiguous lines, 128-byte swizzle
bool make_tmap_lines(CUtensorMap* out, const void* base, bool f16, int64_t lines, int box_lines) {
  static const PFN_cuTensorMapEncodeTiled_v12000 encode = []() {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      fn = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }();
  if (!encode) return false;
  cuuint64_t dims[2] = {f16 ? 64u : 32u, (cuuint64_t)lines};
  cuuint64_t strides[1] = {128u};
  cuuint32_t box[2] = {f16 ? 64u : 32u, (cuuint32_t)box_lines};
  cuuint32_t estr[2] = {1, 1};
  return encode(out, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
                const_cast<void*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

SplitOp split_op(const TcOperand* t, bool second) {
  SplitOp o{};
  if (!t) return o;
  o.X = t->X;
  o.rs = t->rs;
  o.cs = t->cs;
  o.rows = t->rows;
  o.K = t->K;
  o.dst = reinterpret_cast<unsigned char*>(t->buf);
  o.fmt = t->words;
  o.sc = reinterpret_cast<float*>(t->words + 4);
  o.pitch = (t->rows + 3) / 4 * 4;
  o.bit = second ? 4 : 0;
  o.vec = (t->cs == 1 ? t->rs : t->cs) % 4 == 0 && reinterpret_cast<uintptr_t>(t->X) % 16 == 0;
  return o;
}

// Tile width of a product of nk chunks, the tiles computed whole (full waves of
// CTA pairs) and the number of ranges the others are cut into (0: all whole).  The
// modelled time is the longest pair's chunks times the width's chunk time (1.03,
// 0.62, 0.50 us at 256, 128, 64 columns: 4096^3 in 265, 278, 449 us), 7 us of
// start and end, and for cut tiles a launch and their pieces written and read.
// It lies within 4 us of the best of the six choices at 1024^3 (64 columns, whole:
// 13 us), 2048^3 (256, whole: 40), 3001 x 1025 x 5003 (256, cut: 76 + 12),
// 4096 x 128 x 4096 (128, cut: 21 + 5), 8192 x 64 x 8192 (64, cut: 57 + 6) and
// 300 x 40 x 5000 (64, cut: 9 + 7, whole: 38).
//
// A product that leaves half of the pairs idle (at 256 columns) has time for smaller sums,
// as the chains of such products (A^16 at n <= 1500, the rounds of an iteration) add up
// their errors: its choices are those whose pieces add at most 20 chunks one after the
// other, or two thirds of its chunks (all choices where there is none), and up to 32 chunks
// every other one goes to two accumulators, which takes a fifth off the bias that the tensor
// cores' truncation leaves (8.9e-8 of a product; a re-evaluated A^16 has 15 times that).
// Errors against FP64, time: A^16 re-evaluated at n = 1000 1.42e-6 -> 1.19e-6, 95.5 -> 101.4 us;
// 314 x 3654 x 2299 1.73e-7 -> 1.54e-7, 93 -> 95; adjoint of 16 rounds at 2000 x 200 3.1e-7
// -> 2.7e-7, 529 -> 550.  20 chunks add up to no more error than TF32 halves left (n = 1250
// 1.562e-7 of a product against 1.571e-7); with 16 the products of n = 1050 to 1280 were cut for
// nothing (n = 1250 153 us a re-evaluation, 137 so), with all 22 n = 1352 would be 1.598e-7
// against 1.581e-7 (145 us, 174 so).  (Every chunk in halves: 0.99e-6, but 103.6 us, and 16.2 -> 19.9 ms
// for the products of n = 8192, whose epilogue then takes longer than their MMAs.)
void gemm_plan(int M, int N, int nk, int num_sms, int64_t work_floats, GArgs& a, int* bn_out,
               bool* halves) {
  const int pairs = num_sms / 2;
  const long long mt = (M + kGBM - 1) / kGBM;
  const bool small = mt * ((N + 255) / 256) <= pairs / 2;
  const int longest = small ? std::max(20, nk * 2 / 3) : nk;
  double best = 1e30;
  bool best_short = false;
  for (int bn = 256; bn >= 64; bn /= 2) {
    const double chunk = bn == 256 ? 1.03 : (bn == 128 ? 0.62 : 0.50);
    const long long tiles = mt * ((N + bn - 1) / bn);
    for (int c = 0; c < 2; ++c) {
      long long left = c ? tiles % pairs : 0;
      int cut = (int)(left * nk / 4 < pairs ? left * nk / 4 : pairs);  // at least four chunks each
      if (c && (cut <= left || (left + cut) * kGBM * bn > work_floats)) continue;
      double t = 7.0 + (double)((tiles - left + pairs - 1) / pairs) * nk * chunk;
      if (cut)
        t += (double)((left * nk + cut - 1) / cut) * chunk + 3.5 +
             (double)(left + cut) * (kGBM * bn) * 8.0 / 6e6;
      const long long chain = tiles > left ? nk : (left * nk + cut - 1) / cut;
      const bool is_short = chain <= longest;
      if (is_short == best_short ? t < best : is_short) {
        best = t;
        best_short = is_short;
        *bn_out = bn;
        a.dp = (int)(tiles - left);
        a.cut = cut;
      }
    }
  }
  *halves = small && nk <= 32;
}

}  // namespace

int64_t tc_operand_floats(int64_t rows, int64_t K) {
  return (rows + 127) / 128 * 128 * 2 * ((K + 31) / 32 * 32);
}
int64_t tc_work_floats(int64_t a_rows, int64_t b_rows, int64_t K, int num_sms) {
  const int64_t pairs = num_sms / 2, nk = (K + 63) / 64;
  int64_t most = 0;
  for (int bn = 256; bn >= 64; bn /= 2) {
    int64_t left = (a_rows + kGBM - 1) / kGBM * ((b_rows + bn - 1) / bn);
    left = left < pairs ? left : pairs;
    const int64_t cut = left * nk / 4 < pairs ? left * nk / 4 : pairs;
    most = most > (left + cut) * kGBM * bn ? most : (left + cut) * kGBM * bn;
  }
  return most;
}
int64_t tc_split_words(int64_t rows, int64_t K) {
  return 4 + (rows + 3) / 4 * 4 * ((K + 63) / 64);
}

cudaError_t launch_tc_split(const TcOperand* a, const TcOperand* b, unsigned* flag,
                            cudaStream_t s) {
  SplitPair sp{};
  sp.flag = flag;
  const TcOperand* in[2] = {a, b};
  for (int w = 0; w < 2; ++w) {
    if (!in[w]) continue;
    if (in[w]->rows <= 0 || in[w]->K <= 0) return cudaErrorInvalidValue;
    // TMA sources and 128-bit loads of the factors
    if ((reinterpret_cast<uintptr_t>(in[w]->buf) | reinterpret_cast<uintptr_t>(in[w]->words)) & 15)
      return cudaErrorInvalidValue;
    sp.o[w] = split_op(in[w], w == 1);
    sp.o[w].blocks = ((sp.o[w].rows + kSpR - 1) / kSpR) *
                     (((sp.o[w].K + 63) / 64 * 64 + kSpK - 1) / kSpK);
  }
  // the smaller operand first: what it raises spares the larger one's split
  if (sp.o[1].blocks < sp.o[0].blocks) std::swap(sp.o[0], sp.o[1]);
  return launch_pdl(split_f16_kernel, sp.o[0].blocks + sp.o[1].blocks, 256, 0, s, sp);
}

cudaError_t launch_tc_gemm(const TcOperand& a, const TcOperand& b, unsigned* flag, float* D,
                           int64_t ldd, const float* C, int64_t ldc, float alpha, float beta,
                           int num_sms, unsigned* status, cudaStream_t s, float* work,
                           int64_t work_floats, bool reverse, const TcOperand* next,
                           bool* next_split, unsigned* next_flag) {
  const int M = a.rows, N = b.rows, K = a.K;
  if (M <= 0 || N <= 0 || K <= 0 || b.K != K) return cudaErrorInvalidValue;
  SplitPair sp{};
  sp.flag = flag;
  sp.o[0] = split_op(&a, false);
  sp.o[1] = split_op(&b, true);
  const cudaError_t es = launch_pdl(split_tf32_kernel, 4 * num_sms, 256, 0, s, sp);
  if (es != cudaSuccess) return es;
  GArgs g{};
  g.M = M;
  g.N = N;
  g.kp16 = (K + 63) / 64 * 64;
  g.kp32 = (K + 31) / 32 * 32;
  int bn = 256;
  bool halves = false;
  gemm_plan(M, N, g.kp16 / 64, num_sms, work ? work_floats : 0, g, &bn, &halves);
  g.reverse = reverse ? 1 : 0;
  GMaps maps;
  const int64_t ab = (M + 127) / 128 * 256, bb = (N + 127) / 128 * 256;  // lines per chunk
  const int nk16 = g.kp16 / 64, nk32 = g.kp32 / 32, bl = bn == 256 ? 256 : bn / 2;
  if (ab * nk32 > INT32_MAX || bb * nk32 > INT32_MAX) return cudaErrorInvalidValue;
  if (!make_tmap_lines(&maps.a16, a.buf, true, ab * nk16, 256) ||
      !make_tmap_lines(&maps.b16, b.buf, true, bb * nk16, bl) ||
      !make_tmap_lines(&maps.a32, a.buf, false, ab * nk32, 256) ||
      !make_tmap_lines(&maps.b32, b.buf, false, bb * nk32, bl))
    return cudaErrorInvalidValue;
  const bool c_used = C != nullptr && beta != 0.f;
  g.D = D;
  g.ldd = ldd;
  g.C = C;
  g.ldc = ldc;
  g.alpha = alpha;
  g.beta = beta;
  g.vec_ok = (ldd % 4 == 0) && (reinterpret_cast<uintptr_t>(D) % 16 == 0) &&
             (!c_used || (ldc % 4 == 0 && reinterpret_cast<uintptr_t>(C) % 16 == 0));
  g.work = work;
  g.sa = sp.o[0].sc;
  g.sb = sp.o[1].sc;
  g.pa = sp.o[0].pitch;
  g.pb = sp.o[1].pitch;
  g.fmta = a.words;
  g.fmtb = b.words;
  g.flag = flag;
  g.status = status;
  const SplitOp nx = split_op(next, true);
  const SplitOp* np = next ? &nx : nullptr;
  auto run = [&](auto width) {
    constexpr int BN = decltype(width)::value;
    return halves ? launch_tc_gemm_t<BN, true>(maps, g, np, next_split, next_flag, num_sms, s)
                  : launch_tc_gemm_t<BN, false>(maps, g, np, next_split, next_flag, num_sms, s);
  };
  if (bn == 256) return run(std::integral_constant<int, 256>{});
  if (bn == 128) return run(std::integral_constant<int, 128>{});
  return run(std::integral_constant<int, 64>{});
}

static int gemm_simt_splits(int M, int N, int K, int num_sms, int64_t work_elems) {
  const int64_t tiles = (int64_t)((M + kSB - 1) / kSB) * ((N + kSB - 1) / kSB);
  int splits = 1;
  // split long inner dimensions until about two waves of CTAs are running
  while (tiles * splits < 2 * num_sms && K / (splits * 2) >= 8 * kSK &&
         (int64_t)(splits * 2) * M * N <= work_elems)
    splits *= 2;
  return splits;
}

template <typename T>
cudaError_t launch_gemm_simt(int M, int N, int K, T alpha, const T* A, int64_t a_rs, int64_t a_cs,
                             const T* B, int64_t b_rs, int64_t b_cs, T beta, T* C, int64_t c_rs,
                             int64_t c_cs, T* work, int64_t work_elems, int num_sms,
                             cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (K <= 0) return cudaErrorInvalidValue;
  const int splits = work ? gemm_simt_splits(M, N, K, num_sms, work_elems) : 1;
  const int kchunk = ((K + splits - 1) / splits + kSK - 1) / kSK * kSK;
  dim3 grid((N + kSB - 1) / kSB, (M + kSB - 1) / kSB, splits);
  gemm_simt_kernel<T><<<grid, 256, 0, s>>>(M, N, K, kchunk, alpha, A, a_rs, a_cs, B, b_rs, b_cs,
                                           beta, C, c_rs, c_cs, splits > 1 ? work : nullptr);
  if (splits == 1) return cudaGetLastError();
  const int64_t outs = (int64_t)M * N;
  const int blocks = (int)((outs + 7) / 8 < 4096 ? (outs + 7) / 8 : 4096);
  gemm_reduce_kernel<T><<<blocks, 256, 0, s>>>(M, N, splits, alpha, work, beta, C, c_rs, c_cs);
  return cudaGetLastError();
}

template cudaError_t launch_gemm_simt<float>(int, int, int, float, const float*, int64_t, int64_t,
                                             const float*, int64_t, int64_t, float, float*,
                                             int64_t, int64_t, float*, int64_t, int, cudaStream_t);
template cudaError_t launch_gemm_simt<double>(int, int, int, double, const double*, int64_t,
                                              int64_t, const double*, int64_t, int64_t, double,
                                              double*, int64_t, int64_t, double*, int64_t, int,
                                              cudaStream_t);

}  // namespace lv
