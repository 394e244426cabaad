// Products X = P F of an n x n FP32 view with a few factor columns, whole rows at a
// time (the Krylov chain K_j = A K_{j-1} of Appendix B).
#include <cuda_runtime.h>

#include "lv_device.cuh"
#include "lv_internal.h"

namespace lv {

namespace {

// A CTA owns a contiguous range of rows and runs over all columns of each, so X's entries
// leave the kernel complete.  The strip passes (lv_pass_ws.cuh) leave one partial set per
// 512 columns to a kernel of their own, which in a chain of dependent products is another
// link.  Thread t keeps the factor entries of columns 4t .. 4t + 3 of every 1024 in
// registers (at most 64), so four view entries cost one 128-bit shared load and 4 R FMAs: the
// pass is bound by reading the view.  Four rows make a batch: its sums are reduced across the
// lanes by halving the values with each shuffle, then across the warps in a fixed order.  Row
// pieces of 4 KB come by bulk copies into a ring of six 16 KB stages, which the warps refill in
// turn.  Two CTAs per SM: with one, its two warps per scheduler left the reductions' latency in
// the open (n = 8192, two columns: 50 us a link against 37 with two; the strips' pass and sum
// 41).  Rows are exact, not boxes of eight, so the CTAs' ranges differ by one row at most.
// Rounding: a chunk's four products are summed by themselves, the chunks in fours, and once a
// lane holds one value its sums are pairs, to the end.  So an entry passes 9 FP32 roundings of
// a sum's size at every n, as in the strips, which sum their partial sets in pairs: the last
// of 15 links is off by 2.5e-7 (n = 1000), 3.2e-7 (8192), 3.4e-7 (16384, one column) against
// the strips' 3.4e-7, 3.6e-7, 3.5e-7.  With chunks one after the other and plain lane sums it
// was 3.1e-7, 3.8e-7 and 4.3e-7; an update at n = 8192, p = 64 took 652 us (two columns) so,
// 656 now.
// One column up to n = 8192 has room for half of the entries (32 registers; with the 64 that
// n = 16384 needs a link was slower than with two columns, and than a strip pass from n = 1300
// to 4096): n = 300 57.0 -> 45.5 us an update, n = 1318 99 -> 81 (strips 98), n = 4096 205 -> 178,
// n = 8192 665 -> 625.
constexpr int kRpRows = 4, kRpCols = 1024, kRpStages = 6;
constexpr int kRpThreads = 256, kRpWarps = kRpThreads / 32;
constexpr int kRpStageBytes = kRpRows * kRpCols * 4;

struct RpBars {
  uint64_t full[kRpStages], empty[kRpStages];
  int uses[kRpStages];  // loads of a stage so far
  int abort;
};

template <int R>
constexpr int kRpSmem = kRpStages * kRpStageBytes + 2 * kRpWarps * kRpRows * R * (int)sizeof(float2) +
                        (int)sizeof(RpBars);

// (s, low) += v as a pair, Knuth's TwoSum
__device__ __forceinline__ void rp_two_sum(float& s, float& low, float v) {
  const float z = s + v, b = z - s;
  low += (s - (z - b)) + (v - b);
  s = z;
}

// false once a wait of this CTA has run out (status then holds the timeout)
__device__ __forceinline__ bool rp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                        unsigned* status) {
  if (mbar_try_wait(bar, parity)) return true;
  if (*abort_flag) return false;
  if (mbar_wait_bounded(bar, parity, status)) return true;
  *abort_flag = 1;
  return false;
}

// untiled copy of ``bytes`` (a multiple of 16) between 16-byte aligned addresses
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

template <int R, int CH>
__global__ void __launch_bounds__(kRpThreads, 2)
    row_products_kernel(const float* __restrict__ P, int64_t ldp, const float* F, int64_t fs,
                        int n, int r, float* X, int64_t xs, int vec, int reverse,
                        unsigned* status) {
  extern __shared__ __align__(128) unsigned char rp_mem[];
  float* ring = reinterpret_cast<float*>(rp_mem);
  float2* red = reinterpret_cast<float2*>(rp_mem + kRpStages * kRpStageBytes);
  RpBars* bars = reinterpret_cast<RpBars*>(rp_mem + kRpSmem<R> - sizeof(RpBars));
  volatile int* abort_flag = &bars->abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r0 = (int)((int64_t)n * blockIdx.x / gridDim.x);
  const int r1 = (int)((int64_t)n * (blockIdx.x + 1) / gridDim.x);
  const int nb = (r1 - r0 + kRpRows - 1) / kRpRows;
  const int nch = (n + kRpCols - 1) / kRpCols;
  auto batch_row = [&](int b) { return r0 + kRpRows * (reverse ? nb - 1 - b : b); };
  const int total = nb * nch;  // (batch, column chunk) steps
  if (tid == 0) {
    for (int i = 0; i < kRpStages; ++i) {
      mbar_init(&bars->full[i], 1);
      mbar_init(&bars->empty[i], kRpWarps);
      bars->uses[i] = 0;
    }
    bars->abort = 0;
    fence_mbar_init();
  }
  __syncthreads();

  // a whole warp requests the rows of step t
  auto request = [&](int t) {
    const int b = t / nch, c = t - b * nch, st = t % kRpStages;
    const int row0 = batch_row(b), nr = min(kRpRows, r1 - row0);
    // past n: up to three entries of the row's padding (ldp is a multiple of four)
    const uint32_t bytes = 4u * (uint32_t)((min(kRpCols, n - c * kRpCols) + 3) & ~3);
    if (lane == 0) {
      fence_proxy_async();
      mbar_arrive_expect_tx(&bars->full[st], bytes * nr);
      ++bars->uses[st];
    }
    __syncwarp();
    if (lane < nr)
      bulk_load(ring + (st * kRpRows + lane) * kRpCols,
                P + (int64_t)(row0 + lane) * ldp + c * kRpCols, bytes, &bars->full[st]);
  };
  // the kernel before does not write the view, so its first rows are requested at once
  if (warp == 0)
    for (int t = 0; t < kRpStages && t < total; ++t) request(t);
  griddep_wait();
  griddep_launch_dependents();
  float u[CH][4][R];
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int col = c * kRpCols + 4 * tid;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const float* f = F + (int64_t)q * fs + col;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (q < r) {
        if (vec && col + 4 <= n) {
          v = *reinterpret_cast<const float4*>(f);
        } else {
          if (col < n) v.x = f[0];
          if (col + 1 < n) v.y = f[1];
          if (col + 2 < n) v.z = f[2];
          if (col + 3 < n) v.w = f[3];
        }
      }
      u[c][0][q] = v.x;
      u[c][1][q] = v.y;
      u[c][2][q] = v.z;
      u[c][3][q] = v.w;
    }
  }
  constexpr int NV = kRpRows * R;  // sums of a batch
  int st = 0, step = 0;
  uint32_t phase = 0;
  bool ok = true;
  for (int b = 0; b < nb; ++b) {
    const int row0 = batch_row(b), nr = min(kRpRows, r1 - row0);
    constexpr bool GRP = CH > 4;
    float acc[NV], tot[GRP ? NV : 1];  // sums of up to four chunks, of the fours before
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = 0.f;
    if constexpr (GRP)
#pragma unroll
      for (int i = 0; i < NV; ++i) tot[i] = 0.f;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      if (c < nch) {
        ok = ok && rp_wait(&bars->full[st], phase, abort_flag, status);
        float4 x[kRpRows];
#pragma unroll
        for (int j = 0; j < kRpRows; ++j)
          x[j] = *reinterpret_cast<const float4*>(ring + (st * kRpRows + j) * kRpCols + 4 * tid);
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->empty[st]);
        const int left = n - c * kRpCols - 4 * tid;  // entries of the view from this column on
        if (left < 4) {
#pragma unroll
          for (int j = 0; j < kRpRows; ++j) {
            if (left < 1) x[j].x = 0.f;
            if (left < 2) x[j].y = 0.f;
            if (left < 3) x[j].z = 0.f;
            x[j].w = 0.f;
          }
        }
#pragma unroll
        for (int j = 0; j < kRpRows; ++j)
#pragma unroll
          for (int q = 0; q < R; ++q) {
            float t = x[j].x * u[c][0][q];
            t = fmaf(x[j].y, u[c][1][q], t);
            t = fmaf(x[j].z, u[c][2][q], t);
            acc[j * R + q] += fmaf(x[j].w, u[c][3][q], t);
          }
        if (GRP && c % 4 == 3) {
#pragma unroll
          for (int i = 0; i < NV; ++i) {
            tot[GRP ? i : 0] += acc[i];
            acc[i] = 0.f;
          }
        }
        // the stage of the step before is refilled, by each warp in its turn
        if (step >= 1 && step % kRpWarps == warp && step - 1 + kRpStages < total) {
          const int pt = step - 1;
          ok = ok && rp_wait(&bars->empty[pt % kRpStages], (uint32_t)((pt / kRpStages) & 1),
                             abort_flag, status);
          if (__all_sync(0xffffffffu, ok)) request(pt + kRpStages);
        }
        ++step;
        if (++st == kRpStages) {
          st = 0;
          phase ^= 1u;
        }
      }
    }
    if constexpr (GRP)
#pragma unroll
      for (int i = 0; i < NV; ++i) acc[i] += tot[i];
    // lane sums: while there are several values, each shuffle halves their number; lane
    // ends with value lane / (32 / NV), which goes on as a pair
    int cnt = NV;
    float low = 0.f;
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
      if (cnt > 1) {
        cnt >>= 1;
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int i = 0; i < NV / 2; ++i)
          if (i < cnt) {
            const float give = up ? acc[i] : acc[i + cnt], keep = up ? acc[i + cnt] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, m);
          }
      } else {
        const float l = __shfl_xor_sync(0xffffffffu, low, m);
        rp_two_sum(acc[0], low, __shfl_xor_sync(0xffffffffu, acc[0], m));
        low += l;
      }
    }
    float2* rb = red + (b & 1) * kRpWarps * NV;
    if (lane % (32 / NV) == 0) rb[warp * NV + lane / (32 / NV)] = make_float2(acc[0], low);
    __syncthreads();
    if (tid < NV) {
      float s = rb[tid].x;
      low = rb[tid].y;
#pragma unroll
      for (int w = 1; w < kRpWarps; ++w) {
        const float2 v = rb[w * NV + tid];
        rp_two_sum(s, low, v.x);
        low += v.y;
      }
      s += low;
      const int j = tid / R, q = tid % R;
      if (j < nr && q < r && ok) X[(int64_t)q * xs + row0 + j] = s;
    }
  }
  __syncthreads();
  if (*abort_flag && tid < kRpStages && bars->uses[tid] > 0)  // copies in flight land (bounded)
    mbar_wait_bounded(&bars->full[tid], (uint32_t)((bars->uses[tid] - 1) & 1), nullptr);
}

template <int R, int CH>
cudaError_t launch_rows_t(const float* P, int64_t ldp, const float* F, int64_t fs, int n, int r,
                          float* X, int64_t xs, bool reverse, int num_sms, unsigned* status,
                          cudaStream_t s) {
  static const cudaError_t configured = cudaFuncSetAttribute(
      row_products_kernel<R, CH>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRpSmem<R>);
  if (configured != cudaSuccess) return configured;
  // every resident CTA, while there are batches for it
  const int batches = (n + kRpRows - 1) / kRpRows;
  const int resident = 2 * num_sms;
  const int grid = batches < resident ? batches : resident;
  const int vec = fs % 4 == 0 && (reinterpret_cast<uintptr_t>(F) & 15) == 0;
  return launch_pdl(row_products_kernel<R, CH>, grid, kRpThreads, kRpSmem<R>, s, P, ldp, F, fs, n,
                    r, X, xs, vec, reverse ? 1 : 0, status);
}

}  // namespace

bool row_products_fit(const void* P, int64_t ldp, int n, int r) {
  if (ldp % 4 || (reinterpret_cast<uintptr_t>(P) & 15)) return false;  // bulk copies
  return r <= 1 ? n <= 16 * kRpCols : r == 2 ? n <= 8 * kRpCols : r <= 4 && n <= 4 * kRpCols;
}

cudaError_t launch_row_products(const float* P, int64_t ldp, const float* F, int64_t fs, int n,
                                int r, float* X, int64_t xs, bool reverse, int num_sms,
                                unsigned* status, cudaStream_t s) {
  if (n < 1 || r < 1 || !row_products_fit(P, ldp, n, r)) return cudaErrorInvalidValue;
  if (r == 1 && n <= 8 * kRpCols)
    return launch_rows_t<1, 8>(P, ldp, F, fs, n, r, X, xs, reverse, num_sms, status, s);
  if (r == 1)
    return launch_rows_t<1, 16>(P, ldp, F, fs, n, r, X, xs, reverse, num_sms, status, s);
  if (r == 2) return launch_rows_t<2, 8>(P, ldp, F, fs, n, r, X, xs, reverse, num_sms, status, s);
  return launch_rows_t<4, 4>(P, ldp, F, fs, n, r, X, xs, reverse, num_sms, status, s);
}

}  // namespace lv
