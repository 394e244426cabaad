// Products of the general form's n x p panels with narrow factors (Appendix B):
//
//   tdot:   M = T^T V       (columns x w, w <= 64; one read of the panel)
//   outer:  T += K M^T      (rank w per view, in place)
//
// for the T panel of the linear model (all views T_0 .. T_{k-1}, T_1 .. T_k at
// once) and for single panels (the exponential and skip models, B).  Both are
// bound by reading (and writing) the panel, whose rows are row-major, so a
// warp takes 128 adjacent columns of a row.
#include <cuda_runtime.h>

#include "lv_device.cuh"
#include "lv_internal.h"

namespace lv {

namespace {

// ---------------------------------------------------------------- tdot
// part[b][c][col] = sum over the rows j of block b of
//   A0[j lda0 + col] F0[c fs + j]  (+ A1[j lda1 + col] (F1 - F0)[c fs + j]).
// A CTA takes 128 columns and ``rows`` rows; its 8 warps are W/8 factor groups
// of 8 columns times 64/W row groups, a lane holds 4 columns x 8 factors, so a
// panel row costs one 128-bit load for 32 FMAs and is fetched by W/8 warps (from
// L1 after the first).  The row groups are added in a fixed order in shared
// memory.  Eight rows' loads are in flight per warp.
// n = 4096, p = 1024, up to 8 factors: 12 + 3 us with the sums of the row blocks
// (16.8 MB; floor 2.5 us), 16 factors of two panels at once 25 + 5 us; each such
// product took 32 + 4 us as a 64 x 64-tile GEMM that padded the factors to its
// tile width.
constexpr int kTdCols = 128;   // columns per CTA
constexpr int kTdChunk = 64;   // rows of factors staged at once
constexpr int kTdMaxBlocks = 64;

struct TdotArgs {
  const void *A0, *F0, *A1, *F1;
  int64_t lda0, lda1, fs;
  int n, cols, w, rows;
  void* part;
};

template <typename T, int W>
__global__ void __launch_bounds__(256) tdot_kernel(const TdotArgs a) {
  constexpr int WG = W / 8, RG = 8 / WG;
  constexpr int LDF = W + 4;
  constexpr int kRed = RG > 1 ? (RG / 2) * WG * 32 * 32 : 0;
  constexpr int kSm = kTdChunk * LDF > kRed ? kTdChunk * LDF : kRed;
  __shared__ __align__(16) T sm[kSm];
  griddep_wait();
  griddep_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wg = warp % WG, rg = warp / WG;
  const int q = blockIdx.x * kTdCols + 4 * lane;
  const int j0 = blockIdx.y * a.rows;
  const int nr = min(a.rows, a.n - j0);
  T acc[4][8];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[k][c] = T(0);
  for (int src = 0; src < (a.A1 ? 2 : 1); ++src) {
    const T* A = static_cast<const T*>(src ? a.A1 : a.A0);
    const int64_t lda = src ? a.lda1 : a.lda0;
    const T* F = static_cast<const T*>(src ? a.F1 : a.F0);
    const T* Fm = src ? static_cast<const T*>(a.F0) : nullptr;
    // 128-bit loads need every row of this lane's columns on a 16-byte boundary
    const bool vec = (q + 4 <= a.cols) && (lda % 4 == 0) &&
                     (reinterpret_cast<uintptr_t>(A + q) % 16 == 0);
    for (int c0 = 0; c0 < nr; c0 += kTdChunk) {
      __syncthreads();
      for (int e = threadIdx.x; e < kTdChunk * W; e += 256) {
        const int jr = e % kTdChunk, c = e / kTdChunk;
        T v = T(0);
        if (c < a.w && c0 + jr < nr) {
          const int64_t g = (int64_t)c * a.fs + j0 + c0 + jr;
          v = F[g];
          if (Fm) v -= Fm[g];
        }
        sm[jr * LDF + c] = v;
      }
      __syncthreads();
      const int nc = min(kTdChunk, nr - c0);
      const T* base = A + (int64_t)(j0 + c0) * lda + q;
      for (int b = rg; b < nc; b += 8 * RG) {
        T t[8][4];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int jr = b + u * RG;
          if (jr < nc && vec) {
            if constexpr (sizeof(T) == 4) {
              const float4 x = *reinterpret_cast<const float4*>(base + (int64_t)jr * lda);
              t[u][0] = x.x; t[u][1] = x.y; t[u][2] = x.z; t[u][3] = x.w;
            } else {
              const double2 x = *reinterpret_cast<const double2*>(base + (int64_t)jr * lda);
              const double2 y = *reinterpret_cast<const double2*>(base + (int64_t)jr * lda + 2);
              t[u][0] = x.x; t[u][1] = x.y; t[u][2] = y.x; t[u][3] = y.y;
            }
          } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
              t[u][k] = (jr < nc && q + k < a.cols) ? base[(int64_t)jr * lda + k] : T(0);
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int jr = b + u * RG;
          if (jr < nc) {
            const T* f = sm + jr * LDF + wg * 8;
            T fv[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) fv[c] = f[c];
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
              for (int c = 0; c < 8; ++c) acc[k][c] = fma(t[u][k], fv[c], acc[k][c]);
          }
        }
      }
    }
  }
  // the upper half of the row groups hands its sums to the lower half
#pragma unroll
  for (int half = RG / 2; half >= 1; half /= 2) {
    __syncthreads();
    T* red = sm + ((rg % (half > 0 ? half : 1)) * WG + wg) * 1024 + lane;
    if (rg >= half && rg < 2 * half) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int c = 0; c < 8; ++c) red[(k * 8 + c) * 32] = acc[k][c];
    }
    __syncthreads();
    if (rg < half) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[k][c] += red[(k * 8 + c) * 32];
    }
  }
  if (rg != 0) return;
  T* out = static_cast<T*>(a.part) + (int64_t)blockIdx.y * a.w * a.cols;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    if (wg * 8 + c >= a.w) break;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (q + k < a.cols) out[(int64_t)(wg * 8 + c) * a.cols + q + k] = acc[k][c];
  }
}

// M[((k - 1 - i) w + c) ldm + q] = sum_b part[b][c][i p + q] (+ sum_t Yc[t ldy +
// q] S[t s_t + c s_c]), k panels of p columns.  Threads (x, y): 32 columns, the
// partials y, y + 8, ... each; FP32 sums as TwoSum pairs (about 48 bits).
struct TdotSumArgs {
  const void* part;
  int blocks, cols, p, k, w;
  void* M;
  int64_t ldm;
  const void* Yc;
  int64_t ldy;
  int ny;
  const double* S;
  int64_t s_t, s_c;
};

template <typename T>
__device__ __forceinline__ void pair_add(T& hi, T& lo, T x) {
  if constexpr (sizeof(T) == 4) {
    const float t = __fadd_rn(hi, x);
    const float z = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(x, z)));
    hi = t;
  } else {
    hi += x;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) tdot_sum_kernel(const TdotSumArgs a) {
  __shared__ T sh[8][32], sl[8][32];
  griddep_wait();
  griddep_launch_dependents();
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int col = blockIdx.x * 32 + x, c = blockIdx.y;
  T hi = T(0), lo = T(0);
  if (col < a.cols) {
    const T* src = static_cast<const T*>(a.part) + (int64_t)c * a.cols + col;
    const int64_t bs = (int64_t)a.w * a.cols;
    T v[kTdMaxBlocks / 8];
#pragma unroll
    for (int u = 0; u < kTdMaxBlocks / 8; ++u)
      v[u] = (y + 8 * u < a.blocks) ? src[(y + 8 * u) * bs] : T(0);
#pragma unroll
    for (int u = 0; u < kTdMaxBlocks / 8; ++u) pair_add(hi, lo, v[u]);
    const T* yc = static_cast<const T*>(a.Yc);
    for (int t = y; t < a.ny; t += 8)
      pair_add(hi, lo, yc[(int64_t)t * a.ldy + col] * (T)a.S[t * a.s_t + c * a.s_c]);
  }
  sh[y][x] = hi;
  sl[y][x] = lo;
  __syncthreads();
  if (y != 0 || col >= a.cols) return;
#pragma unroll
  for (int u = 1; u < 8; ++u) {
    pair_add(hi, lo, sh[u][x]);
    lo += sl[u][x];
  }
  const int i = col / a.p, q = col - i * a.p;
  static_cast<T*>(a.M)[((int64_t)(a.k - 1 - i) * a.w + c) * a.ldm + q] = hi + lo;
}

// ---------------------------------------------------------------- outer
// Views T_i, i = 1 .. k, side by side (T_i's column q at T1[j ldT + (i - 1) p + q]):
//   T_i(j, q) (+)= sum_{t < i r} K[t fs + j] M[((k - i) r + t) ldm + q]
// (App. B, linear model: view i takes the first i Krylov blocks and the i
// newest M blocks; k = 1 is a plain rank-r update of one panel).  A CTA takes
// 16 RPT rows and 64 columns of the views blockIdx.z + 1, + gridDim.z, ...; the
// rows of K and the columns of M that it needs are staged once in shared
// memory, and a thread owns RPT rows x 4 columns, so that one step of t is two
// 128-bit shared loads for 16 FMAs (RPT = 4; with one row per thread the
// shared-memory pipe bound it: n = 8192, p = 64, k = 16, r = 2 took 42 us,
// 20 us now).  RPT = 1 serves factors too wide for the 64-row stage.
// The next view's entries are loaded before this one's products.  Sums over t
// in increasing order, in T.
template <typename T, int RPT>
__global__ void __launch_bounds__(256)
    outer_kernel(T* T1, int64_t ldT, const T* __restrict__ K, int64_t fs, const T* __restrict__ M,
                 int64_t ldm, int n, int p, int k, int r, int accumulate) {
  constexpr int ROWS = 16 * RPT, COLS = 64;
  extern __shared__ __align__(16) unsigned char outer_sm[];
  const int KR = k * r;
  T* Ks = reinterpret_cast<T*>(outer_sm);  // [KR][ROWS]
  T* Ms = Ks + KR * ROWS;                  // [KR][COLS]
  griddep_wait();
  griddep_launch_dependents();
  const int j0 = blockIdx.x * ROWS, q0 = blockIdx.y * COLS;
  for (int e = threadIdx.x; e < KR * ROWS; e += 256) {
    const int jr = e % ROWS, t = e / ROWS;
    Ks[e] = (j0 + jr < n) ? K[(int64_t)t * fs + j0 + jr] : T(0);
  }
  for (int e = threadIdx.x; e < KR * COLS; e += 256) {
    const int q = e % COLS, t = e / COLS;
    Ms[e] = (q0 + q < p) ? M[(int64_t)t * ldm + q0 + q] : T(0);
  }
  __syncthreads();
  const int jr = (threadIdx.x / 16) * RPT, qa = 4 * (threadIdx.x % 16);
  const int nq = min(4, p - q0 - qa), nj = min(RPT, n - j0 - jr);
  if (nq <= 0 || nj <= 0) return;
  T* base = T1 + (int64_t)(j0 + jr) * ldT + q0 + qa;
  auto load = [&](int i, T (&v)[RPT][4]) {
    T* src = base + (int64_t)(i - 1) * p;
    const bool vec = sizeof(T) == 4 && nq == 4 && ldT % 4 == 0 &&
                     reinterpret_cast<uintptr_t>(src) % 16 == 0;
#pragma unroll
    for (int a = 0; a < RPT; ++a) {
      if (a < nj && vec) {
        const float4 x = *reinterpret_cast<const float4*>(src + (int64_t)a * ldT);
        v[a][0] = x.x; v[a][1] = x.y; v[a][2] = x.z; v[a][3] = x.w;
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) v[a][c] = (a < nj && c < nq) ? src[(int64_t)a * ldT + c] : T(0);
      }
    }
  };
  T tv[RPT][4];
#pragma unroll
  for (int a = 0; a < RPT; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) tv[a][c] = T(0);
  const int step = gridDim.z;
  int i = blockIdx.z + 1;
  if (i <= k && accumulate) load(i, tv);
  for (; i <= k; i += step) {
    T nx[RPT][4];
#pragma unroll
    for (int a = 0; a < RPT; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) nx[a][c] = T(0);
    if (i + step <= k && accumulate) load(i + step, nx);
    T acc[RPT][4];
#pragma unroll
    for (int a = 0; a < RPT; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][c] = T(0);
    const T* kp = Ks + jr;
    const T* mp = Ms + (int64_t)(k - i) * r * COLS + qa;
#pragma unroll 4
    for (int t = 0; t < i * r; ++t) {
      T kv[RPT], mv[4];
#pragma unroll
      for (int a = 0; a < RPT; ++a) kv[a] = kp[t * ROWS + a];
#pragma unroll
      for (int c = 0; c < 4; ++c) mv[c] = mp[t * COLS + c];
#pragma unroll
      for (int a = 0; a < RPT; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = fma(kv[a], mv[c], acc[a][c]);
    }
    T* dst = base + (int64_t)(i - 1) * p;
    const bool vec = sizeof(T) == 4 && nq == 4 && ldT % 4 == 0 &&
                     reinterpret_cast<uintptr_t>(dst) % 16 == 0;
#pragma unroll
    for (int a = 0; a < RPT; ++a) {
      if (a < nj && vec) {
        *reinterpret_cast<float4*>(dst + (int64_t)a * ldT) =
            make_float4(tv[a][0] + acc[a][0], tv[a][1] + acc[a][1], tv[a][2] + acc[a][2],
                        tv[a][3] + acc[a][3]);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (a < nj && c < nq) dst[(int64_t)a * ldT + c] = tv[a][c] + acc[a][c];
      }
    }
#pragma unroll
    for (int a = 0; a < RPT; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) tv[a][c] = nx[a][c];
  }
}

// out(j, q) = sum_i A[j lda + i p + q], i = 0 .. k - 1 in order: the k panels of a row
// are read once (dB = G_1 + .. + G_k took k launches that re-read the sum: 15 x 4.5
// us at n = 8192, p = 64, k = 16).
template <typename T>
__global__ void __launch_bounds__(256) panel_sum_kernel(const T* __restrict__ A, int64_t lda, T* out,
                                                        int64_t ldo, int n, int p, int k) {
  griddep_wait();
  griddep_launch_dependents();
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (idx >= (int64_t)n * p) return;
  int j, q;
  split_index(idx, p, j, q);
  const T* src = A + (int64_t)j * lda + q;
  T acc = src[0];
  int i = 1;
  for (; i + 8 <= k; i += 8) {  // eight loads in flight, added in order
    T v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = src[(int64_t)(i + u) * p];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc += v[u];
  }
  for (; i < k; ++i) acc += src[(int64_t)i * p];
  out[(int64_t)j * ldo + q] = acc;
}

// largest dynamic shared memory a block of this device may opt in to
int smem_optin_max() {
  static const int v = [] {
    int dev = 0, b = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&b, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
      (void)cudaGetLastError();
      return 49152;
    }
    return b;
  }();
  return v;
}

size_t outer_smem(int rpt, int kr, size_t elem) { return elem * (size_t)(16 * rpt + 64) * kr; }

template <typename T, int RPT>
cudaError_t launch_outer_t(T* T1, int64_t ldT, const T* K, int64_t fs, const T* M, int64_t ldm,
                           int n, int p, int k, int r, bool accumulate, int num_sms,
                           cudaStream_t s) {
  const size_t smem = outer_smem(RPT, k * r, sizeof(T));
  if (smem > 49152) {  // opt in once, to the device's limit
    static const cudaError_t configured = cudaFuncSetAttribute(
        outer_kernel<T, RPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin_max());
    if (configured != cudaSuccess) return configured;
  }
  const unsigned gx = (unsigned)((n + 16 * RPT - 1) / (16 * RPT)), gy = (unsigned)((p + 63) / 64);
  // few tiles: the views are spread over CTAs as well (about two CTAs per SM)
  unsigned gz = 1;
  while (gz < (unsigned)k && gz < 64 && (int64_t)gx * gy * gz < 2 * num_sms) gz *= 2;
  if (gz > (unsigned)k) gz = (unsigned)k;
  return launch_pdl(outer_kernel<T, RPT>, dim3(gx, gy, gz), 256, smem, s, T1, ldT, K, fs, M, ldm, n,
                    p, k, r, accumulate ? 1 : 0);
}

// row blocks of a tdot over ``cols`` columns.  FP32: about two CTAs per SM (two waves
// of one would leave the second one nearly empty), at least 64 rows each.  FP64 is bound by
// its FMAs, two a clock and SM, so the blocks are those (of 16 rows and more, and some 24 rows'
// time to start one) that leave the busiest SM the fewest rows: linear iterations of 8 steps
// against FP32's rule at n = 300, p = 3, rank 8 114 -> 104 us, n = 777, p = 64 327 -> 321,
// n = 1500, p = 129, rank 1 198 -> 186 (187 before these kernels).
int tdot_blocks(int elem_bytes, int n, int cols, int num_sms) {
  const int cb = (cols + kTdCols - 1) / kTdCols;
  if (elem_bytes == 8) {
    int best = 1;
    int64_t least = INT64_MAX;
    for (int nb = 1; nb <= kTdMaxBlocks && 16 * nb < n + 16; ++nb) {
      const int rows = ((n + nb - 1) / nb + 7) / 8 * 8;
      const int64_t ctas = (int64_t)cb * ((n + rows - 1) / rows);
      const int64_t busiest = (ctas + num_sms - 1) / num_sms * (rows + 24);
      if (busiest < least) {
        least = busiest;
        best = nb;
      }
    }
    return best;
  }
  int nb = 2 * num_sms / cb;
  if (nb > (n + 63) / 64) nb = (n + 63) / 64;
  if (nb > kTdMaxBlocks) nb = kTdMaxBlocks;
  return nb < 1 ? 1 : nb;
}

}  // namespace

int64_t tdot_work_elems(int elem_bytes, int n, int cols, int w, int num_sms) {
  return (int64_t)tdot_blocks(elem_bytes, n, cols, num_sms) * cols * w;
}

template <typename T>
cudaError_t launch_tdot(const TdotOp<T>& o, int num_sms, cudaStream_t s) {
  const int cols = o.k * o.p;
  if (o.n < 1 || cols < 1 || o.w < 1 || o.w > 64) return cudaErrorInvalidValue;
  // no more row blocks than the work space has room for
  const int64_t room = o.work_elems / ((int64_t)cols * o.w);
  if (room < 1) return cudaErrorInvalidValue;
  int nb0 = tdot_blocks(sizeof(T), o.n, cols, num_sms);
  if (nb0 > room) nb0 = (int)room;
  const int rows = ((o.n + nb0 - 1) / nb0 + 7) / 8 * 8;
  const int nb = (o.n + rows - 1) / rows;
  TdotArgs a{o.A0, o.F0, o.A1, o.F1, o.lda0, o.lda1, o.fs, o.n, cols, o.w, rows, o.work};
  const dim3 grid((unsigned)((cols + kTdCols - 1) / kTdCols), (unsigned)nb);
  auto* kern = o.w <= 8    ? tdot_kernel<T, 8>
               : o.w <= 16 ? tdot_kernel<T, 16>
               : o.w <= 32 ? tdot_kernel<T, 32>
                           : tdot_kernel<T, 64>;
  cudaError_t e = launch_pdl(kern, grid, 256, 0, s, a);
  if (e != cudaSuccess) return e;
  TdotSumArgs b{o.work, nb, cols, o.p, o.k, o.w, o.M, o.ldm, o.Yc, o.ldy, o.ny, o.S, o.s_t, o.s_c};
  return launch_pdl(tdot_sum_kernel<T>, dim3((unsigned)((cols + 31) / 32), (unsigned)o.w), 256, 0,
                    s, b);
}

bool outer_fits(int kr, size_t elem_bytes) {
  return outer_smem(1, kr, elem_bytes) <= (size_t)smem_optin_max();
}

template <typename T>
cudaError_t launch_outer(T* T1, int64_t ldT, const T* K, int64_t fs, const T* M, int64_t ldm, int n,
                         int p, int k, int r, bool accumulate, int num_sms, cudaStream_t s) {
  if (n <= 0 || p <= 0 || k < 1 || r < 1) return cudaSuccess;
  if (!outer_fits(k * r, sizeof(T))) return cudaErrorInvalidValue;
  // FP64 is bound by its FMAs, not by shared memory: tiles of 16 rows while those of 64 are few,
  // which spread more evenly (8 steps, rank 8, p = 129: n = 300 161 -> 145 us, n = 777 415 -> 384
  // (381 before these kernels), but n = 1000, 48 tiles of 64 rows, 411 -> 442)
  const int64_t tiles = (int64_t)((n + 63) / 64) * ((p + 63) / 64);
  if (!(sizeof(T) == 8 && tiles < num_sms * 3 / 10) &&
      outer_smem(4, k * r, sizeof(T)) <= (size_t)smem_optin_max())
    return launch_outer_t<T, 4>(T1, ldT, K, fs, M, ldm, n, p, k, r, accumulate, num_sms, s);
  return launch_outer_t<T, 1>(T1, ldT, K, fs, M, ldm, n, p, k, r, accumulate, num_sms, s);
}

template <typename T>
cudaError_t launch_panel_sum(const T* A, int64_t lda, T* out, int64_t ldo, int n, int p, int k,
                             cudaStream_t s) {
  const int64_t tot = (int64_t)n * p;
  return launch_pdl(panel_sum_kernel<T>, dim3((unsigned)((tot + 255) / 256)), 256, 0, s, A, lda, out,
                    ldo, n, p, k);
}

#define LV_INST(T)                                                                               \
  template cudaError_t launch_tdot<T>(const TdotOp<T>&, int, cudaStream_t);                      \
  template cudaError_t launch_panel_sum<T>(const T*, int64_t, T*, int64_t, int, int, int,        \
                                           cudaStream_t);                                        \
  template cudaError_t launch_outer<T>(T*, int64_t, const T*, int64_t, const T*, int64_t, int,   \
                                       int, int, int, bool, int, cudaStream_t);
LV_INST(float)
LV_INST(double)

}  // namespace lv
