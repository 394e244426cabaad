// Internal declarations shared by the LINVIEW translation units (kernels and
// the C-ABI/engine).  Not part of the public ABI.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace lv {

// Launch ``k`` with programmatic stream serialisation (the kernel calls
// griddep_wait() before it reads what earlier kernels of the stream wrote).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

// return a failed launch's error from a launcher
#define LV_LAUNCH(expr)                    \
  do {                                     \
    const cudaError_t e_ = (expr);         \
    if (e_ != cudaSuccess) return e_;      \
  } while (0)

constexpr int kThreads = 256;   // threads per pass CTA
constexpr int kBatch = 8;       // rows per pipeline stage = TMA box height = warps per CTA
constexpr int kStages = 4;      // TMA ring depth (generic passes)
constexpr int kStagesWs = 6;    // TMA ring depth of the decoupled-ring FP32 passes
constexpr int kBoxBytes = 1024; // bytes per TMA box row (256 floats / 128 doubles)
constexpr int kMaxAsmR = 64;    // widest factor block U_h of one assembly (= the widest Gram block)
constexpr int kMaxFusedR = 8;   // widest factor block of the fused products pass
// Widest factor block of an FP32 products-only pass.  Wider levels run on the tensor-core
// products pass.  At 9 - 16 columns it would take 3 - 5 % off an update from n = 3500 on (A^16
// rank 4 at n = 4096 259 -> 253 us, n = 8192 812 -> 776, with sums 1146 -> 1126), but its split
// TF32 holds less of a product than FP32 FMAs: where the update makes up most of the view, the
// error against FP64 was 1.03e-6 against 9.7e-7 (A^8, n = 3500, rank 3) and 8.4e-7 against
// 7.4e-7 (A^4, rank 8).
constexpr int kMaxProductR = 16;
constexpr int kMaxUpdateR = 32;   // widest factor block of one update pass (shared-memory
                                  // broadcasts of the factor rows bound wider blocks)

// Pass modes: which of X = P Xf, Y = P^T Yf and P += Uu Wu^T a launch does.
enum PassMode : int { kModeXYU = 7, kModeXY = 3, kModeXU = 5, kModeX = 1, kModeY = 2 };
constexpr int kMaxColSumR = 32;  // widest factor block of an FP32 column-sums-only pass (Y)

// Everything a view pass needs.  Factors are column-major with column
// stride ``fs`` (elements); the partial-sum arrays are [block][column][row]
// with column stride ``part_cs`` and block strides ``xp_s`` / ``yp_q``.
struct PassParams {
  void* P;            // view, row-major
  int64_t ldp;        // leading dimension of P (elements)
  int n;              // P is n x n
  const void* Xf;     // X factor (n x r) or null
  const void* Yf;     // Y factor (n x r) or null
  const void* Uu;     // update left factor (n x r) or null
  const void* Wu;     // update right factor (n x r) or null
  int64_t fs;         // factor column stride
  int r;              // valid factor columns (<= template width)
  void* Xpart;        // [gC][r][part_cs] row-sum partials (pre-offset to the column block)
  void* Ypart;        // [gR][r][part_cs] column-sum partials
  int64_t part_cs;
  int64_t xp_s;
  int64_t yp_q;
  int gC, gR;         // column strips x row ranges; grid = gC * gR
  int rows_per_cta;   // multiple of kBatch (FP64 also 2 or 4)
  unsigned* status;   // device status word
  double* Cpart;      // fused XYU pass: per-row-range V^T U partials [gR][r*r] (or null)
  int suffix_rin;     // update pass: >0 applies block suffix sums (block width) to Wu
  int tma_store;      // FP32 passes may store updated tiles with TMA: the tensor map's
                      // row extent is a multiple of 16 bytes (a TMA store writes whole
                      // 16-byte units, so a row ending inside one would overwrite the
                      // elements past the view, e.g. a caller's padding)
  int reverse;        // FP32 passes: each CTA visits its row batches last to first.
                      // Alternating it over consecutive passes on one view makes a
                      // pass start on the rows the previous one read last, which are
                      // still in L2 (the FP64 pass ignores it)
};

// Host: grid geometry for a pass over an n x n view.
struct PassGeom {
  int strip, gC, gR, rows_per_cta;
};
PassGeom fused_geom(int elem_bytes, int n, int num_sms);
// beside: the pass runs next to another one (on a side stream)
PassGeom update_geom(int elem_bytes, int R, int n, int num_sms, bool beside = false);

// Host: 2-D tensor map over a row-major matrix (rows x cols, ld elements),
// box = (kBoxBytes / elem_bytes) columns x kBatch rows.
bool make_tmap(CUtensorMap* out, const void* base, int elem_bytes, int64_t cols, int64_t rows,
               int64_t ld);

// Host: FP32 tensor map with 32-column x box_rows boxes and 128-byte swizzle
// (operand and tile layout of the tensor-core update pass).
bool make_tmap_sw128(CUtensorMap* out, const void* base, int64_t cols, int64_t rows, int64_t ld,
                     int box_rows);
// Floats of the split-factor scratch of the tensor-core update pass (A_cat
// then B_cat, n x 128 each).
int64_t tc_split_floats(int64_t n);
constexpr int kMaxTcR = 64;  // widest factor block of one tensor-core update pass
constexpr int kTpMaxParts = 8;  // K parts (partial sums) of a tensor-core products pass
// Tensor-core products pass (FP32, 1 <= r <= 64): transpose = false: the
// partial sums of X = P F over column ranges of P; true: of Y = P^T F over
// row ranges; ``parts`` = tp_parts(n, num_sms) partial sets, every one
// written.  Partial q, factor column c, output row i lands at
// out[q ps + c cs + i].  F column-major (column stride fs, a multiple of 64,
// >= n); Fsplit is scratch of 128 x fs floats (the split factor; F null: it is there
// already, see launch_level_split).
cudaError_t launch_tc_products(bool transpose, const float* P, int64_t ldp, const float* F,
                               int64_t fs, float* Fsplit, int n, int r, float* out, int64_t ps,
                               int64_t cs, int parts, int num_sms, unsigned* status,
                               cudaStream_t s);
// The splits of a level's factors in one launch: U and V for the products passes (FU, FV,
// 128 x fs floats each) and both for the update P += U V^T (Acat, Bcat).
cudaError_t launch_level_split(const float* U, const float* V, int64_t fs, int n, int r, float* FU,
                               float* FV, float* Acat, float* Bcat, cudaStream_t s);
// whether a products pass over an n x n view has fewer CTAs than the GPU has SMs
bool tp_leaves_sms(int n, int num_sms);
// partial sets the products pass writes for an n x n view (<= kTpMaxParts)
int tp_parts(int n, int num_sms);
// Tensor-core update pass P += U W^T (FP32 view, 17 <= r <= 64 factor
// columns, split TF32): splits U, W into the scratch (presplit: already there), then one persistent
// launch over 128 x 64 tiles.  tmP:
// make_tmap_sw128 over the view P (box rows 128, row stride ldp); tmA / tmB:
// over A_cat (128 columns, box rows 128) / B_cat (128 columns, box rows 32).
cudaError_t launch_tc_update(const CUtensorMap& tmP, const CUtensorMap& tmA,
                             const CUtensorMap& tmB, float* P, int64_t ldp, float* Acat,
                             float* Bcat, const float* U, const float* W, int64_t fs, int n, int r,
                             int num_sms, unsigned* status, cudaStream_t s,
                             bool presplit = false);

// Own dense GEMMs (lv_gemm.cu).
// A split operand of the tensor-core GEMM: element (i, k) of op(X) at X[i * rs +
// k * cs] (rs or cs == 1), its split blocks in ``buf`` (tc_operand_floats(rows,
// K) floats, 16-byte aligned; FP16 halves take half of it) and in ``words`` (tc_split_words(rows,
// K), 16-byte aligned) the buffer's format and the factors of its runs.  X stays
// readable for as long as products use the split: a product that has to fall back
// to TF32 splits it again.
struct TcOperand {
  const float* X;
  int64_t rs, cs;
  int rows, K;
  float* buf;
  unsigned* words;
};
int64_t tc_operand_floats(int64_t rows, int64_t K);
int64_t tc_split_words(int64_t rows, int64_t K);
// floats of ``work`` below that let every product with up to these sizes cut tiles
int64_t tc_work_floats(int64_t a_rows, int64_t b_rows, int64_t K, int num_sms);
// Split a and b (either may be null).  ``flag`` (one word, zeroed by the caller
// before the first split of a scratch) collects what FP16 halves would lose of either
// operand; its bits stay set, so once a product takes TF32 all later ones on the scratch do.
cudaError_t launch_tc_split(const TcOperand* a, const TcOperand* b, unsigned* flag,
                            cudaStream_t s);
// D (M x N, row-major, ldd) = alpha A B^T + beta C on the tensor cores (split
// FP16 or TF32, FP32 accumulation) of split operands with M and N rows.  C may
// alias D (beta == 0 ignores it).  ``work`` (work_floats floats, 16-byte aligned, may
// be null): room for the pieces of tiles that several CTA pairs share along K
// (summed in a fixed order).  ``reverse`` visits K from its end: a product that
// follows another one with the same A then starts on the part still in L2.
// ``next``: D's columns as a split operand (rows N, K = M; its buffer may be b's): they
// are split by the kernel that adds up the cut tiles when every tile is cut and one
// tile column holds D; *next_split says whether they were, and ``next_flag`` (another word
// than ``flag``, with its bits of a) is then the flag of the product that reads them.
cudaError_t launch_tc_gemm(const TcOperand& a, const TcOperand& b, unsigned* flag, float* D,
                           int64_t ldd, const float* C, int64_t ldc, float alpha, float beta,
                           int num_sms, unsigned* status, cudaStream_t s, float* work = nullptr,
                           int64_t work_floats = 0, bool reverse = false,
                           const TcOperand* next = nullptr, bool* next_split = nullptr,
                           unsigned* next_flag = nullptr);
// C (M x N) = alpha A B + beta C on the CUDA cores, A(m, k) = A[m a_rs + k a_cs],
// B(k, n) = B[k b_rs + n b_cs], C(m, n) = C[m c_rs + n c_cs]; long inner
// dimensions are split over ``work`` (work_elems elements, may be null) and
// the partials summed in a fixed order.
template <typename T>
cudaError_t launch_gemm_simt(int M, int N, int K, T alpha, const T* A, int64_t a_rs, int64_t a_cs,
                             const T* B, int64_t b_rs, int64_t b_cs, T beta, T* C, int64_t c_rs,
                             int64_t c_cs, T* work, int64_t work_elems, int num_sms,
                             cudaStream_t s);

// Launchers (return cudaGetLastError()).  R is the runtime factor width,
// bucketed internally to a compiled width.  The passes are launched with
// programmatic stream serialisation, and the FP32 passes request their first
// view tiles before waiting on the kernel before them: that kernel must not
// write the view.  An update launched right after another pass that wrote
// the same view (the second block of a wide update) takes programmatic =
// false: a plain launch, which starts only once that kernel has completed.
template <typename T>
cudaError_t launch_fused(const PassParams& p, const CUtensorMap& tm, int R, int mode,
                         cudaStream_t s);
template <typename T>
cudaError_t launch_update(const PassParams& p, const CUtensorMap& tm, int R, cudaStream_t s,
                          bool programmatic = true);

// X (n x r, column stride xs) = P F for an n x n FP32 view and a few columns (lv_rows.cu),
// without partial sums.  As for the passes, the kernel launched before must not write P.
bool row_products_fit(const void* P, int64_t ldp, int n, int r);
cudaError_t launch_row_products(const float* P, int64_t ldp, const float* F, int64_t fs, int n,
                                int r, float* X, int64_t xs, bool reverse, int num_sms,
                                unsigned* status, cudaStream_t s);

// Factor cores and assembly (lv_core.cu).
// C (r x r, FP64, row-major) = V^T U over n rows; deterministic two-level
// reduction using Cpart (grid x r*r doubles) and a ticket counter.  FP32
// programs may also take C as double-float pairs (Cdf, r x r float2).
template <typename T>
cudaError_t launch_gram(const T* V, const T* U, int64_t fs, int n, int r, double* Cpart,
                        unsigned* ticket, double* C, unsigned* status, cudaStream_t s,
                        float2* Cdf = nullptr);
int gram_grid(int n);
// C (rx x rv, FP64, row-major) = X^T V over n rows (FP32 factors, double-float
// sums; rv <= 64, any rx in blocks of 64), no status check.
cudaError_t launch_cross_gram(const float* X, const float* V, int64_t fs, int n, int rx, int rv,
                              double* Cpart, double* C, cudaStream_t s);

struct AssembleParams {
  int n, r_h;             // rows, current factor width
  int r_out;              // columns of X_h / Y_h to assemble (0 = r_h)
  int64_t fs;             // arena column stride
  const void* Xpart; int gC; int64_t xp_s;   // row-sum partials of P_h U_h
  const void* Ypart; int gR; int64_t yp_q;   // column-sum partials of P_h^T V_h (or null)
  int64_t part_cs;
  const double* C;        // r_h x r_h = V_h^T U_h, summed over nC partial blocks (the first
                          // r_out columns are used)
  int nC;                 // number of [r_h*r_h] partial blocks in C (1 = already reduced)
  const void* Uh;         // U_h (n x r_h)
  void* Unew;             // destination of X_h + U_h C_h (n x r_h), = U arena + r_h columns
  void* Ynew;             // destination of Y_h (n x r_h), = V arena left of V_h
  unsigned* status;       // device status word: a non-finite C_h entry latches
                          // kStatusNonFinite (or null)
};
template <typename T>
cudaError_t launch_assemble(const AssembleParams& a, cudaStream_t s);

// One bounded wait that always expires (diagnostic; see lv_core.cu).
cudaError_t launch_bounded_wait_probe(uint64_t limit_ns, unsigned* status,
                                      unsigned long long* waited_ns, cudaStream_t s);

// Suffix block sums: W[:, a-block] = sum_{b >= a} V[:, b-block] (blocks of r_in).
template <typename T>
cudaError_t launch_suffix_sums(const T* V, T* W, int64_t fs, int n, int width, int r_in,
                               cudaStream_t s);

// Copy a row-major user matrix (rows x cols, ld) into column-major storage
// (column stride fs) -- factor ingest.
template <typename T>
cudaError_t launch_rm_to_cm(const T* src, int64_t ld, T* dst, int64_t fs, int rows, int cols,
                            cudaStream_t s);
// Ingest of an update in one launch: U (nu x cols, row-major) and V (nv x cols) into
// column-major storage; or e_row into du with a copy of v (may be null: du only) in dv.
template <typename T>
cudaError_t launch_ingest_pair(const T* U, int64_t ldu, T* du, int64_t fsu, int nu, const T* V,
                               int64_t ldv, T* dv, int64_t fsv, int nv, int cols, cudaStream_t s);
template <typename T>
cudaError_t launch_ingest_row(T* du, T* dv, const T* v, int n, int row, cudaStream_t s);

// Sum of column-major partial blocks: out[c][j] = sum_b part[b][c][j].
template <typename T>
cudaError_t launch_sum_partials(const T* part, int blocks, int64_t block_stride, int64_t cs,
                                int n, int r, T* out, int64_t out_cs, cudaStream_t s);

// Elementwise helpers.
// blk = ub + tmp - blk, or ub (tmp null); column-major n x r, column stride fs
template <typename T>
cudaError_t launch_s_block(T* blk, const T* ub, const T* tmp, int64_t fs, int n, int r,
                           cudaStream_t s);
// out = x + y, rows x ld elements each (views of one layout)
template <typename T>
cudaError_t launch_add_views(const T* x, const T* y, T* out, int64_t rows, int64_t ld,
                             cudaStream_t s);
template <typename T>
cudaError_t launch_axpy_rows(T* y, int64_t ldy, const T* x, int64_t ldx, T alpha, int rows,
                             int cols, cudaStream_t s);  // y += alpha x (row-major blocks)
template <typename T>
cudaError_t launch_scale_copy(T* y, int64_t ldy, const T* x, int64_t ldx, T alpha, int rows,
                              int cols, cudaStream_t s);  // y = alpha x
// Products of n x p panels with narrow factors (lv_panel.cu).
// M[((k - 1 - i) w + c) ldm + q] = sum_j A0[j lda0 + i p + q] F0[c fs + j] for
// i < k, c < w <= 64, q < p; optionally + sum_j A1[j lda1 + i p + q] (F1 - F0)[c fs +
// j] and + sum_{t < ny} Yc[t ldy + i p + q] S[t s_t + c s_c].  ``work`` holds
// ``work_elems`` elements, tdot_work_elems(sizeof(T), n, k p, w) for as many row blocks as fill the
// GPU; fewer elements mean fewer blocks, and less than one block's k p w is an error.
template <typename T>
struct TdotOp {
  const T* A0;
  int64_t lda0;
  const T* F0;
  int64_t fs;
  int n, p, k, w;
  T* M;
  int64_t ldm;
  T* work;
  int64_t work_elems;
  const T* A1 = nullptr;
  int64_t lda1 = 0;
  const T* F1 = nullptr;
  const T* Yc = nullptr;
  int64_t ldy = 0;
  int ny = 0;
  const double* S = nullptr;
  int64_t s_t = 0, s_c = 0;
};
int64_t tdot_work_elems(int elem_bytes, int n, int cols, int w, int num_sms);
template <typename T>
cudaError_t launch_tdot(const TdotOp<T>& o, int num_sms, cudaStream_t s);
// T_i(j, q) = T1[j ldT + (i - 1) p + q] += sum_{t < i r} K[t fs + j] M[((k - i) r + t) ldm
// + q] for i = 1 .. k (k = 1: one panel, rank r); accumulate = false overwrites.
// The staged factors must fit shared memory: outer_fits(k r).
template <typename T>
cudaError_t launch_outer(T* T1, int64_t ldT, const T* K, int64_t fs, const T* M, int64_t ldm, int n,
                         int p, int k, int r, bool accumulate, int num_sms, cudaStream_t s);
bool outer_fits(int kr, size_t elem_bytes);
// out(j, q) = sum_{i < k} A[j lda + i p + q], in order
template <typename T>
cudaError_t launch_panel_sum(const T* A, int64_t lda, T* out, int64_t ldo, int n, int p, int k,
                             cudaStream_t s);

// OLS pieces (lv_ols.cu).
// Row block exchange: U's column k + t = the old row rows[t] of X, X takes U's column t
// (the new row), Yr's row t = the row rows[t] of Y.
template <typename T>
cudaError_t launch_exchange_rows(T* X, int64_t ldx, const T* Y, int64_t ldy, const int64_t* rows,
                                 int k, int n, int p, T* U, int64_t fs, T* Yr, cudaStream_t s);
// Minv = (diag(+1 x kpos, -1 x (kk - kpos)) + S)^{-1}, kk <= 64: FP64
// programs in FP64 (S and Minv kk x kk doubles); FP32 programs in
// double-float on the FP32 pipe (S and Minv kk x kk float2 pairs).
cudaError_t launch_core_inverse(const double* S, int kk, int kpos, double* Minv, unsigned* status,
                                cudaStream_t s);
cudaError_t launch_core_inverse_df(const float2* S, int kk, int kpos, float2* Minv,
                                   unsigned* status, cudaStream_t s);
// Wu = -G Minv (FP64 core for double views, double-float core for float views)
cudaError_t launch_wu(const double* G, int64_t fs, int n, int kk, const double* Minv, double* Wu,
                      cudaStream_t s);
// (Acat, Bcat: also the split of G and Wu for launch_tc_update's presplit form; may be null)
cudaError_t launch_wu(const float* G, int64_t fs, int n, int kk, const float2* Minv, float* Wu,
                      float* Acat, float* Bcat, cudaStream_t s);
// Newton-Schulz correction of FP32 OLS programs: Z = X^T X as double-float
// pairs (Zh, Zl; n x n, row-major ldz, a multiple of 64 with zero padding)
cudaError_t launch_z_from_lower(const double* L, int64_t ldl, int n, float* Zh, float* Zl,
                                int64_t ldz, cudaStream_t s);
// Z += Hp Hp^T - Hm Hm^T (cnt history columns each, column stride fs >= ldz)
cudaError_t launch_z_flush(float* Zh, float* Zl, int64_t ldz, const float* Hp, const float* Hm,
                           int64_t fs, int n, int cnt, cudaStream_t s);
// R = D - Z B (B n x nb; D the identity if Dh is null, else the pairs Dh + Dl;
// double-float sums, rounded to FP32)
cudaError_t launch_ns_residual(const float* Zh, const float* Zl, int64_t ldz, const float* B,
                               int64_t ldb, int nb, const float* Dh, const float* Dl, int64_t ldd,
                               float* R, int64_t ldr, int n, cudaStream_t s);
// lo = src - (float)src, rounded to FP32 (src FP64 row-major)
cudaError_t launch_low_half(const double* src, int64_t lds, float* lo, int64_t ldl, int rows,
                            int cols, cudaStream_t s);
template <typename T>
cudaError_t launch_xty_update(T* xty, int64_t ld, T* xtyc, int64_t fs, const T* U, int n, int p,
                              int k, const T* Yr, cudaStream_t s,
                              T* xtyl = nullptr);
template <typename T>
cudaError_t launch_to_double(const T* src, int64_t lds, double* dst, int64_t ldd, int rows,
                             int cols, cudaStream_t s);
template <typename T>
cudaError_t launch_sym_lower_to_full(const double* Lcm, int64_t ldl, int n, T* dst, int64_t ldd,
                                     double* full, int64_t ldf, cudaStream_t s);
template <typename T>
cudaError_t launch_from_double(const double* src, int64_t lds, T* dst, int64_t ldd, int rows,
                               int cols, T* cm, int64_t cfs, cudaStream_t s);

}  // namespace lv
