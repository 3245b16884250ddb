// Shared declarations of the library's translation units (internal; the public surface is include/ab.h).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stddef.h>

#include <utility>

#include "ab.h"

namespace ab {

typedef __nv_bfloat16 bf16;

#define AB_CUDA_OK(expr)                                   \
  do {                                                     \
    cudaError_t _e = (expr);                               \
    if (_e != cudaSuccess) return AB_ERR_CUDA;             \
  } while (0)

// Every kernel launch site is followed by AB_LAUNCH_OK(), which also counts the launch.
void count_launches(long long n);

#define AB_LAUNCH_OK()                                     \
  do {                                                     \
    ::ab::count_launches(1);                               \
    if (cudaPeekAtLastError() != cudaSuccess) {            \
      cudaGetLastError();                                  \
      return AB_ERR_CUDA;                                  \
    }                                                      \
  } while (0)

#define AB_TRY(expr)                                       \
  do {                                                     \
    int _s = (expr);                                       \
    if (_s != AB_OK) return _s;                            \
  } while (0)

// Lets a kernel take all the shared memory there is beside its static words.  The limit belongs to the kernel, not to a launch: a
// thread that set its own call's figure could lower it between another thread's setting and launch, and that launch would fail.
constexpr int kMaxSmem = 227 * 1024;
template <typename K>
inline cudaError_t allow_smem(K* kernel, int static_bytes = 0) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem - static_bytes);
}

// Launch with programmatic stream serialisation, in clusters of `cluster` CTAs: the kernel may become resident while the one before it
// in the stream still runs.  Only for kernels that wait for that one (tc::dep_wait) before they touch global memory.
template <typename... KArgs, typename... Args>
inline int launch_after(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem, int cluster, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  if (cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...) != cudaSuccess) { (void)cudaGetLastError(); return AB_ERR_CUDA; }
  AB_LAUNCH_OK();
  return AB_OK;
}

// Multiprocessors of the current device (cached per device; 0 if the query fails).  Grid sizes that are
// meant to fill the GPU are derived from it.
int sm_count();

static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
static inline size_t dtype_size(int dt) { return dt == AB_BF16 ? 2 : 4; }
static inline bool dtype_ok(int dt) { return dt == AB_F32 || dt == AB_BF16; }
static inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Carves 256-byte aligned pieces out of the caller's workspace.
struct Arena {
  char* base;
  size_t used;
  size_t cap;
  Arena(void* p, size_t bytes) : base(static_cast<char*>(p)), used(0), cap(bytes) {}
  void* take(size_t bytes) {
    size_t off = align_up(used, 256);
    used = off + bytes;
    return base ? base + off : nullptr;
  }
  template <typename T> T* take_n(size_t n) { return static_cast<T*>(take(n * sizeof(T))); }
  bool fits() const { return used <= cap; }
};

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(bf16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void from_f32(float& d, float v) { d = v; }
__device__ __forceinline__ void from_f32(bf16& d, float v) { d = __float2bfloat16_rn(v); }

// ---- general strided GEMM on the plain fp32 pipes (ab_gemm_simt.cu) ----------------------------
// C[i,j] = sum_k A(i,k) * B(k,j), A(i,k) at A + i*sAm + k*sAk, B(k,j) at B + k*sBk + j*sBn,
// C row-major with row stride ldc.  fp32 accumulation, k ascending inside a thread: results
// do not depend on the launch.  a_dt/b_dt/c_dt are ab_dtype values.
int gemm_simt(const void* A, int a_dt, int64_t sAm, int64_t sAk,
              const void* B, int b_dt, int64_t sBk, int64_t sBn,
              void* C, int c_dt, int64_t ldc,
              int64_t M, int64_t N, int64_t K, cudaStream_t st);

// The reduction in parts of `per`: part q is M x N (without gaps) at parts + q M N, sums of 16 products in fp32, those in fp64; upper (M
// = N): only tiles that reach the upper triangle are formed.  sum_parts adds them up.
int gemm_parts(const float* A, int64_t sAm, int64_t sAk, const float* B, int64_t sBk, int64_t sBn, double* parts, int M, int N, int K, int per,
               bool upper, cudaStream_t st);
int sum_parts(const double* part, int parts, int64_t count, float* out, cudaStream_t st);

// One fp32 problem of the register-tiled kernel.
struct GemmDesc {
  const float* A; const float* B; void* C;
  int64_t sAm, sAk, sBk, sBn, ldc;
  int M, N, K;
  // Operand prologue that averages group copies (0 / 1 copies: plain operand).  Copy c of A starts a_cstride
  // elements after copy c - 1; the loader adds the copies in ascending c in fp32 and scales by copy_inv, the
  // arithmetic of the group mean.  The CTAs of the first tile column / row also write the averaged operand out.
  int a_copies, b_copies;
  int64_t a_cstride, b_cstride;
  float copy_inv;
  float* a_mean_out;   // optional, M x K row-major
  float* b_mean_out;   // optional, K x N row-major
};
// W = mean_k(A_k) mean_k(B_k) in one kernel (the mean as the product's operand prologue); Abar, Bbar optional outputs.
int recombine_mean_simt(const float* A_copies, int64_t strideA, const float* B_copies, int64_t strideB, int K,
                        float* W, float* Abar, float* Bbar, int m, int n, int r, cudaStream_t st);

// ---- general tensor-core GEMM (ab_gemm_tc.cu) --------------------------------------------------
// C[M x N] = A B^T on the tensor cores; see the head of ab_gemm_tc.cu.
struct TcOperand {
  const void* p;      // bf16
  int64_t ld;         // row stride in elements, a multiple of 8
  bool mn;            // false: stored M x K (resp. N x K); true: stored K x M (resp. K x N)
};
struct TcProblem {
  TcOperand A, B;
  void* C;            // fp32 or bf16, row stride ldc; with ksplit > 1: ksplit partial results, each
  int64_t ldc;        //   round_up(M, 128) rows, one after the other (fp32 only)
  int M, N, K;
  bool c_f32;
  int ksplit;
};
bool gemm_tc_available();
bool gemm_tc_problem_ok(const TcProblem& q);
// One or two problems; status: device int, cleared first, that receives AB_ERR_TIMEOUT if a bounded wait ran out.
int gemm_tc_batched(const TcProblem* probs, int count, int* status, cudaStream_t st);
// count and slice_stride multiples of 4, 16-byte aligned
int sum_slices(const float* part, float* out, int64_t count, int64_t slice_stride, int slices, cudaStream_t st);

// ---- batched fp32-accurate products with the split in the loader (ab_gemm_split.cu) --------------------------
// C[i,j] = rs(i) cs(j) sum_k A(i,k) B(j,k).  A(i,k) at A[i * lda + k] (a_mn 0) or A[k * lda + i] (a_mn 1), B(j,k)
// likewise.  rs, cs from a vector v sorted in descending order: mode 0: 1, 1: sqrt(v), 2: 1/sqrt(v), entries v <= thr v[0]
// count as 0.  Rows >= *live_rows and columns >= *live_cols (device ints, optional) are written as zero.  K >= 1.
struct SplitGemm {
  const void* A; const void* B; void* C;
  int64_t lda, ldb, ldc;
  int M, N, K;
  int a_mn, b_mn;
  int c_bf16;
  int upper_only;           // 1: tiles entirely below the diagonal are skipped
  const float* row_vec; const float* col_vec;
  int row_mode, col_mode;
  float thr;
  const int* live_rows; const int* live_cols;
  int first_tile;           // set by gemm_split_plan
};
struct SplitBatch { int count, tiles, bn; };
SplitBatch gemm_split_plan(SplitGemm* probs, int count);      // fills first_tile; the table then goes to the device
int gemm_split_batched(const SplitGemm* d_probs, const SplitBatch& b, int* status, cudaStream_t st);   // fp32 operands
int gemm_split_one(SplitGemm p, bool src_bf16, int* status, cudaStream_t st);    // one problem; clears *status first

// Copies a host table to the device in pieces the runtime stages without waiting for the stream (a pageable copy of
// more than 64 KB waits until the stream has drained), under stream capture as arguments of kernels: either way the table may go
// when the call returns.
int upload_async(void* dst, const void* src, size_t bytes, cudaStream_t st);

// ---- dense layer of the full-rank phases (ab_dense.cu) ------------------------------------------
size_t dense_forward_ws(int64_t N, int m, int n);
size_t dense_backward_ws(int64_t N, int m, int n);

// ---- fused tensor-core chain (ab_chain_tc.cu) --------------------------------------------------
bool chain_tc_supported(int64_t N, int m, int n, int r, int ldA, int ldB, int dt,
                        const void* x, const void* A, const void* B, const void* y);
size_t chain_tc_forward_ws(int64_t N, int m, int n, int r);
size_t chain_tc_backward_ws(int64_t N, int m, int n, int r);
int chain_tc_forward(const void* x, const void* A, const void* B, void* y, void* T_save,
                     int64_t N, int m, int n, int r, int ldA, int ldB,
                     void* ws, size_t ws_bytes, cudaStream_t st);
int chain_tc_backward(const void* x, const void* dY, const void* A, const void* B,
                      const void* T_saved, void* dX, float* dA, float* dB,
                      int64_t N, int m, int n, int r, int ldA, int ldB,
                      void* ws, size_t ws_bytes, cudaStream_t st);

// ---- bf16 products by tiles (ab_tile_tc.cu) ------------------------------------------------------
// D = X F^T: X is N x K, D is N x P (both without gaps), F is P x K, or, f_mn, K x P; row stride ldF.  K, P, ldF multiples of 8.
struct TileProduct { const void* X; int64_t N; int K; const void* F; int ldF; bool f_mn; void* D; int P; };
int tile_product(const TileProduct& t, bool clear_status, int* status, cudaStream_t st);

// ---- small fp32 products and layers (ab_layer_small.cu) -----------------------------------------
// C[p][q] = sum over k of U[p * u_p + k * u_k] V[q * v_q + k * v_k], row stride ldc; sums of 16 products in fp32, those
// in fp64.  One or two products with the same reduction length in one launch; status: cleared if not null.
struct SmallProduct { const float* U; int64_t u_p, u_k; const float* V; int64_t v_q, v_k; float* C; int64_t ldc; int P, Q; };
int gemm_small(const SmallProduct* jobs, int njobs, int64_t K, int* status, cudaStream_t st);
bool gemm_small_pays(int64_t M, int64_t N, int64_t K);
// S = In F1^T, Out = S F2^T (Out null: only S; S null: not stored) for a layer small enough to be latency-bound;
// F1(j, k) at F1[j * f1_j + k * f1_k], F2(p, j) at F2[p * f2_p + j * f2_j]
bool layer_small_ok(int64_t N, int K1, int P, int r, bool backward);
int layer_small_chain(const float* In, int64_t N, int K1, const float* F1, int64_t f1_j, int64_t f1_k, const float* F2, int64_t f2_p,
                      int64_t f2_j, float* Out, int P, float* S, int r, int* status, cudaStream_t st);

// 3 x 3 convolution with the factorised weight on NHWC activations, im2col rows never formed (ab_chain_tc.cu)
bool conv_tc_supported(int B, int H, int W, int C, int m, int r, int ldA, int ldB, int dt,
                       const void* x, const void* A, const void* Bf);
size_t conv_tc_ws(int B, int H, int W, int C, int m, int r);
int conv_tc_forward(const void* x, const void* A, const void* Bf, void* y, void* T_save, int B, int H, int W, int C,
                    int m, int r, int ldA, int ldB, void* ws, size_t ws_bytes, cudaStream_t st);
int conv_tc_backward(const void* x, const void* dY, const void* A, const void* Bf, const void* T_saved, void* dX,
                     float* dA, float* dB, int B, int H, int W, int C, int m, int r, int ldA, int ldB,
                     void* ws, size_t ws_bytes, cudaStream_t st);

int bounded_wait_selftest(int* dev_status, unsigned limit_us, cudaStream_t st);
size_t chain_stall_selftest_ws();
int chain_stall_selftest(void* ws, size_t ws_bytes, unsigned limit_us, cudaStream_t st);

// ---- SVD pipeline (ab_svd.cu) ------------------------------------------------------------------
struct SvdItem {
  const void* W;     // dense m x n
  int w_dt;
  int m, n, r_max;
  void* A;           // m x r_max
  void* B;           // r_max x n
  int out_dt;
  float* sigma;
  int* r_out;
  int* dev_status;
};
size_t svd_batch_ws(const SvdItem* items, int L);
// Self-test of what follows the direct solver: the first 64 matrices whose bit is set are flagged as if it had left their vectors
// less than orthogonal; a status other than AB_OK stands for a wait that ran out in the solver's first call.
struct SvdSelftest { unsigned long long flagged; int solver_status; };
int svd_batch(const SvdItem* items, int L, float sigma_cutoff, void* ws, size_t ws_bytes, cudaStream_t st,
              const SvdSelftest* selftest = nullptr);

// ---- direct symmetric eigensolver (ab_eig.cu) ---------------------------------------------------
// Leading eigenvectors of `count` symmetric matrices, fp64 inside: any orders up to kEigSmallMax in one call, or
// matrices of one order up to eig_max().  Everything an EigJob points to is device memory; eig_bind carves the
// scratch of one matrix (eig_ws_doubles(s) doubles, 16-byte aligned).
constexpr int kEigSmallMax = 256;
int eig_max();
struct EigJob {
  const float* X;     // s x s, row stride s
  int gram;           // 0: the matrix is X (symmetric); 1: it is X^T X, formed in fp64 from X (s <= kEigSmallMax)
  int s, need;        // order; how many eigenvectors are wanted
  float* rows;        // need x s: unit rows, descending eigenvalue
  float* vals;        // need: the eigenvalue (gram 0) or its square root, 0 below 1e-6 of the largest (gram 1); may be null
  int* flag;          // set to 1 when close vectors came out less than orthogonal (the caller clears it)
  double *xbuf, *refl, *tmat, *zp, *zm, *d, *e, *gam, *lam, *inv, *norm;
  int* order;
};
size_t eig_ws_doubles(int s);
void eig_bind(EigJob& j, double* ws);
// status: device int that receives AB_ERR_TIMEOUT if a bounded wait ran out
// h_jobs: the same table in host memory
int eig_direct(const EigJob* h_jobs, const EigJob* d_jobs, int count, int smax, int* status, cudaStream_t st);

// ---- factored group sync (ab_sync_fast.cu) ------------------------------------------------------
// One-sided Jacobi on the rows of `count` s x s matrices (s <= 256) kept in shared memory, one CTA or
// one cluster of CTAs per matrix (ab_sync_fast.cu).  X: count matrices, s * s apart.  rows: the
// orthogonalised rows scaled to unit length, sorted by descending norm; norms: those norms.  status:
// one int per matrix, status_stride_bytes apart (AB_OK / AB_ERR_NOT_CONVERGED).  scratch: device memory
// of rows_jacobi_scratch_bytes(count).  flags: one int per matrix in device memory; a matrix whose flag is zero is
// left alone.
bool rows_jacobi_fits(int count, int s);
size_t rows_jacobi_scratch_bytes(int count);
int rows_jacobi(const float* X, float* rows, float* norms, int* status, size_t status_stride_bytes, const int* flags,
                int count, int s, void* scratch, cudaStream_t st);
bool sync_factored_supported(const ab_sync_desc* d, int L);
size_t sync_factored_ws(const ab_sync_desc* d, int L);
int sync_factored(const ab_sync_desc* d, int L, int K, float sigma_cutoff, int dt, int* dev_status,
                  void* ws, size_t ws_bytes, cudaStream_t st);

// ---- group mean (ab_average.cu) ----------------------------------------------------------------
// AdamW step on fp32 master values (ab_optim.cu); p_lp: optional bf16 copy of the result.
int adamw_step(float* p, const float* g, float* m, float* v, bf16* p_lp, int64_t count, float lr, float beta1,
               float beta2, float eps, float weight_decay, int step, cudaStream_t st);

// One mean per job in a single launch; results are fp32.  d_jobs is device memory.
// One mean of a batched launch.  first_block: the job's first block in the flat grid (running sum of
// average_job_blocks over the jobs before it); the launch gets the sum over all jobs.
struct AvgJob { const void* base; int64_t stride; int64_t count; float* out; int64_t first_block; };
int64_t average_job_blocks(int64_t count, int in_dt);
int group_average_batched(const AvgJob* d_jobs, int njobs, int K, int in_dt, int64_t total_blocks, cudaStream_t st);
int group_average(const void* base, int64_t stride_elems, int K, int64_t count,
                  int in_dt, int out_dt, void* out, cudaStream_t st);

}  // namespace ab
