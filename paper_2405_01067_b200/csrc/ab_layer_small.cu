// The factorised layer in fp32 storage: forward and backward of the small layers, two kernels in place of one general
// GEMM per product (six and a cast; 11 us each for a 64 x 512 -> 256 layer, of which the arithmetic is a tenth).
//
//   small_chain_kernel:  S = In F1^T,  Out = S F2^T  for a few rows per CTA, S in shared memory (forward: T and y;
//                        backward: dT and dX with A and B read the other way round)
//   small_gemm_kernel:   dA = dY^T T and dB = dT^T x in one launch, 32 x 32 tiles, the rows cut over a cluster; also
//                        every other fp32 product that gemm_small_pays names
//
// Sums: 16 products in fp32, those sums in fp64, in an order fixed by the shape, as in the general kernel.
// What bounds both at the small sizes is latency: a launch, a trip to L2 for the first values, then the factors streamed once per
// CTA (96 KB, about 1 us).  64 x 512 -> 256, rank 32, forward and backward: 82 -> 27 us, seven kernels -> three.
// The tiled product against the general kernel it replaces for fp32 (64 x 64 tiles, one CTA walking the whole reduction):
// backward of a 1024 x 100 layer, rank 30, 50432 rows: 8.8 -> 0.8 ms.
#include <cooperative_groups.h>

#include "ab_common.cuh"
#include "ab_tc_ptx.cuh"

namespace ab {
namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;

struct SmallChain {
  const float* In; int K1;            // N x K1
  const float* F1; int64_t f1_j, f1_k;   // F1(j, k) at F1[j * f1_j + k * f1_k]; one of the strides is 1
  const float* F2; int64_t f2_p, f2_j;   // F2(p, j) likewise
  float* Out; int P;                  // N x P, or null
  float* S;                           // N x r, or null
  int64_t N;
  int r;
  int* status;                        // cleared by the first kernel of a call (null otherwise)
};

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One pass over a reduction for R rows and one column per thread: rows in[i * ld_in + k] (shared memory),
// column c[k * step], k = k0 .. k1 - 1.
template <int R>
__device__ __forceinline__ void column_sums(const float* in, int ld_in, const float* __restrict__ c, int64_t step, int k0, int k1,
                                            double (&acc)[R]) {
#pragma unroll
  for (int i = 0; i < R; ++i) acc[i] = 0.0;
  int k = k0;
  for (; k + 16 <= k1; k += 16) {
    float v[16], part[R];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = c[(k + u) * step];
#pragma unroll
    for (int i = 0; i < R; ++i) part[i] = 0.f;
#pragma unroll
    for (int u = 0; u < 16; u += 4)
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const float4 q = *reinterpret_cast<const float4*>(in + i * ld_in + k + u);
        part[i] = fmaf(q.w, v[u + 3], fmaf(q.z, v[u + 2], fmaf(q.y, v[u + 1], fmaf(q.x, v[u], part[i]))));
      }
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] += (double)part[i];
  }
  if (k < k1) {
    float part[R];
#pragma unroll
    for (int i = 0; i < R; ++i) part[i] = 0.f;
    for (; k < k1; ++k) {
      const float v = c[k * step];
#pragma unroll
      for (int i = 0; i < R; ++i) part[i] = fmaf(in[i * ld_in + k], v, part[i]);
    }
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] += (double)part[i];
  }
}

// R rows per CTA.  A factor whose reduction index is contiguous in memory (forward: B in the first product) is walked by
// warps, a warp per column, lanes along the reduction, sums across the lanes at the end.  One whose other index is
// contiguous (backward: A in the first product, B in the second) is walked by threads, a thread per column; when there
// are fewer columns than threads, groups of warps take parts of the reduction and their sums meet in shared memory.
template <int R>
__global__ void __launch_bounds__(kThreads)
small_chain_kernel(const SmallChain p) {
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r = p.r, ldi = (p.K1 + 3) & ~3, lds = (r + 3) & ~3;     // 16-byte rows
  float* in = sm;                              // R x ldi
  float* S = in + R * ldi;                     // R x lds
  double* red = reinterpret_cast<double*>(S + R * lds);   // kThreads x R
  tc::dep_wait();
  tc::dep_launch();
  if (p.status && blockIdx.x == 0 && tid == 0) *p.status = 0;
  const int64_t row0 = (int64_t)blockIdx.x * R;
  const int rows = (int)(p.N - row0 < R ? p.N - row0 : R);
  for (int i = 0; i < R; ++i)
    for (int k = tid; k < p.K1; k += kThreads) in[i * ldi + k] = i < rows ? p.In[(row0 + i) * p.K1 + k] : 0.f;
  __syncthreads();

  if (p.f1_k == 1) {
    for (int j = warp; j < r; j += kThreads / 32) {
      const float* c = p.F1 + (int64_t)j * p.f1_j;
      double acc[R];
#pragma unroll
      for (int i = 0; i < R; ++i) acc[i] = 0.0;
      for (int kb = 0; kb < p.K1; kb += 512) {            // 16 values a lane
        float v[16], part[R];
#pragma unroll
        for (int u = 0; u < 16; ++u) { const int k = kb + 32 * u + lane; v[u] = k < p.K1 ? c[k] : 0.f; }
#pragma unroll
        for (int i = 0; i < R; ++i) part[i] = 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int k = kb + 32 * u + lane;
          if (k < p.K1) {
#pragma unroll
            for (int i = 0; i < R; ++i) part[i] = fmaf(in[i * ldi + k], v[u], part[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < R; ++i) acc[i] += (double)part[i];
      }
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const double t = warp_sum_d(acc[i]);
        if (lane == i) S[i * lds + j] = (float)t;
      }
    }
  } else {
    const int rp = (r + 31) & ~31, groups = rp >= kThreads ? 1 : kThreads / rp;     // parts of the reduction
    const int g = groups > 1 ? tid / rp : 0, jt = groups > 1 ? tid - g * rp : tid;
    const int per = ((p.K1 + groups - 1) / groups + 15) & ~15;
    for (int j0 = 0; j0 < rp; j0 += kThreads) {
      const int j = j0 + jt;
      double acc[R];
#pragma unroll
      for (int i = 0; i < R; ++i) acc[i] = 0.0;
      if (j < r && g < groups) column_sums<R>(in, ldi, p.F1 + j, p.f1_k, min(g * per, p.K1), min((g + 1) * per, p.K1), acc);
      if (groups > 1) {
#pragma unroll
        for (int i = 0; i < R; ++i) red[i * kThreads + tid] = acc[i];
        __syncthreads();
        for (int e = tid; e < R * r; e += kThreads) {
          const int i = e / r, jj = e - i * r;
          double t = 0.0;
          for (int q = 0; q < groups; ++q) t += red[i * kThreads + q * rp + jj];
          S[i * lds + jj] = (float)t;
        }
      } else if (j < r) {
#pragma unroll
        for (int i = 0; i < R; ++i) S[i * lds + j] = (float)acc[i];
      }
    }
  }
  __syncthreads();
  if (p.S)
    for (int e = tid; e < rows * r; e += kThreads) { const int i = e / r, j = e - i * r; p.S[(row0 + i) * r + j] = S[i * lds + j]; }
  if (!p.Out) return;
  for (int q = tid; q < p.P; q += kThreads) {
    double acc[R];
    column_sums<R>(S, lds, p.F2 + (int64_t)q * p.f2_p, p.f2_j, 0, r, acc);
#pragma unroll
    for (int i = 0; i < R; ++i)
      if (i < rows) p.Out[(row0 + i) * p.P + q] = (float)acc[i];
  }
}

// C[p][q] = sum over k of U(p, k) V(q, k) for up to two problems with the same k at once; U(p, k) at U[p * u_p + k * u_k],
// V likewise.  32 x 32 tiles; the reduction is cut over the CTAs of a cluster, in each over its eight warps.  A warp
// fetches the 16 x 32 values of each operand that it multiplies itself, so no barrier is inside the loop.
//   kMany false: the next slab waits in registers (one CTA per SM; what counts is the latency of a lone tile)
//   kMany true : asynchronous copies into a second buffer, lanes along the index that is contiguous in memory; two CTAs
//                per SM hide each other's waits (768 x 768 x 3072: 290 -> 235 us, but a 256 x 64 layer of 1000 rows 51 -> 61 us)
struct SmallGemm { SmallProduct job[2]; int64_t K; int tiles0, tiles_q[2]; int* status; };

constexpr int kGt = 32, kGk = 128;                 // tile edge, reduction per slab: 16 for each of the eight warps
static_assert(sizeof(float) * 4 * kGk * (kGt + 4) >= sizeof(double) * 8 * 1024, "");
template <bool kMany>
__global__ void __launch_bounds__(kThreads, kMany ? 2 : 1)
small_gemm_kernel(const __grid_constant__ SmallGemm p) {
  // two slabs of both operands; afterwards the eight warps' sums (8 x 1024 doubles) lie over them
  extern __shared__ __align__(16) unsigned char gsm[];
  typedef float Slab[kGk][kGt + 4];
  Slab* us = reinterpret_cast<Slab*>(gsm);
  Slab* vs = us + 2;
  double* gred = reinterpret_cast<double*>(gsm);
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  tc::dep_wait();
  tc::dep_launch();
  if (p.status && blockIdx.x == 0 && tid == 0) *p.status = 0;
  int t = blockIdx.x / C;
  const int jb = t >= p.tiles0 ? 1 : 0;
  const SmallProduct& job = p.job[jb];
  if (jb) t -= p.tiles0;
  const int p0 = (t / p.tiles_q[jb]) * kGt, q0 = (t % p.tiles_q[jb]) * kGt;
  // this CTA's part of the reduction: whole groups of 16
  const int64_t n16 = (p.K + 15) / 16;
  const int64_t k_begin = n16 * rank / C * 16;
  int64_t k_end = n16 * (rank + 1) / C * 16;
  if (k_end > p.K) k_end = p.K;
  const int ty = lane >> 2, tx = lane & 3;
  double acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.0;
  struct Source { const float* p; int64_t step; int row, k, drow, dk; };     // value e of a lane: row + e drow, k + e dk
  auto source = [&](const float* b, int64_t s_row, int64_t s_k, int row0) {
    Source o;
    if (s_k == 1) { o.row = lane >> 4; o.k = lane & 15; o.drow = 2; o.dk = 0; o.step = 2 * s_row; }
    else { o.row = lane; o.k = 0; o.drow = 0; o.dk = 1; o.step = s_k; }
    o.p = b + (int64_t)(row0 + o.row) * s_row + (int64_t)(warp * 16 + o.k) * s_k;
    return o;
  };
  const Source su = source(job.U, job.u_p, job.u_k, p0), sv = source(job.V, job.v_q, job.v_k, q0);
  auto fetch_one = [&](const Source& o, int64_t s_k, int rows, Slab& dst, int64_t k0) {
    const float* g = o.p + k0 * s_k;
    const int left = (int)(k_end - k0 < (int64_t)kGk ? k_end - k0 : (int64_t)kGk) - warp * 16;      // of the reduction
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const int row = o.row + e * o.drow, k = o.k + e * o.dk;
      const int bytes = (row < rows && k < left) ? 4 : 0;                  // nothing read: zero
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tc::smem_u32(&dst[warp * 16 + k][row])),
                   "l"(bytes ? g + e * o.step : job.U), "r"(bytes)
                   : "memory");
    }
  };
  auto fetch = [&](int64_t k0, int buf) {
    if (k0 < k_end) {
      fetch_one(su, job.u_k, job.P - p0, us[buf], k0);
      fetch_one(sv, job.v_k, job.Q - q0, vs[buf], k0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float fu[16], fv[16];
  const float* up = job.U + (int64_t)(p0 + lane) * job.u_p;
  const float* vp = job.V + (int64_t)(q0 + lane) * job.v_q;
  const bool uin = p0 + lane < job.P, vin = q0 + lane < job.Q;
  const bool uvec = job.u_k == 1 && job.u_p % 4 == 0 && (reinterpret_cast<uintptr_t>(job.U) & 15u) == 0;
  const bool vvec = job.v_k == 1 && job.v_q % 4 == 0 && (reinterpret_cast<uintptr_t>(job.V) & 15u) == 0;
  auto load16 = [](float (&f)[16], const float* b, int64_t step, bool in, bool vec, int64_t k, int64_t kend) {
    if (vec && in && k + 16 <= kend) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float4 q = *reinterpret_cast<const float4*>(b + k + 4 * e);
        f[4 * e] = q.x; f[4 * e + 1] = q.y; f[4 * e + 2] = q.z; f[4 * e + 3] = q.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) f[e] = (in && k + e < kend) ? b[(k + e) * step] : 0.f;
    }
  };
  auto fetch_regs = [&](int64_t k0) {
    load16(fu, up, job.u_k, uin, uvec, k0 + warp * 16, k_end);
    load16(fv, vp, job.v_k, vin, vvec, k0 + warp * 16, k_end);
  };
  if constexpr (kMany) fetch(k_begin, 0);
  else if (k_begin < k_end) fetch_regs(k_begin);
  int buf = 0;
  for (int64_t k0 = k_begin; k0 < k_end; k0 += kGk) {
    if constexpr (kMany) {
      fetch(k0 + kGk, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncwarp();
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) { us[0][warp * 16 + e][lane] = fu[e]; vs[0][warp * 16 + e][lane] = fv[e]; }
      __syncwarp();
      if (k0 + kGk < k_end) fetch_regs(k0 + kGk);
    }
    float part[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) part[i][j] = 0.f;
    if (k0 + warp * 16 < k_end) {
#pragma unroll 4
      for (int e = 0; e < 16; ++e) {
        const float4 a = *reinterpret_cast<const float4*>(&us[buf][warp * 16 + e][ty * 4]);
        const float4 b0 = *reinterpret_cast<const float4*>(&vs[buf][warp * 16 + e][tx * 8]), b1 = *reinterpret_cast<const float4*>(&vs[buf][warp * 16 + e][tx * 8 + 4]);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) part[i][j] = fmaf(av[i], bv[j], part[i][j]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] += (double)part[i][j];
    __syncwarp();
    if constexpr (kMany) buf ^= 1;
  }
  if constexpr (kMany) asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) gred[warp * 1024 + (ty * 4 + i) * 32 + tx * 8 + j] = acc[i][j];
  __syncthreads();
  for (int e = tid; e < 1024; e += kThreads) {        // the eight warps' sums, ascending
    double s = gred[e];
#pragma unroll
    for (int w = 1; w < 8; ++w) s += gred[w * 1024 + e];
    gred[e] = s;
  }
  if (C > 1) cluster.sync(); else __syncthreads();
  // CTA `rank` finishes a part of the tile: sums of the cluster's CTAs in ascending order
  const int share = 1024 / C;
  for (int e = rank * share + tid; e < (rank + 1) * share; e += kThreads) {
    double s = 0.0;
    for (int c = 0; c < C; ++c) s += C > 1 ? cluster.map_shared_rank(gred, c)[e] : gred[e];
    const int pp = p0 + (e >> 5), qq = q0 + (e & 31);
    if (pp < job.P && qq < job.Q) job.C[(int64_t)pp * job.ldc + qq] = (float)s;
  }
  if (C > 1) cluster.sync();                          // nobody leaves while a peer reads its sums
}

template <typename P>
int launch_small(void (*kernel)(const P), unsigned grid, int cluster, size_t smem, cudaStream_t st, const P& p) {
  if (smem > 48 * 1024) AB_CUDA_OK(allow_smem(kernel));
  return launch_after(kernel, grid, (unsigned)kThreads, smem, cluster, st, p);
}

size_t chain_smem(int R, int K1, int r) { return sizeof(float) * (size_t)R * (((K1 + 3) & ~3) + ((r + 3) & ~3)) + sizeof(double) * kThreads * R; }

// Rows per CTA: one CTA per SM as long as that takes at most 16 rows.
int rows_per_cta(int64_t N) {
  const int sms = sm_count() > 0 ? sm_count() : 1;
  int R = 1;
  while (R < 16 && (N + R - 1) / R > sms) R *= 2;
  return R;
}

int run_chain(const SmallChain& p, cudaStream_t st) {
  const int R = rows_per_cta(p.N);
  const unsigned grid = (unsigned)((p.N + R - 1) / R);
  const size_t sm = chain_smem(R, p.K1, p.r);
  switch (R) {
    case 1: return launch_small(small_chain_kernel<1>, grid, 1, sm, st, p);
    case 2: return launch_small(small_chain_kernel<2>, grid, 1, sm, st, p);
    case 4: return launch_small(small_chain_kernel<4>, grid, 1, sm, st, p);
    case 8: return launch_small(small_chain_kernel<8>, grid, 1, sm, st, p);
    default: return launch_small(small_chain_kernel<16>, grid, 1, sm, st, p);
  }
}

}  // namespace

// Whether a product goes to small_gemm_kernel.  Its 32 x 32 tiles and cut reductions win where the 64 x 64 kernel would leave half
// of the SMs empty for a long walk; with more tiles, or next to no reduction, that kernel has less to do per result.  Measured at
// 148 SMs, us 64 x 64 / this: 256 x 250, K 3072 194 / 39, K 64 10.3 / 8.5; 512 x 512 (64 of its tiles), K 4608 280 / 176; 4096 x 64,
// K 64 9.9 / 14.4; 128 x 3072 (96 tiles), K 512 37 / 43; 768 x 768 (144), K 3072 190 / 235, K 16384 1350 / 1270, K 50432 4200 / 3900;
// 1024 x 1024 (256), K 1 7.5 / 34, K 50432 4970 / 7420.
bool gemm_small_pays(int64_t M, int64_t N, int64_t K) {
  const int64_t sms = sm_count() > 0 ? sm_count() : 1, tiles = (M + 63) / 64 * ((N + 63) / 64);
  if (2 * tiles >= sms) return tiles <= sms && K >= 16384;
  return K >= 96 || (K >= 64 && (M + kGt - 1) / kGt * ((N + kGt - 1) / kGt) <= sms);
}

int gemm_small(const SmallProduct* jobs, int njobs, int64_t K, int* status, cudaStream_t st) {
  SmallGemm g;
  int64_t tiles = 0;
  for (int i = 0; i < 2; ++i) {
    g.job[i] = jobs[i < njobs ? i : 0];
    g.tiles_q[i] = (g.job[i].Q + kGt - 1) / kGt;
    const int64_t t = (int64_t)((g.job[i].P + kGt - 1) / kGt) * g.tiles_q[i];
    if (i < njobs) tiles += t;
    if (i == 0) g.tiles0 = (int)t;
  }
  if (tiles <= 0) return AB_OK;
  g.K = K;
  g.status = status;
  // the reduction cut over a cluster while each CTA keeps a slab and the device has room for two CTAs an SM
  const int sms = sm_count() > 0 ? sm_count() : 1;
  int C = 1;
  while (C < 8 && K / (2 * C) >= kGk && tiles * 2 * C <= 2LL * sms) C *= 2;
  const size_t sm = sizeof(float) * 4 * kGk * (kGt + 4);
  if (tiles * C > sms) return launch_small(small_gemm_kernel<true>, (unsigned)(tiles * C), C, sm, st, g);
  return launch_small(small_gemm_kernel<false>, (unsigned)(tiles * C), C, sm, st, g);
}

// Whether the fused chain S = In F1^T, Out = S F2^T (In: N x K1, Out: N x P) is faster than a launch per product.  A CTA streams
// both factors for its 1 to 16 rows, by single values: it wins where that is little and the separate products
// are bound by their launches and the length of one reduction.  Forward, a thread's row of F2 = A is its own and its values lie
// apart from its neighbours': that costs r^2 P, backward the lanes read along F2 = B.  Measured, us fused / by products: forward
// 64 x 512 -> 32 -> 256 9.3 / 16.5, 1000 x 256 -> 32 -> 256 14.6 / 20.6, 2368 x 256 -> 32 -> 64 19.3 / 14.5, 600 x 64 -> 64 -> 64 17.3 / 14.4,
// 64 x 768 -> 32 -> 1024 24 / 16.5, 4096 x 256 -> 8 -> 256 17.1 / 26.7, 16384 x 64 -> 16 -> 64 66.9 / 18.5; backward 1000 x 256 -> 128 -> 256
// 23 / 33, 300 x 256 -> 128 -> 512 31.2 / 20.7, 64 x 1024 -> 32 -> 1024 22.9 / 16.3.  Above 16 rows a CTA and SM the
// factors are streamed again, which only a long first reduction into a narrow rank is worth.
bool layer_small_ok(int64_t N, int K1, int P, int r, bool backward) {
  const int64_t sms = sm_count() > 0 ? sm_count() : 1;
  const int64_t wide = (int64_t)r * (K1 > P ? K1 : P), out = (int64_t)r * P;
  const int R = rows_per_cta(N);
  if (chain_smem(R, K1, r) > 200 * 1024 || chain_smem(R, P, r) > 200 * 1024) return false;
  if (N > 64 * sms) return false;
  if (N > 32 * sms) return r <= 8 && K1 >= 1024;
  if (N > 16 * sms) {
    if (backward) return K1 >= 256 && r <= 32 && (P <= 512 || out <= 1024) && P >= 64;
    return K1 >= 256 && r <= 16 && out <= 4096;
  }
  if (backward) {
    if (N > 4 * sms) return wide <= 65536;
    return r <= 64 && wide <= 32768 && (N > sms || out <= 16384);
  }
  if (r > (N <= 2 * sms ? 64 : 32) || wide > 32768) return false;
  if (N <= 8 * sms) return r * out <= 600000;
  return K1 >= 256 ? r * out <= 300000 : r <= 16 && r * out <= 70000;
}

int layer_small_chain(const float* In, int64_t N, int K1, const float* F1, int64_t f1_j, int64_t f1_k, const float* F2, int64_t f2_p,
                      int64_t f2_j, float* Out, int P, float* S, int r, int* status, cudaStream_t st) {
  SmallChain p;
  p.In = In; p.K1 = K1; p.F1 = F1; p.f1_j = f1_j; p.f1_k = f1_k; p.F2 = F2; p.f2_p = f2_p; p.f2_j = f2_j; p.Out = Out; p.P = P;
  p.S = S; p.N = N; p.r = r; p.status = status;
  return run_chain(p, st);
}

}  // namespace ab
