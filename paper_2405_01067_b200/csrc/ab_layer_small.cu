// The factorised layer in fp32 storage: forward and backward of the small layers, two kernels in place of one general
// GEMM per product (six and a cast; 11 us each for a 64 x 512 -> 256 layer, of which the arithmetic is a tenth).
//
//   small_chain_kernel:  S = In F1^T,  Out = S F2^T  for a few rows per CTA, S in shared memory (forward: T and y;
//                        backward: dT and dX with A and B read the other way round)
//   small_grad_kernel:   dA = dY^T T and dB = dT^T x in one launch, 32 x 32 tiles, the rows cut over a cluster
//
// Sums: 16 products in fp32, those sums in fp64, in an order fixed by the shape, as in the general kernel.
// What bounds both at the small sizes is latency: a launch, a trip to L2 for the first values, then the factors streamed once per
// CTA (96 KB, about 1 us).  64 x 512 -> 256, rank 32, forward and backward: 70 us of kernels -> three kernels.
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

// C[p][q] = sum over rows k of U[k][p] V[k][q] for two problems at once.
struct SmallGradJob { const float* U; const float* V; float* C; int P, Q, tiles_q, tiles; };
struct SmallGrad { SmallGradJob job[2]; int64_t N; int* status; };

constexpr int kGt = 32, kGk = 128;                 // tile edge, rows per slab: 16 for each of the eight warps
__global__ void __launch_bounds__(kThreads)
small_grad_kernel(const SmallGrad p) {
  __shared__ __align__(16) float us[kGk][kGt + 4], vs[kGk][kGt + 4];
  extern __shared__ __align__(16) double gred[];     // 8 warps x 1024
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  tc::dep_wait();
  tc::dep_launch();
  if (p.status && blockIdx.x == 0 && tid == 0) *p.status = 0;
  int t = blockIdx.x / C;
  const int jb = t >= p.job[0].tiles ? 1 : 0;
  const SmallGradJob& job = p.job[jb];
  if (jb) t -= p.job[0].tiles;
  const int p0 = (t / job.tiles_q) * kGt, q0 = (t % job.tiles_q) * kGt;
  // this CTA's rows: whole 16-row groups
  const int64_t n16 = (p.N + 15) / 16;
  const int64_t k_begin = n16 * rank / C * 16;
  int64_t k_end = n16 * (rank + 1) / C * 16;
  if (k_end > p.N) k_end = p.N;
  const int ty = lane >> 2, tx = lane & 3;
  double acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.0;
  float fu[16], fv[16];                              // a column of the slab per lane, 16 rows per thread
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const int64_t k = k0 + warp * 16 + e;
      fu[e] = (k < k_end && p0 + lane < job.P) ? job.U[k * job.P + p0 + lane] : 0.f;
      fv[e] = (k < k_end && q0 + lane < job.Q) ? job.V[k * job.Q + q0 + lane] : 0.f;
    }
  };
  // a warp multiplies the rows it has fetched itself: no barrier inside the loop
  if (k_begin < k_end) fetch(k_begin);
  for (int64_t k0 = k_begin; k0 < k_end; k0 += kGk) {
#pragma unroll
    for (int e = 0; e < 16; ++e) { us[warp * 16 + e][lane] = fu[e]; vs[warp * 16 + e][lane] = fv[e]; }
    __syncwarp();
    if (k0 + kGk < k_end) fetch(k0 + kGk);
    float part[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) part[i][j] = 0.f;
    if (k0 + warp * 16 < k_end) {
#pragma unroll 4
      for (int e = 0; e < 16; ++e) {
        const float4 a = *reinterpret_cast<const float4*>(&us[warp * 16 + e][ty * 4]);
        const float4 b0 = *reinterpret_cast<const float4*>(&vs[warp * 16 + e][tx * 8]), b1 = *reinterpret_cast<const float4*>(&vs[warp * 16 + e][tx * 8 + 4]);
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
  }
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
    if (pp < job.P && qq < job.Q) job.C[(int64_t)pp * job.Q + qq] = (float)s;
  }
  if (C > 1) cluster.sync();                          // nobody leaves while a peer reads its sums
}

template <typename K, typename P>
int launch_small(K* kernel, unsigned grid, int cluster, size_t smem, cudaStream_t st, const P& p) {
  if (smem > 48 * 1024) AB_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  if (cudaLaunchKernelEx(&cfg, kernel, p) != cudaSuccess) { (void)cudaGetLastError(); return AB_ERR_CUDA; }
  AB_LAUNCH_OK();
  return AB_OK;
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

// Where a product gives the register-tiled kernel enough tiles to fill the device twice, that one is the better;
// the row blocks also have to fit shared memory.
bool layer_small_ok(int64_t N, int m, int n, int r) {
  const int64_t wide = m > n ? m : n;
  if (((N + 63) / 64) * ((wide + 63) / 64) >= 296) return false;
  const int R = rows_per_cta(N);
  return chain_smem(R, n, r) <= 200 * 1024 && chain_smem(R, m, r) <= 200 * 1024;
}

int layer_small_forward(const float* x, const float* A, const float* B, float* y, float* T_save, int64_t N, int m, int n, int r,
                        int ldA, int ldB, int* status, cudaStream_t st) {
  SmallChain p;
  p.In = x; p.K1 = n; p.F1 = B; p.f1_j = ldB; p.f1_k = 1; p.F2 = A; p.f2_p = ldA; p.f2_j = 1; p.Out = y; p.P = m; p.S = T_save;
  p.N = N; p.r = r; p.status = status;
  return run_chain(p, st);
}

int layer_small_backward(const float* x, const float* dY, const float* A, const float* B, const float* T_saved, float* dX, float* dA,
                         float* dB, int64_t N, int m, int n, int r, int ldA, int ldB, float* wsT, float* wsdT, int* status,
                         cudaStream_t st) {
  int* clear = status;                // the first kernel of the call clears the status word
  if (dX || dB) {
    SmallChain p;
    p.In = dY; p.K1 = m; p.F1 = A; p.f1_j = 1; p.f1_k = ldA; p.F2 = B; p.f2_p = 1; p.f2_j = ldB; p.Out = dX; p.P = n;
    p.S = dB ? wsdT : nullptr; p.N = N; p.r = r; p.status = clear;
    AB_TRY(run_chain(p, st));
    clear = nullptr;
  }
  const float* T = T_saved;
  if (dA && !T) {
    SmallChain p;
    p.In = x; p.K1 = n; p.F1 = B; p.f1_j = ldB; p.f1_k = 1; p.F2 = nullptr; p.f2_p = p.f2_j = 0; p.Out = nullptr; p.P = 0;
    p.S = wsT; p.N = N; p.r = r; p.status = clear;
    AB_TRY(run_chain(p, st));
    clear = nullptr;
    T = wsT;
  }
  if (dA || dB) {
    SmallGrad g;
    auto job = [](const float* U, const float* V, float* C, int P, int Q) {
      SmallGradJob j;
      j.U = U; j.V = V; j.C = C; j.P = P; j.Q = Q; j.tiles_q = (Q + kGt - 1) / kGt; j.tiles = ((P + kGt - 1) / kGt) * j.tiles_q;
      return j;
    };
    const SmallGradJob ja = job(dY, T, dA, m, r), jb = job(wsdT, x, dB, r, n);
    g.job[0] = dA ? ja : jb;
    g.job[1] = jb;
    if (!(dA && dB)) g.job[1].tiles = 0;
    g.N = N;
    g.status = clear;
    const int tiles = g.job[0].tiles + g.job[1].tiles, sms = sm_count() > 0 ? sm_count() : 1;
    // the rows cut over a cluster while that leaves each CTA 256 of them and the device room for the clusters
    int C = 1;
    while (C < 8 && N / (2 * C) >= 256 && (long long)tiles * 2 * C <= 2LL * sms) C *= 2;
    AB_TRY(launch_small(small_grad_kernel, (unsigned)(tiles * C), C, sizeof(double) * 8 * 1024, st, g));
    clear = nullptr;
  }
  if (clear) AB_CUDA_OK(cudaMemsetAsync(status, 0, sizeof(int), st));    // nothing was asked for
  return AB_OK;
}

}  // namespace ab
