// Factored group synchronisation: the split of W = Abar Bbar (Algorithm 1, the decomposition that
// follows the all-reduces and "W <- AB") without ever forming the m x n matrix.  W has rank <= r,
// so everything reduces to r x r problems:
//   G_A = Abar^T Abar = R_A^T R_A,   G_B = Bbar Bbar^T = R_B^T R_B      (Cholesky, r x r, upper R)
//   Abar = Q_A R_A,  Bbar^T = Q_B R_B   with Q_A = Abar R_A^-1, Q_B = Bbar^T R_B^-1 orthonormal
//   W = Q_A M Q_B^T,  M = R_A R_B^T  (r x r),   M = U_M S V_M^T         (SVD, r x r)
//   A' = Abar Z_A,  Z_A = R_A^-1 (M V_M) S^(-1/2);   B' = Z_B Bbar,  Z_B = S^(1/2) V_M^T R_B^-T
// One CTA per Gram matrix factors it in shared memory and inverts the triangle in place.  The SVD of M is the
// direct eigensolver of ab_eig.cu on M^T M in fp64 (whole ViT-B/16, 72 cores of order 192: 2183 -> 770 us for its four
// kernels against the one-sided Jacobi alone; a lone core of order 64: 234 -> 106 us).  A core whose vectors that solver could not
// keep orthogonal goes through the Jacobi kernel below, which returns at once for all others: one CTA or cluster
// per M keeps it in shared memory and orthogonalises its ROWS with one-sided rotations (the rows of the result are
// sigma_i v_i^T), so no kernel boundary and no global traffic sits
// between rotations.  Cholesky pivots below 1e-6 of the largest diagonal entry of G are treated
// as zero: the row of R and the row and column of its inverse are dropped, which is exactly right
// for factors truncated by the rank rule (zero columns of A, zero rows of B).  Otherwise the
// factors need a condition number below about 300 -- all workloads here are far inside.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <vector>

#include <cooperative_groups.h>

#include "ab_common.cuh"
#include "ab_tc_ptx.cuh"

namespace ab {
namespace {

namespace cg = cooperative_groups;

constexpr int kJMaxSweeps = 40;
constexpr float kJDead2 = 1e-12f;    // rows below 1e-6 of the largest norm are zero rows
constexpr float kJCount2 = 1e-8f;    // rows below 1e-4 of the largest norm do not hold up convergence
constexpr float kJEarly2 = 4e-6f;    // a sweep whose largest rotated cosine was below 2e-3 is the last one: one-sided
                                     // Jacobi converges quadratically, so what it leaves is of the order 4e-6 <= tol
constexpr float kEigThr = 1e-6f;     // relative pivot cut of G_A, G_B (and of sigma in the scalings)
// Accuracy domain of the factored route: the relative error of a singular value grows as it falls below the
// largest and the worse conditioned the factors are (measured: at most 7e-5 down to 1 % of the largest for
// factors of condition number up to 1e4; 1e-4 to 5e-3 below that); a kept value between
// kFZeroRel and kFDomainRel of the largest, or a Cholesky pivot that was dropped although it was not exactly
// zero, is reported through the status word.
constexpr float kFDomainRel = 1e-2f, kFZeroRel = 1e-6f;
constexpr int kCThreads = 512;
constexpr int kStatics = 256;          // the few static words of the kernels here, rounded up

struct JacobiJob {
  const float* X;   // k x r input (row stride r)
  float* rows;      // k x r output: unit rows, sorted by descending norm (zero rows stay zero)
  float* norms;     // k
  int* status;      // AB_OK / AB_ERR_NOT_CONVERGED (may be null)
  const int* flag;  // run only if *flag is set
  int k, r;
};

__device__ __forceinline__ void rr_pair2(int ne, int t, int idx, int& p, int& q) {
  // t < ne - 1 and idx < ne / 2: one conditional subtraction replaces each modulo
  const int n1 = ne - 1;
  if (idx == 0) { p = n1; q = t; }
  else {
    p = t + idx; if (p >= n1) p -= n1;
    q = t - idx + n1; if (q >= n1) q -= n1;
  }
  if (p > q) { int tmp = p; p = q; q = tmp; }
}

// One matrix per cluster of kC CTAs.  Rows are grouped in blocks of 4; block b lives in the shared
// memory of CTA b % kC, and every CTA reads and writes any row through distributed shared memory.
// Each row carries its squared norm in the padding element behind it.  In each round a warp takes
// one pair of blocks, pulls its 8 rows into registers (r/32 elements per lane and row), rotates the
// 16 cross pairs (4 steps of 4 disjoint pairs worked on side by side; in the first round of a
// sweep also the pairs inside each block) and writes the rows back: shared memory is touched once
// per 16 rotations.  Rounds end with a cluster barrier (a hardware barrier: every CTA of the
// cluster runs the same number of them, since sweep and round counts depend only on values all
// CTAs agree on).
template <int kEL, int kC>      // kEL elements per lane and row in registers: r <= 32 kEL
__global__ void __launch_bounds__((kC == 1 && kEL == 6) ? 768 : 512, 1)
jacobi_rows_cluster_kernel(const JacobiJob* __restrict__ jobs, float tol) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) float sm[];
  const int crank = (kC == 1) ? 0 : (int)cluster.block_rank();
  tc::dep_wait();
  tc::dep_launch();
  const JacobiJob job = jobs[blockIdx.x / kC];
  if (*job.flag == 0) return;                  // the same for every CTA of the cluster
  const int k = job.k, r = job.r, ld = r + 1;
  const int nb = (k + 3) / 4;                  // blocks of 4 rows
  const int nbl = (nb + kC - 1) / kC;          // blocks held by each CTA (same layout in all)
  float* X = sm;                               // 4 nbl x ld; X[i * ld + r] = squared norm of local row i
  float* zrow = X + (size_t)4 * nbl * ld;      // ld zeros: stands in for rows beyond k (rotations leave it zero)
  float* lmax = zrow + ld;                     // kC: largest squared norm seen by each CTA
  int* lflag = reinterpret_cast<int*>(lmax + kC);   // kC: per CTA, the largest squared cosine it rotated (float bits)
  int* rank = lflag + kC;                      // 4 nbl
  __shared__ int wflag;
  __shared__ float wmax;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nthreads = blockDim.x, nwarps = nthreads >> 5;
  auto csync = [&]() {                         // all CTAs that hold a part of this matrix
    if constexpr (kC == 1) __syncthreads(); else cluster.sync();
  };

  auto row_ptr = [&](int row) -> float* {      // any row of the matrix, wherever it lives
    const int b = row >> 2;
    float* p = X + (size_t)(((b / kC) << 2) + (row & 3)) * ld;
    if (kC == 1) return p;
    return cluster.map_shared_rank(p, b % kC);
  };
  auto global_row = [&](int lr) { return (((lr >> 2) * kC + crank) << 2) + (lr & 3); };
  const int nlocal = 4 * nbl;

  for (int lr = warp; lr < nlocal; lr += nwarps) {
    const int g = global_row(lr);
    for (int t = lane; t < r; t += 32) X[lr * ld + t] = (g < k) ? job.X[(size_t)g * r + t] : 0.f;
  }
  for (int t = tid; t < ld; t += nthreads) zrow[t] = 0.f;
  csync();                              // every CTA of the cluster is running and loaded

  // exact squared norms of the local rows into their padding element; the cluster-wide maximum
  auto refresh_norms = [&]() -> float {
    if (tid == 0) { wmax = 0.f; wflag = 0; }
    __syncthreads();
    for (int lr = warp; lr < nlocal; lr += nwarps) {
      float a = 0.f;
      for (int t = lane; t < r; t += 32) { const float v = X[lr * ld + t]; a = fmaf(v, v, a); }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) { X[lr * ld + r] = a; atomicMax(reinterpret_cast<int*>(&wmax), __float_as_int(a)); }
    }
    __syncthreads();
    if (tid < kC) {
      float* dst = (kC == 1) ? lmax : cluster.map_shared_rank(lmax, tid);
      dst[crank] = wmax;
    }
    csync();
    float m = 0.f;
#pragma unroll
    for (int c = 0; c < kC; ++c) m = fmaxf(m, lmax[c]);
    return m;
  };

  const int nbe = nb + (nb & 1);
  const int brounds = nbe > 2 ? nbe - 1 : 1;
  int sweeps = 0;
  bool converged = (k < 2);
  for (; sweeps < kJMaxSweeps && !converged; ++sweeps) {
    const float max_n2 = refresh_norms();      // the running updates drift: exact norms every sweep
    const float dead2 = kJDead2 * max_n2, count2 = kJCount2 * max_n2;
    for (int round = 0; round < brounds; ++round) {
      for (int task = crank + kC * warp; task < nbe / 2; task += kC * nwarps) {
        int bi, bj;
        rr_pair2(nbe, round, task, bi, bj);
        const bool has_j = bj < nb;
        if (bi >= nb) continue;
        if (!has_j && round != 0) continue;
        float x[8][kEL];
        float nn[8];
        // where each of the 8 rows lives: an offset into X for a single CTA (fewer registers and
        // plain shared-memory addressing), a pointer that may lead to a peer's shared memory otherwise
        typename std::conditional<kC == 1, int, float*>::type ref[8];
        auto at = [&](int a) -> float* {
          if constexpr (kC == 1) return X + ref[a]; else return ref[a];
        };
#pragma unroll
        for (int a = 0; a < 8; ++a) {
          const int row = (a < 4 ? bi * 4 + a : bj * 4 + (a - 4));
          const bool in = row < k && (a < 4 || has_j);
          if constexpr (kC == 1) ref[a] = in ? row * ld : 4 * nbl * ld;
          else ref[a] = in ? row_ptr(row) : zrow;
        }
        const bool full = (r == 32 * kEL);       // every lane element exists: no per-element checks
#pragma unroll
        for (int a = 0; a < 8; ++a) {
          const float* rp = at(a);
          nn[a] = rp[r];
          if (full) {
#pragma unroll
            for (int e = 0; e < kEL; ++e) x[a][e] = rp[lane + 32 * e];
          } else {
#pragma unroll
            for (int e = 0; e < kEL; ++e) {
              const int t = lane + 32 * e;
              x[a][e] = (t < r) ? rp[t] : 0.f;
            }
          }
        }
        unsigned counted = 0u;                  // largest squared cosine among the pairs rotated here (float bits)
#pragma unroll
        for (int stp = 0; stp < 7; ++stp) {     // fully unrolled: every register index below is a constant
          if (stp >= 4 && round != 0) break;
          // pairs of this step: cross steps pair row a with row 4 + (a + stp) % 4; the three extra
          // steps of round 0 are the rest of an 8-player tournament (pairs inside the blocks)
          float g[4], c[4], sn[4];
          int pa[4], pb[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (stp < 4) { pa[u] = u; pb[u] = 4 + ((u + stp) & 3); }
            else if (stp == 4) { pa[u] = (u < 2) ? 0 + 2 * u : 4 + 2 * (u - 2); pb[u] = pa[u] + 1; }          // (0,1)(2,3)(4,5)(6,7)
            else if (stp == 5) { pa[u] = (u < 2) ? u : 4 + (u - 2); pb[u] = pa[u] + 2; }                         // (0,2)(1,3)(4,6)(5,7)
            else { pa[u] = (u < 2) ? u : 4 + (u - 2); pb[u] = (u < 2) ? 3 - u : 7 - (u - 2); }                  // (0,3)(1,2)(4,7)(5,6)
            g[u] = 0.f;
          }
          // dot products (register indices are resolved by full unrolling over the 8 x 8 choices)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
              for (int bb = 0; bb < 8; ++bb)
                if (a == pa[u] && bb == pb[u]) {
#pragma unroll
                  for (int e = 0; e < kEL; ++e) g[u] = fmaf(x[a][e], x[bb][e], g[u]);
                }
          }
          // four sums across the warp in 6 shuffles: each exchange halves what a lane still carries
          // (two of the four values after the first, one after the second); the lanes of octet u
          // (lanes 8u .. 8u+7) end up with the whole of g[u]
          float gsum;
          {
            const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
            float k0 = h16 ? g[2] : g[0], k1 = h16 ? g[3] : g[1];
            const float s0 = h16 ? g[0] : g[2], s1 = h16 ? g[1] : g[3];
            k0 += __shfl_xor_sync(0xffffffffu, s0, 16);
            k1 += __shfl_xor_sync(0xffffffffu, s1, 16);
            gsum = h8 ? k1 : k0;
            const float sd = h8 ? k0 : k1;
            gsum += __shfl_xor_sync(0xffffffffu, sd, 8);
            gsum += __shfl_xor_sync(0xffffffffu, gsum, 4);
            gsum += __shfl_xor_sync(0xffffffffu, gsum, 2);
            gsum += __shfl_xor_sync(0xffffffffu, gsum, 1);
          }
          // rotation parameters: the lanes of octet u work out pair u, then the results are broadcast
          float appv[4], aqqv[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            appv[u] = 0.f; aqqv[u] = 0.f;
#pragma unroll
            for (int a = 0; a < 8; ++a) { if (a == pa[u]) appv[u] = nn[a]; if (a == pb[u]) aqqv[u] = nn[a]; }
          }
          const int lu = lane >> 3;
          const float my_g = gsum;
          const float my_app = lu == 0 ? appv[0] : lu == 1 ? appv[1] : lu == 2 ? appv[2] : appv[3];
          const float my_aqq = lu == 0 ? aqqv[0] : lu == 1 ? aqqv[1] : lu == 2 ? aqqv[2] : aqqv[3];
          const bool my_act = my_app > dead2 && my_aqq > dead2 && my_app > 0.f && my_aqq > 0.f &&
                              my_g * my_g > tol * tol * my_app * my_aqq;
          float my_c = 1.f, my_s = 0.f, my_dn = 0.f;
          if (my_act) {
            float zeta = __fdividef(my_aqq - my_app, 2.f * my_g);
            zeta = fminf(fmaxf(zeta, -1e15f), 1e15f);
            const float h = fmaf(zeta, zeta, 1.f);
            const float t1 = __fdividef(copysignf(1.f, zeta), fabsf(zeta) + h * rsqrtf(h));
            my_c = rsqrtf(fmaf(t1, t1, 1.f));
            my_s = my_c * t1;
            my_dn = t1 * my_g;
          }
          const bool my_counted = my_act && my_app > count2 && my_aqq > count2;
          const float my_cos2 = my_counted ? __fdividef(my_g * my_g, my_app * my_aqq) : 0.f;
          counted = max(counted, __reduce_max_sync(0xffffffffu, __float_as_uint(my_cos2)));
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            c[u] = __shfl_sync(0xffffffffu, my_c, 8 * u);
            sn[u] = __shfl_sync(0xffffffffu, my_s, 8 * u);
            const float dn = __shfl_sync(0xffffffffu, my_dn, 8 * u);
#pragma unroll
            for (int a = 0; a < 8; ++a) { if (a == pa[u]) nn[a] = appv[u] - dn; if (a == pb[u]) nn[a] = aqqv[u] + dn; }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
              for (int bb = 0; bb < 8; ++bb)
                if (a == pa[u] && bb == pb[u]) {
#pragma unroll
                  for (int e = 0; e < kEL; ++e) {
                    const float xp = x[a][e], xq = x[bb][e];
                    x[a][e] = c[u] * xp - sn[u] * xq;
                    x[bb][e] = sn[u] * xp + c[u] * xq;
                  }
                }
          }
        }
#pragma unroll
        for (int a = 0; a < 8; ++a) {
          float* rp = at(a);
          if (full) {
#pragma unroll
            for (int e = 0; e < kEL; ++e) rp[lane + 32 * e] = x[a][e];
          } else {
#pragma unroll
            for (int e = 0; e < kEL; ++e) {
              const int t = lane + 32 * e;
              if (t < r) rp[t] = x[a][e];
            }
          }
          if (lane == 0) rp[r] = nn[a];
        }
        if (lane == 0 && counted) atomicMax(&wflag, (int)counted);
      }
      csync();                          // all rows of this round are back in place
    }
    if (tid < kC) {
      int* dst = (kC == 1) ? lflag : cluster.map_shared_rank(lflag, tid);
      dst[crank] = wflag;
    }
    csync();
    int any = 0;
#pragma unroll
    for (int c = 0; c < kC; ++c) any = max(any, lflag[c]);
    converged = (__int_as_float(any) <= kJEarly2);     // nothing rotated, or only by angles whose square is noise
  }

  // norms, descending order, unit rows: each CTA finishes the rows it holds
  const float max_n2 = refresh_norms();
  for (int lr = tid; lr < nlocal; lr += nthreads) {
    const int gi = global_row(lr);
    if (gi >= k) continue;
    const float li = X[lr * ld + r];
    int rk = 0;
    for (int j = 0; j < k; ++j) { const float lj = row_ptr(j)[r]; rk += (lj > li) || (lj == li && j < gi); }
    rank[lr] = rk;
  }
  __syncthreads();
  const float dead2 = kJDead2 * max_n2;
  for (int lr = warp; lr < nlocal; lr += nwarps) {
    if (global_row(lr) >= k) continue;
    const float a = X[lr * ld + r];
    const bool live = a > dead2 && a > 0.f;
    const float nrm = live ? sqrtf(a) : 0.f, inv = live ? 1.f / nrm : 0.f;
    float* dst = job.rows + (size_t)rank[lr] * r;
    for (int t = lane; t < r; t += 32) dst[t] = X[lr * ld + t] * inv;
    if (lane == 0) job.norms[rank[lr]] = nrm;
  }
  if (crank == 0 && tid == 0 && job.status) *job.status = converged ? AB_OK : AB_ERR_NOT_CONVERGED;
  csync();                              // nobody leaves while a peer may still read its rows
}

size_t jacobi_smem_bytes(int k, int r, int C) {
  const int nbl = ((k + 3) / 4 + C - 1) / C;
  return sizeof(float) * ((size_t)(4 * nbl + 1) * (r + 1) + C) + sizeof(int) * ((size_t)C + 4 * nbl) + 64;
}

template <int EL, int C>
cudaLaunchConfig_t jacobi_config(int count, int rmax, cudaStream_t st, cudaLaunchAttribute* attr) {
  const int tasks = ((rmax + 3) / 4 + 1) / 2;                         // block pairs per round
  const int max_warps = (C == 1 && EL == 6) ? 24 : 16;              // matches the kernel's launch bounds
  const int warps = std::max(1, std::min(max_warps, (tasks + C - 1) / C));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(count * C));
  cfg.blockDim = dim3((unsigned)(32 * warps));
  cfg.dynamicSmemBytes = jacobi_smem_bytes(rmax, rmax, C);
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cfg;
}
// Launches with clusters of C CTAs if `count` such clusters can be resident at once (or if C == 1).
// Returns 1 when it declined, so that the caller tries a narrower cluster.
template <int EL, int C>
int try_launch_jacobi(const JacobiJob* jobs, int count, int rmax, float tol, cudaStream_t st) {
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = jacobi_config<EL, C>(count, rmax, st, attr);
  if (cfg.dynamicSmemBytes > (size_t)(kMaxSmem - kStatics)) return C == 1 ? AB_ERR_UNSUPPORTED : 1;
  AB_CUDA_OK(allow_smem(jacobi_rows_cluster_kernel<EL, C>, kStatics));
  if (C > 1) {
    // one CTA per SM: CTAs that share an SM would only take turns on its issue slots
    int resident = 0;
    const int sms = sm_count();
    if (sms <= 0) return AB_ERR_CUDA;
    if (rmax < 16 * C || (long long)count * C > sms) return 1;
    if (cudaOccupancyMaxActiveClusters(&resident, jacobi_rows_cluster_kernel<EL, C>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      return 1;
    }
    if (resident < count) return 1;
  }
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  AB_CUDA_OK(cudaLaunchKernelEx(&cfg, jacobi_rows_cluster_kernel<EL, C>, jobs, tol));
  AB_LAUNCH_OK();
  return AB_OK;
}
// Clusters of 8 or 4 CTAs per matrix when that many SMs are free for every matrix, else one CTA each
// (measured: a pair of CTAs gains nothing over one CTA with twice the warps; the round time is then
// set by the latency of one warp's 16 rotations, not by issue slots).
template <int EL>
int launch_jacobi_el(const JacobiJob* jobs, int count, int rmax, float tol, cudaStream_t st) {
  int s = try_launch_jacobi<EL, 8>(jobs, count, rmax, tol, st);
  if (s == 1) s = try_launch_jacobi<EL, 4>(jobs, count, rmax, tol, st);
  if (s == 1) s = try_launch_jacobi<EL, 1>(jobs, count, rmax, tol, st);
  if (s == AB_ERR_UNSUPPORTED) {            // too large for one CTA's shared memory: two CTAs hold half each
    s = try_launch_jacobi<EL, 2>(jobs, count, rmax, tol, st);
    if (s == 1) s = AB_ERR_UNSUPPORTED;
  }
  return s;
}
int launch_jacobi(const JacobiJob* jobs, int count, int rmax, float tol, cudaStream_t st) {
  if (rmax <= 64) return launch_jacobi_el<2>(jobs, count, rmax, tol, st);
  if (rmax <= 128) return launch_jacobi_el<4>(jobs, count, rmax, tol, st);
  if (rmax <= 192) return launch_jacobi_el<6>(jobs, count, rmax, tol, st);
  return launch_jacobi_el<8>(jobs, count, rmax, tol, st);
}

constexpr int kTaskRows = 4;     // rows of a step of the elimination below a panel
constexpr int kCPanel = 8;       // rows per panel of the Cholesky elimination (kCThreads / 64)

struct CholJob {
  const float* G;   // nparts partial sums of an r x r symmetric positive semi-definite matrix (row stride r,
                    // r * r apart); only the upper triangle is read
  int nparts;
  float* R;         // r x r upper triangular, G = R^T R; zeros below the diagonal, dropped rows zero
  float* Rinv;      // r x r upper triangular inverse of the kept part; dropped rows and columns zero
  int* status;      // receives AB_OK (may be null)
  int r;
};

// 1 / sqrt(x) to about one unit in the last place: one Newton step on the hardware's approximation.  The pivots follow from one
// another, and a square root and a division cost 400 cycles of that chain.
__device__ __forceinline__ float rsqrt_close(float x) {
  const float y = rsqrtf(x);
  return fmaf(0.5f * y, fmaf(-x * y, y, 1.f), y);
}
// Right-looking Cholesky of one Gram matrix in shared memory (r <= 256), then the inverse of the
// triangle by back substitution, four columns per warp at a time.  R lives in the upper triangle; column j of
// the inverse is parked in the strict lower triangle of row j (contiguous), its diagonal in dinv[].
// 144 matrices of 192 rows, one CTA each (us): 228 -> 138; the factor 232000 -> 154000 cycles, of them 64000 in the panels'
// chains of pivots and 90000 below them, bound by shared memory; the inverse 134000 -> 60000.
__global__ void __launch_bounds__(kCThreads, 1) chol_inv_kernel(const CholJob* __restrict__ jobs) {
  extern __shared__ __align__(16) float sm[];
  tc::dep_wait();
  tc::dep_launch();
  const CholJob job = jobs[blockIdx.x];
  const int r = job.r, ld = r + 1;
  float* S = sm;                       // r x ld
  float* dinv = S + (size_t)r * ld;    // r
  __shared__ float maxdiag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nwarps = kCThreads / 32;

  __shared__ int dropped_live;          // pivots taken as zero although they were not exactly zero
  if (tid == 0) { maxdiag = 0.f; dropped_live = 0; }
  {
    const float* __restrict__ G = job.G;
    const size_t part = (size_t)r * r;
    if ((r & 3) == 0 && (reinterpret_cast<uintptr_t>(G) & 15u) == 0) {
      // groups of four values of the upper triangle, four a thread and three parts at a time: up to twelve 16-byte loads in flight
      const int rc = r >> 2, n = r * rc;
      const size_t part4 = part >> 2;
      const float4* G4 = reinterpret_cast<const float4*>(G);
      for (int c0 = tid; c0 < n; c0 += 4 * kCThreads) {
        float4 v[4];
        int at[4];                                               // place in S, or -1
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int c = c0 + u * kCThreads, row = c / rc, col = 4 * (c - row * rc);
          at[u] = c < n && col + 3 >= row ? row * ld + col : -1;
          v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int q0 = 0; q0 < job.nparts; q0 += 3) {             // ascending part order
          float4 t[3][4];
#pragma unroll
          for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              t[q][u] = make_float4(0.f, 0.f, 0.f, 0.f);
              if (at[u] >= 0 && q0 + q < job.nparts) t[q][u] = __ldcg(G4 + (q0 + q) * part4 + c0 + u * kCThreads);
            }
#pragma unroll
          for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int u = 0; u < 4; ++u) { v[u].x += t[q][u].x; v[u].y += t[q][u].y; v[u].z += t[q][u].z; v[u].w += t[q][u].w; }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (at[u] >= 0) { S[at[u]] = v[u].x; S[at[u] + 1] = v[u].y; S[at[u] + 2] = v[u].z; S[at[u] + 3] = v[u].w; }
      }
    } else
    for (int i0 = 2 * warp; i0 < r; i0 += 2 * nwarps) {           // two rows per warp; the loads of both are all in flight
      float v[2][8];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 8; ++e) v[h][e] = 0.f;
      for (int q = 0; q < job.nparts; ++q) {                                       // ascending part order
        float t[2][8];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (i0 + h < r && 32 * e + lane < r) t[h][e] = G[q * part + (size_t)(i0 + h) * r + 32 * e + lane];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (i0 + h < r && 32 * e + lane < r) v[h][e] = q == 0 ? t[h][e] : v[h][e] + t[h][e];
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (i0 + h < r && 32 * e + lane < r) S[(i0 + h) * ld + 32 * e + lane] = v[h][e];
    }
  }
  __syncthreads();
  for (int i = tid; i < r; i += kCThreads)
    atomicMax(reinterpret_cast<int*>(&maxdiag), __float_as_int(fmaxf(S[i * ld + i], 0.f)));
  __syncthreads();
  const float cut = kEigThr * maxdiag;

  // Panels of kCPanel rows.  Every thread eliminates the panel's diagonal block for itself, in registers, and takes its own
  // column through it beside that: two barriers a panel, not two a row.  Then all rows below the panel take its kCPanel
  // rank-one terms in one pass, in ascending j -- the same sums per entry as a column-by-column elimination.
  for (int j0 = 0; j0 < r; j0 += kCPanel) {
    const int np = (r - j0 < kCPanel) ? r - j0 : kCPanel, jend = j0 + np;
    const int k = j0 + tid;                // r <= 256 <= kCThreads: one column a thread
    float d[kCPanel][kCPanel], p[kCPanel];
    if (k < r) {
#pragma unroll
      for (int a = 0; a < kCPanel; ++a) {
        p[a] = a < np ? S[(j0 + a) * ld + k] : 0.f;
#pragma unroll
        for (int b = a; b < kCPanel; ++b) d[a][b] = b < np ? S[(j0 + a) * ld + j0 + b] : 0.f;
      }
    }
    __syncthreads();
    if (k < r) {
#pragma unroll
      for (int q = 0; q < kCPanel; ++q) {
        const float dj = d[q][q];
        const bool live = dj > cut && dj > 0.f;
        const float inv = live ? rsqrt_close(dj) : 0.f;
        if (q < np) {
          if (k > j0 + q) {
            p[q] *= inv;                                                          // a dropped row becomes zero
            S[(j0 + q) * ld + k] = p[q];
          } else if (k == j0 + q) {
            S[k * ld + k] = dj * inv;
            dinv[k] = inv;
            if (!live && dj != 0.f) dropped_live = 1;
          }
        }
#pragma unroll
        for (int b = q + 1; b < kCPanel; ++b) d[q][b] *= inv;
#pragma unroll
        for (int a = q + 1; a < kCPanel; ++a) {
          p[a] = fmaf(-d[q][a], p[q], p[a]);
#pragma unroll
          for (int b = a; b < kCPanel; ++b) d[a][b] = fmaf(-d[q][a], d[q][b], d[a][b]);
        }
      }
    }
    __syncthreads();
    if (jend >= r) break;
    // steps of kTaskRows rows x 64 columns, a multiplier read once for two columns a lane; not the last panel: np == kCPanel
    const int nrg = (r - jend + kTaskRows - 1) / kTaskRows, ntasks = nrg * ((r + 63) >> 6);
    for (int t = warp; t < ntasks; t += nwarps) {
      const int cb = t / nrg, i0 = jend + (t - cb * nrg) * kTaskRows, c0 = 64 * cb + lane, c1 = c0 + 32;
      if (c0 - lane + 63 < i0) continue;
      float pk0[kCPanel], pk1[kCPanel], acc0[kTaskRows], acc1[kTaskRows];
#pragma unroll
      for (int q = 0; q < kCPanel; ++q) {
        pk0[q] = c0 < r ? S[(j0 + q) * ld + c0] : 0.f;
        pk1[q] = c1 < r ? S[(j0 + q) * ld + c1] : 0.f;
      }
#pragma unroll
      for (int h = 0; h < kTaskRows; ++h) {
        acc0[h] = (c0 >= i0 + h && c0 < r) ? S[(i0 + h) * ld + c0] : 0.f;
        acc1[h] = (c1 >= i0 + h && c1 < r) ? S[(i0 + h) * ld + c1] : 0.f;
      }
#pragma unroll
      for (int h = 0; h < kTaskRows; ++h) {
        const int i = i0 + h < r ? i0 + h : r - 1;
#pragma unroll
        for (int q = 0; q < kCPanel; ++q) {
          const float f = S[(j0 + q) * ld + i];
          acc0[h] = fmaf(-f, pk0[q], acc0[h]);
          acc1[h] = fmaf(-f, pk1[q], acc1[h]);
        }
      }
#pragma unroll
      for (int h = 0; h < kTaskRows; ++h) {
        if (c0 >= i0 + h && c0 < r) S[(i0 + h) * ld + c0] = acc0[h];
        if (c1 >= i0 + h && c1 < r) S[(i0 + h) * ld + c1] = acc1[h];
      }
    }
    __syncthreads();
  }

  // X = R^-1 restricted to the kept rows, one warp per column j, by back substitution in update
  // form: lane l owns rows l, l + 32, ... of the column.  b starts as e_j; going down from k = j,
  // x_k = b_k / R_kk is final (one shuffle hands it to all lanes) and every row i < k takes
  // b_i -= R_ik x_k -- no reduction across lanes, and only the upper triangle (R) is read.
  // Four neighbouring columns at a time: what a step reads of R serves all four, and their chains of shuffle and update hide one
  // another's latency.  A column's entries below its j stay zero, so its steps above j change nothing.
  {
    float dk[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) dk[e] = (32 * e + lane < r) ? dinv[32 * e + lane] : 0.f;
    const int ngroups = (r + 3) >> 2;
    for (int t = 0; t * nwarps < ngroups; ++t) {
      const int gi = t * nwarps + ((t & 1) ? nwarps - 1 - warp : warp);       // long and short columns shared out
      if (gi >= ngroups) continue;
      const int j0 = 4 * gi, jtop = (j0 + 3 < r - 1) ? j0 + 3 : r - 1;
      float b[4][8];
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int e = 0; e < 8; ++e) b[c][e] = (32 * e + lane == j0 + c) ? 1.f : 0.f;
#pragma unroll
      for (int e = 7; e >= 0; --e) {
        if (32 * e > jtop) continue;                  // uniform over the warp
        const int ltop = (jtop - 32 * e < 31) ? jtop - 32 * e : 31;
        for (int l = ltop; l >= 0; --l) {
          const int k = 32 * e + l;
          float xk[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            xk[c] = __shfl_sync(0xffffffffu, b[c][e] * dk[e], l);
            if (lane == l) b[c][e] = xk[c];
          }
#pragma unroll
          for (int e2 = 0; e2 <= e; ++e2) {
            const int i = 32 * e2 + lane;
            if (i < k) {
              const float Sik = S[i * ld + k];
#pragma unroll
              for (int c = 0; c < 4; ++c) b[c][e2] = fmaf(-Sik, xk[c], b[c][e2]);
            }
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int i = 32 * e + lane;
          if (j0 + c < r && i < j0 + c) S[(j0 + c) * ld + i] = b[c][e];           // column j of X, parked in row j below the diagonal
        }
    }
  }
  __syncthreads();
  for (int i = warp; i < r; i += nwarps) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int k = 32 * e + lane;
      if (k < r) {
        job.R[(size_t)i * r + k] = (k >= i) ? S[i * ld + k] : 0.f;
        job.Rinv[(size_t)i * r + k] = (k > i) ? S[k * ld + i] : (k == i ? dinv[i] : 0.f);
      }
    }
  }
  if (tid == 0 && job.status) *job.status = dropped_live ? (int)AB_ERR_ACCURACY : (int)AB_OK;
}

size_t chol_smem_bytes(int r) { return sizeof(float) * ((size_t)r * (r + 1) + r) + 64; }

// r' = #{ i < r : sigma_i >= cutoff * sigma_0 } (at least 1); folds the three solver statuses.  A warp per matrix (one
// thread per matrix walked its values one load after the other: 31 us for 72 matrices of rank 192).
__global__ void __launch_bounds__(128)
fast_rank_rule_kernel(const float* const* __restrict__ sigma, const int* __restrict__ rs,
                      float cutoff, int* const* __restrict__ r_out,
                      const int* __restrict__ jstatus, int* __restrict__ dev_status, int L) {
  tc::dep_wait();
  tc::dep_launch();
  const int i = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= L) return;
  const float* sg = sigma[i];
  const int r = rs[i];
  float v[8], top = 0.f;               // r <= 256
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    v[e] = lane + 32 * e < r ? sg[lane + 32 * e] : 0.f;
    top = fmaxf(top, v[e]);
  }
  top = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(top)));
  int keep = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) keep += (lane + 32 * e < r && v[e] >= cutoff * top) ? 1 : 0;
  keep = max(1, __reduce_add_sync(0xffffffffu, keep));
  int low = 0;                         // a kept value below the accuracy domain
#pragma unroll
  for (int e = 0; e < 8; ++e) low |= (lane + 32 * e < keep && v[e] < kFDomainRel * top && v[e] > kFZeroRel * top) ? 1 : 0;
  low = __any_sync(0xffffffffu, low);
  if (lane != 0) return;
  *r_out[i] = keep;
  if (dev_status) {
    int st = low ? AB_ERR_ACCURACY : AB_OK;
    for (int j = 0; j < 3; ++j) if (jstatus[3 * i + j] == AB_ERR_ACCURACY) st = AB_ERR_ACCURACY;
    for (int j = 0; j < 3; ++j)          // a solver that did not converge outranks the accuracy note
      if (jstatus[3 * i + j] != AB_OK && jstatus[3 * i + j] != AB_ERR_ACCURACY) st = jstatus[3 * i + j];
    dev_status[i] = st;
  }
}

// A bounded wait that ran out inside one of the tensor-core launches or the eigensolver of the call reaches every matrix's status.
__global__ void fold_tc_status_kernel(const int* __restrict__ tc_status, int* __restrict__ dev_status, int L) {
  tc::dep_wait();
  tc::dep_launch();
  int bad = AB_OK;
  for (int k = 0; k < 4; ++k) if (tc_status[k] != AB_OK) bad = tc_status[k];
  if (bad == AB_OK) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < L; i += gridDim.x * blockDim.x) dev_status[i] = bad;
}

// The long index of a Gram product is cut into slices, whose partial sums the Cholesky kernel adds in ascending order.  Short ones
// give a few matrices more CTAs for the product (2 us a slab of 64 with its start and end), long ones leave the one CTA that adds
// them less to load (22 us a part of rank 192, 2.4 of rank 64): 8 r, and no shorter than gives every SM a tile, from 128 (two slabs)
// to 768, at most kGramMaxParts slices.  Group sync, us, slices of 128 / 256 / 512 / 768: 3072 x 768, rank 192 776 / 727 / 662 / 643;
// 3072 x 3072, rank 128 494 / 473 / 454 / 453; 512 x 4608, rank 64 231 / 230 / 226 / 230; 3072 x 3072, rank 32 158 / 159 / 162 / 163; 3072 x 64,
// rank 16 129 / 132 / 133 / 139; all of ViT-B/16 1935 / 1755 / 1581 / 1548; 100 of 3072 x 3072, rank 32 at 256 / 768: 565 / 539.
constexpr int kGramMaxParts = 16;
int gram_fill(const ab_sync_desc* d, int L) {       // the slice length with which every SM has a tile
  int64_t work = 0;                     // tiles x length
  for (int i = 0; i < L; ++i) {
    const int64_t t = (d[i].r + 127) / 128;
    work += t * (t + 1) / 2 * ((int64_t)d[i].m + d[i].n);
  }
  return (int)std::min<int64_t>(768, (work / std::max(sm_count(), 1) + 63) / 64 * 64);
}
int gram_slice(int r, int fill) { return std::max(128, std::min(768, std::max(8 * r, fill))); }
int gram_per(int len, int slice) {      // length of a part, a multiple of 64
  const int parts = std::max(1, std::min(kGramMaxParts, (len + slice - 1) / slice));
  return ((len + parts - 1) / parts + 63) / 64 * 64;
}
int gram_parts(int len, int slice) { const int per = gram_per(len, slice); return (len + per - 1) / per; }

struct FastWs {
  std::vector<float*> Abar, Bbar, GA, GB, RA, RB, IA, IB, M, Vs, Y1, ZA, ZB;
  SplitGemm* gemms;     // the products of all launches, one after the other: up to (2 kGramMaxParts + 7) L
  CholJob* cjobs;       // 2 L
  AvgJob* ajobs;        // 2 L
  JacobiJob* jobs;      // L
  EigJob* ejobs;        // L
  int* jstatus;         // 3 L
  const float** sig_ptrs;
  int** rout_ptrs;
  int* rs;
  int* tc_status;       // 64 (what the products' and the eigensolver's waits report), and behind them one fallback flag per matrix (see EigJob)
  std::vector<double*> eig;   // scratch of the eigensolver
  size_t bytes;
};

FastWs fast_layout(const ab_sync_desc* d, int L, void* ws) {
  FastWs w;
  Arena ar(ws, 0);
  const int fill = gram_fill(d, L);
  auto each = [&](std::vector<float*>& v, auto count) {
    v.resize(L);
    for (int i = 0; i < L; ++i) v[i] = ar.take_n<float>(count(d[i]));
  };
  each(w.Abar, [](const ab_sync_desc& x) { return (size_t)x.m * x.r; });
  each(w.Bbar, [](const ab_sync_desc& x) { return (size_t)x.r * x.n; });
  auto rr = [](const ab_sync_desc& x) { return (size_t)x.r * x.r; };
  each(w.GA, [=](const ab_sync_desc& x) { return (size_t)gram_parts(x.m, gram_slice(x.r, fill)) * x.r * x.r; });
  each(w.GB, [=](const ab_sync_desc& x) { return (size_t)gram_parts(x.n, gram_slice(x.r, fill)) * x.r * x.r; });
  each(w.RA, rr); each(w.RB, rr); each(w.IA, rr); each(w.IB, rr);
  each(w.M, rr); each(w.Vs, rr); each(w.Y1, rr); each(w.ZA, rr); each(w.ZB, rr);
  size_t ngemm = (size_t)7 * L;
  for (int i = 0; i < L; ++i) ngemm += gram_parts(d[i].m, gram_slice(d[i].r, fill)) + gram_parts(d[i].n, gram_slice(d[i].r, fill));
  w.gemms = ar.take_n<SplitGemm>(ngemm);
  w.cjobs = ar.take_n<CholJob>((size_t)2 * L);
  w.ajobs = ar.take_n<AvgJob>((size_t)2 * L);
  w.jobs = ar.take_n<JacobiJob>((size_t)L);
  w.ejobs = ar.take_n<EigJob>((size_t)L);
  w.jstatus = ar.take_n<int>((size_t)3 * L);
  w.sig_ptrs = ar.take_n<const float*>(L);
  w.rout_ptrs = ar.take_n<int*>(L);
  w.rs = ar.take_n<int>(L);
  w.tc_status = ar.take_n<int>(64 + (size_t)L);
  w.eig.resize(L);
  for (int i = 0; i < L; ++i) w.eig[i] = ar.take_n<double>(eig_ws_doubles(d[i].r));
  w.bytes = align_up(ar.used, 256);
  return w;
}

SplitGemm product(const void* A, int64_t lda, int a_mn, const void* B, int64_t ldb, int b_mn, void* C, int64_t ldc, int M, int N,
                  int K) {
  SplitGemm g;
  std::memset(&g, 0, sizeof(g));
  g.A = A; g.lda = lda; g.a_mn = a_mn; g.B = B; g.ldb = ldb; g.b_mn = b_mn; g.C = C; g.ldc = ldc; g.M = M; g.N = N; g.K = K;
  g.thr = kEigThr;
  return g;
}

}  // namespace

// One helper stream per device (lowest priority, created on first use, kept for the life of the
// process): the optional product W = Abar Bbar depends only on the means, so it runs there beside the
// Cholesky and Jacobi kernels, which leave half of the SMs idle.
cudaStream_t side_stream() {
  static std::mutex mu;
  static cudaStream_t streams[64] = {};
  static bool tried[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!tried[dev]) {
    tried[dev] = true;
    int lo = 0, hi = 0;
    if (cudaDeviceGetStreamPriorityRange(&lo, &hi) != cudaSuccess ||
        cudaStreamCreateWithPriority(&streams[dev], cudaStreamNonBlocking, lo) != cudaSuccess) {
      (void)cudaGetLastError();
      streams[dev] = nullptr;
    }
  }
  return streams[dev];
}

float rows_jacobi_tol(int s) { return 5e-7f * sqrtf((float)s) < 4e-6f ? 4e-6f : 5e-7f * sqrtf((float)s); }

bool rows_jacobi_fits(int count, int s) {
  if (s < 1 || s > 256 || count < 1) return false;
  if (jacobi_smem_bytes(s, s, 1) <= kMaxSmem - kStatics) return true;
  const int sms = sm_count();
  return sms > 0 && (long long)count * 2 <= sms && s >= 32;
}

size_t rows_jacobi_scratch_bytes(int count) { return align_up((size_t)count * sizeof(JacobiJob), 256); }

int rows_jacobi(const float* X, float* rows, float* norms, int* status, size_t status_stride_bytes, const int* flags,
                int count, int s, void* scratch, cudaStream_t st) {
  std::vector<JacobiJob> jb((size_t)count);
  for (int j = 0; j < count; ++j) {
    int* stj = reinterpret_cast<int*>(reinterpret_cast<char*>(status) + (size_t)j * status_stride_bytes);
    jb[j] = JacobiJob{X + (size_t)j * s * s, rows + (size_t)j * s * s, norms + (size_t)j * s, stj, flags + j, s, s};
  }
  AB_TRY(upload_async(scratch, jb.data(), jb.size() * sizeof(JacobiJob), st));
  return launch_jacobi(static_cast<const JacobiJob*>(scratch), count, s, rows_jacobi_tol(s), st);
}

bool sync_factored_supported(const ab_sync_desc* d, int L) {
  // dynamic shared memory of the two single-CTA kernels, with room for their few static words
  const size_t cap = kMaxSmem - kStatics;
  for (int i = 0; i < L; ++i)
    if (chol_smem_bytes(d[i].r) > cap || jacobi_smem_bytes(d[i].r, d[i].r, 1) > cap) return false;
  return true;
}

size_t sync_factored_ws(const ab_sync_desc* d, int L) { return fast_layout(d, L, nullptr).bytes; }

int sync_factored(const ab_sync_desc* d, int L, int K, float sigma_cutoff, int dt, int* dev_status,
                  void* ws, size_t ws_bytes, cudaStream_t st) {
  FastWs w = fast_layout(d, L, ws);
  if (w.bytes > ws_bytes) return AB_ERR_WORKSPACE;
  if (!gemm_tc_available()) return AB_ERR_UNSUPPORTED;
  const int out_bf16 = (dt == AB_BF16) ? 1 : 0;
  const int fill = gram_fill(d, L);
  int rmax = 0;
  bool any_w = false;
  for (int i = 0; i < L; ++i) { rmax = std::max(rmax, d[i].r); any_w = any_w || d[i].W_out != nullptr; }
  // ---- host-built tables, uploaded together.  The products, by launch:
  enum { kGram, kM, kZ1, kZ2, kOut, kW, kLaunches };
  std::vector<SplitGemm> g[kLaunches];
  std::vector<CholJob> cj((size_t)2 * L);
  std::vector<JacobiJob> jb((size_t)L);
  std::vector<EigJob> ej((size_t)L);
  std::vector<const float*> sigp(L);
  std::vector<int*> routp(L);
  std::vector<int> rs(L);
  for (int i = 0; i < L; ++i) {
    const int m = d[i].m, n = d[i].n, r = d[i].r;
    float *Ab = w.Abar[i], *Bb = w.Bbar[i];
    // G_A = Abar^T Abar, G_B = Bbar Bbar^T, upper tiles only, in slices of the long index
    const int slice = gram_slice(d[i].r, fill), pa = gram_parts(m, slice), pb = gram_parts(n, slice);
    for (int q = 0; q < pa; ++q) {
      const int per = gram_per(m, slice), k0 = q * per, k1 = std::min(m, k0 + per);
      const float* src = Ab + (size_t)k0 * r;
      g[kGram].push_back(product(src, r, 1, src, r, 1, w.GA[i] + (size_t)q * r * r, r, r, r, k1 - k0));
      g[kGram].back().upper_only = 1;
    }
    for (int q = 0; q < pb; ++q) {
      const int per = gram_per(n, slice), k0 = q * per, k1 = std::min(n, k0 + per);
      g[kGram].push_back(product(Bb + k0, n, 0, Bb + k0, n, 0, w.GB[i] + (size_t)q * r * r, r, r, r, k1 - k0));
      g[kGram].back().upper_only = 1;
    }
    // M = R_A R_B^T
    g[kM].push_back(product(w.RA[i], r, 0, w.RB[i], r, 0, w.M[i], r, r, r, r));
    // Y1 = M Vs^T;  Z_B = diag(sqrt sig) Vs R_B^-T
    g[kZ1].push_back(product(w.M[i], r, 0, w.Vs[i], r, 0, w.Y1[i], r, r, r, r));
    g[kZ1].push_back(product(w.Vs[i], r, 0, w.IB[i], r, 0, w.ZB[i], r, r, r, r));
    g[kZ1].back().row_vec = d[i].sigma; g[kZ1].back().row_mode = 1;
    // Z_A = R_A^-1 Y1 diag(sig^-1/2)
    g[kZ2].push_back(product(w.IA[i], r, 0, w.Y1[i], r, 1, w.ZA[i], r, r, r, r));
    g[kZ2].back().col_vec = d[i].sigma; g[kZ2].back().col_mode = 2;
    // A' = Abar Z_A (columns at or beyond r' zero), B' = Z_B Bbar (rows at or beyond r' zero)
    g[kOut].push_back(product(Ab, r, 0, w.ZA[i], r, 1, d[i].A_out, r, m, r, r));
    g[kOut].back().c_bf16 = out_bf16; g[kOut].back().live_cols = d[i].r_out;
    g[kOut].push_back(product(w.ZB[i], r, 0, Bb, n, 1, d[i].B_out, n, r, n, r));
    g[kOut].back().c_bf16 = out_bf16; g[kOut].back().live_rows = d[i].r_out;
    if (d[i].W_out) g[kW].push_back(product(Ab, r, 0, Bb, n, 1, d[i].W_out, n, m, n, r));      // W = Abar Bbar
    cj[i] = CholJob{w.GA[i], pa, w.RA[i], w.IA[i], w.jstatus + 3 * i, r};
    cj[L + i] = CholJob{w.GB[i], pb, w.RB[i], w.IB[i], w.jstatus + 3 * i + 1, r};
    int* flag = w.tc_status + 64 + i;
    jb[i] = JacobiJob{w.M[i], w.Vs[i], d[i].sigma, w.jstatus + 3 * i + 2, flag, r, r};
    EigJob& q = ej[i];
    q.X = w.M[i]; q.gram = 1; q.s = r; q.need = r; q.rows = w.Vs[i]; q.vals = d[i].sigma; q.flag = flag;
    eig_bind(q, w.eig[i]);
    sigp[i] = d[i].sigma; routp[i] = d[i].r_out; rs[i] = r;
  }
  // All tables sit back to back in the workspace (gemms ... rs): one host image.
  SplitBatch batch[kLaunches];
  const SplitGemm* table[kLaunches];
  std::vector<AvgJob> aj((size_t)2 * L);
  int64_t avg_blocks = 0;            // flat grid of the batched mean: one 16-byte group per thread
  for (int i = 0; i < L; ++i) {
    aj[2 * i] = AvgJob{d[i].A_copies, d[i].strideA, (int64_t)d[i].m * d[i].r, w.Abar[i], 0};
    aj[2 * i + 1] = AvgJob{d[i].B_copies, d[i].strideB, (int64_t)d[i].r * d[i].n, w.Bbar[i], 0};
    for (int h = 0; h < 2; ++h) {
      aj[2 * i + h].first_block = avg_blocks;
      avg_blocks += average_job_blocks(aj[2 * i + h].count, dt);
    }
  }
  {
    char* base = reinterpret_cast<char*>(w.gemms);
    const size_t span = (size_t)(reinterpret_cast<char*>(w.rs + L) - base);
    std::vector<char> img(span, 0);
    auto put = [&](const void* dev_ptr, const void* src, size_t bytes) {
      std::memcpy(img.data() + (reinterpret_cast<const char*>(dev_ptr) - base), src, bytes);
    };
    SplitGemm* at = w.gemms;
    for (int k = 0; k < kLaunches; ++k) {
      batch[k] = gemm_split_plan(g[k].data(), (int)g[k].size());
      table[k] = at;
      put(at, g[k].data(), g[k].size() * sizeof(SplitGemm));
      at += g[k].size();
    }
    put(w.cjobs, cj.data(), cj.size() * sizeof(CholJob));
    put(w.ajobs, aj.data(), aj.size() * sizeof(AvgJob));
    put(w.jobs, jb.data(), jb.size() * sizeof(JacobiJob));
    put(w.ejobs, ej.data(), ej.size() * sizeof(EigJob));
    put(w.sig_ptrs, sigp.data(), L * sizeof(float*));
    put(w.rout_ptrs, routp.data(), L * sizeof(int*));
    put(w.rs, rs.data(), L * sizeof(int));
    AB_TRY(upload_async(base, img.data(), span, st));
  }

  // ---- a7: means of the K copies (fp32), all matrices in one launch
  AB_TRY(group_average_batched(w.ajobs, 2 * L, K, dt, avg_blocks, st));
  const float tol = rows_jacobi_tol(rmax);
  // a8 (optional): forked off where the Jacobi kernel starts (the kernels before it fill every SM
  // themselves), joined at the end
  cudaStream_t side = any_w ? side_stream() : nullptr;
  // the two events live for this call only; every return below destroys them (destroying an event that
  // has been recorded releases it once the recorded work is done)
  struct EventPair {
    cudaEvent_t fork = nullptr, join = nullptr;
    bool create() {
      if (cudaEventCreateWithFlags(&fork, cudaEventDisableTiming) == cudaSuccess &&
          cudaEventCreateWithFlags(&join, cudaEventDisableTiming) == cudaSuccess)
        return true;
      (void)cudaGetLastError();
      return false;
    }
    ~EventPair() {
      if (fork) cudaEventDestroy(fork);
      if (join) cudaEventDestroy(join);
    }
  } evs;
  if (side && !evs.create()) side = nullptr;
  cudaEvent_t fork = evs.fork, join = evs.join;
  auto run = [&](int k, int* status, cudaStream_t s2) -> int { return gemm_split_batched(table[k], batch[k], status, s2); };
  AB_CUDA_OK(cudaMemsetAsync(w.tc_status, 0, (64 + (size_t)L) * sizeof(int), st));          // wait reports and flags
  if (any_w && !side) AB_TRY(run(kW, w.tc_status + 2, st));
  AB_TRY(run(kGram, w.tc_status, st));
  const size_t csm = chol_smem_bytes(rmax);
  AB_CUDA_OK(allow_smem(chol_inv_kernel, kStatics));
  AB_TRY(launch_after(chol_inv_kernel, dim3((unsigned)(2 * L)), kCThreads, csm, 1, st, (const CholJob*)w.cjobs));       // R_A, R_B and inverses
  AB_TRY(run(kM, w.tc_status, st));
  int side_rc = AB_OK;
  if (side && cudaEventRecord(fork, st) != cudaSuccess) side_rc = AB_ERR_CUDA;
  AB_TRY(eig_direct(ej.data(), w.ejobs, L, rmax, w.tc_status + 3, st));                                                 // SVD of M: right vectors, sigma
  AB_TRY(launch_jacobi(w.jobs, L, rmax, tol, st));                                          // of flagged matrices, from M
  if (side) {
    if (side_rc == AB_OK && cudaStreamWaitEvent(side, fork, 0) != cudaSuccess) side_rc = AB_ERR_CUDA;
    if (side_rc == AB_OK) side_rc = run(kW, w.tc_status + 2, side);
    if (side_rc == AB_OK && cudaEventRecord(join, side) != cudaSuccess) side_rc = AB_ERR_CUDA;
  }
  AB_TRY(launch_after(fast_rank_rule_kernel, dim3((unsigned)((L + 3) / 4)), 128, 0, 1, st, (const float* const*)w.sig_ptrs, (const int*)w.rs, sigma_cutoff,
                      (int* const*)w.rout_ptrs, (const int*)w.jstatus, dev_status, L));
  AB_TRY(run(kZ1, w.tc_status, st));
  AB_TRY(run(kZ2, w.tc_status, st));
  AB_TRY(run(kOut, w.tc_status + 1, st));
  if (side) {
    if (side_rc == AB_OK && cudaStreamWaitEvent(st, join, 0) != cudaSuccess) side_rc = AB_ERR_CUDA;
    if (side_rc != AB_OK) { (void)cudaGetLastError(); return side_rc; }
  }
  if (dev_status) {
    AB_TRY(launch_after(fold_tc_status_kernel, dim3(1), 128, 0, 1, st, (const int*)w.tc_status, dev_status, L));
  }
  return AB_OK;
}
}  // namespace ab
