// Direct eigensolver for symmetric matrices, batched: the r x r core of the factored group synchronisation and
// the Gram matrices of the dense split (short side up to eig_max()).
//
//   1. tridiag_small_kernel : Householder reduction C = H T H^T, order up to kEigSmallMax (a cluster of CTAs per
//      matrix, C in registers); tridiag_grid_kernel above that (eight rows of C in the registers of each CTA)
//   2. tri_values_kernel    : eigenvalues of T, multisection on Sturm counts
//   3. tri_vectors_kernel   : eigenvectors of T, twisted factorisation at each eigenvalue
//   4. back_transform_kernel: u = H z, rows sorted by descending eigenvalue, rounded to fp32
//
// Everything up to the last rounding is fp64.  C = M^T M is formed in fp64 from the fp32 matrix M, so an
// eigenvalue carries an absolute error of up to 4e-15 of the largest (2e-14 above order 256, where the words that cross the device
// keep 44 bits) and squaring costs no accuracy: a singular value of 1 % of the largest is good to 2e-11 before it is
// rounded to fp32.
//
// Why not the one-sided Jacobi that this replaces (it stays as the fallback, see below): its sweeps are chains of
// dependent steps -- s - 1 rounds a sweep, eight to thirteen sweeps, every step a dot product, a reduction across a warp, a
// rotation and a write-back -- while the reduction to tridiagonal form has s - 2 steps in all.
//
// Vectors of eigenvalues that are closer than about 1e-10 of the norm and not separated by a zero off-diagonal
// come out of step 3 less than orthogonal.  Step 4 checks every pair that is close and not null (one that is zero to
// the caller contributes nothing to either factor) and raises the matrix's flag when a pair fails; the caller then runs the Jacobi route for that matrix (a kernel that returns at once when
// the flag is clear).
#include <cooperative_groups.h>

#include <algorithm>

#include "ab_common.cuh"
#include "ab_tc_ptx.cuh"

namespace ab {
namespace {

namespace cg = cooperative_groups;

constexpr double kSplitRel = 2.3e-16;   // an off-diagonal below this fraction of the norm splits T
constexpr double kCloseRel = 1e-7;      // eigenvalues closer than this fraction of the norm are checked for orthogonality
constexpr double kOrthTol = 4e-6;       // what the Jacobi route leaves at small orders
constexpr int kMaxOrder = 1280;         // masks are sized for this order
constexpr double kLive2 = 1e-290;       // a column whose squared norm is below this needs no reflector
constexpr int kGroup = 8;               // reflectors applied together in the back transform
constexpr int kFewClose = 12;           // up to this many close vectors above one are compared with it one by one

// Reflectors are rows of an even number of doubles (bulk copies of whole rows start and end on 16 bytes), zero before and
// behind their elements.
__host__ __device__ __forceinline__ int refl_ld(int s) { return (s + 1) & ~1; }

// Eigenvalues (fractions of the norm) that carry nothing: a core's sigma below 1e-6 of the largest is zero to its
// caller; a Gram matrix that was rounded to fp32 has noise of 2^-24 of its entries for eigenvalues down there.
__device__ __forceinline__ double null_rel(const EigJob& job) { return job.gram ? 1e-12 : 1e-7; }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// 16 bytes to a CTA of the cluster; its barrier counts them.
__device__ __forceinline__ void st_async(uint32_t addr, double x, double y, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(addr), "d"(x), "d"(y),
               "r"(bar)
               : "memory");
}

// ---- 1. Householder reduction ---------------------------------------------------------------------------
// The matrix lives in registers: element (i, k) in warp i mod (warps of the cluster), lane k mod 32, so a warp
// holds R whole rows, E elements of each per lane.  Step j:
//   - warp 0 of each CTA has received p = A v of the reflector before (v, gamma) and column j of
//     the matrix as it was before that reflector's update, a;  w = gamma p - c v, c = gamma^2 p.v / 2;  column j of the updated
//     matrix is (a - x p) + y v with x = v1 gamma, y = 2 c v1 - gamma p_j, where v1 is the first element of v, and only y waits for a
//     sum.  w and the next reflector v' go to the other warps;
//   - all warps pass over their rows in registers: A -= v w^T + w v^T, p' = A v' without the first element of v';  every row's p'_i
//     and A[i][j+1] go to warp 0 of every CTA of the cluster;
//   - while they travel, warp 0 sums the squares of the column and takes their root, which gives the first element of v';  it adds that
//     element's products A[i][j+1] v1' to the p' that it receives.
// The squares are those of the column's own entries.  Sums over b = a - x p, known a reduction earlier (b.b + 2 y b.v + y^2 v.v), cancel:
// reflectors were then orthogonal to 1e-13 in place of 7e-16.  With the root in front of warp 0's pass a split of 256 x 2304 took 515 us
// against 503.
// So the rank-two update and the product with the next vector touch an element once, and a step is a chain of one
// warp reduction, the pass and one exchange.  The vectors are worked out by one warp because fp64 issues
// at half rate: with every warp doing it for itself (no hand-over) the copies took more issue slots than the pass (8100 cycles a step
// at order 192).  Finished 32-column groups are dropped at compile time (segment<E0>).
// The exchange is st.async onto an mbarrier of each receiver (two, used in turn): the data carry their own
// completion.  With a cluster barrier in its place, whose release also waits for the step's global stores, a step
// of order 256 (8 CTAs) took 2.6 us against 1.9 us (1.2 as the steps are now).  A CTA may overwrite a peer's buffer of step j once it has everything of step
// j + 1 from that peer: warp 0 of each CTA sends a 16-byte token once it has read its buffer.
// Where the matrix fits one CTA (kSingle) plain shared memory and named barriers take the place of the exchange.
constexpr int kMaxCl = 8;

__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

template <int E, int R, int W, bool kSingle>
struct Tridiag {
  static_assert(R % 4 == 0, "rows go through the warp reduction in fours");
  static constexpr int S = 32 * E;
  static constexpr int kChunk = 16;
  static constexpr int kThreads = 32 * W;
  struct Shared {
    double2 pa[2][S + kMaxCl];   // p and the next column; behind them the peers' tokens
    double2 stage_or_col[kChunk * S / 2];   // start: rows of X as fp64; afterwards each row warp's piece of column j + 1
    double v[2][S], w[S];
    double first[2];                        // v1 of the reflectors
    uint64_t bar[2];
    int dead;
  };

  Shared& sh;
  const EigJob& job;
  int s, CL, rank, warp, lane;
  int* status;

  struct Rows { double A[R][E]; double v[E]; double gam, v1; bool ok; uint32_t dst, dbar; };

  // Warp 0, step j: from p and the column to w and the next reflector but its first element (left in shared memory).  Returns
  // through vn, dj, alpha what is to be stored and what the first element and gamma follow from.
  template <int E0>
  __device__ __forceinline__ void vec_step(Rows& x, int j, double (&vn)[E], double& dj, double& alpha) {
    const int par = j & 1;
    if constexpr (kSingle) tc::named_bar_sync(2, kThreads);
    else x.ok = x.ok && tc::mbar_wait(&sh.bar[par], (j >> 1) & 1);
    const double2* pb = sh.pa[par];
    const double xg = x.v1 * x.gam;
    double p[E], pv = 0.0;
#pragma unroll
    for (int e = E0; e < E; ++e) {
      const double2 q = pb[lane + 32 * e];
      p[e] = fma(q.y, x.v1, q.x);
      vn[e] = fma(-xg, p[e], q.y);
      pv = fma(p[e], x.v[e], pv);
    }
    const int j1 = j + 1 < s ? j + 1 : j;
    const double2 qj = pb[j], qj1 = pb[j1];
    const double vj1 = sh.v[par][j1], pj = fma(qj.y, x.v1, qj.x), pj1 = fma(qj1.y, x.v1, qj1.x);
    pv = warp_sum(pv);
    const double c = 0.5 * x.gam * (x.gam * pv);    // gamma alone may be as large as 1e290
    const double y = 2.0 * c * x.v1 - x.gam * pj, wj = x.gam * pj - c * x.v1;
#pragma unroll
    for (int e = E0; e < E; ++e) {
      const bool ahead = e > E0 + 1 || lane + 32 * e > j + 1;
      sh.w[lane + 32 * e] = x.gam * p[e] - c * x.v[e];
      vn[e] = ahead ? fma(y, x.v[e], vn[e]) : 0.0;
      sh.v[par ^ 1][lane + 32 * e] = vn[e];
    }
    dj = qj.y - 2.0 * x.v1 * wj;
    alpha = (j + 1 < s) ? fma(y, vj1, fma(-xg, pj1, qj1.y)) : 0.0;
    if constexpr (!kSingle) {
      if (lane == 0 && !x.ok) sh.dead = 1;                 // a peer never answered: all warps leave
      if (x.ok && j + 1 < s) open_step(par ^ 1, s - 1 - j);
    }
  }
  // opens the barrier of buffer buf for the bytes of a step with n live rows; the token says that this CTA has
  // read the buffer of the step before
  __device__ __forceinline__ void open_step(int buf, int n) {
    if (lane == 0) tc::mbar_arrive_expect_tx(&sh.bar[buf], (uint32_t)(16 * (n + CL)));
    if (lane < CL) st_async(map_rank(tc::smem_u32(&sh.pa[buf][S + rank]), lane), 0.0, 0.0, map_rank(tc::smem_u32(&sh.bar[buf]), lane));
  }

  __device__ __forceinline__ void send(const Rows& x, int buf, int row, double p, double a) {
    if constexpr (kSingle) {
      if ((lane & 7) == 0) sh.pa[buf][row] = make_double2(p, a);
    } else {
      if ((lane & 7) < CL) st_async(x.dst + (uint32_t)((buf * (S + kMaxCl) + row) * 16), p, a, x.dbar + (uint32_t)(buf * 8));
    }
  }
  // steps whose first live column lies in the 32-column group E0; groups before it are finished
  template <int E0>
  __device__ __forceinline__ void segment(Rows& x) {
    const int gw = rank * W + warp, gs = CL * W;
    double* col = reinterpret_cast<double*>(sh.stage_or_col) + warp * R;
    const int jend = min(32 * E0 + 32, s);
    for (int j = 32 * E0; j < jend; ++j) {
      const int par = j & 1;
      double w[E], vn[E], dj = 0.0, alpha = 0.0, beta = 0.0, den = 0.0;
      if (warp == 0) vec_step<E0>(x, j, vn, dj, alpha);
      tc::named_bar_sync(1, kThreads);               // w and v' are there
      if (warp != 0 && lane == (j & 31)) x.v[E0] = sh.first[par];      // v of the step before was without its first element, j
      if constexpr (!kSingle) {
        if (*reinterpret_cast<volatile int*>(&sh.dead)) return;
      }
      if (gw + gs * (R - 1) > j) {                   // this warp still has a live row
#pragma unroll
        for (int e = E0; e < E; ++e) {
          w[e] = sh.w[lane + 32 * e];
          vn[e] = sh.v[par ^ 1][lane + 32 * e];
        }
#pragma unroll
        for (int g = 0; g < R / 4; ++g) {
          if (gw + gs * (4 * g + 3) <= j) continue;  // rows of a live group that are finished are updated for nothing
          double ps[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int r = 4 * g + q;
            const int i = min(gw + gs * r, S - 1);
            const double vi = sh.v[par][i], wi = sh.w[i];
            double acc = 0.0;
#pragma unroll
            for (int e = E0; e < E; ++e) {
              x.A[r][e] = fma(-vi, w[e], fma(-wi, x.v[e], x.A[r][e]));
              acc = fma(x.A[r][e], vn[e], acc);
            }
            ps[q] = acc;
          }
          if (lane == ((j + 1) & 31)) {              // column j + 1 of the rows
            const bool next = ((j + 1) >> 5) > E0;
#pragma unroll
            for (int q = 0; q < 4; ++q) col[4 * g + q] = (next && E0 + 1 < E) ? x.A[4 * g + q][E0 + 1 < E ? E0 + 1 : E0] : x.A[4 * g + q][E0];
          }
          __syncwarp();                              // other lanes send what this one wrote
          // four row sums across the warp, each exchange halving what a lane still carries: lanes 8 q .. hold sum q
          const bool h2 = (lane & 16) != 0, h1 = (lane & 8) != 0;
          double t0 = (h2 ? ps[2] : ps[0]) + __shfl_xor_sync(0xffffffffu, h2 ? ps[0] : ps[2], 16);
          double t1 = (h2 ? ps[3] : ps[1]) + __shfl_xor_sync(0xffffffffu, h2 ? ps[1] : ps[3], 16);
          double t = (h1 ? t1 : t0) + __shfl_xor_sync(0xffffffffu, h1 ? t0 : t1, 8);
          t += __shfl_xor_sync(0xffffffffu, t, 4);
          t += __shfl_xor_sync(0xffffffffu, t, 2);
          t += __shfl_xor_sync(0xffffffffu, t, 1);
          const int row = gw + gs * (4 * g + (lane >> 3));
          if (row > j && row < s) send(x, par ^ 1, row, t, col[4 * g + (lane >> 3)]);
        }
      }
      if constexpr (kSingle) { if (warp != 0) bar_arrive(2, kThreads); }
      if (warp == 0) {                               // beside the exchange: the first element, gamma, and what later kernels need
        double sq = 0.0;
#pragma unroll
        for (int e = E0; e < E; ++e) sq = fma(vn[e], vn[e], sq);
        sq = warp_sum(sq);
        const bool live = sq > kLive2;
        const double nrm = sqrt(fma(alpha, alpha, sq));
        beta = live ? (alpha > 0.0 ? -nrm : nrm) : alpha;
        x.v1 = live ? alpha - beta : 0.0;
        den = live ? nrm * (nrm + fabs(alpha)) : 0.0;
        if (lane == 0) sh.first[par ^ 1] = x.v1;     // for the other warps' next pass
        x.gam = den > 0.0 ? 1.0 / den : 0.0;
#pragma unroll
        for (int e = E0; e < E; ++e)
          if (e <= E0 + 1 && lane + 32 * e == j + 1) vn[e] = x.v1;
        if (rank == j % CL) {
          const int ld = refl_ld(s);
          double* dst = job.refl + (size_t)j * ld;
#pragma unroll
          for (int e = 0; e < E; ++e)
            if (lane + 32 * e < ld) dst[lane + 32 * e] = e < E0 ? 0.0 : vn[e];
          if (lane == 0) { job.d[j] = dj; job.e[j] = (j + 1 < s) ? beta : 0.0; job.gam[j] = x.gam; }
        }
      }
#pragma unroll
      for (int e = E0; e < E; ++e) x.v[e] = vn[e];
    }
    if constexpr (E0 + 1 < E) {
      if (32 * (E0 + 1) < s) segment<E0 + 1>(x);
    }
  }

  __device__ __forceinline__ void load_rows(Rows& x) {
    const int gw = rank * W + warp, gs = CL * W;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int e = 0; e < E; ++e) x.A[r][e] = 0.0;
    if (job.gram) {           // C = X^T X, rows of X staged a chunk at a time as fp64
      double (*stage)[S] = reinterpret_cast<double (*)[S]>(sh.stage_or_col);
      for (int t0 = 0; t0 < s; t0 += kChunk) {
        const int tn = min(kChunk, s - t0);
        tc::named_bar_sync(3, 32 * W);
        for (int idx = 32 * warp + lane; idx < tn * S; idx += 32 * W) {
          const int t = idx / S, k = idx - t * S;
          stage[t][k] = (k < s) ? (double)job.X[(size_t)(t0 + t) * s + k] : 0.0;
        }
        tc::named_bar_sync(3, 32 * W);
        for (int t = 0; t < tn; ++t) {
          double xk[E];
#pragma unroll
          for (int e = 0; e < E; ++e) xk[e] = stage[t][lane + 32 * e];
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const double xi = stage[t][min(gw + gs * r, S - 1)];
#pragma unroll
            for (int e = 0; e < E; ++e) x.A[r][e] = fma(xi, xk[e], x.A[r][e]);
          }
        }
      }
      tc::named_bar_sync(3, 32 * W);
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = gw + gs * r;
        if (i < s) {
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const int k = lane + 32 * e;
            if (k < s) x.A[r][e] = (double)job.X[(size_t)i * s + k];
          }
        }
      }
    }
  }

  __device__ __forceinline__ void run() {
    for (int i = threadIdx.x; i < S + kMaxCl; i += kThreads) sh.pa[0][i] = sh.pa[1][i] = make_double2(0.0, 0.0);
    for (int i = threadIdx.x; i < S; i += kThreads) sh.v[0][i] = sh.v[1][i] = sh.w[i] = 0.0;
    if (threadIdx.x == 0) {
      sh.dead = 0;
      sh.first[0] = sh.first[1] = 0.0;
      if (!kSingle) { tc::mbar_init(&sh.bar[0], 1); tc::mbar_init(&sh.bar[1], 1); tc::fence_barrier_init(); }
    }
    if constexpr (kSingle) __syncthreads(); else cg::this_cluster().sync();   // buffers and barriers are ready before a peer writes
    Rows x;
    load_rows(x);
#pragma unroll
    for (int e = 0; e < E; ++e) x.v[e] = 0.0;
    x.gam = 0.0; x.v1 = 0.0; x.ok = true;
    x.dst = x.dbar = 0;
    if constexpr (!kSingle) {
      const int c = (lane & 7) < CL ? (lane & 7) : 0;
      x.dst = map_rank(tc::smem_u32(&sh.pa[0][0]), c);
      x.dbar = map_rank(tc::smem_u32(&sh.bar[0]), c);
      if (warp == 0) open_step(0, s);
    }
    const int gw = rank * W + warp, gs = CL * W;
    double* col = reinterpret_cast<double*>(sh.stage_or_col) + warp * R;
    if (lane == 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) col[r] = x.A[r][0];
    }
    __syncwarp();
#pragma unroll
    for (int g = 0; g < R / 4; ++g) {
      const int row = gw + gs * (4 * g + (lane >> 3));
      if (row < s) send(x, 0, row, 0.0, col[4 * g + (lane >> 3)]);
    }
    __syncwarp();
    if constexpr (kSingle) { if (warp != 0) bar_arrive(2, kThreads); }
    segment<0>(x);
    if (!x.ok && lane == 0) atomicExch(status, (int)AB_ERR_TIMEOUT);
    if constexpr (!kSingle) cg::this_cluster().sync();         // nobody leaves while a peer may still send to it
  }
};

template <int E, int R, int W, bool kSingle>
__global__ void __launch_bounds__(32 * W, 1)
tridiag_small_kernel(const EigJob* __restrict__ jobs, int* status) {
  using T = Tridiag<E, R, W, kSingle>;
  extern __shared__ __align__(16) unsigned char tri_sm[];
  tc::dep_wait();
  // A batch leaves a few SMs empty, and the blocks of the kernel behind would crowd there (72 matrices of order 192: + 120 us).
  if (gridDim.x <= 32) tc::dep_launch();
  const int CL = kSingle ? 1 : (int)cg::this_cluster().num_blocks();
  const EigJob job = jobs[blockIdx.x / CL];
  T t{*reinterpret_cast<typename T::Shared*>(tri_sm), job, job.s, CL, kSingle ? 0 : (int)cg::this_cluster().block_rank(),
      (int)threadIdx.x >> 5, (int)threadIdx.x & 31, status};
  t.run();
}

// ---- 1b. Householder reduction over the whole device ------------------------------------------------------
// The same steps for orders a cluster cannot hold.  CTA c of the matrix's C (s / kGridRows, whole clusters) keeps rows c, c + C,
// ... in registers; thread t owns columns t, t + 256, ... of all of them, so the vectors are spread over the CTA (every
// CTA works out w and the next reflector for itself) and what crosses the device in a step is one (p_i, A[i][j+1]) pair per row.
// A pair is two 8-byte words, each carrying the step in its eight lowest mantissa bits (2^-44 of the value): a reader
// polls the words until the step matches, so data and signal are one trip through L2.  Every CTA needs all pairs, but
// each CTA of a cluster polls a share of them only and passes it on to the others (st.async onto a barrier of each receiver, two buffers
// in turn): all CTAs polling everything was 1.2 MB a round at order 768, and the rounds held up the stores they waited for (3.1 us a step).
// Who may overwrite what.  Buffers of a cluster: the barrier of step j + 1 counts a token of each CTA, sent once it
// has read step j.  Pairs in memory: a cluster stays until its last row is finished, so whoever has all pairs of step j + 1
// has one from every cluster that is still here, sent by a CTA that had all of step j, which its mates had read and passed on
// by then; the buffer of step j may be written (two buffers, cleared before the launch).
// All CTAs of a matrix have to be resident together: cooperative launch.  The waits are bounded.
constexpr int kGridRows = 8;

__device__ __forceinline__ double tag_word(double x, unsigned tag) {
  return __longlong_as_double((__double_as_longlong(x) & ~0xffll) | (long long)tag);
}
__device__ __forceinline__ unsigned word_tag(double x) { return (unsigned)__double2loint(x) & 0xffu; }
__device__ __forceinline__ double2 ld_relaxed(const double2* p) {
  double2 v;
  asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(double2* p, double x, double y) {
  asm volatile("st.relaxed.gpu.global.v2.f64 [%0], {%1, %2};" ::"l"(p), "d"(x), "d"(y) : "memory");
}
__device__ __forceinline__ unsigned step_tag(int j) { return 1u + (unsigned)(j % 255); }
// waits for the pair of a step; false after about a second
__device__ __forceinline__ bool poll_pair(const double2* p, unsigned tag, double2& v) {
  v = ld_relaxed(p);
  if (word_tag(v.x) == tag && word_tag(v.y) == tag) return true;
  const uint64_t t0 = tc::globaltimer_ns();
  for (unsigned it = 0;; ++it) {
    v = ld_relaxed(p);
    if (word_tag(v.x) == tag && word_tag(v.y) == tag) return true;
    if ((it & 1023u) == 1023u && tc::globaltimer_ns() - t0 > tc::kWaitLimitNs) return false;
  }
}
// sum over the CTA's W warps of a value each warp has left in red[warp]
template <int W>
__device__ __forceinline__ double sum_warps(const double* red) {
  const double2* r = reinterpret_cast<const double2*>(red);
  double2 a = r[0], b = r[1];
  double t = (a.x + a.y) + (b.x + b.y);
  if constexpr (W == 8) { a = r[2]; b = r[3]; t += (a.x + a.y) + (b.x + b.y); }
  return t;
}

// A step.  With x = v1 gamma and y = 2 c v1 - gamma p_j (c = gamma^2 p.v / 2) column j + 1 of the updated matrix is
// (a - x p) + y v, where only y waits for a sum.  The sum of its squares goes through the CTA's reduction of the row sums: their root
// is needed for element j + 1 of the reflector alone, whose products are added as the row sums leave.  Split of 3072 x 768
// 2130 us, 2000 x 600 1700; with the squares reduced and their root taken between the halves of the pass (a barrier more) 2240 and 1811.
template <int E, int W>
__global__ void __launch_bounds__(32 * W, 1)
tridiag_grid_kernel(const EigJob* __restrict__ jobs, int count, int C, int* status) {
  constexpr int R = kGridRows, T = 32 * W, S = T * E;
  extern __shared__ __align__(16) double2 pairs[];                        // [2][S + kMaxCl]: the pairs of a step, behind them the mates' tokens
  __shared__ __align__(16) double red_pv[W], red_sq[W], red_row[R][W], vrow[R];      // vrow: v of this CTA's rows
  __shared__ double colbuf[R], vnext;                                     // column j + 1 of the rows; v_j+1
  __shared__ uint64_t bar[2];
  __shared__ int dead;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int CL = (int)cg::this_cluster().num_blocks(), rank = (int)cg::this_cluster().block_rank();
  const int ngroups = gridDim.x / C, group = blockIdx.x / C, cta = blockIdx.x - group * C;
  const uint32_t pairs_at = tc::smem_u32(pairs), bar_off = tc::smem_u32(bar) - pairs_at;
  uint32_t mate[kMaxCl];
#pragma unroll
  for (int c = 0; c < kMaxCl; ++c) mate[c] = map_rank(pairs_at, c < CL ? c : 0);
  for (int k = tid; k < 2 * (S + kMaxCl); k += T) pairs[k] = make_double2(0.0, 0.0);       // columns behind the last stay zero
  if (tid == 0) {
    dead = 0;
    tc::mbar_init(&bar[0], 1); tc::mbar_init(&bar[1], 1);
    tc::fence_barrier_init();
  }
  cg::this_cluster().sync();             // barriers are ready before a mate sends
  int uses = 0;                          // steps so far, over all matrices: buffer and parity
  for (int mat = group; mat < count; mat += ngroups) {
    const EigJob job = jobs[mat];
    const int s = job.s;
    double2* xb = reinterpret_cast<double2*>(job.xbuf);        // 2 x s pairs
    double A[R][E];
    int slot[E];                         // which of this CTA's rows column k is, or -1
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int k = tid + T * e;
      slot[e] = (k < s && k % C == cta) ? k / C : -1;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = cta + C * r;
        A[r][e] = (i < s && k < s) ? (double)job.X[(size_t)i * s + k] : 0.0;
      }
    }
    int last = -1;                       // the cluster's last row
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = cta - rank + C * r;
      if (i < s) last = min(s, i + CL) - 1;
    }
    if (tid < R) {
      const int i = cta + C * tid;
      if (i < s) st_relaxed(xb + i, tag_word(0.0, step_tag(0)), tag_word((double)job.X[(size_t)i * s], step_tag(0)));
      vrow[tid] = 0.0;
    }
    if (tid == 0) vnext = 0.0;
    __syncthreads();
    const int share = (s + CL - 1) / CL, from = share * rank, upto = min(s, from + share);
    if (tid < CL && last > 0) {          // tokens of the first step: this CTA has read the last step of the matrix before
      const int buf = uses & 1;
      const uint32_t m = map_rank(pairs_at, tid);
      st_async(m + (uint32_t)(buf * (S + kMaxCl) + S + rank) * 16, 0.0, 0.0, m + bar_off + buf * 8);
    }
    double v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = 0.0;
    double gam = 0.0, v1 = 0.0, x = 0.0;
    unsigned tag = step_tag(0);
    for (int j = 0; j < last; ++j, ++uses) {
      const int buf = uses & 1;
      const double2* pb = pairs + buf * (S + kMaxCl);
      if (tid == 0) tc::mbar_arrive_expect_tx(&bar[buf], (uint32_t)(16 * (s - j + CL)));
      bool ok = true;
      for (int k = max(from, j) + tid; k < upto; k += T) {
        double2 q;
        ok = poll_pair(xb + (size_t)(j & 1) * s + k, tag, q) && ok;
        const uint32_t off = (uint32_t)(buf * (S + kMaxCl) + k) * 16;
#pragma unroll
        for (int c = 0; c < kMaxCl; ++c)
          if (c < CL) st_async(mate[c] + off, q.x, q.y, mate[c] + bar_off + buf * 8);
      }
      const unsigned next_tag = tag == 255u ? 1u : tag + 1u;
      // (v, p) of this CTA's rows, the two entries that everybody needs, and this thread's columns
      double vr[R], pr[R];
#pragma unroll
      for (int r = 0; r < R; ++r) vr[r] = vrow[r];
      const double vj1 = vnext;
      ok = tc::mbar_wait(&bar[buf], (uses >> 1) & 1) && ok;
      if (!ok) *reinterpret_cast<volatile int*>(&dead) = 1;
      double p[E], vn[E], pv = 0.0;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int k = tid + T * e;
        const double2 q = pb[k];
        p[e] = k >= j ? q.x : 0.0;                       // what is before j is of an earlier step
        vn[e] = fma(-x, q.x, q.y);
        pv = fma(p[e], v[e], pv);
      }
      const double2 qj = pb[j], qj1 = pb[j + 1];
#pragma unroll
      for (int r = 0; r < R; ++r) pr[r] = pb[min(cta + C * r, S - 1)].x;
      pv = warp_sum(pv);
      if (lane == 0) red_pv[warp] = pv;
      __syncthreads();
      if (*reinterpret_cast<volatile int*>(&dead)) break;      // the same for all threads: a peer never answered
      if (tid < CL && j + 1 < last) {
        const uint32_t m = map_rank(pairs_at, tid);
        st_async(m + (uint32_t)((buf ^ 1) * (S + kMaxCl) + S + rank) * 16, 0.0, 0.0, m + bar_off + (buf ^ 1) * 8);
      }
      pv = sum_warps<W>(red_pv);
      const double c = 0.5 * gam * (gam * pv);           // gamma alone may be as large as 1e290
      const double y = 2.0 * c * v1 - gam * qj.x, wj = gam * qj.x - c * v1;
      double w[E], sq = 0.0;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int k = tid + T * e;
        w[e] = fma(gam, p[e], -(c * v[e]));
        vn[e] = k > j + 1 ? fma(y, v[e], vn[e]) : 0.0;
        sq = fma(vn[e], vn[e], sq);
      }
      const double dj = qj.y - 2.0 * v1 * wj, alpha = fma(y, vj1, fma(-x, qj1.x, qj1.y));
      double ps[R];
#pragma unroll
      for (int h = 0; h < R; h += 4) {
#pragma unroll
        for (int r = h; r < h + 4; ++r) ps[r] = 0.0;
        if (cta + C * (h + 3) > j) {                     // of four rows that are not all finished
#pragma unroll
          for (int r = h; r < h + 4; ++r) {
            const double wr = fma(gam, pr[r], -(c * vr[r]));      // the bits of w
#pragma unroll
            for (int e = 0; e < E; ++e) {
              A[r][e] = fma(-vr[r], w[e], fma(-wr, v[e], A[r][e]));
              ps[r] = fma(A[r][e], vn[e], ps[r]);
            }
          }
        }
      }
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int k = tid + T * e;
        if (k == j + 1) {
#pragma unroll
          for (int r = 0; r < R; ++r) colbuf[r] = A[r][e];
        }
        if (k == j + 2) vnext = vn[e];
        if (slot[e] >= 0) vrow[slot[e]] = vn[e];
      }
      {
        // eight row sums across the warp: lanes 4 r ... hold sum r
        const bool h3 = (lane & 16) != 0, h2 = (lane & 8) != 0, h1 = (lane & 4) != 0;
        double t8[4], t2[2];
#pragma unroll
        for (int q = 0; q < 4; ++q) t8[q] = (h3 ? ps[q + 4] : ps[q]) + __shfl_xor_sync(0xffffffffu, h3 ? ps[q] : ps[q + 4], 16);
#pragma unroll
        for (int q = 0; q < 2; ++q) t2[q] = (h2 ? t8[q + 2] : t8[q]) + __shfl_xor_sync(0xffffffffu, h2 ? t8[q] : t8[q + 2], 8);
        double t = (h1 ? t2[1] : t2[0]) + __shfl_xor_sync(0xffffffffu, h1 ? t2[0] : t2[1], 4);
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        if ((lane & 3) == 0) red_row[lane >> 2][warp] = t;
        sq = warp_sum(sq);
        if (lane == 0) red_sq[warp] = sq;
      }
      __syncthreads();
      sq = sum_warps<W>(red_sq);                         // the same in all CTAs: they work on the same bits
      const bool live = sq > kLive2;
      const double nrm = sqrt(fma(alpha, alpha, sq));
      const double beta = live ? (alpha > 0.0 ? -nrm : nrm) : alpha;
      v1 = live ? alpha - beta : 0.0;
      if (tid < R) {
        const int i = cta + C * tid;
        if (i > j && i < s) {
          const double a = colbuf[tid], sum = live ? fma(a, v1, sum_warps<W>(red_row[tid])) : 0.0;
          st_relaxed(xb + (size_t)((j + 1) & 1) * s + i, tag_word(sum, next_tag), tag_word(a, next_tag));
        }
      }
      gam = live ? 1.0 / (nrm * (nrm + fabs(alpha))) : 0.0;
      x = v1 * gam;
      tag = next_tag;
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = tid + T * e == j + 1 ? v1 : live ? vn[e] : 0.0;
      // what later kernels need, from the owner of row j + 1 (its cluster is still here)
      if ((j + 1) % C == cta) {
        const int ld = refl_ld(s);
        double* dst = job.refl + (size_t)j * ld;
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (tid + T * e < ld) dst[tid + T * e] = v[e];
        if (tid == 0) { job.d[j] = dj; job.e[j] = beta; job.gam[j] = gam; }
      }
    }
    if (*reinterpret_cast<volatile int*>(&dead)) break;
    if ((s - 1) % C == cta) {            // the last diagonal element is what its row would have sent
      double* dst = job.refl + (size_t)(s - 1) * refl_ld(s);
      for (int k = tid; k < refl_ld(s); k += T) dst[k] = 0.0;
      if (tid == 0) { job.d[s - 1] = colbuf[(s - 1) / C]; job.e[s - 1] = 0.0; job.gam[s - 1] = 0.0; }
    }
    __syncthreads();                     // colbuf is read before the next matrix writes it
  }
  if (tid == 0 && dead) atomicExch(status, (int)AB_ERR_TIMEOUT);
  cg::this_cluster().sync();             // nobody leaves while a mate may still send to it
}

// ---- 2. and 3. the tridiagonal problem ------------------------------------------------------------------
// Shared by both kernels: d and e of T scaled by 1 / norm, the positions where T splits.
struct TriShared {
  double2* de;               // (d[k], e[k]); e[k] couples k and k + 1 and is zero where T splits
  unsigned* mask;            // bit k set: T splits between k and k + 1
  double norm;
};
// sm: s entries; one pass over global memory with the loads of four rounds in flight
__device__ __forceinline__ void tri_load(const EigJob& job, TriShared& t, double2* sm, unsigned* mask, double* red) {
  const int s = job.s;
  t.de = sm; t.mask = mask;
#pragma unroll 4
  for (int k = threadIdx.x; k < s; k += blockDim.x) sm[k] = make_double2(job.d[k], k + 1 < s ? job.e[k] : 0.0);
  for (int k = threadIdx.x; k < (s + 31) / 32; k += blockDim.x) mask[k] = 0u;
  __syncthreads();
  double big = 0.0;
  for (int k = threadIdx.x; k < s; k += blockDim.x) {
    const double2 q = sm[k];
    big = fmax(big, fabs(q.x) + (k > 0 ? fabs(sm[k - 1].y) : 0.0) + fabs(q.y));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = big;
  __syncthreads();
  big = 0.0;
  for (int k = 0; k < (int)(blockDim.x >> 5); ++k) big = fmax(big, red[k]);
  t.norm = big;
  const double inv = big > 0.0 ? 1.0 / big : 0.0;
  for (int k = threadIdx.x; k < s; k += blockDim.x) {
    const double2 q = sm[k];
    const double e = q.y * inv;
    const bool cut = fabs(e) <= kSplitRel;
    sm[k] = make_double2(q.x * inv, cut ? 0.0 : e);
    if (cut) atomicOr(&mask[k >> 5], 1u << (k & 31));
  }
  __syncthreads();
}
// the unreduced block [b0, b1) that position i lies in
__device__ __forceinline__ void tri_block(const TriShared& t, int s, int i, int& b0, int& b1) {
  b0 = 0;
  for (int w = (i - 1) >> 5; w >= 0 && i > 0; --w) {
    unsigned m = t.mask[w];
    if (w == ((i - 1) >> 5)) m &= 0xffffffffu >> (31 - ((i - 1) & 31));
    if (m) { b0 = 32 * w + 32 - __clz(m); break; }
  }
  b1 = s;
  for (int w = i >> 5; w < (s + 31) / 32; ++w) {
    unsigned m = t.mask[w];
    if (w == (i >> 5)) m &= 0xffffffffu << (i & 31);
    if (m) { b1 = 32 * w + __ffs(m); break; }
  }
}

// T splits somewhere inside (the bit of the last row is always set)
__device__ __forceinline__ bool tri_splits(const TriShared& t, int s) {
  for (int w = 0; w < (s + 31) / 32; ++w)
    if (t.mask[w] & (w == (s - 1) >> 5 ? ~(1u << ((s - 1) & 31)) : 0xffffffffu)) return true;
  return false;
}

// the power of two that brings the larger of two numbers to unit size
__device__ __forceinline__ double pair_scale(double p0, double p1) {
  const int h = max(__double2hiint(p0) & 0x7ff00000, __double2hiint(p1) & 0x7ff00000);
  return (h > 0 && h < 0x7fe00000) ? __hiloint2double(0x7fe00000 - h, 0) : 1.0;
}

// Eigenvalues below x of the block [b0, b1): sign changes of the leading principal minors p[k] of T - x I, scaled by
// factors s[k] > 0 with s[k + 1] = s[k - 1] / e[k - 1]^2, which leaves
//   p[k + 1] = beta[k] (d[k] - x) p[k] - p[k - 1],   beta[k] = s[k + 1] / s[k]:
// two multiply-adds a step, one of them dependent (8.5 cycles), and the signs are collected by one shift.  ab: (beta d, beta).
// Every eight steps the pair is brought back to unit size and beta starts at 1 again, for which the older of the two is scaled
// by ratio: between splits e^2 >= 5e-32, so eight steps stay within 1e127.  The coefficients are fetched eight steps ahead.
// Cycles a step, one warp and four warps a scheduler: 15 and 40 (unscaled, a difference, a product and a multiply-add a step: 23 and 49).
__device__ __forceinline__ int sturm_count(const double2* ab, const double* ratio, int b0, int b1, double x) {
  double p0 = 0.0, p1 = 1.0, sc = 1.0;
  unsigned m = 0;
  int cnt = 0, k0 = b0 & ~7;
  auto step = [&](const double2 q) {
    const double p2 = fma(fma(-x, q.y, q.x), p1, -p0);
    m = __funnelshift_l((unsigned)__double2hiint(p2), m, 1);
    p0 = p1; p1 = p2;
  };
  if (k0 < b0) {                                         // the rest of a group that the block starts inside of
    for (int u = b0 - k0; u < 8; ++u) step(ab[k0 + u]);
    unsigned keep = 0xffu >> (b0 - k0);
    if (k0 + 8 > b1) keep &= 0xffu << (k0 + 8 - b1);
    cnt = __popc((m ^ (m >> 1)) & keep);
    k0 += 8;
    if (k0 >= b1) return cnt;
    sc = pair_scale(p0, p1);
    p0 = p0 * ratio[k0 >> 3] * sc; p1 *= sc;
  }
  double2 q[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) q[u] = ab[k0 + u];         // padded to whole pairs of groups, and a group behind
  for (;;) {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const double rn = ratio[(k0 >> 3) + g + 1];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        step(q[u]);
        q[u] = ab[k0 + 8 * g + 8 + u];
        if (u == 5) sc = pair_scale(p0, p1);             // two steps early, off the chain: they add 1e32 at most
      }
      p0 = p0 * rn * sc; p1 *= sc;
    }
    k0 += 16;
    const unsigned chg = m ^ (m >> 1);
    if (k0 >= b1) return cnt + __popc(chg & 0xffffu & (0xffffu << (k0 - b1)));
    cnt += __popc(chg & 0xffffu);
  }
}

// Position i of T carries the (i - b0)-th smallest eigenvalue of its block.  kLanes lanes share the position: each
// pass cuts the interval into kLanes + 1 parts, so a lone matrix takes 32 lanes (11 passes) and a batch that fills the
// device by itself 4 (24 passes, least time in all: 2 take 35, and one warp a scheduler costs half of what four do).
// Where T does not split, the positions below s - need carry values that nobody asks for: they get -2, below everything.
template <int kLanes>
__global__ void __launch_bounds__(128)
tri_values_kernel(const EigJob* __restrict__ jobs) {
  extern __shared__ __align__(16) double2 eig_sm[];
  __shared__ unsigned mask[kMaxOrder / 32];
  __shared__ double red[4];
  __shared__ double ratio[kMaxOrder / 8 + 4];
  tc::dep_wait();
  tc::dep_launch();
  const EigJob job = jobs[blockIdx.y];
  const int s = job.s;
  constexpr int per = 128 / kLanes;
  if ((int)blockIdx.x * per >= s) return;
  TriShared t;
  tri_load(job, t, eig_sm, mask, red);
  const int i = blockIdx.x * per + threadIdx.x / kLanes, sub = threadIdx.x % kLanes;
  const int unasked = tri_splits(t, s) ? 0 : s - job.need;
  if ((int)(blockIdx.x + 1) * per <= unasked) {          // the same for the whole block
    if (sub == 0) job.lam[i] = -2.0;
    return;
  }
  int b0 = 0, b1 = 1;
  const bool in = i < s && i >= unasked;
  if (in) tri_block(t, s, i, b0, b1);
  double lo = -1.0000001, hi = 1.0000001;
  if (in && b1 - b0 == 1) { lo = hi = t.de[b0].x; }
  __syncthreads();                                       // before the diagonal is scaled
  for (int g = threadIdx.x; 8 * g < s; g += 128) {
    double beta = 1.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = 8 * g + u;
      const double2 q = k < s ? eig_sm[k] : make_double2(2.0, 0.0);
      eig_sm[k] = make_double2(q.x * beta, beta);
      const double eb = q.y * q.y * beta;
      if (u == 7) ratio[g + 1] = eb;
      else beta = eb > 0.0 ? 1.0 / eb : 1.0;
    }
  }
  __syncthreads();
  const int want = i - b0;
  const unsigned gmask = (0xffffffffu >> (32 - kLanes)) << ((threadIdx.x & 31) / kLanes * kLanes);
  constexpr int kPasses = kLanes == 4 ? 24 : kLanes == 8 ? 18 : 11;
  for (int pass = 0; pass < kPasses; ++pass) {
    const double wdt = (hi - lo) * (1.0 / (kLanes + 1));
    const double x = lo + wdt * (sub + 1);
    const bool open = in && hi - lo > 2e-16 * fmax(fabs(lo), fabs(hi)) + 1e-18;
    const bool below = open && sturm_count(t.de, ratio, b0, b1, x) <= want;        // x is at or below the wanted eigenvalue
    const unsigned bal = __ballot_sync(0xffffffffu, below) & gmask;
    if (open) {
      const int nb = __popc(bal);                     // counts rise with x: the first nb points are below
      const double l0 = lo;
      if (nb > 0) lo = l0 + wdt * nb;
      if (nb < kLanes) hi = l0 + wdt * (nb + 1);
    }
  }
  if (i < s && sub == 0) { job.lam[i] = in ? 0.5 * (lo + hi) : -2.0; if (i == s - 1) job.norm[0] = t.norm; }
}

// Eigenvector z of T at lam (twisted factorisation; Fernando, and Dhillon and Parlett), without its divisions.  u
// solves all rows of (T - lam) u = 0 but the last from the top, w all but the first from the bottom; z is u down to a row tw, w from
// there on, joined at size 1.  The residual is the joint pivot in row tw, which is the constant e[k] (u[k] w[k+1] - u[k+1] w[k])
// over u[tw] w[tw], so tw is where |u w| is largest.  A step is
//   u[k+1] = ((lam - d[k]) u[k] - e[k-1] u[k-1]) / e[k],   the quotients of e worked out once for all lanes:
// one dependent multiply-add, where the factorisation had a dependent division (145 cycles).  Every eight steps the pair is brought back to
// unit size and the exponent noted.  A split (e = 0) starts the recurrence anew; outside its block a vector is zero.
// A block works on 32 eigenvalues, a lane each: warp 0 from the top, warp 1 from the bottom, then all warps share the rows.
// z[k][i]: component k of vector i, not normalised.
// The block also sorts its vectors among all: order[rank] is the position of the vector with that rank (descending).
// The blocks behind the vector blocks form the factors of the groups of reflectors (group_factor).
constexpr int kVecWarps = 8;
constexpr int kNoKey = -2147483647 - 1;

// order of the size of |v| 2^e among values of any exponent: exponent and 13 bits
__device__ __forceinline__ int size_key(double v, int e) {
  const int hi = __double2hiint(v) & 0x7fffffff;
  return hi < 0x00100000 ? kNoKey : ((hi >> 20) + e) * 8192 + ((hi >> 7) & 0x1fff);
}
inline size_t vectors_smem(int smax) {
  const size_t n = (size_t)(smax + 7) / 8 * 8;
  return n * (sizeof(double2) * 3 + 2 * sizeof(double) + 8 * sizeof(int));
}

// H[j0] ... H[j0 + 7] = I - V T V^T, T upper triangular (compact WY form; Schreiber and Van Loan), one warp a group.
// A reflector of a small column has gamma up to 1e290 and v of 1e-145: the sums below pair a gamma with a dot product first.
__device__ __forceinline__ void group_factor(const EigJob& job, int g, int j0, int lane) {
  const int s = job.s, ld = refl_ld(s);
  double dot[kGroup][kGroup];
#pragma unroll
  for (int a = 0; a < kGroup; ++a)
#pragma unroll
    for (int b = a + 1; b < kGroup; ++b) dot[a][b] = 0.0;
  for (int k = (j0 & ~31) + lane; k < s; k += 32) {
    double f[kGroup];
#pragma unroll
    for (int a = 0; a < kGroup; ++a) f[a] = j0 + a < s ? job.refl[(size_t)(j0 + a) * ld + k] : 0.0;
#pragma unroll
    for (int a = 0; a < kGroup; ++a)
#pragma unroll
      for (int b = a + 1; b < kGroup; ++b) dot[a][b] = fma(f[a], f[b], dot[a][b]);
  }
  double row[kGroup];                   // lane i: row i of T
#pragma unroll
  for (int b = 0; b < kGroup; ++b) {
    const double gm = j0 + b < s ? job.gam[j0 + b] : 0.0;
    double acc = 0.0;
#pragma unroll
    for (int a = 0; a < b; ++a) acc = fma(a >= lane ? row[a] : 0.0, warp_sum(dot[a][b]), acc);
    row[b] = b == lane ? gm : b > lane ? -gm * acc : 0.0;
  }
  if (lane < kGroup) {
#pragma unroll
    for (int b = 0; b < kGroup; ++b) job.tmat[(size_t)g * kGroup * kGroup + lane * kGroup + b] = row[b];
  }
}

__global__ void __launch_bounds__(32 * kVecWarps)
tri_vectors_kernel(const EigJob* __restrict__ jobs, int vec_blocks, int smax) {
  extern __shared__ __align__(16) double2 eig_sm[];
  __shared__ unsigned mask[kMaxOrder / 32];
  __shared__ double red[kVecWarps];
  __shared__ double part[kVecWarps][32];
  __shared__ int best_key[kVecWarps][32], best_row[kVecWarps][32], rank_part[kVecWarps][32];
  tc::dep_wait();
  tc::dep_launch();
  const EigJob job = jobs[blockIdx.y];
  const int s = job.s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int)blockIdx.x >= vec_blocks) {
    const int g = ((int)blockIdx.x - vec_blocks) * kVecWarps + warp, j0 = g * kGroup;
    if (j0 < s) group_factor(job, g, j0, lane);
    return;
  }
  if ((int)blockIdx.x * 32 >= s) return;
  TriShared t;
  tri_load(job, t, eig_sm, mask, red);
  if (!tri_splits(t, s) && (int)blockIdx.x * 32 + 32 <= s - job.need) return;      // vectors that nobody asks for
  const int pad = (smax + 7) & ~7;            // whole groups of eight rows; those behind the last are zero
  double2* fwd = eig_sm + pad;                // (1 / e[k], e[k-1] / e[k])
  double2* bwd = fwd + pad;                   // (1 / e[k-1], e[k] / e[k-1])
  double* dd = reinterpret_cast<double*>(bwd + pad);
  double* lams = dd + pad;
  int* ex = reinterpret_cast<int*>(lams + pad);                // exponents of u, then of w: [group of eight rows][lane]
  int* exw = ex + pad * 4;
  for (int k = threadIdx.x; k < pad; k += 32 * kVecWarps) {
    const double2 q = k < s ? t.de[k] : make_double2(0.0, 0.0);
    const double el = k > 0 && k < s ? t.de[k - 1].y : 0.0;
    const double ir = q.y != 0.0 ? 1.0 / q.y : 0.0, il = el != 0.0 ? 1.0 / el : 0.0;
    fwd[k] = make_double2(ir, el * ir);
    bwd[k] = make_double2(il, q.y * il);
    dd[k] = q.x;
    if (k < s) lams[k] = job.lam[k];
  }
  const int i = blockIdx.x * 32 + lane;
  const bool in = i < s;
  double* up = job.zp + i;
  double* wp = job.zm + i;
  int b0 = s, b1 = 0;
  double lam = 0.0;
  if (in) { tri_block(t, s, i, b0, b1); lam = job.lam[i]; }
  // rows any lane of the block works on, in whole groups of eight
  const int g0 = __reduce_min_sync(0xffffffffu, b0) >> 3, g1 = (__reduce_max_sync(0xffffffffu, b1) + 7) >> 3;
  __syncthreads();
  if (warp < 2) {
    const double2* cf = warp == 0 ? fwd : bwd;
    double* out = warp == 0 ? up : wp;
    int* exs = warp == 0 ? ex : exw;
    const int first = warp == 0 ? b0 : b1 - 1;           // where this lane's block starts
    double u = 0.0, um = 0.0;
    int E = 0;
    double2 q[8];
    double d[8];
    const int dir = warp == 0 ? 1 : -1, flip = warp == 0 ? 0 : 7;
    int g = warp == 0 ? g0 : g1 - 1;
#pragma unroll
    for (int v = 0; v < 8; ++v) { q[v] = cf[8 * g + (v ^ flip)]; d[v] = dd[8 * g + (v ^ flip)]; }
    for (int n = g1 - g0; n > 0; --n, g += dir) {
      const int h = max(__double2hiint(u) & 0x7ff00000, __double2hiint(um) & 0x7ff00000);
      if (h > 0 && h < 0x7fe00000) {
        const double sc = __hiloint2double(0x7fe00000 - h, 0);
        u *= sc; um *= sc; E += (h >> 20) - 1023;
      }
      exs[g * 32 + lane] = E;
      const bool starts = __any_sync(0xffffffffu, first >> 3 == g);
      const int gn = n > 1 ? g + dir : g;
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        const int k = 8 * g + (v ^ flip);
        if (starts && k == first) { u = 1.0; um = 0.0; }
        if (in && k < s) out[(size_t)k * s] = u;
        const double un = fma((lam - d[v]) * q[v].x, u, -(q[v].y * um));
        um = u; u = un;
        q[v] = cf[8 * gn + (v ^ flip)]; d[v] = dd[8 * gn + (v ^ flip)];       // the next group's
      }
    }
  }
  __syncthreads();
  {                           // where |u w| is largest
    int key = kNoKey, row = min(b0, s - 1);
    for (int g = g0 + warp; g < g1; g += kVecWarps) {
      const int k0 = 8 * g, n = in ? min(8, s - k0) : 0;
      double a[8], c[8], top = 0.0;
      int at = k0;
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        a[v] = v < n ? up[(size_t)(k0 + v) * s] : 0.0;
        c[v] = v < n ? wp[(size_t)(k0 + v) * s] : 0.0;
      }
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        const double p = fabs(a[v] * c[v]);
        if (p > top) { top = p; at = k0 + v; }
      }
      const int ky = size_key(top, ex[g * 32 + lane] + exw[g * 32 + lane]);
      if (ky > key) { key = ky; row = at; }
    }
    best_key[warp][lane] = key;
    best_row[warp][lane] = row;
  }
  __syncthreads();
  int tw = best_row[0][lane], key = best_key[0][lane];
#pragma unroll
  for (int v = 1; v < kVecWarps; ++v)
    if (best_key[v][lane] > key) { key = best_key[v][lane]; tw = best_row[v][lane]; }
  const double ui = in ? 1.0 / up[(size_t)tw * s] : 0.0, wi = in ? 1.0 / wp[(size_t)tw * s] : 0.0;
  const int eu = ex[(tw >> 3) * 32 + lane], ew = exw[(tw >> 3) * 32 + lane];
  {
    int above = 0;
#pragma unroll 8
    for (int k = warp; k < s; k += kVecWarps) {
      const double lk = lams[k];
      above += (lk > lam || (lk == lam && k < i)) ? 1 : 0;
    }
    rank_part[warp][lane] = above;
  }
  __syncthreads();            // before row tw is overwritten
  if (in && warp == 0) {
    int above = 0;
#pragma unroll
    for (int v = 0; v < kVecWarps; ++v) above += rank_part[v][lane];
    job.order[above] = i;
  }
  double n2 = 0.0;
  for (int g = warp; 8 * g < s; g += kVecWarps) {
    const int k0 = 8 * g, n = in ? min(8, s - k0) : 0;
    const bool live = g >= g0 && g < g1;
    double a[8], c[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      a[v] = live && v < n && k0 + v <= tw ? up[(size_t)(k0 + v) * s] : 0.0;
      c[v] = live && v < n && k0 + v > tw ? wp[(size_t)(k0 + v) * s] : 0.0;
    }
    const double fu = live ? ldexp(ui, ex[g * 32 + lane] - eu) : 0.0, fw = live ? ldexp(wi, exw[g * 32 + lane] - ew) : 0.0;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const double z = k0 + v <= tw ? a[v] * fu : c[v] * fw;
      n2 = fma(z, z, n2);
      if (v < n) up[(size_t)(k0 + v) * s] = z;
    }
  }
  part[warp][lane] = n2;
  __syncthreads();
  if (in && warp == 0) {
    n2 = 0.0;
#pragma unroll
    for (int v = 0; v < kVecWarps; ++v) n2 += part[v][lane];
    job.inv[i] = 1.0 / sqrt(n2);
  }
}

// ---- 4. back transform ----------------------------------------------------------------------------------
// Z <- (I - V T V^T) Z for groups of eight reflectors, last group first: y = V^T z, w = T y, z -= V w.  Each is a product of
// 8 x 8 pieces on the fp64 tensor path (mma.sync m8n8k4; there is no tcgen05 form for fp64).  Its rate is that of plain
// multiply-adds, but the sums across lanes and most of the instructions go: with a vector a warp, its dot products reduced by
// shuffles, order 768 (192 vectors) took 407 us, now 121; 72 matrices of order 192 took 192, now 65.
// A warp holds Z^T of eight vectors as accumulator pieces: piece t, lane l, element i is vector l / 4, component
// 8 t + 2 (l % 4) + i.  That is at once the left operand of y^T = Z^T V, if step i of the reduction takes the components
// 8 t + 2 (l % 4) + i; likewise y^T and w^T are passed on as they come out.  Column c of y and w stands for
// reflector row_of(c) of the group, an order in which all reads of shared memory are free of bank conflicts.
// RS warps share the components of the same eight vectors (pieces dealt in turn) and add their parts of y through shared memory: a
// lone matrix, whose chain of groups is what counts; RS = 1: a batch.  The reflectors of a group and its T come by bulk copies, the next
// groups' on their way while one is applied.  Columns that a group's reflectors do not reach are dropped kBlock pieces at a time.
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}
__device__ __forceinline__ int row_of(int c) { return (c & 1) ? 4 + (((c >> 1) + 2) & 3) : c >> 1; }

template <int TW, int RS, int W>
struct BackShape {
  static constexpr int kCols = 8 * TW * RS;
  static constexpr int kPitch = (kCols + 15) / 16 * 16 + 4;       // rows 32 bytes apart modulo the 128 of the banks
  static constexpr int kBlock = RS > 1 ? (TW % 2 ? 1 : 2) : 4;     // pieces of a warp that are dropped together
  static constexpr int kGroups = W / RS;                           // vector groups of a CTA
  static constexpr int kY = RS > 1 ? 2 * kGroups * RS * 32 : 0;
  static constexpr size_t kStageBytes = sizeof(double) * (kGroup * kPitch + kGroup * kGroup);
  static constexpr int kStages = std::min(4, (int)((kMaxSmem - 1024 - sizeof(double2) * kY) / kStageBytes));      // groups in flight
  static constexpr size_t kBytes = kStages * kStageBytes + sizeof(double2) * kY;
  static_assert(TW % kBlock == 0 && W % RS == 0, "shape");
};

template <int TW, int RS, int W>
struct BackState {
  using B = BackShape<TW, RS, W>;
  const double *fs, *ts;
  double2* ys;
  uint64_t* bars;
  int* dead;
  int stage, parity, g, sub, vg, lane;
  // the groups whose first column lies in the pieces [Q0, Q0 + kBlock) of the warps, then the groups before them
  template <int Q0, typename F>
  __device__ __forceinline__ void segment(double (&z)[TW][2], F& fetch) {
    constexpr int kPitch = B::kPitch, kStages = B::kStages;
    const int lr = lane >> 2, lc = lane & 3, frow = row_of(lr), wrow0 = row_of(2 * lc), wrow1 = row_of(2 * lc + 1);
    for (; g >= RS * Q0; --g) {
      if (!tc::mbar_wait(&bars[stage], parity)) *reinterpret_cast<volatile int*>(dead) = 1;
      __syncthreads();                     // group g is here, and nobody reads the stage of group g + 1 any more
      if (*reinterpret_cast<volatile int*>(dead)) return;
      if (threadIdx.x == 0 && g >= kStages - 1) fetch(g - (kStages - 1), stage == 0 ? kStages - 1 : stage - 1);
      const double* f = fs + stage * kGroup * kPitch;
      const double* t = ts + stage * kGroup * kGroup;
      const double t0 = t[frow * kGroup + wrow0], t1 = t[frow * kGroup + wrow1];
      double y[2] = {0.0, 0.0}, y1[2] = {0.0, 0.0}, w[2] = {0.0, 0.0};
#pragma unroll
      for (int q = Q0; q < TW; ++q) {
        const double2 v = *reinterpret_cast<const double2*>(f + frow * kPitch + 8 * (sub + RS * q) + 2 * lc);
        dmma(y, z[q][0], v.x);
        dmma(y1, z[q][1], v.y);
      }
      y[0] += y1[0]; y[1] += y1[1];
      if constexpr (RS > 1) {
        double2* yw = ys + ((g & 1) * B::kGroups + vg) * RS * 32;
        yw[sub * 32 + lane] = make_double2(y[0], y[1]);
        tc::named_bar_sync(1 + vg, 32 * RS);
        double2 p[RS];
#pragma unroll
        for (int r = 0; r < RS; ++r) p[r] = yw[r * 32 + lane];
#pragma unroll
        for (int o = 1; o < RS; o *= 2)
#pragma unroll
          for (int r = 0; r < RS; r += 2 * o) { p[r].x += p[r + o].x; p[r].y += p[r + o].y; }
        y[0] = p[0].x; y[1] = p[0].y;
      }
      dmma(w, y[0], t0);
      dmma(w, y[1], t1);
      w[0] = -w[0]; w[1] = -w[1];
#pragma unroll
      for (int q = Q0; q < TW; ++q) {
        const int c = 8 * (sub + RS * q) + lr;
        dmma(z[q], w[0], f[wrow0 * kPitch + c]);
        dmma(z[q], w[1], f[wrow1 * kPitch + c]);
      }
      if (++stage == kStages) { stage = 0; parity ^= 1; }
    }
    if constexpr (Q0 > 0) {
      if (*reinterpret_cast<volatile int*>(dead) == 0) segment<Q0 - B::kBlock>(z, fetch);
    }
  }
};

template <int TW, int RS, int W>
__global__ void __launch_bounds__(32 * W)
back_transform_kernel(const EigJob* __restrict__ jobs, int* status) {
  using B = BackShape<TW, RS, W>;
  constexpr int kPitch = B::kPitch, kBlock = B::kBlock;
  extern __shared__ __align__(128) double back_sm[];
  constexpr int kStages = B::kStages;
  double* fs = back_sm;                                    // [kStages][kGroup][kPitch]
  double* ts = fs + kStages * kGroup * kPitch;             // [kStages][kGroup][kGroup]
  double2* ys = reinterpret_cast<double2*>(ts + kStages * kGroup * kGroup);
  __shared__ uint64_t bars[kStages];
  __shared__ int dead;
  tc::dep_wait();
  tc::dep_launch();
  const EigJob job = jobs[blockIdx.y];
  const int s = job.s, ld = refl_ld(s), ngroups = (s + kGroup - 1) / kGroup;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lr = lane >> 2, lc = lane & 3;
  const int sub = warp % RS, vg = warp / RS;
  if ((int)blockIdx.x * 8 * B::kGroups >= job.need) return;
  // what no copy fills: columns behind the rows, rows behind the last reflector (in the stage of the last group, the first one used)
  for (int r = warp; r < kStages * kGroup; r += W) {
    const bool none = r < kGroup && (ngroups - 1) * kGroup + r >= s;
    for (int k = (none ? 0 : ld) + lane; k < kPitch; k += 32) fs[r * kPitch + k] = 0.0;
  }
  if (tid == 0) {
    dead = 0;
    for (int i = 0; i < kStages; ++i) tc::mbar_init(&bars[i], 1);
    tc::fence_barrier_init();
  }
  tc::fence_proxy_async_smem();
  __syncthreads();
  auto fetch = [&](int g, int stage) {
    const int j0 = g * kGroup, n = min(kGroup, s - j0), k0 = 8 * RS * kBlock * (g / (RS * kBlock));
    const uint32_t bytes = (uint32_t)(ld - k0) * 8;
    uint64_t* bar = &bars[stage];
    tc::mbar_arrive_expect_tx(bar, n * bytes + kGroup * kGroup * 8);
    for (int a = 0; a < n; ++a) tc::bulk_load(fs + (stage * kGroup + a) * kPitch + k0, job.refl + (size_t)(j0 + a) * ld + k0, bytes, bar);
    tc::bulk_load(ts + stage * kGroup * kGroup, job.tmat + (size_t)g * kGroup * kGroup, kGroup * kGroup * 8, bar);
  };
  if (tid == 0)
    for (int i = 0; i < kStages - 1 && i < ngroups; ++i) fetch(ngroups - 1 - i, i);
  const int q0 = (blockIdx.x * B::kGroups + vg) * 8, mine = q0 + lr;
  auto position = [&](int q) { const int i = job.order[q]; return (unsigned)i < (unsigned)s ? i : q; };   // NaN leaves holes in the order
  double z[TW][2];
  double lam = 0.0;
  {
    const int i = mine < job.need ? position(mine) : 0;
    const double inv = mine < job.need ? job.inv[i] : 0.0;
    lam = mine < job.need ? job.lam[i] : 0.0;
#pragma unroll
    for (int q = 0; q < TW; ++q)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int k = 8 * (sub + RS * q) + 2 * lc + e;
        z[q][e] = (mine < job.need && k < s) ? job.zp[(size_t)k * s + i] * inv : 0.0;
      }
  }
  // Neighbours too close for the factorisation to keep apart: is this vector orthogonal to those above it?  A few pairs are formed by
  // the whole warp, one after the other, more of them side by side, a lane each: neighbours in the order are neighbours in memory.
  // Split of a flat spectrum, all one by one / as it is: 256 x 256 685 / 541 us, 1024 x 1024 at rank 512 5540 / 3610.  With six pairs as the
  // line 256 x 256 with all values equal took 517 us, with twelve 488.
  for (int q = q0 + sub; q < min(q0 + 8, job.need); q += RS) {
    const int i = position(q);
    const double li = job.lam[i];
    if (!(li > null_rel(job))) continue;
    for (int top = q - 1; top >= 0; top -= 32) {           // a lane a neighbour
      const int p = top - lane, k = p >= 0 ? position(p) : i;
      const unsigned apart = __ballot_sync(0xffffffffu, !(p >= 0 && fabs(job.lam[k] - li) < kCloseRel));
      const int n = apart ? __ffs(apart) - 1 : 32;
      double acc = 0.0;
      if (n > kFewClose) {
        if (lane < n) {
          const double *zi = job.zp + i, *zk = job.zp + k;
#pragma unroll 16
          for (int c = 0; c < s; ++c) acc = fma(zi[(size_t)c * s], zk[(size_t)c * s], acc);
        }
      } else {
        for (int u = 0; u < n; ++u) {
          const int ku = __shfl_sync(0xffffffffu, k, u);
          double t = 0.0;
#pragma unroll 4
          for (int c = lane; c < s; c += 32) t = fma(job.zp[(size_t)c * s + i], job.zp[(size_t)c * s + ku], t);
          t = warp_sum(t);
          if (lane == u) acc = t;
        }
      }
      if (lane < n && !(fabs(acc * job.inv[i] * job.inv[k]) <= kOrthTol)) *job.flag = 1;
      if (n < 32) break;
    }
  }
  BackState<TW, RS, W> x{fs, ts, ys, bars, &dead, 0, 0, ngroups - 1, sub, vg, lane};
  x.template segment<TW - kBlock>(z, fetch);
  if (*reinterpret_cast<volatile int*>(&dead)) {           // a copy never arrived
    if (tid == 0) atomicExch(status, (int)AB_ERR_TIMEOUT);
    return;
  }
  if (mine >= job.need) return;
  float* dst = job.rows + (size_t)mine * s;
#pragma unroll
  for (int q = 0; q < TW; ++q)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int k = 8 * (sub + RS * q) + 2 * lc + e;
      if (k < s) dst[k] = (float)z[q][e];
    }
  if (lc == 0 && sub == 0 && job.vals) {
    const double norm = job.norm[0], l = lam * norm;
    job.vals[mine] = (float)(job.gram ? (l > 1e-12 * norm ? sqrt(l) : 0.0) : l);
  }
}

template <int E, int R, int W, bool kSingle>
int launch_tridiag(const EigJob* jobs, int count, int CL, int* status, cudaStream_t st) {
  const size_t sm = sizeof(typename Tridiag<E, R, W, kSingle>::Shared);
  AB_CUDA_OK(cudaFuncSetAttribute(tridiag_small_kernel<E, R, W, kSingle>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  return launch_after(tridiag_small_kernel<E, R, W, kSingle>, dim3((unsigned)(count * CL)), 32 * W, sm, CL, st, jobs, status);
}

template <int L>
int launch_values(const EigJob* jobs, int count, int smax, cudaStream_t st) {
  const int per = 128 / L;
  return launch_after(tri_values_kernel<L>, dim3((unsigned)((smax + per - 1) / per), (unsigned)count), 128, (smax + 32) * sizeof(double2), 1, st, jobs);
}

template <int E, int W>
int launch_grid(const EigJob* jobs, int count, int smax, int* status, cudaStream_t st) {
  const size_t sm = 2 * (size_t)(32 * W * E + kMaxCl) * sizeof(double2);
  AB_CUDA_OK(allow_smem(tridiag_grid_kernel<E, W>, 2048));
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(32 * W);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  // The size of clusters that leaves room for the most matrices at a time, the largest of those.
  int best = 0, size = 0, groups = 0;
  for (int CL = kMaxCl; CL >= 1; CL /= 2) {
    const int C = ((smax + kGridRows - 1) / kGridRows + CL - 1) / CL * CL;
    int clusters = 0;
    attr[0].val.clusterDim.x = CL;
    cfg.gridDim = dim3((unsigned)C);
    cfg.numAttrs = 1;
    AB_CUDA_OK(cudaOccupancyMaxActiveClusters(&clusters, tridiag_grid_kernel<E, W>, &cfg));
    const int g = std::min(count, clusters * CL / C);
    if (g > groups) { best = CL; size = C; groups = g; }
  }
  if (groups < 1) return AB_ERR_UNSUPPORTED;
  attr[0].val.clusterDim.x = best;
  cfg.gridDim = dim3((unsigned)(groups * size));
  cfg.numAttrs = 2;
  AB_CUDA_OK(cudaLaunchKernelEx(&cfg, tridiag_grid_kernel<E, W>, jobs, count, size, status));
  AB_LAUNCH_OK();
  return AB_OK;
}

template <int TW, int RS, int W>
int launch_back(const EigJob* jobs, int count, int need, int* status, cudaStream_t st) {
  using B = BackShape<TW, RS, W>;
  constexpr int per = 8 * W / RS;
  AB_CUDA_OK(allow_smem(back_transform_kernel<TW, RS, W>, 1024));
  return launch_after(back_transform_kernel<TW, RS, W>, dim3((unsigned)((need + per - 1) / per), (unsigned)count), 32 * W, B::kBytes, 1, st, jobs,
                      status);
}

}  // namespace

static size_t xbuf_doubles(int s) { return s > kEigSmallMax ? (size_t)4 * s : 0; }

size_t eig_ws_doubles(int s) {
  const size_t n = (size_t)s, groups = (n + kGroup - 1) / kGroup;
  return align_up(xbuf_doubles(s) + n * refl_ld(s) + 2 * n * n + groups * kGroup * kGroup + (5 + 1) * n + 8, 2);
}

// The largest order: the grid kernel needs all CTAs of a matrix resident together.
int eig_max() { return std::min(1184, kGridRows * std::max(sm_count(), 1)); }

void eig_bind(EigJob& j, double* ws) {
  const size_t s = (size_t)j.s, groups = (s + kGroup - 1) / kGroup;
  j.xbuf = ws; j.refl = j.xbuf + xbuf_doubles(j.s); j.tmat = j.refl + s * refl_ld(j.s);      // each of these 16-byte aligned
  j.zp = j.tmat + groups * kGroup * kGroup; j.zm = j.zp + s * s;
  j.d = j.zm + s * s; j.e = j.d + s; j.gam = j.e + s; j.lam = j.gam + s; j.inv = j.lam + s; j.norm = j.inv + s;
  j.order = reinterpret_cast<int*>(j.norm + 1);
}

int eig_direct(const EigJob* h_jobs, const EigJob* d_jobs, int count, int smax, int* status, cudaStream_t st) {
  if (smax > eig_max()) return AB_ERR_UNSUPPORTED;
  const int sms = sm_count();
  if (sms <= 0) return AB_ERR_CUDA;
  int rc;
  if (smax > kEigSmallMax) {
    for (int i = 0; i < count; ++i)       // no word of a step is there yet
      AB_CUDA_OK(cudaMemsetAsync(h_jobs[i].xbuf, 0, xbuf_doubles(h_jobs[i].s) * sizeof(double), st));
    if (smax <= 512) rc = launch_grid<4, 4>(d_jobs, count, smax, status, st);
    else if (smax <= 768) rc = launch_grid<6, 4>(d_jobs, count, smax, status, st);
    else if (smax <= 1024) rc = launch_grid<4, 8>(d_jobs, count, smax, status, st);
    else rc = launch_grid<5, 8>(d_jobs, count, smax, status, st);
  } else if (smax <= 64) rc = launch_tridiag<2, 8, 8, true>(d_jobs, count, 1, status, st);
  else if (smax <= 128) rc = launch_tridiag<4, 16, 8, true>(d_jobs, count, 1, status, st);
  else if (smax <= 192)
    rc = 6 * count <= sms ? launch_tridiag<6, 4, 8, false>(d_jobs, count, 6, status, st) : launch_tridiag<6, 12, 8, false>(d_jobs, count, 2, status, st);
  else
    rc = 8 * count <= sms ? launch_tridiag<8, 4, 8, false>(d_jobs, count, 8, status, st) : launch_tridiag<8, 8, 8, false>(d_jobs, count, 4, status, st);
  AB_TRY(rc);
  long long values = 0;
  for (int i = 0; i < count; ++i) values += h_jobs[i].need;
  if (values <= 16LL * sms) rc = launch_values<32>(d_jobs, count, smax, st);
  else if (values <= 64LL * sms) rc = launch_values<8>(d_jobs, count, smax, st);
  else rc = launch_values<4>(d_jobs, count, smax, st);
  AB_TRY(rc);
  const int vb = (smax + 31) / 32, gb = ((smax + kGroup - 1) / kGroup + kVecWarps - 1) / kVecWarps;
  AB_CUDA_OK(allow_smem(tri_vectors_kernel, 8192));
  AB_TRY(launch_after(tri_vectors_kernel, dim3((unsigned)(vb + gb), (unsigned)count), 32 * kVecWarps, vectors_smem(smax), 1, st, d_jobs, vb, smax));
  // A warp to eight vectors where that gives a scheduler more than one warp, else eight warps to them (72 matrices of
  // order 192, 23 warps of vectors an SM: 65 us against 137).
  int need = 1;
  for (int i = 0; i < count; ++i) need = std::max(need, h_jobs[i].need);
  if (smax <= kEigSmallMax && values >= 48LL * sms) {
    if (smax <= 64) return launch_back<8, 1, 4>(d_jobs, count, need, status, st);
    if (smax <= 128) return launch_back<16, 1, 4>(d_jobs, count, need, status, st);
    if (smax <= 192) return launch_back<24, 1, 4>(d_jobs, count, need, status, st);
    return launch_back<32, 1, 4>(d_jobs, count, need, status, st);
  }
  if (smax <= 64) return launch_back<1, 8, 8>(d_jobs, count, need, status, st);
  if (smax <= 128) return launch_back<2, 8, 8>(d_jobs, count, need, status, st);
  if (smax <= 192) return launch_back<3, 8, 8>(d_jobs, count, need, status, st);
  if (smax <= 256) return launch_back<4, 8, 8>(d_jobs, count, need, status, st);
  if (smax <= 512) return launch_back<8, 8, 8>(d_jobs, count, need, status, st);
  if (smax <= 768) return launch_back<12, 8, 8>(d_jobs, count, need, status, st);
  if (smax <= 1024) return launch_back<16, 8, 8>(d_jobs, count, need, status, st);
  return launch_back<20, 8, 8>(d_jobs, count, need, status, st);
}

}  // namespace ab
