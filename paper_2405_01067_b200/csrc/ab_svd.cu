// Truncated SVD and sqrt-sigma split (Eq. 3 with the rank rule), batched over matrices.
//
// Route: Gram matrix of the shorter side, G = W^T W (m >= n) or W W^T (m < n) -- the paper's
// "transpose when n > m" is this choice of side -- then a block one-sided Jacobi eigensolve on
// X = G with the rotations accumulated in V^T, all in fp32:
//   * vectors are stored as ROWS (X is s x s, V^T is s x s), split into blocks of b rows;
//   * a sweep is nb-1 rounds of disjoint block pairs (round-robin); one CTA per pair keeps the
//     2b x s panel in shared memory (b = 16), forms its 32 x 32 Gram matrix M, runs a few
//     sweeps of a two-sided cyclic Jacobi on M in shared memory (accumulating Q),
//     applies Q^T to the panel and to the matching panel of V^T;
//   * sweeps repeat until no pair of rows has |x_i.x_j| > tol |x_i||x_j| (a device flag; the
//     host enqueues a fixed number of sweeps and converged matrices return at once).
// At convergence the rows of V^T are eigenvectors of G (singular vectors of the short side)
// and |x_i| = sigma_i^2.  The long-side factor is W V_r (or V_r^T W) by a GEMM; sigma_i is
// re-measured as the norm of that product, which makes A^T A = B B^T = diag(sigma) hold by
// construction.  The Jacobi kernels launched round by round wait for nothing: every loop has a fixed trip count.  The fallback in
// one cooperative launch (grid_meet) and the direct solver wait for other CTAs; those waits are bounded and reach the status word.
//
// Short sides up to eig_max() (1184) take the direct solver of ab_eig.cu; the Jacobi in shared memory (up to
// kEigSmallMax) or the block Jacobi in one cooperative launch is its fallback.  Larger ones take the block Jacobi.
// Eigensolve of 256 x 2304: 2.87 ms in the shared-memory Jacobi -> 0.47 ms; of 3072 x 768: 21.9 ms in 1410 launches of the
// block Jacobi -> 2.94 ms.
#include <vector>
#include <algorithm>
#include <map>

#include <cooperative_groups.h>

#include "ab_common.cuh"
#include "ab_tc_ptx.cuh"

namespace ab {
namespace {

struct JState {
  int done;            // 1 once converged (or sweep cap reached)
  unsigned off_bits;   // max relative off-orthogonality seen in the running sweep (float bits)
  int sweeps;
  unsigned maxn2_bits;      // largest squared row norm of the previous sweep (float bits)
  unsigned next_maxn2_bits; // the same, being collected in the running sweep
  int status;
  float off_hist[26];       // off-orthogonality after each sweep (diagnostics)
};

constexpr int kMaxSweeps = 30;
constexpr int kInnerSweeps = 1;
constexpr float kCountRel2 = 1e-8f;  // rows below 1e-4 of the largest norm do not hold up convergence
constexpr float kDeadRel2 = 1e-12f;   // rows below 1e-6 of the largest norm count as zero
// Accuracy domain of this route: a kept singular value between kZeroRel and kDomainRel of the largest has lost
// relative accuracy to the squaring in the Gram matrix (measured: 2e-7 above 2 %, up to 1.3e-4 at 1-2 %, 5e-3 at
// 0.5-1 %); the status word then says so.  Below kZeroRel a value is zero to working precision (a W of lower rank than asked for).
constexpr float kDomainRel = 2e-2f, kZeroRel = 1e-5f;

// Rows count as orthogonal when |x_i.x_j| <= tol |x_i||x_j|.  An fp32 dot product of length s
// carries rounding noise of about 6e-8 sqrt(s) relative to |x_i||x_j|; the maximum over all
// pairs sits a few times above that, so tol is placed at eight times the noise.
__host__ __device__ inline float jacobi_tol(int s) {
  float t = 5e-7f * sqrtf((float)s);
  return t < 4e-6f ? 4e-6f : t;
}

// flags: null, or one int per matrix; a matrix whose flag is zero is left alone (also in the kernels below)
__global__ void init_state_kernel(float* __restrict__ Vt, JState* __restrict__ st, int s, const int* __restrict__ flags) {
  const int mat = blockIdx.y;
  if (flags && flags[mat] == 0) return;
  float* V = Vt + (size_t)mat * s * s;
  const size_t total = (size_t)s * s;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
    V[i] = (i / s == i % s) ? 1.f : 0.f;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    JState z;
    z.done = 0; z.off_bits = 0; z.sweeps = 0; z.maxn2_bits = 0; z.next_maxn2_bits = 0; z.status = AB_OK;
    for (int i = 0; i < 26; ++i) z.off_hist[i] = 0.f;
    st[mat] = z;
  }
}

__device__ __forceinline__ void sweep_end(JState* st, int i, float tol) {
  JState z = st[i];
  if (z.done) return;
  if (z.sweeps < 26) z.off_hist[z.sweeps] = __uint_as_float(z.off_bits);
  z.sweeps += 1;
  if (__uint_as_float(z.off_bits) <= tol) z.done = 1;
  else if (z.sweeps >= kMaxSweeps) { z.done = 1; z.status = AB_ERR_NOT_CONVERGED; }
  z.off_bits = 0;
  if (z.next_maxn2_bits) z.maxn2_bits = z.next_maxn2_bits;
  z.next_maxn2_bits = 0;
  st[i] = z;
}
__global__ void sweep_end_kernel(JState* __restrict__ st, int count, float tol) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) sweep_end(st, i, tol);
}

// Index pair k of round t in a round-robin over an even number `ne` of players.
__device__ __forceinline__ void rr_pair(int ne, int t, int k, int& p, int& q) {
  const int n1 = ne - 1;
  if (k == 0) { p = n1; q = t % n1; }
  else { p = (t + k) % n1; q = (t - k + n1) % n1; }
  if (p > q) { int tmp = p; p = q; q = tmp; }
}

// ---- 32 x 32 symmetric eigenproblem of a panel ---------------------------------------------------
// Two-sided cyclic Jacobi: 31 steps of 16 disjoint pairs (round-robin tournament) cover every pair once.
// Solved by the whole CTA (256 threads) in shared memory, two barriers and a few dozen instructions per thread
// and step; an earlier version that kept the matrix
// in one warp's registers and moved columns by shuffles took a few hundred dependent shuffles per step
// (measured on the 3072 x 768 split: 118 us per round of the block Jacobi with it).
// Ms: the symmetric matrix (leading dimension ldm), Qs: receives Q (identity on entry is set here).
// Rotation that annihilates M[p][q].  Approximate reciprocal and square-root units are enough here: an error in
// c scales both rotated vectors alike (their orthogonality is untouched, and the singular vectors are
// normalised at the end), an error in t leaves a residue of second order that the next sweep removes.
__device__ __forceinline__ void jacobi_rotation(const float* Ms, int ldm, int pp, int qq, float thr, float dead2,
                                                float& c, float& sn) {
  const float app = Ms[pp * ldm + pp], aqq = Ms[qq * ldm + qq], g = Ms[pp * ldm + qq];
  c = 1.f; sn = 0.f;
  if (app > dead2 && aqq > dead2 && app > 0.f && aqq > 0.f && g * g > thr * thr * app * aqq) {
    float zeta = __fdividef(aqq - app, 2.f * g);
    zeta = fminf(fmaxf(zeta, -1e15f), 1e15f);
    const float h = fmaf(zeta, zeta, 1.f);
    const float t = __fdividef(copysignf(1.f, zeta), fabsf(zeta) + h * rsqrtf(h));
    c = rsqrtf(fmaf(t, t, 1.f));
    sn = c * t;
  }
}

// Thread (k, k2) of the 16 x 16 grid owns the 2 x 2 block of M at the rows of pair k and the columns of pair k2.
// Per step: 16 threads work out the 16 rotations (the pairs of all 31 steps come from a table built once); after
// a barrier every thread reads its block, applies J_k^T B J_k2 and writes it back (the blocks of a step are
// disjoint), and carries two rows of Q through the column rotation of pair k2; a second barrier ends the step.
struct EigScratch {
  unsigned char pp[31 * 16], qq[31 * 16];
  float c[16], s[16];
  int flag;
};
__device__ __forceinline__ void cta_eig32(float* Ms, float* Qs, int ldm, float thr, float dead2, int max_sweeps, EigScratch* es) {
  const int tid = threadIdx.x;
  const int k = tid >> 4, k2 = tid & 15;
  for (int idx = tid; idx < 32 * 32; idx += 256) Qs[(idx >> 5) * ldm + (idx & 31)] = ((idx >> 5) == (idx & 31)) ? 1.f : 0.f;
  for (int idx = tid; idx < 31 * 16; idx += 256) {
    int a, b;
    rr_pair(32, idx >> 4, idx & 15, a, b);
    es->pp[idx] = (unsigned char)a; es->qq[idx] = (unsigned char)b;
  }
  __syncthreads();
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    if (tid == 0) es->flag = 0;
    __syncthreads();
    for (int step = 0; step < 31; ++step) {
      if (tid < 16) {
        float c, sn;
        jacobi_rotation(Ms, ldm, es->pp[step * 16 + tid], es->qq[step * 16 + tid], thr, dead2, c, sn);
        es->c[tid] = c; es->s[tid] = sn;
        if (sn != 0.f) es->flag = 1;
      }
      __syncthreads();
      const float c1 = es->c[k], s1 = es->s[k], c2 = es->c[k2], s2 = es->s[k2];
      const int p1 = es->pp[step * 16 + k], q1 = es->qq[step * 16 + k], p2 = es->pp[step * 16 + k2], q2 = es->qq[step * 16 + k2];
      if (s1 != 0.f || s2 != 0.f) {
        const float b00 = Ms[p1 * ldm + p2], b01 = Ms[p1 * ldm + q2], b10 = Ms[q1 * ldm + p2], b11 = Ms[q1 * ldm + q2];
        // rows (pair k), then columns (pair k2)
        const float r00 = c1 * b00 - s1 * b10, r10 = s1 * b00 + c1 * b10;
        const float r01 = c1 * b01 - s1 * b11, r11 = s1 * b01 + c1 * b11;
        Ms[p1 * ldm + p2] = c2 * r00 - s2 * r01; Ms[p1 * ldm + q2] = s2 * r00 + c2 * r01;
        Ms[q1 * ldm + p2] = c2 * r10 - s2 * r11; Ms[q1 * ldm + q2] = s2 * r10 + c2 * r11;
      }
      if (s2 != 0.f) {
        const int i0 = k, i1 = k + 16;                // the two rows of Q this thread rotates (columns p2, q2)
        const float qa0 = Qs[i0 * ldm + p2], qb0 = Qs[i0 * ldm + q2], qa1 = Qs[i1 * ldm + p2], qb1 = Qs[i1 * ldm + q2];
        Qs[i0 * ldm + p2] = c2 * qa0 - s2 * qb0; Qs[i0 * ldm + q2] = s2 * qa0 + c2 * qb0;
        Qs[i1 * ldm + p2] = c2 * qa1 - s2 * qb1; Qs[i1 * ldm + q2] = s2 * qa1 + c2 * qb1;
      }
      __syncthreads();
    }
    if (!es->flag) break;
  }
}

// One cluster of kCl CTAs (8, or 1 when a batch already fills the device) per block pair: PB = 32 rows (16 + 16)
// or PB = 16 (8 + 8).  A panel is only PB rows, so
// one CTA per pair would leave most of the device idle (24 CTAs for a 768 x 768 matrix: 116 us per round); the
// columns of the panel are cut into kCl slices instead, one per CTA of the cluster.  Each CTA forms the Gram matrix
// of its slice; the partial matrices are added through distributed shared memory in ascending CTA order, so every
// CTA of the cluster holds the same M to the bit, solves the same small eigenproblem and rotates its own slice of
// the X panel and of the V^T panel.  No wait spins: the only waits are cluster barriers that every CTA of the
// cluster reaches (all early exits depend on values the whole cluster agrees on).
template <int PB, int kCl>
__device__ __forceinline__ void jacobi_pair(float* Xall, float* Vall, int s, int nb, int round, int mat, int pair, int crank,
                                            float tol, JState* states) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int HB = PB / 2;          // rows per block
  constexpr int LDM = 33;
  constexpr int LDQ = PB + 4;
  extern __shared__ __align__(16) float smem[];
  JState* st = states + mat;
  if (*reinterpret_cast<volatile int*>(&st->done)) return;               // the same for the whole cluster
  const int nbe = nb + (nb & 1);
  int bi, bj;
  rr_pair(nbe, round, pair, bi, bj);
  if (bj >= nb && nb > 1) return;     // this block sits the round out (whole cluster)
  // this CTA's slice of the columns: multiples of 4, as equal as they come
  const int s4 = (s + 3) >> 2;
  const int c_lo = (int)((long long)crank * s4 / kCl) * 4;
  int c_hi = (int)((long long)(crank + 1) * s4 / kCl) * 4;
  if (c_hi > s) c_hi = s;
  const int w = c_hi > c_lo ? c_hi - c_lo : 0;     // width of the slice
  const int ldp = (((s4 + kCl - 1) / kCl) * 4) + 4;  // the same in every CTA
  float* P = smem;                    // PB x ldp
  float* Mp = P + (size_t)PB * ldp;   // 32 x LDM: this CTA's partial Gram matrix (zero beyond PB)
  float* Ms = Mp + 32 * LDM;          // 32 x LDM: the sum
  float* Qs = Ms + 32 * LDM;          // 32 x LDM
  float* Qt = Qs + 32 * LDM + 1;      // PB x LDQ, Qt[c][i] = Q[i][c]; realigned below
  Qt = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(Qt) + 15) & ~(uintptr_t)15);
  __shared__ int any_rot;
  __shared__ EigScratch eig_scratch;
  const int tid = threadIdx.x;
  float* X = Xall + (size_t)mat * s * s;
  float* V = Vall + (size_t)mat * s * s;
  const float maxn2 = __uint_as_float(st->maxn2_bits);
  const float dead2 = kDeadRel2 * maxn2;
  const float count2 = kCountRel2 * maxn2;

  auto grow = [&](int lr) -> int {    // local panel row -> global row (or -1)
    int g = (lr < HB) ? bi * HB + lr : bj * HB + (lr - HB);
    if (lr >= HB && bj >= nb) return -1;
    return g < s ? g : -1;
  };
  auto load_panel = [&](const float* src) {
    for (int lr = tid >> 5; lr < PB; lr += 8) {      // a warp per row: coalesced
      const int g = grow(lr);
      for (int k = tid & 31; k < ldp - 4; k += 32)
        P[(size_t)lr * ldp + k] = (g >= 0 && k < w) ? src[(size_t)g * s + c_lo + k] : 0.f;
    }
  };
  auto store_panel = [&](float* dst) {
    for (int lr = tid >> 5; lr < PB; lr += 8) {
      const int g = grow(lr);
      if (g < 0) continue;
      for (int k = tid & 31; k < w; k += 32) dst[(size_t)g * s + c_lo + k] = P[(size_t)lr * ldp + k];
    }
  };
  auto apply_q = [&]() {              // P <- Q^T P, one panel column per thread at a time
    for (int k = tid; k < w; k += 256) {
      float col[PB];
#pragma unroll
      for (int j = 0; j < PB; ++j) col[j] = P[(size_t)j * ldp + k];
#pragma unroll 4
      for (int i = 0; i < PB; ++i) {
        const float4* qrow = reinterpret_cast<const float4*>(Qt + i * LDQ);
        float acc = 0.f;
#pragma unroll
        for (int j4 = 0; j4 < PB / 4; ++j4) {
          float4 q4 = qrow[j4];
          acc = fmaf(q4.x, col[4 * j4], acc);
          acc = fmaf(q4.y, col[4 * j4 + 1], acc);
          acc = fmaf(q4.z, col[4 * j4 + 2], acc);
          acc = fmaf(q4.w, col[4 * j4 + 3], acc);
        }
        P[(size_t)i * ldp + k] = acc;
      }
    }
  };

  load_panel(X);
  for (int idx = tid; idx < 32 * LDM; idx += 256) Mp[idx] = 0.f;
  if (tid == 0) any_rot = 0;
  __syncthreads();

  // ---- partial Gram matrix of this slice: entry (i, j) by thread i * PB + j (and + 256 ...), k ascending
  for (int e = tid; e < PB * PB; e += 256) {
    const int i = e / PB, jj = e - i * PB;
    if (jj < i) continue;             // symmetric: the upper triangle is computed, the lower mirrored
    const float4* a = reinterpret_cast<const float4*>(P + (size_t)i * ldp);
    const float4* b = reinterpret_cast<const float4*>(P + (size_t)jj * ldp);
    float acc = 0.f;
    for (int k = 0; k < (ldp - 4) / 4; ++k) {
      const float4 x = a[k], y = b[k];
      acc = fmaf(x.x, y.x, acc); acc = fmaf(x.y, y.y, acc); acc = fmaf(x.z, y.z, acc); acc = fmaf(x.w, y.w, acc);
    }
    Mp[i * LDM + jj] = acc;
    Mp[jj * LDM + i] = acc;
  }
  if constexpr (kCl > 1) cluster.sync(); else __syncthreads();     // every CTA's partial matrix is complete
  for (int idx = tid; idx < 32 * LDM; idx += 256) {
    float acc = 0.f;
    if constexpr (kCl > 1) {
#pragma unroll
      for (int c = 0; c < kCl; ++c) acc += cluster.map_shared_rank(Mp, c)[idx];   // ascending CTA order in every CTA
    } else {
      acc = Mp[idx];
    }
    Ms[idx] = acc;
  }
  if constexpr (kCl > 1) cluster.sync(); else __syncthreads();     // nobody reads a peer's partial matrix after this

  // ---- how far from orthogonal is this panel?  (also collects the largest squared norm)
  {
    float worst = 0.f, big = 0.f;
    int rot = 0;
    for (int idx = tid; idx < PB * PB; idx += 256) {
      int i = idx / PB, jj = idx - i * PB;
      float mii = Ms[i * LDM + i], mjj = Ms[jj * LDM + jj];
      if (i == jj) { big = fmaxf(big, mii); continue; }
      if (i < jj && mii > dead2 && mjj > dead2 && mii > 0.f && mjj > 0.f) {
        float rel = fabsf(Ms[i * LDM + jj]) / (sqrtf(mii) * sqrtf(mjj));
        if (rel > tol) rot = 1;
        // rows far below the largest norm are rounding noise of the large ones: they are still
        // rotated, but the sweep counts as converged without them
        if (mii > count2 && mjj > count2) worst = fmaxf(worst, rel);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, o));
      big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
    }
    if ((tid & 31) == 0 && crank == 0) {
      atomicMax(&st->off_bits, __float_as_uint(worst));
      atomicMax(&st->next_maxn2_bits, __float_as_uint(big));
    }
    if (rot) atomicExch(&any_rot, 1);
  }
  __syncthreads();
  if (!any_rot) return;               // panel already orthogonal: nothing to write (the same M in every CTA)

  // ---- diagonalise M (all threads; the same arithmetic in every CTA of the cluster), then Qt[c][i] = Q[i][c]
  cta_eig32(Ms, Qs, LDM, 0.25f * tol, dead2, kInnerSweeps, &eig_scratch);
  for (int idx = tid; idx < PB * PB; idx += 256) {
    const int c = idx / PB, i = idx - c * PB;
    Qt[c * LDQ + i] = Qs[i * LDM + c];
  }
  __syncthreads();

  // ---- rotate this slice of the panel of X, then of the same rows of V^T
  apply_q();
  __syncthreads();
  store_panel(X);
  __syncthreads();
  load_panel(V);
  __syncthreads();
  apply_q();
  __syncthreads();
  store_panel(V);
}

template <int PB, int kCl>
__global__ void __launch_bounds__(256, 2)
jacobi_pair_kernel(float* __restrict__ Xall, float* __restrict__ Vall, int s, int nb, int round,
                   float tol, JState* __restrict__ states) {
  jacobi_pair<PB, kCl>(Xall, Vall, s, nb, round, blockIdx.y, blockIdx.x / kCl, blockIdx.x % kCl, tol, states);
}

// All sweeps of the flagged matrices in one launch, for when the block Jacobi is the fallback of the direct solver:
// nearly always no flag is set and one empty launch is all it costs.  The blocks meet between rounds (cooperative
// launch, so all of them are resident); bar[0] counts arrivals, bar[1] is set when a wait gave up.
__device__ __forceinline__ bool grid_meet(unsigned* bar, unsigned& round_no) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ++round_no;
    __threadfence();
    atomicAdd(bar, 1u);
    const unsigned want = round_no * gridDim.x;
    const uint64_t t0 = tc::globaltimer_ns();
    ok = 1;
    for (unsigned it = 0; *reinterpret_cast<volatile unsigned*>(bar) < want; ++it) {
      if (*reinterpret_cast<volatile unsigned*>(bar + 1) || ((it & 1023u) == 1023u && tc::globaltimer_ns() - t0 > tc::kWaitLimitNs)) {
        atomicExch(bar + 1, 1u);
        ok = 0;
        break;
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}
template <int PB>
__global__ void __launch_bounds__(256)
jacobi_sweeps_kernel(float* Xall, float* Vall, int s, int nb, int count, float tol, JState* states, const int* flags, unsigned* bar) {
  bool any = false;
  for (int m = 0; m < count; ++m) any = any || flags[m] != 0;
  if (!any) return;
  const int nbe = nb + (nb & 1), pairs = nbe / 2, rounds = nbe > 2 ? nbe - 1 : 1;
  unsigned round_no = 0;
  bool met = true;
  for (int sweep = 0; sweep < kMaxSweeps && met; ++sweep) {
    for (int r = 0; r < rounds && met; ++r) {
      for (int t = blockIdx.x; t < pairs * count; t += gridDim.x) {
        const int mat = t / pairs;
        __syncthreads();                               // the panel of the task before is no longer read
        if (flags[mat]) jacobi_pair<PB, 1>(Xall, Vall, s, nb, r, mat, t - mat * pairs, 0, tol, states);
      }
      met = grid_meet(bar, round_no);
    }
    if (!met) break;
    if (blockIdx.x == 0)
      for (int m = threadIdx.x; m < count; m += blockDim.x) if (flags[m]) sweep_end(states, m, tol);
    met = grid_meet(bar, round_no);
    bool busy = false;
    for (int m = 0; m < count; ++m) busy = busy || (flags[m] && !*reinterpret_cast<volatile int*>(&states[m].done));
    if (!busy) return;
  }
  if (!met && blockIdx.x == 0)
    for (int m = threadIdx.x; m < count; m += blockDim.x) if (flags[m]) states[m].status = AB_ERR_TIMEOUT;
}

constexpr int kJacobiStatics = 2048;      // static shared memory of the kernels above, rounded up
template <int PB, int kCl>
size_t jacobi_smem_bytes(int s) {
  const int s4 = (s + 3) >> 2;
  const int ldp = (((s4 + kCl - 1) / kCl) * 4) + 4;
  return sizeof(float) * ((size_t)PB * ldp + 3 * 32 * 33 + 8 + (size_t)PB * (PB + 4));
}

// lam[i] = |row i of X|, perm = indices by descending lam (ties by index).  One CTA per matrix.
__global__ void __launch_bounds__(256)
norms_sort_kernel(const float* __restrict__ Xall, int s, float* __restrict__ lam_all, int* __restrict__ perm_all,
                  const int* __restrict__ flags) {
  extern __shared__ float lam_s[];
  const int mat = blockIdx.x;
  if (flags && flags[mat] == 0) return;
  const float* X = Xall + (size_t)mat * s * s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = warp; i < s; i += 8) {
    double acc = 0.0;
    for (int k = lane; k < s; k += 32) { float v = X[(size_t)i * s + k]; acc += (double)v * v; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) lam_s[i] = (float)sqrt(acc);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < s; i += 256) {
    // Compared by their bits, which for values that are not negative is the order of the values: NaN has a place as well, and perm
    // is a permutation whatever the matrix holds (a rank that nothing took would leave an index of old workspace contents).
    const unsigned li = __float_as_uint(lam_s[i]);
    int rank = 0;
    for (int j = 0; j < s; ++j) {
      const unsigned lj = __float_as_uint(lam_s[j]);
      rank += (lj > li) || (lj == li && j < i);
    }
    perm_all[(size_t)mat * s + rank] = i;
    lam_all[(size_t)mat * s + i] = lam_s[i];
  }
}

// After the in-shared-memory solver: rows (unit length, sorted by descending lam) whose lam is below
// 1e-4 of the largest carry directions of rounding noise, not eigenvectors.  Each of them is made
// orthogonal to every row before it (Gram-Schmidt, two passes) and rescaled, so that the rows stay an
// orthonormal set and W v picks up nothing of the resolved directions; a row that does not survive the
// projection becomes zero (it then contributes nothing to either factor).  Only the first r_need rows
// are ever used.  One CTA per matrix.
__global__ void __launch_bounds__(256)
complete_basis_kernel(float* __restrict__ rows_all, const float* __restrict__ lam_all, const int* __restrict__ flags, int s,
                      int r_need) {
  if (flags[blockIdx.x] == 0) return;
  extern __shared__ float cb_sm[];
  float* v = cb_sm;            // s
  float* coef = cb_sm + s;     // s
  __shared__ float red[8];
  __shared__ int k_first;
  float* rows = rows_all + (size_t)blockIdx.x * s * s;
  const float* lam = lam_all + (size_t)blockIdx.x * s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    int k = 0;
    const float thr = 1e-4f * lam[0];
    while (k < s && lam[k] >= thr && lam[k] > 0.f) ++k;
    k_first = k;
  }
  __syncthreads();
  const int k_end = r_need < s ? r_need : s;
  for (int k = k_first; k < k_end; ++k) {
    for (int u = tid; u < s; u += 256) v[u] = rows[(size_t)k * s + u];
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
      for (int j = warp; j < k; j += 8) {
        float a = 0.f;
        for (int u = lane; u < s; u += 32) a = fmaf(rows[(size_t)j * s + u], v[u], a);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) coef[j] = a;
      }
      __syncthreads();
      for (int u = tid; u < s; u += 256) {
        float a = v[u];
        for (int j = 0; j < k; ++j) a = fmaf(-coef[j], rows[(size_t)j * s + u], a);
        v[u] = a;
      }
      __syncthreads();
    }
    float a = 0.f;
    for (int u = tid; u < s; u += 256) a = fmaf(v[u], v[u], a);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) red[warp] = a;
    __syncthreads();
    float n2 = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) n2 += red[i];
    const float inv = n2 > 1e-6f ? rsqrtf(n2) : 0.f;       // the row started at unit length (or zero)
    for (int u = tid; u < s; u += 256) rows[(size_t)k * s + u] = v[u] * inv;
    __syncthreads();                                         // the next row reads this one from global memory
  }
}

// Vr[k][:] = Vt[perm[k]][:] scaled to unit length, k < r_cap (thousands of fp32 rotations leave
// the rows orthogonal but let their norms wander by ~1e-6)
__global__ void __launch_bounds__(256)
gather_rows_kernel(const float* __restrict__ Vt, const int* __restrict__ perm, int s, int r_cap,
                   float* __restrict__ Vr, const int* __restrict__ flag) {
  if (flag && *flag == 0) return;
  __shared__ double red[8];
  const int k = blockIdx.x;
  if (k >= r_cap) return;
  const float* src = Vt + (size_t)perm[k] * s;
  double acc = 0.0;
  for (int u = threadIdx.x; u < s; u += 256) { float v = src[u]; acc += (double)v * v; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  double tot = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) tot += red[i];
  const float inv = tot > 0.0 ? (float)(1.0 / sqrt(tot)) : 0.f;
  for (int u = threadIdx.x; u < s; u += 256) Vr[(size_t)k * s + u] = src[u] * inv;
}

// sigma[k] = norm over t of Ylong(k,t), Ylong(k,t) = Y[t*st_ + k*sk].
// Neighbouring k adjacent in memory: a cluster of kNormCl CTAs takes 32 values of k, a lane each, the warps of all of them
// sharing the t; the parts are added in the order of the warps.  One CTA to 32 values walked 3072 rows in
// 384 dependent rounds: 57 us for 192 values, 10 now.  Neighbouring t adjacent: a CTA a k (70 us -> 5, 128 values of 2304).
constexpr int kNormCl = 8;
__global__ void __launch_bounds__(256)
long_norms_kernel(const float* __restrict__ Y, int64_t st_, int L, int r_cap, float* __restrict__ sigma) {
  __shared__ double red[8][32];
  __shared__ double part[kNormCl][32];
  auto cluster = cooperative_groups::this_cluster();
  auto started = cluster.barrier_arrive();
  tc::dep_wait();
  tc::dep_launch();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, rank = blockIdx.x % kNormCl;
  const int k = blockIdx.x / kNormCl * 32 + lane;
  double acc = 0.0;
  if (k < r_cap) {
#pragma unroll 8
    for (int t = rank * 8 + warp; t < L; t += 8 * kNormCl) { const float v = Y[(int64_t)t * st_ + k]; acc += (double)v * v; }
  }
  red[warp][lane] = acc;
  __syncthreads();
  cluster.barrier_wait(std::move(started));      // rank 0 runs: its shared memory may be written
  if (warp == 0) {
    acc = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc += red[i][lane];
    *cluster.map_shared_rank(&part[rank][lane], 0) = acc;
  }
  cluster.sync();
  if (rank == 0 && warp == 0 && k < r_cap) {
    acc = 0.0;
#pragma unroll
    for (int i = 0; i < kNormCl; ++i) acc += part[i][lane];
    sigma[k] = (float)sqrt(acc);
  }
}
__global__ void __launch_bounds__(256)
long_norms_rows_kernel(const float* __restrict__ Y, int64_t sk, int L, float* __restrict__ sigma) {
  __shared__ double red[8];
  tc::dep_wait();
  tc::dep_launch();
  const float* y = Y + (int64_t)blockIdx.x * sk;
  double acc = 0.0;
#pragma unroll 4
  for (int t = threadIdx.x; t < L; t += 256) { const float v = y[t]; acc += (double)v * v; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    acc = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc += red[i];
    sigma[blockIdx.x] = (float)sqrt(acc);
  }
}

// The rank rule, by every block of 256 threads for itself: how many values reach cutoff times the largest (at least one);
// outside: whether one of those that are kept lies outside the accuracy domain.
__device__ __forceinline__ int rank_rule(const float* __restrict__ sigma, int r_cap, float cutoff, bool& outside) {
  __shared__ float red[8];
  float top = 0.f;
  for (int k = threadIdx.x; k < r_cap; k += 256) top = fmaxf(top, sigma[k]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = top;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) top = fmaxf(top, red[i]);
  const float thr = cutoff * top;
  int keep = 0;
  for (int k0 = 0; k0 < r_cap; k0 += 256) {
    const int k = k0 + (int)threadIdx.x;
    keep += __syncthreads_count(k < r_cap && sigma[k] >= thr);
  }
  if (keep < 1) keep = 1;
  bool out = false;
  for (int k = threadIdx.x; k < keep; k += 256) out = out || (sigma[k] < kDomainRel * top && sigma[k] > kZeroRel * top);
  outside = __syncthreads_or(out) != 0;
  return keep;
}

// What the self-test of the fallback makes of the direct solver's verdicts (see SvdSelftest).
__global__ void force_fallback_kernel(int* __restrict__ flags, int count, int* __restrict__ solver, unsigned long long flagged, int status) {
  const int i = threadIdx.x;
  if (i < count && (flagged >> i & 1ull)) flags[i] = 1;
  if (i == 0 && status != AB_OK) *solver = status;
}

// Applies the rank rule and writes the factors.
// long factor: F(t,k) = Ylong(k,t) / sqrt(sigma_k); short factor: F(k,u) = sqrt(sigma_k) Vr[k][u].
// Columns/rows k >= r' (and k >= r_cap) are written as zero.  tall: the long factor is A (L x r_max), the short one B (r_max x s);
// else the long one is B (r_max x L), the short one A (s x r_max).  A warp a row of the results.
// solver: null, or what the direct solver's waits reported for the call this matrix was part of
template <typename TO>
__global__ void __launch_bounds__(256)
write_factors_kernel(const float* __restrict__ Y, const float* __restrict__ Vr, const float* __restrict__ sigma, int tall, int L, int s,
                     int r_cap, int r_max, float cutoff, TO* __restrict__ Flong, TO* __restrict__ Fshort, int* __restrict__ r_out,
                     const JState* __restrict__ st, const int* __restrict__ solver, int* __restrict__ dev_status) {
  tc::dep_wait();
  tc::dep_launch();
  bool outside;
  const int rk = rank_rule(sigma, r_cap, cutoff, outside), keep = rk < r_cap ? rk : r_cap;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *r_out = rk;
    if (dev_status) {
      const int code = solver && *solver != AB_OK ? *solver : st->status;
      *dev_status = code == AB_OK && outside ? (int)AB_ERR_ACCURACY : code;
    }
  }
  const int lane = threadIdx.x & 31, nlong = tall ? L : r_max, nshort = tall ? r_max : s;
  for (int row = blockIdx.x * 8 + (threadIdx.x >> 5); row < nlong + nshort; row += gridDim.x * 8) {
    const bool is_long = row < nlong;
    const int i = is_long ? row : row - nlong;
    if (is_long == (tall != 0)) {          // a row runs over k
      TO* dst = (is_long ? Flong : Fshort) + (int64_t)i * r_max;
      for (int k = lane; k < r_max; k += 32) {
        float v = 0.f;
        if (k < keep) {
          const float sg = sigma[k];
          if (is_long) v = sg > 0.f ? Y[(int64_t)i * r_cap + k] * rsqrtf(sg) : 0.f;
          else v = sqrtf(sg) * Vr[(int64_t)k * s + i];
        }
        from_f32(dst[k], v);
      }
    } else {                               // a row is one k
      const int n = is_long ? L : s;
      TO* dst = (is_long ? Flong : Fshort) + (int64_t)i * n;
      const float* src = is_long ? Y + (int64_t)i * L : Vr + (int64_t)i * s;
      float f = 0.f;
      if (i < keep) f = !is_long ? sqrtf(sigma[i]) : sigma[i] > 0.f ? rsqrtf(sigma[i]) : 0.f;
      const bool zero = i >= keep || (is_long && !(sigma[i] > 0.f));
      for (int t = lane; t < n; t += 32) from_f32(dst[t], zero ? 0.f : src[t] * f);
    }
  }
}

// X = the sum of `parts` partial Gram matrices of which the upper triangle counts, added in fp64 in ascending order, and its mirror
// image.  A block a pair of 32 x 32 tiles.
__global__ void __launch_bounds__(256)
sum_gram_kernel(const double* __restrict__ part, int parts, float* __restrict__ X, int s) {
  __shared__ float t[32][33];
  tc::dep_wait();
  tc::dep_launch();
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj < bi) return;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, col = 32 * bj + tx;
  const size_t stride = (size_t)s * s;
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const int row = 32 * bi + ty + 8 * h;
    double acc = 0.0;
    if (row < s && col < s && row <= col) {
#pragma unroll 3
      for (int q = 0; q < parts; ++q) acc += part[q * stride + (size_t)row * s + col];
      X[(size_t)row * s + col] = (float)acc;
    }
    t[ty + 8 * h][tx] = (float)acc;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const int row = 32 * bj + ty + 8 * h, c = 32 * bi + tx;      // the mirror image's
    if (row < s && c < s && row > c) X[(size_t)row * s + c] = t[tx][ty + 8 * h];
  }
}

struct Plan {
  int s, L, r_cap, pb, nb;
  bool tall;           // m >= n
};

Plan make_plan(const SvdItem& it) {
  Plan p;
  p.tall = it.m >= it.n;
  p.s = p.tall ? it.n : it.m;
  p.L = p.tall ? it.m : it.n;
  p.r_cap = std::min(it.r_max, p.s);
  p.pb = p.s <= 1536 ? 32 : 16;
  int hb = p.pb / 2;
  p.nb = (p.s + hb - 1) / hb;
  return p;
}

struct ItemWs {
  float *lam, *Vr, *Y, *Wf;
  int* perm;
};

// Lays out the workspace: per group (equal s) X, Vt and states; per item the rest.
struct Layout {
  std::map<int, std::vector<int>> groups;     // s -> item indices
  std::map<int, float*> X, Vt;
  std::map<int, JState*> st;
  std::map<int, void*> jobs;                  // short side up to kEigSmallMax: the in-shared-memory Jacobi's scratch
  std::map<int, double*> eig;                 // direct solver: its scratch, EigJobs, fallback flags (and behind the flags of a
  std::map<int, int*> flags;                  //   group two words on which the blocks of the fallback meet and the solver's status)
  std::map<int, EigJob*> ejobs;
  std::vector<ItemWs> item;
  size_t bytes;
};

// Matrices of one order that are solved (and hold scratch) at the same time: two or three of the large ones fill the
// device in the reduction, a dozen in the steps behind it.
int eig_chunk(int s) { return s <= kEigSmallMax ? 1 << 20 : 12; }
// one status word per call of the direct solver: a wait that runs out leaves every matrix of that call undone
int eig_calls(int s, int count) { return (count + eig_chunk(s) - 1) / eig_chunk(s); }

Layout make_layout(const SvdItem* items, int L, void* ws) {
  Layout lo;
  Arena ar(ws, 0);
  for (int i = 0; i < L; ++i) lo.groups[make_plan(items[i]).s].push_back(i);
  for (auto& g : lo.groups) {
    size_t s = (size_t)g.first, cnt = g.second.size();
    lo.X[g.first] = ar.take_n<float>(cnt * s * s);
    lo.Vt[g.first] = ar.take_n<float>(cnt * s * s);
    lo.st[g.first] = ar.take_n<JState>(cnt);
    if (g.first <= kEigSmallMax) lo.jobs[g.first] = ar.take_n<char>(rows_jacobi_scratch_bytes((int)cnt));
    if (g.first <= eig_max()) {
      lo.ejobs[g.first] = ar.take_n<EigJob>(cnt);
      lo.flags[g.first] = ar.take_n<int>(cnt + 2 + eig_calls(g.first, (int)cnt));
      lo.eig[g.first] = ar.take_n<double>(std::min(cnt, (size_t)eig_chunk(g.first)) * eig_ws_doubles(g.first));
    }
  }
  lo.item.resize(L);
  for (int i = 0; i < L; ++i) {
    Plan p = make_plan(items[i]);
    lo.item[i].lam = nullptr;
    lo.item[i].perm = nullptr;
    lo.item[i].Vr = ar.take_n<float>((size_t)p.r_cap * p.s);
    lo.item[i].Y = ar.take_n<float>((size_t)p.L * p.r_cap);
    lo.item[i].Wf = nullptr;
  }
  for (auto& g : lo.groups) {   // lam/perm are group-contiguous (one sort launch per group)
    size_t s = (size_t)g.first, cnt = g.second.size();
    float* lam = ar.take_n<float>(cnt * s);
    int* perm = ar.take_n<int>(cnt * s);
    for (size_t j = 0; j < cnt; ++j) {
      lo.item[g.second[j]].lam = lam ? lam + j * s : nullptr;
      lo.item[g.second[j]].perm = perm ? perm + j * s : nullptr;
    }
  }
  lo.bytes = align_up(ar.used, 256);
  return lo;
}

template <int PB, int CL>
int run_jacobi_cl(float* X, float* Vt, JState* st, int s, int nb, int count, cudaStream_t stream) {
  const size_t smem = jacobi_smem_bytes<PB, CL>(s);
  if (smem > kMaxSmem - kJacobiStatics) return AB_ERR_UNSUPPORTED;
  AB_CUDA_OK(allow_smem(jacobi_pair_kernel<PB, CL>, kJacobiStatics));
  const int nbe = nb + (nb & 1);
  const int rounds = nbe > 2 ? nbe - 1 : 1;
  const float tol = jacobi_tol(s);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nbe / 2) * CL, (unsigned)count);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  for (int sw = 0; sw < kMaxSweeps; ++sw) {
    for (int r = 0; r < rounds; ++r) {
      AB_CUDA_OK(cudaLaunchKernelEx(&cfg, jacobi_pair_kernel<PB, CL>, X, Vt, s, nb, r, tol, st));
    }
    sweep_end_kernel<<<(count + 127) / 128, 128, 0, stream>>>(st, count, tol);
  }
  count_launches((long long)kMaxSweeps * (rounds + 1) - 1);
  AB_LAUNCH_OK();
  return AB_OK;
}

// Clusters of 8 CTAs per block pair while that leaves the device room for every pair of a round (a lone matrix);
// one CTA per pair for batches, whose pairs fill the device by themselves.
template <int PB>
int run_jacobi(float* X, float* Vt, JState* st, int s, int nb, int count, cudaStream_t stream) {
  const int nbe = nb + (nb & 1);
  const long long pairs = (long long)(nbe / 2) * count;
  int sms = sm_count();
  if (sms <= 0) sms = 1;
  if (pairs * 8 <= 2LL * sms + 8) return run_jacobi_cl<PB, 8>(X, Vt, st, s, nb, count, stream);
  return run_jacobi_cl<PB, 1>(X, Vt, st, s, nb, count, stream);
}

template <int PB>
int run_jacobi_fallback(float* X, float* Vt, JState* st, int* flags, int s, int nb, int count, cudaStream_t stream) {
  const size_t smem = jacobi_smem_bytes<PB, 1>(s);
  if (smem > kMaxSmem - kJacobiStatics) return AB_ERR_UNSUPPORTED;
  AB_CUDA_OK(allow_smem(jacobi_sweeps_kernel<PB>, kJacobiStatics));
  int per_sm = 0;
  AB_CUDA_OK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, jacobi_sweeps_kernel<PB>, 256, smem));
  const int sms = sm_count();
  if (sms <= 0 || per_sm <= 0) return AB_ERR_CUDA;
  const int pairs = (nb + 1) / 2;
  const unsigned grid = (unsigned)std::min<long long>((long long)pairs * count, (long long)per_sm * sms);
  float tol = jacobi_tol(s);
  unsigned* bar = reinterpret_cast<unsigned*>(flags + count);
  const int* cflags = flags;
  void* args[] = {&X, &Vt, &s, &nb, &count, &tol, &st, &cflags, &bar};
  AB_CUDA_OK(cudaLaunchCooperativeKernel(jacobi_sweeps_kernel<PB>, dim3(grid), dim3(256), args, smem, stream));
  AB_LAUNCH_OK();
  return AB_OK;
}

// Gram matrix and long product of a large fp32 matrix: the reduction in parts that together fill the device (gemm_parts); the scratch of
// the solver, in use only between the two, holds kParts s x s partial results in fp64.  On the tensor cores as six bf16 terms
// the two are faster still, but their sums are cut off, not rounded: sigma was off by 7e-7 of itself instead of 5e-8.
// Lower line, by the products to form: below, parts leave each CTA too few slabs and their sum is a launch more.  Split of 2304 x 256 at
// rank 128 (1.5e8 products in the Gram matrix) by gemm_simt / in parts 513 / 546 us, 3072 x 320 at rank 80 (3.1e8) 828 / 851, 2048 x 400
// (3.3e8) 1116 / 1100, 2600 x 400 (4.2e8) 1162 / 1139.
// The Gram matrix also needs half as many CTAs as there are SMs: with three parts at most, fewer tiles leave the device idle however long
// the reduction is, while gemm_simt's kernel for few tiles cuts it over clusters.  21 tiles (63 CTAs): 2800 x 384 962 / 992, 40000 x 384
// 1811 / 2058; 10 tiles: 20000 x 256 750 / 1011; one: 100000 x 64 641 / 2648.  28 tiles (84 CTAs): 8000 x 448 1389 / 1277, 40000 x 448
// 2697 / 2273; 55: 40000 x 640 4631 / 3464.
// Long product, also against the 8 x 8 kernel that gemm_simt has from 296 tiles on: 3072 x 768 at rank 192 (144 tiles) 2292 / 2216, at 400
// (336) 2425 / 2363, at 576 (432) 2399 / 2384; 4096 x 1024 at rank 320 3431 / 3285, at 512 3467 / 3435; 768 x 3072 at rank 480
// 2404 / 2403.  There sigma is off by 3.3e-8 of the largest where that kernel's fp32 sums left 5.5e-8.
constexpr int kParts = 3;
constexpr int64_t kPartsWork = 400000000;
bool in_parts(const SvdItem& it, const Plan& p, int64_t rows, int64_t len) {
  return it.w_dt == AB_F32 && p.s <= eig_max() && rows * p.s * len >= kPartsWork;
}
bool gram_in_parts(const SvdItem& it, const Plan& p) {
  const int64_t t = (p.s + 63) / 64, ctas = kParts * (t * (t + 1) / 2);
  return in_parts(it, p, p.s, p.L) && 2 * ctas >= sm_count();
}
bool long_in_parts(const SvdItem& it, const Plan& p) {      // room for one part at least
  return in_parts(it, p, p.r_cap, p.L) && (int64_t)p.r_cap * p.L <= (int64_t)kParts * p.s * p.s;
}
int part_len(int64_t tiles, int len, int most) {
  const int want = (int)std::max<int64_t>(1, std::min<int64_t>(most, (2LL * std::max(sm_count(), 1) + tiles / 2) / tiles));
  return ((len + want - 1) / want + 15) / 16 * 16;
}
// G = W^T W (tall) or W W^T
int gram_parts(const SvdItem& it, const Plan& p, float* G, double* parts, cudaStream_t st) {
  const float* W = static_cast<const float*>(it.W);
  const int64_t t = (p.s + 63) / 64, sr = p.tall ? 1 : it.n, sk = p.tall ? it.n : 1;
  const int per = part_len(t * (t + 1) / 2, p.L, kParts), n = (p.L + per - 1) / per;
  AB_TRY(gemm_parts(W, sr, sk, W, sk, sr, parts, p.s, p.s, p.L, per, true, st));
  const unsigned t32 = (unsigned)(p.s + 31) / 32;
  sum_gram_kernel<<<dim3(t32, t32), 256, 0, st>>>(parts, n, G, p.s);
  AB_LAUNCH_OK();
  return AB_OK;
}
// Y (L x r_cap) = W Vr^T (tall) or Y (r_cap x L) = Vr W
int long_parts(const SvdItem& it, const Plan& p, const float* Vr, float* Y, double* parts, cudaStream_t st) {
  const float* W = static_cast<const float*>(it.W);
  const int M = p.tall ? p.L : p.r_cap, N = p.tall ? p.r_cap : p.L;
  const int64_t tiles = (int64_t)((M + 63) / 64) * ((N + 63) / 64), count = (int64_t)M * N;
  const int per = part_len(tiles, p.s, (int)std::min<int64_t>(kParts, (int64_t)kParts * p.s * p.s / count)), n = (p.s + per - 1) / per;
  if (p.tall) AB_TRY(gemm_parts(W, it.n, 1, Vr, 1, p.s, parts, M, N, p.s, per, false, st));
  else AB_TRY(gemm_parts(Vr, p.s, 1, W, it.n, 1, parts, M, N, p.s, per, false, st));
  return sum_parts(parts, n, count, Y, st);
}

// Whether a group of `count` matrices of short side s goes to the direct solver (its fallback has to fit as well).
bool direct(int s, int count) { return s <= kEigSmallMax ? rows_jacobi_fits(count, s) : s <= eig_max(); }

}  // namespace

size_t svd_batch_ws(const SvdItem* items, int L) {
  return make_layout(items, L, nullptr).bytes;
}

int svd_batch(const SvdItem* items, int L, float sigma_cutoff, void* ws, size_t ws_bytes, cudaStream_t stream,
              const SvdSelftest* selftest) {
  Layout lo = make_layout(items, L, ws);
  if (lo.bytes > ws_bytes) return AB_ERR_WORKSPACE;
  // 1. Gram matrices into X
  for (auto& g : lo.groups) {
    const int s = g.first;
    for (size_t j = 0; j < g.second.size(); ++j) {
      const SvdItem& it = items[g.second[j]];
      float* G = lo.X[s] + j * (size_t)s * s;
      const Plan p = make_plan(it);
      if (gram_in_parts(it, p)) AB_TRY(gram_parts(it, p, G, lo.eig[s], stream));
      else if (it.m >= it.n)   // G = W^T W
        AB_TRY(gemm_simt(it.W, it.w_dt, 1, it.n, it.W, it.w_dt, it.n, 1, G, AB_F32, s, s, s, it.m, stream));
      else                // G = W W^T
        AB_TRY(gemm_simt(it.W, it.w_dt, it.n, 1, it.W, it.w_dt, 1, it.n, G, AB_F32, s, s, s, it.n, stream));
    }
  }
  // 2. eigen-decomposition of every group
  for (auto& g : lo.groups) {
    const int s = g.first, count = (int)g.second.size();
    Plan p = make_plan(items[g.second[0]]);
    float* lam = lo.item[g.second[0]].lam;
    int* perm = lo.item[g.second[0]].perm;
    if (direct(s, count)) {
      // The direct solver leaves the leading eigenvectors as unit rows in descending order in Vr (for a group that may
      // fall back to the Jacobi in shared memory: in Vt, where that leaves its rows).  Flagged matrices go on to the
      // Jacobi route of their size, whose kernels return at once for the others.
      const bool small = s <= kEigSmallMax;
      const int chunk = std::min(count, eig_chunk(s));
      std::vector<EigJob> ej((size_t)count);
      for (int j = 0; j < count; ++j) {
        EigJob& q = ej[j];
        const int idx = g.second[j];
        q.X = lo.X[s] + (size_t)j * s * s; q.gram = 0; q.s = s; q.need = make_plan(items[idx]).r_cap;
        q.rows = small ? lo.Vt[s] + (size_t)j * s * s : lo.item[idx].Vr; q.vals = nullptr; q.flag = lo.flags[s] + j;
        eig_bind(q, lo.eig[s] + (size_t)(j % chunk) * eig_ws_doubles(s));
      }
      AB_CUDA_OK(cudaMemsetAsync(lo.st[s], 0, sizeof(JState) * count, stream));
      AB_CUDA_OK(cudaMemsetAsync(lo.flags[s], 0, sizeof(int) * (count + 2 + eig_calls(s, count)), stream));
      AB_TRY(upload_async(lo.ejobs[s], ej.data(), ej.size() * sizeof(EigJob), stream));
      for (int j = 0; j < count; j += chunk)
        AB_TRY(eig_direct(ej.data() + j, lo.ejobs[s] + j, std::min(chunk, count - j), s, lo.flags[s] + count + 2 + j / chunk, stream));
      if (selftest) {
        force_fallback_kernel<<<1, 64, 0, stream>>>(lo.flags[s], count, lo.flags[s] + count + 2, selftest->flagged, selftest->solver_status);
        AB_LAUNCH_OK();
      }
      if (small) {
        AB_TRY(rows_jacobi(lo.X[s], lo.Vt[s], lam, &lo.st[s]->status, sizeof(JState), lo.flags[s], count, s, lo.jobs[s], stream));
        int r_need = 0;
        for (int idx : g.second) r_need = std::max(r_need, make_plan(items[idx]).r_cap);
        complete_basis_kernel<<<count, 256, 2 * (size_t)s * sizeof(float), stream>>>(lo.Vt[s], lam, lo.flags[s], s, r_need);
        AB_LAUNCH_OK();
      } else {
        init_state_kernel<<<dim3(64, (unsigned)count), 256, 0, stream>>>(lo.Vt[s], lo.st[s], s, lo.flags[s]);
        AB_LAUNCH_OK();
        AB_TRY(run_jacobi_fallback<32>(lo.X[s], lo.Vt[s], lo.st[s], lo.flags[s], s, p.nb, count, stream));
        norms_sort_kernel<<<count, 256, (size_t)s * sizeof(float), stream>>>(lo.X[s], s, lam, perm, lo.flags[s]);
        AB_LAUNCH_OK();
      }
      continue;
    }
    dim3 ig(64, (unsigned)count);
    init_state_kernel<<<ig, 256, 0, stream>>>(lo.Vt[s], lo.st[s], s, nullptr);
    AB_LAUNCH_OK();
    int rc;
    if (p.pb == 32) rc = run_jacobi<32>(lo.X[s], lo.Vt[s], lo.st[s], s, p.nb, count, stream);
    else rc = run_jacobi<16>(lo.X[s], lo.Vt[s], lo.st[s], s, p.nb, count, stream);
    AB_TRY(rc);
    norms_sort_kernel<<<count, 256, (size_t)s * sizeof(float), stream>>>(
        lo.X[s], s, lam, perm, nullptr);
    AB_LAUNCH_OK();
  }
  // 3. per matrix: leading vectors, long-side product, sigma, rank rule, factors
  for (auto& g : lo.groups) {
    const int s = g.first;
    for (size_t j = 0; j < g.second.size(); ++j) {
      const int i = g.second[j];
      const SvdItem& it = items[i];
      Plan p = make_plan(it);
      ItemWs w = lo.item[i];
      float* Vt = lo.Vt[s] + j * (size_t)s * s;
      const bool solved = direct(s, (int)g.second.size());
      if (solved && s <= kEigSmallMax) {
        w.Vr = Vt;                  // unit rows in order already
      } else {
        gather_rows_kernel<<<p.r_cap, 256, 0, stream>>>(Vt, w.perm, s, p.r_cap, w.Vr, solved ? lo.flags[s] + j : nullptr);
        AB_LAUNCH_OK();
      }
      int64_t yt, yk;   // Ylong(k,t) = Y[t*yt + k*yk]
      const bool parts = long_in_parts(it, p);
      if (parts) AB_TRY(long_parts(it, p, w.Vr, w.Y, lo.eig[s], stream));
      if (p.tall) {     // Y (m x r_cap) = W Vr^T
        if (!parts) AB_TRY(gemm_simt(it.W, it.w_dt, it.n, 1, w.Vr, AB_F32, 1, s, w.Y, AB_F32, p.r_cap, it.m, p.r_cap, it.n, stream));
        yt = p.r_cap; yk = 1;
      } else {          // Y (r_cap x n) = Vr W
        if (!parts) AB_TRY(gemm_simt(w.Vr, AB_F32, s, 1, it.W, it.w_dt, it.n, 1, w.Y, AB_F32, it.n, p.r_cap, it.n, it.m, stream));
        yt = 1; yk = it.n;
      }
      if (p.tall) {
        AB_TRY(launch_after(long_norms_kernel, dim3((unsigned)((p.r_cap + 31) / 32 * kNormCl)), 256, 0, kNormCl, stream, (const float*)w.Y, yt, p.L,
                            p.r_cap, it.sigma));
      } else {
        AB_TRY(launch_after(long_norms_rows_kernel, dim3((unsigned)p.r_cap), 256, 0, 1, stream, (const float*)w.Y, yk, p.L, it.sigma));
      }
      const int count = (int)g.second.size();
      const int* solver = solved ? lo.flags[s] + count + 2 + j / eig_chunk(s) : nullptr;
      const int rows = p.tall ? p.L + it.r_max : it.r_max + p.s;
      const unsigned grid = (unsigned)std::min((rows + 7) / 8, std::max(sm_count(), 1) * 4);
      void* Fl = p.tall ? it.A : it.B;
      void* Fs = p.tall ? it.B : it.A;
      if (it.out_dt == AB_F32)
        AB_TRY(launch_after(write_factors_kernel<float>, dim3(grid), 256, 0, 1, stream, (const float*)w.Y, (const float*)w.Vr, (const float*)it.sigma,
                            (int)p.tall, p.L, p.s, p.r_cap, it.r_max, sigma_cutoff, (float*)Fl, (float*)Fs, it.r_out, (const JState*)(lo.st[s] + j),
                            solver, it.dev_status));
      else
        AB_TRY(launch_after(write_factors_kernel<bf16>, dim3(grid), 256, 0, 1, stream, (const float*)w.Y, (const float*)w.Vr, (const float*)it.sigma,
                            (int)p.tall, p.L, p.s, p.r_cap, it.r_max, sigma_cutoff, (bf16*)Fl, (bf16*)Fs, it.r_out, (const JState*)(lo.st[s] + j),
                            solver, it.dev_status));
    }
  }
  return AB_OK;
}

}  // namespace ab
