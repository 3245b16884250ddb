// Batched products of fp32 (or bf16) matrices on the tensor cores, the operands cut into bf16 pieces on the way in.
//
//   C[M x N] = diag(rs) (A B^T) diag(cs)      A: M x K, B: N x K, either one stored with either index contiguous
//
// An fp32 value is hi + mid + lo, three bf16 pieces that carry 24 bits; the product is the six terms mid*mid,
// lo*hi, hi*lo, mid*hi, hi*mid (one accumulator) and hi*hi (another, added to the first in the epilogue), each bf16
// product exact in fp32: what is lost is the three products of order 2^-24 and the rounding of the fp32 sums.  bf16
// operands are one term.
//
// This is every product of the factored group synchronisation -- Gram matrices, r x r products, the new factors,
// W = Abar Bbar -- and ab_recombine.  The pieces used to be made by a kernel of their own, written to memory and fetched
// through tensor maps, and the r x r products ran on the fp32 pipes.  Here the converter warps read the operand as it
// lies, and write the pieces straight into the swizzled tiles that the MMAs read: no pieces in memory, no tensor
// maps to encode and upload, one launch where there were three.  Per slab of 64 of the reduction the conversion runs
// beside the 24 MMAs (1570 cycles at 128 columns) of the slab before it.
//
// Persistent CTAs: CTA b takes tiles b, b + grid, ... of all problems of the launch.  Warps 0..7 convert, warps
// 8..11 empty the accumulators (two pairs, used in turn), warp 12 issues the MMAs, warp 13 finds the tiles' problems
// and hands their records round through shared memory.  Every wait is bounded.
#include "ab_common.cuh"
#include "ab_tc_ptx.cuh"

namespace ab {
namespace {

using namespace tc;

constexpr int kM = 128;                  // rows of a tile
constexpr int kConvWarps = 8;
constexpr int kConvThreads = 32 * kConvWarps;
constexpr int kMmaWarp = kConvWarps + 4, kFindWarp = kMmaWarp + 1;
constexpr int kThreads = 32 * (kConvWarps + 8);          // four warpgroups; the last holds the MMA warp
// Registers a thread by role, of the 4 x 128 the block is launched with.
constexpr int kRegsConv = 152, kRegsEpi = 120, kRegsMma = 80;
static_assert(2 * kRegsConv + kRegsEpi + kRegsMma <= 512, "");
constexpr int kRing = 4;                 // tile records on their way to the other warps

// Bytes of a piece of an operand tile: where the index of the rows is contiguous, its lines are 64 values long, also of 32 rows.
constexpr int piece_bytes(int rows) { return (rows < 64 ? 64 : rows) * 128; }

template <int BN, bool kBf16>
struct Cfg {
  static constexpr int kPieces = kBf16 ? 1 : 3;
  static constexpr int kStages = kBf16 ? 4 : 2;
  static constexpr int kABytes = piece_bytes(kM), kBBytes = piece_bytes(BN);
  static constexpr int kStage = kPieces * (kABytes + kBBytes);
  static constexpr size_t kSmem = (size_t)kStages * kStage + 4 * 4096 + 1024 + 2048;
};

struct TileRecord { SplitGemm P; int m0, n0, last; };
struct SplitBars {
  uint64_t full[4], empty[4], acc_full[2], acc_empty[2], rec_full[kRing], rec_empty[kRing];
  uint32_t tmem_base;
  int abort_any;
  TileRecord rec[kRing];
};
static_assert(sizeof(SplitBars) <= 2048 && sizeof(SplitGemm) % 8 == 0, "");

// the whole warp waits, one lane polls; the verdict is a vote, on which the compiler branches uniformly
__device__ __forceinline__ bool split_warp_wait(SplitBars* b, uint64_t* bar, uint32_t parity, int* status) {
  bool ok = true;
  if ((threadIdx.x & 31) == 0) {
    ok = mbar_wait(bar, parity);
    if (!ok) {
      *reinterpret_cast<volatile int*>(&b->abort_any) = 1;
      atomicExch(status, (int)AB_ERR_TIMEOUT);
    }
  }
  return __all_sync(0xffffffffu, ok);
}

// A consumer warp's walk over its CTA's tiles.  Several problems: records handed round by the finder warp.  One problem: it lies
// in the kernel's parameters and a tile follows from its number, so no warp waits for another (through records 3300 cycles
// passed from the start to the first load, as many as two slabs take; 768 x 768 x 192 11.4 -> 7.9 us, of it also
// the epilogue without scaling code, 4300 -> 2200 cycles).
struct TileAt { const SplitGemm* P; int m0, n0; };
template <bool kOne, int BN>
struct TileReader {
  int slot = 0, ph = 0;
  // the next tile; P is null after the last one (or when a wait gave up)
  __device__ __forceinline__ TileAt next(SplitBars* b, const SplitGemm* probs, int ntiles, int* status) {
    if constexpr (kOne) {
      const int tile = (int)blockIdx.x + slot++ * (int)gridDim.x;
      if (tile >= ntiles) return {nullptr, 0, 0};
      const int tn = (probs->N + BN - 1) / BN, tm = tile / tn;
      return {probs, tm * kM, (tile - tm * tn) * BN};
    } else {
      if (!split_warp_wait(b, &b->rec_full[slot], ph, status)) return {nullptr, 0, 0};
      const TileRecord* r = &b->rec[slot];
      if (__any_sync(0xffffffffu, r->last)) return {nullptr, 0, 0};
      return {&r->P, r->m0, r->n0};
    }
  }
  __device__ __forceinline__ void done(SplitBars* b) {     // the record has been read
    if constexpr (kOne) return;
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&b->rec_empty[slot]);
    if (++slot == kRing) { slot = 0; ph ^= 1; }
  }
};

__device__ __forceinline__ float split_diag(const float* v, int idx, int mode, float thr) {
  if (mode == 0 || v == nullptr) return 1.f;
  const float x = v[idx];
  if (!(x > thr * v[0]) || !(x > 0.f)) return 0.f;
  return mode == 1 ? sqrtf(x) : 1.f / sqrtf(x);
}

// One operand's share of a slab, kRows x 64 values, as a thread holds it: kF groups of 16 bytes.
// Element (row, k) of the operand is at p[row * ld + k] (mn false) or p[k * ld + row] (mn true).  What lies past the
// reduction arrives as zero; rows past the operand feed only rows or columns that are never stored.
// A thread's groups lie kStep lines apart (a line: the 64 or kRows contiguous values of a row or of a k), a multiple
// of 8, so their places in the swizzled tile differ by a constant.
template <int kRows, bool kBf16>
struct OperandSlab {
  static constexpr int kPer = kBf16 ? 8 : 4;                        // values per group
  static constexpr int kF = kRows * 64 / kPer / kConvThreads;
  static constexpr int kStepK = kConvThreads / (64 / kPer), kStepMn = kConvThreads / (kRows / kPer);
  static_assert(kF >= 1 && kStepK % 8 == 0 && kStepMn % 8 == 0, "");
  uint4 q[kF];
};
template <int kRows, bool kBf16>
struct OperandCursor {
  using Slab = OperandSlab<kRows, kBf16>;
  static constexpr int kPer = Slab::kPer, kF = Slab::kF;
  static constexpr int64_t kSize = kBf16 ? 2 : 4;
  const char* p;            // this thread's first group of the next slab
  int64_t step, adv;        // bytes from group to group, from slab to slab
  uint32_t soff;            // place of the first group in the tile
  int line, left;           // k of the first group (mn) or its offset in the slab; values of a group that exist
  uint32_t mask;            // groups whose row exists
  bool mn, vec;

  __device__ __forceinline__ void start(const void* base, int64_t ld, bool mn_, int row0, int rows, int tid) {
    mn = mn_;
    constexpr int al = kBf16 ? 8 : 4;
    vec = (reinterpret_cast<uintptr_t>(base) & 15u) == 0 && ld % al == 0;
    if (mn) {
      const int c = (tid % (kRows / kPer)) * kPer;
      line = tid / (kRows / kPer);
      left = rows - (row0 + c);
      mask = left > 0 ? 0xffffffffu : 0u;
      p = static_cast<const char*>(base) + ((int64_t)line * ld + row0 + c) * kSize;
      step = Slab::kStepMn * ld * kSize;
      adv = 64 * ld * kSize;
      soff = (c >> 6) * 8192 + line * 128 + ((((c & 63) >> 3) ^ (line & 7)) << 4) + (kBf16 ? 0 : (c & 4) * 2);
    } else {
      const int c = (tid % (64 / kPer)) * kPer, r = tid / (64 / kPer);
      line = c;
      left = kPer;
      mask = 0u;
#pragma unroll
      for (int e = 0; e < kF; ++e) if (row0 + r + e * Slab::kStepK < rows) mask |= 1u << e;
      p = static_cast<const char*>(base) + ((int64_t)(row0 + r) * ld + c) * kSize;
      step = Slab::kStepK * ld * kSize;
      adv = 64 * kSize;
      soff = r * 128 + (((c >> 3) ^ (r & 7)) << 4) + (kBf16 ? 0 : (c & 4) * 2);
    }
  }
  // klen: values of the reduction in this slab (64 but for the last)
  __device__ __forceinline__ void load(Slab& s, int klen) {
    if (vec && klen == 64 && left >= kPer) {
#pragma unroll
      for (int e = 0; e < kF; ++e) {
        s.q[e] = make_uint4(0u, 0u, 0u, 0u);
        if (mask >> e & 1u) s.q[e] = *reinterpret_cast<const uint4*>(p + e * step);
      }
    } else {
#pragma unroll
      for (int e = 0; e < kF; ++e) {
        const int n = mn ? (line + e * Slab::kStepMn < klen ? left : 0) : klen - line;     // values of the group that exist
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (mask >> e & 1u) {
          const char* g = p + e * step;
#pragma unroll
          for (int j = 0; j < kPer; ++j)
            if (j < n) {
              if constexpr (kBf16) w[j >> 1] |= (uint32_t)reinterpret_cast<const uint16_t*>(g)[j] << (16 * (j & 1));
              else w[j] = reinterpret_cast<const uint32_t*>(g)[j];
            }
        }
        s.q[e] = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    p += adv;
  }
};
// into the 128-byte-swizzled tile(s): lines of 128 bytes (64 values); piece p at dst + p * kPieceBytes
template <int kRows, bool kBf16>
__device__ __forceinline__ void store_slab(const OperandSlab<kRows, kBf16>& s, uint8_t* dst, uint32_t estep) {
  constexpr int kPieceBytes = piece_bytes(kRows);
#pragma unroll
  for (int e = 0; e < OperandSlab<kRows, kBf16>::kF; ++e) {
    uint8_t* b = dst + e * estep;
    const uint4 q = s.q[e];
    if constexpr (kBf16) {
      *reinterpret_cast<uint4*>(b) = q;
    } else {
      const float x[4] = {__uint_as_float(q.x), __uint_as_float(q.y), __uint_as_float(q.z), __uint_as_float(q.w)};
      uint32_t h[2], m[2], l[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        __nv_bfloat162 t = __floats2bfloat162_rn(x[2 * u], x[2 * u + 1]);
        h[u] = *reinterpret_cast<uint32_t*>(&t);
        const float r0 = x[2 * u] - __uint_as_float(h[u] << 16), r1 = x[2 * u + 1] - __uint_as_float(h[u] & 0xffff0000u);
        t = __floats2bfloat162_rn(r0, r1);
        m[u] = *reinterpret_cast<uint32_t*>(&t);
        t = __floats2bfloat162_rn(r0 - __uint_as_float(m[u] << 16), r1 - __uint_as_float(m[u] & 0xffff0000u));
        l[u] = *reinterpret_cast<uint32_t*>(&t);
      }
      *reinterpret_cast<uint2*>(b) = make_uint2(h[0], h[1]);
      *reinterpret_cast<uint2*>(b + kPieceBytes) = make_uint2(m[0], m[1]);
      *reinterpret_cast<uint2*>(b + 2 * kPieceBytes) = make_uint2(l[0], l[1]);
    }
  }
}

template <int BN, bool kBf16, bool kOne>
__device__ __forceinline__ void gemm_split_body(const SplitGemm* probs, int nprobs, int ntiles, int* status) {
  using C = Cfg<BN, kBf16>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* stg = smem + C::kStages * C::kStage;
  SplitBars* bars = reinterpret_cast<SplitBars*>(stg + 4 * 4096);
  const int tid = threadIdx.x, warp = (int)uniform((uint32_t)tid >> 5), lane = tid & 31;

  if (tid == 0) {
    for (int i = 0; i < C::kStages; ++i) { mbar_init(&bars->full[i], kConvWarps); mbar_init(&bars->empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&bars->acc_full[i], 1); mbar_init(&bars->acc_empty[i], 4); }
    for (int i = 0; i < kRing; ++i) { mbar_init(&bars->rec_full[i], 1); mbar_init(&bars->rec_empty[i], kConvWarps + 5); }
    bars->abort_any = 0;
    fence_barrier_init();
  }
  if (warp == kMmaWarp) tmem_alloc(&bars->tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);
  if constexpr (!kOne) {       // one problem: each role finds its first tile before it waits
    dep_wait();
    dep_launch();
  }

  if (warp < kConvWarps) {
    // ------------------------------------------------------------ converters
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsConv));
    using SA = OperandSlab<kM, kBf16>;
    using SB = OperandSlab<BN, kBf16>;
    OperandCursor<kM, kBf16> ca;
    OperandCursor<BN, kBf16> cb;
    TileReader<kOne, BN> rd;
    int K = 0, k0 = 0, slot = 0, ph = 1;
    auto open = [&]() -> bool {
      const TileAt t = rd.next(bars, probs, ntiles, status);
      if (!t.P) return false;
      ca.start(t.P->A, t.P->lda, t.P->a_mn, t.m0, t.P->M, tid);
      cb.start(t.P->B, t.P->ldb, t.P->b_mn, t.n0, t.P->N, tid);
      K = t.P->K;
      k0 = 0;
      rd.done(bars);
      return true;
    };
    auto load = [&](SA& a, SB& b) { ca.load(a, min(64, K - k0)); cb.load(b, min(64, K - k0)); k0 += 64; };
    auto fetch = [&](SA& a, SB& b) -> bool {
      if (k0 >= K && !open()) return false;
      load(a, b);
      return true;
    };
    auto put = [&](const SA& a, const SB& b) -> bool {
      if (!split_warp_wait(bars, &bars->empty[slot], ph, status)) return false;
      uint8_t* dst = smem + (size_t)slot * C::kStage;
      store_slab<kM, kBf16>(a, dst + ca.soff, (ca.mn ? SA::kStepMn : SA::kStepK) * 128);
      store_slab<BN, kBf16>(b, dst + C::kPieces * C::kABytes + cb.soff, (cb.mn ? SB::kStepMn : SB::kStepK) * 128);
      fence_proxy_async_smem();                          // before the next loads: it waits for what is in flight
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->full[slot]);
      if (++slot == C::kStages) { slot = 0; ph ^= 1; }
      return true;
    };
    bool h0 = open();
    if constexpr (kOne) {
      dep_wait();
      dep_launch();
      // a wait gives up only after about a second: this cannot wipe a raised error
      if (blockIdx.x == 0 && tid == 0) atomicExch(status, 0);
    }
    SA a0;
    SB b0;
    if (h0) load(a0, b0);
    while (h0) {
      if (!put(a0, b0)) break;
      h0 = fetch(a0, b0);
    }
  } else if (warp >= kMmaWarp) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsMma));
    if (warp == kMmaWarp) {
      // ---------------------------------------------------------- MMA issuer (see elect_one for the uniform loop)
      if constexpr (kOne) {
        dep_launch();            // the kernel behind may set itself up already: it waits for this one as a whole
        dep_wait();              // no bounded wait starts before the kernel in front is done: it may take longer than a wait may
      }
      TileReader<kOne, BN> rd;
      int slot = 0, ph = 0;
      bool ok = true;
      const uint32_t sbase = uniform(smem_u32(smem)), tbase = uniform(tmem_base);
      for (int it = 0; ok; ++it) {
        const TileAt t = rd.next(bars, probs, ntiles, status);
        if (!t.P) break;
        const int amn = (int)uniform(t.P->a_mn), bmn = (int)uniform(t.P->b_mn), K = (int)uniform(t.P->K),
                  ncols = (int)uniform(min(BN, t.P->N - t.n0));
        rd.done(bars);
        const uint32_t idesc = instr_desc_bf16(kM, (ncols + 15) & ~15, amn, bmn);
        const int buf = it & 1;
        if (!split_warp_wait(bars, &bars->acc_empty[buf], ((it >> 1) & 1) ^ 1, status)) break;
        tc_fence_after();
        const uint32_t acc = tbase + 256 * buf;             // hi * hi; the five small terms at + 128
        const uint64_t da0 = smem_desc_sw128(sbase, amn ? 8192 : 16);
        const uint64_t db0 = smem_desc_sw128(sbase + C::kPieces * C::kABytes, bmn ? 8192 : 16);
        const uint64_t as = amn ? 128u : 2u, bs = bmn ? 128u : 2u;       // 16 of the reduction, in 16-byte units
        for (int k0 = 0; k0 < K; k0 += 64) {
          ok = split_warp_wait(bars, &bars->full[slot], ph, status);
          if (!ok) break;
          tc_fence_after();
          const uint64_t da = da0 + (uint64_t)(slot * (C::kStage >> 4)), db = db0 + (uint64_t)(slot * (C::kStage >> 4));
          const int ksteps = min(4, (K - k0 + 15) >> 4);
          if (elect_one()) {
            if constexpr (kBf16) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                if (kk < ksteps) tc_mma_bf16(acc, da + as * kk, db + bs * kk, idesc, (k0 | kk) ? 1u : 0u);
            } else {
              constexpr uint64_t pa = C::kABytes >> 4, pb = C::kBBytes >> 4;
              constexpr int ta[6] = {1, 2, 0, 1, 0, 0}, tb[6] = {1, 0, 2, 0, 1, 0};
#pragma unroll
              for (int u = 0; u < 6; ++u)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                  if (kk < ksteps)
                    tc_mma_bf16(u < 5 ? acc + 128 : acc, da + pa * ta[u] + as * kk, db + pb * tb[u] + bs * kk, idesc,
                                (k0 | kk | (u % 5)) ? 1u : 0u);
            }
            tc_commit(&bars->empty[slot]);
          }
          __syncwarp();
          if (++slot == C::kStages) { slot = 0; ph ^= 1; }
        }
        if (ok && elect_one()) tc_commit(&bars->acc_full[buf]);
        __syncwarp();
      }
    } else if (!kOne && warp == kFindWarp) {
      // ---------------------------------------------------------- tile finder
      int idx = 0, slot = 0, ph = 1;
      for (int tile = blockIdx.x;; tile += gridDim.x) {
        TileRecord* r = &bars->rec[slot];
        int m0 = 0, n0 = 0;
        const bool last = tile >= ntiles;
        if (!last) {
          for (;;) {                      // the last problem whose first tile is <= tile; 32 candidates at a time
            const int c = idx + 1 + lane;
            const int n = __popc(__ballot_sync(0xffffffffu, c < nprobs && probs[c < nprobs ? c : idx].first_tile <= tile));
            idx += n;
            if (n < 32) break;
          }
          const SplitGemm* P = probs + idx;
          const int k = tile - P->first_tile, tn = (P->N + BN - 1) / BN;
          m0 = (k / tn) * kM;
          n0 = (k - (k / tn) * tn) * BN;
          if (P->upper_only && n0 + BN <= m0) continue;
        }
        if (!split_warp_wait(bars, &bars->rec_empty[slot], ph, status)) break;
        if (!last)
          for (int w = lane; w < (int)(sizeof(SplitGemm) / 8); w += 32)
            reinterpret_cast<uint64_t*>(&r->P)[w] = reinterpret_cast<const uint64_t*>(probs + idx)[w];
        if (lane == 0) { r->m0 = m0; r->n0 = n0; r->last = last; }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->rec_full[slot]);
        if (last) break;
        if (++slot == kRing) { slot = 0; ph ^= 1; }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    const int qw = warp & 3;                             // the quarter of the TMEM lanes this warp may read
    uint8_t* mystg = stg + qw * 4096;
    const uint32_t lane_base = (uint32_t)(qw * 32) << 16;
    if constexpr (kOne) {
      dep_wait();
      dep_launch();
    }
    TileReader<kOne, BN> rd;
    for (int it = 0;; ++it) {
      const TileAt t = rd.next(bars, probs, ntiles, status);
      if (!t.P) break;
      const int M = t.P->M, N = t.P->N, c_bf16 = t.P->c_bf16, m0 = t.m0, n0 = t.n0;
      const int64_t ldc = t.P->ldc;
      void* Cp = t.P->C;
      const float *row_vec = t.P->row_vec, *col_vec = t.P->col_vec, thr = t.P->thr;
      const int row_mode = t.P->row_mode, col_mode = t.P->col_mode;
      const int *lr = t.P->live_rows, *lc = t.P->live_cols;
      rd.done(bars);
      const int live_r = lr ? min(*lr, M) : M, live_c = lc ? min(*lc, N) : N;
      const int row = m0 + qw * 32 + lane;
      const float rs = row < live_r ? split_diag(row_vec, row, row_mode, thr) : 0.f;
      const bool cvec = (reinterpret_cast<uintptr_t>(Cp) & 15u) == 0 && ldc % 4 == 0;
      const bool rows_in = m0 + qw * 32 < M;
      const int ncols = min(BN, N - n0);
      const int buf = it & 1;
      if (!split_warp_wait(bars, &bars->acc_full[buf], (it >> 1) & 1, status)) break;
      tc_fence_after();
      const uint32_t acc = tmem_base + 256 * buf + lane_base;
      for (int c0 = 0; c0 < ncols; c0 += 32) {
        uint32_t v[2][16], u[2][16];
        if (rows_in) {
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            tmem_ld16_nowait(acc + c0 + 16 * g, v[g]);
            if constexpr (!kBf16) tmem_ld16_nowait(acc + 128 + c0 + 16 * g, u[g]);
          }
          tmem_wait_ld();
        }
        if (c0 + 32 >= ncols) {                          // the last piece is in registers: hand the accumulators back
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->acc_empty[buf]);
        }
        if (!rows_in) continue;
        __syncwarp();                                    // the staging tile has been read
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
          float x[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int g = ch >> 2, e = (ch & 3) * 4 + j;
            x[j] = __uint_as_float(v[g][e]);
            if constexpr (!kBf16) x[j] += __uint_as_float(u[g][e]);
            x[j] = rs == 0.f ? 0.f : x[j] * rs;
          }
          *reinterpret_cast<float4*>(mystg + lane * 128 + ((ch ^ (lane & 7)) << 4)) = make_float4(x[0], x[1], x[2], x[3]);
        }
        __syncwarp();
        const int ch = lane & 7, col = n0 + c0 + ch * 4;        // 8 lanes a row, 4 rows at a time
        float cs[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) cs[j] = col + j < live_c ? split_diag(col_vec, col + j, col_mode, thr) : 0.f;
        const bool plain = cs[0] == 1.f && cs[1] == 1.f && cs[2] == 1.f && cs[3] == 1.f;
        const int nrows = min(32, M - (m0 + qw * 32)), ncol = N - col, r0 = lane >> 3;
        const int64_t off0 = (int64_t)(m0 + qw * 32 + r0) * ldc + col;
        float4 q[8];
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) q[rr] = *reinterpret_cast<const float4*>(mystg + (rr * 4 + r0) * 128 + ((ch ^ ((rr * 4 + r0) & 7)) << 4));
        if (!plain) {
#pragma unroll
          for (int rr = 0; rr < 8; ++rr) {
            q[rr].x = cs[0] == 0.f ? 0.f : q[rr].x * cs[0]; q[rr].y = cs[1] == 0.f ? 0.f : q[rr].y * cs[1];
            q[rr].z = cs[2] == 0.f ? 0.f : q[rr].z * cs[2]; q[rr].w = cs[3] == 0.f ? 0.f : q[rr].w * cs[3];
          }
        }
        if (cvec && nrows == 32 && n0 + c0 + 32 <= N) {          // a whole piece: no checks between the stores
          if (c_bf16) {
            uint2* o = reinterpret_cast<uint2*>(static_cast<bf16*>(Cp) + off0);
#pragma unroll
            for (int rr = 0; rr < 8; ++rr) {
              __nv_bfloat162 lo = __floats2bfloat162_rn(q[rr].x, q[rr].y), hi = __floats2bfloat162_rn(q[rr].z, q[rr].w);
              o[rr * ldc] = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
            }
          } else {
            float4* o = reinterpret_cast<float4*>(static_cast<float*>(Cp) + off0);
#pragma unroll
            for (int rr = 0; rr < 8; ++rr) o[rr * ldc] = q[rr];      // 4 rows of 4-value groups: ldc groups on
          }
        } else {
#pragma unroll
          for (int rr = 0; rr < 8; ++rr) {
            if (rr * 4 + r0 >= nrows) continue;
            const float x[4] = {q[rr].x, q[rr].y, q[rr].z, q[rr].w};
            const int64_t off = off0 + rr * 4 * ldc;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              if (j >= ncol) continue;
              if (c_bf16) static_cast<bf16*>(Cp)[off + j] = __float2bfloat16_rn(x[j]);
              else static_cast<float*>(Cp)[off + j] = x[j];
            }
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (*reinterpret_cast<volatile int*>(&bars->abort_any)) {     // MMAs that were issued finish before TMEM is given back
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) { }
    __syncthreads();
  }
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
gemm_split_batched_kernel(const SplitGemm* __restrict__ probs, int nprobs, int ntiles, int* status) {
  gemm_split_body<BN, false, false>(probs, nprobs, ntiles, status);
}
template <int BN, bool kBf16>
__global__ void __launch_bounds__(kThreads, 1)
gemm_split_one_kernel(const __grid_constant__ SplitGemm p, int ntiles, int* status) {
  gemm_split_body<BN, kBf16, true>(&p, 1, ntiles, status);
}

template <typename... KArgs, typename... Args>
int launch(void (*kernel)(KArgs...), size_t smem, int tiles, cudaStream_t st, Args... args) {
  const int sms = sm_count();
  if (sms <= 0) return AB_ERR_CUDA;
  AB_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  return launch_after(kernel, (unsigned)(tiles < sms ? tiles : sms), (unsigned)kThreads, smem, 1, st, args...);
}

int tiles_of(const SplitGemm& p, int bn) { return ((p.M + kM - 1) / kM) * ((p.N + bn - 1) / bn); }

// Tiles of a batch, and of a problem too large for narrow_tiles: 128 or 64 columns wide, whichever takes less time: a wide one about one
// and a half times a narrow one (its A is converted once instead of twice).  768 x 768: 36 or 72 tiles, one round of either: 64.  3072 x 768: 144 wide ones in one round, 288
// narrow ones in two: 128 (10.4 us against 12.4 us).
int tile_width(int tiles64, int tiles128) {
  const int sms = sm_count() > 0 ? sm_count() : 1;
  return 2 * ((tiles64 + sms - 1) / sms) >= 3 * ((tiles128 + sms - 1) / sms) ? 128 : 64;
}

// Up to how many tiles of 32 columns a lone problem takes them.  What a CTA converts and writes is a chain of latencies, so less of it
// is faster as long as every tile has an SM, and the CTAs of the launch behind find room beside.  us a launch in a row of twelve, 64 wide
// / 32 wide: 256 x 256, rank 64, fp32 4.9 / 4.4, bf16 3.4 / 3.2; 512 x 512, rank 192 7.5 / 6.8, 4.6 / 4.2; 1000 x 448 (112
// tiles), rank 192 7.7 / 7.3, 4.8 / 4.6.  With nearly every SM taken the next launch waits outside, which a reduction of one slab
// and the lighter bf16 conversion do not make up for: 768 x 768 (144 tiles), rank 64 5.4 / 5.6, 3.6 / 4.0, rank 192 7.7 / 7.6, 4.7 / 4.8.
int narrow_tiles(bool src_bf16, int K) {
  const int sms = sm_count();
  return !src_bf16 && K > 64 ? sms : sms / 5 * 4;
}

}  // namespace

SplitBatch gemm_split_plan(SplitGemm* probs, int count) {
  SplitBatch b;
  int t64 = 0, t128 = 0;
  for (int i = 0; i < count; ++i) { t64 += tiles_of(probs[i], 64); t128 += tiles_of(probs[i], 128); }
  b.count = count;
  b.bn = tile_width(t64, t128);
  b.tiles = 0;
  for (int i = 0; i < count; ++i) { probs[i].first_tile = b.tiles; b.tiles += tiles_of(probs[i], b.bn); }
  return b;
}

int gemm_split_batched(const SplitGemm* d_probs, const SplitBatch& b, int* status, cudaStream_t st) {
  if (b.count <= 0 || b.tiles <= 0) return AB_OK;
  if (b.bn == 128) return launch(gemm_split_batched_kernel<128>, Cfg<128, false>::kSmem, b.tiles, st, d_probs, b.count, b.tiles, status);
  return launch(gemm_split_batched_kernel<64>, Cfg<64, false>::kSmem, b.tiles, st, d_probs, b.count, b.tiles, status);
}

int gemm_split_one(SplitGemm p, bool src_bf16, int* status, cudaStream_t st) {
  const int t32 = tiles_of(p, 32);
  if (t32 <= narrow_tiles(src_bf16, p.K)) {
    if (src_bf16) return launch(gemm_split_one_kernel<32, true>, Cfg<32, true>::kSmem, t32, st, p, t32, status);
    return launch(gemm_split_one_kernel<32, false>, Cfg<32, false>::kSmem, t32, st, p, t32, status);
  }
  const SplitBatch b = gemm_split_plan(&p, 1);
  if (src_bf16) {
    if (b.bn == 128) return launch(gemm_split_one_kernel<128, true>, Cfg<128, true>::kSmem, b.tiles, st, p, b.tiles, status);
    return launch(gemm_split_one_kernel<64, true>, Cfg<64, true>::kSmem, b.tiles, st, p, b.tiles, status);
  }
  if (b.bn == 128) return launch(gemm_split_one_kernel<128, false>, Cfg<128, false>::kSmem, b.tiles, st, p, b.tiles, status);
  return launch(gemm_split_one_kernel<64, false>, Cfg<64, false>::kSmem, b.tiles, st, p, b.tiles, status);
}

}  // namespace ab
