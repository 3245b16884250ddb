// Fused tensor-core chain for bf16 storage (fp32 accumulation) on sm_100a.
//
// chain_kernel: persistent CTAs; for a block of 128 rows  S = In F1^T  (128 x r, K-loop over the input
// width, accumulator in TMEM), S rounded to bf16 into shared memory, multiplied on:  Out = S F2^T  in
// 256-column chunks.  The rank-r intermediate never goes to HBM unless the caller asks for a copy.
//   forward : In = x,  F1 = B   (r x n), F2 = A   (m x r), Out = y,  S = T
//   backward: In = dY, F1 = A^T (r x m), F2 = B^T (n x r), Out = dX, S = dT   (A and B read as they lie)
// grad_kernel: dA = dY^T T and dB^T = x^T dT are reductions over the rows; a CTA owns 256 output rows (a
// slice of m or of n) and one slice of the N rows and streams 64-row slabs of both operands (both "MN-major": the reduction
// index is the slow one in memory).  Where a tile has several slices each leaves its sums in memory and
// reduce_partials_kernel adds them in a fixed order.
//
// All operand tiles are TMA boxes of 64 bf16 (128 bytes) x rows with 128-byte swizzle.  Every mbarrier
// wait gives up after about a second, raises AB_ERR_TIMEOUT in the status word and unwinds to the common
// exit, where TMEM is released.
#include <cooperative_groups.h>

#include <cstring>
#include <mutex>

#include "ab_common.cuh"
#include "ab_tc_ptx.cuh"

namespace ab {
namespace {

using namespace tc;

constexpr int kAtomBytes = 16384;      // 128 rows x 128 bytes
constexpr int kMaxStages = 10;
constexpr int kMaxStages2 = 6;         // 32 KB slots of the second product, carved from the same ring memory
constexpr int kChunk = 256;            // output columns per accumulator of the second product
constexpr int kAtom2Bytes = kChunk * 128;   // one 256 x 64 tile of F2
constexpr int kSmemLimit = kMaxSmem;
constexpr int kTmemCols = 512;
constexpr int kEpiThreads = 128;

constexpr int kEpiWarps = 4;                         // one per quarter of the TMEM lanes
constexpr int kStgTiles = 2;                         // staging tiles per epilogue warp
constexpr int kChainThreads = 32 * (2 + kEpiWarps);
constexpr int kGroupRows = 32;                   // rows are dealt to CTAs, loaded and stored in groups of 32
constexpr int kGroupBytes = kGroupRows * 128;    // one group of one 64-column tile
constexpr int kF1AtomBytes = 8192;               // 64 x 64 box of an MN-major factor

// Convolution mode (3 x 3, stride 1, padding 1, activations NHWC): the rows of In are never materialised.  A
// block is a tile of whole image rows (bh rows of one image, or bb whole images when an image has at most 128
// pixels), i.e. a run of consecutive pixels; slab kr of the reduction is tap kr / cslabs and 64 channels, and the
// block's In tile for it is the 4-D box of the activation shifted by the tap (what falls outside an image
// arrives as zeros: the padding).  The factor's slab is found at column tap * tap_stride (+ f1_col_off).
struct ConvGeom {
  int on;
  int B, H, W;
  int in_ch;       // channels of the In tensor
  int cslabs;      // ceil(in_ch / 64)
  int bh, bb;      // tile: bh image rows (bb == 1) or bb whole images (bh == H)
  int tpi;         // tiles per image (bb == 1) or 1
  int box_rows;    // W * bh * bb: rows one In box delivers
  int sign;        // +1: In pixel = out pixel + (tap - 1); -1: In pixel = out pixel - (tap - 1)
  int tap_stride;  // columns of the factor between taps
  int f1_col_off;  // first column of this launch's factor window inside a tap
  int s_col_off;   // first column of S in the output it is stored to
};

struct ChainParams {
  int K1;        // width of In (reduction length of the first product)
  int P;         // width of Out (0: first product only)
  int r;         // rank, padded to a multiple of 16
  int nk1;       // ceil(K1 / 64)
  int nchunks;   // ceil(P / 256)
  int natoms;    // ceil(r / 64)
  int max_blocks;          // 128-row blocks per unit: 1 or 2
  int ns, slot_bytes;      // first product: slots of max_blocks In tiles + one slab of F1
  int ns2;                 // second product: 32 KB slots at the start of shared memory
  int f1_bytes;            // bytes of one F1 slab as the loads deliver it
  int f1_mn, f2_mn;        // 1: the factor is held with the reduction index as the slow one (MN-major operand)
  int save_s;              // 1: copy S to global through tmS
  int groups;              // work items in all: 32-row groups, or tiles of a convolution (see ConvGeom)
  int deal;                // items are dealt to the CTAs in runs of this many
  ConvGeom cv;
  bf16* out_ptr;           // convolution mode: Out and S as plain pointers for the rows of a tile's last, partial
  bf16* s_ptr;             //   group of 32 (row strides P and s_ld)
  int s_ld, s_cols;        // s_cols: true width of S
  int clear_status;        // 1: this is the first kernel of a call and zeroes the status word (see clear_status_word)
  int stall_selftest;      // 1: the producer loads nothing, so every wait of the kernel runs out (failure-path self-test)
  unsigned long long wait_ns;   // limit of every on-chip wait
  int* status;
};

struct Bars {
  uint64_t full[kMaxStages], empty[kMaxStages];
  uint64_t full2[kMaxStages2], empty2[kMaxStages2];
  uint64_t t_full, s_ready, unit_done;
  uint64_t acc_full[2], acc_empty[2];
  uint32_t tmem_base;
  int abort_any;   // set by any role that gave up
  int epi_abort;   // used by the gradient kernel's epilogue warps around their own barrier
};

__device__ __forceinline__ void raise_timeout(Bars* b, int* status) {
  *reinterpret_cast<volatile int*>(&b->abort_any) = 1;
  atomicExch(status, (int)AB_ERR_TIMEOUT);
}

// The status word of a call starts at zero.  The first kernel of the call clears it itself (block 0,
// right after dep_wait) instead of a memset in the stream, which would sit between this kernel and the
// one before it and undo the overlap of dep_wait.  Block 0 runs in the first wave and gets here within
// microseconds of the launch; a kernel raises AB_ERR_TIMEOUT only after a wait of about a second, so
// the clear cannot wipe a raised error.
__device__ __forceinline__ void clear_status_word(int enabled, int* status) {
  if (enabled && blockIdx.x == 0 && threadIdx.x == 0) atomicExch(status, 0);
}

// epilogue-wide wait of the gradient kernel: every epilogue thread calls it; the verdict is uniform
__device__ __forceinline__ bool epi_wait(Bars* b, uint64_t* bar, uint32_t parity, int* status) {
  if (!mbar_wait(bar, parity)) {
    *reinterpret_cast<volatile int*>(&b->epi_abort) = 1;
    raise_timeout(b, status);
  }
  named_bar_sync(1, kEpiThreads);
  return *reinterpret_cast<volatile int*>(&b->epi_abort) == 0;
}

// one warp waits; the verdict is a vote, on which the compiler branches uniformly
__device__ __forceinline__ bool warp_wait(Bars* b, uint64_t* bar, uint32_t parity, unsigned long long limit, int* status) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) {          // one lane polls; the others rest at the shuffle
    ok = mbar_wait(bar, parity, limit) ? 1 : 0;
    if (!ok) raise_timeout(b, status);
  }
  return __all_sync(0xffffffffu, ok);
}

__device__ __forceinline__ void store_bf16x16_swizzled(uint8_t* row_base, int row, int c0, const uint32_t* v) {
  // 16 consecutive columns c0..c0+15 (c0 % 16 == 0) of a 128-byte row inside a swizzled atom
  uint32_t w[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
    w[i] = *reinterpret_cast<uint32_t*>(&h);
  }
  const int ch = (c0 & 63) >> 3;
  uint4* p0 = reinterpret_cast<uint4*>(row_base + (((ch) ^ (row & 7)) << 4));
  uint4* p1 = reinterpret_cast<uint4*>(row_base + (((ch + 1) ^ (row & 7)) << 4));
  *p0 = make_uint4(w[0], w[1], w[2], w[3]);
  *p1 = make_uint4(w[4], w[5], w[6], w[7]);
}

// One unit of a CTA's run: up to two blocks, each with its first row, its count of valid rows and (convolution
// mode) the image and image row its tile starts at.
struct Unit { int nt, adv; int row0[2], nrows[2], b0[2], y0[2]; };
__device__ __forceinline__ Unit make_unit(const ChainParams& p, int it, int it_end) {
  Unit u;
  if (!p.cv.on) {
    const int cap = 4 * p.max_blocks;
    const int ng = (it_end - it < cap) ? it_end - it : cap;
    u.nt = ng > 4 ? 2 : 1;
    u.adv = ng;
    u.row0[0] = it * kGroupRows; u.row0[1] = u.row0[0] + 128;
    u.nrows[0] = (ng < 4 ? ng : 4) * kGroupRows; u.nrows[1] = (ng - 4) * kGroupRows;
    u.b0[0] = u.b0[1] = u.y0[0] = u.y0[1] = 0;
  } else {
    u.nt = (it_end - it < p.max_blocks) ? it_end - it : p.max_blocks;
    u.adv = u.nt;
    for (int tt = 0; tt < 2; ++tt) {
      const int t = it + tt;
      const int grp = t / p.cv.tpi, ty = t - grp * p.cv.tpi;
      u.b0[tt] = grp * p.cv.bb;
      u.y0[tt] = ty * p.cv.bh;
      u.row0[tt] = (u.b0[tt] * p.cv.H + u.y0[tt]) * p.cv.W;
      int nb = p.cv.B - u.b0[tt]; if (nb > p.cv.bb) nb = p.cv.bb;
      int nh = p.cv.H - u.y0[tt]; if (nh > p.cv.bh) nh = p.cv.bh;
      u.nrows[tt] = nb * nh * p.cv.W;
    }
  }
  return u;
}

// The rows of a partial group (fewer than 32) of a staged 32 x 64 tile go out with plain 16-byte stores.
__device__ __forceinline__ void store_partial_group(const uint8_t* buf, bf16* dst, int64_t ld, int rows, int cols_left) {
  const int lane = threadIdx.x & 31;
  for (int idx = lane; idx < rows * 8; idx += 32) {
    const int rr = idx >> 3, ch = idx & 7;
    if (ch * 8 >= cols_left) continue;
    const uint4 v = *reinterpret_cast<const uint4*>(buf + rr * 128 + ((ch ^ (rr & 7)) << 4));
    *reinterpret_cast<uint4*>(dst + (int64_t)rr * ld + ch * 8) = v;
  }
}

// ---------------------------------------------------------------------------------------------
// chain_kernel:  S = In F1^T (rows x r, accumulated in TMEM over the width of In), S rounded to bf16 into
// shared memory, Out = S F2^T in 256-column chunks, stored as bf16.  One persistent CTA per SM.
//
// Rows.  The rows are cut into groups of 32 and every CTA owns a contiguous run of groups, as equal as the
// group count allows, so the CTAs finish together whatever the row count is.  A CTA works through its run
// in units of up to two blocks of 128 rows (one block when max_blocks == 1).  Both blocks of a unit share
// every factor tile that is loaded -- each slab of F1 feeds two first-product MMAs, each tile of F2 two
// second-product MMAs -- so a row costs half the factor bytes from L2.  A block at the end of a run may
// hold fewer than four groups: only its groups are stored; the block is loaded and multiplied whole (rows are
// independent in every product, and the rows past the run are never stored).
//
// Warps (192 threads): 0 = TMA producer, 1 = MMA issuer and TMEM owner, 2..5 = epilogue.  An epilogue
// warp may read the quarter of the TMEM lanes given by its index modulo 4, i.e. the 32 rows of one group.
// Each warp converts its 32 x 64 pieces, two at a time, into two staging tiles of its own and stores them
// with TMA stores of its own: no barrier spans the epilogue warps.  (Measured: two warps per quarter with
// one staging tile each are slower, 129 against 110 us for a ViT forward; more pollers, no more overlap.)
//
// TMEM: block b of a unit keeps its S accumulator at column 256 b while the first product runs; the
// accumulators of the second product take the same columns afterwards (in a two-block unit accumulator b
// belongs to block b; in a one-block unit the two alternate between chunks).
//
// Factors.  F1 is r x K1 and F2 is P x r as operands.  Either may be given as it lies in memory (K-major:
// the reduction index is the fast one -- B and A in the forward pass) or transposed (MN-major: the
// reduction index is the slow one -- A and B in the backward pass, where F1 = A^T and F2 = B^T), which the
// shared-memory descriptors of the MMAs express directly; nothing is transposed in memory.
__global__ void __launch_bounds__(kChainThreads, 1)
chain_kernel(const __grid_constant__ CUtensorMap tmIn, const __grid_constant__ CUtensorMap tmIn4,
             const __grid_constant__ CUtensorMap tmF1, const __grid_constant__ CUtensorMap tmF2,
             const __grid_constant__ CUtensorMap tmOut, const __grid_constant__ CUtensorMap tmS, const ChainParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  // [ second-product ring | S of block 0 | S of block 1 | staging tiles of the epilogue warps | barriers ]; the
  // first product's ring lies over all of the first four regions, which it has to itself while it runs (the
  // staging tiles are written only after the unit's first product is complete, and a unit ends only when the
  // stores that read them are done)
  uint8_t* ring = smem;
  uint8_t* S0 = smem + (size_t)p.ns2 * kAtom2Bytes;
  uint8_t* stg = S0 + (size_t)p.max_blocks * p.natoms * kAtomBytes;
  Bars* bars = reinterpret_cast<Bars*>(stg + kEpiWarps * kStgTiles * kGroupBytes);

  const int warp = (int)uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  // items are dealt in runs of p.deal (1, or 4 = whole 128-row blocks when every CTA gets at least two blocks:
  // a block costs the same whether full or not, so whole blocks waste none, and the CTAs with one block fewer
  // leave their SMs to the kernel that follows)
  const int nruns = (p.groups + p.deal - 1) / p.deal;
  const int g_begin = (int)((int64_t)blockIdx.x * nruns / gridDim.x) * p.deal;
  int g_end = (int)((int64_t)(blockIdx.x + 1) * nruns / gridDim.x) * p.deal;
  if (g_end > p.groups) g_end = p.groups;
  // All CTAs walk the same factor tiles.  Started together they would all ask L2 for the same few lines at
  // the same moment; each CTA therefore starts its walk at a different slab / chunk and wraps round.
  const int rot1 = blockIdx.x % p.nk1;
  const int rot2 = p.nchunks > 0 ? (blockIdx.x * 5) % p.nchunks : 0;

  if (threadIdx.x == 0) {
    for (int i = 0; i < p.ns; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
    for (int i = 0; i < p.ns2; ++i) { mbar_init(&bars->full2[i], 1); mbar_init(&bars->empty2[i], 1); }
    mbar_init(&bars->t_full, 1);
    mbar_init(&bars->s_ready, kEpiWarps);
    mbar_init(&bars->unit_done, 1 + kEpiWarps);   // the MMA issuer's commit and every epilogue warp
    for (int i = 0; i < 2; ++i) { mbar_init(&bars->acc_full[i], 1); mbar_init(&bars->acc_empty[i], kEpiWarps); }
    bars->abort_any = 0;
    bars->epi_abort = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmIn); tma_prefetch_desc(&tmIn4); tma_prefetch_desc(&tmF1); tma_prefetch_desc(&tmF2);
    tma_prefetch_desc(&tmOut); tma_prefetch_desc(&tmS);
  }
  if (warp == 1) tmem_alloc(&bars->tmem_base, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);
  dep_wait();            // nothing above touches global memory
  dep_launch();
  clear_status_word(p.clear_status, p.status);
  const unsigned long long lim = p.wait_ns;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (one elected lane, as the MMA issuer)
    if (!p.stall_selftest) {
      int u = 0;
      int slot1 = 0, ph1 = 1, slot2 = 0, ph2 = 1;       // ring positions; parity of the next wait for an empty slot
      bool ok = true;
      for (int g = g_begin; g < g_end && ok; ++u) {
        const Unit un = make_unit(p, g, g_end);
        const int nt = un.nt;
        // the shared memory of the last unit is free once its MMAs are done and its stores have been read
        if (u > 0 && !mbar_wait_warp(&bars->unit_done, (u - 1) & 1, lim)) { raise_timeout(bars, p.status); ok = false; break; }
        int kr = rot1;
        int tap = p.cv.on ? rot1 / p.cv.cslabs : 0, cs = p.cv.on ? rot1 - tap * p.cv.cslabs : 0;
        const uint32_t tx1 = (p.cv.on ? nt * p.cv.box_rows * 128 : nt * kAtomBytes) + p.f1_bytes;
        for (int ks = 0; ks < p.nk1; ++ks) {
          if (!mbar_wait_warp(&bars->empty[slot1], ph1, lim)) { raise_timeout(bars, p.status); ok = false; break; }
          if (elect_one()) {
            uint8_t* dst = smem + (size_t)slot1 * p.slot_bytes;
            uint8_t* f1 = dst + p.max_blocks * kAtomBytes;
            uint64_t* bar = &bars->full[slot1];
            mbar_arrive_expect_tx(bar, tx1);
            if (!p.cv.on) {
              // a block at the end of the run is loaded whole as well: the rows past the run are a neighbour's
              // (or zeros past the last row) and cost less than four separate 32-row loads
              for (int tt = 0; tt < nt; ++tt) tma_load_2d(dst + tt * kAtomBytes, &tmIn, bar, kr * 64, un.row0[tt]);
              if (p.f1_mn)
                for (int a = 0; a < p.natoms; ++a) tma_load_2d(f1 + a * kF1AtomBytes, &tmF1, bar, a * 64, kr * 64);
              else
                tma_load_2d(f1, &tmF1, bar, kr * 64, 0);
            } else {
              // slab kr = (tap, 64 channels): the tile's box of the activation, shifted by the tap
              const int ty = tap / 3, dy = (ty - 1) * p.cv.sign, dx = (tap - 3 * ty - 1) * p.cv.sign;
              for (int tt = 0; tt < nt; ++tt)
                tma_load_4d(dst + tt * kAtomBytes, &tmIn4, bar, cs * 64, dx, un.y0[tt] + dy, un.b0[tt]);
              const int fcol = tap * p.cv.tap_stride + p.cv.f1_col_off;
              if (p.f1_mn)
                for (int a = 0; a < p.natoms; ++a) tma_load_2d(f1 + a * kF1AtomBytes, &tmF1, bar, fcol + a * 64, cs * 64);
              else
                tma_load_2d(f1, &tmF1, bar, fcol + cs * 64, 0);
            }
          }
          __syncwarp();
          if (++slot1 == p.ns) { slot1 = 0; ph1 ^= 1; }
          if (++cs == p.cv.cslabs) { cs = 0; ++tap; }
          if (++kr == p.nk1) { kr = 0; tap = 0; cs = 0; }
        }
        if (!ok) break;
        // the second product's slots lie over the first product's: wait until its MMAs have read them
        if (!mbar_wait_warp(&bars->t_full, u & 1, lim)) { raise_timeout(bars, p.status); ok = false; break; }
        int col0 = rot2 * kChunk;
        for (int c = 0; c < p.nchunks && ok; ++c) {
          for (int j = 0; j < p.natoms; ++j) {
            if (!mbar_wait_warp(&bars->empty2[slot2], ph2, lim)) { raise_timeout(bars, p.status); ok = false; break; }
            if (elect_one()) {
              uint8_t* d = ring + (size_t)slot2 * kAtom2Bytes;
              uint64_t* bar = &bars->full2[slot2];
              mbar_arrive_expect_tx(bar, kAtom2Bytes);
              if (p.f2_mn)
                for (int b = 0; b < 4; ++b) tma_load_2d(d + b * kF1AtomBytes, &tmF2, bar, col0 + 64 * b, j * 64);
              else
                tma_load_2d(d, &tmF2, bar, j * 64, col0);
            }
            __syncwarp();
            if (++slot2 == p.ns2) { slot2 = 0; ph2 ^= 1; }
          }
          col0 += kChunk;
          if (col0 >= p.nchunks * kChunk) col0 = 0;
        }
        g += un.adv;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // The descriptors of slot 0 are built once, a slot is an addition, a K step is an addition (32 bytes along a K-major
    // row, 2048 bytes -- 16 rows -- down an MN-major tile), and the four K steps are unrolled.  The whole warp walks the
    // loop and one elected lane issues (see elect_one).
    {
      const uint32_t tmem = uniform(tmem_base);
      const uint32_t idesc1 = instr_desc_bf16(128, p.r, 0, p.f1_mn);
      const uint32_t idesc2 = instr_desc_bf16(128, kChunk, 0, p.f2_mn);
      const uint32_t s_base = uniform(smem_u32(smem));
      const uint64_t dA1 = smem_desc_sw128(s_base, 16);                          // In tile of block 0, slot 0
      const uint64_t dF1 = p.f1_mn ? smem_desc_sw128(s_base + p.max_blocks * kAtomBytes, kF1AtomBytes)
                                   : smem_desc_sw128(s_base + p.max_blocks * kAtomBytes, 16);
      const uint64_t f1_step = p.f1_mn ? (2048u >> 4) : 2u;
      const uint64_t slot_step = (uint64_t)(p.slot_bytes >> 4);
      const uint64_t dS = smem_desc_sw128(uniform(smem_u32(S0)), 16);                     // S tile 0 of block 0
      const uint64_t dF2 = p.f2_mn ? smem_desc_sw128(s_base, kF1AtomBytes) : smem_desc_sw128(s_base, 16);
      const uint64_t f2_step = p.f2_mn ? (2048u >> 4) : 2u;
      const uint64_t blk_step = (uint64_t)(kAtomBytes >> 4);
      int u = 0;
      int slot1 = 0, ph1 = 0, slot2 = 0, ph2 = 0;                  // ring positions
      int q0 = 0, q1 = 0;                      // uses of each accumulator so far
      bool ok = true;
      for (int g = g_begin; g < g_end && ok; ++u) {
        const Unit un = make_unit(p, g, g_end);
        const int nt = un.nt;
        int kr = rot1, cs = p.cv.on ? rot1 % p.cv.cslabs : 0;
        for (int ks = 0; ks < p.nk1; ++ks) {
          if (!mbar_wait_warp(&bars->full[slot1], ph1, lim)) { raise_timeout(bars, p.status); ok = false; break; }
          tc_fence_after();
          const uint64_t da0 = dA1 + slot_step * slot1, db0 = dF1 + slot_step * slot1;
          const int ksteps = p.cv.on ? (p.cv.in_ch - cs * 64 + 15) >> 4 : (p.K1 - kr * 64 + 15) >> 4;
          const uint32_t acc0 = ks != 0;
          if (elect_one()) {
            if (nt == 2) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              if (kk < ksteps) {
                tc_mma_bf16(tmem, da0 + 2 * kk, db0 + f1_step * kk, idesc1, kk ? 1u : acc0);
                tc_mma_bf16(tmem + 256, da0 + blk_step + 2 * kk, db0 + f1_step * kk, idesc1, kk ? 1u : acc0);
              }
            }
          } else {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              if (kk < ksteps) tc_mma_bf16(tmem, da0 + 2 * kk, db0 + f1_step * kk, idesc1, kk ? 1u : acc0);
          }
            tc_commit(&bars->empty[slot1]);
          }
          __syncwarp();
          if (++slot1 == p.ns) { slot1 = 0; ph1 ^= 1; }
          if (++cs == p.cv.cslabs) cs = 0;
          if (++kr == p.nk1) { kr = 0; cs = 0; }
        }
        if (!ok) break;
        if (elect_one()) tc_commit(&bars->t_full);
        __syncwarp();
        if (p.nchunks > 0) {
          if (!mbar_wait_warp(&bars->s_ready, u & 1, lim)) { raise_timeout(bars, p.status); ok = false; break; }
          tc_fence_after();
        }
        for (int c = 0; c < p.nchunks && ok; ++c) {
          int slot = slot2, ph = ph2;          // every block of the unit walks the same tiles
          for (int tt = 0; tt < nt && ok; ++tt) {
            const int b = (nt == 2) ? tt : (c & 1);
            slot = slot2; ph = ph2;
            if (!mbar_wait_warp(&bars->acc_empty[b], ((b ? q1 : q0) & 1) ^ 1, lim)) { raise_timeout(bars, p.status); ok = false; break; }
            tc_fence_after();
            const uint32_t tacc = tmem + kChunk * b;
            const uint64_t dSb = dS + blk_step * (uint64_t)(tt * p.natoms);
            for (int j = 0; j < p.natoms; ++j) {
              if (!mbar_wait_warp(&bars->full2[slot], ph, lim)) { raise_timeout(bars, p.status); ok = false; break; }
              tc_fence_after();
              const uint64_t da = dSb + blk_step * j;
              const uint64_t db = dF2 + (uint64_t)(kAtom2Bytes >> 4) * slot;
              const int ksteps = (p.r - j * 64) >> 4;
              const uint32_t acc0 = j != 0;
              if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                  if (kk < ksteps) tc_mma_bf16(tacc, da + 2 * kk, db + f2_step * kk, idesc2, kk ? 1u : acc0);
                if (tt == nt - 1) tc_commit(&bars->empty2[slot]);     // the last block of the unit is done with this tile
              }
              __syncwarp();
              if (++slot == p.ns2) { slot = 0; ph ^= 1; }
            }
            if (ok) { if (elect_one()) tc_commit(&bars->acc_full[b]); __syncwarp(); if (b) ++q1; else ++q0; }
          }
          slot2 = slot; ph2 = ph;
        }
        if (ok && elect_one()) tc_commit(&bars->unit_done);
        __syncwarp();
        g += un.adv;
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..5)
    const int qw = warp & 3;                // TMEM lane quarter this warp may read = the 32-row group it serves
    const int row = qw * 32 + lane;         // row of the 128-row block
    const uint32_t lane_base = (uint32_t)(qw * 32) << 16;
    uint8_t* mystg = stg + (size_t)(warp - 2) * kStgTiles * kGroupBytes;
    int q0 = 0, q1 = 0;
    int u = 0;
    bool ok = true;
    for (int g = g_begin; g < g_end && ok; ++u) {
      const Unit un = make_unit(p, g, g_end);
      const int nt = un.nt;
      ok = warp_wait(bars, &bars->t_full, u & 1, lim, p.status);
      if (!ok) break;
      tc_fence_after();
      // S of every block of the unit
      for (int tt = 0; tt < nt; ++tt) {
        uint8_t* Sb = S0 + (size_t)tt * p.natoms * kAtomBytes;
        for (int j = 0; j < p.natoms; ++j) {
          const int c0 = j * 64;
          uint32_t v[4][16];
#pragma unroll
          for (int gq = 0; gq < 4; ++gq)
            if (c0 + gq * 16 < p.r) tmem_ld16_nowait(tmem_base + 256 * tt + lane_base + c0 + gq * 16, v[gq]);
          tmem_wait_ld();
#pragma unroll
          for (int gq = 0; gq < 4; ++gq)
            if (c0 + gq * 16 < p.r) store_bf16x16_swizzled(Sb + j * kAtomBytes + row * 128, row, c0 + gq * 16, v[gq]);
        }
      }
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->s_ready);
      if (p.save_s) {                        // this warp's 32 rows, if the block has them
        for (int tt = 0; tt < nt; ++tt) {
          const int grows = (int)uniform(un.nrows[tt] - qw * kGroupRows);      // rows of this warp's group in the block
          if (grows <= 0) continue;
          const int grow0 = un.row0[tt] + qw * kGroupRows;
          for (int j = 0; j < p.natoms; ++j) {
            const uint8_t* src = S0 + ((size_t)tt * p.natoms + j) * kAtomBytes + qw * kGroupBytes;
            if (grows >= kGroupRows) {
              if (elect_one()) tma_store_2d(&tmS, src, j * 64 + p.cv.s_col_off, grow0);
              __syncwarp();
            } else {
              store_partial_group(src, p.s_ptr + (int64_t)grow0 * p.s_ld + p.cv.s_col_off + j * 64, p.s_ld, grows,
                                  p.s_cols - j * 64);
            }
          }
        }
        if (elect_one()) tma_store_commit();
        __syncwarp();
      }
      int col0 = rot2 * kChunk;
      for (int c = 0; c < p.nchunks && ok; ++c) {
        for (int tt = 0; tt < nt && ok; ++tt) {
          const int b = (nt == 2) ? tt : (c & 1);
          ok = warp_wait(bars, &bars->acc_full[b], (b ? q1 : q0) & 1, lim, p.status);
          if (!ok) break;
          if (b) ++q1; else ++q0;
          tc_fence_after();
          const int grows = (int)uniform(un.nrows[tt] - qw * kGroupRows);   // rows of this warp's group in the block
          const int grow0 = un.row0[tt] + qw * kGroupRows;
          const uint32_t tacc = tmem_base + kChunk * b + lane_base;
          const int npairs = grows > 0 ? min(2, (p.P - col0 + 127) >> 7) : 0;     // 128-column pairs of pieces this warp stores
          // two 64-column pieces at a time: TMEM -> registers (bf16 pairs) while the stores of the pair before them still
          // read the staging tiles; the accumulator is handed back as soon as its last piece is in registers
#pragma unroll
          for (int pr = 0; pr < 2; ++pr) {
            uint32_t w[2][32];
            if (pr < npairs) {
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint32_t v[4][16];
#pragma unroll
                for (int gq = 0; gq < 4; ++gq) tmem_ld16_nowait(tacc + pr * 128 + h * 64 + gq * 16, v[gq]);
                tmem_wait_ld();
#pragma unroll
                for (int gq = 0; gq < 4; ++gq)
#pragma unroll
                  for (int e = 0; e < 8; ++e) {
                    __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(v[gq][2 * e]), __uint_as_float(v[gq][2 * e + 1]));
                    w[h][gq * 8 + e] = *reinterpret_cast<uint32_t*>(&h2);
                  }
              }
            }
            if (pr == (npairs == 2 ? 1 : 0)) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&bars->acc_empty[b]);
            }
            if (pr >= npairs) continue;
            if (elect_one()) tma_store_wait_read<0>();     // the stores that last read the staging tiles
            __syncwarp();
            const int pcol = col0 + pr * 128;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              uint8_t* rowp = mystg + h * kGroupBytes + lane * 128;
#pragma unroll
              for (int ch = 0; ch < 8; ++ch)                 // 16-byte chunk ch of the row goes to slot ch ^ (row & 7)
                *reinterpret_cast<uint4*>(rowp + ((ch ^ (lane & 7)) << 4)) =
                    make_uint4(w[h][4 * ch], w[h][4 * ch + 1], w[h][4 * ch + 2], w[h][4 * ch + 3]);
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (grows >= kGroupRows) {
              if (elect_one()) {
                tma_store_2d(&tmOut, mystg, pcol, grow0);
                if (pcol + 64 < p.P) tma_store_2d(&tmOut, mystg + kGroupBytes, pcol + 64, grow0);
                tma_store_commit();
              }
              __syncwarp();
            } else {        // the last rows of a convolution tile: fewer than 32
              for (int h = 0; h < 2; ++h)
                if (pcol + 64 * h < p.P)
                  store_partial_group(mystg + h * kGroupBytes, p.out_ptr + (int64_t)grow0 * p.P + pcol + 64 * h, p.P, grows, p.P - (pcol + 64 * h));
              __syncwarp();
            }
          }
        }
        col0 += kChunk;
        if (col0 >= p.nchunks * kChunk) col0 = 0;
      }
      // this warp has read all it will of the unit's accumulators; once its stores have read their
      // shared memory (S tiles and staging) the next unit may overwrite both
      if (ok) {
        if (elect_one()) { tma_store_wait_read<0>(); mbar_arrive(&bars->unit_done); }
        __syncwarp();
      }
      g += un.adv;
    }
    if (elect_one()) tma_store_wait_all();
    __syncwarp();
  }

  // ------------------------------------------------------------ common exit
  tc_fence_before();
  __syncthreads();
  if (*reinterpret_cast<volatile int*>(&bars->abort_any)) {
    // give loads that are still in flight time to land before the shared memory is released
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// The MMA warp of both gradient kernels: nk slabs of 64, two 128-row accumulators sharing every slab of `small`.
__device__ __forceinline__ void grad_mma_loop(Bars* bars, uint8_t* ring, int nk, int ns, int slot_bytes, int r, uint32_t tmem_base,
                                              int* status) {
  const uint32_t idesc = instr_desc_bf16(128, r, 1, 1), tmem = uniform(tmem_base);
  const uint64_t d0 = smem_desc_sw128(uniform(smem_u32(ring)), 8192), slot_step = (uint64_t)(slot_bytes >> 4);
  int slot = 0, ph = 0;
  for (int i = 0; i < nk; ++i) {
    if (!mbar_wait_warp(&bars->full[slot], ph)) { raise_timeout(bars, status); return; }
    tc_fence_after();
    const uint64_t d = d0 + slot_step * slot;
    if (elect_one()) {
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const uint64_t da = d + 128 * kk, db = da + (32768 >> 4);
        tc_mma_bf16(tmem, da, db, idesc, (i | kk) != 0);
        tc_mma_bf16(tmem + 256, da + (16384 >> 4), db, idesc, (i | kk) != 0);
      }
      tc_commit(&bars->empty[slot]);
    }
    __syncwarp();
    if (++slot == ns) { slot = 0; ph ^= 1; }
  }
  if (elect_one()) tc_commit(&bars->t_full);
  __syncwarp();
}

// ---------------------------------------------------------------------------------------------
// grad kernel: partial[slice][p][j] = sum_{k in slice} act[k][p] * small[k][j]
// Where a tile's sums go: element (row, col) to dst[row * ld + col], or, transposed, to dst[col * ld + row].  A tile with
// several slices leaves one set of sums per slice, `stride` elements apart.
struct GradOut {
  float* dst;
  int64_t ld, stride;
  int rows, cols;
  int transposed;
};
struct GradJob {
  int chunks;     // 256-row tiles of the output
  GradOut out;
};
struct GradParams {
  GradJob job[2];
  int r, natoms, ns, slot_bytes;
  int slices, rows_per_slice;   // rows_per_slice is a multiple of 64
  int N;
  int clear_status;
  int job0_independent;   // 1: job 0 reads nothing the kernel before this one in the stream writes (see grad_kernel)
  int* status;
};

// The end of both gradient kernels: 2 x 128 accumulator rows of r columns -> this CTA's shared memory -> global memory, two
// rows per warp instruction (from the registers a warp instruction would touch 32 rows).  Every thread of the CTA
// comes here, also after a wait that gave up (the outputs are then undefined, the status says so).
// A row takes r + 4 floats of shared memory: with r a multiple of 16 eight lanes' 16-byte accesses then fall into different
// banks.  Slices were also added inside clusters: through distributed shared memory the sums come at 10 to 15
// bytes a cycle and SM, and 8-CTA clusters leave 20 SMs empty (convolution of the ResNet layer: 57.5 us against 22 us,
// and 6 to 9 us for the separate reduction).
__device__ __forceinline__ void grad_finish(uint8_t* ring, int ring_bytes, uint32_t tmem_base, bool have, int r, int row0,
                                            int slice, const GradOut& o) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* tile = reinterpret_cast<float*>(ring);
  const int ldt = r + 4;
  const int halves = 256 * ldt * 4 <= ring_bytes ? 2 : 1;      // accumulators per pass
  float* dst = o.dst + (int64_t)slice * o.stride;
  for (int m0 = 0; m0 < 2 && row0 + 128 * m0 < o.rows; m0 += halves) {
    const int grow0 = row0 + 128 * m0;
    int rows = o.rows - grow0;
    if (rows > 128 * halves) rows = 128 * halves;
    if (warp >= 2) {
      for (int h = 0; 128 * h < rows; ++h) {
        const int q = warp & 3, row = 128 * h + q * 32 + lane;
        const uint32_t t = tmem_base + 256 * (m0 + h) + ((uint32_t)(q * 32) << 16);
        for (int c0 = 0; c0 < r; c0 += 64) {
          uint32_t v[4][16];
          if (have) {
#pragma unroll
            for (int g = 0; g < 4; ++g) if (c0 + 16 * g < r) tmem_ld16_nowait(t + c0 + 16 * g, v[g]);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int g = 0; g < 4; ++g)
#pragma unroll
              for (int i = 0; i < 16; ++i) v[g][i] = 0u;
          }
          uint4* d = reinterpret_cast<uint4*>(tile + row * ldt + c0);
#pragma unroll
          for (int g = 0; g < 4; ++g)
            if (c0 + 16 * g < r) {
#pragma unroll
              for (int i = 0; i < 4; ++i) d[4 * g + i] = make_uint4(v[g][4 * i], v[g][4 * i + 1], v[g][4 * i + 2], v[g][4 * i + 3]);
            }
        }
      }
    }
    __syncthreads();
    if (o.transposed) {              // neighbouring lanes take neighbouring rows
      for (int c = warp; c < o.cols; c += 6)
        for (int row = lane; row < rows; row += 32) dst[(int64_t)c * o.ld + grow0 + row] = tile[row * ldt + c];
    } else {
      for (int c = 4 * (lane & 15); c < o.cols; c += 64) {         // cols and ld are multiples of 4
        float* d = dst + (int64_t)grow0 * o.ld + c;
#pragma unroll 4
        for (int row = 2 * warp + (lane >> 4); row < rows; row += 12)
          *reinterpret_cast<float4*>(d + (int64_t)row * o.ld) = *reinterpret_cast<const float4*>(tile + row * ldt + c);
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(192, 1)
grad_kernel(const __grid_constant__ CUtensorMap tmAct0, const __grid_constant__ CUtensorMap tmSmall0,
            const __grid_constant__ CUtensorMap tmAct1, const __grid_constant__ CUtensorMap tmSmall1,
            const GradParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* ring = smem;
  Bars* bars = reinterpret_cast<Bars*>(ring + (size_t)p.ns * p.slot_bytes);
  const int warp = (int)uniform(threadIdx.x >> 5);

  // which job, which 128-row chunk of its output, which slice of the N rows
  int tile = blockIdx.x;
  const int slice = tile % p.slices;
  tile /= p.slices;
  int jb = 0;
  if (tile >= p.job[0].chunks) { jb = 1; tile -= p.job[0].chunks; }
  const int chunk = tile;
  const CUtensorMap* tmAct = jb ? &tmAct1 : &tmAct0;
  const CUtensorMap* tmSmall = jb ? &tmSmall1 : &tmSmall0;
  const int k_begin = slice * p.rows_per_slice;
  int k_end = k_begin + p.rows_per_slice;
  if (k_end > p.N) k_end = p.N;
  const int nk = k_end > k_begin ? (k_end - k_begin + 63) / 64 : 0;

  if (threadIdx.x == 0) {
    for (int i = 0; i < p.ns; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
    mbar_init(&bars->t_full, 1);
    bars->abort_any = 0;
    bars->epi_abort = 0;
    fence_barrier_init();
    tma_prefetch_desc(tmAct); tma_prefetch_desc(tmSmall);
  }
  if (warp == 1) tmem_alloc(&bars->tmem_base, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);
  // In a full backward the kernel before this one is the dT/dX chain, which writes dT and dX: the dB
  // job reads dT and has to wait for it, the dA job reads only dY and T.  This kernel becomes resident
  // only after every CTA of the chain kernel has passed its own dep_wait, i.e. after everything
  // earlier in the stream (T included) is complete, so the dA CTAs start at once on the SMs that the
  // chain kernel's short CTAs have already left (its last third runs on two thirds of the SMs).
  if (!(p.job0_independent && jb == 0)) dep_wait();
  dep_launch();
  clear_status_word(p.clear_status, p.status);

  if (warp == 0) {
    int slot = 0, ph = 1;
    for (int i = 0; i < nk; ++i) {
      if (!mbar_wait_warp(&bars->empty[slot], ph)) { raise_timeout(bars, p.status); break; }
      if (elect_one()) {
        uint8_t* dst = ring + (size_t)slot * p.slot_bytes;
        uint64_t* bar = &bars->full[slot];
        const int k0 = k_begin + i * 64;
        // two 128-row accumulators share every slab of `small`: four 64-wide boxes of act, then small
        mbar_arrive_expect_tx(bar, (4 + p.natoms) * 8192);
        for (int a = 0; a < 4; ++a) tma_load_2d(dst + a * 8192, tmAct, bar, chunk * 256 + a * 64, k0);
        for (int a = 0; a < p.natoms; ++a) tma_load_2d(dst + 32768 + a * 8192, tmSmall, bar, a * 64, k0);
      }
      __syncwarp();
      if (++slot == p.ns) { slot = 0; ph ^= 1; }
    }
  } else if (warp == 1) {
    grad_mma_loop(bars, ring, nk, p.ns, p.slot_bytes, p.r, tmem_base, p.status);
  } else if (nk > 0) {
    if (epi_wait(bars, &bars->t_full, 0, p.status)) tc_fence_after();
  }
  __syncwarp();
  __syncthreads();          // the MMAs have read the ring, which now takes the sums
  const bool failed = *reinterpret_cast<volatile int*>(&bars->abort_any) != 0;
  if (failed) {             // give copies that are still in flight time to land
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) { }
    __syncthreads();
  }
  tc_fence_after();
  grad_finish(ring, p.ns * p.slot_bytes, tmem_base, nk > 0 && !failed, p.r, chunk * 256, slice, p.job[jb].out);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
  // Whatever is launched behind this kernel waits for this kernel alone.  Without a dB job (whose CTAs have waited above) it could
  // be through while the chain kernel still writes dX and reads the workspace: no CTA leaves before that kernel is done.
  dep_wait();
}

// ---------------------------------------------------------------------------------------------
// conv_grad_kernel: dB of a 3 x 3 convolution without materialised im2col rows,
//   dB[j][tap * C + c] = sum over pixels of dT[pixel][j] * x[pixel shifted by the tap][c].
// Same shape as grad_kernel (two 128-row accumulators per CTA, a slice of the reduction each, fp32 partials),
// but the reduction runs over boxes of whole image rows (at most 64 pixels: bhk rows of one image, or kb whole
// images), loaded with 4-D boxes: x shifted by the tap (zeros outside an image: the padding), dT unshifted.
// A box may hold fewer than 64 pixels; the ring is zeroed once, so the rows no box ever writes stay zero in
// both operands and add nothing.
struct ConvGradParams {
  int B, H, W, C;
  int r, natoms, ns, slot_bytes;
  int spi, kb, bhk, box_rows;    // slabs per image (kb == 1) or 1; images per slab; image rows per slab; pixels per box
  int cpt;                       // 256-channel windows per tap
  int slices, slabs_per_slice, nslabs;
  GradOut out;                   // rows: 9 C
  int* status;
};

__global__ void __launch_bounds__(192, 1)
conv_grad_kernel(const __grid_constant__ CUtensorMap tmX4, const __grid_constant__ CUtensorMap tmT4,
                 const ConvGradParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* ring = smem;
  Bars* bars = reinterpret_cast<Bars*>(ring + (size_t)p.ns * p.slot_bytes);
  const int warp = (int)uniform(threadIdx.x >> 5);
  int tile = blockIdx.x;
  const int slice = tile % p.slices;
  const int chunk = tile / p.slices;
  const int tap = chunk / p.cpt, cwin = (chunk - tap * p.cpt) * 256;
  const int s_begin = slice * p.slabs_per_slice;
  int s_end = s_begin + p.slabs_per_slice;
  if (s_end > p.nslabs) s_end = p.nslabs;
  const int nk = s_end > s_begin ? s_end - s_begin : 0;

  if (threadIdx.x == 0) {
    for (int i = 0; i < p.ns; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
    mbar_init(&bars->t_full, 1);
    bars->abort_any = 0;
    bars->epi_abort = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmX4); tma_prefetch_desc(&tmT4);
  }
  {
    // a box has box_rows of a tile's 64 rows: the rest stay zero
    const int per = (64 - p.box_rows) * 8, n16 = p.ns * (p.slot_bytes / 8192) * per;
    for (int i = threadIdx.x; i < n16; i += blockDim.x) {
      const int t = i / per;
      reinterpret_cast<uint4*>(ring + (size_t)t * 8192 + p.box_rows * 128)[i - t * per] = make_uint4(0u, 0u, 0u, 0u);
    }
    fence_proxy_async_smem();
  }
  if (warp == 1) tmem_alloc(&bars->tmem_base, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);
  dep_wait();
  dep_launch();

  if (warp == 0) {
    const int dy = tap / 3 - 1, dx = tap % 3 - 1;
    int slot = 0, ph = 1;
    int grp = s_begin / p.spi, ty = s_begin - grp * p.spi;
    for (int i = 0; i < nk; ++i) {
      if (!mbar_wait_warp(&bars->empty[slot], ph)) { raise_timeout(bars, p.status); break; }
      if (elect_one()) {
        uint8_t* dst = ring + (size_t)slot * p.slot_bytes;
        uint64_t* bar = &bars->full[slot];
        const int b0 = grp * p.kb, y0 = ty * p.bhk;
        mbar_arrive_expect_tx(bar, (4 + p.natoms) * p.box_rows * 128);
        for (int a = 0; a < 4; ++a) tma_load_4d(dst + a * 8192, &tmX4, bar, cwin + a * 64, dx, y0 + dy, b0);
        for (int a = 0; a < p.natoms; ++a) tma_load_4d(dst + 32768 + a * 8192, &tmT4, bar, a * 64, 0, y0, b0);
      }
      __syncwarp();
      if (++slot == p.ns) { slot = 0; ph ^= 1; }
      if (++ty == p.spi) { ty = 0; ++grp; }
    }
  } else if (warp == 1) {
    grad_mma_loop(bars, ring, nk, p.ns, p.slot_bytes, p.r, tmem_base, p.status);
  } else if (nk > 0) {
    if (epi_wait(bars, &bars->t_full, 0, p.status)) tc_fence_after();
  }
  __syncwarp();
  __syncthreads();
  const bool failed = *reinterpret_cast<volatile int*>(&bars->abort_any) != 0;
  if (failed) {
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) { }
    __syncthreads();
  }
  tc_fence_after();
  // the tile's rows are channels cwin .. of one tap: rows end with the tap
  GradOut o = p.out;
  o.dst += p.out.transposed ? (int64_t)tap * p.C : (int64_t)tap * p.C * p.out.ld;
  o.rows = p.C;
  grad_finish(ring, p.ns * p.slot_bytes, tmem_base, nk > 0 && !failed, p.r, cwin, slice, o);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// Sums the slices' partials in a fixed order (identical bits every run).
//   blocks [0, nA):  dA[p][j]  = sum_s pA[s][p][j]
//   blocks [nA, ..): dB[j][q]  = sum_s pB[s][q][j]            (tiles transposed through shared memory)
// The partials lie in L2 and the kernel waits for them: a thread that walks the slices alone makes slices / 4 trips of
// about 800 cycles (104 slices of 256 x 128: 38 us).  So G threads share an element (4 columns), each sums every G-th
// slice, and the first adds the G sums (6 us).
constexpr int kReduceT = 256;
__host__ __device__ inline int reduce_groups(int slices) { return slices >= 24 ? 8 : slices >= 12 ? 4 : slices >= 6 ? 2 : 1; }
// rows x float4 columns of a transposed tile: 256 / G of them, rows as long as a 128-byte line as far as they go
__host__ __device__ inline int reduce_rows(int G) { return G == 8 ? 16 : 32; }
__device__ __forceinline__ float4 sum_slices(const float* src, int64_t stride, int first, int slices, int step) {
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  int k = first;
  for (; k + 7 * step < slices; k += 8 * step) {
    float4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __ldcg(reinterpret_cast<const float4*>(src + (k + i * step) * stride));
#pragma unroll
    for (int i = 0; i < 8; ++i) { acc.x += v[i].x; acc.y += v[i].y; acc.z += v[i].z; acc.w += v[i].w; }
  }
#pragma unroll 4
  for (; k < slices; k += step) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(src + k * stride));
    acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
  }
  return acc;
}
__global__ void __launch_bounds__(kReduceT)
reduce_partials_kernel(const float* __restrict__ pA, float* __restrict__ dA, int PA, int nA,
                       const float* __restrict__ pB, float* __restrict__ dB, int PB, int slices, int r, int rp) {
  // r: columns of the results, a multiple of 4; rp: row length of the partials (r rounded up to 16)
  __shared__ float4 part[kReduceT];
  __shared__ float turned[32][33];
  const int G = reduce_groups(slices), items = kReduceT / G;
  const int g = threadIdx.x / items, e = threadIdx.x - g * items;
  const bool first = (int)blockIdx.x < nA;
  const int r4 = r >> 2, rows = reduce_rows(G), c4 = items / rows;
  const int tiles_j = (r4 + c4 - 1) / c4, t = (int)blockIdx.x - nA;
  int64_t row;
  int col;
  int64_t i4 = 0;
  if (first) {
    i4 = (int64_t)blockIdx.x * items + e;
    row = i4 / r4;
    col = 4 * (int)(i4 - row * r4);
  } else {
    row = (int64_t)(t / tiles_j) * rows + e / c4;
    col = 4 * ((t % tiles_j) * c4 + e % c4);
  }
  const bool live = col < r && row < (first ? PA : PB);
  dep_wait();
  dep_launch();
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (live) acc = sum_slices((first ? pA : pB) + row * rp + col, (int64_t)(first ? PA : PB) * rp, g, slices, G);
  part[threadIdx.x] = acc;
  __syncthreads();
  if (g == 0) {
    for (int i = 1; i < G; ++i) {
      const float4 v = part[i * items + e];
      acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    if (first) {
      if (live) reinterpret_cast<float4*>(dA)[i4] = acc;
    } else {
      float* d = &turned[e / c4][4 * (e % c4)];
      d[0] = acc.x; d[1] = acc.y; d[2] = acc.z; d[3] = acc.w;
    }
  }
  if (first) return;
  __syncthreads();
  const int64_t q0 = (int64_t)(t / tiles_j) * rows;
  const int j0 = (t % tiles_j) * c4 * 4;
  for (int i = threadIdx.x; i < rows * c4 * 4; i += kReduceT) {
    const int j = i / rows, q = i - j * rows;
    if (j0 + j < r && q0 + q < PB) dB[(int64_t)(j0 + j) * PB + q0 + q] = turned[q][j];
  }
}

// Self-test of the bounded wait every pipeline stage of the kernels above relies on: one thread waits on
// an mbarrier that nobody ever arrives at.  The wait gives up after limit_ns and the kernel reports
// AB_ERR_TIMEOUT through the status word, exactly as the chain kernels do; nothing spins for ever and the
// context stays usable.
__global__ void bounded_wait_selftest_kernel(int* status, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) *status = mbar_wait(&bar, 0, limit_ns) ? (int)AB_OK : (int)AB_ERR_TIMEOUT;
}

// ---------------------------------------------------------------------------------------------
// host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

bool device_is_sm100() {
  static std::mutex mu;
  static int cache[64];
  static bool init = false;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  std::lock_guard<std::mutex> lock(mu);
  if (!init) { for (int i = 0; i < 64; ++i) cache[i] = -1; init = true; }
  if (cache[dev] < 0) {
    int major = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return false;
    cache[dev] = (major == 10) ? 1 : 0;
  }
  return cache[dev] == 1;
}

// Ranks that are multiples of 8 but not of 16 run as the next multiple of 16: the tensor maps keep the
// true extents, so the extra rows / columns of every factor tile arrive as zeros.
int pad16(int r) { return (r + 15) & ~15; }

// Shared-memory plan of chain_kernel for a (padded) rank and a number of blocks per unit.
struct ChainPlan { int natoms, max_blocks, ns, slot_bytes, ns2, f1_bytes; size_t smem; bool ok; };
ChainPlan chain_plan(int rp, int max_blocks, bool f1_mn) {
  ChainPlan pl;
  pl.natoms = (rp + 63) / 64;
  pl.max_blocks = max_blocks;
  pl.f1_bytes = f1_mn ? pl.natoms * kF1AtomBytes : rp * 128;
  pl.slot_bytes = max_blocks * kAtomBytes + pl.f1_bytes;
  const int s_bytes = max_blocks * pl.natoms * kAtomBytes;
  const int fixed = s_bytes + kEpiWarps * kStgTiles * kGroupBytes + (int)sizeof(Bars) + 1024;
  pl.ns2 = (kSmemLimit - fixed) / kAtom2Bytes;
  if (pl.ns2 > kMaxStages2) pl.ns2 = kMaxStages2;
  if (pl.ns2 < 0) pl.ns2 = 0;
  // the first product's ring lies over the second product's ring, S and the staging tiles (all idle while it runs)
  pl.ns = (pl.ns2 * kAtom2Bytes + s_bytes + kEpiWarps * kStgTiles * kGroupBytes) / pl.slot_bytes;
  if (pl.ns > kMaxStages) pl.ns = kMaxStages;
  pl.smem = (size_t)fixed + (size_t)pl.ns2 * kAtom2Bytes;
  // a two-block unit keeps every tile of a chunk of F2 until its second block has used it
  pl.ok = pl.ns >= 2 && pl.ns2 >= 2 && (max_blocks == 1 || pl.ns2 >= pl.natoms);
  return pl;
}

// How the slabs of a gradient reduction are dealt: slices per 256-row tile, slabs per slice.  The split with the least time by
// what was measured: 0.55 us a slab, 5 us to fill and empty a CTA and to write its sums; several slices
// take a reduction launch of 3 us that reads them all at 3 TB/s.  Few slabs thus go to fewer CTAs than there are SMs.
struct GradSplit { int slices, per; };
GradSplit grad_split(int64_t slabs, int tiles, int rp) {
  const int sms = sm_count() > 0 ? sm_count() : 1;
  GradSplit best = {1, (int)slabs};
  double best_t = 1e30;
  for (int want = 1; want <= sms && want <= slabs; ++want) {
    const int64_t per = (slabs + want - 1) / want;
    const int slices = (int)((slabs + per - 1) / per);
    if (slices != want) continue;
    const int waves = (tiles * slices + sms - 1) / sms;
    double t = waves * (0.55 * (double)per + 5.0);
    if (slices > 1) t += 3.0 + (double)slices * tiles * 256.0 * rp * 4.0 / 3e6;
    if (t < best_t) { best_t = t; best = {slices, (int)per}; }
  }
  return best;
}
int tiles256(int v) { return (v + 255) / 256; }

struct GradPlan { int natoms, ns, slot_bytes; GradSplit sp; size_t smem; };
GradPlan grad_plan(int64_t N, int m, int n, int r) {
  GradPlan pl;
  pl.natoms = (r + 63) / 64;
  pl.slot_bytes = 32768 + pl.natoms * 8192;
  const int fixed = (int)sizeof(Bars) + 1024;
  pl.ns = (kSmemLimit - fixed) / pl.slot_bytes;
  if (pl.ns > kMaxStages) pl.ns = kMaxStages;
  pl.smem = (size_t)fixed + (size_t)pl.ns * pl.slot_bytes;      // the ring also takes 128 x (r + 4) sums: at most 133 KB of it
  pl.sp = grad_split((N + 63) / 64, tiles256(m) + tiles256(n), pad16(r));
  return pl;
}
// floats of the slices' sums of an output of `rows` rows, where there is more than one slice
size_t grad_partial(const GradSplit& s, int64_t rows, int rp) { return s.slices > 1 ? (size_t)s.slices * rows * rp : 0; }
GradOut grad_out(const GradSplit& sp, float* partial, float* dst, int rows, int r, bool transposed) {
  GradOut o;
  const int rp = pad16(r);
  o.rows = rows;
  if (sp.slices > 1) { o.dst = partial; o.ld = rp; o.stride = (int64_t)rows * rp; o.cols = rp; o.transposed = 0; }
  else { o.dst = dst; o.ld = transposed ? rows : r; o.stride = 0; o.cols = r; o.transposed = transposed ? 1 : 0; }
  return o;
}
struct ReduceGrid { int a, b; };          // blocks of reduce_partials_kernel
ReduceGrid reduce_grid(const GradSplit& sp, int64_t rowsA, int64_t rowsB, int r) {
  const int G = reduce_groups(sp.slices), items = kReduceT / G, rows = reduce_rows(G), c4 = items / rows, r4 = r / 4;
  return {(int)((rowsA * r4 + items - 1) / items), (int)((rowsB + rows - 1) / rows) * ((r4 + c4 - 1) / c4)};
}

struct BwdWs { int* status; bf16 *T, *dT; float *pA, *pB; size_t bytes; };
BwdWs bwd_ws(void* ws, int64_t N, int m, int n, int r) {
  const GradSplit sp = grad_plan(N, m, n, r).sp;
  Arena ar(ws, 0);
  BwdWs w;
  w.status = ar.take_n<int>(64);
  w.T = ar.take_n<bf16>((size_t)N * r);
  w.dT = ar.take_n<bf16>((size_t)N * r);
  w.pA = ar.take_n<float>(grad_partial(sp, m, pad16(r)));
  w.pB = ar.take_n<float>(grad_partial(sp, n, pad16(r)));
  w.bytes = align_up(ar.used, 256);
  return w;
}

// Everything one launch of chain_kernel needs.  Regular mode: In is N x K1.  Convolution mode (cv != null): In is
// the NHWC activation cv describes, N = B H W pixels, K1 is not used; F1 is the factor that holds the nine taps
// side by side (r x 9 C as an operand, or, MN-major, stored (reduction index) x (9 C)).
struct ChainLaunch {
  const void* In; int64_t N; int K1;
  const void* F1; int ldF1; int f1_rows, f1_cols;   // extents of F1 as it lies in memory
  const void* F2; int ldF2; int P;
  bool f_mn;
  void* Out; void* Sg; int s_ld, s_cols;   // S is stored to Sg (row stride s_ld) at column cv->s_col_off
  int r;                                   // width of S
  const ConvGeom* cv;
  int* status; bool clear_status;
  bool stall_selftest; unsigned long long wait_ns;
};

int launch_chain_ex(const ChainLaunch& L, cudaStream_t st) {
  const int rp = pad16(L.r);
  const bool second = L.Out != nullptr && L.P > 0;
  const int sms = sm_count();
  if (sms <= 0) return AB_ERR_CUDA;
  const bool conv = L.cv != nullptr;
  int64_t items, per_unit;
  if (conv) {
    const int groups_of_images = (L.cv->B + L.cv->bb - 1) / L.cv->bb;
    items = (int64_t)groups_of_images * L.cv->tpi;
    per_unit = 1;
  } else {
    items = (L.N + kGroupRows - 1) / kGroupRows;
    per_unit = 4;
  }
  const int grid = (int)(items < sms ? items : sms);
  const int64_t per_cta = (items + grid - 1) / grid;
  ChainPlan pl = chain_plan(rp, per_cta > per_unit ? 2 : 1, L.f_mn);
  if (!pl.ok && pl.max_blocks == 2) pl = chain_plan(rp, 1, L.f_mn);
  if (!pl.ok) return AB_ERR_UNSUPPORTED;
  CUtensorMap tmIn, tmIn4, tmF1, tmF2, tmOut, tmS;
  if (conv) {
    AB_TRY(make_tensor_map_nhwc(&tmIn4, L.In, L.cv->B, L.cv->H, L.cv->W, L.cv->in_ch, L.cv->W, L.cv->bh, L.cv->bb));
    AB_TRY(make_tensor_map_2d(&tmF1, L.F1, false, L.f1_rows, L.f1_cols, L.ldF1, 64, L.f_mn ? 64 : rp));
    tmIn = tmF1;
  } else {
    AB_TRY(make_tensor_map_2d(&tmIn, L.In, false, (uint64_t)L.N, L.K1, L.K1, 64, 128));
    tmIn4 = tmIn;
    if (L.f_mn) AB_TRY(make_tensor_map_2d(&tmF1, L.F1, false, L.K1, L.r, L.ldF1, 64, 64));
    else AB_TRY(make_tensor_map_2d(&tmF1, L.F1, false, L.r, L.K1, L.ldF1, 64, rp));
  }
  // unused maps still have to be valid objects: alias them to another operand
  if (second) {
    if (L.f_mn) AB_TRY(make_tensor_map_2d(&tmF2, L.F2, false, L.r, L.P, L.ldF2, 64, 64));
    else AB_TRY(make_tensor_map_2d(&tmF2, L.F2, false, L.P, L.r, L.ldF2, 64, kChunk));
    AB_TRY(make_tensor_map_2d(&tmOut, L.Out, false, (uint64_t)L.N, L.P, L.P, 64, kGroupRows));
  } else {
    tmF2 = tmF1;
    tmOut = tmF1;
  }
  if (L.Sg) AB_TRY(make_tensor_map_2d(&tmS, L.Sg, false, (uint64_t)L.N, conv ? L.cv->s_col_off + L.s_cols : L.s_cols, L.s_ld, 64, kGroupRows));
  else tmS = tmF1;
  ChainParams q;
  std::memset(&q, 0, sizeof(q));
  q.K1 = L.K1; q.P = second ? L.P : 0; q.r = rp;
  q.nk1 = conv ? 9 * L.cv->cslabs : (L.K1 + 63) / 64;
  q.nchunks = second ? (L.P + kChunk - 1) / kChunk : 0;
  q.natoms = pl.natoms; q.max_blocks = pl.max_blocks; q.ns = pl.ns; q.slot_bytes = pl.slot_bytes; q.ns2 = pl.ns2;
  q.f1_bytes = pl.f1_bytes; q.f1_mn = L.f_mn ? 1 : 0; q.f2_mn = L.f_mn ? 1 : 0; q.save_s = L.Sg ? 1 : 0;
  q.groups = (int)items;
  q.deal = (!conv && items >= (int64_t)8 * grid) ? 4 : 1;
  q.clear_status = L.clear_status ? 1 : 0; q.stall_selftest = L.stall_selftest ? 1 : 0;
  q.wait_ns = L.wait_ns; q.status = L.status;
  if (conv) q.cv = *L.cv;
  q.out_ptr = static_cast<bf16*>(L.Out); q.s_ptr = static_cast<bf16*>(L.Sg); q.s_ld = L.s_ld; q.s_cols = L.s_cols;
  AB_CUDA_OK(allow_smem(chain_kernel));
  AB_TRY(launch_after(chain_kernel, (unsigned)grid, kChainThreads, pl.smem, 1, st, tmIn, tmIn4, tmF1, tmF2, tmOut, tmS, q));
  return AB_OK;
}

// Whether the chain runs as two products by tiles.  The fused kernel takes every row through whole factors on one SM: with
// few rows that is a long walk on few SMs, and S in memory costs next to nothing.  Measured (us, fused / by tiles,
// 768 -> 192 -> 3072): 64 rows 21.8 / 8.5, 6173 26.2 / 17.4, 8800 26.5 / 23.1, 10500 28.7 / 32.5; 776 -> 120 -> 1000: 64 rows
// 14.2 / 8.3, 8800 20.0 / 14.5, 25088 30.7 / 34.4: hence up to one 128-row block for every two SMs.  Factors of a few tiles
// are no long walk (256 -> 32 -> 256: 5.9 / 6.9); between (512 -> 64 -> 512) a lone forward is bound by the host's second launch, 8.6 / 11.4,
// and the backward of 6173 rows, where the launches overlap, gains, 19.6 / 18.1.
// The first product alone (us, chain kernel / tiles): K 3072 12608 rows 24.1 / 17.0, 25088 33.2 / 44.7; K 256, rank 128 25088 rows
// 6.3 / 4.7, 50432 9.2 / 6.1; with the gradient behind it K 64 to 512, rank 32, 200704 rows 82 to 111 / 76 to 102, but rank 24, K 512
// 118 / 138 and rank 8, K 256 102 / 120: many rows of a rank below 32 stay with the chain kernel.
bool by_tiles(int64_t N, int K1, int r, int P) {
  const int64_t blocks = (N + 127) / 128;
  const int sms = sm_count();
  if (P == 0) return 3 * blocks <= 2 * sms || (K1 <= 512 && r >= 32);
  const int walk = (K1 + 63) / 64 + (P + kChunk - 1) / kChunk * ((r + 63) / 64);
  return 2 * blocks <= sms && walk > 6;
}

// S = In F1^T (saved to Sg if not null), Out = S F2^T (skipped if Out is null).
// f_mn = false: F1 is given as r x K1 (row stride ldF1) and F2 as P x r (row stride ldF2);
// f_mn = true : F1 is given transposed, K1 x r, and F2 transposed, r x P (the factors A and B as they lie in
//               memory when the chain runs backwards).
// P is given even where Out is not wanted: which kernels run, and with that the bits of S, depends on the shape and on whether
// there is room for S, not on what is wanted.  scratch: N x r for S where Sg is null; without it the fused kernel runs.
int launch_chain(const void* In, int64_t N, int K1, const void* F1, int ldF1, const void* F2, int ldF2, int P,
                 bool f_mn, void* Out, void* Sg, void* scratch, int r, int* status, bool clear_status, cudaStream_t st,
                 bool stall_selftest = false, unsigned long long wait_ns = kWaitLimitNs) {
  void* S = Sg ? Sg : scratch;
  if (!stall_selftest && S && by_tiles(N, K1, r, P)) {
    const TileProduct first = {In, N, K1, F1, ldF1, f_mn, S, r}, second = {S, N, r, F2, ldF2, f_mn, Out, P};
    AB_TRY(tile_product(first, clear_status, status, st));
    if (Out && P > 0) AB_TRY(tile_product(second, false, status, st));
    return AB_OK;
  }
  ChainLaunch L;
  L.In = In; L.N = N; L.K1 = K1; L.F1 = F1; L.ldF1 = ldF1; L.f1_rows = 0; L.f1_cols = 0; L.F2 = F2; L.ldF2 = ldF2; L.P = P;
  L.f_mn = f_mn; L.Out = Out; L.Sg = Sg; L.s_ld = r; L.s_cols = r; L.r = r; L.cv = nullptr; L.status = status;
  L.clear_status = clear_status; L.stall_selftest = stall_selftest; L.wait_ns = wait_ns;
  return launch_chain_ex(L, st);
}

}  // namespace

int bounded_wait_selftest(int* dev_status, unsigned limit_us, cudaStream_t st) {
  bounded_wait_selftest_kernel<<<1, 32, 0, st>>>(dev_status, (unsigned long long)limit_us * 1000ull);
  AB_LAUNCH_OK();
  return AB_OK;
}

// The chain kernel itself with a producer that loads nothing: the MMA issuer's and the epilogue warps'
// waits run out after limit_us, every role unwinds to the common exit, TMEM is released and the status
// word (first int of ws) holds AB_ERR_TIMEOUT.  The operands are carved from ws; their contents do not
// matter, since nothing is ever loaded.
size_t chain_stall_selftest_ws() { return 256 + 4 * 65536; }
int chain_stall_selftest(void* ws, size_t ws_bytes, unsigned limit_us, cudaStream_t st) {
  if (!ws || !aligned(ws, 256) || ws_bytes < chain_stall_selftest_ws()) return AB_ERR_WORKSPACE;
  if (!device_is_sm100() || !encode_fn()) return AB_ERR_UNSUPPORTED;
  char* base = static_cast<char*>(ws);
  int* status = reinterpret_cast<int*>(base);
  void* In = base + 256;                 // 256 x 64 bf16
  void* F1 = base + 256 + 65536;         // 16 x 64
  void* F2 = base + 256 + 2 * 65536;     // 64 x 16
  void* Out = base + 256 + 3 * 65536;    // 256 x 64
  return launch_chain(In, 256, 64, F1, 64, F2, 16, 64, false, Out, nullptr, nullptr, 16, status, true, st, true,
                      (unsigned long long)limit_us * 1000ull);
}

int make_tensor_map_2d(CUtensorMap* m, const void* ptr, bool f32, uint64_t rows, uint64_t cols, uint64_t ld,
                       uint32_t box_cols, uint32_t box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return AB_ERR_CUDA;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {ld * (f32 ? 4 : 2)};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult rc = fn(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr),
                   dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return rc == CUDA_SUCCESS ? AB_OK : AB_ERR_CUDA;
}

int make_tensor_map_nhwc(CUtensorMap* m, const void* ptr, uint64_t B, uint64_t H, uint64_t W, uint64_t C,
                         uint32_t bw, uint32_t bh, uint32_t bb) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return AB_ERR_CUDA;
  cuuint64_t dims[4] = {C, W, H, B};
  cuuint64_t strides[3] = {C * 2, W * C * 2, H * W * C * 2};
  cuuint32_t box[4] = {64, bw, bh, bb};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult rc = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptr), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return rc == CUDA_SUCCESS ? AB_OK : AB_ERR_CUDA;
}

bool tc_device_ok() { return device_is_sm100() && encode_fn() != nullptr; }

bool chain_tc_supported(int64_t N, int m, int n, int r, int ldA, int ldB, int dt,
                        const void* x, const void* A, const void* B, const void* y) {
  if (dt != AB_BF16) return false;
  if (r % 8 != 0 || r < 8 || r > 256) return false;
  if (m % 8 != 0 || n % 8 != 0 || ldA % 8 != 0 || ldB % 8 != 0) return false;
  if (N > (int64_t)1 << 30) return false;
  if (!aligned(x, 16) || !aligned(A, 16) || !aligned(B, 16) || !aligned(y, 16)) return false;
  if (!device_is_sm100() || !encode_fn()) return false;
  return chain_plan(pad16(r), 1, false).ok && chain_plan(pad16(r), 1, true).ok;
}

size_t chain_tc_forward_ws(int64_t N, int, int, int r) { return 256 + align_up((size_t)N * r * sizeof(bf16), 256); }
size_t chain_tc_backward_ws(int64_t N, int m, int n, int r) {
  if (r % 8 != 0 || r < 8 || r > 256) return 0;
  return bwd_ws(nullptr, N, m, n, r).bytes;
}

int chain_tc_forward(const void* x, const void* A, const void* B, void* y, void* T_save,
                     int64_t N, int m, int n, int r, int ldA, int ldB,
                     void* ws, size_t ws_bytes, cudaStream_t st) {
  if (!ws || ws_bytes < 256) return AB_ERR_WORKSPACE;
  if (T_save && !aligned(T_save, 16)) return AB_ERR_INVALID_ARG;
  int* status = static_cast<int*>(ws);
  // S has room behind the status word in a workspace of the size that was asked for
  void* scratch = ws_bytes >= chain_tc_forward_ws(N, m, n, r) ? static_cast<char*>(ws) + 256 : nullptr;
  return launch_chain(x, N, n, B, ldB, A, ldA, m, false, y, T_save, scratch, r, status, true, st);
}

int chain_tc_backward(const void* x, const void* dY, const void* A, const void* B,
                      const void* T_saved, void* dX, float* dA, float* dB,
                      int64_t N, int m, int n, int r, int ldA, int ldB,
                      void* ws, size_t ws_bytes, cudaStream_t st) {
  if (!ws) return AB_ERR_WORKSPACE;
  BwdWs w = bwd_ws(ws, N, m, n, r);
  if (w.bytes > ws_bytes) return AB_ERR_WORKSPACE;
  if ((dX && !aligned(dX, 16)) || (T_saved && !aligned(T_saved, 16)) || (dA && !aligned(dA, 16)) ||
      (dB && !aligned(dB, 16)))
    return AB_ERR_INVALID_ARG;
  bool first = true;     // the first kernel of the call zeroes the status word
  bool after_chain = false;   // the dT/dX chain kernel is the launch right before the gradient kernel
  const bf16* T = static_cast<const bf16*>(T_saved);
  if (dA && !T) {   // recompute T = x B^T (first product only)
    AB_TRY(launch_chain(x, N, n, B, ldB, A, ldA, m, false, nullptr, w.T, nullptr, r, w.status, first, st));
    first = false;
    T = w.T;
  }
  if (dX || dB) {
    // dT = dY A (kept for dB), dX = dT B: the chain with F1 = A^T and F2 = B^T, i.e. A and B as they lie
    AB_TRY(launch_chain(dY, N, m, A, ldA, B, ldB, n, true, dX, dB ? w.dT : nullptr, w.dT, r, w.status, first, st));
    first = false;
    after_chain = true;
  }
  if (dA || dB) {
    const GradPlan gp = grad_plan(N, m, n, r);     // the same split whichever is asked for: the same bits
    const int rp = pad16(r), slices = gp.sp.slices;
    GradParams p;
    std::memset(&p, 0, sizeof(p));
    CUtensorMap tmAct[2], tmSmall[2];
    int nj = 0;
    if (dA) {
      AB_TRY(make_tensor_map_2d(&tmAct[nj], dY, false, (uint64_t)N, m, m, 64, 64));
      AB_TRY(make_tensor_map_2d(&tmSmall[nj], T, false, (uint64_t)N, r, r, 64, 64));
      p.job[nj].chunks = tiles256(m); p.job[nj].out = grad_out(gp.sp, w.pA, dA, m, r, false);
      ++nj;
    }
    if (dB) {
      AB_TRY(make_tensor_map_2d(&tmAct[nj], x, false, (uint64_t)N, n, n, 64, 64));
      AB_TRY(make_tensor_map_2d(&tmSmall[nj], w.dT, false, (uint64_t)N, r, r, 64, 64));
      p.job[nj].chunks = tiles256(n); p.job[nj].out = grad_out(gp.sp, w.pB, dB, n, r, true);
      ++nj;
    }
    if (nj == 1) { tmAct[1] = tmAct[0]; tmSmall[1] = tmSmall[0]; p.job[1] = p.job[0]; p.job[1].chunks = 0; }
    p.r = rp; p.natoms = gp.natoms; p.ns = gp.ns; p.slot_bytes = gp.slot_bytes;
    p.slices = slices; p.rows_per_slice = gp.sp.per * 64; p.N = (int)N; p.clear_status = first ? 1 : 0; p.status = w.status;
    p.job0_independent = (after_chain && dA) ? 1 : 0;   // job 0 is the dA job whenever dA is asked for
    AB_CUDA_OK(allow_smem(grad_kernel));
    const unsigned grid = (unsigned)((p.job[0].chunks + p.job[1].chunks) * slices);
    AB_TRY(launch_after(grad_kernel, grid, 192, gp.smem, 1, st, tmAct[0], tmSmall[0], tmAct[1], tmSmall[1], p));
    if (slices > 1) {
      const ReduceGrid rg = reduce_grid(gp.sp, dA ? m : 0, dB ? n : 0, r);
      const int nA = rg.a, nB = rg.b;
      AB_TRY(launch_after(reduce_partials_kernel, (unsigned)(nA + nB), kReduceT, 0, 1, st, static_cast<const float*>(w.pA), dA,
                          m, nA, static_cast<const float*>(w.pB), dB, n, slices, r, rp));
    }
    first = false;
  }
  if (first) AB_CUDA_OK(cudaMemsetAsync(w.status, 0, sizeof(int), st));   // nothing was asked for
  return AB_OK;
}

// ---------------------------------------------------------------------------------------------
// 3 x 3 convolution (stride 1, padding 1, NHWC) with the factorised weight, im2col rows never materialised.
namespace {

ConvGeom conv_geom(int B, int H, int W, int in_ch, int sign, int tap_stride, int f1_col_off, int s_col_off) {
  ConvGeom g;
  g.on = 1; g.B = B; g.H = H; g.W = W; g.in_ch = in_ch; g.cslabs = (in_ch + 63) / 64;
  if (H * W <= 128) { g.bb = 128 / (H * W); g.bh = H; g.tpi = 1; }
  else {
    const int bhmax = 128 / W;
    g.bb = 1; g.tpi = (H + bhmax - 1) / bhmax; g.bh = (H + g.tpi - 1) / g.tpi;
  }
  g.box_rows = W * g.bh * g.bb;
  g.sign = sign; g.tap_stride = tap_stride; g.f1_col_off = f1_col_off; g.s_col_off = s_col_off;
  return g;
}

struct ConvGradPlan { int natoms, ns, slot_bytes, spi, kb, bhk, box_rows, cpt, nslabs; GradSplit sp; size_t smem; bool ok; };
ConvGradPlan conv_grad_plan(int B, int H, int W, int C, int rp) {
  ConvGradPlan pl;
  pl.natoms = (rp + 63) / 64;
  pl.slot_bytes = 32768 + pl.natoms * 8192;
  const int fixed = (int)sizeof(Bars) + 1024;
  pl.ns = (kSmemLimit - fixed) / pl.slot_bytes;
  if (pl.ns > kMaxStages) pl.ns = kMaxStages;
  pl.smem = (size_t)fixed + (size_t)pl.ns * pl.slot_bytes;
  pl.ok = W <= 64 && pl.ns >= 2;
  if (H * W <= 64) { pl.kb = 64 / (H * W); pl.bhk = H; pl.spi = 1; pl.nslabs = (B + pl.kb - 1) / pl.kb; }
  else { pl.kb = 1; pl.bhk = W <= 64 ? 64 / W : 1; pl.spi = (H + pl.bhk - 1) / pl.bhk; pl.nslabs = B * pl.spi; }
  pl.box_rows = W * pl.bhk * pl.kb;
  pl.cpt = (C + 255) / 256;
  pl.sp = grad_split(pl.nslabs, 9 * pl.cpt, rp);
  return pl;
}

struct ConvWs { int* status; bf16 *T, *dT; float *pA, *pB; size_t bytes; };
ConvWs conv_ws(void* ws, int B, int H, int W, int C, int m, int r) {
  const int64_t N = (int64_t)B * H * W;
  const int rp = pad16(r);
  const GradSplit ga = grad_plan(N, m, 0, r).sp, gb = conv_grad_plan(B, H, W, C, rp).sp;
  Arena ar(ws, 0);
  ConvWs w;
  w.status = ar.take_n<int>(64);
  w.T = ar.take_n<bf16>((size_t)N * r);
  w.dT = ar.take_n<bf16>((size_t)N * r);
  w.pA = ar.take_n<float>(grad_partial(ga, m, rp));
  w.pB = ar.take_n<float>(grad_partial(gb, 9 * (int64_t)C, rp));
  w.bytes = align_up(ar.used, 256);
  return w;
}

}  // namespace

bool conv_tc_supported(int B, int H, int W, int C, int m, int r, int ldA, int ldB, int dt,
                       const void* x, const void* A, const void* Bf) {
  if (dt != AB_BF16) return false;
  if (r % 8 != 0 || r < 8 || r > 256 || C % 8 != 0 || m % 8 != 0 || ldA % 8 != 0 || ldB % 8 != 0) return false;
  if (B < 1 || H < 1 || W < 1 || W > 64 || H > 256 || (int64_t)B * H * W > ((int64_t)1 << 30)) return false;
  if (!aligned(x, 16) || !aligned(A, 16) || !aligned(Bf, 16)) return false;
  if (!device_is_sm100() || !encode_fn()) return false;
  const int cw = C < 256 ? C : 256;
  return chain_plan(pad16(r), 1, false).ok && chain_plan(pad16(r), 1, true).ok && chain_plan(pad16(cw), 1, true).ok &&
         conv_grad_plan(B, H, W, C, pad16(r)).ok;
}

size_t conv_tc_ws(int B, int H, int W, int C, int m, int r) { return conv_ws(nullptr, B, H, W, C, m, r).bytes; }

// y[pixel][:] = (sum over taps of x[pixel + tap][:] B_tap^T) A^T, B_tap = columns tap C .. tap C + C of B
int conv_tc_forward(const void* x, const void* A, const void* Bf, void* y, void* T_save, int B, int H, int W, int C,
                    int m, int r, int ldA, int ldB, void* ws, size_t ws_bytes, cudaStream_t st) {
  if (!ws || ws_bytes < 256) return AB_ERR_WORKSPACE;
  if ((T_save && !aligned(T_save, 16)) || !aligned(y, 16)) return AB_ERR_INVALID_ARG;
  const ConvGeom g = conv_geom(B, H, W, C, +1, C, 0, 0);
  ChainLaunch L;
  L.In = x; L.N = (int64_t)B * H * W; L.K1 = 0; L.F1 = Bf; L.ldF1 = ldB; L.f1_rows = r; L.f1_cols = 9 * C;
  L.F2 = A; L.ldF2 = ldA; L.P = m; L.f_mn = false; L.Out = y; L.Sg = T_save; L.s_ld = r; L.s_cols = r; L.r = r; L.cv = &g;
  L.status = static_cast<int*>(ws); L.clear_status = true; L.stall_selftest = false; L.wait_ns = kWaitLimitNs;
  return launch_chain_ex(L, st);
}

// dT = dY A; dX[pixel][c] = sum over taps of dT[pixel - tap][:] B[:, tap C + c] (the col2im sum, folded into the
// reduction); dA = dY^T T; dB[j][tap C + c] = sum over pixels of dT[pixel][j] x[pixel + tap][c].
int conv_tc_backward(const void* x, const void* dY, const void* A, const void* Bf, const void* T_saved, void* dX,
                     float* dA, float* dB, int B, int H, int W, int C, int m, int r, int ldA, int ldB,
                     void* ws, size_t ws_bytes, cudaStream_t st) {
  if (!ws) return AB_ERR_WORKSPACE;
  ConvWs w = conv_ws(ws, B, H, W, C, m, r);
  if (w.bytes > ws_bytes) return AB_ERR_WORKSPACE;
  if ((dX && !aligned(dX, 16)) || (T_saved && !aligned(T_saved, 16)) || (dA && !aligned(dA, 16)) || (dB && !aligned(dB, 16)))
    return AB_ERR_INVALID_ARG;
  const int64_t N = (int64_t)B * H * W;
  const int rp = pad16(r);
  bool first = true;
  const bf16* T = static_cast<const bf16*>(T_saved);
  if (dA && !T) {      // T rebuilt from x (first product of the forward pass only)
    const ConvGeom g = conv_geom(B, H, W, C, +1, C, 0, 0);
    ChainLaunch L;
    L.In = x; L.N = N; L.K1 = 0; L.F1 = Bf; L.ldF1 = ldB; L.f1_rows = r; L.f1_cols = 9 * C; L.F2 = nullptr; L.ldF2 = 0; L.P = 0;
    L.f_mn = false; L.Out = nullptr; L.Sg = w.T; L.s_ld = r; L.s_cols = r; L.r = r; L.cv = &g; L.status = w.status;
    L.clear_status = first; L.stall_selftest = false; L.wait_ns = kWaitLimitNs;
    AB_TRY(launch_chain_ex(L, st));
    first = false;
    T = w.T;
  }
  if (dX || dB) {
    AB_TRY(launch_chain(dY, N, m, A, ldA, nullptr, 0, 0, true, nullptr, w.dT, nullptr, r, w.status, first, st));   // dT = dY A
    first = false;
  }
  if (dX) {
    for (int c0 = 0; c0 < C; c0 += 256) {      // 256 channels of dX per launch: the width of one accumulator
      const int cw = C - c0 < 256 ? C - c0 : 256;
      const ConvGeom g = conv_geom(B, H, W, r, -1, C, c0, c0);
      ChainLaunch L;
      L.In = w.dT; L.N = N; L.K1 = 0; L.F1 = Bf; L.ldF1 = ldB; L.f1_rows = r; L.f1_cols = 9 * C; L.F2 = nullptr; L.ldF2 = 0;
      L.P = 0; L.f_mn = true; L.Out = nullptr; L.Sg = dX; L.s_ld = C; L.s_cols = cw; L.r = cw; L.cv = &g; L.status = w.status;
      L.clear_status = false; L.stall_selftest = false; L.wait_ns = kWaitLimitNs;
      AB_TRY(launch_chain_ex(L, st));
    }
  }
  if (dA) {
    GradPlan gp = grad_plan(N, m, 0, r);
    GradParams p;
    std::memset(&p, 0, sizeof(p));
    CUtensorMap tmAct, tmSmall;
    AB_TRY(make_tensor_map_2d(&tmAct, dY, false, (uint64_t)N, m, m, 64, 64));
    AB_TRY(make_tensor_map_2d(&tmSmall, T, false, (uint64_t)N, r, r, 64, 64));
    p.job[0].chunks = tiles256(m); p.job[0].out = grad_out(gp.sp, w.pA, dA, m, r, false);
    p.job[1] = p.job[0]; p.job[1].chunks = 0;
    const int slices = gp.sp.slices;
    p.r = rp; p.natoms = gp.natoms; p.ns = gp.ns; p.slot_bytes = gp.slot_bytes;
    p.slices = slices; p.rows_per_slice = gp.sp.per * 64; p.N = (int)N; p.clear_status = first ? 1 : 0;
    p.status = w.status; p.job0_independent = 0;
    AB_CUDA_OK(allow_smem(grad_kernel));
    AB_TRY(launch_after(grad_kernel, (unsigned)(p.job[0].chunks * slices), 192, gp.smem, 1, st, tmAct, tmSmall, tmAct, tmSmall, p));
    first = false;
    if (slices > 1) {
      const int nA = reduce_grid(gp.sp, m, 0, r).a;
      AB_TRY(launch_after(reduce_partials_kernel, (unsigned)(nA), kReduceT, 0, 1, st, static_cast<const float*>(w.pA), dA, m, nA,
                          static_cast<const float*>(w.pA), static_cast<float*>(nullptr), 0, slices, r, rp));
    }
  }
  if (dB) {
    ConvGradPlan gp = conv_grad_plan(B, H, W, C, rp);
    ConvGradParams p;
    std::memset(&p, 0, sizeof(p));
    CUtensorMap tmX4, tmT4;
    AB_TRY(make_tensor_map_nhwc(&tmX4, x, B, H, W, C, W, gp.bhk, gp.kb));
    AB_TRY(make_tensor_map_nhwc(&tmT4, w.dT, B, H, W, r, W, gp.bhk, gp.kb));
    p.B = B; p.H = H; p.W = W; p.C = C; p.r = rp; p.natoms = gp.natoms; p.ns = gp.ns; p.slot_bytes = gp.slot_bytes;
    const int slices = gp.sp.slices;
    p.spi = gp.spi; p.kb = gp.kb; p.bhk = gp.bhk; p.box_rows = gp.box_rows; p.cpt = gp.cpt; p.slices = slices;
    p.slabs_per_slice = gp.sp.per; p.nslabs = gp.nslabs; p.out = grad_out(gp.sp, w.pB, dB, 9 * C, r, true); p.status = w.status;
    AB_CUDA_OK(allow_smem(conv_grad_kernel));
    AB_TRY(launch_after(conv_grad_kernel, (unsigned)(9 * gp.cpt * slices), 192, gp.smem, 1, st, tmX4, tmT4, p));
    if (slices > 1) {
      const int nB = reduce_grid(gp.sp, 0, 9 * (int64_t)C, r).b;
      AB_TRY(launch_after(reduce_partials_kernel, (unsigned)(nB), kReduceT, 0, 1, st, static_cast<const float*>(w.pB),
                          static_cast<float*>(nullptr), 0, 0, static_cast<const float*>(w.pB), dB, 9 * C, slices, r, rp));
    }
  }
  if (first) AB_CUDA_OK(cudaMemsetAsync(w.status, 0, sizeof(int), st));
  return AB_OK;
}

}  // namespace ab
