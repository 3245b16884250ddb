// D = X F^T for bf16 storage (fp32 accumulation), one tile of D per CTA: the two products of the factorised chain as two
// launches, for layers of few rows and for single products.
//
// A CTA is bound by the arrival of its operands (a 128-byte row of a TMA box every 2 cycles, 64 bytes a cycle and SM) and
// by the trips of a tile: barriers, TMEM, first load, accumulator to memory, about 2.4 us in all.  So tiles are small where there
// are few (64 rows, 64 columns) and several CTAs share an SM, each with a short ring, so that one stores while another loads.
// Measured against the fused chain kernel: 197 rows 768 -> 192 -> 3072 8.5 us (22), 6173 rows 776 -> 120 -> 1000 12.7 us (20.7);
// the product dT = dY A of a convolution, 25088 rows, K 256, rank 128: 5.3 us (10.7).
#include <cstring>

#include "ab_common.cuh"
#include "ab_tc_ptx.cuh"

namespace ab {
namespace {

using namespace tc;

constexpr int kTileThreads = 192;             // 0 = TMA producer, 1 = MMA issuer and TMEM owner, 2..5 = epilogue
constexpr int kXBytes = 16384;                // 128 rows x 64 bf16
constexpr int kMaxTileStages = 6;

struct TileParams {
  int K, nk;                // reduction length, slabs of 64
  int rows, cols;           // rows loaded and stored per tile (64 or 128), columns (a multiple of 16)
  int ncol;                 // tiles across D
  int N, P;                 // rows and width of D
  int ns, slot_bytes;
  int f_mn, f_bytes;        // F held with the reduction index as the slow one; bytes of one slab of it
  int tmem_cols;
  int clear_status;
  int* status;
};

struct TileBars {
  uint64_t full[kMaxTileStages], empty[kMaxTileStages];
  uint64_t done;
  uint32_t tmem_base;
  int abort_any;
};

__device__ __forceinline__ void tile_timeout(TileBars* b, int* status) {
  *reinterpret_cast<volatile int*>(&b->abort_any) = 1;
  atomicExch(status, (int)AB_ERR_TIMEOUT);
}

__global__ void __launch_bounds__(kTileThreads)
tile_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmF,
            const __grid_constant__ CUtensorMap tmD, const TileParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  TileBars* bars = reinterpret_cast<TileBars*>(ring + (size_t)p.ns * p.slot_bytes);
  const int warp = (int)uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int rt = (int)blockIdx.x / p.ncol, row0 = rt * p.rows, col0 = ((int)blockIdx.x - rt * p.ncol) * p.cols;

  if (threadIdx.x == 0) {
    for (int i = 0; i < p.ns; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
    mbar_init(&bars->done, 1);
    bars->abort_any = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmF); tma_prefetch_desc(&tmD);
  }
  __syncthreads();
  dep_wait();            // nothing above touches global memory
  if (p.clear_status && blockIdx.x == 0 && threadIdx.x == 0) atomicExch(p.status, 0);
  // TMEM is taken here, while the first loads are on their way, and not above: a CTA that waited for the kernel before with
  // columns in hand would keep that kernel's own CTAs on this SM from theirs (two such launches 20.7 us, apart 13.9 us).  The
  // next kernel is let in only after that: it may take its columns at once and then wait for this one.
  uint32_t tmem_base = 0;
  if (warp != 0) {
    if (warp == 1) tmem_alloc(&bars->tmem_base, p.tmem_cols);
    tc_fence_before();
    named_bar_sync(1, kTileThreads - 32);
    tc_fence_after();
    dep_launch();
    tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);
  }

  if (warp == 0) {
    int slot = 0, ph = 1;
    const uint32_t tx = p.rows * 128 + p.f_bytes;
    for (int i = 0; i < p.nk; ++i) {
      if (!mbar_wait_warp(&bars->empty[slot], ph)) { tile_timeout(bars, p.status); break; }
      if (elect_one()) {
        uint8_t* dst = ring + (size_t)slot * p.slot_bytes;
        uint64_t* bar = &bars->full[slot];
        mbar_arrive_expect_tx(bar, tx);
        tma_load_2d(dst, &tmX, bar, i * 64, row0);
        if (p.f_mn)
          for (int a = 0; a * 8192 < p.f_bytes; ++a) tma_load_2d(dst + kXBytes + a * 8192, &tmF, bar, col0 + a * 64, i * 64);
        else
          tma_load_2d(dst + kXBytes, &tmF, bar, i * 64, col0);
      }
      __syncwarp();
      if (++slot == p.ns) { slot = 0; ph ^= 1; }
    }
  } else if (warp == 1) {
    // rows past the ones that are loaded hold whatever the shared memory held: rows of D are independent, and these are
    // never stored
    const uint32_t idesc = instr_desc_bf16(128, p.cols, 0, p.f_mn), tmem = uniform(tmem_base);
    const uint32_t base = uniform(smem_u32(ring));
    const uint64_t dX = smem_desc_sw128(base, 16), dF = smem_desc_sw128(base + kXBytes, p.f_mn ? 8192 : 16);
    const uint64_t f_step = p.f_mn ? (2048u >> 4) : 2u, slot_step = (uint64_t)(p.slot_bytes >> 4);
    int slot = 0, ph = 0;
    for (int i = 0; i < p.nk; ++i) {
      if (!mbar_wait_warp(&bars->full[slot], ph)) { tile_timeout(bars, p.status); break; }
      tc_fence_after();
      const uint64_t da = dX + slot_step * slot, db = dF + slot_step * slot;
      const int ksteps = (p.K - i * 64 + 15) >> 4;
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          if (kk < ksteps) tc_mma_bf16(tmem, da + 2 * kk, db + f_step * kk, idesc, (i | kk) != 0);
        tc_commit(&bars->empty[slot]);
      }
      __syncwarp();
      if (++slot == p.ns) { slot = 0; ph ^= 1; }
    }
    if (elect_one()) tc_commit(&bars->done);
    __syncwarp();
  } else {
    const int q = warp & 3;                  // quarter of the TMEM lanes this warp may read = its 32 rows of the tile
    const bool ok = mbar_wait_warp(&bars->done, 0);
    if (!ok) tile_timeout(bars, p.status);
    else if (q * 32 < p.rows && row0 + q * 32 < p.N) {
      tc_fence_after();
      // the MMAs have read the ring, which now takes the tile: 32 rows x 64 columns at a time
      uint8_t* stg = ring + (size_t)q * (((p.cols + 63) >> 6) * 4096);
      const uint32_t t = tmem_base + ((uint32_t)(q * 32) << 16);
      for (int c0 = 0; c0 < p.cols && col0 + c0 < p.P; c0 += 64) {
        uint32_t v[4][16];
#pragma unroll
        for (int g = 0; g < 4; ++g) if (c0 + 16 * g < p.cols) tmem_ld16_nowait(t + c0 + 16 * g, v[g]);
        tmem_wait_ld();
        uint8_t* buf = stg + (c0 >> 6) * 4096;
        uint8_t* rowp = buf + lane * 128;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          uint32_t w[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(v[g][2 * e]), __uint_as_float(v[g][2 * e + 1]));
            w[e] = *reinterpret_cast<uint32_t*>(&h2);
          }
          *reinterpret_cast<uint4*>(rowp + (((2 * g) ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
          *reinterpret_cast<uint4*>(rowp + (((2 * g + 1) ^ (lane & 7)) << 4)) = make_uint4(w[4], w[5], w[6], w[7]);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (elect_one()) {
          tma_store_2d(&tmD, buf, col0 + c0, row0 + q * 32);
          tma_store_commit();
        }
        __syncwarp();
      }
      if (elect_one()) tma_store_wait_all();
      __syncwarp();
    }
  }

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
    tmem_dealloc(tmem_base, p.tmem_cols);
  }
}

// What one launch costs in SM cycles, by what was measured on tiles of 32 to 128 rows (32 never pays) and 64 to 256 columns:
// a 128-byte row arrives every 2 cycles, an MMA step of 16 takes 51 / 65 / 98 / 130 cycles at 64 / 128 / 192 / 256 columns, a slab
// 200 besides; a load takes 1100 cycles (2200 from many megabytes) and the stages of the CTAs on an SM hide it; a CTA starts, fills
// and stores in about 4500, which those on the SM beside it hide.
struct TilePlan { int rows, cols, ns; double cycles; };
int tile_slot_bytes(int cols, bool f_mn) {
  const int f = f_mn ? (cols + 63) / 64 * 8192 : cols * 128;
  return kXBytes + (f + 1023) / 1024 * 1024;
}
TilePlan tile_plan(int64_t N, int K, int P, bool f_mn) {
  const int sms = sm_count() > 0 ? sm_count() : 1;
  const int nk = (K + 63) / 64;
  const double trip = (double)N * K * 2 > 32e6 ? 2200.0 : 1100.0;
  TilePlan best = {128, 64, 2, 1e30};
  for (int rows = 64; rows <= 128; rows *= 2) {
    for (int cols = 64; cols <= 256; cols += 64) {
      // a store takes whole 64-column pieces and stops at D's edge, not at the tile's: narrower pieces only where one tile is
      // all of D across
      const int c = P <= cols ? (P + 15) / 16 * 16 : cols;
      const int fw = f_mn ? (c + 63) / 64 * 64 : c;
      const int64_t tiles = (N + rows - 1) / rows * ((P + c - 1) / c);
      const double t = (double)((tiles + sms - 1) / sms);
      for (int ns = 2; ns <= 4; ++ns) {
        int k = (225 * 1024) / (ns * tile_slot_bytes(c, f_mn) + 2048);
        if (k * (c <= 64 ? 64 : c <= 128 ? 128 : 256) > 512) k = 512 / (c <= 64 ? 64 : c <= 128 ? 128 : 256);
        if (k < 1) continue;
        const double live = t < k ? t : k;
        double slab = 2.0 * (rows + fw);
        const double mma = 200.0 + 4.0 * (c <= 64 ? 51 : c <= 128 ? 65 : c <= 192 ? 98 : 130);
        if (mma > slab) slab = mma;
        if (nk > ns && trip / (ns * live) > slab) slab = trip / (ns * live);
        const double cycles = t * nk * slab + (double)(int64_t)((t + k - 1) / k) * 4500.0;
        if (cycles < best.cycles) best = {rows, c, ns, cycles};
      }
      if (P <= cols) break;
    }
  }
  return best;
}

int launch_tiles(const TileProduct& t, const TilePlan& pl, bool clear_status, int* status, cudaStream_t st) {
  const int rows = pl.rows, cols = pl.cols, ns = pl.ns;
  TileParams p;
  std::memset(&p, 0, sizeof(p));
  p.K = t.K; p.nk = (t.K + 63) / 64; p.rows = rows; p.cols = cols; p.N = (int)t.N; p.P = t.P; p.ncol = (t.P + cols - 1) / cols;
  p.f_mn = t.f_mn ? 1 : 0; p.f_bytes = t.f_mn ? (cols + 63) / 64 * 8192 : cols * 128;
  p.slot_bytes = tile_slot_bytes(cols, t.f_mn); p.ns = ns;
  p.tmem_cols = cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : 256;
  p.clear_status = clear_status ? 1 : 0; p.status = status;
  CUtensorMap tmX, tmF, tmD;
  AB_TRY(make_tensor_map_2d(&tmX, t.X, false, (uint64_t)t.N, t.K, t.K, 64, rows));
  if (t.f_mn) AB_TRY(make_tensor_map_2d(&tmF, t.F, false, t.K, t.P, t.ldF, 64, 64));
  else AB_TRY(make_tensor_map_2d(&tmF, t.F, false, t.P, t.K, t.ldF, 64, cols));
  AB_TRY(make_tensor_map_2d(&tmD, t.D, false, (uint64_t)t.N, t.P, t.P, 64, 32));
  const size_t smem = 1024 + (size_t)ns * p.slot_bytes + sizeof(TileBars);
  AB_CUDA_OK(allow_smem(tile_kernel));
  return launch_after(tile_kernel, (unsigned)((t.N + rows - 1) / rows * p.ncol), (unsigned)kTileThreads, smem, 1, st, tmX, tmF, tmD, p);
}

}  // namespace

int tile_product(const TileProduct& t, bool clear_status, int* status, cudaStream_t st) {
  return launch_tiles(t, tile_plan(t.N, t.K, t.P, t.f_mn), clear_status, status, st);
}

}  // namespace ab
