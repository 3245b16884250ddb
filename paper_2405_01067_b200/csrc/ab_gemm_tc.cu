// General tensor-core GEMM on sm_100a: the products of the path that are plain contractions.
//
//   C[M x N] = A[M x K] * B[N x K]^T        (bf16 operands, fp32 accumulation in TMEM)
//
// the dense layer of the full-rank phases: y = x W^T, dX = dY W, dW = dY^T x.
//
// Either operand may lie K-major (M x K resp. N x K, row-major) or MN-major (stored K x M resp. K x N,
// row-major); the shared-memory descriptors of the MMAs express the difference, nothing is transposed.
// Up to two problems run in one launch; their records (tensor maps included) are kernel parameters and a CTA finds its problem
// and its 128 x 256 tile from its block index.  (In a table in device memory they cost a copy in front of every launch, which
// also kept the launch from overlapping the kernel before it.)  K may be cut into slices, each writing its own partial
// result (summed afterwards in ascending order: fixed bits).  A slab of 64 is bound by the arrival of its 48 KB at 64 bytes a
// cycle and SM, 768 cycles; its MMAs take 520.
//
// Warps (192 threads): 0 = TMA producer, 1 = MMA issuer and TMEM owner, 2..5 = epilogue (TMEM -> registers
// -> a staging tile of the warp's own -> TMA store of 32 rows).  Every wait is bounded (see ab_tc_ptx.cuh).
#include <cstring>

#include "ab_common.cuh"
#include "ab_tc_ptx.cuh"

namespace ab {
namespace {

using namespace tc;

constexpr int kBM = 128, kBN = 256, kBK = 64;
constexpr int kAStage = kBM * 128;        // 16 KB: 128 x 64 bf16
constexpr int kBStage = kBN * 128;        // 32 KB
constexpr int kStage = kAStage + kBStage;
constexpr int kStages = 4;
constexpr int kStgBytes = 4096;           // 32 rows x 128 bytes
constexpr int kTcThreads = 192;
constexpr int kMaxProbs = 2;

struct TcBars {
  uint64_t full[kStages], empty[kStages];
  uint64_t acc_full[2], acc_empty[2];
  uint32_t tmem_base;
  int abort_any;
};

struct alignas(64) TcProblemDev {
  CUtensorMap a, b;
  CUtensorMap c;            // output, boxes of 32 rows x 128 bytes
  int M, N, K;
  int a_mn, b_mn;           // 1: stored K x M / K x N
  int c_f32;                // 1: fp32 output (32 columns per box), 0: bf16 (64 columns per box)
  int tiles_n;              // column tiles
  int ksplit;               // slices of K
  int kslice;               // K per slice, a multiple of 64
  int c_rows;               // rows of one partial result in the output map (M when ksplit == 1)
  int first_tile;           // index of this problem's first tile among all tiles of the batch
};
struct TcBatch {
  TcProblemDev prob[kMaxProbs];
  int nprobs, ntiles;
  int* status;
};

__device__ __forceinline__ void tc_raise(TcBars* b, int* status) {
  *reinterpret_cast<volatile int*>(&b->abort_any) = 1;
  atomicExch(status, (int)AB_ERR_TIMEOUT);
}

// What one tile of the batch is: its problem, its corner, its slice of K.
struct TileInfo {
  const TcProblemDev* P;
  int m0, n0, slice, k_begin, k_end, nslab, ncols, nmma;
};
__device__ __forceinline__ TileInfo decode_tile(const TcBatch& p, int tile) {
  TileInfo ti;
  ti.P = p.prob + (p.nprobs > 1 && tile >= p.prob[1].first_tile ? 1 : 0);
  int t = tile - ti.P->first_tile;
  ti.slice = t % ti.P->ksplit;
  t /= ti.P->ksplit;
  ti.n0 = (t % ti.P->tiles_n) * kBN;
  ti.m0 = (t / ti.P->tiles_n) * kBM;
  ti.k_begin = ti.slice * ti.P->kslice;
  ti.k_end = ti.k_begin + ti.P->kslice;
  if (ti.k_end > ti.P->K) ti.k_end = ti.P->K;
  ti.nslab = ti.k_end > ti.k_begin ? (ti.k_end - ti.k_begin + kBK - 1) / kBK : 0;
  ti.ncols = ti.P->N - ti.n0;
  if (ti.ncols > kBN) ti.ncols = kBN;
  ti.nmma = (ti.ncols + 15) & ~15;
  return ti;
}

// Persistent CTAs: CTA b takes the tiles b, b + gridDim.x, ... of the batch.  Two 256-column accumulators in
// TMEM alternate between a CTA's tiles, so the epilogue of one tile (TMEM -> staging -> TMA stores) runs
// beside the loads and MMAs of the next.
__global__ void __launch_bounds__(kTcThreads, 1)
gemm_tc_kernel(const __grid_constant__ TcBatch p) {
  int* const status = p.status;
  const int ntiles = p.ntiles;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* ring = smem;
  uint8_t* stg = smem + kStages * kStage;
  TcBars* bars = reinterpret_cast<TcBars*>(stg + 4 * 2 * kStgBytes);
  const int warp = (int)uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&bars->acc_full[i], 1); mbar_init(&bars->acc_empty[i], 4); }
    bars->abort_any = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&bars->tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);
  dep_wait();            // nothing above touches global memory
  dep_launch();
  // a wait gives up only after about a second: this cannot wipe a raised error
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(status, 0);

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    {
      int slot = 0, ph = 1;
      bool ok = true;
      for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const TileInfo ti = decode_tile(p, tile);
        const TcProblemDev* P = ti.P;
        const int a_mn = (int)uniform(P->a_mn), b_mn = (int)uniform(P->b_mn), nslab = (int)uniform(ti.nslab);
        const CUtensorMap *ma = &P->a, *mb = &P->b;
        for (int ks = 0; ks < nslab; ++ks) {
          if (!mbar_wait_warp(&bars->empty[slot], ph)) { tc_raise(bars, status); ok = false; break; }
          if (elect_one()) {
            uint8_t* da = ring + (size_t)slot * kStage;
            uint8_t* db = da + kAStage;
            uint64_t* bar = &bars->full[slot];
            const int k0 = ti.k_begin + ks * kBK;
            mbar_arrive_expect_tx(bar, kStage);
            if (a_mn) { for (int h = 0; h < 2; ++h) tma_load_2d(da + h * 8192, ma, bar, ti.m0 + 64 * h, k0); }
            else tma_load_2d(da, ma, bar, k0, ti.m0);
            if (b_mn) { for (int h = 0; h < 4; ++h) tma_load_2d(db + h * 8192, mb, bar, ti.n0 + 64 * h, k0); }
            else tma_load_2d(db, mb, bar, k0, ti.n0);
          }
          __syncwarp();
          if (++slot == kStages) { slot = 0; ph ^= 1; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    {
      int slot = 0, ph = 0, it = 0;
      bool ok = true;
      const uint32_t sbase = uniform(smem_u32(ring)), tmem = uniform(tmem_base);
      for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++it) {
        const TileInfo ti = decode_tile(p, tile);
        const int nslab = (int)uniform(ti.nslab), klen = (int)uniform(ti.k_end - ti.k_begin);
        const int a_mn = (int)uniform(ti.P->a_mn), b_mn = (int)uniform(ti.P->b_mn);
        const uint32_t idesc = instr_desc_bf16(kBM, (int)uniform(ti.nmma), a_mn, b_mn);
        const uint64_t da0 = smem_desc_sw128(sbase, a_mn ? 8192 : 16), db0 = smem_desc_sw128(sbase + kAStage, b_mn ? 8192 : 16);
        const uint64_t as = a_mn ? 128u : 2u, bs = b_mn ? 128u : 2u;      // 16 of the reduction, in 16-byte units
        const int b = it & 1;
        if (!mbar_wait_warp(&bars->acc_empty[b], ((it >> 1) & 1) ^ 1)) { tc_raise(bars, status); ok = false; break; }
        tc_fence_after();
        const uint32_t tacc = tmem + 256 * b;
        for (int ks = 0; ks < nslab; ++ks) {
          if (!mbar_wait_warp(&bars->full[slot], ph)) { tc_raise(bars, status); ok = false; break; }
          tc_fence_after();
          const uint64_t da = da0 + (uint64_t)(slot * (kStage >> 4)), db = db0 + (uint64_t)(slot * (kStage >> 4));
          const int ksteps = (klen - ks * kBK + 15) >> 4;
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              if (kk < ksteps) tc_mma_bf16(tacc, da + as * kk, db + bs * kk, idesc, (ks | kk) ? 1u : 0u);
            tc_commit(&bars->empty[slot]);
          }
          __syncwarp();
          if (++slot == kStages) { slot = 0; ph ^= 1; }
        }
        if (ok && elect_one()) tc_commit(&bars->acc_full[b]);
        __syncwarp();
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..5)
    const int qw = warp & 3;
    const uint32_t lane_base = (uint32_t)(qw * 32) << 16;
    uint8_t* mystg = stg + (size_t)(warp - 2) * 2 * kStgBytes;
    int nst = 0, it = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++it) {
      const TileInfo ti = decode_tile(p, tile);
      const TcProblemDev* P = ti.P;
      const int b = it & 1;
      const bool have_acc = ti.nslab > 0;      // an empty reduction leaves zeros
      {
        int w = 1;
        if (lane == 0) { w = mbar_wait(&bars->acc_full[b], (it >> 1) & 1) ? 1 : 0; if (!w) tc_raise(bars, status); }
        ok = __shfl_sync(0xffffffffu, w, 0) != 0;
      }
      if (!ok) break;
      tc_fence_after();
      const bool rows_in = ti.m0 + qw * 32 < P->M;
      const int c_f32 = P->c_f32;
      const int pcols = c_f32 ? 32 : 64;                 // columns of one 128-byte piece
      const int crow = ti.slice * P->c_rows + ti.m0 + qw * 32;
      const uint32_t tacc = tmem_base + 256 * b + lane_base;
      for (int c0 = 0; c0 < ti.ncols; c0 += pcols) {
        uint32_t v[4][16];
        if (have_acc && rows_in) {
#pragma unroll
          for (int gq = 0; gq < 4; ++gq)
            if (gq * 16 < pcols) tmem_ld16_nowait(tacc + c0 + gq * 16, v[gq]);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int gq = 0; gq < 4; ++gq)
#pragma unroll
            for (int e = 0; e < 16; ++e) v[gq][e] = 0u;
        }
        if (c0 + pcols >= ti.ncols) {                    // the last piece is in registers: hand the accumulator back
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->acc_empty[b]);
        }
        if (!rows_in) continue;
        uint8_t* buf = mystg + (nst & 1) * kStgBytes;
        ++nst;
        if (lane == 0) tma_store_wait_read<1>();
        __syncwarp();
        uint8_t* rowp = buf + lane * 128;
        if (c_f32) {
#pragma unroll
          for (int ch = 0; ch < 8; ++ch)
            *reinterpret_cast<uint4*>(rowp + ((ch ^ (lane & 7)) << 4)) =
                make_uint4(v[ch >> 2][(ch & 3) * 4], v[ch >> 2][(ch & 3) * 4 + 1], v[ch >> 2][(ch & 3) * 4 + 2],
                           v[ch >> 2][(ch & 3) * 4 + 3]);
        } else {
#pragma unroll
          for (int ch = 0; ch < 8; ++ch) {
            uint32_t w4[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int idx = ch * 8 + 2 * e;          // column within the 64-column piece
              __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(v[idx >> 4][idx & 15]),
                                                        __uint_as_float(v[(idx + 1) >> 4][(idx + 1) & 15]));
              w4[e] = *reinterpret_cast<uint32_t*>(&h2);
            }
            *reinterpret_cast<uint4*>(rowp + ((ch ^ (lane & 7)) << 4)) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          tma_store_2d(&P->c, buf, ti.n0 + c0, crow);
          tma_store_commit();
        }
      }
    }
    if (lane == 0) tma_store_wait_all();
  }

  tc_fence_before();
  __syncthreads();
  if (*reinterpret_cast<volatile int*>(&bars->abort_any)) {
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// out[i] = sum over slices of part[s][i], ascending s (fixed order); four values a thread (count and stride are multiples of 4), up
// to eight slices' loads in flight
__global__ void __launch_bounds__(256)
sum_slices_kernel(const float4* __restrict__ part, float4* __restrict__ out, int64_t count4, int64_t stride4, int slices) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  dep_wait();
  dep_launch();
  if (i >= count4) return;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int s0 = 0; s0 < slices; s0 += 8) {
    float4 v[8];
#pragma unroll
    for (int s = 0; s < 8; ++s)
      if (s0 + s < slices) v[s] = __ldcg(part + i + (s0 + s) * stride4);
#pragma unroll
    for (int s = 0; s < 8; ++s)
      if (s0 + s < slices) { acc.x += v[s].x; acc.y += v[s].y; acc.z += v[s].z; acc.w += v[s].w; }
  }
  out[i] = acc;
}

}  // namespace

int sum_slices(const float* part, float* out, int64_t count, int64_t slice_stride, int slices, cudaStream_t st) {
  if (count <= 0) return AB_OK;
  if (count % 4 != 0 || slice_stride % 4 != 0 || !aligned(part, 16) || !aligned(out, 16)) return AB_ERR_INVALID_ARG;
  return launch_after(sum_slices_kernel, (unsigned)((count / 4 + 255) / 256), 256u, 0, 1, st, reinterpret_cast<const float4*>(part),
                      reinterpret_cast<float4*>(out), count / 4, slice_stride / 4, slices);
}

bool gemm_tc_available() { return tc_device_ok(); }

bool gemm_tc_problem_ok(const TcProblem& q) {
  if (q.M <= 0 || q.N <= 0 || q.K <= 0) return false;
  if (q.A.ld % 8 != 0 || q.B.ld % 8 != 0 || !aligned(q.A.p, 16) || !aligned(q.B.p, 16)) return false;
  if (!aligned(q.C, 16) || (q.ldc * (q.c_f32 ? 4 : 2)) % 16 != 0) return false;
  if (q.ksplit < 1 || (q.ksplit > 1 && !q.c_f32)) return false;
  return true;
}

int gemm_tc_batched(const TcProblem* probs, int count, int* status, cudaStream_t st) {
  if (count <= 0) return AB_OK;
  if (count > kMaxProbs || !tc_device_ok()) return AB_ERR_UNSUPPORTED;
  TcBatch batch;
  std::memset(&batch, 0, sizeof(batch));
  int tiles = 0;
  for (int i = 0; i < count; ++i) {
    const TcProblem& q = probs[i];
    if (!gemm_tc_problem_ok(q)) return AB_ERR_UNSUPPORTED;
    TcProblemDev& d = batch.prob[i];
    if (q.A.mn) AB_TRY(make_tensor_map_2d(&d.a, q.A.p, false, q.K, q.M, q.A.ld, 64, 64));
    else AB_TRY(make_tensor_map_2d(&d.a, q.A.p, false, q.M, q.K, q.A.ld, 64, kBM));
    if (q.B.mn) AB_TRY(make_tensor_map_2d(&d.b, q.B.p, false, q.K, q.N, q.B.ld, 64, 64));
    else AB_TRY(make_tensor_map_2d(&d.b, q.B.p, false, q.N, q.K, q.B.ld, 64, kBN));
    d.M = q.M; d.N = q.N; d.K = q.K;
    d.a_mn = q.A.mn ? 1 : 0; d.b_mn = q.B.mn ? 1 : 0; d.c_f32 = q.c_f32 ? 1 : 0;
    d.tiles_n = (q.N + kBN - 1) / kBN;
    d.ksplit = q.ksplit;
    const int slabs = (q.K + kBK - 1) / kBK;
    d.kslice = ((slabs + q.ksplit - 1) / q.ksplit) * kBK;
    d.c_rows = q.ksplit > 1 ? (q.M + kBM - 1) / kBM * kBM : q.M;
    AB_TRY(make_tensor_map_2d(&d.c, q.C, q.c_f32, (uint64_t)d.c_rows * q.ksplit, q.N, q.ldc,
                              q.c_f32 ? 32 : 64, 32));
    d.first_tile = tiles;
    tiles += ((q.M + kBM - 1) / kBM) * d.tiles_n * q.ksplit;
  }
  const size_t smem = (size_t)kStages * kStage + 4 * 2 * kStgBytes + sizeof(TcBars) + 1024;
  AB_CUDA_OK(cudaFuncSetAttribute(gemm_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int sms = sm_count();
  if (sms <= 0) return AB_ERR_CUDA;
  const int grid = tiles < sms ? tiles : sms;
  batch.nprobs = count; batch.ntiles = tiles; batch.status = status;
  return launch_after(gemm_tc_kernel, (unsigned)grid, (unsigned)kTcThreads, smem, 1, st, batch);
}

}  // namespace ab
