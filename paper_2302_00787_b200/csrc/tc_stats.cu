// Set statistics of Theorems 4.2 and 4.3 on the tensor cores, for bf16 tokens with d = 64:
// M1 = L^-1 sum x x^T, M2 = L^-1 sum y y^T, mu4 = mean x, mu5 = mean y.
//
// A 128-token tile X [128 x 64] sits in shared memory once (TMA, 128-byte swizzle) and is read
// by the MMA as both operands: D = [X | E]^T X with E the constant tile whose first column is 1.
// Rows 0..63 of D are the tile's Gram matrix, row 64 its column sums.  Products of bf16 values
// are exact in fp32; the fp32 sums of ST_FOLD tiles at a time are folded into fp64 registers (the fold, 64
// conversions and additions per thread, is what a tile's arrival rate from HBM has to cover), and the
// blocks of one group are combined with fp64 atomics.  The kernel is bound by the HBM read of Q and K.
// d = 128 (tc_stats128_kernel): D = [X_a | X_b]^T [X_a | X_b | E] from the two 64-column panels of a token tile, the column sums
// in column 128; twice the epilogue, one block per SM.
#include "common.cuh"
#include "tc_common.cuh"
#include "tc_layout.cuh"

using namespace tc;
using namespace tcl;

namespace {

constexpr int ST_STAGES = 4;                 // ring of token tiles in flight (two blocks share an SM: eight tiles per SM)
constexpr int ST_FOLD = 2;                   // tiles summed in one fp32 accumulator before it is folded into fp64
constexpr int ST_EPI_WARPS = 3;              // rows 0..95 of D; only 0..64 carry data
constexpr int ST_WARP_TMA = 3, ST_WARP_MMA = 4, ST_THREADS = 160;
constexpr uint32_t ST_TMEM_COLS = 128;       // two accumulators of 64 columns

struct StSmem {
  static constexpr uint32_t X0 = 0, ONES = ST_STAGES * TILE_BYTES, MISC = ONES + TILE_BYTES, TOTAL = MISC + 256;
};
struct StMisc {
  uint64_t full[ST_STAGES], empty[ST_STAGES], acc_full[2], acc_free[2];
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(StMisc) <= 256, "misc block");

__global__ void __launch_bounds__(ST_THREADS, 2)
tc_stats_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, int H, int Lq, int Lk,
                int Bpool, double qk_scale, int tiles_per_split, double* __restrict__ stats,
                int* __restrict__ status) {
  constexpr int NST = ST_STAGES;
  fs_grid_dependency_wait();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  StMisc* misc = reinterpret_cast<StMisc*>(sm + StSmem::MISC);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int side = blockIdx.z;
  // One group's tokens are one stream of tiles: the Bpool sequences that the group pools, one after the other.  A block takes a
  // range of the stream (a block per sequence and range, 64 x 12 sequences of four tiles pooled per head: 1536 blocks, each
  // adding its 4160 sums into one of 24 matrices, 43 us; 288 blocks of 22 tiles now, 24 us).
  const int g = blockIdx.y, h = g % H, b0 = g / H;          // (pooled per head: b0 = 0)
  const int L = side ? Lk : Lq;
  const CUtensorMap* tm = side ? &tmK : &tmQ;
  const int seq_tiles = (L + TILE - 1) / TILE;
  const int tile0 = blockIdx.x * tiles_per_split;
  const int ntiles = min(tiles_per_split, Bpool * seq_tiles - tile0);
  if (ntiles <= 0) return;                    // uniform over the block, before anything is allocated
  volatile int* abortp = &misc->abort_flag;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NST; i++) { mbar_init(&misc->full[i], 1); mbar_init(&misc->empty[i], 1); }
    for (int i = 0; i < 2; i++) { mbar_init(&misc->acc_full[i], 1); mbar_init(&misc->acc_free[i], ST_EPI_WARPS); }
    misc->abort_flag = 0;
    fence_barrier_init();
  }
  for (int i = threadIdx.x; i < TILE_BYTES / 16; i += ST_THREADS) reinterpret_cast<uint4*>(sm + StSmem::ONES)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  if (threadIdx.x < TILE)
    *reinterpret_cast<__nv_bfloat16*>(sm + StSmem::ONES + sw128_offset(threadIdx.x, 0)) = __float2bfloat16(1.f);
  fence_proxy_async_smem();
  if (warp == ST_WARP_MMA) {
    tmem_alloc(&misc->tmem_base, ST_TMEM_COLS);
    tmem_relinquish();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = misc->tmem_base;

  if (warp == ST_WARP_TMA) {
    if (lane == 0) {
      prefetch_tmap(tm);
      int issued = 0, b = b0 + tile0 / seq_tiles, t = tile0 % seq_tiles;
      for (int it = 0; it < ntiles; it++) {
        const int st = it % NST;
        if (!mbar_wait(&misc->empty[st], ((it / NST) & 1) ^ 1, abortp, status)) break;
        mbar_expect_tx(&misc->full[st], TILE_BYTES);
        tma_load_4d(sm + StSmem::X0 + st * TILE_BYTES, tm, &misc->full[st], 0, t * TILE, h, b);
        issued = it + 1;
        if (++t == seq_tiles) { t = 0; b++; }
      }
      // no copy of this block may still be in flight when it exits
      for (int it = max(0, issued - NST); it < issued; it++)
        mbar_wait(&misc->full[it % NST], (it / NST) & 1, abortp, status, false);
    }
  } else if (warp == ST_WARP_MMA) {
    // The whole warp walks the schedule (waits and descriptor arithmetic stay warp-uniform); lane 0 issues.
    // An MMA issued by a single lane of a diverged warp costs its thread two to three times as long.
    constexpr uint32_t ID = idesc_bf16(128, TC_D, 1, 1);      // both operands MN-major (feature index contiguous)
    const uint32_t sX0 = smem_u32(sm + StSmem::X0), sOnes = smem_u32(sm + StSmem::ONES);
    for (int it = 0; it < ntiles; it++) {
      const int st = it % NST, grp = it / ST_FOLD, buf = grp & 1, sub = it % ST_FOLD;
      if (!__all_sync(0xffffffffu, mbar_wait(&misc->full[st], (it / NST) & 1, abortp, status))) break;
      if (sub == 0 && !__all_sync(0xffffffffu, mbar_wait(&misc->acc_free[buf], ((grp >> 1) & 1) ^ 1, abortp, status))) break;
      tcgen05_fence_after();
      const uint32_t sX = sX0 + st * TILE_BYTES;
      // A = [X | E]: block 0 the tile, block 1 the constant tile (leading offset = their distance); a step's
      // descriptors are the tile's plus a constant in the low word (start address / 16)
      const uint64_t dA = smem_desc(sX, sOnes - sX, 1024, SWZ_128B);
      const uint64_t dB = smem_desc(sX, TILE_BYTES, 1024, SWZ_128B);
      uint32_t al = (uint32_t)dA, bl = (uint32_t)dB;
      const uint32_t ah = (uint32_t)(dA >> 32), bh = (uint32_t)(dB >> 32);
      opaque(al); opaque(bl);
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < TILE / 16; k++)
          mma_bf16_lh(tmem + buf * TC_D, al + k * 128, ah, bl + k * 128, bh, ID, (k > 0 || sub > 0) ? 1u : 0u);
        if (sub == ST_FOLD - 1 || it == ntiles - 1) mma_commit(&misc->acc_full[buf]);
        mma_commit(&misc->empty[st]);
      }
      __syncwarp();
    }
  } else {
    // epilogue: thread = row of D (rows 0..63 Gram, row 64 column sums), 64 columns
    const int row = warp * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
    double acc[TC_D];
#pragma unroll
    for (int j = 0; j < TC_D; j++) acc[j] = 0.0;
    bool alive = true;
    const int ngroups = (ntiles + ST_FOLD - 1) / ST_FOLD;
    for (int it = 0; it < ngroups && alive; it++) {
      const int buf = it & 1;
      if (!mbar_wait(&misc->acc_full[buf], (it >> 1) & 1, abortp, status, false)) { alive = false; break; }
      __syncwarp();
      tcgen05_fence_after();
#pragma unroll
      for (int c = 0; c < TC_D / 16; c++) {
        uint32_t t[16];
        tmem_ld16(lane_addr + buf * TC_D + c * 16, t);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 16; j++) acc[c * 16 + j] += (double)__uint_as_float(t[j]);
      }
      tcgen05_fence_before();
      mbar_arrive_warp(&misc->acc_free[buf], lane);
    }
    if (alive && row <= TC_D) {
      const double inv = 1.0 / ((double)L * (double)Bpool);
      StatsLayout sl{TC_D};
      double* out = stats + (size_t)g * sl.total();
      bool bad = false;
      if (row < TC_D) {
        // the Gram matrix is symmetric: row `row` is stored as column `row`, so a warp's atomics coalesce
        double* Mo = out + sl.M(side + 1);
        const double f = inv * qk_scale * qk_scale;
#pragma unroll
        for (int j = 0; j < TC_D; j++) {
          if (!isfinite(acc[j])) bad = true;
          atomicAdd(&Mo[(size_t)j * TC_D + row], acc[j] * f);
        }
      } else {
        double* mu = out + sl.mu(side + 4);
        const double f = inv * qk_scale;
#pragma unroll
        for (int j = 0; j < TC_D; j++) {
          if (!isfinite(acc[j])) bad = true;
          atomicAdd(&mu[j], acc[j] * f);
        }
      }
      if (bad) atomicExch(status, FSHARP_E_NONFINITE);
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == ST_WARP_MMA) {
    tcgen05_fence_after();
    tmem_dealloc(tmem, ST_TMEM_COLS);
  }
}

// d = 128.  Stage: [X_a | X_b | E], E (first column 1) written once per stage; a 128 x 144 accumulator, two of them; thread of the
// epilogue = (row of D, half of its columns).  As four blocks of the matrix on blocks of their own every panel came in four
// times: 1 x 16 x 65536 tokens 207 us, 98 us now (HBM 81).
constexpr int SW_STAGES = 4, SW_EPI_WARPS = 8, SW_WARP_TMA = 8, SW_WARP_MMA = 9, SW_THREADS = 320, SW_N = 144;
struct SwSmem {
  static constexpr uint32_t STAGE = 3 * TILE_BYTES, MISC = SW_STAGES * STAGE, TOTAL = MISC + 256;
};
static_assert(SwSmem::TOTAL + 1024 <= 232448, "shared memory budget");

__global__ void __launch_bounds__(SW_THREADS, 1)
tc_stats128_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, int H, int Lq, int Lk,
                   int Bpool, double qk_scale, int tiles_per_split, double* __restrict__ stats, int* __restrict__ status) {
  constexpr int DD = 2 * TC_D;
  fs_grid_dependency_wait();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  StMisc* misc = reinterpret_cast<StMisc*>(sm + SwSmem::MISC);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int side = blockIdx.z, g = blockIdx.y, h = g % H, b0 = g / H;          // (the stream of tiles: as above)
  const int L = side ? Lk : Lq;
  const CUtensorMap* tm = side ? &tmK : &tmQ;
  const int seq_tiles = (L + TILE - 1) / TILE;
  const int tile0 = blockIdx.x * tiles_per_split;
  const int ntiles = min(tiles_per_split, Bpool * seq_tiles - tile0);
  if (ntiles <= 0) return;                    // uniform over the block, before anything is allocated
  volatile int* abortp = &misc->abort_flag;

  if (threadIdx.x == 0) {
    for (int i = 0; i < SW_STAGES; i++) { mbar_init(&misc->full[i], 1); mbar_init(&misc->empty[i], 1); }
    for (int i = 0; i < 2; i++) { mbar_init(&misc->acc_full[i], 1); mbar_init(&misc->acc_free[i], SW_EPI_WARPS); }
    misc->abort_flag = 0;
    fence_barrier_init();
  }
  for (int i = threadIdx.x; i < SW_STAGES * (int)(TILE_BYTES / 16); i += SW_THREADS)
    reinterpret_cast<uint4*>(sm + (i >> 10) * SwSmem::STAGE + 2 * TILE_BYTES)[i & 1023] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  for (int i = threadIdx.x; i < SW_STAGES * TILE; i += SW_THREADS)
    *reinterpret_cast<__nv_bfloat16*>(sm + (i >> 7) * SwSmem::STAGE + 2 * TILE_BYTES + sw128_offset(i & 127, 0)) = __float2bfloat16(1.f);
  fence_proxy_async_smem();
  if (warp == SW_WARP_MMA) {
    tmem_alloc(&misc->tmem_base, 512);
    tmem_relinquish();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = misc->tmem_base;

  if (warp == SW_WARP_TMA) {
    if (lane == 0) {
      prefetch_tmap(tm);
      int issued = 0, b = b0 + tile0 / seq_tiles, t = tile0 % seq_tiles;
      for (int it = 0; it < ntiles; it++) {
        const int st = it % SW_STAGES;
        if (!mbar_wait(&misc->empty[st], ((it / SW_STAGES) & 1) ^ 1, abortp, status)) break;
        mbar_expect_tx(&misc->full[st], 2 * TILE_BYTES);
        tma_load_4d(sm + st * SwSmem::STAGE, tm, &misc->full[st], 0, t * TILE, h, b);
        tma_load_4d(sm + st * SwSmem::STAGE + TILE_BYTES, tm, &misc->full[st], TC_D, t * TILE, h, b);
        issued = it + 1;
        if (++t == seq_tiles) { t = 0; b++; }
      }
      // no copy of this block may still be in flight when it exits
      for (int it = max(0, issued - SW_STAGES); it < issued; it++)
        mbar_wait(&misc->full[it % SW_STAGES], (it / SW_STAGES) & 1, abortp, status, false);
    }
  } else if (warp == SW_WARP_MMA) {
    constexpr uint32_t ID = idesc_bf16(128, SW_N, 1, 1);      // both operands MN-major (feature index contiguous)
    for (int it = 0; it < ntiles; it++) {
      const int st = it % SW_STAGES, grp = it / ST_FOLD, buf = grp & 1, sub = it % ST_FOLD;
      if (!__all_sync(0xffffffffu, mbar_wait(&misc->full[st], (it / SW_STAGES) & 1, abortp, status))) break;
      if (sub == 0 && !__all_sync(0xffffffffu, mbar_wait(&misc->acc_free[buf], ((grp >> 1) & 1) ^ 1, abortp, status))) break;
      tcgen05_fence_after();
      const uint64_t d = smem_desc(smem_u32(sm + st * SwSmem::STAGE), TILE_BYTES, 1024, SWZ_128B);
      uint32_t dl = (uint32_t)d;
      const uint32_t dh = (uint32_t)(d >> 32);
      opaque(dl);
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < TILE / 16; k++)
          mma_bf16_lh(tmem + buf * 256, dl + k * 128, dh, dl + k * 128, dh, ID, (k > 0 || sub > 0) ? 1u : 0u);
        if (sub == ST_FOLD - 1 || it == ntiles - 1) mma_commit(&misc->acc_full[buf]);
        mma_commit(&misc->empty[st]);
      }
      __syncwarp();
    }
  } else {
    const int half = warp >> 2, row = (warp & 3) * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    double acc[TC_D], sum = 0.0;
#pragma unroll
    for (int j = 0; j < TC_D; j++) acc[j] = 0.0;
    bool alive = true;
    const int ngroups = (ntiles + ST_FOLD - 1) / ST_FOLD;
    for (int it = 0; it < ngroups && alive; it++) {
      const int buf = it & 1;
      if (!mbar_wait(&misc->acc_full[buf], (it >> 1) & 1, abortp, status, false)) { alive = false; break; }
      __syncwarp();
      tcgen05_fence_after();
      uint32_t s0;
      tmem_ld1(lane_addr + buf * 256 + DD, s0);
#pragma unroll
      for (int c = 0; c < TC_D / 16; c++) {
        uint32_t t[16];
        tmem_ld16(lane_addr + buf * 256 + half * TC_D + c * 16, t);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 16; j++) acc[c * 16 + j] += (double)__uint_as_float(t[j]);
      }
      sum += (double)__uint_as_float(s0);
      tcgen05_fence_before();
      mbar_arrive_warp(&misc->acc_free[buf], lane);
    }
    if (alive) {
      const double inv = 1.0 / ((double)L * (double)Bpool);
      StatsLayout sl{DD};
      double* out = stats + (size_t)g * sl.total();
      // (the Gram matrix is symmetric: row `row` is stored as column `row`, so a warp's atomics coalesce)
      double* Mo = out + sl.M(side + 1) + (size_t)(half * TC_D) * DD;
      const double f = inv * qk_scale * qk_scale;
      bool bad = false;
#pragma unroll
      for (int j = 0; j < TC_D; j++) {
        if (!isfinite(acc[j])) bad = true;
        atomicAdd(&Mo[(size_t)j * DD + row], acc[j] * f);
      }
      if (half == 0) {
        if (!isfinite(sum)) bad = true;
        atomicAdd(&out[sl.mu(side + 4) + row], sum * (inv * qk_scale));
      }
      if (bad) atomicExch(status, FSHARP_E_NONFINITE);
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == SW_WARP_MMA) {
    tcgen05_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

bool aligned16(const void* p, TensorAddr a) {
  return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && a.sl % 8 == 0 && a.sh % 8 == 0 && a.sb % 8 == 0;
}

}  // namespace

namespace tchost {
int make_map_tokens(CUtensorMap* map, const void* base, TensorAddr a, int B, int H, int L, int inner);
}

int fs_tc_stats_supported(const void* Q, const void* K, const fsharp_dims* dm, int dtype) {
  if (dtype != FSHARP_BF16 || (dm->d != TC_D && dm->d != 2 * TC_D) || dm->Lq <= 0 || dm->Lk <= 0) return 0;
  return aligned16(Q, fs_addr(dm->q_stride, dm->H, dm->Lq, dm->d)) && aligned16(K, fs_addr(dm->k_stride, dm->H, dm->Lk, dm->d));
}

// The statistics block must already be zero (the blocks add into it).
int fs_tc_stats(fsharp_ctx* ctx, const void* Q, const void* K, const fsharp_dims* dm, float qk_scale, double* stats) {
  const int B = dm->B, H = dm->H, BH = B * H;
  const int Lmax = dm->Lq > dm->Lk ? dm->Lq : dm->Lk;
  const int Bpool = dm->pool == FSHARP_POOL_PER_BH ? 1 : B, G = BH / Bpool;
  const int tiles = Bpool * ((Lmax + TILE - 1) / TILE);                // of one group
  const bool wide = dm->d == 2 * TC_D;
  // two blocks per SM (each block has one MMA-issuing thread, and issuing is what bounds a block; d = 128: one): the split of
  // a group's tiles with the fewest (waves x tiles per block)
  const int slots = (wide ? 1 : 2) * ctx->sm_count;
  int best = 1, best_cost = 0x7fffffff, tps = tiles;
  for (int ns = 1; ns <= tiles && ns <= 4 * ctx->sm_count; ns++) {
    const int t = (tiles + ns - 1) / ns;
    if ((tiles + t - 1) / t != ns) continue;
    const long long blocks = 2LL * G * ns;
    const int waves = (int)((blocks + slots - 1) / slots);
    const int cost = waves * (t + 6);        // fill, drain and the final atomics cost about six tiles
    if (cost < best_cost) { best_cost = cost; best = ns; tps = t; }
  }
  CUtensorMap tmQ, tmK;
  FS_TRY(tchost::make_map_tokens(&tmQ, Q, fs_addr(dm->q_stride, H, dm->Lq, dm->d), B, H, dm->Lq, dm->d));
  FS_TRY(tchost::make_map_tokens(&tmK, K, fs_addr(dm->k_stride, H, dm->Lk, dm->d), B, H, dm->Lk, dm->d));
  if (wide) {
    FS_CUDA_OK(cudaFuncSetAttribute(tc_stats128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SwSmem::TOTAL + 1024));
    FS_TIME_BEGIN(ctx, FS_K_TC_STATS);
    (void)fs_launch_chained(tc_stats128_kernel, dim3(best, G, 2), dim3(SW_THREADS), SwSmem::TOTAL + 1024, ctx->stream,
        tmQ, tmK, H, dm->Lq, dm->Lk, Bpool, (double)qk_scale, tps, stats, ctx->d_status);
    FS_TIME_END(ctx);
  } else {
    FS_CUDA_OK(cudaFuncSetAttribute(tc_stats_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)StSmem::TOTAL + 1024));
    FS_TIME_BEGIN(ctx, FS_K_TC_STATS);
    (void)fs_launch_chained(tc_stats_kernel, dim3(best, G, 2), dim3(ST_THREADS), StSmem::TOTAL + 1024, ctx->stream,
        tmQ, tmK, H, dm->Lq, dm->Lk, Bpool, (double)qk_scale, tps, stats, ctx->d_status);
    FS_TIME_END(ctx);
  }
  FS_LAUNCH_CHECK(ctx);
  return FSHARP_OK;
}
