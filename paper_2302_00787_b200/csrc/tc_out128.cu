// Query side of the causal chunked form (Section 2.2 with Khat = P S^T under the lower-triangular mask) on the tensor
// cores for the shapes that have no fused kernel (bf16, dv = 128, M a multiple of 128, chunks of 128 or 256):
//   [num | den]_i = phi(Q)_i KV_c + sum_{j <= i in chunk c} (phi(Q)_i . phi(K)_j) [V_j | 1],   Y_i = num_i / den_i
// with KV_c the sum of the earlier chunks' key-side sums (tc_kv128.cu: bf16, [M][128] and the normaliser's column).
//
// Blocks are persistent, one per SM, each with a range of consecutive 128-token tiles.  Per tile: stages of 64 features, of which
// phi(Q) (K-major A operand) multiplies the rows of KV_c (MN-major, N = 128), the normaliser's row (N = 16) and the phi(K) tiles of
// the chunk up to the query's own (K-major, N = 128 each): numerators, normalisers and scores at once.  Then the scores are
// masked, rounded to bf16 and put back into tensor memory, from where they multiply [V | 1] (V MN-major, the ones column from
// a constant tile) into the same accumulator; the epilogue divides and writes bf16 rows.
// Bound: HBM (phi(Q), phi(K), KV_c, V, Y: 390 KB per tile).  The chain at a tile's end (scores to bf16, their product, the
// output) is some 2.5 us, the next tile's copies go on under it: three stages are 4 us of this SM's share of the copy rate.
// (The scores by a kernel of their own, 423 us for 1 x 16 x 65536 tokens, M = 512, chunks of 256, and this kernel on what it
// left in HBM, 450 us, read phi(Q) twice and moved the scores out and in; 612 us now.  DRAM counters for a quarter of the tokens: 886 MB in
// 156 us, 87 % of the copy rate, tensor pipe 35 % busy.)
#include "common.cuh"
#include "tc_common.cuh"
#include "tc_layout.cuh"

using namespace tc;
using namespace tcl;

namespace {

constexpr int OU_ST = 3;
constexpr int OUE_WARPS = 8, OUW_TMA = 8, OUW_MMA = 9, OUT_T = 320;
constexpr uint32_t OU_TMEM_COLS = 512;                 // 128 numerators, 16 (normaliser in the first), two score tiles
constexpr uint32_t OU_DEN = 128, OU_S = 160;
constexpr uint32_t OU_PANEL = 8192;                    // 64 rows x 128 bytes of KV_c
// phi(Q); KV_c columns 0..63, 64..127; the normaliser's row (16 rows of 128 bytes); phi(K) tiles 0, 1.  After the features: V tiles
constexpr uint32_t OU_OFF_S = TILE_BYTES, OU_OFF_D = OU_OFF_S + 2 * OU_PANEL, OU_OFF_K = OU_OFF_D + 2048, OU_STAGE = OU_OFF_K + 2 * TILE_BYTES;
static_assert(4 * TILE_BYTES <= OU_STAGE, "two tiles of V in a stage");

struct OuSm {
  static constexpr uint32_t A0 = 0, ONES = OU_ST * OU_STAGE, MISC = ONES + TILE_BYTES, TOTAL = MISC + 256;
};
struct OuMs {
  uint64_t full[OU_ST], empty[OU_ST], s_full, s_ready, o_full, o_free;
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(OuMs) <= 256, "misc block");
static_assert(OU_STAGE % 1024 == 0 && OuSm::TOTAL + 1024 <= 232448, "shared memory budget");

__global__ void __launch_bounds__(OUT_T, 1)
tc_out128_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmS,
                 const __grid_constant__ CUtensorMap tmD, const __grid_constant__ CUtensorMap tmV, __nv_bfloat16* __restrict__ Y,
                 TensorAddr ay, int H, int M, int C, int nch, int total, int* __restrict__ status) {
  fs_grid_dependency_wait();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  OuMs* misc = reinterpret_cast<OuMs*>(sm + OuSm::MISC);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tpc = C / TILE, nf = M / 64;       // tiles per chunk (1 or 2); stages over the features, then one with V
  // tiles of all (batch, head)s in a row: item w = tile w % (nch tpc) of (batch, head) w / (nch tpc)
  const int w0 = (int)((int64_t)total * blockIdx.x / gridDim.x), w1 = (int)((int64_t)total * (blockIdx.x + 1) / gridDim.x);
  volatile int* abortp = &misc->abort_flag;

  if (threadIdx.x == 0) {
    for (int i = 0; i < OU_ST; i++) { mbar_init(&misc->full[i], 1); mbar_init(&misc->empty[i], 1); }
    mbar_init(&misc->s_full, 1);
    mbar_init(&misc->s_ready, OUE_WARPS);
    mbar_init(&misc->o_full, 1);
    mbar_init(&misc->o_free, OUE_WARPS);
    misc->abort_flag = 0;
    fence_barrier_init();
  }
  for (int i = threadIdx.x; i < (int)(TILE_BYTES / 16); i += OUT_T) reinterpret_cast<uint4*>(sm + OuSm::ONES)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  if (threadIdx.x < TILE)
    *reinterpret_cast<__nv_bfloat16*>(sm + OuSm::ONES + sw128_offset(threadIdx.x, 0)) = __float2bfloat16(1.f);
  fence_proxy_async_smem();
  if (warp == OUW_MMA) {
    tmem_alloc(&misc->tmem_base, OU_TMEM_COLS);
    tmem_relinquish();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = misc->tmem_base;

  if (warp == OUW_TMA) {
    if (lane == 0) {
      prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmS); prefetch_tmap(&tmD); prefetch_tmap(&tmV);
      int issued = 0;
      bool ok = true;
      for (int w = w0; w < w1 && ok; w++) {
        const int bh = w / (nch * tpc), tile = w % (nch * tpc), c = tile / tpc, nkt = tile % tpc + 1;
        const int tok = tile * TILE, first = c * C, unit = bh * nch + c, h = bh % H, b = bh / H;
        for (int it = 0; it <= nf; it++, issued++) {
          const int s = issued % OU_ST;
          if (!mbar_wait(&misc->empty[s], ((issued / OU_ST) & 1) ^ 1, abortp, status)) { ok = false; break; }
          uint8_t* base = sm + OuSm::A0 + s * OU_STAGE;
          uint64_t* bar = &misc->full[s];
          if (it < nf) {
            const int x = it * 64;
            mbar_expect_tx(bar, OU_OFF_K + nkt * TILE_BYTES);
            tma_load_4d(base, &tmQ, bar, x, tok, bh, 0);
            tma_load_4d(base + OU_OFF_S, &tmS, bar, 0, x, unit, 0);
            tma_load_4d(base + OU_OFF_S + OU_PANEL, &tmS, bar, 64, x, unit, 0);
            // (rows 1 .. 15 belong to later chunks, or are zeros past the last one: columns that nothing reads)
            tma_load_4d(base + OU_OFF_D, &tmD, bar, x, unit, 0, 0);
            for (int kt = 0; kt < nkt; kt++) tma_load_4d(base + OU_OFF_K + kt * TILE_BYTES, &tmK, bar, x, first + kt * TILE, bh, 0);
          } else {
            mbar_expect_tx(bar, 2 * nkt * TILE_BYTES);
            for (int kt = 0; kt < nkt; kt++) {
              tma_load_4d(base + 2 * kt * TILE_BYTES, &tmV, bar, 0, first + kt * TILE, h, b);
              tma_load_4d(base + (2 * kt + 1) * TILE_BYTES, &tmV, bar, 64, first + kt * TILE, h, b);
            }
          }
        }
      }
      // no copy of this block may still be in flight when it exits
      for (int it = max(0, issued - OU_ST); it < issued; it++)
        mbar_wait(&misc->full[it % OU_ST], (it / OU_ST) & 1, abortp, status, false);
    }
  } else if (warp == OUW_MMA) {
    // The whole warp walks the schedule (waits and descriptor arithmetic stay warp-uniform); an elected lane issues.
    constexpr uint32_t ID_KK = idesc_bf16(128, 128, 0, 0), ID_KK16 = idesc_bf16(128, 16, 0, 0);    // both K-major
    constexpr uint32_t ID_KM = idesc_bf16(128, 128, 0, 1), ID_KM16 = idesc_bf16(128, 16, 0, 1);    // B MN-major
    const uint32_t sA0 = smem_u32(sm + OuSm::A0), sOnes = smem_u32(sm + OuSm::ONES);
    int it = 0, n = 0;
    bool ok = true;
    auto wait = [&](uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abortp, status)) != 0; };
    for (int w = w0; w < w1 && ok; w++, n++) {
      const int nkt = w % (nch * tpc) % tpc + 1;
      ok = wait(&misc->o_free, (n & 1) ^ 1);
      for (int f = 0; f < nf && ok; f++, it++) {
        const int s = it % OU_ST;
        if (!(ok = wait(&misc->full[s], (it / OU_ST) & 1))) break;
        tcgen05_fence_after();
        const uint32_t base = sA0 + s * OU_STAGE;
        const uint64_t dA = smem_desc(base, 16, 1024, SWZ_128B), dS = smem_desc(base + OU_OFF_S, OU_PANEL, 1024, SWZ_128B);
        uint32_t al = (uint32_t)dA, sl = (uint32_t)dS;
        const uint32_t ah = (uint32_t)(dA >> 32), sh = (uint32_t)(dS >> 32);
        opaque(al); opaque(sl);
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < 4; k++) {
            const uint32_t more = (f | k) ? 1u : 0u;
            mma_bf16_lh(tmem, al + 2 * k, ah, sl + 128 * k, sh, ID_KM, more);
            mma_bf16_lh(tmem + OU_DEN, al + 2 * k, ah, al + OU_OFF_D / 16 + 2 * k, ah, ID_KK16, more);
            mma_bf16_lh(tmem + OU_S, al + 2 * k, ah, al + OU_OFF_K / 16 + 2 * k, ah, ID_KK, more);
            if (nkt > 1) mma_bf16_lh(tmem + OU_S + 128, al + 2 * k, ah, al + (OU_OFF_K + TILE_BYTES) / 16 + 2 * k, ah, ID_KK, more);
          }
          mma_commit(&misc->empty[s]);
          if (f == nf - 1) mma_commit(&misc->s_full);
        }
        __syncwarp();
      }
      if (!ok) break;
      const int s = it % OU_ST;
      if (!(ok = wait(&misc->full[s], (it / OU_ST) & 1) && wait(&misc->s_ready, n & 1))) break;
      tcgen05_fence_after();
      // V: two 64-column panels (leading offset = their distance), 16 keys per step = 16 rows of 128 bytes
      const uint64_t dV = smem_desc(sA0 + s * OU_STAGE, TILE_BYTES, 1024, SWZ_128B), dE = smem_desc(sOnes, TILE_BYTES, 1024, SWZ_128B);
      uint32_t vl = (uint32_t)dV, el = (uint32_t)dE;
      const uint32_t vh = (uint32_t)(dV >> 32), eh = (uint32_t)(dE >> 32);
      opaque(vl); opaque(el);
      if (elect_one()) {
        for (int kt = 0; kt < nkt; kt++) {
          // (a chunk's first tile has its scores' bf16 copy where a second tile's scores would be)
          const uint32_t p = tmem + OU_S + (nkt == 1 ? 128 : kt * 128);
#pragma unroll
          for (int k = 0; k < 8; k++) {
            mma_bf16_ta_lh(tmem, p + 8 * k, vl + kt * (2 * TILE_BYTES / 16) + k * 128, vh, ID_KM, 1u);
            mma_bf16_ta_lh(tmem + OU_DEN, p + 8 * k, el + k * 128, eh, ID_KM16, 1u);
          }
        }
        mma_commit(&misc->empty[s]);
        mma_commit(&misc->o_full);
      }
      __syncwarp();
      it++;
    }
  } else {
    // epilogue: thread = token; the two warpgroups share a tile's columns
    const int wg = warp >> 2, row = (warp & 3) * 32 + lane;
    const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    for (int w = w0, n = 0; w < w1; w++, n++) {
      const int bh = w / (nch * tpc), tile = w % (nch * tpc), nkt = tile % tpc + 1;
      if (!mbar_wait(&misc->s_full, n & 1, abortp, status, false)) break;
      __syncwarp();
      tcgen05_fence_after();
      // scores -> masked, bf16.  Two score tiles: one per warpgroup, in place (a piece's packed values go where values already read
      // were).  One: half of its columns each, to the second tile's place, since in place one group would write what the
      // other has yet to read.
      const uint32_t src = lanes + OU_S + (nkt > 1 ? wg * 128 : wg * 64), dst = lanes + OU_S + (nkt > 1 ? wg * 128 : 128 + wg * 32);
      const int cols = nkt > 1 ? 128 : 64, last = nkt > 1 ? (wg ? row : TILE) : row - wg * 64;      // columns up to `last` are kept
      for (int c = 0; c < cols; c += 32) {
        uint32_t t[32], o[16];
        tmem_ld16(src + c, *reinterpret_cast<uint32_t(*)[16]>(t));
        tmem_ld16(src + c + 16, *reinterpret_cast<uint32_t(*)[16]>(t + 16));
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; j++) t[j] = c + j <= last ? t[j] : 0u;
#pragma unroll
        for (int j = 0; j < 16; j++) o[j] = pack_bf16(__uint_as_float(t[2 * j]), __uint_as_float(t[2 * j + 1]));
        tmem_st16(dst + c / 2, o);
      }
      tmem_wait_st();
      tcgen05_fence_before();
      mbar_arrive_warp(&misc->s_ready, lane);
      if (!mbar_wait(&misc->o_full, n & 1, abortp, status, false)) break;
      __syncwarp();
      tcgen05_fence_after();
      uint32_t d[8], t[64];
      tmem_ld8(lanes + OU_DEN, d);
#pragma unroll
      for (int q = 0; q < 4; q++) tmem_ld16(lanes + wg * 64 + q * 16, *reinterpret_cast<uint32_t(*)[16]>(t + q * 16));
      tmem_wait_ld();
      tcgen05_fence_before();
      mbar_arrive_warp(&misc->o_free, lane);
      const float den = __uint_as_float(d[0]), inv = 1.f / den;
      if (!(den > 0.f) || !isfinite(den)) atomicExch(status, FSHARP_E_NONFINITE);
      __nv_bfloat16* out = Y + bh / H * ay.sb + bh % H * ay.sh + ((int64_t)tile * TILE + row) * ay.sl + wg * 64;
#pragma unroll
      for (int q = 0; q < 8; q++) {                    // (rows are 16-byte aligned)
        uint32_t o[4];
#pragma unroll
        for (int j = 0; j < 4; j++) o[j] = pack_bf16(inv * __uint_as_float(t[8 * q + 2 * j]), inv * __uint_as_float(t[8 * q + 2 * j + 1]));
        *reinterpret_cast<uint4*>(out + 8 * q) = make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == OUW_MMA) {
    tcgen05_fence_after();
    tmem_dealloc(tmem, OU_TMEM_COLS);
  }
}

}  // namespace

namespace tchost {
int make_map_tokens(CUtensorMap* map, const void* base, TensorAddr a, int B, int H, int L, int inner);
int make_map_rows(CUtensorMap* map, const void* base, TensorAddr a, int B, int H, int L, int inner, int box_rows);
}

// Y: bf16 [B,H,L,128] with 16-byte aligned rows
int fs_tc_out128_supported(const void* Y, TensorAddr ay) {
  if (reinterpret_cast<uintptr_t>(Y) % 16 != 0) return 0;
  return (ay.sl * 2) % 16 == 0 && (ay.sh * 2) % 16 == 0 && (ay.sb * 2) % 16 == 0;
}

// phiQ16, phiK16 [BH][L][M], st16 [BH * L / C][M][128] and z16 [BH * L / C][M] (sums of the earlier chunks), all bf16;
// V, Y [B,H,L,128] bf16; L a multiple of C
int fs_tc_out128(fsharp_ctx* ctx, const void* phiQ16, const void* phiK16, const void* st16, const void* z16, const void* V, TensorAddr av,
                 void* Y, TensorAddr ay, int B, int H, int L, int M, int C) {
  const int BH = B * H, nch = L / C, total = BH * (L / TILE);
  CUtensorMap tmQ, tmK, tmS, tmD, tmV;
  TensorAddr ap{(int64_t)BH * L * M, (int64_t)L * M, (int64_t)M};
  TensorAddr as{(int64_t)BH * nch * 128 * M, (int64_t)128 * M, 128};
  TensorAddr ad{(int64_t)BH * nch * M, (int64_t)BH * nch * M, (int64_t)M};
  FS_TRY(tchost::make_map_tokens(&tmQ, phiQ16, ap, 1, BH, L, M));
  FS_TRY(tchost::make_map_tokens(&tmK, phiK16, ap, 1, BH, L, M));
  FS_TRY(tchost::make_map_rows(&tmS, st16, as, 1, BH * nch, M, 128, 64));
  FS_TRY(tchost::make_map_rows(&tmD, z16, ad, 1, 1, BH * nch, M, 16));
  FS_TRY(tchost::make_map_tokens(&tmV, V, av, B, H, L, 128));
  FS_CUDA_OK(cudaFuncSetAttribute(tc_out128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OuSm::TOTAL + 1024));
  FS_TIME_BEGIN(ctx, FS_K_TC_OUT128);
  tc_out128_kernel<<<dim3(total < ctx->sm_count ? total : ctx->sm_count), OUT_T, OuSm::TOTAL + 1024, ctx->stream>>>(
      tmQ, tmK, tmS, tmD, tmV, (__nv_bfloat16*)Y, ay, H, M, C, nch, total, ctx->d_status);
  FS_TIME_END(ctx);
  FS_LAUNCH_CHECK(ctx);
  return FSHARP_OK;
}
