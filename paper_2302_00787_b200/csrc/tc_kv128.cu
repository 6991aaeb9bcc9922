// Key side of the causal chunked form, the running sums KV_c = sum over the chunks before c of S^T [V | 1] (Section 2.1's
// O(L M n) order), on the tensor cores for the shapes that have no fused kernel: bf16 copy of phi(K) [B*H][L][M], V [B,H,L,128]
// bf16.  Output, both bf16: st16 [B*H * L/C][M][128] and the normaliser's column z16 [B*H * L/C][M].
//
// One block = (segment of consecutive chunks, block of 128 features, (batch, head)).  Tokens are the contraction: a stage holds
// 128 tokens of the feature block (two 64-feature panels) and of V (two 64-column panels), all "MN-major" operands
// (the contracted index is the row of the tile).  Per 16 tokens: D[:, 0..127] += phi^T V (N = 128) and
// D[:, 128..143] += phi^T E with E the constant tile whose first column is 1 (N = 16).  Two accumulators in tensor
// memory: the epilogue takes chunk c while chunk c + 1 is multiplied.  A chunk's sum is added in fp32 to the running one, which
// the epilogue warps keep in registers and write, rounded to bf16, in front of every chunk: nothing else leaves the block.  (Sums
// of single chunks written in fp32, 505 us for 1 x 16 x 65536 tokens, M = 512, chunks of 256, and scanned by a kernel of its own,
// 265 us, moved 2.2 GB that never had to; the two launches take 139 and 292 us.)
// Segments: as many as there are SMs for all (segment, block, (batch, head)); where there is more than one, a first launch
// (EMIT = false) adds up the earlier ones, cut finer so that it fills the chip too, and the scan kernel turns the pieces' sums into
// what precedes every piece.  From half as many (block, (batch, head))s as SMs there is one segment each, also where that leaves SMs without
// work or a second wave short: the totals would read everything once more.  (Steps before, with single chunks' sums and their scan, and now, us:
// 25 x 4096 tokens, M = 512, 100 blocks, 481 and 334; 38 x 4096, M = 512, 152 blocks, 608 and 470; 75 x 2048, M = 256, 150, 438 and 349; 76 x 4096,
// M = 128, 76, 521 and 385.)
#include "common.cuh"
#include "tc_common.cuh"
#include "tc_layout.cuh"

using namespace tc;
using namespace tcl;

namespace {

constexpr int KV_ST = 3;
constexpr int KVE_WARPS = 8, KVW_TMA = 8, KVW_MMA = 9, KVT = 320;
constexpr uint32_t KV_ACC_COLS = 160;                  // 128 + 16, kept apart by a multiple of 32
constexpr uint32_t KV_TMEM_COLS = 512;                 // two accumulators (power of two)
constexpr uint32_t KV_STAGE = 4 * TILE_BYTES;          // feature panels 0, 1, then V panels 0, 1

struct KvSm {
  static constexpr uint32_t A0 = 0, ONES = KV_ST * KV_STAGE, MISC = ONES + TILE_BYTES, TOTAL = MISC + 256;
};
struct KvMs {
  uint64_t full[KV_ST], empty[KV_ST], acc_full[2], acc_free[2];
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(KvMs) <= 256, "misc block");
static_assert(KvSm::TOTAL + 1024 <= 232448, "shared memory budget");

// cps: chunks per segment; sub: pieces that the launch of the totals cuts a segment into, cpp chunks each (none is empty).
struct KvCut {
  int nch, cps, sub, cpp;
  __host__ __device__ int segments() const { return (nch + cps - 1) / cps; }
  __host__ __device__ int slots() const { return (segments() - 1) * sub + 1; }       // pieces, and one for what precedes the last segment
};

template <bool EMIT>
__global__ void __launch_bounds__(KVT, 1)
tc_kv128_kernel(const __grid_constant__ CUtensorMap tmP, const __grid_constant__ CUtensorMap tmV, float* __restrict__ tot,
                __nv_bfloat16* __restrict__ st16, __nv_bfloat16* __restrict__ z16, int H, int M, int C, KvCut cut,
                int* __restrict__ status) {
  fs_grid_dependency_wait();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  KvMs* misc = reinterpret_cast<KvMs*>(sm + KvSm::MISC);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int fblk = blockIdx.y, bh = blockIdx.z, b = bh / H, h = bh % H;
  const int seg = EMIT ? (int)blockIdx.x : (int)blockIdx.x / cut.sub, piece = EMIT ? 0 : (int)blockIdx.x % cut.sub;
  const int c0 = seg * cut.cps + piece * cut.cpp;
  const int ncs = min(EMIT ? cut.cps : min(cut.cpp, cut.cps - piece * cut.cpp), cut.nch - c0);
  if (ncs <= 0) return;                        // uniform over the block, before anything is allocated
  const int sums = EMIT ? ncs - 1 : ncs;       // chunks that are multiplied (nothing follows a segment's last one)
  const int tpc = C / TILE;                    // token tiles per chunk
  const int ntiles = sums * tpc;
  volatile int* abortp = &misc->abort_flag;
  constexpr int N = 129;

  if (threadIdx.x == 0) {
    for (int i = 0; i < KV_ST; i++) { mbar_init(&misc->full[i], 1); mbar_init(&misc->empty[i], 1); }
    for (int i = 0; i < 2; i++) { mbar_init(&misc->acc_full[i], 1); mbar_init(&misc->acc_free[i], KVE_WARPS); }
    misc->abort_flag = 0;
    fence_barrier_init();
  }
  for (int i = threadIdx.x; i < (int)(TILE_BYTES / 16); i += KVT) reinterpret_cast<uint4*>(sm + KvSm::ONES)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  if (threadIdx.x < TILE)
    *reinterpret_cast<__nv_bfloat16*>(sm + KvSm::ONES + sw128_offset(threadIdx.x, 0)) = __float2bfloat16(1.f);
  fence_proxy_async_smem();
  if (warp == KVW_MMA) {
    tmem_alloc(&misc->tmem_base, KV_TMEM_COLS);
    tmem_relinquish();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = misc->tmem_base;

  if (warp == KVW_TMA) {
    if (lane == 0) {
      prefetch_tmap(&tmP);
      prefetch_tmap(&tmV);
      int issued = 0;
      for (int it = 0; it < ntiles; it++) {
        const int s = it % KV_ST;
        const int tok = (c0 * tpc + it) * TILE;
        if (!mbar_wait(&misc->empty[s], ((it / KV_ST) & 1) ^ 1, abortp, status)) break;
        uint8_t* base = sm + KvSm::A0 + s * KV_STAGE;
        mbar_expect_tx(&misc->full[s], KV_STAGE);
        tma_load_4d(base, &tmP, &misc->full[s], fblk * 128, tok, bh, 0);
        tma_load_4d(base + TILE_BYTES, &tmP, &misc->full[s], fblk * 128 + 64, tok, bh, 0);
        tma_load_4d(base + 2 * TILE_BYTES, &tmV, &misc->full[s], 0, tok, h, b);
        tma_load_4d(base + 3 * TILE_BYTES, &tmV, &misc->full[s], 64, tok, h, b);
        issued = it + 1;
      }
      // no copy of this block may still be in flight when it exits
      for (int it = max(0, issued - KV_ST); it < issued; it++)
        mbar_wait(&misc->full[it % KV_ST], (it / KV_ST) & 1, abortp, status, false);
    }
  } else if (warp == KVW_MMA) {
    // The whole warp walks the schedule (waits and descriptor arithmetic stay warp-uniform); lane 0 issues.
    constexpr uint32_t ID_V = idesc_bf16(128, 128, 1, 1), ID_E = idesc_bf16(128, 16, 1, 1);   // both operands MN-major
    const uint32_t sA0 = smem_u32(sm + KvSm::A0), sOnes = smem_u32(sm + KvSm::ONES);
    for (int it = 0; it < ntiles; it++) {
      const int s = it % KV_ST, ch = it / tpc, sub = it % tpc, buf = ch & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&misc->full[s], (it / KV_ST) & 1, abortp, status))) break;
      if (sub == 0 && !__all_sync(0xffffffffu, mbar_wait(&misc->acc_free[buf], ((ch >> 1) & 1) ^ 1, abortp, status))) break;
      tcgen05_fence_after();
      const uint32_t sP = sA0 + s * KV_STAGE, sV = sP + 2 * TILE_BYTES;
      // operands of 128 (features / columns) = two 64-wide panels: the leading offset is the panels' distance
      const uint64_t dA = smem_desc(sP, TILE_BYTES, 1024, SWZ_128B);
      const uint64_t dB = smem_desc(sV, TILE_BYTES, 1024, SWZ_128B);
      const uint64_t dE = smem_desc(sOnes, TILE_BYTES, 1024, SWZ_128B);
      uint32_t al = (uint32_t)dA, bl = (uint32_t)dB, el = (uint32_t)dE;
      const uint32_t ah = (uint32_t)(dA >> 32), bhh = (uint32_t)(dB >> 32), eh = (uint32_t)(dE >> 32);
      opaque(al); opaque(bl); opaque(el);
      if (lane == 0) {
        const uint32_t acc = tmem + buf * KV_ACC_COLS;
#pragma unroll
        for (int k = 0; k < TILE / 16; k++) {
          mma_bf16_lh(acc, al + k * 128, ah, bl + k * 128, bhh, ID_V, (k > 0 || sub > 0) ? 1u : 0u);
          mma_bf16_lh(acc + 128, al + k * 128, ah, el + k * 128, eh, ID_E, (k > 0 || sub > 0) ? 1u : 0u);
        }
        if (sub == tpc - 1) mma_commit(&misc->acc_full[buf]);
        mma_commit(&misc->empty[s]);
      }
      __syncwarp();
    }
  } else {
    // epilogue: thread = feature row of D and 64 of its columns; the warps of the first half also take the ones column
    const int half = warp >> 2, row = (warp & 3) * 32 + lane, f = fblk * 128 + row;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    float run[64], z = 0.f;
#pragma unroll
    for (int j = 0; j < 64; j++) run[j] = 0.f;
    // totals [(batch, head)][piece][129][M]: the pieces' own sums, or (EMIT) those of the pieces before
    float* t = tot + (((size_t)bh * cut.slots() + seg * cut.sub + piece) * N + half * 64) * M + f;
    if (EMIT && seg > 0) {
#pragma unroll
      for (int j = 0; j < 64; j++) run[j] = t[(size_t)j * M];
      if (half == 0) z = t[(size_t)128 * M];
    }
    auto emit = [&](int c) {
      const size_t at = ((size_t)bh * cut.nch + c) * M + f;
      uint32_t* out = reinterpret_cast<uint32_t*>(st16 + at * 128 + half * 64);
#pragma unroll
      for (int q = 0; q < 4; q++) {                    // 32 bytes each
        uint32_t o[8];
#pragma unroll
        for (int j = 0; j < 8; j++) o[j] = pack_bf16(run[q * 16 + 2 * j], run[q * 16 + 2 * j + 1]);
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out + q * 8), "r"(o[0]), "r"(o[1]), "r"(o[2]),
                     "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
                     : "memory");
      }
      if (half == 0) z16[at] = __float2bfloat16_rn(z);
    };
    if (EMIT) emit(c0);
    for (int ch = 0; ch < sums; ch++) {
      const int buf = ch & 1;
      if (!mbar_wait(&misc->acc_full[buf], (ch >> 1) & 1, abortp, status, false)) break;
      __syncwarp();
      tcgen05_fence_after();
#pragma unroll
      for (int cc = 0; cc < 4; cc++) {
        uint32_t t[16];
        tmem_ld16(lane_addr + buf * KV_ACC_COLS + half * 64 + cc * 16, t);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 16; j++) run[cc * 16 + j] += __uint_as_float(t[j]);
      }
      if (half == 0) {
        uint32_t t[8];
        tmem_ld8(lane_addr + buf * KV_ACC_COLS + 128, t);
        tmem_wait_ld();
        z += __uint_as_float(t[0]);
      }
      tcgen05_fence_before();
      mbar_arrive_warp(&misc->acc_free[buf], lane);
      if (EMIT) emit(c0 + ch + 1);
    }
    if (!EMIT) {
#pragma unroll
      for (int j = 0; j < 64; j++) t[(size_t)j * M] = run[j];
      if (half == 0) t[(size_t)128 * M] = z;
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == KVW_MMA) {
    tcgen05_fence_after();
    tmem_dealloc(tmem, KV_TMEM_COLS);
  }
}

KvCut cut_of(const fsharp_ctx* ctx, int BH, int M, int nch) {
  const int units = BH * (M / 128);
  int ns = ctx->sm_count / units;
  ns = ns < 1 ? 1 : (ns > nch ? nch : ns);
  KvCut cut;
  cut.nch = nch;
  cut.cps = (nch + ns - 1) / ns;
  ns = cut.segments();
  int k = ns > 1 ? ctx->sm_count / (units * (ns - 1)) : 1;
  k = k < 1 ? 1 : (k > cut.cps ? cut.cps : k);
  cut.cpp = (cut.cps + k - 1) / k;
  cut.sub = (cut.cps + cut.cpp - 1) / cut.cpp;
  return cut;
}

}  // namespace

namespace tchost {
int make_map_tokens(CUtensorMap* map, const void* base, TensorAddr a, int B, int H, int L, int inner);
}

// bf16 tensors, dv = 128, M a multiple of 128, chunks of 128 or 256 tokens, 16-byte aligned V rows
int fs_tc_kv128_supported(const void* V, TensorAddr av, int dv, int M, int C) {
  if (dv != 128 || M % 128 != 0 || (C != 128 && C != 256)) return 0;
  if (reinterpret_cast<uintptr_t>(V) % 16 != 0) return 0;
  return (av.sl * 2) % 16 == 0 && (av.sh * 2) % 16 == 0 && (av.sb * 2) % 16 == 0;
}

// Totals per (batch, head) of [129][M] fp32; one: there is a single segment and no totals are needed.
int fs_tc_kv128_slots(const fsharp_ctx* ctx, int BH, int M, int nch) { return cut_of(ctx, BH, M, nch).slots(); }

// phiK16 [BH][L][M] bf16, V [B,H,L,128] bf16 (strides av).  st16 = null: the sums of the pieces of all segments but the last to
// tot [BH][slots][129][M]; else st16 [BH * L / C][M][128] and z16 [BH * L / C][M], from tot as the exclusive scan over slots.
int fs_tc_kv128(fsharp_ctx* ctx, const void* phiK16, const void* V, TensorAddr av, int B, int H, int L, int M, int C, float* tot,
                void* st16, void* z16) {
  const int BH = B * H, nch = L / C;
  const KvCut cut = cut_of(ctx, BH, M, nch);
  CUtensorMap tmP, tmV;
  TensorAddr ap{(int64_t)BH * L * M, (int64_t)L * M, (int64_t)M};
  FS_TRY(tchost::make_map_tokens(&tmP, phiK16, ap, 1, BH, L, M));
  FS_TRY(tchost::make_map_tokens(&tmV, V, av, B, H, L, 128));
  const auto kernel = st16 ? tc_kv128_kernel<true> : tc_kv128_kernel<false>;
  const size_t smem = KvSm::TOTAL + 1024;
  FS_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  FS_TIME_BEGIN(ctx, FS_K_TC_KV128);
  kernel<<<dim3(st16 ? cut.segments() : cut.slots() - 1, M / 128, BH), KVT, smem, ctx->stream>>>(
      tmP, tmV, tot, (__nv_bfloat16*)st16, (__nv_bfloat16*)z16, H, M, C, cut, ctx->d_status);
  FS_TIME_END(ctx);
  FS_LAUNCH_CHECK(ctx);
  return FSHARP_OK;
}
