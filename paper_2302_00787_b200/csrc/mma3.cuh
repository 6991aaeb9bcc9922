// Block product at fp32 precision on the tensor cores: D[128 x NT] = sum over segments of A_s B_s, operands read from
// global memory through caller-supplied loaders, turned into three-part bf16 operands (split3.cuh) on the way into shared
// memory, accumulated by tcgen05 in tensor memory.  It is what the fp32-precision kernels (attention, backward pass) are
// built from.
//
// 288 threads: warps 0-7 load, convert and store operand slices of 32 values of K (two stages) and later read the result;
// warp 8 issues the MMAs.  Two blocks fit on an SM (96 KB of stages, 256 columns of tensor memory each), so one block's
// conversion and epilogue run under the other's products.  Per slice of 128 x 128: 12 MMAs of 65 cycles (both operands
// fp32) against about 400 issue cycles of conversion.
// Two accumulators: h h products in one, everything with an m or l part in the other.  The tensor core truncates the
// accumulator at every MMA, so the large sum must not take the small products' steps too (tc_pairs.cu has the figures).  Where
// K exceeds 128 and the columns leave room (80 of them at most) the h h products take turns in two accumulators, slice by
// slice, so that each is truncated half as often; callers with K > 256 cut wider products into tiles of 64 columns for it.
// (Attention outputs, d = 64, L = 2048, relative error at M = 512 and 1024: 2.3e-6 and 4.9e-6 with one, 1.3e-6 and 2.5e-6 with
// two, 1.5e-6 and 1.6e-6 for fp32 multiply-adds.)
//
// Operand slices: contracted index contiguous ("K-major"): rows of 64 bytes, 64-byte swizzle; row / column index
// contiguous ("MN-major"): panels of 64 x 32, rows of 128 bytes, 128-byte swizzle.  Nothing is transposed on the way.
#pragma once
#include "common.cuh"
#include "split3.cuh"

namespace mma3 {

constexpr int THREADS = 288, PRODUCERS = 256, KS = 32, ROWS = 128;
constexpr uint32_t PART = 8192;                       // 128 x 32 bf16
constexpr uint32_t STAGE = 6 * PART;                  // A: h, m, l; B: h, m, l
// main accumulator at column 0, the small products' at 128; or the two main ones at 0 and SECOND, the small products' at CORR2
constexpr uint32_t TMEM = 256, CORR = 128, SECOND = 80, CORR2 = 160;
constexpr int LONG_K = 256;                           // from here on two main accumulators are worth narrower tiles

struct Misc {
  uint64_t full[2], empty[2], done;
  uint32_t tmem_base;
  int abort_flag;
};
constexpr size_t SMEM = 1024 + 2 * STAGE + 64;
static_assert(sizeof(Misc) <= 64, "misc block");

__device__ __forceinline__ uint4 zero4() { return make_uint4(0u, 0u, 0u, 0u); }

// eight consecutive fp32 / bf16 values; the pointers are 16-byte aligned
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
// One 8-value piece of an operand as it waits in registers for its stage: eight floats (PARTS = 3) or eight bf16
// (PARTS = 1, exact in bf16).
template <int PARTS> struct Piece;
template <> struct Piece<3> {
  float v[8];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int j = 0; j < 8; j++) v[j] = 0.f;
  }
  __device__ __forceinline__ void load(const float* p) { load8(p, v); }
  __device__ __forceinline__ void unit() { zero(); v[0] = 1.f; }                  // (1, 0, ..., 0): the ones column
  __device__ __forceinline__ void store(uint8_t* dst) const {
    uint4 h, m, l;
    split3::split8(v, h, m, l);
    *reinterpret_cast<uint4*>(dst) = h;
    *reinterpret_cast<uint4*>(dst + PART) = m;
    *reinterpret_cast<uint4*>(dst + 2 * PART) = l;
  }
};
template <> struct Piece<1> {
  uint4 r;
  __device__ __forceinline__ void zero() { r = zero4(); }
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { r = *reinterpret_cast<const uint4*>(p); }
  __device__ __forceinline__ void unit() { r = make_uint4(0x3f80u, 0u, 0u, 0u); }
  __device__ __forceinline__ void store(uint8_t* dst) const { *reinterpret_cast<uint4*>(dst) = r; }
};
// parts of a tensor's own values
template <typename T> struct PartsOf { static constexpr int N = 3; };
template <> struct PartsOf<__nv_bfloat16> { static constexpr int N = 1; };

// Which unit (z coordinate) a block takes.  Kernels of a chain walk the units up and down in turn: the matrices that one leaves behind
// are larger than the L2, and what it touched last is still there for the next one (causal training step of 2 x 12 x 4096 tokens: 1223 -> 1208 us).
__device__ __forceinline__ int unit_of(int flip) { return flip ? gridDim.z - 1 - blockIdx.z : blockIdx.z; }

// rows of `bytes` contiguous bytes, `stride` bytes apart, asked into L2 by the whole block ahead of its slices: a slice takes 128
// bytes of a row at a time, one slice ahead of its use, which is not enough against the latency of HBM.  For the matrices that a long
// sequence leaves in HBM: the tokens' own rows of bwd_dfeat and bwd_dx (gradients of 5 x 4 x 16722 bf16 tokens, d = 64, M = 256, 1783 us with none,
// 1741 with bwd_dfeat's, 1724 with both; of 2 x 12 x 4096, causal, 941 and 937).  The chunk's other rows too: 954, the first slices wait
// behind all of them; those of bwd_numden and bwd_dv: the same within 1 %.
__device__ __forceinline__ void prefetch_rows(const void* base, int64_t stride, int rows, int64_t bytes) {
  const int lines = (int)((bytes + 127) >> 7);
  for (int e = threadIdx.x; e < rows * lines; e += THREADS) {
    const int r = e / lines;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char*>(base) + r * stride + (int64_t)(e - r * lines) * 128));
  }
}

struct Block {
  uint8_t* sm;
  Misc* misc;
  int* status;
  uint32_t tmem, corr;                                // corr: first column of the small products' accumulator
  bool two;                                           // two main accumulators
  int nt, it;                                         // columns of the product; slices so far
  int warp, lane;

  // every thread of the block; `columns` a multiple of 16, at most 128; K: length of all segments together (where it
  // exceeds 128 there are two slices at least)
  __device__ __forceinline__ void begin(uint8_t* raw, int columns, int K, int* status_word) {
    sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
    misc = reinterpret_cast<Misc*>(sm + 2 * STAGE);
    status = status_word;
    nt = columns;
    two = columns <= (int)SECOND && K > 128;
    corr = two ? CORR2 : CORR;
    it = 0;
    warp = threadIdx.x >> 5;
    lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
      for (int i = 0; i < 2; i++) { tc::mbar_init(&misc->full[i], PRODUCERS / 32); tc::mbar_init(&misc->empty[i], 1); }
      tc::mbar_init(&misc->done, 1);
      misc->abort_flag = 0;
      tc::fence_barrier_init();
    }
    if (warp == 8) {
      tc::tmem_alloc(&misc->tmem_base, TMEM);
      tc::tmem_relinquish();
    }
    tc::tcgen05_fence_before();
    __syncthreads();
    tc::tcgen05_fence_after();
    tmem = misc->tmem_base;
  }

  // D += A B over k in [0, K).  AK / BK: that operand is K-major.  fa(row, k, piece) fills eight values of A: k .. k + 7
  // of one row (AK) or rows row .. row + 7 at one k; fb(column, k, piece) likewise.  Both are called with k < K only; K is
  // the same for all threads, and a multiple of 8 where an operand is K-major.
  template <bool AK, int AP, bool BK, int BP, class FA, class FB>
  __device__ __forceinline__ void segment(int K, FA fa, FB fb) {
    const int ns = (K + KS - 1) / KS;
    if (warp == 8) {
      const uint32_t idesc = tc::idesc_bf16(ROWS, nt, AK ? 0 : 1, BK ? 0 : 1);
      const uint32_t base = tc::smem_u32(sm);
      const uint64_t da = tc::smem_desc(base, AK ? 16 : 4096, AK ? 512 : 1024, AK ? 4 : tc::SWZ_128B);
      const uint64_t db = tc::smem_desc(base + 3 * PART, BK ? 16 : 4096, BK ? 512 : 1024, BK ? 4 : tc::SWZ_128B);
      constexpr uint32_t ka = AK ? 2 : 128, kb = BK ? 2 : 128, P = PART / 16;      // descriptor units (16 bytes)
      const uint32_t ah = (uint32_t)(da >> 32), bh = (uint32_t)(db >> 32);
      for (int s = 0; s < ns; s++, it++) {
        const int st = it & 1;
        if (!__all_sync(0xffffffffu, tc::mbar_wait(&misc->full[st], (it >> 1) & 1, &misc->abort_flag, status))) break;
        tc::tcgen05_fence_after();
        const int steps = K - s * KS > 16 ? 2 : 1;
        uint32_t al = (uint32_t)da + st * (STAGE / 16), bl = (uint32_t)db + st * (STAGE / 16);
        tc::opaque(al); tc::opaque(bl);
        if (lane == 0) {
#pragma unroll
          for (int k = 0; k < 2; k++) {
            if (k < steps) {
              const uint32_t a = al + k * ka, b = bl + k * kb, more = (it | k) ? 1u : 0u, small = tmem + corr;
              if (AP == 3) {
                tc::mma_bf16_lh(small, a + 2 * P, ah, b, bh, idesc, more);
                tc::mma_bf16_lh(small, a + P, ah, b, bh, idesc, 1u);
              }
              if (BP == 3) {
                tc::mma_bf16_lh(small, a, ah, b + 2 * P, bh, idesc, AP == 3 ? 1u : more);
                tc::mma_bf16_lh(small, a, ah, b + P, bh, idesc, 1u);
              }
              if (AP == 3 && BP == 3) tc::mma_bf16_lh(small, a + P, ah, b + P, bh, idesc, 1u);
              const bool other = two && (it & 1);
              tc::mma_bf16_lh(other ? tmem + SECOND : tmem, a, ah, b, bh, idesc, it > (two ? 1 : 0) || k > 0 ? 1u : 0u);
            }
          }
          tc::mma_commit(&misc->empty[st]);
        }
        __syncwarp();
      }
    } else {
      const int tid = threadIdx.x;
      // this thread's pieces: [2] of A, up to [2] of B
      int ar[2], akk[2], br[2], bkk[2];
      uint32_t ao[2], bo[2];
      bool bon[2];
      const int nch = nt >> 3;
#pragma unroll
      for (int u = 0; u < 2; u++) {
        const int i = tid + u * PRODUCERS;
        if (AK) { ar[u] = i >> 2; akk[u] = (i & 3) * 8; ao[u] = (i >> 2) * 64 + (((i & 3) ^ ((i >> 3) & 3)) << 4); }
        else { const int c = i & 15, k = i >> 4; ar[u] = c * 8; akk[u] = k; ao[u] = (c >> 3) * 4096 + k * 128 + (((c & 7) ^ (k & 7)) << 4); }
        if (BK) { br[u] = i >> 2; bkk[u] = (i & 3) * 8; bon[u] = br[u] < nt; bo[u] = (i >> 2) * 64 + (((i & 3) ^ ((i >> 3) & 3)) << 4); }
        else { const int c = i % nch, k = i / nch; br[u] = c * 8; bkk[u] = k; bon[u] = k < KS; bo[u] = (c >> 3) * 4096 + k * 128 + (((c & 7) ^ (k & 7)) << 4); }
      }
      Piece<AP> pa[2];
      Piece<BP> pb[2];
      auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
          if (k0 + akk[u] < K) fa(ar[u], k0 + akk[u], pa[u]); else pa[u].zero();
          if (bon[u] && k0 + bkk[u] < K) fb(br[u], k0 + bkk[u], pb[u]); else pb[u].zero();
        }
      };
      if (ns > 0) fetch(0);
      for (int s = 0; s < ns; s++, it++) {
        const int st = it & 1;
        // (a wait that runs out has latched its status: the thread goes on, so that the block still leaves together)
        tc::mbar_wait(&misc->empty[st], ((it >> 1) & 1) ^ 1, &misc->abort_flag, status);
        uint8_t* base = sm + st * STAGE;
#pragma unroll
        for (int u = 0; u < 2; u++) {
          pa[u].store(base + ao[u]);
          if (bon[u]) pb[u].store(base + 3 * PART + bo[u]);
        }
        tc::fence_proxy_async_smem();
        tc::mbar_arrive_warp(&misc->full[st], lane);
        if (s + 1 < ns) fetch((s + 1) * KS);
      }
    }
  }

  // After the last segment (at least one slice in all): waits for the products.
  __device__ __forceinline__ void finish() {
    if (warp == 8) {
      if (lane == 0) tc::mma_commit(&misc->done);
      __syncwarp();
    } else {
      tc::mbar_wait(&misc->done, 0, &misc->abort_flag, status);
      __syncwarp();
      tc::tcgen05_fence_after();
    }
  }

  // One column of the product; thread (warps 0-3) = row.
  __device__ __forceinline__ float column(int c) const {
    uint32_t a[8], b[8], d[8];
    const uint32_t at = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(c & ~7);
    tc::tmem_ld8(at, a);
    tc::tmem_ld8(at + corr, b);
    if (two) tc::tmem_ld8(at + SECOND, d);
    tc::tmem_wait_ld();
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < 8; j++)
      if (j == (c & 7)) v = __uint_as_float(a[j]) + (two ? __uint_as_float(b[j]) + __uint_as_float(d[j]) : __uint_as_float(b[j]));
    return v;
  }

  // Hands the product out in pieces of four columns, arranged so that a warp's global accesses coalesce:
  // emit(row, column, float4), every lane of a warp at the same time (eight lanes per row and 32 columns, or four lanes
  // per row where 16 columns are left).  Warps 0-7; the stages serve as a transposing buffer, one 4 KB piece per warp.
  template <class F>
  __device__ __forceinline__ void rows(F emit) {
    rows([](int, int) { return 0; }, [&](int r, int c, float4 v, int, int) { emit(r, c, v); });
  }
  // The same with something fetched for every piece: emit(row, column, float4, load(row, column), i).  The loads of eight pieces
  // are issued together, ahead of what emit does with them.  i: number of the row among the lane's eight (its row is
  // 32 (warp % 4) + 4 i + lane / 8), or -1 where 16 columns are left.
  template <class L, class F>
  __device__ __forceinline__ void rows(L load, F emit) {
    if (warp == 8) return;
    const int half = ((nt >> 1) + 15) & ~15;
    const int c1 = warp < 4 ? half : nt;
    const int row0 = (warp & 3) * 32;
    const uint32_t lanes = tmem + ((uint32_t)row0 << 16);
    float* buf = reinterpret_cast<float*>(sm + warp * 4096);          // [32][32], 16-byte pieces XORed with row % 8
    for (int c = warp < 4 ? 0 : half; c < c1; c += 32) {
      const int wide = c1 - c >= 32 ? 2 : 1;
#pragma unroll
      for (int q = 0; q < 2; q++) {
        if (q < wide) {
          uint32_t a[16], b[16];
          tc::tmem_ld16(lanes + c + q * 16, a);
          tc::tmem_ld16(lanes + corr + c + q * 16, b);
          tc::tmem_wait_ld();
          if (two) {
            uint32_t d[16];
            tc::tmem_ld16(lanes + SECOND + c + q * 16, d);
            tc::tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; j++) b[j] = __float_as_uint(__uint_as_float(b[j]) + __uint_as_float(d[j]));
          }
#pragma unroll
          for (int j = 0; j < 4; j++)
            *reinterpret_cast<float4*>(buf + lane * 32 + (((q * 4 + j) ^ (lane & 7)) << 2)) =
                make_float4(__uint_as_float(a[4 * j]) + __uint_as_float(b[4 * j]), __uint_as_float(a[4 * j + 1]) + __uint_as_float(b[4 * j + 1]),
                            __uint_as_float(a[4 * j + 2]) + __uint_as_float(b[4 * j + 2]), __uint_as_float(a[4 * j + 3]) + __uint_as_float(b[4 * j + 3]));
        }
      }
      __syncwarp();
      if (wide == 2) {
        float4 f[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
          const int r = i * 4 + (lane >> 3), cc = lane & 7;
          f[i] = *reinterpret_cast<const float4*>(buf + r * 32 + ((cc ^ (r & 7)) << 2));
        }
        decltype(load(0, 0)) g[8];
#pragma unroll
        for (int i = 0; i < 8; i++) g[i] = load(row0 + i * 4 + (lane >> 3), c + (lane & 7) * 4);
#pragma unroll
        for (int i = 0; i < 8; i++) emit(row0 + i * 4 + (lane >> 3), c + (lane & 7) * 4, f[i], g[i], i);
      } else {
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const int r = i * 8 + (lane >> 2), cc = lane & 3;
          emit(row0 + r, c + cc * 4, *reinterpret_cast<const float4*>(buf + r * 32 + ((cc ^ (r & 7)) << 2)),
               load(row0 + r, c + cc * 4), -1);
        }
      }
      __syncwarp();
    }
  }

  // Sums over the columns that the callers of rows() kept per lane (wide pieces): sum[i] is added to out[row] for the lane's rows.
  __device__ __forceinline__ void add_row_sums(const float (&sum)[8], float* out) const {
    if (warp == 8) return;
#pragma unroll
    for (int i = 0; i < 8; i++) {
      float s = sum[i];
#pragma unroll
      for (int o = 1; o < 8; o *= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
      if ((lane & 7) == 0) atomicAdd(&out[(warp & 3) * 32 + i * 4 + (lane >> 3)], s);
    }
  }

  __device__ __forceinline__ void end() {
    tc::tcgen05_fence_before();
    __syncthreads();
    if (warp == 8) {
      tc::tcgen05_fence_after();
      tc::tmem_dealloc(tmem, TMEM);
    }
  }
};

// Host side: a launch with the stages' shared memory, timed and checked like every other.
template <typename... KArgs, typename... Args>
inline int launch(fsharp_ctx* ctx, int tag, void (*kernel)(KArgs...), dim3 grid, Args... args) {
  FS_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM));
  FS_TIME_BEGIN(ctx, tag);
  (void)fs_launch_chained(kernel, grid, dim3(THREADS), SMEM, ctx->stream, args...);
  FS_TIME_END(ctx);
  FS_LAUNCH_CHECK(ctx);
  return FSHARP_OK;
}

}  // namespace mma3
