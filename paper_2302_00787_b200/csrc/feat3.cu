// Features at fp32 precision (Section 4 definition with Section 2.1's M^-1/2) on the tensor cores, for every shape and both
// types: phi = exp(e - shift), e_im = bias + a_m + w_m . x_i + c_i, c_i = x_i^T C x_i.
//
// The fp32 operands enter the MMAs as three bf16 parts (split3.cuh); bf16 tokens are exact.  The feature matrix is written
// once: the row shift is found in tensor memory before the exponentials, the group shift by a pass of the same products
// that writes nothing (the products of a tile cost a quarter of what its 128 x 256 features cost in HBM time).  The kernels
// they replace (fp32 multiply-adds; exponents written, read for the maximum, read and written again as features) took
// 441 + 98 + 38 us for 2 x 160 k tokens, d = 64, M = 256, and 360 us for the dense quadratic terms.
#include <math.h>

#include "feat3.cuh"
#include "split3.cuh"
#include "tc_layout.cuh"

using namespace tc;
using namespace tcl;
using feat3::Task;

namespace tchost {
int make_map_tokens(CUtensorMap* map, const void* base, TensorAddr a, int B, int H, int L, int inner);
int make_map_features(CUtensorMap* map, void* base, int BH, int L, int M, int bf16, int box_bytes);
}

namespace {

__device__ __forceinline__ int group_of(int bh, int H, int pool) { return pool == FSHARP_POOL_PER_BH ? bh : bh % H; }

// Order-preserving map float -> unsigned, so that atomicMax on words gives the float maximum (0 lies below every float).
__device__ __forceinline__ unsigned f2ord(float f) {
  unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(unsigned u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Float maximum by integer atomics (start value -inf; bit patterns of non-negative floats ascend, of negative ones descend).
__device__ __forceinline__ void atomic_max_float(float* p, float v) {
  v += 0.f;                                        // -0 -> +0
  if (v >= 0.f) atomicMax(reinterpret_cast<int*>(p), __float_as_int(v));
  else atomicMin(reinterpret_cast<unsigned*>(p), __float_as_uint(v));
}

// 2^x with subnormal results
__device__ __forceinline__ float ex2_full(float x) {
  float y;
  asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 32 bytes (eight words) as one store; p is 32-byte aligned
__device__ __forceinline__ void store32(float* p, const uint32_t* x) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]),
               "r"(x[5]), "r"(x[6]), "r"(x[7])
               : "memory");
}

// A factor as a float and its remainder: fmaf(hi, x, lo * x) is the product with the unrounded factor, rounded once.  (The same
// factor multiplies every exponent: rounded to fp32 it moves exponents of 60 nats by 2e-6, all of them in one direction.)
struct Factor {
  float hi, lo;
  __host__ __device__ explicit constexpr Factor(double f = 0.0) : hi((float)f), lo((float)(f - (double)(float)f)) {}
  __device__ __forceinline__ float times(float x) const { return fmaf(hi, x, lo * x); }
};
constexpr double LOG2E = 1.4426950408889634074;
// The accumulator is cut off after every MMA, never rounded up: over the d / 16 steps of the large products a sum that grows
// from 0 loses on average LOST_W units of 2^-23 of itself, and what it starts with (a_m) LOST_A units.  Measured by regression
// of the exponents' errors on w . x and a_m: 0.34, 0.37, 0.51, 0.85 units at d = 16, 32, 64, 128 for the sum.  W and a are scaled up
// by as much, so that the errors centre on zero.
template <int D> constexpr double LOST_W = (0.17 + 0.085 * (D / 16)) / 8388608.0;
template <int D> constexpr double LOST_A = 0.17 * (D / 16) / 8388608.0;
#define FS_TO_LOG2(x) fmaf(1.44269502f, (x), 1.92596299e-8f * (x))      // x log2(e)

struct Args {
  CUtensorMap map[2];     // per task: the tokens (BP = 2)
  CUtensorMap out[2];     // per task: the features, where staged[i]
  bool staged[2];
  Task t[2];
  int first[3];           // running number of work items: task i owns [first[i], first[i + 1])
  int tiles[2];           // token tiles per (batch, head)
  int H, M, pool, nmb;
  const float* prep;
  const uint8_t* img[2];  // per task: operand images of W (nullptr: blocks build them from prep)
  Factor wscale;          // log2e qk_scale (1 + LOST_W)
  float pow2;             // power of two next to qk_scale: tokens times this do not overflow when squared
  double quad;            // log2e (qk_scale / pow2)^2
  bool own_terms;         // the feature kernels compute the quadratic terms of groups with C = gamma I themselves
  bool row_init;          // a pass raises logscale from -inf
  float4* zero;           // cleared by the kernel of the quadratic terms
  size_t zero4;
  int* status;
};

// Eight values of a token row as the parts of an MMA operand (16-byte pieces `part` bytes apart).
__device__ __forceinline__ void put8(uint8_t* dst, uint32_t part, const float* p, bool in) {
  float v[8] = {};
  if (in) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
  uint4 h, m, l;
  split3::split8(v, h, m, l);
  *reinterpret_cast<uint4*>(dst) = h;
  *reinterpret_cast<uint4*>(dst + part) = m;
  *reinterpret_cast<uint4*>(dst + 2 * part) = l;
}

template <typename T, int D> struct Geo {
  static constexpr int NKS = (D + 63) / 64;                  // slices of 64 values of K
  static constexpr int KSTEPS = D < 64 ? D / 16 : 4;         // MMA steps per slice
  static constexpr int CH = D < 64 ? D / 8 : 8;              // 16-byte pieces of a row and slice
  static constexpr int AP = sizeof(T) == 2 ? 1 : 3;          // parts of a token
  static constexpr uint32_t A_BYTES = NKS * AP * TILE_BYTES; // [slice][part][128 rows x 128 bytes]
};

// Token tile -> operand parts, thread i of N; consecutive lanes take one row's pieces.  The global loads are a step of
// their own, so that they can be in flight while the buffer is still being read.
template <typename T, int D, int N> struct Stage {
  using G = Geo<T, D>;
  static constexpr int PER_ROW = G::NKS * G::CH, COUNT = TILE * PER_ROW / N;
  static constexpr int BATCH = COUNT < 8 ? COUNT : 8;           // pieces in flight per thread
  uint4 r[BATCH][sizeof(T) == 2 ? 1 : 2];
  __device__ __forceinline__ void load(const T* X, int64_t sl, int rows, int i, int batch) {
#pragma unroll
    for (int u = 0; u < BATCH; u++) {
      const int e = i + (batch * BATCH + u) * N, row = e / PER_ROW, c = e % PER_ROW;
      const uint4* src = reinterpret_cast<const uint4*>(X + (int64_t)row * sl + 8 * c);
      const bool in = row < rows;
      r[u][0] = in ? src[0] : make_uint4(0, 0, 0, 0);
      if (sizeof(T) == 4) r[u][sizeof(T) == 4 ? 1 : 0] = in ? src[1] : make_uint4(0, 0, 0, 0);
    }
  }
  __device__ __forceinline__ void store(uint8_t* sA, int i, int batch) const {
#pragma unroll
    for (int u = 0; u < BATCH; u++) {
      const int e = i + (batch * BATCH + u) * N, row = e / PER_ROW, c = e % PER_ROW, s = c / 8, cc = c % 8;
      uint8_t* dst = sA + s * (G::AP * TILE_BYTES) + row * 128 + ((cc ^ (row & 7)) << 4);
      if (sizeof(T) == 2) {
        *reinterpret_cast<uint4*>(dst) = r[u][0];
      } else {
        const uint4 a = r[u][0], b = r[u][sizeof(T) == 4 ? 1 : 0];
        const float v[8] = {__uint_as_float(a.x), __uint_as_float(a.y), __uint_as_float(a.z), __uint_as_float(a.w),
                            __uint_as_float(b.x), __uint_as_float(b.y), __uint_as_float(b.z), __uint_as_float(b.w)};
        uint4 h, m, l;
        split3::split8(v, h, m, l);
        *reinterpret_cast<uint4*>(dst) = h;
        *reinterpret_cast<uint4*>(dst + TILE_BYTES) = m;
        *reinterpret_cast<uint4*>(dst + 2 * TILE_BYTES) = l;
      }
    }
  }
  // all pieces of a tile but those of batch 0, which `load` has fetched ahead
  __device__ __forceinline__ void finish(uint8_t* sA, const T* X, int64_t sl, int rows, int i) {
    store(sA, i, 0);
#pragma unroll
    for (int b = 1; b < COUNT / BATCH; b++) {
      load(X, sl, rows, i, b);
      store(sA, i, b);
    }
  }
};

// Feature blocks of M (all of M when it fits: a row's largest exponent is then known inside the block) and their images:
// [block][slice][BP parts][rows of 128 bytes, 128-byte swizzle], already scaled by log2e qk_scale.
// BP = 2 (16 significant bits of W) goes with features that are rounded to bf16.
template <int D, int BP> struct WGeo {
  static constexpr int NKS = (D + 63) / 64, MB = D == 128 && BP == 3 ? 128 : 256;
};
template <int D, int BP>
__device__ __forceinline__ void put_w(uint8_t* img, int mb, int f, int c, const float* w, Factor scale, bool& bad) {
  float v[8];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    v[j] = scale.times(w[j]);
    bad |= !isfinite(v[j]);
  }
  uint4 h, m, l;
  split3::split8(v, h, m, l);
  uint8_t* dst = img + (c / 8) * (BP * mb * 128) + f * 128 + (((c % 8) ^ (f & 7)) << 4);
  *reinterpret_cast<uint4*>(dst) = h;
  *reinterpret_cast<uint4*>(dst + mb * 128) = m;
  if (BP == 3) *reinterpret_cast<uint4*>(dst + 2 * mb * 128) = l;
}
template <int D, int BP>
__global__ void __launch_bounds__(256)
w3_images_kernel(const float* __restrict__ prep, int side0, int sides, int M, Factor scale, uint8_t* __restrict__ img,
                 int* __restrict__ status) {
  fs_grid_dependency_wait();
  using G = WGeo<D, BP>;
  const int g = blockIdx.y, k = blockIdx.z;                          // group; which of the `sides` sides
  const size_t per_group = (size_t)G::NKS * BP * M * 128;
  const float* W = prep + ((size_t)g * 2 + (side0 - 1 + k)) * PrepLayout{D, M}.total();
  uint8_t* out = img + ((size_t)k * gridDim.y + g) * per_group;
  bool bad = false;
  for (int e = blockIdx.x * 256 + threadIdx.x; e < M * (D / 8); e += gridDim.x * 256) {
    const int m = e / (D / 8), c = e % (D / 8), blk = m / G::MB, mb = min(G::MB, M - blk * G::MB);
    put_w<D, BP>(out + (size_t)blk * G::MB * (G::NKS * BP * 128), mb, m - blk * G::MB, c, W + (size_t)m * D + 8 * c, scale, bad);
  }
  if (bad) atomicExch(status, FSHARP_E_NONFINITE);
}

// acc[128 x N] = A B^T with A = staged tokens, B = [slice][BP parts][N rows x 128 bytes], by one lane: the products with m or l
// parts (those of the first USE parts of B) first, h h last (the accumulator is truncated at every step; see tc_pairs.cu).
// sOne / sRow (may be null): one more step of K = 16 with operands [128 x 16] and [N x 16] in core matrices, for a term per column.
template <typename T, int D, int BP = 3, int USE = BP>
__device__ __forceinline__ void issue_products(uint32_t acc, const uint8_t* sA, const uint8_t* sB, int N, const uint8_t* sOne = nullptr,
                                               const uint8_t* sRow = nullptr) {
  using G = Geo<T, D>;
  const uint32_t idesc = idesc_bf16(128, N, 0, 0);
  const uint64_t da = smem_desc(smem_u32(sA), 16, 1024, SWZ_128B), db = smem_desc(smem_u32(sB), 16, 1024, SWZ_128B);
  const uint32_t ah = (uint32_t)(da >> 32), bh = (uint32_t)(db >> 32), P = TILE_BYTES / 16, Q = (uint32_t)N * 8;
#pragma unroll
  for (int s = 0; s < (USE > 1 ? G::NKS : 0); s++) {
    const uint32_t a0 = (uint32_t)da + s * G::AP * P, b0 = (uint32_t)db + s * BP * Q;
#pragma unroll
    for (int k = 0; k < G::KSTEPS; k++) {
      const uint32_t a = a0 + 2 * k, b = b0 + 2 * k;
      if (USE == 3) mma_bf16_lh(acc, a, ah, b + 2 * Q, bh, idesc, (s | k) ? 1u : 0u);
      if (G::AP == 3) {
        mma_bf16_lh(acc, a + 2 * P, ah, b, bh, idesc, 1u);
        mma_bf16_lh(acc, a + P, ah, b + Q, bh, idesc, 1u);
        mma_bf16_lh(acc, a + P, ah, b, bh, idesc, 1u);
      }
      mma_bf16_lh(acc, a, ah, b + Q, bh, idesc, USE == 3 || (s | k) ? 1u : 0u);
    }
  }
  if (sOne != nullptr)
    mma_bf16(acc, smem_desc(smem_u32(sOne), 128, 256, SWZ_NONE), smem_desc(smem_u32(sRow), 128, 256, SWZ_NONE), idesc, USE > 1 ? 1u : 0u);
#pragma unroll
  for (int s = 0; s < G::NKS; s++)
#pragma unroll
    for (int k = 0; k < G::KSTEPS; k++)
      mma_bf16_lh(acc, (uint32_t)da + s * G::AP * P + 2 * k, ah, (uint32_t)db + s * BP * Q + 2 * k, bh, idesc, 1u);
}

// ---- c_i = x_i^T C x_i; also clears the maxima that later passes raise ------------------------
// Block = 128 tokens at a time: T = X C on the tensor cores, c_i = t_i . x_i; C = gamma I needs no product.
constexpr int RT_THREADS = 256;
struct RtMisc {
  uint64_t done;
  uint32_t tmem_base;
  int abort_flag;
  float part[2][TILE];
};
template <typename T, int D> constexpr size_t rt_smem() { return 1024 + Geo<T, D>::A_BYTES + Geo<T, D>::NKS * 3 * D * 128 + sizeof(RtMisc); }

template <typename T, int D>
__global__ void __launch_bounds__(RT_THREADS, D == 128 ? 1 : 3)
rowterm3_kernel(const __grid_constant__ Args a) {
  fs_grid_dependency_wait();
  using G = Geo<T, D>;
  using St = Stage<T, D, RT_THREADS>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sA = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sC = sA + G::A_BYTES;
  RtMisc* misc = reinterpret_cast<RtMisc*>(sC + G::NKS * 3 * D * 128);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr uint32_t COLS = D < 32 ? 32 : D;
  PrepLayout pr{D, a.M};
  const int total = a.first[2];
  const int w0 = (int)((int64_t)total * blockIdx.x / gridDim.x), w1 = (int)((int64_t)total * (blockIdx.x + 1) / gridDim.x);
  for (size_t i = blockIdx.x * (size_t)RT_THREADS + tid; i < a.zero4; i += (size_t)gridDim.x * RT_THREADS) a.zero[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (a.own_terms) {
    // nothing but the start values where all groups of this block have C = gamma I
    bool all = true;
    for (int w = w0; w < w1;) {
      const int ti = w >= a.first[1] ? 1 : 0, bh = (w - a.first[ti]) / a.tiles[ti], tile = (w - a.first[ti]) % a.tiles[ti];
      const Task& t = a.t[ti];
      all &= a.prep[((size_t)group_of(bh, a.H, a.pool) * 2 + (t.side - 1)) * pr.total() + pr.scal() + PS_CSCALAR] != 0.f;
      if (tile == 0 && tid == 0 && t.gmax) t.gmax[bh] = 0u;
      if (t.stab == FSHARP_STAB_ROW && a.row_init) {
        const int i1 = min(t.L, (tile + min(a.tiles[ti] - tile, w1 - w)) * TILE);
        for (int i = tile * TILE + tid; i < i1; i += RT_THREADS) t.logscale[(int64_t)bh * t.L + i] = __int_as_float(0xff800000);
      }
      w += a.tiles[ti] - tile;
    }
    if (all) return;
  }
  if (tid == 0) {
    mbar_init(&misc->done, 1);
    misc->abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc(&misc->tmem_base, COLS);
    tmem_relinquish();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = misc->tmem_base;
  int have = -1, phase = 0;                       // (task, group) whose C is staged
  bool scalar = false, bad = false;
  Factor quad;
  St st;
  auto tokens = [&](int w, int& rows, int64_t& sl) {
    const int ti = w >= a.first[1] ? 1 : 0;
    const Task& t = a.t[ti];
    const int bh = (w - a.first[ti]) / a.tiles[ti], tile = (w - a.first[ti]) % a.tiles[ti];
    rows = t.L - tile * TILE;
    sl = t.ax.sl;
    return reinterpret_cast<const T*>(t.X) + (bh / a.H) * t.ax.sb + (bh % a.H) * t.ax.sh + (int64_t)tile * TILE * sl;
  };
  int rows = 0;
  int64_t sl = 0;
  const T* X = nullptr;
  if (w0 < w1) {
    X = tokens(w0, rows, sl);
    st.load(X, sl, rows, tid, 0);
  }
  for (int w = w0; w < w1; w++) {
    const int ti = w >= a.first[1] ? 1 : 0;
    const Task& t = a.t[ti];
    const int bh = (w - a.first[ti]) / a.tiles[ti], tile = (w - a.first[ti]) % a.tiles[ti];
    const int g = group_of(bh, a.H, a.pool), key = ti * 65536 + g;
    if (key != have) {
      have = key;
      const float* pp = a.prep + ((size_t)g * 2 + (t.side - 1)) * pr.total();
      scalar = pp[pr.scal() + PS_CSCALAR] != 0.f;
      quad = Factor(scalar ? a.quad * (double)pp[pr.scal() + PS_CGAMMA] : a.quad);
      if (!scalar) {
        // row j of the operand: column j of C, its index i contiguous (the same matrix in the quadratic form: row j of C)
        const float* Cm = pp + pr.Cmat();
        for (int e = tid; e < D * G::NKS * G::CH; e += RT_THREADS) {
          const int j = e / (G::NKS * G::CH), c = e % (G::NKS * G::CH), s = c / 8, cc = c % 8;
          put8(sC + s * (3 * D * 128) + j * 128 + ((cc ^ (j & 7)) << 4), D * 128, Cm + j * D + 8 * c, true);
        }
      }
    }
    const int64_t out0 = (int64_t)bh * t.L + (int64_t)tile * TILE;
    const int row = tid & 127, half = tid >> 7;
    const int valid = rows;
    st.finish(sA, X, sl, rows, tid);
    if (w + 1 < w1) {                             // the next tile's loads fly under this tile's product
      X = tokens(w + 1, rows, sl);
      st.load(X, sl, rows, tid, 0);
    }
    if (!scalar) {
      fence_proxy_async_smem();
      __syncthreads();
      if (warp == 0) {
        tcgen05_fence_after();
        if (lane == 0) {
          issue_products<T, D>(tmem, sA, sC, D);
          mma_commit(&misc->done);
        }
        __syncwarp();
      }
      mbar_wait(&misc->done, phase & 1, &misc->abort_flag, a.status, false);
      phase++;
      __syncwarp();
      tcgen05_fence_after();
    } else {
      __syncthreads();
    }
    // x from its parts (the row's pieces are conflict-free to read), half of the columns per warpgroup
    float sum[4] = {};
    const uint32_t lanes = tmem + ((uint32_t)(row & ~31) << 16);
#pragma unroll
    for (int c = 0; c < D / 16; c++) {
      const int c8 = half * (D / 16) + c, s = c8 / 8, cc = c8 % 8;            // eight columns
      const uint8_t* src = sA + s * (G::AP * TILE_BYTES) + row * 128 + ((cc ^ (row & 7)) << 4);
      float x[8];
#pragma unroll
      for (int p = 0; p < G::AP; p++) {
        const uint4 q = *reinterpret_cast<const uint4*>(src + p * TILE_BYTES);
        const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const float lo = __uint_as_float(u[j] << 16), hi = __uint_as_float(u[j] & 0xffff0000u);
          x[2 * j] = p ? x[2 * j] + lo : lo;
          x[2 * j + 1] = p ? x[2 * j + 1] + hi : hi;
        }
      }
#pragma unroll
      for (int j = 0; j < 8; j++) x[j] *= a.pow2;
      if (scalar) {
#pragma unroll
        for (int j = 0; j < 8; j++) sum[j & 3] = fmaf(x[j], x[j], sum[j & 3]);
      } else {
        uint32_t tv[8];
        tmem_ld8(lanes + c8 * 8, tv);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; j++) sum[j & 3] = fmaf(a.pow2 * __uint_as_float(tv[j]), x[j], sum[j & 3]);
      }
    }
    if (!scalar) tcgen05_fence_before();
    misc->part[half][row] = (sum[0] + sum[1]) + (sum[2] + sum[3]);
    __syncthreads();
    if (half == 0 && row < valid) {
      const float c = quad.times(misc->part[0][row] + misc->part[1][row]);
      bad |= !isfinite(c);                        // so is x then (or C): one test per token instead of one per exponent
      t.rowc[out0 + row] = c;
      if (t.stab == FSHARP_STAB_ROW && a.row_init) t.logscale[out0 + row] = __int_as_float(0xff800000);
    }
    if (tile == 0 && tid == 0 && t.gmax) t.gmax[bh] = 0u;
    // (the next tile's staging overwrites sA: its readers are behind the barrier above)
  }
  if (bad) atomicExch(a.status, FSHARP_E_NONFINITE);
  tcgen05_fence_before();
  __syncthreads();
  if (warp == 0) {
    tcgen05_fence_after();
    tmem_dealloc(tmem, COLS);
  }
}

// ---- the exponents' maxima (WRITE = false), the features (WRITE = true) -------------------------
// Persistent blocks, one per SM; a block owns a range of (task, (batch, head), feature block, token tile) and fetches the
// parts of W = Omega B when the group changes.  Everything is in powers of two (W, a, c and the bias carry log2e), so a
// feature is one ex2 of one addition: the per-feature term a_m rides on the products as one more K step (its three parts
// against ones).  Warps 8-11 stage token tiles, warp 12 issues the products, the two warpgroups of warps 0-7 take one
// accumulator each and work on alternate tiles: thread = token, all columns of a row in one thread, so the row's maximum
// needs no exchange.  A warp's rows go through shared memory and leave as copies of whole lines (32 rows of 128 bytes; 64 where d = 128
// leaves little room).  Bound of the writing pass: HBM (128 KB per tile of 128 x 256: 6.5 k cycles of this SM's share of the rate of writes)
// against 3.4 k cycles of products;
// 2 x 8 x 10007 fp32 tokens, d = 64, M = 256, both sides: 217.6 us with each lane storing its own row in 32-byte pieces (a store instruction
// then touches 32 lines: 3.5 TB/s at best, whole lines 5.7), 212 us so.  Measured inside: 12 k cycles per tile, the two warpgroups' stores
// taking turns at some 15 bytes per cycle, and 3.5 k of each 23 k waiting for the next tile's products.
constexpr int FT_AHEAD = 4;                                        // tiles pulled into L2 ahead of the two buffers (BP = 2)
constexpr int FT_STAGE0 = 8, FT_MMA = 12, FT_THREADS = 416;
struct FtMisc {
  uint64_t a_full[2], a_free[2], t_full[2], t_free[2], max_full[2][2], w_full;
  uint32_t tmem_base;
  int abort_flag;
};
struct FtMax {
  float row[2][2][TILE];      // PAIR: the other block's maxima, two places (and barriers) per warpgroup
  float term[2][TILE];        // x^T C x of the warpgroups' tiles
};
template <typename T, int D, int BP, bool WRITE> struct FtGeo : Geo<T, D> {
  static_assert(BP == 3 || Geo<T, D>::AP == 1, "two parts of W: bf16 tokens");
  static constexpr int MB = WGeo<D, BP>::MB;
  static constexpr bool SMALL = D == 128;                              // little room beside W and the tokens
  // token tiles in shared memory (one where fp32 tokens leave room for no second one beside the staged features: their conversion and
  // the products, 1.5 k + 3.2 k cycles, stay below what the stores of a tile take)
  static constexpr int NBUF = sizeof(T) == 4 && (D == 128 || WRITE) ? 1 : 2;
  static constexpr uint32_t STAGE = SMALL ? 2048 : 4096;               // per warp: 32 rows of features, STAGE / 32 bytes each
  static constexpr int NSTAGE = SMALL ? 1 : 2;
  static constexpr uint32_t W_BYTES = Geo<T, D>::NKS * BP * MB * 128;
  static constexpr uint32_t OFF_A = W_BYTES, OFF_OUT = OFF_A + NBUF * Geo<T, D>::A_BYTES, OFF_ONE = OFF_OUT + (WRITE ? 8 * NSTAGE * STAGE : 0),
                            OFF_ROW = OFF_ONE + TILE * 32, OFF_MISC = OFF_ROW + MB * 32;
  static constexpr uint32_t OFF_MAX = OFF_MISC + sizeof(FtMisc);
  static constexpr size_t SMEM = 1024 + OFF_MAX + (BP == 2 ? sizeof(FtMax) : 0);
  static_assert(SMEM <= 232448, "shared memory budget");
};

// BP = 2: bf16 features of the chain of d = 128 kernels.  A row's shift is its largest exponent, so that its largest feature, which
// counts most, is a power of two and loses nothing to bf16 (with a maximum from the leading part of W, half the products, the
// outputs' error rose from 2.83e-3 to 2.88e-3; the pass for it took 80 us of 3435 for 1 x 16 x 65536 tokens, M = 512).  The shift of a group may be any value near
// its maximum (it cancels in the normalisation, and bf16 has the range of fp32): that pass takes the leading part of W alone.
// PAIR: row shifts where M takes two blocks of features: two blocks of a cluster walk the same tiles, one half of the features each, and
// tell each other their rows' maxima through shared memory.  (A pass of its own for the maxima, 200 us for 1 x 16 x 65536 tokens and
// M = 512, made all the products of the pass that writes; that pass takes 430 us as pairs, 380 with the shifts given.)
// BP = 2, C = gamma I: the first pass over the tokens takes x^T C x from the tile in shared memory, in the order of
// rowterm3_kernel (which read all tokens once more for it: 85 us for the same tokens).
template <typename T, int D, bool WRITE, int BP, bool PAIR = false>
__global__ void __launch_bounds__(FT_THREADS, 1)
feat3_kernel(const __grid_constant__ Args a) {
  fs_grid_dependency_wait();
  using G = FtGeo<T, D, BP, WRITE>;
  constexpr bool OUT16 = BP == 2;
  static_assert(!PAIR || (WRITE && OUT16), "pairs write bf16 features");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sW = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = sW + G::OFF_A;
  uint8_t* sOne = sW + G::OFF_ONE;
  uint8_t* sRow = sW + G::OFF_ROW;
  FtMisc* misc = reinterpret_cast<FtMisc*>(sW + G::OFF_MISC);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = PAIR ? (int)cluster_rank() : 0;
  // the first pass over the tokens: its epilogue warps read them too
  const bool terms = OUT16 && (!WRITE || PAIR || (a.t[0].stab == FSHARP_STAB_ROW && a.nmb == 1));
  if (tid == 0) {
    for (int i = 0; i < 2; i++) {
      mbar_init(&misc->a_full[i], OUT16 ? 1 : 4);
      mbar_init(&misc->a_free[i], terms ? 5 : 1);
      if (PAIR) {
        mbar_init(&misc->max_full[i][0], 4);
        mbar_init(&misc->max_full[i][1], 4);
      }
      mbar_init(&misc->t_full[i], 1);
      mbar_init(&misc->t_free[i], 4);
    }
    mbar_init(&misc->w_full, 1);
    misc->abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == FT_MMA) {
    tmem_alloc(&misc->tmem_base, 512);
    tmem_relinquish();
  }
  for (int e = tid; e < (TILE + G::MB) * 8; e += FT_THREADS) reinterpret_cast<uint32_t*>(sOne)[e] = 0u;
  __syncthreads();
  if (tid < TILE) {                                                // [1, 1, 1, 0, ...]
    *reinterpret_cast<uint2*>(sOne + core16_offset(tid, 0)) = make_uint2(0x3f803f80u, 0x00003f80u);
  }
  tcgen05_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();                                        // the other block's barriers are initialised
  tcgen05_fence_after();
  const uint32_t tmem = misc->tmem_base;
  FtMax* maxima = reinterpret_cast<FtMax*>(sW + G::OFF_MAX);
  PrepLayout pr{D, a.M};
  const int total = a.first[2], me = PAIR ? (int)blockIdx.x >> 1 : (int)blockIdx.x, blocks = PAIR ? (int)gridDim.x >> 1 : (int)gridDim.x;
  const int w1 = (int)((int64_t)total * (me + 1) / blocks);
  int w = (int)((int64_t)total * me / blocks);
  int copies = 0;
  int n = 0, runs = 0;                                             // tiles and runs done by this block (every role counts alike)
  bool bad = false;
  while (w < w1) {
    // a run: consecutive tiles of one (task, (batch, head), feature block)
    const int ti = w >= a.first[1] ? 1 : 0;
    const Task& t = a.t[ti];
    const int u = (w - a.first[ti]) / a.tiles[ti], tile0 = (w - a.first[ti]) % a.tiles[ti];
    const int bh = PAIR ? u : u / a.nmb, mblk = PAIR ? rank : u % a.nmb, m0 = mblk * G::MB, mb = min(G::MB, a.M - m0);
    const int ntiles = min(a.tiles[ti] - tile0, w1 - w);
    w += ntiles;
    const int g = group_of(bh, a.H, a.pool);
    const float* pp = a.prep + ((size_t)g * 2 + (t.side - 1)) * pr.total();
    const float bias = FS_TO_LOG2(pp[pr.scal() + PS_BIAS]);
    __syncthreads();                                               // the previous run's products have been read
    if (a.img[ti] != nullptr) {
      if (tid == 0) {
        const uint32_t bytes = (uint32_t)mb * (G::NKS * BP * 128);
        mbar_expect_tx(&misc->w_full, bytes);
        bulk_load(sW, a.img[ti] + ((size_t)g * a.M + m0) * (G::NKS * BP * 128), bytes, &misc->w_full);
      }
    } else {
      const float* W = pp + pr.W() + (size_t)m0 * D;
      for (int e = tid; e < mb * (D / 8); e += FT_THREADS)
        put_w<D, BP>(sW, mb, e / (D / 8), e % (D / 8), W + (size_t)e * 8, a.wscale, bad);
    }
    for (int e = tid; e < mb; e += FT_THREADS) {
      const float v = Factor(LOG2E * (1.0 + LOST_A<D>)).times(pp[pr.a() + m0 + e]);
      bad |= !isfinite(v);
      uint32_t h, m, l;
      split3::split_pair(v, 0.f, h, m, l);
      *reinterpret_cast<uint2*>(sRow + core16_offset(e, 0)) = make_uint2((h & 0xffffu) | (m << 16), l & 0xffffu);
    }
    bad |= !isfinite(bias);
    fence_proxy_async_smem();
    __syncthreads();
    if (OUT16 && warp >= FT_STAGE0 && warp < FT_MMA) {
      // the tokens are operands as they are: one lane has them copied, panel by panel.  (Through registers, half of a tile's
      // loads ahead, a tile of the maxima pass took 3.3 k cycles for 1.2 k of products.)
      if (warp == FT_STAGE0 && lane == 0) {
        const int b4 = bh / a.H, h4 = bh - b4 * a.H;
        for (int it = 0; it < ntiles; it++) {
          const int k = n + it, b = k % G::NBUF, tok = (tile0 + it) * TILE;
          mbar_wait(&misc->a_free[b], ((k / G::NBUF) & 1) ^ 1, &misc->abort_flag, a.status);
          mbar_expect_tx(&misc->a_full[b], G::A_BYTES);
#pragma unroll
          for (int s = 0; s < G::NKS; s++) tma_load_4d(sA + b * G::A_BYTES + s * TILE_BYTES, &a.map[ti], &misc->a_full[b], 64 * s, tok, h4, b4);
          if (it + FT_AHEAD < ntiles) {
#pragma unroll
            for (int s = 0; s < G::NKS; s++) tma_prefetch_4d(&a.map[ti], 64 * s, tok + FT_AHEAD * TILE, h4, b4);
          }
        }
      }
      __syncwarp();
      n += ntiles;
    } else if (warp >= FT_STAGE0 && warp < FT_MMA) {
      const T* X = reinterpret_cast<const T*>(t.X) + (bh / a.H) * t.ax.sb + (bh % a.H) * t.ax.sh;
      const int i = tid - FT_STAGE0 * 32;
      Stage<T, D, 128> st;
      st.load(X + (int64_t)tile0 * TILE * t.ax.sl, t.ax.sl, t.L - tile0 * TILE, i, 0);
      for (int it = 0; it < ntiles; it++, n++) {
        const int b = n % G::NBUF, tok = (tile0 + it) * TILE;
        mbar_wait(&misc->a_free[b], ((n / G::NBUF) & 1) ^ 1, &misc->abort_flag, a.status);
        st.finish(sA + b * G::A_BYTES, X + (int64_t)tok * t.ax.sl, t.ax.sl, t.L - tok, i);
        fence_proxy_async_smem();
        mbar_arrive_warp(&misc->a_full[b], lane);
        if (it + 1 < ntiles) st.load(X + (int64_t)(tok + TILE) * t.ax.sl, t.ax.sl, t.L - tok - TILE, i, 0);
      }
    } else if (warp == FT_MMA) {
      if (a.img[ti] != nullptr) mbar_wait(&misc->w_full, runs & 1, &misc->abort_flag, a.status, false);
      for (int it = 0; it < ntiles; it++, n++) {
        const int b = n & 1, ab = n % G::NBUF;
        mbar_wait(&misc->a_full[ab], (n / G::NBUF) & 1, &misc->abort_flag, a.status);
        mbar_wait(&misc->t_free[b], ((n >> 1) & 1) ^ 1, &misc->abort_flag, a.status);
        __syncwarp();
        tcgen05_fence_after();
        if (elect_one()) {
          if (OUT16 && !WRITE && t.stab == FSHARP_STAB_GROUP) issue_products<T, D, BP, 1>(tmem + b * 256, sA + ab * G::A_BYTES, sW, mb, sOne, sRow);
          else issue_products<T, D, BP>(tmem + b * 256, sA + ab * G::A_BYTES, sW, mb, sOne, sRow);
          mma_commit(&misc->t_full[b]);
          mma_commit(&misc->a_free[ab]);
        }
        __syncwarp();
      }
    } else {
      const int wg = warp >> 2;
      float gmx = -3.0e38f;
      const float gshift = (WRITE && t.stab == FSHARP_STAB_GROUP) ? ord2f(t.gmax[bh]) : 0.f;
      const bool own = PAIR || (t.stab == FSHARP_STAB_ROW && a.nmb == 1);
      const bool wide = WRITE && !OUT16 && (reinterpret_cast<uintptr_t>(t.phi) & 31) == 0;
      const bool scalar = terms && pp[pr.scal() + PS_CSCALAR] != 0.f;
      const Factor quad(scalar ? a.quad * (double)pp[pr.scal() + PS_CGAMMA] : 0.0);
      // 32 rows of ROW_BYTES of features from the lanes' registers to the warp's place in shared memory, and out by a copy that
      // drops rows and columns past the end
      constexpr int ROW_BYTES = G::STAGE / 32;
      uint8_t* place = sW + G::OFF_OUT + warp * (G::NSTAGE * G::STAGE);
      const auto put_rows = [&](const uint32_t* x, int column, int row0) {
        if (lane == 0) {
          if (G::NSTAGE == 2) bulk_wait_read1(); else bulk_wait_read0();
        }
        __syncwarp();
        uint8_t* dst = place + (G::NSTAGE == 2 ? (copies & 1) * G::STAGE : 0);
        copies++;
#pragma unroll
        for (int j = 0; j < ROW_BYTES / 16; j++) {
          const int piece = ROW_BYTES == 128 ? j ^ (lane & 7) : j ^ ((lane >> 1) & 3);
          *reinterpret_cast<uint4*>(dst + lane * ROW_BYTES + piece * 16) = make_uint4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (row0 < t.L) tma_store_3d(&a.out[ti], dst, column, row0, bh);
          bulk_commit();
        }
      };
      // x ln 2, x + y being rounded to x: one rounding in all
      const auto to_nat = [](float x, float y) { return fmaf(0.693147182f, x, fmaf(0.693147182f, y, -1.90465421e-9f * x)); };
      if (WRITE && t.stab == FSHARP_STAB_GROUP && t.logscale && tile0 == 0 && mblk == 0 && tid == 0) t.logscale[bh] = to_nat(gshift, 0.f);
      const uint32_t acc = tmem + wg * 256 + ((uint32_t)((warp & 3) * 32) << 16);
      for (int it = 0; it < ntiles; it++, n++) {
        if ((n & 1) != wg) continue;
        const int tok0 = (tile0 + it) * TILE + (warp & 3) * 32, tok = tok0 + lane;
        const int64_t at = (int64_t)bh * t.L + tok;
        const bool in = tok < t.L;
        float ci = bias;
        if (OUT16 && terms) {
          const int ab = n % G::NBUF, row = (warp & 3) * 32 + lane;
          if (scalar) {
            mbar_wait(&misc->a_full[ab], (n / G::NBUF) & 1, &misc->abort_flag, a.status);
            float half[2] = {};
#pragma unroll
            for (int s = 0; s < G::NKS; s++) {
              float sum[4] = {};
              const uint8_t* src = sA + ab * G::A_BYTES + s * TILE_BYTES + row * 128;
#pragma unroll
              for (int cc = 0; cc < G::CH; cc++) {
                const uint4 q = *reinterpret_cast<const uint4*>(src + ((cc ^ (row & 7)) << 4));
                const uint32_t v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int j = 0; j < 4; j++) {
                  const float lo = a.pow2 * __uint_as_float(v[j] << 16), hi = a.pow2 * __uint_as_float(v[j] & 0xffff0000u);
                  sum[(2 * j) & 3] = fmaf(lo, lo, sum[(2 * j) & 3]);
                  sum[(2 * j + 1) & 3] = fmaf(hi, hi, sum[(2 * j + 1) & 3]);
                }
              }
              half[s & 1] = (sum[0] + sum[1]) + (sum[2] + sum[3]);
            }
            const float c = quad.times(half[0] + half[1]);
            bad |= in && !isfinite(c);
            ci += c;
            if (!WRITE && in && mblk == 0) t.rowc[at] = c;
            // Stored before the tile is handed back: the store needs every value of the row.  Nothing else uses c on this side of
            // the arrival, behind which the last loads could still be on their way out of shared memory when the next tile lands.
            *const_cast<volatile float*>(&maxima->term[wg][row]) = c;
          } else {
            ci += in ? t.rowc[at] : 0.f;
          }
          mbar_arrive_warp(&misc->a_free[ab], lane);
        } else {
          ci += in ? t.rowc[at] : 0.f;
        }
        // exponent = acc + add, minus `shift` where that does not come from this block's own maximum: in this order the largest
        // exponent of the group or row, rounded as it was when the maximum was taken, gives 1 and nothing gives more
        float add = ci, shift = gshift - t.lift;
        if (WRITE && t.stab == FSHARP_STAB_ROW && !own) shift = (in ? FS_TO_LOG2(t.logscale[at]) : 0.f) - t.lift;
        const bool shifted = WRITE && !own && t.stab != FSHARP_STAB_NONE;
        mbar_wait(&misc->t_full[wg], (n >> 1) & 1, &misc->abort_flag, a.status);
        __syncwarp();
        tcgen05_fence_after();
        // The next columns' loads from tensor memory are in flight under the current ones' arithmetic: a warpgroup has one
        // warp per scheduler, so the latencies are its own to hide.  The last piece may reach past mb: columns of the other
        // accumulator, whose values are not used.
        uint32_t v[32];
        auto fetch = [&](int c) {
          tmem_ld16(acc + c, *reinterpret_cast<uint32_t(*)[16]>(v));
          tmem_ld16(acc + min(c + 16, 240), *reinterpret_cast<uint32_t(*)[16]>(v + 16));
        };
        auto arrived = [&](uint32_t (&x)[32]) {
          tmem_wait_ld();
          pin16(v); pin16(v + 16);
#pragma unroll
          for (int j = 0; j < 32; j++) x[j] = v[j];
        };
        fetch(0);
        if (!WRITE || own) {
          float mx = -3.0e38f, my = -3.0e38f;
          for (int c = 0; c < mb; c += 32) {
            uint32_t x[32];
            arrived(x);
            fetch(c + 32 < mb ? c + 32 : 0);           // (the features start again at column 0)
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
              mx = max3(mx, __uint_as_float(x[j]), __uint_as_float(x[j + 1]));
              my = max3(my, __uint_as_float(x[j + 2]), __uint_as_float(x[j + 3]));
            }
            if (c + 16 < mb) {
#pragma unroll
              for (int j = 16; j < 32; j += 4) {
                mx = max3(mx, __uint_as_float(x[j]), __uint_as_float(x[j + 1]));
                my = max3(my, __uint_as_float(x[j + 2]), __uint_as_float(x[j + 3]));
              }
            }
          }
          mx = fmaxf(mx, my);
          if (PAIR) {
            // The other block's warps can be one of this warpgroup's tiles ahead, no more: past it they wait for warps here.  So
            // consecutive tiles have places and barriers of their own (with one barrier, the next tile's four arrivals could
            // complete a second phase before a slow warp here had seen the first, and its wait for that parity would not end).
            const int k = n >> 1, row = (warp & 3) * 32 + lane;
            float* place = &maxima->row[wg][k & 1][row];
            uint64_t* bar = &misc->max_full[wg][k & 1];
            store_cluster(map_cluster(smem_u32(place), rank ^ 1), mx);
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_cluster(smem_u32(bar), rank ^ 1));
            mbar_wait_cluster(bar, (k >> 1) & 1, &misc->abort_flag, a.status);
            __syncwarp();
            mx = fmaxf(mx, *reinterpret_cast<volatile float*>(place));
          }
          if (WRITE) {
            add = t.lift - mx;
            const float top = mx + ci, big = fabsf(mx) > fabsf(ci) ? mx : ci, small = fabsf(mx) > fabsf(ci) ? ci : mx;
            if (t.logscale && in) t.logscale[at] = to_nat(top, small - (top - big));
          } else if (t.stab == FSHARP_STAB_GROUP) {
            if (in) gmx = fmaxf(gmx, mx + ci);
          } else {
            // (nudged upwards by the rounding of the two conversions, so that no feature exceeds one)
            const float ls = to_nat(mx + ci, 0.f);
            if (in) atomic_max_float(t.logscale + at, fmaf(fabsf(ls), 2.4e-7f, ls));
          }
        }
        if (WRITE) {
          for (int c = 0; c < mb; c += 32) {
            uint32_t x[32];
            arrived(x);
            if (c + 32 < mb) fetch(c + 32);
#pragma unroll
            for (int j = 0; j < 32; j += 2) add2(x[j], x[j + 1], add, add);
            if (shifted) {
#pragma unroll
              for (int j = 0; j < 32; j += 2) add2(x[j], x[j + 1], -shift, -shift);
            }
#pragma unroll
            for (int j = 0; j < 32; j++) x[j] = __float_as_uint(OUT16 ? ex2(__uint_as_float(x[j])) : ex2_full(__uint_as_float(x[j])));
            if (OUT16) {
              uint32_t h[16];
#pragma unroll
              for (int j = 0; j < 16; j++) h[j] = pack_bf16(__uint_as_float(x[2 * j]), __uint_as_float(x[2 * j + 1]));
              put_rows(h, m0 + c, tok0);
            } else if (a.staged[ti]) {
#pragma unroll
              for (int j = 0; j < 32; j += ROW_BYTES / 4)
                if (c + j < mb) put_rows(x + j, m0 + c + j, tok0);
            } else if (in) {
              float* dst = t.phi + at * a.M + m0 + c;
              if (wide) {
#pragma unroll
                for (int j = 0; j < 4; j++)
                  if (j < 2 || c + 16 < mb) store32(dst + 8 * j, &x[8 * j]);
              } else {
#pragma unroll
                for (int j = 0; j < 32; j++)
                  if (j < 16 || c + 16 < mb) dst[j] = __uint_as_float(x[j]);
              }
            }
          }
        } else {
          tmem_wait_ld();                              // the wrapped-around fetch
        }
        tcgen05_fence_before();
        mbar_arrive_warp(&misc->t_free[wg], lane);
      }
      if (!WRITE && t.stab == FSHARP_STAB_GROUP) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) gmx = fmaxf(gmx, __shfl_xor_sync(0xffffffffu, gmx, o));
        if (lane == 0) atomicMax(t.gmax + bh, f2ord(gmx));
      }
    }
    runs++;
  }
  if (bad) atomicExch(a.status, FSHARP_E_NONFINITE);
  // no copy of this block may still be in flight when it exits
  if (WRITE && warp < FT_STAGE0 && lane == 0) bulk_wait0();
  if (OUT16 && warp == FT_STAGE0 && lane == 0)
    for (int k = max(0, n - G::NBUF); k < n; k++)
      mbar_wait(&misc->a_full[k % G::NBUF], (k / G::NBUF) & 1, &misc->abort_flag, a.status, false);
  tcgen05_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();                                        // (the other block writes here until its last tile)
  if (warp == FT_MMA) {
    tcgen05_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// Tiles per block up to which each lane stores its own row: where a block has only a few, nothing runs under the latency of staging and
// copying, and lines that a row does not fill are written in parts either way.  Staged and direct, us, row shifts, 148 SMs.  d = 64, M = 256,
// fp32: 24.8 and 24.6 with half a tile per block, 29.2 and 30.7 with one or two, 49.3 and 51.6 with four.  Rows of partial lines, d = 32, M = 208,
// bf16: 18.0 and 17.4 with one, 40.8 and 39.8 with six, 46.0 and 46.2 with eight; d = 64, M = 48, fp32: 18.2 and 17.8, 33.8 and 33.7, 55.6 and 57.1 with
// twelve; M = 16, half of a staged tile: 12.7 and 12.3, 35.7 and 33.7 with twenty.  d = 128, in halves of a line: fp32, M = 256, 71.7 and
// 70.1 with two, 81.6 and 81.6 with three, 91.2 and 92.7 with four; bf16, 96 x 687 tokens, M = 256 (eight tiles per block, in pieces of sequences),
// 169 and 164, 8 x 9472 87.4 and 89.0; one block of features, M = 64, 32.6 and 32.9 with three.
int direct_tiles(int bits, int d, int M) {
  if (d == 128) return bits == 16 && M > 128 ? 8 : 3;
  return M < 32 ? 1 << 24 : M % 32 ? 6 : 1;
}

template <typename T, int D, int BP>
int launch_t(fsharp_ctx* ctx, Args& a, const Task* tasks, int ntasks, int BH, int G_groups, float qk_scale, uint8_t* img) {
  using G = FtGeo<T, D, BP, true>;
  constexpr size_t max_smem = FtGeo<T, D, BP, false>::SMEM;
  a.wscale = Factor(LOG2E * (1.0 + LOST_W<D>) * (double)qk_scale);
  a.nmb = (a.M + G::MB - 1) / G::MB;
  CUtensorMap maps[2] = {};
  if (BP == 2)
    for (int i = 0; i < ntasks; i++) FS_TRY(tchost::make_map_tokens(&maps[i], tasks[i].X, tasks[i].ax, BH / a.H, a.H, tasks[i].L, D));
  CUtensorMap outs[2] = {};
  bool staged[2] = {};
  int64_t items = 0;
  for (int i = 0; i < ntasks; i++) items += (int64_t)BH * a.nmb * ((tasks[i].L + TILE - 1) / TILE);
  const bool few = BP == 3 && items <= (int64_t)direct_tiles(sizeof(T) * 8, D, a.M) * ctx->sm_count;
  for (int i = 0; i < ntasks; i++) {
    void* phi = BP == 2 ? (void*)tasks[i].phi16 : (void*)tasks[i].phi;
    const uintptr_t at = reinterpret_cast<uintptr_t>(phi);
    staged[i] = at % 16 == 0 && !(few && at % 32 == 0);              // (the library's own are on 256-byte boundaries)
    if (staged[i]) FS_TRY(tchost::make_map_features(&outs[i], phi, BH, tasks[i].L, a.M, BP == 2, G::STAGE / 32));
  }
  const uint8_t* side_img[2] = {nullptr, nullptr};     // by side - 1
  const bool pair = BP == 2 && ntasks == 1 && tasks[0].stab == FSHARP_STAB_ROW && a.nmb == 2;
  a.own_terms = BP == 2;
  a.row_init = a.nmb > 1 && !pair;
  // (a set with a row shift over several feature blocks has its maxima pass instead: its blocks convert W themselves)
  if (img != nullptr && !(ntasks == 1 && tasks[0].stab == FSHARP_STAB_ROW && a.nmb > 1 && !pair)) {
    const int side0 = ntasks == 2 ? 1 : tasks[0].side;
    const size_t per_side = (size_t)G_groups * G::NKS * BP * a.M * 128;
    for (int k = 0; k < ntasks; k++) side_img[side0 - 1 + k] = img + k * per_side;
    const dim3 grid((a.M * (D / 8) + 255) / 256, G_groups, ntasks);
    FS_TIME_BEGIN(ctx, FS_K_W3);
    (void)fs_launch_chained(w3_images_kernel<D, BP>, grid, dim3(256), 0, ctx->stream, a.prep, side0, ntasks, a.M, a.wscale, img, ctx->d_status);
    FS_TIME_END(ctx);
    FS_LAUNCH_CHECK(ctx);
  }
  const auto set = [&](int units_per_bh, bool (*take)(const Task&, int)) {
    int k = 0;
    a.first[0] = 0;
    for (int i = 0; i < ntasks; i++) {
      if (!take(tasks[i], a.nmb)) continue;
      a.t[k] = tasks[i];
      a.map[k] = maps[i];
      a.out[k] = outs[i];
      a.staged[k] = staged[i];
      a.img[k] = side_img[tasks[i].side - 1];
      a.tiles[k] = (tasks[i].L + TILE - 1) / TILE;
      a.first[k + 1] = a.first[k] + BH * units_per_bh * a.tiles[k];
      k++;
    }
    for (; k < 2; k++) a.first[k + 1] = a.first[k];
    return a.first[2];
  };
  {
    const int total = set(1, [](const Task&, int) { return true; });
    constexpr size_t smem = rt_smem<T, D>();
    FS_CUDA_OK(cudaFuncSetAttribute(rowterm3_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int most = (D == 128 ? 1 : 3) * ctx->sm_count;
    // A block per tile; where tiles are few, enough blocks for what is cleared (four stores per thread), up to one per SM.  (All of it by the
    // blocks of one or two tiles: the attention of 2 x 64 tokens, d = 128, M = 1024, 84 -> 90 us, 85 so; up to three per SM: 64 x 100 tokens,
    // d = 64, M = 256, 69.7 -> 71.3.)
    const size_t clear = (a.zero4 + 4 * RT_THREADS - 1) / (4 * RT_THREADS);
    int blocks = clear < (size_t)ctx->sm_count ? (int)clear : ctx->sm_count;
    if (total > blocks) blocks = total < most ? total : most;
    FS_TIME_BEGIN(ctx, FS_K_ROWTERM);
    (void)fs_launch_chained(rowterm3_kernel<T, D>, dim3(blocks), dim3(RT_THREADS), smem, ctx->stream, a);
    FS_TIME_END(ctx);
    FS_LAUNCH_CHECK(ctx);
  }
  if constexpr (BP == 2) {
    if (pair) {
      const auto kernel = feat3_kernel<T, D, true, BP, true>;
      const int total = set(1, [](const Task&, int) { return true; }), most = ctx->sm_count / 2;
      FS_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM));
      FS_TIME_BEGIN(ctx, FS_K_FEAT);
      (void)fs_launch_chained_cluster(kernel, dim3(2 * (total < most ? total : most)), dim3(FT_THREADS), 2, G::SMEM, ctx->stream, a);
      FS_TIME_END(ctx);
      FS_LAUNCH_CHECK(ctx);
      return FSHARP_OK;
    }
  }
  const int maxed = set(a.nmb, [](const Task& t, int nmb) { return t.stab == FSHARP_STAB_GROUP || (t.stab == FSHARP_STAB_ROW && nmb > 1); });
  if (maxed > 0) {
    FS_CUDA_OK(cudaFuncSetAttribute(feat3_kernel<T, D, false, BP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem));
    FS_TIME_BEGIN(ctx, FS_K_GROUPMAX);
    (void)fs_launch_chained(feat3_kernel<T, D, false, BP>, dim3(maxed < ctx->sm_count ? maxed : ctx->sm_count), dim3(FT_THREADS), max_smem, ctx->stream, a);
    FS_TIME_END(ctx);
    FS_LAUNCH_CHECK(ctx);
  }
  const int total = set(a.nmb, [](const Task&, int) { return true; });
  FS_CUDA_OK(cudaFuncSetAttribute(feat3_kernel<T, D, true, BP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM));
  FS_TIME_BEGIN(ctx, FS_K_FEAT);
  (void)fs_launch_chained(feat3_kernel<T, D, true, BP>, dim3(total < ctx->sm_count ? total : ctx->sm_count), dim3(FT_THREADS), G::SMEM, ctx->stream, a);
  FS_TIME_END(ctx);
  FS_LAUNCH_CHECK(ctx);
  return FSHARP_OK;
}

// Two token sets share their launches, four instead of seven (the attention of 4 x 8 x 1501 tokens, d = 32, M = 128, and its gradients
// 360 -> 332 us, the kernel operator on 20011 x 30000 points 141 -> 121 us).  At d = 128 W is the larger part of what a block
// reads, and a launch of its own lets blocks keep one for longer: there only while both sets together leave SMs without a tile.
template <typename T, int D, int BP>
int run_t(fsharp_ctx* ctx, Args& a, const Task* tasks, int ntasks, int BH, int groups, float qk_scale, uint8_t* img) {
  if constexpr (BP == 3 && D == 128 && sizeof(T) == 2) {
    if (tasks[0].phi16 != nullptr) return run_t<T, D, 2>(ctx, a, tasks, ntasks, BH, groups, qk_scale, img);
  }
  int64_t items = 0;
  for (int i = 0; i < ntasks; i++) items += (int64_t)BH * ((tasks[i].L + TILE - 1) / TILE) * ((a.M + WGeo<D, BP>::MB - 1) / WGeo<D, BP>::MB);
  if (items > 2147483647LL) return FSHARP_E_SHAPE;     // items are numbered in 32 bits
  if (ntasks == 1 || (BP == 3 && (D < 128 || items <= ctx->sm_count))) return launch_t<T, D, BP>(ctx, a, tasks, ntasks, BH, groups, qk_scale, img);
  for (int i = 0; i < ntasks; i++) {
    FS_TRY((launch_t<T, D, BP>(ctx, a, tasks + i, 1, BH, groups, qk_scale, img)));
    a.zero4 = 0;
  }
  return FSHARP_OK;
}

}  // namespace

// Images of very many groups (none beyond 1 GB) are not worth their memory: a group's tokens are then few, and every block converts
// the W of its own.
size_t feat3::image_bytes(int groups, int d, int M, int ntasks) {
  const size_t bytes = ws_round((size_t)ntasks * groups * ((d + 63) / 64) * 3 * M * 128);
  return bytes <= ((size_t)1 << 30) ? bytes : 0;
}

int feat3::run(fsharp_ctx* ctx, const Task* tasks, int ntasks, int dtype, int B, int H, int d, int M, int pool, const float* prep,
               float qk_scale, uint8_t* img, float* zero, size_t zero_floats) {
  Args a{};
  a.zero = reinterpret_cast<float4*>(zero);
  a.zero4 = zero_floats / 4;
  a.H = H; a.M = M; a.pool = pool; a.prep = prep; a.status = ctx->d_status;
  int e = 0;
  (void)frexp((double)qk_scale, &e);
  a.pow2 = (float)ldexp(1.0, e < -100 ? -100 : (e > 100 ? 100 : e));
  a.quad = LOG2E * (double)qk_scale * (double)qk_scale / ((double)a.pow2 * (double)a.pow2);
  const int groups = pool == FSHARP_POOL_PER_BH ? B * H : H;
  if (image_bytes(groups, d, M, ntasks) == 0) img = nullptr;
#define FS_FEAT3(DD)                                                                                          \
  return dtype == FSHARP_F32 ? run_t<float, DD, 3>(ctx, a, tasks, ntasks, B * H, groups, qk_scale, img)                    \
                             : run_t<__nv_bfloat16, DD, 3>(ctx, a, tasks, ntasks, B * H, groups, qk_scale, img)
  switch (d) {
    case 16: FS_FEAT3(16);
    case 32: FS_FEAT3(32);
    case 64: FS_FEAT3(64);
    case 128: FS_FEAT3(128);
    default: return FSHARP_E_SHAPE;
  }
#undef FS_FEAT3
}
