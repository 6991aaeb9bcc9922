// Per-group precomputation for the feature kernels (Section 4, cost paragraph):
// W^(k) = Omega B^(k) (row m = (B^(k)T w_m)^T), a_m = w_m^T A w_m, the constant
// log D - 1/2 log M.
#include <cuda_fp16.h>

#include "common.cuh"
#include "mma3.cuh"
#include "tc_common.cuh"
#include "tc_layout.cuh"

namespace {

constexpr int PREP_MB = mma3::ROWS;           // features per block
constexpr int PREP_THREADS = mma3::THREADS;

// C, the scalars and the flags of one (group, side); every thread of the block
template <int D>
__device__ __forceinline__ void scalars_of(int g, int side, const double* __restrict__ params, int64_t params_stride, int M,
                                           double half_log_m, float* __restrict__ prep, float qk_scale, uint8_t* __restrict__ images,
                                           int* __restrict__ img_flags, double alpha, uint8_t* raw) {
  constexpr int d = D;
  const int tid = threadIdx.x;
  ParamsLayout pl{d};
  PrepLayout pr{d, M};
  const double* P = params + (size_t)g * params_stride;
  float* out = prep + ((size_t)g * 2 + (side - 1)) * pr.total();
  const double* Cm = P + pl.C(side);
  const double* tail = P + pl.tail();
  float* scal = out + pr.scal();
  float* Cf = out + pr.Cmat();
  // C = gamma I exactly?  The operand images (row j, column i = C[i][j], 128-byte swizzle) are put together in shared
  // memory and leave in 16-byte pieces: element-wise stores of a transposed 2-byte layout would touch a sector each.
  int cscalar = 1, lo_nonzero = 0;
  const double gamma = Cm[0] + alpha;
  uint8_t* simg = raw;             // [hi image | lo image], IMG_C_BYTES each (d = 64 only)
  for (int e0 = tid; e0 < d * d; e0 += 8 * PREP_THREADS) {
    double cv[8];
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int e = e0 + q * PREP_THREADS;
      cv[q] = e < d * d ? Cm[e] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int e = e0 + q * PREP_THREADS;
      if (e >= d * d) continue;
      const int i = e / d, j = e % d;
      if (i == j) cv[q] += alpha;                                    // (0, but for the operator with exp(alpha |x|^2))
      if (images == nullptr) Cf[e] = (float)cv[q];
      if (i == j ? (cv[q] != gamma) : (cv[q] != 0.0)) cscalar = 0;
      if (images != nullptr) {
        // log2e * qk_scale^2 * C[i][j] goes to row j, column i of the MMA operand
        const float v = (float)cv[q] * (FS_LOG2E * qk_scale * qk_scale);
        const __nv_bfloat16 hi = __float2bfloat16_rn(v), lo = __float2bfloat16_rn(v - __bfloat162float(hi));
        if (__bfloat162float(lo) != 0.f) lo_nonzero = 1;
        *reinterpret_cast<__nv_bfloat16*>(simg + tc::sw128_offset(j, i)) = hi;
        *reinterpret_cast<__nv_bfloat16*>(simg + tcl::IMG_C_BYTES + tc::sw128_offset(j, i)) = lo;
      }
    }
  }
  lo_nonzero = __syncthreads_or(lo_nonzero);
  if (images != nullptr) {
    // the two images are adjacent in the operand image block as well (IMG_CLO = IMG_CHI + IMG_C_BYTES)
    uint4* dst = reinterpret_cast<uint4*>(images + ((size_t)g * 2 + (side - 1)) * tcl::IMG_BYTES + tcl::IMG_CHI);
    const uint4* src = reinterpret_cast<const uint4*>(simg);
    for (int e = tid; e < (int)(2 * tcl::IMG_C_BYTES / 16); e += PREP_THREADS) dst[e] = src[e];
  }
  cscalar = __syncthreads_and(cscalar);
  if (tid == 0) {
    for (int i = 0; i < 8; i++) scal[i] = 0.f;
    scal[PS_BIAS] = (float)(tail[PT_LOGD] - half_log_m);
    scal[PS_CSCALAR] = cscalar ? 1.f : 0.f;
    scal[PS_CGAMMA] = (float)gamma;
    if (images != nullptr) {
      int* fl = img_flags + ((size_t)g * 2 + (side - 1)) * tcl::FLAG_WORDS;
      fl[0] = (cscalar ? 0 : tcl::FLAG_C_DENSE) | (lo_nonzero ? tcl::FLAG_C_LO : 0);
      fl[1] = __float_as_int((float)gamma * (FS_LOG2E * qk_scale * qk_scale));
    }
  }
}

// One block = one (group, role, chunk of 128 features).  Roles: W = Omega B of SIDES sides; a = diag(Omega A Omega^T), the same for
// both sides and written for both; C, the scalars and the flags of side blockIdx.z + 1 (in front of the blocks of a, these made a
// launch 3 us longer, also with the sum for diagonal A).  The products run on the tensor cores at fp32
// precision (mma3.cuh): 64 groups of 256 x 64 features are 200 million multiply-adds, which as fp32 instructions on operands in shared
// memory took 20 us (bound by the shared-memory reads).  What is left is the latency of loads, products and stores one after the
// other, in as many waves as it takes: two blocks on an SM (96 registers: three warps of each of two blocks' nine share a scheduler.  With more, one
// block: features of 400 x 128 fp32 tokens, d = 128, M = 512, 744 us, 641 so).  d = 64 and below: a W block takes one side while that
// makes at most two waves (d = 64) or one, both side by side beyond that (features of 128-token groups, d = 64, M = 256, us, one side and both: 24
// groups 25.6 and 30.2, 64 36.3 and 40.8, 74 37.4 and 38.1, 200 86.6 and 81.8; d = 32: 37 16.7 and 17.9, 64 18.2 and 18.7, 100 21.6 and 19.8).
template <int D, int SIDES>
__global__ void __launch_bounds__(PREP_THREADS, 2)
prep_kernel(const float* __restrict__ Omega, int64_t omega_head_stride, const double* __restrict__ params,
            int64_t params_stride, int H, int pool, int M, float* __restrict__ prep, float qk_scale,
            uint8_t* __restrict__ images, int* __restrict__ img_flags, double half_log_m, double alpha, int* __restrict__ status) {
  fs_grid_dependency_wait();
  // images != nullptr (d = 64, M = 256 only): the tensor-core path's operand images of this (group, side)
  // are written as well, in the layouts of tc_layout.cuh
  constexpr int d = D, NW = 2 / SIDES;                                 // W roles
  static_assert(SIDES * D <= 128, "columns of one product");
  extern __shared__ __align__(1024) uint8_t raw[];
  const int g = blockIdx.x, role = blockIdx.y, tid = threadIdx.x;
  if (reinterpret_cast<uintptr_t>(raw) & 1023) {                       // (there is no room to align the stages)
    if (tid == 0) atomicExch(status, FSHARP_E_INTERNAL);
    return;
  }
  if (role == NW + 1) {
    if (blockIdx.z < 2) scalars_of<D>(g, blockIdx.z + 1, params, params_stride, M, half_log_m, prep, qk_scale, images, img_flags, alpha, raw);
    return;
  }
  const int m0 = blockIdx.z * PREP_MB, side0 = role;                  // (a W block's first side, from 0)
  const bool is_a = role == NW;
  if (m0 >= M) return;
  const int h = pool == FSHARP_POOL_PER_BH ? g % H : g;
  const float* Om = Omega + (int64_t)h * omega_head_stride;
  ParamsLayout pl{d};
  PrepLayout pr{d, M};
  const double* P = params + (size_t)g * params_stride;
  float* out = prep + (size_t)g * 2 * pr.total();                     // side 1; side 2 follows
  const bool aligned = (reinterpret_cast<uintptr_t>(Om) & 15) == 0;
  const auto omega = [&](int m, int k, auto& piece) {
    if (m0 + m >= M) { piece.zero(); return; }
    const float* p = Om + (size_t)(m0 + m) * d + k;
    if (aligned) { piece.load(p); return; }
#pragma unroll
    for (int j = 0; j < 8; j++) piece.v[j] = p[j];
  };
  const auto matrix = [&](int c, int k, auto& piece) {              // eight columns of row k of A or of [B^(1) | B^(2)]
    const double* p = P + (is_a ? pl.A() : pl.B(side0 + 1 + c / d)) + (size_t)k * d + c % d;
#pragma unroll
    for (int j = 0; j < 8; j++) piece.v[j] = (float)p[j];
  };
  const auto put_a = [&](int m, float a) {
#pragma unroll
    for (int side = 0; side < 2; side++) {
      out[(size_t)side * pr.total() + pr.a() + m] = a;
      if (images != nullptr)
        reinterpret_cast<float*>(images + ((size_t)g * 2 + side) * tcl::IMG_BYTES + tcl::IMG_A2)[m] = 2.f * FS_LOG2E * a;
    }
  };
  if (is_a) {
    // A is diagonal in all fits: a_m = sum_k A_kk Omega_mk^2, in fp64, and no product (which takes the same time, but ends in fp32:
    // error of the gradients at d = 16 4.3e-7 and 6.4e-7)
    double* diag = reinterpret_cast<double*>(raw);
    const double* A = P + pl.A();
    int off = 0;
    constexpr int BATCH = D == 128 ? 16 : 8;
    for (int e0 = tid; e0 < d * d; e0 += BATCH * PREP_THREADS) {
      double v[BATCH];
#pragma unroll
      for (int q = 0; q < BATCH; q++) v[q] = e0 + q * PREP_THREADS < d * d ? A[e0 + q * PREP_THREADS] : 0.0;
#pragma unroll
      for (int q = 0; q < BATCH; q++) {
        const int e = e0 + q * PREP_THREADS;
        if (e >= d * d) continue;
        if (e % (d + 1) == 0) diag[e / (d + 1)] = v[q];
        else if (v[q] != 0.0) off = 1;
      }
    }
    if (!__syncthreads_or(off)) {
      const int m = m0 + (tid >> 1), k0 = (tid & 1) * (d / 2);        // two threads per feature
      if (tid < 2 * PREP_MB) {
        double s[4] = {};
        if (m < M) {
          const float* o = Om + (size_t)m * d + k0;
#pragma unroll
          for (int k = 0; k < d / 2; k += 4) {
            float4 w;
            if (aligned) w = *reinterpret_cast<const float4*>(o + k);
            else w = make_float4(o[k], o[k + 1], o[k + 2], o[k + 3]);
            const float v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int j = 0; j < 4; j++) s[j] = fma(diag[k0 + k + j] * v[j], (double)v[j], s[j]);
          }
        }
        double sum = (s[0] + s[1]) + (s[2] + s[3]);
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        const float a = (float)sum;
        if (m < M && (tid & 1) == 0) put_a(m, a);
      }
      return;
    }
  }
  mma3::Block b;
  b.begin(raw, is_a ? d : SIDES * d, d, status);
  b.template segment<true, 3, false, 3>(d, omega, matrix);
  b.finish();
  if (!is_a) {
    b.rows([&](int row, int c, float4 v) {
      const int m = m0 + row, side = side0 + c / d, j = c % d;
      if (m >= M) return;
      if (images == nullptr) {           // (the fp32 copy serves the fp32 kernels only; the tensor-core path reads the operand image)
        float* w = out + (size_t)side * pr.total() + pr.W() + (size_t)m * d + j;
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
      } else {                           // log2e * qk_scale * W rounded to fp16
        const float sw = FS_LOG2E * qk_scale;
        const __half2 lo = __floats2half2_rn(v.x * sw, v.y * sw), hi = __floats2half2_rn(v.z * sw, v.w * sw);
        *reinterpret_cast<uint2*>(images + ((size_t)g * 2 + side) * tcl::IMG_BYTES + tcl::IMG_WH + tc::sw128_offset(m, j)) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
      }
    });
  } else {
    // a_m = sum_j (Omega A)_mj Omega_mj: the lanes that hold row m, piece by piece, then the two warps
    float (*part)[PREP_MB] = reinterpret_cast<float (*)[PREP_MB]>(b.sm + 65536);
    __syncthreads();                                                // (the products have been waited for by warps 0-7)
    if (tid < PREP_MB) part[0][tid] = part[1][tid] = 0.f;
    __syncthreads();
    b.rows([&](int row, int c, float4 v) {
      float s = 0.f;
      if (m0 + row < M) {
        const float* o = Om + (size_t)(m0 + row) * d + c;
        s = fmaf(v.x, o[0], fmaf(v.y, o[1], fmaf(v.z, o[2], v.w * o[3])));
      }
#pragma unroll
      for (int x = 1; x < (d >= 64 ? 8 : 4); x *= 2) s += __shfl_xor_sync(0xffffffffu, s, x);
      if ((b.lane & (d >= 64 ? 7 : 3)) == 0) part[b.warp >> 2][row] += s;
    });
    __syncthreads();
    if (tid < PREP_MB && m0 + tid < M) {
      const int m = m0 + tid;
      put_a(m, part[0][tid] + part[1][tid]);
    }
  }
  b.end();
}

}  // namespace

int fs_run_prep(fsharp_ctx* ctx, const float* Omega, int64_t omega_head_stride, const double* params,
                int64_t params_stride, int G, int H, int pool, int d, int M, float* prep, double alpha) {
  return fs_run_prep_images(ctx, Omega, omega_head_stride, params, params_stride, G, H, pool, d, M, prep, 1.f, nullptr, nullptr, alpha);
}

int fs_run_prep_images(fsharp_ctx* ctx, const float* Omega, int64_t omega_head_stride, const double* params,
                       int64_t params_stride, int G, int H, int pool, int d, int M, float* prep, float qk_scale,
                       uint8_t* images, int* flags, double alpha) {
  FS_RANGE("operand images");
  if (G == 0) return FSHARP_OK;
  if (images != nullptr && (d != tcl::TC_D || M != tcl::TC_M)) return FSHARP_E_SHAPE;
  const int nchunks = (M + PREP_MB - 1) / PREP_MB;
  const int nz = nchunks > 2 ? nchunks : 2;
  const bool apart = d == 128 || (int64_t)G * 4 * nz <= (d == 64 ? 4 : 2) * ctx->sm_count;
  const dim3 grid(G, apart ? 4 : 3, nz);
  // Shared memory: one block on an SM while there are no more blocks than SMs, two beyond that; and never so much that an SM is set up with its
  // largest share of it, as it is for the kernels around this one: with the same share the kernels that follow take longer (seen, not
  // explained; launched one by one: step of 1 x 17613 queries and 23266 keys 84.5 to 89 us, 81 so; 2^20 pairs, 32 draws, 3960 and 3905).
  constexpr size_t ONE = 116 * 1024, TWO = mma3::SMEM - 1024;          // 132 and 196 KB (1 KB more per block); the stages start at 0
  static_assert(2 * (TWO + 1024) <= 196 * 1024 && 2 * (ONE + 1024) > 228 * 1024, "shares");
  const size_t smem = (int64_t)grid.x * grid.y * grid.z <= ctx->sm_count ? ONE : TWO;
#define FS_PREP(DD, SS)                                                                                              \
  do {                                                                                                               \
    FS_CUDA_OK(cudaFuncSetAttribute(prep_kernel<DD, SS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ONE));    \
    FS_TIME_BEGIN(ctx, FS_K_PREP);                                                                                    \
    (void)fs_launch_chained(prep_kernel<DD, SS>, grid, dim3(PREP_THREADS), smem, ctx->stream, Omega, omega_head_stride, params, params_stride, H,   \
                                                               pool, M, prep, qk_scale, images, flags, 0.5 * log((double)M), alpha, ctx->d_status);  \
  } while (0)
  switch (d) {
    case 16: if (apart) FS_PREP(16, 1); else FS_PREP(16, 2); break;
    case 32: if (apart) FS_PREP(32, 1); else FS_PREP(32, 2); break;
    case 64: if (apart) FS_PREP(64, 1); else FS_PREP(64, 2); break;
    case 128: FS_PREP(128, 1); break;
    default: return FSHARP_E_SHAPE;
  }
#undef FS_PREP
  FS_TIME_END(ctx);
  FS_LAUNCH_CHECK(ctx);
  return FSHARP_OK;
}
