// Kernel estimation for (x, y) pairs (Section 2.1: Khat = sum_m P_m S_m; the estimates themselves: tc_pairs.cu) and the
// closed-form variance of Theorem 4.1 divided by M (Section 2.1).
#include "common.cuh"

size_t fs_tc_pairs_scratch_bytes(int d, int M, int R);
int fs_tc_pairs(fsharp_ctx* ctx, const float* X, const float* Y, int64_t np, int d, int M, int R, const float* prep, float* est,
                WsAlloc* ws);

namespace {

constexpr int NTH = 256;

// With z = (x, y) the closed form's exponent is z^T F z, F upper triangular (2 d x 2 d):
// x^T E1 x + y^T E2 y + x^T E12 y, E1 = C1 + 2 B1^T R B1, E2 = C2 + 2 B2^T R B2, E12 = 4 B1^T R B2 with R = (I - 8A)^-1 (A
// diagonal), off-diagonal entries of E1 and E2 doubled and kept on one side, and k0 = 4 log D - 1/2 log det(I - 8A).
// ev: the 8 x 8 blocks on and above the diagonal, block column by block column, each in the order in which a warp reads it as an operand
// of the fp64 tensor cores (frag()); then k0.
__host__ __device__ constexpr int pv_blocks(int columns) { return columns * (columns + 1) / 2; }      // of the first block columns
__device__ __forceinline__ int frag(int k, int j) {
  return ((pv_blocks(j >> 3) + (k >> 3)) * 32 + (j & 7) * 4 + ((k & 7) >> 1)) * 2 + (k & 1);
}
// One block per row k; 256 / d threads per column share the inner products' terms, whose loads are in flight together.  (One thread
// per column, four terms at a time: 30 us at d = 64, a third of a call with few pairs; a single block took 172 us.)
constexpr int PP_THREADS = 256;
__global__ void __launch_bounds__(PP_THREADS)
pairvar_prep_kernel(const double* __restrict__ params, int d, double* __restrict__ ev, int* __restrict__ status) {
  fs_grid_dependency_wait();
  ParamsLayout pl{d};
  const double* A = params + pl.A();
  const double* B1 = params + pl.B(1);
  const double* B2 = params + pl.B(2);
  const double* C1 = params + pl.C(1);
  const double* C2 = params + pl.C(2);
  __shared__ double rinv[128], lg[128], part_s[3][PP_THREADS];
  const int k = blockIdx.x, tid = threadIdx.x, j = tid % d, parts = PP_THREADS / d, len = d / parts, l0 = tid / d * len;
  double c1 = 0.0, c2 = 0.0, a = 0.0;
  if (tid < d) {
    const double v = 1.0 - 8.0 * A[j * d + j];
    c1 = C1[k * d + j] + C1[j * d + k];
    c2 = C2[k * d + j] + C2[j * d + k];
    a = A[k * d + j];
    rinv[j] = 1.0 / v;
    if (k == 0) lg[j] = log(v);
    if (k == 0 && !(v > 0.0)) atomicExch(status, FSHARP_E_CONSTRAINT);
    if (k != j && a != 0.0) atomicExch(status, FSHARP_E_CONSTRAINT);
  }
  __syncthreads();
  double s1 = 0.0, s2 = 0.0, s12 = 0.0;
#pragma unroll 16
  for (int l = l0; l < l0 + len; l++) {
    const double r = rinv[l], b1k = B1[l * d + k] * r, b2j = B2[l * d + j];
    s1 = fma(b1k, B1[l * d + j], s1);
    s2 = fma(B2[l * d + k] * r, b2j, s2);
    s12 = fma(b1k, b2j, s12);
  }
  part_s[0][tid] = s1;
  part_s[1][tid] = s2;
  part_s[2][tid] = s12;
  __syncthreads();
  if (tid < d) {
    for (int p = 1; p < parts; p++) {
      s1 += part_s[0][p * d + j];
      s2 += part_s[1][p * d + j];
      s12 += part_s[2][p * d + j];
    }
    if (k >> 3 <= j >> 3) {
      ev[frag(k, j)] = k < j ? 2.0 * (c1 + 2.0 * s1) : (k == j ? c1 + 2.0 * s1 : 0.0);
      ev[frag(d + k, d + j)] = k < j ? 2.0 * (c2 + 2.0 * s2) : (k == j ? c2 + 2.0 * s2 : 0.0);
    }
    ev[frag(k, d + j)] = 4.0 * s12;
  }
  if (k == 0 && tid < 32) {
    double ld = 0.0;
    for (int l = tid; l < d; l += 32) ld += lg[l];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ld += __shfl_xor_sync(0xffffffffu, ld, o);
    if (tid == 0) ev[64 * pv_blocks(d / 4)] = 4.0 * params[pl.tail() + PT_LOGD] - 0.5 * ld;
  }
}

// c += A B, 8 x 8 x 4 on the fp64 tensor cores: lane holds A[lane / 4][lane % 4], B[lane % 4][lane / 4] and C[lane / 4][2 (lane % 4) + {0, 1}].
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
  asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}

// Var = (exp(k0 + z^T F z) - exp(2 x^T y)) / M per pair, in fp64, and (pooled != nullptr) the
// pooled relative variances of Section 5.1: the unbiased sample variance of a pair's R estimates and its closed-form
// variance, both over K^2 = exp(2 x^T y), averaged over the pairs (pooled[0], pooled[1] += ..., fp64 atomics; zero on entry).
//
// Bound: fp64 multiply-adds (2 d^2 per pair).  A warp has 8 MT pairs, whose z stay in registers as the A operand of Z F for all
// columns; F comes from shared memory, 512 bytes per 8 x 8 block and 2 MT MMAs.  The contracted index is taken in an order
// in which a lane's A values of an 8-block, z[2 t] and z[2 t + 1] (t = lane % 4), belong to the columns of its part of the product,
// so that z^T (F z) needs no other values of z.  The warps go their own ways (loads of one run under the products of another),
// the pooling included.  d = 128: half of F fits, so two launches, the first of which leaves its share of the exponent in var.
// (Scalar multiply-adds, x and y as doubles in shared memory and F through L1, which it did not fit: 1.57 ms for 2^20 pairs, d = 64, R = 32; 0.69 ms now, 0.52 at
// the rate of the fp64 units.  16 warps of eight pairs each instead of eight of sixteen: the same.)
template <int D> struct PvGeo {
  static constexpr int NB = D / 4, MT = D == 128 ? 1 : 2, P = 64 * MT, SPLIT = D == 128 ? 23 : NB;    // block columns; those of the first launch
  static constexpr int BLOCKS0 = pv_blocks(SPLIT), BLOCKS1 = pv_blocks(NB) - BLOCKS0;
  static constexpr size_t smem(int pass) { return (size_t)(pass ? BLOCKS1 : BLOCKS0) * 512; }
};
template <int D, int PASS>
__global__ void __launch_bounds__(NTH, D < 64 ? 2 : 1)
pairvar_kernel(const float* __restrict__ X, const float* __restrict__ Y, int64_t np, int M, int R, const double* __restrict__ ev,
               const float* __restrict__ est, double* __restrict__ var, double* __restrict__ pooled) {
  fs_grid_dependency_wait();
  using G = PvGeo<D>;
  constexpr int NB = G::NB, MT = G::MT, J0 = PASS ? G::SPLIT : 0, J1 = PASS ? NB : G::SPLIT, FIRST = pv_blocks(J0);
  constexpr bool LAST = J1 == NB;
  extern __shared__ __align__(16) double2 sf[];        // blocks FIRST .. of F
  __shared__ double red[2][NTH / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, g = lane >> 2, t = lane & 3;
  for (int e = tid; e < (pv_blocks(J1) - FIRST) * 32; e += NTH) sf[e] = reinterpret_cast<const double2*>(ev)[FIRST * 32 + e];
  const double k0 = ev[64 * pv_blocks(NB)];
  const bool vec = ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 7) == 0;
  __syncthreads();
  double acc_e = 0.0, acc_c = 0.0;
  for (int64_t p0 = (int64_t)blockIdx.x * G::P + w * (8 * MT); p0 < np; p0 += (int64_t)gridDim.x * G::P) {
    double z[MT][2 * NB];
#pragma unroll
    for (int m = 0; m < MT; m++) {
      const int64_t p = p0 + 8 * m + g;
      float2 v[NB];
#pragma unroll
      for (int b = 0; b < NB; b++) {
        const float* src = (b < NB / 2 ? X : Y) + p * D + 8 * (b % (NB / 2)) + 2 * t;
        v[b] = make_float2(0.f, 0.f);
        if (p < np) v[b] = vec ? *reinterpret_cast<const float2*>(src) : make_float2(src[0], src[1]);
      }
#pragma unroll
      for (int b = 0; b < NB; b++) { z[m][2 * b] = v[b].x; z[m][2 * b + 1] = v[b].y; }
    }
    double q[MT], xy[MT];
#pragma unroll
    for (int m = 0; m < MT; m++) {
      q[m] = xy[m] = 0.0;
#pragma unroll
      for (int k = 0; k < NB; k++) xy[m] = fma(z[m][k], z[m][NB + k], xy[m]);
    }
#pragma unroll
    for (int jb = J0; jb < J1; jb++) {
      double c[MT][2][2] = {};
#pragma unroll
      for (int kb = 0; kb <= jb; kb++) {
        const double2 f = sf[(pv_blocks(jb) + kb - FIRST) * 32 + lane];
#pragma unroll
        for (int m = 0; m < MT; m++) {
          dmma(c[m][0], z[m][2 * kb], f.x);
          dmma(c[m][1], z[m][2 * kb + 1], f.y);
        }
      }
#pragma unroll
      for (int m = 0; m < MT; m++)
        q[m] = fma(c[m][0][0] + c[m][1][0], z[m][2 * jb], fma(c[m][0][1] + c[m][1][1], z[m][2 * jb + 1], q[m]));
    }
    // a pair's sums over its four lanes; then pair lane % (8 MT) of the warp, its draws shared by the lanes that have it
    double qq = 0.0, dot = 0.0;
    constexpr int N = 8 * MT, SHARE = 32 / N;
#pragma unroll
    for (int m = 0; m < MT; m++) {
#pragma unroll
      for (int o = 1; o < 4; o *= 2) {
        q[m] += __shfl_xor_sync(0xffffffffu, q[m], o);
        xy[m] += __shfl_xor_sync(0xffffffffu, xy[m], o);
      }
      const double a = __shfl_sync(0xffffffffu, q[m], 4 * (lane & 7)), b = __shfl_sync(0xffffffffu, xy[m], 4 * (lane & 7));
      if (((lane >> 3) & (MT - 1)) == m) { qq = a; dot = b; }
    }
    const int64_t p = p0 + lane % N;
    const bool in = p < np;
    if (PASS > 0 && in) qq += var[p];
    __syncwarp();
    if (!LAST) {
      if (in && lane < N) var[p] = qq;
      continue;
    }
    const double v = (exp(k0 + qq) - exp(2.0 * dot)) / (double)M;
    if (in && lane < N) var[p] = v;
    if (pooled != nullptr) {
      // about the first draw: one pass over the estimates, and what the difference of the sums loses is some R roundings in fp64
      double s1 = 0.0, s2 = 0.0;
      const double e0 = in ? (double)est[p] : 0.0;
#pragma unroll 8
      for (int r = lane / N; r < R; r += SHARE) {
        const double dv = (in ? (double)est[(int64_t)r * np + p] : 0.0) - e0;
        s1 += dv;
        s2 = fma(dv, dv, s2);
      }
#pragma unroll
      for (int o = N; o < 32; o *= 2) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      }
      if (in && lane < N) {
        const double ik2 = exp(-2.0 * dot);
        acc_e += (R > 1 ? fma(-s1 / (double)R, s1, s2) / (double)(R - 1) : 0.0) * ik2;
        acc_c += v * ik2;
      }
    }
  }
  if (LAST && pooled != nullptr) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      acc_e += __shfl_xor_sync(0xffffffffu, acc_e, o);
      acc_c += __shfl_xor_sync(0xffffffffu, acc_c, o);
    }
    if (lane == 0) { red[0][w] = acc_e; red[1][w] = acc_c; }
    __syncthreads();
    if (tid == 0) {
      double e = 0.0, c = 0.0;
      for (int i = 0; i < NTH / 32; i++) { e += red[0][i]; c += red[1][i]; }
      atomicAdd(&pooled[0], e / (double)np);
      atomicAdd(&pooled[1], c / (double)np);
    }
  }
}

template <int D, int PASS>
int launch_pairvar(fsharp_ctx* ctx, const float* X, const float* Y, int64_t np, int M, int R, const double* ev, const float* est, double* var,
                   double* pooled) {
  constexpr size_t smem = PvGeo<D>::smem(PASS);
  FS_CUDA_OK(cudaFuncSetAttribute(pairvar_kernel<D, PASS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int64_t most = (D < 64 ? 2 : 1) * (int64_t)ctx->sm_count, blocks = (np + PvGeo<D>::P - 1) / PvGeo<D>::P;
  FS_TIME_BEGIN(ctx, FS_K_PAIRVAR);
  (void)fs_launch_chained(pairvar_kernel<D, PASS>, dim3((unsigned)(blocks < most ? blocks : most)), dim3(NTH), smem, ctx->stream, X, Y, np, M, R, ev,
                          est, var, pooled);
  FS_TIME_END(ctx);
  FS_LAUNCH_CHECK(ctx);
  return FSHARP_OK;
}

}  // namespace

// Draws that go through together: as many as prepared operands and images of 1 GB hold (a multiple of 128, so that column tiles of
// several draws are cut as in one go), all of them in any study but one of thousands of draws.
static int draws_per_batch(int d, int M, int R) {
  const size_t per = 2 * PrepLayout{d, M}.total() * sizeof(float) + fs_tc_pairs_scratch_bytes(d, M, 128) / 128;
  const size_t n = ((size_t)1 << 30) / per / 128 * 128;
  return (size_t)R <= n ? R : (int)n;
}

size_t fs_pairs_scratch_bytes(int d, int M, int R) {
  const int n = draws_per_batch(d, M, R);
  return ws_round((size_t)n * 2 * PrepLayout{d, M}.total() * sizeof(float)) +
         ws_round((64 * (size_t)pv_blocks(d / 4) + 1) * sizeof(double)) + fs_tc_pairs_scratch_bytes(d, M, n);
}

int fs_run_pairs(fsharp_ctx* ctx, const float* X, const float* Y, const float* Omega, const double* params,
                 int64_t npairs, int d, int M, int R, float* est, double* var_cf, double* pooled, WsAlloc* ws) {
  const int batch = draws_per_batch(d, M, R);
  float* prep = ws->take<float>((size_t)batch * 2 * PrepLayout{d, M}.total());
  double* ev = ws->take<double>(64 * (size_t)pv_blocks(d / 4) + 1);
  for (int r = 0; r < R; r += batch) {
    const int n = R - r < batch ? R - r : batch;
    // one "group" per draw, all reading the same parameter blob
    FS_TRY(fs_run_prep(ctx, Omega + (int64_t)r * M * d, (int64_t)M * d, params, 0, n, n, FSHARP_POOL_PER_HEAD, d, M, prep));
    WsAlloc rest = *ws;
    if (npairs > 0) FS_TRY(fs_tc_pairs(ctx, X, Y, npairs, d, M, n, prep, est + (int64_t)r * npairs, &rest));
  }
  if (npairs == 0) return FSHARP_OK;
  if (var_cf) {
    FS_TIME_BEGIN(ctx, FS_K_PAIRVAR_PREP);
    (void)fs_launch_chained(pairvar_prep_kernel, dim3(d), dim3(PP_THREADS), 0, ctx->stream, params, d, ev, ctx->d_status);
    FS_TIME_END(ctx);
    FS_LAUNCH_CHECK(ctx);
    if (pooled) FS_CUDA_OK(cudaMemsetAsync(pooled, 0, 2 * sizeof(double), ctx->stream));
    switch (d) {
      case 16: return launch_pairvar<16, 0>(ctx, X, Y, npairs, M, R, ev, est, var_cf, pooled);
      case 32: return launch_pairvar<32, 0>(ctx, X, Y, npairs, M, R, ev, est, var_cf, pooled);
      case 64: return launch_pairvar<64, 0>(ctx, X, Y, npairs, M, R, ev, est, var_cf, pooled);
      default:
        FS_TRY((launch_pairvar<128, 0>(ctx, X, Y, npairs, M, R, ev, est, var_cf, pooled)));
        return launch_pairvar<128, 1>(ctx, X, Y, npairs, M, R, ev, est, var_cf, pooled);
    }
  }
  return FSHARP_OK;
}
