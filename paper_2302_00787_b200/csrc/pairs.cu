// Kernel estimation for (x, y) pairs (Section 2.1: Khat = sum_m P_m S_m; the estimates themselves: tc_pairs.cu) and the
// closed-form variance of Theorem 4.1 divided by M (Section 2.1).
#include "common.cuh"

size_t fs_tc_pairs_scratch_bytes(int d, int M, int R);
int fs_tc_pairs(fsharp_ctx* ctx, const float* X, const float* Y, int64_t np, int d, int M, int R, const float* prep, float* est,
                WsAlloc* ws);

namespace {

constexpr int NTH = 256;
template <typename T, T V> struct integral_constant_t {
  __host__ __device__ constexpr operator T() const { return V; }
};

// E1 = 2 (C1 + B1^T R B1), E2 = 2 (C2 + B2^T R B2), E12 = 4 B1^T R B2 with R = (I - 8A)^-1 (A diagonal), and
// k0 = 4 log D - 1/2 log det(I - 8A).   ev: [3 d^2 + 1] doubles.  The two quadratic forms are folded into triangles
// (E1: k <= j, E2: k >= j, off-diagonal entries of both sides added), which halves their multiply-adds.
// One block per row k, one thread per column: the serial length is that of one inner product (a single block took
// 172 us at d = 64).
__global__ void __launch_bounds__(128)
pairvar_prep_kernel(const double* __restrict__ params, int d, double* __restrict__ ev, int* __restrict__ status) {
  fs_grid_dependency_wait();
  ParamsLayout pl{d};
  const double* A = params + pl.A();
  const double* B1 = params + pl.B(1);
  const double* B2 = params + pl.B(2);
  const double* C1 = params + pl.C(1);
  const double* C2 = params + pl.C(2);
  __shared__ double rinv[128], lg[128];
  const int k = blockIdx.x, j = threadIdx.x;
  if (j < d) {
    const double v = 1.0 - 8.0 * A[j * d + j];
    rinv[j] = 1.0 / v;
    if (k == 0) lg[j] = log(v);
    if (k == 0 && !(v > 0.0)) atomicExch(status, FSHARP_E_CONSTRAINT);
  }
  __syncthreads();
  if (j < d) {
    if (k != j && A[k * d + j] != 0.0) atomicExch(status, FSHARP_E_CONSTRAINT);
    double s1 = 0.0, s2 = 0.0, s12 = 0.0;
#pragma unroll 4
    for (int l = 0; l < d; l++) {
      const double r = rinv[l], b1k = B1[l * d + k] * r, b2j = B2[l * d + j];
      s1 = fma(b1k, B1[l * d + j], s1);
      s2 = fma(B2[l * d + k] * r, b2j, s2);
      s12 = fma(b1k, b2j, s12);
    }
    const double c1 = C1[k * d + j] + C1[j * d + k], c2 = C2[k * d + j] + C2[j * d + k];
    const int e = k * d + j;
    ev[e] = k < j ? 2.0 * (c1 + 2.0 * s1) : (k == j ? c1 + 2.0 * s1 : 0.0);
    ev[d * d + e] = k > j ? 2.0 * (c2 + 2.0 * s2) : (k == j ? c2 + 2.0 * s2 : 0.0);
    ev[2 * d * d + e] = 4.0 * s12;
  }
  if (k == 0 && j == 0) {
    double ld = 0.0;
    for (int l = 0; l < d; l++) ld += lg[l];
    ev[3 * d * d] = 4.0 * params[pl.tail() + PT_LOGD] - 0.5 * ld;
  }
}

// Var = (exp(k0 + x^T E1 x + y^T E2 y + x^T E12 y) - exp(2 x^T y)) / M per pair, in fp64, and (pooled != nullptr) the
// pooled relative variances of Section 5.1: the unbiased sample variance of a pair's R estimates and its closed-form
// variance, both over K^2 = exp(2 x^T y), averaged over the pairs (pooled[0], pooled[1] += ..., fp64 atomics; zero on entry).
//
// Bound: fp64 multiply-adds (2 d^2 per pair).  Block = P pairs, their x and y as doubles in shared memory, k index
// first; a lane carries P / 32 pairs and a warp D / 8 columns, so a row of E feeds a warp as broadcast loads and x, y as
// consecutive ones.  Column group w takes k <= j of E1 and k >= j of E2: every warp has the same work.  One warp per pair
// walking whole rows of the three matrices issued three loads per three multiply-adds: 4.2 ms for 2^20 pairs at d = 64
// and 0.64 ms for the pooling in a kernel of its own, now 1.57 ms for both.
template <int D>
__global__ void __launch_bounds__(NTH)
pairvar_kernel(const float* __restrict__ X, const float* __restrict__ Y, int64_t np, int M, int R, const double* __restrict__ ev,
               const float* __restrict__ est, double* __restrict__ var, double* __restrict__ pooled) {
  fs_grid_dependency_wait();
  constexpr int PL = D == 128 ? 2 : 4, P = 32 * PL, NC = D / 8;
  extern __shared__ __align__(16) double smd[];
  double* xs = smd;                       // [D][P]
  double* ys = smd + D * P;
  double* red = smd + 2 * D * P;          // [2][8][P]: q and x.y of the eight column groups
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const double k0 = ev[3 * D * D];
  const bool vec = ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15) == 0;
  double acc_e = 0.0, acc_c = 0.0;
  for (int64_t p0 = (int64_t)blockIdx.x * P; p0 < np; p0 += (int64_t)gridDim.x * P) {
    __syncthreads();
    // lanes run over the pairs: the stores hit consecutive words, the lines of the row-wise loads are met again in L1
#pragma unroll 2
    for (int e = tid; e < P * (D / 4); e += NTH) {
      const int p = e % P, k = e / P * 4;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
      if (p0 + p < np) {
        const float* xp = X + (p0 + p) * D + k;
        const float* yp = Y + (p0 + p) * D + k;
        if (vec) {
          x = *reinterpret_cast<const float4*>(xp);
          y = *reinterpret_cast<const float4*>(yp);
        } else {
          x = make_float4(xp[0], xp[1], xp[2], xp[3]);
          y = make_float4(yp[0], yp[1], yp[2], yp[3]);
        }
      }
      xs[k * P + p] = x.x; xs[(k + 1) * P + p] = x.y; xs[(k + 2) * P + p] = x.z; xs[(k + 3) * P + p] = x.w;
      ys[k * P + p] = y.x; ys[(k + 1) * P + p] = y.y; ys[(k + 2) * P + p] = y.z; ys[(k + 3) * P + p] = y.w;
    }
    __syncthreads();
    const int j0 = w * NC;
    double q[PL], xy[PL];
#pragma unroll
    for (int i = 0; i < PL; i++) q[i] = xy[i] = 0.0;
    // columns in groups of at most eight, so that the running products stay in registers
    constexpr int CG = NC < 8 ? NC : 8;
    for (int jg = j0; jg < j0 + NC; jg += CG) {
      double t1[PL][CG], t2[PL][CG];
#pragma unroll
      for (int i = 0; i < PL; i++)
#pragma unroll
        for (int c = 0; c < CG; c++) t1[i][c] = t2[i][c] = 0.0;
      auto step = [&](int k, auto use1, auto use2) {
        double x[PL], y[PL];
#pragma unroll
        for (int i = 0; i < PL; i += 2) {
          const double2 xv = *reinterpret_cast<const double2*>(xs + k * P + lane * PL + i);
          x[i] = xv.x; x[i + 1] = xv.y;
          if (use2) {
            const double2 yv = *reinterpret_cast<const double2*>(ys + k * P + lane * PL + i);
            y[i] = yv.x; y[i + 1] = yv.y;
          }
        }
#pragma unroll
        for (int c = 0; c < CG; c += 2) {
          const double2 e12 = __ldg(reinterpret_cast<const double2*>(ev + 2 * D * D + k * D + jg + c));
          double2 e1{}, e2{};
          if (use1) e1 = __ldg(reinterpret_cast<const double2*>(ev + k * D + jg + c));
          if (use2) e2 = __ldg(reinterpret_cast<const double2*>(ev + D * D + k * D + jg + c));
#pragma unroll
          for (int i = 0; i < PL; i++) {
            t2[i][c] = fma(x[i], e12.x, t2[i][c]);
            t2[i][c + 1] = fma(x[i], e12.y, t2[i][c + 1]);
            if (use1) { t1[i][c] = fma(x[i], e1.x, t1[i][c]); t1[i][c + 1] = fma(x[i], e1.y, t1[i][c + 1]); }
            if (use2) { t2[i][c] = fma(y[i], e2.x, t2[i][c]); t2[i][c + 1] = fma(y[i], e2.y, t2[i][c + 1]); }
          }
        }
      };
      using yes = integral_constant_t<bool, true>;
      using no = integral_constant_t<bool, false>;
#pragma unroll 2
      for (int k = 0; k < jg; k++) step(k, yes{}, no{});
      for (int k = jg; k < jg + CG; k++) step(k, yes{}, yes{});
#pragma unroll 2
      for (int k = jg + CG; k < D; k++) step(k, no{}, yes{});
#pragma unroll
      for (int c = 0; c < CG; c++)
#pragma unroll
        for (int i = 0; i < PL; i++) {
          const double xj = xs[(jg + c) * P + lane * PL + i], yj = ys[(jg + c) * P + lane * PL + i];
          q[i] = fma(t1[i][c], xj, fma(t2[i][c], yj, q[i]));
          xy[i] = fma(xj, yj, xy[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < PL; i++) {
      red[w * P + lane * PL + i] = q[i];
      red[(8 + w) * P + lane * PL + i] = xy[i];
    }
    __syncthreads();
    const int64_t p = p0 + tid;
    if (tid < P && p < np) {
      double qq = 0.0, dot = 0.0;
#pragma unroll
      for (int i = 0; i < 8; i++) { qq += red[i * P + tid]; dot += red[(8 + i) * P + tid]; }
      const double v = (exp(k0 + qq) - exp(2.0 * dot)) / (double)M;
      var[p] = v;
      if (pooled != nullptr) {
        double s1 = 0.0, s2 = 0.0;
#pragma unroll 8
        for (int r = 0; r < R; r++) s1 += (double)est[(int64_t)r * np + p];
        const double mean = s1 / (double)R;
#pragma unroll 8
        for (int r = 0; r < R; r++) {
          const double dv = (double)est[(int64_t)r * np + p] - mean;
          s2 = fma(dv, dv, s2);
        }
        const double ik2 = exp(-2.0 * dot);
        acc_e += (R > 1 ? s2 / (double)(R - 1) : 0.0) * ik2;
        acc_c += v * ik2;
      }
    }
  }
  if (pooled != nullptr) {
    __syncthreads();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      acc_e += __shfl_xor_sync(0xffffffffu, acc_e, o);
      acc_c += __shfl_xor_sync(0xffffffffu, acc_c, o);
    }
    if (lane == 0) { red[w] = acc_e; red[8 + w] = acc_c; }
    __syncthreads();
    if (tid == 0) {
      double e = 0.0, c = 0.0;
      for (int i = 0; i < NTH / 32; i++) { e += red[i]; c += red[8 + i]; }
      atomicAdd(&pooled[0], e / (double)np);
      atomicAdd(&pooled[1], c / (double)np);
    }
  }
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
         ws_round((3 * (size_t)d * d + 1) * sizeof(double)) + fs_tc_pairs_scratch_bytes(d, M, n);
}

int fs_run_pairs(fsharp_ctx* ctx, const float* X, const float* Y, const float* Omega, const double* params,
                 int64_t npairs, int d, int M, int R, float* est, double* var_cf, double* pooled, WsAlloc* ws) {
  const int batch = draws_per_batch(d, M, R);
  float* prep = ws->take<float>((size_t)batch * 2 * PrepLayout{d, M}.total());
  double* ev = ws->take<double>(3 * (size_t)d * d + 1);
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
    (void)fs_launch_chained(pairvar_prep_kernel, dim3(d), dim3(128), 0, ctx->stream, params, d, ev, ctx->d_status);
    FS_TIME_END(ctx);
    FS_LAUNCH_CHECK(ctx);
    if (pooled) FS_CUDA_OK(cudaMemsetAsync(pooled, 0, 2 * sizeof(double), ctx->stream));
#define FS_PV(DD)                                                                                                       \
  do {                                                                                                                   \
    constexpr int P = DD == 128 ? 64 : 128;                                                                              \
    const size_t smem = (2 * (size_t)DD * P + 16 * P) * sizeof(double);                                                  \
    FS_CUDA_OK(cudaFuncSetAttribute(pairvar_kernel<DD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));         \
    int64_t blocks = (npairs + P - 1) / P;                                                                               \
    const int64_t most = (DD < 64 ? 2 : 1) * (int64_t)ctx->sm_count;                                                     \
    if (blocks > most) blocks = most;                                                                                    \
    FS_TIME_BEGIN(ctx, FS_K_PAIRVAR);                                                                                    \
    (void)fs_launch_chained(pairvar_kernel<DD>, dim3((unsigned)blocks), dim3(NTH), smem, ctx->stream, X, Y, npairs, M, R, ev, est, var_cf, pooled);       \
    FS_TIME_END(ctx);                                                                                                    \
  } while (0)
    switch (d) {
      case 16: FS_PV(16); break;
      case 32: FS_PV(32); break;
      case 64: FS_PV(64); break;
      default: FS_PV(128); break;
    }
#undef FS_PV
    FS_LAUNCH_CHECK(ctx);
  }
  return FSHARP_OK;
}
