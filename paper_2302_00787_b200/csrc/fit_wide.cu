// ADERF / SDERF fits for d = 64 and d = 128 as a chain of kernels, fp64.
//
// One block per matrix for the whole fit (fit.cu) leaves two thirds of the chip idle and walks every phase at one block's
// latency: 217 us (ADERF) / 145 us (SDERF) at d = 64, and 6.7 ms of Jacobi sweeps at d = 128.  Here the sequential phases
// (Cholesky, tridiagonalisation) keep one block per matrix with the matrix in registers, and everything that splits by rows,
// columns or vectors goes to several blocks per matrix:
//   chol      M1 = L L^T and L^-1                                              (ADERF)     1 block
//   zform     Z = L^T M2 L, column blocks                                      (ADERF)     d / SPLIT blocks
//   tridiag   Householder tridiagonalisation of Z, or of N = M1 + mu4 mu5^T + mu5 mu4^T + M2     1 block
//   vectors   16 eigenvalues (multisection on Sturm counts) and vectors (twisted factorisation, reflectors applied back)
//   polish    one first-order symmetric orthogonalisation, Rayleigh quotients, residuals, products with L^-1 and L^T
//   finish    A, B, C, D of the theorems
// Every launch is a programmatic dependent of the one before.  A matrix whose vectors are not orthonormal to 1e-6 before the
// orthogonalisation, or whose residual exceeds 1e-12 of its norm after it (eigenvalues that agree to rounding, a matrix
// that splits), is flagged and fitted by the Jacobi solver of fit.cu instead.
#include "fit_common.cuh"
#include "fit_wide.cuh"
#include "tc_common.cuh"

using namespace fitw;

namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// c += A B for one 8 x 8 x 4 step on the fp64 tensor cores: lane holds A[lane / 4][lane % 4], B[lane % 4][lane / 4] and
// C[lane / 4][2 (lane % 4) + {0, 1}].
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
  asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}
// Product of a block of eight warps, [NR x K] [K x NC] with NR NC = 2048: one 16 x 16 tile per warp, out(row, column, value).
// A step of K = 4 costs a lane four 8-byte loads for the 1024 multiply-adds of its warp; with one output per thread and
// scalar multiply-adds the same work takes five loads per four of them, and the shared-memory pipe is the limit.
// UNROLL: steps whose loads are in flight together (operands in global memory: the latency of the L2).
template <int NR, int NC, int K, int UNROLL = 4, class FA, class FB, class FO>
__device__ __forceinline__ void product8(FA fa, FB fb, FO out) {
  static_assert(NR * NC == 2048, "eight tiles");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lr = lane >> 2, lk = lane & 3;
  const int r0 = warp % (NR / 16) * 16, c0 = warp / (NR / 16) * 16;
  double c[2][2][2] = {};
#pragma unroll UNROLL
  for (int k = 0; k < K; k += 4) {
    const double a0 = fa(r0 + lr, k + lk), a1 = fa(r0 + 8 + lr, k + lk), b0 = fb(k + lk, c0 + lr), b1 = fb(k + lk, c0 + 8 + lr);
    dmma(c[0][0], a0, b0);
    dmma(c[0][1], a0, b1);
    dmma(c[1][0], a1, b0);
    dmma(c[1][1], a1, b1);
  }
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int j = 0; j < 2; j++)
#pragma unroll
      for (int q = 0; q < 2; q++) out(r0 + 8 * i + lr, c0 + 8 * j + 2 * lk + q, c[i][j][q]);
}
// Rows (columns) of a matrix that one block of such products takes, and the leading dimension of a matrix in shared memory:
// 4 mod 16 doubles, so that the 4 x 4 quarters that a half-warp touches fall into different banks.
template <int D> constexpr int SPLIT = 2048 / D;
template <int D> constexpr int LDS_ = D + 4;

// Distribution of a D x D matrix over the registers of a block for the sequential factorisations: sixteen lanes share a row
// (columns part + 16 u), a lane has the four rows h + NH q.  A step then moves D / 16 doubles of a row or vector and four
// row scalars per lane: what a lane receives from shared memory (broadcast or not) is what the pipe is paid in, and four
// lanes per row with all their columns kept it busy for 1.3 k cycles per step.
template <int D> struct Dist {
  static constexpr int NT = 4 * D, NH = NT / 16, NU = D / 16, NQ = 4;
  static_assert(NH * NQ == D, "rows");
};

// ---- Cholesky M1 = L L^T and L^-1 -------------------------------------------------------------------
// By elimination, one column per step, the matrix in registers: the slot of column c of row i holds M1[i][c] while c > j and
// the row of L^-1 (without its scale 1 / l_ii) afterwards; only the pivot row goes through shared memory, and one barrier
// separates two steps.  The unscaled columns of L are collected in shared memory and leave at the end.
template <int D> constexpr size_t chol_smem() { return (size_t)D * (D + 1) * sizeof(double); }
template <int D>
__global__ void __launch_bounds__(Dist<D>::NT)
chol_kernel(const double* __restrict__ stats, double ridge, double* __restrict__ scratch, int* __restrict__ status) {
  fs_grid_dependency_wait();
  constexpr int NT = Dist<D>::NT, NH = Dist<D>::NH, NU = Dist<D>::NU, NQ = Dist<D>::NQ, LD = D + 1;
  extern __shared__ __align__(16) double sl[];          // [D][LD]: a_ij at the step that eliminates column j
  __shared__ double rowbuf[2][D], tr[D], pv[D];
  const int g = blockIdx.x, tid = threadIdx.x, part = tid & 15, h = tid >> 4;
  const double* M1 = stats + (size_t)g * StatsLayout{D}.total() + StatsLayout{D}.M(1);
  double* sc = scratch + (size_t)g * Layout{D}.total();
  double a[NQ][NU];
#pragma unroll
  for (int q = 0; q < NQ; q++)
#pragma unroll
    for (int u = 0; u < NU; u++) a[q][u] = M1[(h + NH * q) * D + part + 16 * u];
  if (tid < D) tr[tid] = M1[tid * D + tid];
  __syncthreads();
  double t1 = 0.0;
  for (int i = 0; i < D; i++) t1 += tr[i];             // (broadcast reads)
  const double rg1 = ridge * t1 / D, floor_piv = 1e-12 * (t1 + D * rg1) / D;
#pragma unroll
  for (int q = 0; q < NQ; q++)
#pragma unroll
    for (int u = 0; u < NU; u++)
      if (part + 16 * u == h + NH * q) a[q][u] += rg1;
  if (h == 0)
#pragma unroll
    for (int u = 0; u < NU; u++) rowbuf[0][part + 16 * u] = a[0][u];
  __syncthreads();
  bool raised = false;
  for (int j = 0; j < D; j++) {
    const double* rb = rowbuf[j & 1];
    double* nb = rowbuf[(j + 1) & 1];
    double piv = rb[j], p[NU], f[NQ];
#pragma unroll
    for (int u = 0; u < NU; u++) p[u] = rb[part + 16 * u];
#pragma unroll
    for (int q = 0; q < NQ; q++) f[q] = rb[h + NH * q];  // M1[i][j] = M1[j][i]
    if (!(piv > floor_piv)) { raised = true; piv = floor_piv + 1e-300; }
    if (tid == 0) pv[j] = piv;
    const double rp = recip_fast(piv);
    const int qn = (j + 1) / NH;
#pragma unroll
    for (int q = 0; q < NQ; q++) {
      if (NH * q + NH - 1 <= j) continue;               // (rows of this slot are all done)
      const int i = h + NH * q;
      if (i > j && part == (j & 15)) sl[i * LD + j] = f[q];
      const double m = i > j ? -f[q] * rp : 0.0;
#pragma unroll
      for (int u = 0; u < NU; u++) a[q][u] = part + 16 * u == j && i > j ? m : fma(m, p[u], a[q][u]);     // W[j][j] = 1
      if (q == qn && i == j + 1)
#pragma unroll
        for (int u = 0; u < NU; u++) nb[part + 16 * u] = a[q][u];
    }
    __syncthreads();
  }
  double* rs = tr;
  if (tid < D) rs[tid] = rsqrt_fast(pv[tid]);           // 1 / l_jj
  __syncthreads();
  double* Li = sc + Layout{D}.Li();
  double* L = sc + Layout{D}.L();
  double* LT = sc + Layout{D}.LT();
#pragma unroll
  for (int q = 0; q < NQ; q++) {
    const int i = h + NH * q;
    const double ri = rs[i];
#pragma unroll
    for (int u = 0; u < NU; u++) {
      const int c = part + 16 * u;
      Li[i * D + c] = c > i ? 0.0 : (c == i ? ri : a[q][u] * ri);
    }
  }
  for (int e = tid; e < D * D; e += NT) {
    const int i = e / D, c = e % D;
    L[e] = c > i ? 0.0 : (c == i ? pv[c] : sl[i * LD + c]) * rs[c];
    LT[e] = i > c ? 0.0 : (c == i ? pv[c] : sl[c * LD + i]) * rs[i];
  }
  if (raised) atomicExch(status, FSHARP_E_CONSTRAINT);
}

// ---- Z = L^T (M2 L), SPLIT columns per block -----------------------------------------------------------------
constexpr int PR_THREADS = 256;
template <int D>
__global__ void __launch_bounds__(PR_THREADS)
zform_kernel(const double* __restrict__ stats, double ridge, double* __restrict__ scratch) {
  fs_grid_dependency_wait();
  constexpr int CB = SPLIT<D>, LB = CB + 4;
  __shared__ __align__(16) double lc[D * LB], t1[D * LB];
  __shared__ double tr[D];
  const int g = blockIdx.x, c0 = blockIdx.y * CB, tid = threadIdx.x;
  const double* M2 = stats + (size_t)g * StatsLayout{D}.total() + StatsLayout{D}.M(2);
  double* sc = scratch + (size_t)g * Layout{D}.total();
  const double* L = sc + Layout{D}.L();
#pragma unroll 8
  for (int e = tid; e < D * CB; e += PR_THREADS) lc[(e / CB) * LB + e % CB] = L[(e / CB) * D + c0 + e % CB];
  if (tid < D) tr[tid] = M2[tid * D + tid];
  __syncthreads();
  double t2 = 0.0;
  for (int k = 0; k < D; k++) t2 += tr[k];
  const double rg2 = ridge * t2 / D;
  product8<D, CB, D, 16>([&](int r, int k) { return M2[r * D + k]; }, [&](int k, int c) { return lc[k * LB + c]; },
                         [&](int r, int c, double v) { t1[r * LB + c] = fma(rg2, lc[r * LB + c], v); });
  __syncthreads();
  double* Z = sc + Layout{D}.V();                       // (free until the vectors are formed)
  product8<D, CB, D, 16>([&](int r, int k) { return L[k * D + r]; }, [&](int k, int c) { return t1[k * LB + c]; },
                         [&](int r, int c, double v) { Z[r * D + c0 + c] = v; });
}

// ---- A -> Q^T A Q = T (tridiagonal) -----------------------------------------------------------------------
// Reflector k, I - beta_k v v^T with v = x - alpha e_1, acts on indices k+1..D-1 (x: column k below the diagonal).  With A22
// the trailing block, y = A22 x and n = A22 e_1 (its first column):
//   p = beta A22 v = beta (y - alpha n),   v.p = beta (x.y - 2 alpha y_1 + alpha^2 n_1),   w = p - (beta/2 v.p) v,
//   A22 -= v w^T + w v^T
// One barrier per step: y, n and x.y (as the sum of x_r a_rc x_c) cross the block together, |x|^2, alpha and beta are worked out
// by every group of lanes on its own copy of x, and the next x, row k + 1 of the updated block, follows from n, v and w
// without asking its owners.  What bounds a step is its chain of reductions and exchanges and the shared-memory pipe, which
// is paid for what every lane receives: P lanes share a row (eight columns part + P u each), a lane has NQ rows h + 16 q, and
// the block is as small as the registers allow.  (Sixteen lanes per row and twice the threads: 1.7 k cycles per step at
// d = 64.)  The loop over k is cut where a slot of columns is used up, so that the work shrinks with the block.
template <int D> struct Tri {
  static constexpr int NU = 8, P = D / NU, NG = 16, NT = NG * P, NQ = D / NG, NW = NT / 32;
  static_assert(P == 2 * NQ && NG * NQ == D, "distribution");
};
template <int D>
struct TriState {
  double a[Tri<D>::NQ][Tri<D>::NU];                     // the own part of the matrix
  double xv[Tri<D>::NU], xr[Tri<D>::NQ];                // x at the own columns and rows, zero up to index k
  double x0, alpha, beta;
};

// Step k begins: x is in the registers; alpha, beta; y, n and the partial sums of x.y go out.  UB: first slot in use.
template <int D, int UB>
__device__ __forceinline__ void tri_begin(TriState<D>& s, int k, double2* __restrict__ yn, double* __restrict__ pt, int part, int h, int lane, int warp) {
  constexpr int NU = Tri<D>::NU, P = Tri<D>::P, NQ = Tri<D>::NQ, U1 = UB + 1 < NU ? UB + 1 : UB;
  constexpr int Q0 = P * UB >= 15 ? (P * UB - 15 + 15) / 16 : 0;       // first row slot in use
  const bool second = k + 1 >= P * (UB + 1);            // column k + 1 lies in slot UB + 1
  const int pk = (k + 1) & (P - 1);
  s.x0 = __shfl_sync(0xffffffffu, second ? s.xv[U1] : s.xv[UB], pk, P);
  double y[NQ], s2 = 0.0, t = 0.0;
#pragma unroll
  for (int q = 0; q < NQ; q++) y[q] = 0.0;
#pragma unroll
  for (int u = UB; u < NU; u++) {
    const double x = (u == UB || u == UB + 1) && part + P * u == k + 1 ? 0.0 : s.xv[u];
    s2 = fma(x, x, s2);
#pragma unroll
    for (int q = Q0; q < NQ; q++) y[q] = fma(s.a[q][u], s.xv[u], y[q]);
  }
  if (part == pk) {
#pragma unroll
    for (int q = Q0; q < NQ; q++) yn[h + 16 * q].y = second ? s.a[q][U1] : s.a[q][UB];
  }
#pragma unroll
  for (int q = Q0; q < NQ; q++) t = fma(s.xr[q], y[q], t);
  // NQ sums over P lanes: every exchange but the last halves the number of values a lane keeps
  int row = 0;
#pragma unroll
  for (int n = NQ / 2, o = P / 2; n >= 1; n >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < NQ / 2; i++) {
      if (i < n) {
        const double give = up ? y[i] : y[i + n], keep = up ? y[i + n] : y[i];
        y[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
    row += up ? n : 0;
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  y[0] += __shfl_xor_sync(0xffffffffu, y[0], 1);
  s2 += __shfl_xor_sync(0xffffffffu, s2, 1);
  if ((lane & 1) == 0) yn[h + 16 * row].x = y[0];
  t = warp_sum(t);
  if (lane == 0) pt[warp] = t;
  s.alpha = s.x0;
  s.beta = 0.0;
  if (s2 > 0.0) {
    const double nrm2 = fma(s.x0, s.x0, s2);
    const double anorm = nrm2 * rsqrt_fast(nrm2);                   // |x|
    s.alpha = -copysign(anorm, s.x0);
    s.beta = recip_fast(fma(fabs(s.x0), anorm, nrm2));              // 2 / |v|^2 = 1 / (|x|^2 + |x_0| |x|)
  }
}

// Step k ends (after the barrier): the update, and the next x.
template <int D, int UB>
__device__ __forceinline__ void tri_end(TriState<D>& s, int k, const double2* __restrict__ yn, const double* __restrict__ pt, double* __restrict__ diag,
                                        double* __restrict__ rf, int part, int h) {
  constexpr int NU = Tri<D>::NU, P = Tri<D>::P, NQ = Tri<D>::NQ, NW = Tri<D>::NW;
  constexpr int Q0 = P * UB >= 15 ? (P * UB - 15 + 15) / 16 : 0;
  const double alpha = s.alpha, b = s.beta;
  const double2 yn0 = yn[k + 1];
  double2 c[NU], r[NQ];
#pragma unroll
  for (int u = UB; u < NU; u++) c[u] = yn[part + P * u];
#pragma unroll
  for (int q = Q0; q < NQ; q++) r[q] = yn[h + 16 * q];
  double sxy = 0.0;
#pragma unroll
  for (int w = 0; w < NW; w += 2) {
    const double2 p = *reinterpret_cast<const double2*>(pt + w);
    sxy += p.x + p.y;
  }
  const double kk = 0.5 * b * b * fma(alpha, fma(alpha, yn0.y, -2.0 * yn0.x), sxy);
  const double v0 = s.x0 - alpha, w0 = fma(-kk, v0, b * fma(-alpha, yn0.y, yn0.x));
  if (h == Tri<D>::NG - 1) {
#pragma unroll
    for (int u = 0; u < NU; u++) rf[part + P * u] = u < UB ? 0.0 : (part + P * u == k + 1 ? v0 : s.xv[u]);
  }
  if (h == 0 && part == 0) {
    diag[k + 1] = fma(-2.0 * v0, w0, yn0.y);
    diag[D + k] = alpha;
    diag[2 * D + k] = b;
  }
  double vr[NQ], wr[NQ];
#pragma unroll
  for (int q = Q0; q < NQ; q++) {
    const int i = h + 16 * q;
    vr[q] = i == k + 1 ? v0 : s.xr[q];
    wr[q] = i > k ? fma(-kk, vr[q], b * fma(-alpha, r[q].y, r[q].x)) : 0.0;
    s.xr[q] = i > k + 1 ? fma(-v0, wr[q], fma(-w0, vr[q], r[q].y)) : 0.0;
  }
#pragma unroll
  for (int u = UB; u < NU; u++) {
    const int j = part + P * u;
    const double vc = j == k + 1 ? v0 : s.xv[u];
    const double wc = j > k ? fma(-kk, vc, b * fma(-alpha, c[u].y, c[u].x)) : 0.0;
    s.xv[u] = j > k + 1 ? fma(-v0, wc, fma(-w0, vc, c[u].y)) : 0.0;
#pragma unroll
    for (int q = Q0; q < NQ; q++) s.a[q][u] = fma(-vr[q], wc, fma(-wr[q], vc, s.a[q][u]));
  }
}

template <int D, int UB, class Bar>
__device__ __forceinline__ void tri_blocks(TriState<D>& s, double2 (*yn)[D], double (*pt)[Tri<D>::NW], double* diag, double* rf, int part, int h, int lane, int warp, Bar bar) {
  constexpr int P = Tri<D>::P, K1 = P * (UB + 1) < D - 2 ? P * (UB + 1) : D - 2;
#pragma unroll 1
  for (int k = P * UB; k < K1; k++) {
    bar();
    tri_end<D, UB>(s, k, yn[k & 1], pt[k & 1], diag, rf + (size_t)k * D, part, h);
    if (k < D - 3) tri_begin<D, UB>(s, k + 1, yn[(k + 1) & 1], pt[(k + 1) & 1], part, h, lane, warp);
  }
  if constexpr (UB + 1 < Tri<D>::NU) tri_blocks<D, UB + 1>(s, yn, pt, diag, rf, part, h, lane, warp, bar);
}

template <int D>
__global__ void __launch_bounds__(Tri<D>::NT)
tridiag_kernel(const double* __restrict__ stats, int variant, double ridge, double* __restrict__ scratch, int* __restrict__ status) {
  fs_grid_dependency_wait();
  constexpr int NT = Tri<D>::NT, NU = Tri<D>::NU, P = Tri<D>::P, NQ = Tri<D>::NQ, NW = Tri<D>::NW;
  __shared__ __align__(16) double2 yn[2][D];
  __shared__ __align__(16) double pt[2][NW];
  __shared__ double mu[2][D], red[5][NW], row0[D];
  const int g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, part = tid & (P - 1), h = tid / P;
  const StatsLayout sl{D};
  const double* st = stats + (size_t)g * sl.total();
  double* sc = scratch + (size_t)g * Layout{D}.total();
  const double* Z = sc + Layout{D}.V();
  double* A0 = sc + Layout{D}.A0();
  double* diag = sc + Layout{D}.diag();
  // traces, mu4 . mu5, finiteness
  double t1 = 0.0, t2 = 0.0, mm = 0.0, bad = 0.0, tot = 0.0;
  if (tid < D) {
    t1 = st[sl.M(1) + tid * D + tid];
    t2 = st[sl.M(2) + tid * D + tid];
    const double a = st[sl.mu(4) + tid], b = st[sl.mu(5) + tid];
    mm = a * b;
    mu[0][tid] = a;
    mu[1][tid] = b;
  }
  // (one double per load: a caller's statistics are aligned to 8 bytes, no more)
#pragma unroll 32
  for (int e = tid; e < (int)sl.total(); e += NT)
    if (!isfinite(st[e])) bad = 1.0;
  t1 = warp_sum(t1); t2 = warp_sum(t2); mm = warp_sum(mm); bad = warp_sum(bad);
  if (lane == 0) { red[0][warp] = t1; red[1][warp] = t2; red[2][warp] = mm; red[3][warp] = bad; }
  __syncthreads();
  t1 = t2 = mm = bad = 0.0;
  for (int w = 0; w < NW; w++) { t1 += red[0][w]; t2 += red[1][w]; mm += red[2][w]; bad += red[3][w]; }
  const double rg1 = ridge * t1 / D, rg2 = ridge * t2 / D;
  TriState<D> s;
  // (the two reads of an element are of opposite order in memory: their sums are the same bits for (r, c) and (c, r))
#pragma unroll
  for (int q = 0; q < NQ; q++)
#pragma unroll
    for (int u = 0; u < NU; u++) {
      const int r = h + 16 * q, c = part + P * u;
      double v;
      if (variant == FSHARP_ADERF) v = 0.5 * (Z[r * D + c] + Z[c * D + r]);
      else v = st[sl.M(1) + r * D + c] + st[sl.M(2) + r * D + c] + mu[0][r] * mu[1][c] + mu[1][r] * mu[0][c] + (r == c ? rg1 + rg2 : 0.0);
      s.a[q][u] = v;
      A0[r * D + c] = v;
      tot = fma(v, v, tot);
      if (r == 0) row0[c] = v;
    }
  tot = warp_sum(tot);
  if (lane == 0) red[4][warp] = tot;
  __syncthreads();
  if (tid == 0) {
    double sum = 0.0;
    for (int w = 0; w < NW; w++) sum += red[4][w];
    double* o = sc + Layout{D}.scal();
    o[FS_T1] = t1 + D * rg1;
    o[FS_T2] = t2 + D * rg2;
    o[FS_MM] = mm;
    o[FS_TOT] = sum;
    o[FS_FLAG] = 0.0;
    diag[0] = row0[0];
    if (bad > 0.0) atomicExch(status, FSHARP_E_NONFINITE);
  }
#pragma unroll
  for (int u = 0; u < NU; u++) s.xv[u] = part + P * u > 0 ? row0[part + P * u] : 0.0;
#pragma unroll
  for (int q = 0; q < NQ; q++) s.xr[q] = h + 16 * q > 0 ? row0[h + 16 * q] : 0.0;
  tri_begin<D, 0>(s, 0, yn[0], pt[0], part, h, lane, warp);
  tri_blocks<D, 0>(s, yn, pt, diag, sc + Layout{D}.RF(), part, h, lane, warp, [] { __syncthreads(); });
  // what is left: rows D - 2 (in xv) and D - 1
  if (tid == NT - 1) {
    diag[D - 1] = s.a[NQ - 1][NU - 1];
    diag[D + D - 2] = s.xv[NU - 1];
    diag[D + D - 1] = 0.0;
  }
}

// ---- 16 eigenvalues and vectors per block, eight lanes per vector --------------------------------------------------
// (A warp per vector needs five instead of eight multisection steps per 16 bits, but nearly three times the Sturm counts: with
// 4 x 48 blocks on the chip their fp64 throughput is the limit.)
constexpr int VC_THREADS = 128, VP = 8;
template <int D> constexpr size_t vectors_smem() { return ((size_t)(D - 2) * D + 16 * (2 * D + 2)) * sizeof(double); }
template <int D>
__global__ void __launch_bounds__(VC_THREADS)
vectors_kernel(int variant, double* __restrict__ scratch, int* __restrict__ status) {
  fs_grid_dependency_wait();
  constexpr int NU = D / VP;
  extern __shared__ __align__(16) double smv[];
  double* rf = smv;                                     // [D - 2][D] reflectors
  __shared__ __align__(16) double2 de[D];               // (d_i, e_{i-1}^2), scaled
  __shared__ double dd[D], ee[D], beta[D], bounds[2][VC_THREADS / 32];
  __shared__ int cnt[VC_THREADS];
  __shared__ uint64_t rf_full;
  __shared__ int abort_flag;
  const int g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, vec = tid / VP, part = tid % VP, r = blockIdx.y * 16 + vec;
  auto gsum = [](double v) {
#pragma unroll
    for (int o = VP >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  double* sc = scratch + (size_t)g * Layout{D}.total();
  const double* diag = sc + Layout{D}.diag();
  // the reflectors arrive under the search for the eigenvalues
  if (tid == 0) {
    tc::mbar_init(&rf_full, 1);
    abort_flag = 0;
    tc::fence_barrier_init();
    tc::mbar_expect_tx(&rf_full, (D - 2) * D * 8);
    tc::bulk_load(rf, sc + Layout{D}.RF(), (D - 2) * D * 8, &rf_full);
  }
  double* Lp = smv + (size_t)(D - 2) * D + vec * (2 * D + 2);  // P+, then l+, then the vector
  double* Lm = Lp + D;                                    // P-, then l-
  // Gershgorin interval; T is scaled by a power of two so that it is of order one (the vectors do not change)
  double lo = 1e300, hi = -1e300;
  if (tid < D) {
    const double rad = fabs(diag[D + tid]) + (tid > 0 ? fabs(diag[D + tid - 1]) : 0.0);
    lo = diag[tid] - rad;
    hi = diag[tid] + rad;
    beta[tid] = tid < D - 2 ? diag[2 * D + tid] : 0.0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) { bounds[0][warp] = lo; bounds[1][warp] = hi; }
  __syncthreads();
  for (int w = 0; w < VC_THREADS / 32; w++) { lo = fmin(lo, bounds[0][w]); hi = fmax(hi, bounds[1][w]); }
  const double nrm = fmax(fabs(lo), fabs(hi));
  if (!(nrm > 1e-290) || !(nrm < 1e290)) {              // zero, non-finite or absurdly scaled: the fall-back takes it
    if (tid == 0) sc[Layout{D}.scal() + FS_FLAG] = 1.0;
    tc::mbar_wait(&rf_full, 0, &abort_flag, status, false);
    return;
  }
  const int nex = ((__double2hiint(nrm) >> 20) & 0x7ff) - 1023;
  const double scale = __hiloint2double((1023 - nex) << 20, 0);       // 2^-nex: nrm * scale in [1, 2)
  if (tid < D) {
    const double ep = tid > 0 ? diag[D + tid - 1] * scale : 0.0;
    dd[tid] = diag[tid] * scale;
    ee[tid] = diag[D + tid] * scale;
    de[tid] = make_double2(diag[tid] * scale, ep * ep);
  }
  __syncthreads();
  lo *= scale; hi *= scale;
  // Number of eigenvalues below x: sign changes along the leading principal minors p_i of T - x I,
  // p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2}, p_{-1} = 1.  The pair of minors is brought back to order one
  // every eight steps.
  auto below = [&](double x) {
    double pm2 = 1.0, pm1 = de[0].x - x;
    int c = (unsigned)__double2hiint(pm1) >> 31;
#pragma unroll 8
    for (int i = 1; i < D; i++) {
      const double2 t = de[i];
      const double p = fma(t.x - x, pm1, -(t.y * pm2));
      c += (unsigned)(__double2hiint(p) ^ __double2hiint(pm1)) >> 31;
      pm2 = pm1; pm1 = p;
      if ((i & 7) == 0) {
        const int ex = max((__double2hiint(pm1) >> 20) & 0x7ff, (__double2hiint(pm2) >> 20) & 0x7ff);
        if (ex > 0 && ex < 0x7fe) {
          const double s = __hiloint2double((2046 - ex) << 20, 0);
          pm1 *= s; pm2 *= s;
        }
      }
    }
    return c;
  };
  double sigma;
  {
    // a grid of 512 points over the whole interval: every fourth by one thread each, the three between by this group's lanes;
    // then VP points per step inside this group's bracket, to 2^-50.  (Where the spectrum is so crowded that the vectors fail the
    // check below, the precision of sigma decides it, and with it which solver's order of rows a caller gets: the points are
    // those of the one-block kernel in fit.cu.)
    double a = lo - 0.001 * (hi - lo) - 1e-3, b = hi + 0.001 * (hi - lo) + 1e-3;
    constexpr int GRID = 4 * VC_THREADS;
    const double h0 = (b - a) * (1.0 / (GRID + 1));
    cnt[tid] = below(fma(h0, (double)(4 * tid + 4), a));
    __syncthreads();
    int lo_i = 0, hi_i = VC_THREADS;                    // first of these points with more than r eigenvalues below it
    while (lo_i < hi_i) {
      const int mid = (lo_i + hi_i) >> 1;
      if (cnt[mid] >= r + 1) hi_i = mid; else lo_i = mid + 1;
    }
    const int g0 = 4 * lo_i;                            // points g0 .. g0 + 2 of the grid lie below point g0 + 3
    const bool under = part < 3 && g0 + part < GRID && below(fma(h0, (double)(g0 + part + 1), a)) >= r + 1;
    const unsigned m3 = (__ballot_sync(0xffffffffu, under) >> (lane & ~(VP - 1))) & 7u;
    const int gi = lo_i < VC_THREADS ? g0 + (m3 ? __ffs(m3) - 1 : 3) : GRID;        // first point of the grid with more than r below
    const double na = gi > 0 ? fma(h0, (double)gi, a) : a;
    b = gi < GRID ? fma(h0, (double)(gi + 1), a) : b;
    a = na;
    for (int it = 0; it < 13; it++) {
      const double h = (b - a) * (1.0 / (VP + 1)), x = fma(h, (double)(part + 1), a);
      const unsigned mask = (__ballot_sync(0xffffffffu, below(x) >= r + 1) >> (lane & ~(VP - 1))) & ((1u << VP) - 1u);
      const int first = mask ? __ffs(mask) - 1 : VP;    // first point with the r-th eigenvalue below it
      const double ma = first > 0 ? fma(h, (double)first, a) : a;
      b = first < VP ? fma(h, (double)(first + 1), a) : b;
      a = ma;
    }
    sigma = 0.5 * (a + b);
  }
  // Eigenvector of T for sigma from the twisted factorisation.  With P+_i the leading and P-_i the trailing principal minors
  // of T - sigma I (P+_{-1} = P-_D = 1), the pivots of the elimination from the top and from the bottom are
  // D+_i = P+_i / P+_{i-1} and D-_i = P-_i / P-_{i+1}, and gamma_i = D+_i + D-_i - (d_i - sigma).  The vector starts with 1 at
  // the index of the smallest |gamma| and runs outwards: z_i = -l+_i z_{i+1} with l+_i = e_i / D+_i,
  // z_{i+1} = -l-_{i+1} z_i with l-_i = e_{i-1} / D-_i.  Two lanes run the two recurrences; the minors are rescaled every
  // eight steps by powers of two, whose exponents the quotients take into account.  A minor that is exactly zero gives a
  // non-finite vector, which the orthogonality check rejects.
  __shared__ int exps[16][2][D / 8], cums[16][2][D / 8];      // [q]: exponent taken out before step 8 q + 1; their sums
  if (part < 2) {
    const bool fwd = part == 0;
    double* out = fwd ? Lp : Lm;
    const int i0 = fwd ? 0 : D - 1, di = fwd ? 1 : -1;
    double pm2 = 1.0, pm1 = de[i0].x - sigma;
    out[i0] = pm1;
    int* ex_out = exps[vec][part];
    int* cum_out = cums[vec][part];
    ex_out[0] = cum_out[0] = 0;
    int cum = 0;
    for (int s0 = 1; s0 < D; s0 += 8) {                 // eight steps' operands are loaded ahead of the chain
      double dv[8], ev[8], pv[8];
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int i = i0 + di * (s0 + q);
        const bool in = s0 + q < D;
        dv[q] = in ? de[i].x - sigma : 0.0;
        ev[q] = in ? de[fwd ? i : i + 1].y : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 8; q++) {
        pv[q] = fma(dv[q], pm1, -(ev[q] * pm2));
        pm2 = pm1; pm1 = pv[q];
      }
#pragma unroll
      for (int q = 0; q < 8; q++)
        if (s0 + q < D) out[i0 + di * (s0 + q)] = pv[q];
      const int ex = max((__double2hiint(pm1) >> 20) & 0x7ff, (__double2hiint(pm2) >> 20) & 0x7ff);
      int sh = 0;
      if (ex > 0 && ex < 0x7fe) {
        sh = 1023 - ex;
        const double s = __hiloint2double((1023 + sh) << 20, 0);
        pm1 *= s; pm2 *= s;
      }
      cum += sh;
      if (s0 + 8 < D) {                                 // the minors from step s0 + 8 on carry 2^sh against those before
        ex_out[(s0 + 8) >> 3] = sh;
        cum_out[(s0 + 8) >> 3] = cum;
      }
    }
  }
  __syncwarp();
  // First steps of the recurrences whose minors, without the rescaling, leave the range of normal numbers.  At d = 64 such a
  // minor of an ADERF fit counts as zero: many crowded eigenvalues then go to the Jacobi solver, whose order of the rows of B
  // (Theorem 4.2 leaves it free; here it is that of the eigenvalues) is what callers get for such spectra.  The first of them
  // still takes part in the choice of the starting index, with the bits it has as a subnormal number.
  auto subnormal = [](double v, int cum) {
    const int k = min(max(1074 - cum, -1000), 1000);    // v 2^-cum in units of 2^-1074
    return rint(v * __hiloint2double((1023 + k) << 20, 0)) * __hiloint2double((1023 - k) << 20, 0);
  };
  int deadf = D, deadb = D;
  if (D == 64 && variant == FSHARP_ADERF) {
#pragma unroll
    for (int u = 0; u < NU; u++) {
      const int i = part + VP * u, sf = i, sb = D - 1 - i;
      const int ef = ((__double2hiint(Lp[i]) >> 20) & 0x7ff) - cums[vec][0][sf > 0 ? (sf - 1) >> 3 : 0];
      const int eb = ((__double2hiint(Lm[i]) >> 20) & 0x7ff) - cums[vec][1][sb > 0 ? (sb - 1) >> 3 : 0];
      if (ef < 1) deadf = min(deadf, sf);
      if (eb < 1) deadb = min(deadb, sb);
    }
#pragma unroll
    for (int o = VP >> 1; o > 0; o >>= 1) {
      deadf = min(deadf, __shfl_xor_sync(0xffffffffu, deadf, o));
      deadb = min(deadb, __shfl_xor_sync(0xffffffffu, deadb, o));
    }
  }
  double gbest = 1e300;
  int ibest = 0;
  {
    double lp[NU], lm[NU];
#pragma unroll
    for (int u = 0; u < NU; u++) {
      const int i = part + VP * u;
      // step numbers: forward s = i, backward s = D - 1 - i; a step s = 1 mod 8, s > 1, divides by a minor of the block before
      const int sf = i, sb = D - 1 - i;
      double pp = Lp[i], pq = Lm[i];
      double ppm = i > 0 ? Lp[i - 1] : 1.0, pqp = i < D - 1 ? Lm[i + 1] : 1.0;
      if (sf > 1 && (sf & 7) == 1) ppm *= __hiloint2double((1023 + exps[vec][0][sf >> 3]) << 20, 0);
      if (sb > 1 && (sb & 7) == 1) pqp *= __hiloint2double((1023 + exps[vec][1][sb >> 3]) << 20, 0);
      const double rp = recip_fast(pp), rq = recip_fast(pq);
      lp[u] = ee[i] * ppm * rp;                         // l+_i (unused for i = D - 1: e = 0)
      lm[u] = (i > 0 ? ee[i - 1] : 0.0) * pqp * rq;     // l-_i
      if (sf == deadf) pp = subnormal(pp, cums[vec][0][sf > 0 ? (sf - 1) >> 3 : 0]);
      if (sb == deadb) pq = subnormal(pq, cums[vec][1][sb > 0 ? (sb - 1) >> 3 : 0]);
      const double gm = fabs(fma(pp, recip_fast(ppm), fma(pq, recip_fast(pqp), -(dd[i] - sigma))));
      if (sf >= deadf) lp[u] = __longlong_as_double(-1ll);           // NaN: the check below rejects a vector that uses it
      if (sb >= deadb) lm[u] = __longlong_as_double(-1ll);
      if (gm < gbest && sf <= deadf && sb <= deadb) { gbest = gm; ibest = i; }        // NaN never wins
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < NU; u++) {
      Lp[part + VP * u] = lp[u];
      Lm[part + VP * u] = lm[u];
    }
  }
#pragma unroll
  for (int o = VP >> 1; o > 0; o >>= 1) {
    const double go = __shfl_xor_sync(0xffffffffu, gbest, o);
    const int io = __shfl_xor_sync(0xffffffffu, ibest, o);
    if (go < gbest || (go == gbest && io < ibest)) { gbest = go; ibest = io; }
  }
  __syncwarp();
  double zz = 0.0;
  if (part < 2) {
    const bool up = part == 0;
    const double* mul = up ? Lp : Lm;
    const int di = up ? -1 : 1, steps = up ? ibest : D - 1 - ibest;
    double z = 1.0;
    zz = up ? 1.0 : 0.0;
    for (int s0 = 1; s0 <= steps; s0 += 8) {
      double mv[8], zv[8];
#pragma unroll
      for (int q = 0; q < 8; q++) mv[q] = s0 + q <= steps ? mul[ibest + di * (s0 + q)] : 0.0;
#pragma unroll
      for (int q = 0; q < 8; q++) {
        z = -mv[q] * z;
        zv[q] = z;
        zz = fma(z, z, zz);
      }
#pragma unroll
      for (int q = 0; q < 8; q++)
        if (s0 + q <= steps) Lp[ibest + di * (s0 + q)] = zv[q];
    }
  }
  __syncwarp();
  if (part == 0) Lp[ibest] = 1.0;
  zz = gsum(zz);
  __syncwarp();
  const double zn = rsqrt(zz);
  double z[NU];
#pragma unroll
  for (int u = 0; u < NU; u++) z[u] = Lp[part + VP * u] * zn;
  // Eigenvector of A = Q z: the reflectors in reverse order, the next one's loads ahead of the current one's reduction
  tc::mbar_wait(&rf_full, 0, &abort_flag, status, false);
  __syncwarp();
  double vi[NU];
#pragma unroll
  for (int u = 0; u < NU; u++) vi[u] = rf[(size_t)(D - 3) * D + part + VP * u];
  for (int k = D - 3; k >= 0; k--) {
    const double b = beta[k];
    const double* next = rf + (size_t)max(k - 1, 0) * D; // (a reflector is zero up to index k)
    double nv[NU], da = 0.0, db = 0.0;
#pragma unroll
    for (int u = 0; u < NU; u += 2) {
      da = fma(vi[u], z[u], da);
      db = fma(vi[u + 1], z[u + 1], db);
    }
#pragma unroll
    for (int u = 0; u < NU; u++) nv[u] = next[part + VP * u];
    const double dot = gsum(da + db) * b;
#pragma unroll
    for (int u = 0; u < NU; u++) {
      z[u] = fma(-dot, vi[u], z[u]);
      vi[u] = nv[u];
    }
  }
  double* V = sc + Layout{D}.V() + (size_t)r * D;
#pragma unroll
  for (int u = 0; u < NU; u++) V[part + VP * u] = z[u];
}

// ---- orthogonalisation, Rayleigh quotients, residuals; SPLIT rows of V per block -----------------------------------
template <int D> constexpr size_t polish_smem() { return ((size_t)D + 2 * SPLIT<D>) * LDS_<D> * sizeof(double); }
template <int D>
__global__ void __launch_bounds__(PR_THREADS)
polish_kernel(int variant, double* __restrict__ scratch) {
  fs_grid_dependency_wait();
  constexpr int R = SPLIT<D>, LD = LDS_<D>;
  extern __shared__ __align__(16) double smv[];
  double* vs = smv;                                     // [D][LD] all vectors
  double* gs = vs + D * LD;                             // [R][LD]: G = V V^T - I, later V' A
  double* vp = gs + R * LD;                             // [R][LD]: V'
  const int g = blockIdx.x, r0 = blockIdx.y * R, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* sc = scratch + (size_t)g * Layout{D}.total();
  double* flag = sc + Layout{D}.scal() + FS_FLAG;
  {
    const double2* V = reinterpret_cast<const double2*>(sc + Layout{D}.V());
#pragma unroll 8
    for (int e = tid; e < D * D / 2; e += PR_THREADS) *reinterpret_cast<double2*>(vs + (2 * e / D) * LD + 2 * e % D) = V[e];
  }
  __syncthreads();
  double gmax = 0.0;
  product8<R, D, D>([&](int r, int k) { return vs[(r0 + r) * LD + k]; }, [&](int k, int c) { return vs[c * LD + k]; },
                    [&](int r, int c, double v) {
                      v -= r0 + r == c ? 1.0 : 0.0;
                      gs[r * LD + c] = v;
                      gmax = fmax(gmax, isfinite(v) ? fabs(v) : 1e300);
                    });
  if (!(gmax <= 1e-6)) *flag = 1.0;                     // (several threads may write the same value)
  __syncthreads();
  // V' = (I - G / 2) V: orthonormal to second order in G
  double* Vo = sc + Layout{D}.RF();                     // (the reflectors are no longer needed)
  product8<R, D, D>([&](int r, int k) { return gs[r * LD + k]; }, [&](int k, int c) { return vs[k * LD + c]; },
                    [&](int r, int c, double v) {
                      v = fma(-0.5, v, vs[(r0 + r) * LD + c]);
                      vp[r * LD + c] = v;
                      Vo[(size_t)(r0 + r) * D + c] = v;
                    });
  __syncthreads();
  const double* A0 = sc + Layout{D}.A0();
  auto rows = [&](int r, int k) { return vp[r * LD + k]; };
  product8<R, D, D, 16>(rows, [&](int k, int c) { return A0[k * D + c]; }, [&](int r, int c, double v) { gs[r * LD + c] = v; });
  if (variant == FSHARP_ADERF) {
    const double* Li = sc + Layout{D}.Li();
    const double* LT = sc + Layout{D}.LT();
    double* U1 = sc + Layout{D}.U1() + (size_t)r0 * D;
    double* U2 = sc + Layout{D}.U2() + (size_t)r0 * D;
    product8<R, D, D, 16>(rows, [&](int k, int c) { return Li[k * D + c]; }, [&](int r, int c, double v) { U1[r * D + c] = v; });
    product8<R, D, D, 16>(rows, [&](int k, int c) { return LT[k * D + c]; }, [&](int r, int c, double v) { U2[r * D + c] = v; });
  }
  __syncthreads();
  const double tot = sc[Layout{D}.scal() + FS_TOT];
  for (int i = warp; i < R; i += PR_THREADS / 32) {
    double s = 0.0;
    for (int k = lane; k < D; k += 32) s = fma(gs[i * LD + k], vp[i * LD + k], s);
    const double lam = warp_sum(s);
    double res = 0.0;
    for (int k = lane; k < D; k += 32) {
      const double e = fma(-lam, vp[i * LD + k], gs[i * LD + k]);
      res = fma(e, e, res);
    }
    res = warp_sum(res);
    if (lane == 0) {
      sc[Layout{D}.lam() + r0 + i] = lam;
      // the rows' residuals are the off-diagonal rows of V' A V'^T: together at most 1e-24 of |A|^2
      if (!(res <= 1e-24 * tot / D)) *flag = 1.0;
    }
  }
}

// ---- A, B, C, D of the theorems; SPLIT rows per block -------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(PR_THREADS)
finish_kernel(int variant, const double* __restrict__ scratch, double* __restrict__ params, int* __restrict__ status) {
  fs_grid_dependency_wait();
  constexpr int R = SPLIT<D>;
  __shared__ double lam[D], w1[D], w2[D], red[2][PR_THREADS / 32];
  __shared__ int perm[D];
  const int g = blockIdx.x, r0 = blockIdx.y * R, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* sc = scratch + (size_t)g * Layout{D}.total();
  const double* scal = sc + Layout{D}.scal();
  if (scal[FS_FLAG] != 0.0) return;                      // the fall-back writes this group
  const ParamsLayout pl{D};
  double* out = params + (size_t)g * pl.total();
  double* oA = out + pl.A();
  double* oB1 = out + pl.B(1);
  double* oB2 = out + pl.B(2);
  double* oC1 = out + pl.C(1);
  double* oC2 = out + pl.C(2);
  auto block_sum = [&](double v, int slot) {
    v = warp_sum(v);
    if (lane == 0) red[slot][warp] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < PR_THREADS / 32; w++) s += red[slot][w];
    return s;
  };
  double logD, obj, phi;
  if (tid < D) lam[tid] = sc[Layout{D}.lam() + tid];
  __syncthreads();
  if (variant == FSHARP_SDERF) {
    // eigenvalues non-ascending
    double al = 0.0, sl = 0.0, so = 0.0;
    if (tid < D) {
      const double li = lam[tid];
      int rank = 0;
      for (int j = 0; j < D; j++) rank += (lam[j] > li) || (lam[j] == li && j < tid);
      perm[rank] = tid;
      const double lv = fmax(li, 0.0);                   // N is PSD; rounding may give -1e-17
      al = lemma_a1(lv);
      sl = log(1.0 - 4.0 * al);
      so = sl - 0.5 * log(1.0 - 8.0 * al) + (1.0 + 1.0 / (1.0 - 8.0 * al)) * lv;
      w1[tid] = al;
      w2[tid] = sqrt(1.0 - 4.0 * al);
    }
    sl = block_sum(sl, 0);
    so = block_sum(so, 1);
    const double* V = sc + Layout{D}.RF();
#pragma unroll 8
    for (int e = tid; e < R * D; e += PR_THREADS) {
      const int l = r0 + e / D, c = e % D, p = perm[l];
      const double dg = l == c ? 1.0 : 0.0, b = w2[p] * V[(size_t)p * D + c];       // B = (I-4A)^1/2 Q3^T
      oA[l * D + c] = w1[p] * dg;
      oB1[l * D + c] = b;
      oB2[l * D + c] = b;
      oC1[l * D + c] = -0.5 * dg;
      oC2[l * D + c] = -0.5 * dg;
    }
    logD = 0.25 * sl;
    obj = so - scal[FS_T1] - scal[FS_T2];
    phi = fmax(lam[perm[0]], 0.0);
  } else {
    // Sigma from the eigenvalues of L^T M2 L; B1 = r Sigma^1/2 U^T L^-1, B2 = r Sigma^-1/2 U^T L^T
    double sg = 0.0, smin = 1e300, smax = 0.0;
    if (tid < D) smin = smax = sg = sqrt(fmax(lam[tid], 0.0));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      smin = fmin(smin, __shfl_xor_sync(0xffffffffu, smin, o));
      smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, o));
    }
    if (lane == 0 && warp < D / 32) { w1[warp] = smin; w2[warp] = smax; }
    const double ssum = block_sum(sg, 0), mu3 = scal[FS_MM] / D;
    for (int w = 0; w < D / 32; w++) { smin = fmin(smin, w1[w]); smax = fmax(smax, w2[w]); }
    __syncthreads();                                      // (w1, w2 are written again)
    phi = 2.0 * ssum / D + 2.0 * mu3;
    const double A = lemma_a1(phi), r = sqrt(1.0 - 4.0 * A);
    if (!(smin > 1e-12 * smax) && tid == 0 && r0 == 0) atomicExch(status, FSHARP_E_CONSTRAINT);
    if (tid < D) {
      const double s = fmax(sg, 1e-300 + 1e-12 * smax);
      w1[tid] = r * sqrt(s);
      w2[tid] = r / sqrt(s);
    }
    __syncthreads();
    const double* U1 = sc + Layout{D}.U1();
    const double* U2 = sc + Layout{D}.U2();
    const double cf = -1.0 / (2.0 * (1.0 - 4.0 * A));     // C = -B^T B / (2 (1 - 4A))
    product8<R, D, D, 8>([&](int i, int l) { return w1[l] * w1[l] * U1[(size_t)l * D + r0 + i]; }, [&](int l, int j) { return U1[(size_t)l * D + j]; },
                         [&](int i, int j, double v) { oC1[(r0 + i) * D + j] = cf * v; });
    product8<R, D, D, 8>([&](int i, int l) { return w2[l] * w2[l] * U2[(size_t)l * D + r0 + i]; }, [&](int l, int j) { return U2[(size_t)l * D + j]; },
                         [&](int i, int j, double v) { oC2[(r0 + i) * D + j] = cf * v; });
#pragma unroll 8
    for (int e = tid; e < R * D; e += PR_THREADS) {
      const int l = r0 + e / D, c = e % D;
      oB1[l * D + c] = w1[l] * U1[(size_t)l * D + c];
      oB2[l * D + c] = w2[l] * U2[(size_t)l * D + c];
      oA[l * D + c] = l == c ? A : 0.0;
    }
    logD = 0.25 * D * log(1.0 - 4.0 * A);
    obj = D * (log(1.0 - 4.0 * A) - 0.5 * log(1.0 - 8.0 * A) + 2.0 / (1.0 - 8.0 * A) * (ssum / D + mu3) + 2.0 * mu3);
  }
  if (r0 == 0 && tid == 0) {
    double* tail = out + pl.tail();
    tail[PT_LOGD] = logD;
    tail[PT_OBJ] = obj;
    tail[PT_PHI] = phi;
    for (int i = 3; i < 8; i++) tail[i] = 0.0;            // [3]: no Jacobi sweeps
  }
}

// Dynamic shared memory that spreads `blocks` blocks evenly over the SMs: a launch that begins while its predecessor drains puts
// as many blocks as fit on the first SMs that come free, where they share one fp64 pipe and one shared-memory pipe (64
// tridiagonalisations: 70 us so, 51 us spread).
size_t spread(const fsharp_ctx* ctx, size_t static_bytes, int blocks, size_t need) {
  const int per_sm = (blocks + ctx->sm_count - 1) / ctx->sm_count;
  if (per_sm > 4) return need;
  // more than a (per_sm + 1)-th of the SM's 228 KB (1 KB per block is the system's)
  const size_t room = (size_t)(228 * 1024) / (per_sm + 1) + 128, fixed = static_bytes + 1024;
  const size_t want = room > fixed ? room - fixed : 0;
  return want > need ? want : need;
}

template <int D>
int run_d(fsharp_ctx* ctx, const double* stats, int G, int variant, double ridge, double* params, double* scratch) {
  cudaStream_t st = ctx->stream;
#define FITW_LAUNCH(kernel, grid, threads, smem, ...)                                       \
  do {                                                                                      \
    const dim3 gr = grid;                                                                   \
    cudaFuncAttributes at;                                                                  \
    FS_CUDA_OK(cudaFuncGetAttributes(&at, kernel));                                         \
    FS_CUDA_OK(fs_allow_smem(kernel, at.sharedSizeBytes));                                  \
    const size_t sm = spread(ctx, at.sharedSizeBytes, (int)(gr.x * gr.y), smem);            \
    FS_TIME_BEGIN(ctx, FS_K_FIT);                                                           \
    (void)fs_launch_chained(kernel, gr, dim3(threads), sm, st, __VA_ARGS__);                \
    FS_TIME_END(ctx);                                                                       \
    FS_LAUNCH_CHECK(ctx);                                                                   \
  } while (0)
  if (variant == FSHARP_ADERF) {
    FITW_LAUNCH(chol_kernel<D>, dim3(G), Dist<D>::NT, chol_smem<D>(), stats, ridge, scratch, ctx->d_status);
    FITW_LAUNCH(zform_kernel<D>, dim3(G, D / SPLIT<D>), PR_THREADS, 0, stats, ridge, scratch);
  }
  FITW_LAUNCH(tridiag_kernel<D>, dim3(G), Tri<D>::NT, 0, stats, variant, ridge, scratch, ctx->d_status);
  FITW_LAUNCH(vectors_kernel<D>, dim3(G, D / 16), VC_THREADS, vectors_smem<D>(), variant, scratch, ctx->d_status);
  FITW_LAUNCH(polish_kernel<D>, dim3(G, D / SPLIT<D>), PR_THREADS, polish_smem<D>(), variant, scratch);
  FITW_LAUNCH(finish_kernel<D>, dim3(G, D / SPLIT<D>), PR_THREADS, 0, variant, scratch, params, ctx->d_status);
#undef FITW_LAUNCH
  return FSHARP_OK;
}

}  // namespace

int fitw::run(fsharp_ctx* ctx, const double* stats, int G, int d, int variant, double ridge, double* params, double* scratch) {
  return d == 64 ? run_d<64>(ctx, stats, G, variant, ridge, params, scratch)
                 : run_d<128>(ctx, stats, G, variant, ridge, params, scratch);
}
