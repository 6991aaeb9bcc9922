// Backward pass of featurize + attend (Section 5.3 trains Transformers through the attention of
// Section 2.2): given dY, the gradients with respect to Q, K and V, the random features Omega and
// the fitted parameters being constants.  Every product is a block product at fp32 precision on the tensor cores (mma3.cuh).
//
// With P = phi(Q) (L x M), S = phi(K), [num | den] = P KV_i, KV_i = sum_{j <= i} S_j [V_j | 1]^T
// (all j when bidirectional), Y = num / den:
//   G_i   = [dY_i / den_i | -(dY_i . Y_i) / den_i]                                (L x (dv + 1))
//   dP_i  = G_i KV_i^T,                     dlogP = dP * P
//   R_j   = sum_{i >= j} P_i G_i^T          (M x (dv + 1); all i when bidirectional)
//   dS_j  = [V_j | 1] R_j^T,                dlogS = dS * S,      dV_j = S_j R_j[:, :dv]
//   logit = a_m + w_m^T B x + x^T C x:      dx = dlog W + rowsum(dlog) (C + C^T) x,   dQ = qk_scale dx
// Causal sequences go chunk by chunk: KV_i = (sum over earlier chunks) + the masked part inside the
// chunk, R_j = (sum over later chunks) + the masked part, with tril(P_c S_c^T) and tril(G_c [V_c | 1]^T)
// formed per chunk.  The feature kernels' shifts (per query row, per (batch, head) for the keys)
// cancel in every product above exactly as they do in Y.  Their factor 2^LIFT on either side (feat3.cuh)
// would leave G with 2^-2 LIFT; it is given half of that back, so that R and G KV^T are what they are without the factor (a
// query that sees distant keys only has G near the top of the range), and the gradients' last products take off 2^LIFT.
#include "f32_parts.cuh"
#include "feat3.cuh"

namespace {

using mma3::Piece;
using mma3::ROWS;

constexpr float LIFTED = (float)(1 << feat3::LIFT), UNLIFT = 1.f / LIFTED;

struct BwdDims {
  int H, Lq, Lk, d, dv, M, NP, causal, C, nch;      // NP = dv + 16: [V | 1] rows, G rows and sums are padded to it
};

__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}

// ---- masked blocks tril(G_c [V_c | 1]^T) of a chunk ----------------------------------------------
template <typename T>
__global__ void __launch_bounds__(mma3::THREADS, 2)
bwd_tri_kernel(const float* __restrict__ G, const T* __restrict__ V, TensorAddr av, BwdDims q, float* __restrict__ out,
               int flip, int* __restrict__ status) {
  fs_grid_dependency_wait();
  const int zi = mma3::unit_of(flip);
  extern __shared__ uint8_t smem[];
  const int bh = zi / q.nch, c = zi % q.nch, b = bh / q.H, h = bh % q.H;
  const int i0 = blockIdx.x * ROWS, j0 = blockIdx.y * ROWS, C = q.C, dv = q.dv;
  if (j0 > i0) return;
  mma3::Block blk;
  blk.begin(smem, ROWS, q.NP, status);
  const int rows = min(C, q.Lq - c * C);
  const float* Gc = G + ((int64_t)bh * q.Lq + (int64_t)c * C + i0) * q.NP;
  const T* Vc = V + b * av.sb + h * av.sh + ((int64_t)c * C + j0) * av.sl;
  constexpr int VP = mma3::PartsOf<T>::N;
  blk.template segment<true, 3, true, VP>(
      q.NP, [&](int r, int k, Piece<3>& p) { if (i0 + r < rows) p.load(Gc + (int64_t)r * q.NP + k); else p.zero(); },
      [&](int n, int k, Piece<VP>& p) {
        if (j0 + n >= rows || k > dv) p.zero();
        else if (k < dv) p.load(Vc + (int64_t)n * av.sl + k);
        else p.unit();
      });
  blk.finish();
  float* S = out + (int64_t)zi * C * C;
  blk.rows([&](int r, int n, float4 v) {
    const int i = i0 + r, j = j0 + n;
    if (j > i) v.x = 0.f;
    if (j + 1 > i) v.y = 0.f;
    if (j + 2 > i) v.z = 0.f;
    if (j + 3 > i) v.w = 0.f;
    *reinterpret_cast<float4*>(S + (int64_t)i * C + j) = v;
  });
  blk.end();
}

// ---- [num | den] = phiQ KV (+ masked scores times [V_c | 1]), and from it G = [dY / den | -(dY . Y) / den] -----------
// dv <= 64: one column tile holds the whole row and G is written; dv = 128 (two tiles): [num | den] is, for bwd_g_kernel.
template <typename T>
__global__ void __launch_bounds__(mma3::THREADS, 2)
bwd_numden_kernel(const float* __restrict__ phiQ, const float* __restrict__ KV, const float* __restrict__ sc,
                  const T* __restrict__ V, TensorAddr av, const T* __restrict__ dY, TensorAddr ay, BwdDims q, float* __restrict__ G,
                  int flip, int* __restrict__ status) {
  fs_grid_dependency_wait();
  const int zi = mma3::unit_of(flip);
  extern __shared__ uint8_t smem[];
  __shared__ float inv_s[ROWS], dot_s[ROWS];
  const int bh = zi, b = bh / q.H, h = bh % q.H, i0 = blockIdx.x * ROWS;
  const int C = q.C, M = q.M, NP = q.NP, dv = q.dv, L = q.Lq;
  const ColTile ct(dv, blockIdx.y);
  mma3::Block blk;
  blk.begin(smem, ct.nt(), M + (q.causal ? C : 0), status);
  const int chunk = q.causal ? i0 / C : 0;
  const float* PQ = phiQ + ((int64_t)bh * L + i0) * M;
  const float* S = KV + ((int64_t)bh * q.nch + chunk) * M * NP;
  blk.template segment<true, 3, false, 3>(
      M, [&](int r, int k, Piece<3>& p) { if (i0 + r < L) p.load(PQ + (int64_t)r * M + k); else p.zero(); },
      [&](int c, int k, Piece<3>& p) { p.load(S + (int64_t)k * NP + ct.at(dv, c)); });
  if (q.causal) {
    const int ic = i0 - chunk * C, keys = min(ic + ROWS, L - chunk * C);
    const float* SC = sc + (((int64_t)bh * q.nch + chunk) * C + ic) * C;
    const T* Vc = V + b * av.sb + h * av.sh + (int64_t)chunk * C * av.sl;
    constexpr int VP = mma3::PartsOf<T>::N;
    blk.template segment<true, 3, false, VP>(
        (keys + 7) & ~7, [&](int r, int k, Piece<3>& p) { p.load(SC + (int64_t)r * C + k); },
        [&](int c, int k, Piece<VP>& p) {
          if (k >= keys) p.zero();
          else if (c < ct.wt) p.load(Vc + (int64_t)k * av.sl + ct.v0 + c);
          else if (c == ct.wt) p.unit();
          else p.zero();
        });
  }
  blk.finish();
  float* Gb = G + ((int64_t)bh * L + i0) * NP;
  if (gridDim.y > 1) {
    blk.rows([&](int r, int c, float4 v) {
      if (i0 + r < L && (c < ct.wt || blockIdx.y == 0)) *reinterpret_cast<float4*>(Gb + (int64_t)r * NP + ct.at(dv, c)) = v;
    });
    blk.end();
    return;
  }
  if (threadIdx.x < ROWS) {
    const float den = blk.column(ct.wt);
    if (i0 + (int)threadIdx.x < L && (!(den > 0.f) || !isfinite(den))) atomicExch(status, FSHARP_E_NONFINITE);
    inv_s[threadIdx.x] = 1.f / den;
    dot_s[threadIdx.x] = 0.f;
  }
  __syncthreads();
  const T* dYb = dY + b * ay.sb + h * ay.sh + (int64_t)i0 * ay.sl;
  float sum[8] = {};
  blk.rows([&](int r, int c) { return i0 + r < L && c < dv ? load4(dYb + (int64_t)r * ay.sl + c) : make_float4(0.f, 0.f, 0.f, 0.f); },
           [&](int r, int c, float4 v, float4 y, int i) {
             float s = 0.f;
             if (i0 + r < L && c < dv) {
               const float inv = inv_s[r];
               s = fmaf(y.x, v.x * inv, fmaf(y.y, v.y * inv, fmaf(y.z, v.z * inv, y.w * (v.w * inv))));
               const float gi = LIFTED * inv;
               *reinterpret_cast<float4*>(Gb + (int64_t)r * NP + c) = make_float4(y.x * gi, y.y * gi, y.z * gi, y.w * gi);
             }
             if (i >= 0) { sum[i < 0 ? 0 : i] += s; return; }
             // (four neighbouring lanes hold the row's last 16 columns)
             s += __shfl_xor_sync(0xffffffffu, s, 1);
             s += __shfl_xor_sync(0xffffffffu, s, 2);
             if ((threadIdx.x & 3) == 0) atomicAdd(&dot_s[r], s);
           });
  blk.add_row_sums(sum, dot_s);
  __syncthreads();
  for (int e = threadIdx.x; e < ROWS * 4; e += mma3::THREADS) {
    const int r = e >> 2, part = e & 3;
    if (i0 + r < L) *reinterpret_cast<float4*>(Gb + (int64_t)r * NP + dv + 4 * part) = make_float4(part ? 0.f : -dot_s[r] * (LIFTED * inv_s[r]), 0.f, 0.f, 0.f);
  }
  blk.end();
}

// ---- G from [num | den], in place; one warp per row (dv = 128) --------------------------------------
template <typename T>
__global__ void __launch_bounds__(NTH)
bwd_g_kernel(float* __restrict__ ND, const T* __restrict__ dY, TensorAddr ay, BwdDims q, int* __restrict__ status) {
  fs_grid_dependency_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int bh = blockIdx.y, b = bh / q.H, h = bh % q.H, dv = q.dv;
  const T* dYb = dY + b * ay.sb + h * ay.sh;
  for (int i = blockIdx.x * 8 + warp; i < q.Lq; i += gridDim.x * 8) {
    float* row = ND + ((int64_t)bh * q.Lq + i) * q.NP;
    const float den = row[dv], inv = 1.f / den, gi = LIFTED * inv;
    float s = 0.f;
    for (int c = 4 * lane; c < dv; c += 128) {
      const float4 y = load4(dYb + (int64_t)i * ay.sl + c), n = *reinterpret_cast<const float4*>(row + c);
      s = fmaf(y.x, n.x * inv, fmaf(y.y, n.y * inv, fmaf(y.z, n.z * inv, fmaf(y.w, n.w * inv, s))));
      *reinterpret_cast<float4*>(row + c) = make_float4(y.x * gi, y.y * gi, y.z * gi, y.w * gi);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      row[dv] = -s * gi;
      if (!(den > 0.f) || !isfinite(den)) atomicExch(status, FSHARP_E_NONFINITE);
    }
  }
}

// ---- E = dphi * phi (the gradient with respect to the exponents), and its row sums per feature tile ----------------
// SIDE 1: dphiQ_c = G_c KV_c^T + tril(G_c [V_c | 1]^T) phiK_c;   SIDE 2: dphiK_c = [V_c | 1] R_c^T + tril(...)^T phiQ_c
// rs [feature tile][BH][L]
// (2 x 12 x 4096 tokens, M = 256, causal: 183 us with a load of phi, a product and a shared-memory atomic per piece of the
// epilogue, one after the other; 160 us with the loads of eight pieces issued together and the row sums kept in registers)
template <typename T, int SIDE>
__global__ void __launch_bounds__(mma3::THREADS, 2)
bwd_dfeat_kernel(const float* __restrict__ phiQ, const float* __restrict__ phiK, const float* __restrict__ G,
                 const float* __restrict__ St, const float* __restrict__ gv, const T* __restrict__ V, TensorAddr av,
                 BwdDims q, float* __restrict__ E, float* __restrict__ rs, int flip, int* __restrict__ status) {
  fs_grid_dependency_wait();
  const int zi = mma3::unit_of(flip);
  extern __shared__ uint8_t smem[];
  __shared__ float rs_s[ROWS];
  const int bh = zi, b = bh / q.H, h = bh % q.H;
  // (token tiles run along x, the only coordinate that takes more than 65535; the feature tiles of one token tile are neighbours)
  const int mtiles = (q.M + ROWS - 1) / ROWS, mt = blockIdx.x % mtiles, m0 = mt * ROWS, i0 = blockIdx.x / mtiles * ROWS;
  const int C = q.C, M = q.M, NP = q.NP, dv = q.dv, L = SIDE == 1 ? q.Lq : q.Lk;
  const int chunk = q.causal ? i0 / C : 0, ic = q.causal ? i0 - chunk * C : 0;
  mma3::Block blk;
  blk.begin(smem, min(ROWS, M - m0), NP + (q.causal ? C : 0), status);
  const float* S = St + ((int64_t)bh * q.nch + chunk) * M * NP + (int64_t)m0 * NP;
  const float* GV = q.causal ? gv + ((int64_t)bh * q.nch + chunk) * C * C : nullptr;
  mma3::prefetch_rows((SIDE == 1 ? phiQ : phiK) + ((int64_t)bh * L + i0) * M + m0, 4LL * M, min(ROWS, L - i0), 4LL * min(ROWS, M - m0));
  if (SIDE == 1) {
    const float* Gb = G + ((int64_t)bh * L + i0) * NP;
    blk.template segment<true, 3, true, 3>(
        NP, [&](int r, int k, Piece<3>& p) { if (i0 + r < L) p.load(Gb + (int64_t)r * NP + k); else p.zero(); },
        [&](int n, int k, Piece<3>& p) { p.load(S + (int64_t)n * NP + k); });
    if (q.causal) {
      const int keys = min(ic + ROWS, L - chunk * C);
      const float* PK = phiK + ((int64_t)bh * L + (int64_t)chunk * C) * M + m0;
      blk.template segment<true, 3, false, 3>(
          (keys + 7) & ~7, [&](int r, int k, Piece<3>& p) { p.load(GV + (int64_t)(ic + r) * C + k); },
          [&](int c, int k, Piece<3>& p) { if (k < keys) p.load(PK + (int64_t)k * M + c); else p.zero(); });
    }
  } else {
    const T* Vb = V + b * av.sb + h * av.sh + (int64_t)i0 * av.sl;
    constexpr int VP = mma3::PartsOf<T>::N;
    blk.template segment<true, VP, true, 3>(
        NP,
        [&](int r, int k, Piece<VP>& p) {
          if (i0 + r >= L || k > dv) p.zero();
          else if (k < dv) p.load(Vb + (int64_t)r * av.sl + k);
          else p.unit();
        },
        [&](int n, int k, Piece<3>& p) { p.load(S + (int64_t)n * NP + k); });
    if (q.causal) {
      // rows ic + k of the masked block, k >= 0: the queries of this chunk at or after this tile's first key
      const float* PQ = phiQ + ((int64_t)bh * L + (int64_t)chunk * C + ic) * M + m0;
      blk.template segment<false, 3, false, 3>(
          min(C, L - chunk * C) - ic, [&](int r, int k, Piece<3>& p) { p.load(GV + (int64_t)(ic + k) * C + ic + r); },
          [&](int c, int k, Piece<3>& p) { p.load(PQ + (int64_t)k * M + c); });
    }
  }
  blk.finish();
  if (threadIdx.x < ROWS) rs_s[threadIdx.x] = 0.f;
  __syncthreads();
  const int64_t base = ((int64_t)bh * L + i0) * M + m0;
  const float* Ph = (SIDE == 1 ? phiQ : phiK) + base;
  float sum[8] = {};
  blk.rows([&](int r, int c) { return i0 + r < L ? *reinterpret_cast<const float4*>(Ph + (int64_t)r * M + c) : make_float4(0.f, 0.f, 0.f, 0.f); },
           [&](int r, int c, float4 v, float4 f, int i) {
             v.x = UNLIFT * v.x * f.x; v.y = UNLIFT * v.y * f.y; v.z = UNLIFT * v.z * f.z; v.w = UNLIFT * v.w * f.w;
             float s = 0.f;
             if (i0 + r < L) {
               *reinterpret_cast<float4*>(E + base + (int64_t)r * M + c) = v;
               s = (v.x + v.y) + (v.z + v.w);
             }
             if (i >= 0) { sum[i < 0 ? 0 : i] += s; return; }
             // (four neighbouring lanes hold the row's last 16 columns)
             s += __shfl_xor_sync(0xffffffffu, s, 1);
             s += __shfl_xor_sync(0xffffffffu, s, 2);
             if ((threadIdx.x & 3) == 0) atomicAdd(&rs_s[r], s);
           });
  blk.add_row_sums(sum, rs_s);
  __syncthreads();
  if (threadIdx.x < ROWS && i0 + (int)threadIdx.x < L)
    rs[((int64_t)mt * gridDim.z + bh) * L + i0 + threadIdx.x] = rs_s[threadIdx.x];
  blk.end();
}

// ---- dV_c = phiK_c R_c[:, :dv] + tril(phiQ_c phiK_c^T)^T G_c[:, :dv] ------------------------------
template <typename T>
__global__ void __launch_bounds__(mma3::THREADS, 2)
bwd_dv_kernel(const float* __restrict__ phiK, const float* __restrict__ Rt, const float* __restrict__ sc,
              const float* __restrict__ G, BwdDims q, T* __restrict__ dV, TensorAddr av, int flip, int* __restrict__ status) {
  fs_grid_dependency_wait();
  const int zi = mma3::unit_of(flip);
  extern __shared__ uint8_t smem[];
  const int bh = zi, b = bh / q.H, h = bh % q.H, j0 = blockIdx.x * ROWS;
  const int C = q.C, M = q.M, NP = q.NP, L = q.Lk, cols = tile_columns(q.dv, M), c0 = blockIdx.y * cols;
  const int chunk = q.causal ? j0 / C : 0, jc = q.causal ? j0 - chunk * C : 0;
  mma3::Block blk;
  blk.begin(smem, cols, M + (q.causal ? C - jc : 0), status);
  const float* PK = phiK + ((int64_t)bh * L + j0) * M;
  const float* R = Rt + ((int64_t)bh * q.nch + chunk) * M * NP;
  blk.template segment<true, 3, false, 3>(
      M, [&](int r, int k, Piece<3>& p) { if (j0 + r < L) p.load(PK + (int64_t)r * M + k); else p.zero(); },
      [&](int c, int k, Piece<3>& p) { p.load(R + (int64_t)k * NP + c0 + c); });
  if (q.causal) {
    const float* SC = sc + ((int64_t)bh * q.nch + chunk) * C * C;
    const float* Gc = G + ((int64_t)bh * L + (int64_t)chunk * C + jc) * NP;
    blk.template segment<false, 3, false, 3>(
        min(C, L - chunk * C) - jc, [&](int r, int k, Piece<3>& p) { p.load(SC + (int64_t)(jc + k) * C + jc + r); },
        [&](int c, int k, Piece<3>& p) { p.load(Gc + (int64_t)k * NP + c0 + c); });
  }
  blk.finish();
  T* Ob = dV + b * av.sb + h * av.sh + (int64_t)j0 * av.sl;
  blk.rows([&](int r, int c, float4 v) {
    if (j0 + r < L) store4(Ob + (int64_t)r * av.sl + c0 + c, make_float4(UNLIFT * v.x, UNLIFT * v.y, UNLIFT * v.z, UNLIFT * v.w));
  });
  blk.end();
}

// ---- dX = qk_scale (E W + rowsum(E) x^T (C + C^T)),  x = qk_scale X ------------------------------
template <typename T>
__global__ void __launch_bounds__(mma3::THREADS, 2)
bwd_dx_kernel(const float* __restrict__ E, const float* __restrict__ rs, int mtiles, const T* __restrict__ X, TensorAddr ax, int H, int L,
              int d, int M, int pool, int side, const float* __restrict__ prep, float qk_scale, T* __restrict__ dX,
              int flip, int* __restrict__ status) {
  fs_grid_dependency_wait();
  const int zi = mma3::unit_of(flip);
  extern __shared__ uint8_t smem[];
  __shared__ float rs_s[ROWS];
  const int bh = zi, b = bh / H, h = bh % H, i0 = blockIdx.x * ROWS, cols = tile_columns(d, M), c0 = blockIdx.y * cols;
  PrepLayout pr{d, M};
  const float* pp = prep + ((size_t)(pool == FSHARP_POOL_PER_BH ? bh : h) * 2 + (side - 1)) * pr.total();
  const float* W = pp + pr.W();
  const float* Cm = pp + pr.Cmat();
  const bool cscalar = pp[pr.scal() + PS_CSCALAR] != 0.f;
  const float gamma = pp[pr.scal() + PS_CGAMMA];
  mma3::Block blk;
  blk.begin(smem, cols, M + d, status);
  if (threadIdx.x < ROWS) {
    float s = 0.f;
    if (i0 + (int)threadIdx.x < L)
      for (int t = 0; t < mtiles; t++) s += rs[((int64_t)t * gridDim.z + bh) * L + i0 + threadIdx.x];
    rs_s[threadIdx.x] = qk_scale * s;
  }
  __syncthreads();
  const float* Eb = E + ((int64_t)bh * L + i0) * M;
  mma3::prefetch_rows(Eb, 4LL * M, min(ROWS, L - i0), 4LL * M);
  const T* Xb = X + b * ax.sb + h * ax.sh + (int64_t)i0 * ax.sl;
  blk.template segment<true, 3, false, 3>(
      M, [&](int r, int k, Piece<3>& p) { if (i0 + r < L) p.load(Eb + (int64_t)r * M + k); else p.zero(); },
      [&](int c, int k, Piece<3>& p) { p.load(W + (size_t)k * d + c0 + c); });
  if (!cscalar)
    blk.template segment<true, 3, false, 3>(
        d,
        [&](int r, int k, Piece<3>& p) {
          if (i0 + r >= L) { p.zero(); return; }
          const float4 a = load4(Xb + (int64_t)r * ax.sl + k), c = load4(Xb + (int64_t)r * ax.sl + k + 4);
          const float s = rs_s[r];
          p.v[0] = s * a.x; p.v[1] = s * a.y; p.v[2] = s * a.z; p.v[3] = s * a.w;
          p.v[4] = s * c.x; p.v[5] = s * c.y; p.v[6] = s * c.z; p.v[7] = s * c.w;
        },
        [&](int c, int k, Piece<3>& p) {
          p.load(Cm + (size_t)k * d + c0 + c);
#pragma unroll
          for (int j = 0; j < 8; j++) p.v[j] += Cm[(size_t)(c0 + c + j) * d + k];
        });
  blk.finish();
  T* Ob = dX + b * ax.sb + h * ax.sh + (int64_t)i0 * ax.sl;
  bool bad = false;
  blk.rows([&](int r, int column, float4 v) {
    const int c = c0 + column;
    if (i0 + r >= L) return;
    if (cscalar) {
      const float s = 2.f * gamma * rs_s[r];
      const float4 x = load4(Xb + (int64_t)r * ax.sl + c);
      v.x = fmaf(s, x.x, v.x); v.y = fmaf(s, x.y, v.y); v.z = fmaf(s, x.z, v.z); v.w = fmaf(s, x.w, v.w);
    }
    v.x *= qk_scale; v.y *= qk_scale; v.z *= qk_scale; v.w *= qk_scale;
    if (!isfinite(v.x) || !isfinite(v.y) || !isfinite(v.z) || !isfinite(v.w)) bad = true;
    store4(Ob + (int64_t)r * ax.sl + c, v);
  });
  if (bad) atomicExch(status, FSHARP_E_NONFINITE);
  blk.end();
}

struct Yes { static constexpr bool value = true; };
struct No { static constexpr bool value = false; };

template <typename T>
int backward_t(fsharp_ctx* ctx, const void* Qv, const void* Kv, const void* Vv, const void* dYv, const fsharp_dims* dm,
               int dtype, int causal, int chunk, float qk_scale, const float* prep, void* dQv, void* dKv, void* dVv,
               WsAlloc* ws) {
  const T* Q = (const T*)Qv; const T* K = (const T*)Kv; const T* V = (const T*)Vv; const T* dY = (const T*)dYv;
  const int B = dm->B, H = dm->H, BH = B * H, Lq = dm->Lq, Lk = dm->Lk, d = dm->d, dv = dm->dv, M = dm->M;
  const int NP = dv + 16, C = causal ? inner_chunk(chunk) : 0, nch = causal ? (Lq + C - 1) / C : 1;
  const int mt = (M + ROWS - 1) / ROWS, ctiles = (dv + 63) / 64, qt = (Lq + ROWS - 1) / ROWS, kt = (Lk + ROWS - 1) / ROWS;
  const BwdDims q{H, Lq, Lk, d, dv, M, NP, causal ? 1 : 0, C, nch};
  TensorAddr aq = fs_addr(dm->q_stride, H, Lq, d), ak = fs_addr(dm->k_stride, H, Lk, d);
  TensorAddr av = fs_addr(dm->v_stride, H, Lk, dv), ay = fs_addr(dm->y_stride, H, Lq, dv);
  float* phiQ = ws->take<float>((size_t)BH * Lq * M);
  float* phiK = ws->take<float>((size_t)BH * Lk * M);
  float* E = ws->take<float>((size_t)BH * (Lq > Lk ? Lq : Lk) * M);      // one side after the other
  float* rs = ws->take<float>((size_t)mt * BH * (Lq > Lk ? Lq : Lk));
  float* rowcq = ws->take<float>((size_t)BH * Lq);
  float* rowck = ws->take<float>((size_t)BH * Lk);
  unsigned* gmax = ws->take<unsigned>((size_t)BH);
  float* lsq = ws->take<float>((size_t)BH * Lq);
  float* lsk = ws->take<float>((size_t)BH);
  float* G = ws->take<float>((size_t)BH * Lq * NP);
  float* KV = ws->take<float>((size_t)BH * nch * M * NP);
  float* Rt = ws->take<float>((size_t)BH * nch * M * NP);
  float* sc = causal ? ws->take<float>((size_t)BH * nch * C * C) : nullptr;
  float* gv = causal ? ws->take<float>((size_t)BH * nch * C * C) : nullptr;
  uint8_t* img = ws->take<uint8_t>(feat3::image_bytes(fs_groups(dm), d, M, 2));
  int* status = ctx->d_status;
  const int64_t elems = (int64_t)M * NP;
  const dim3 gscan((unsigned)((elems + NTH - 1) / NTH), BH);

  const feat3::Task tasks[2] = {{K, ak, Lk, 2, FSHARP_STAB_GROUP, rowck, gmax, phiK, nullptr, lsk, feat3::LIFT},
                                {Q, aq, Lq, 1, FSHARP_STAB_ROW, rowcq, nullptr, phiQ, nullptr, lsq, feat3::LIFT}};
  // (KV and Rt are neighbours, with less than 256 bytes between them)
  FS_TRY(feat3::run(ctx, tasks, 2, dtype, B, H, d, M, dm->pool, prep, qk_scale, img, KV, causal ? 0 : (size_t)(Rt - KV) + (size_t)BH * elems));
  // sums over tokens: the total (bidirectional), or one per chunk turned into the sum over earlier / later chunks (causal)
  auto sums = [&](auto from_g, const float* F, int L, float* out, int reverse, int flip) -> int {
    constexpr bool FG = decltype(from_g)::value;
    int slen = C, nsl = nch;
    if (!causal) nsl = fs_token_slices(ctx, BH * mt * ctiles, BH, L, &slen);
    FS_TRY(mma3::launch(ctx, FS_K_BWD_STATE, state_kernel<T, FG>, dim3(mt, ctiles, BH * nsl), F, V, av, G, H, L, M, dv, slen, nsl,
                        causal ? 1 : 0, out, flip, status));
    if (causal) {
      FS_TIME_BEGIN(ctx, FS_K_PREFIX);
      (void)fs_launch_chained(prefix_kernel, gscan, dim3(NTH), 0, ctx->stream, out, nch, elems, reverse, 1 - flip);
      FS_TIME_END(ctx);
      FS_LAUNCH_CHECK(ctx);
    }
    return FSHARP_OK;
  };
  const dim3 gtri(causal ? C / ROWS : 1, causal ? C / ROWS : 1, BH * nch), gsc(gtri.x, causal ? C / tile_columns(ROWS, M) : 1, BH * nch);
  const int dtiles = d / tile_columns(d, M);
  FS_TRY(sums(No{}, phiK, Lk, KV, 0, 0));
  if (causal) FS_TRY(mma3::launch(ctx, FS_K_SCORES, scores_kernel, gsc, phiQ, phiK, Lq, M, C, nch, sc, 1, status));
  FS_TRY(mma3::launch(ctx, FS_K_BWD_NUMDEN, bwd_numden_kernel<T>, dim3(qt, ctiles, BH), phiQ, KV, sc, V, av, dY, ay, q, G, 0, status));
  if (ctiles > 1) {
    int gx = (Lq + 7) / 8;
    if (gx > 4 * ctx->sm_count) gx = 4 * ctx->sm_count;
    FS_TIME_BEGIN(ctx, FS_K_BWD_NUMDEN);
    (void)fs_launch_chained(bwd_g_kernel<T>, dim3(gx, BH), dim3(NTH), 0, ctx->stream, G, dY, ay, q, status);
    FS_TIME_END(ctx);
    FS_LAUNCH_CHECK(ctx);
  }
  FS_TRY(sums(Yes{}, phiQ, Lq, Rt, 1, 1));
  if (causal) FS_TRY(mma3::launch(ctx, FS_K_SCORES, bwd_tri_kernel<T>, gtri, G, V, av, q, gv, 1, status));
  FS_TRY(mma3::launch(ctx, FS_K_BWD_DFEAT, bwd_dfeat_kernel<T, 1>, dim3(mt * qt, 1, BH), phiQ, phiK, G, KV, gv, V, av, q, E, rs, 0, status));
  FS_TRY(mma3::launch(ctx, FS_K_BWD_DX, bwd_dx_kernel<T>, dim3(qt, dtiles, BH), E, rs, mt, Q, aq, H, Lq, d, M, dm->pool, 1, prep, qk_scale,
                      (T*)dQv, 1, status));
  FS_TRY(mma3::launch(ctx, FS_K_BWD_DFEAT, bwd_dfeat_kernel<T, 2>, dim3(mt * kt, 1, BH), phiQ, phiK, G, Rt, gv, V, av, q, E, rs, 0, status));
  FS_TRY(mma3::launch(ctx, FS_K_BWD_DX, bwd_dx_kernel<T>, dim3(kt, dtiles, BH), E, rs, mt, K, ak, H, Lk, d, M, dm->pool, 2, prep, qk_scale,
                      (T*)dKv, 1, status));
  return mma3::launch(ctx, FS_K_BWD_DV, bwd_dv_kernel<T>, dim3(kt, dv / tile_columns(dv, M), BH), phiK, Rt, sc, G, q, (T*)dVv, av, 0, status);
}

}  // namespace

size_t fs_backward_scratch_bytes(const fsharp_dims* dm, int causal, int chunk) {
  const size_t BH = (size_t)dm->B * dm->H, NP = dm->dv + 16, M = dm->M;
  const size_t Lq = dm->Lq, Lk = dm->Lk, Lmax = Lq > Lk ? Lq : Lk, C = causal ? inner_chunk(chunk) : 0;
  const size_t nch = causal ? (Lq + C - 1) / C : 1, mt = (M + ROWS - 1) / ROWS;
  size_t b = ws_round(BH * Lq * M * 4) + ws_round(BH * Lk * M * 4) + ws_round(BH * Lmax * M * 4) + ws_round(mt * BH * Lmax * 4) +
             2 * ws_round(BH * Lq * 4) + ws_round(BH * Lk * 4) + 2 * ws_round(BH * 4) + ws_round(BH * Lq * NP * 4) +
             2 * ws_round(BH * nch * M * NP * 4);
  b += feat3::image_bytes(fs_groups(dm), dm->d, dm->M, 2);
  if (causal) b += 2 * ws_round(BH * nch * C * C * 4);
  return b;
}

int fs_backward(fsharp_ctx* ctx, const void* Q, const void* K, const void* V, const void* dY, const fsharp_dims* dm,
                int dtype, int causal, int chunk, float qk_scale, const float* prep, void* dQ, void* dK, void* dV,
                WsAlloc* ws) {
  if (dtype == FSHARP_F32)
    return backward_t<float>(ctx, Q, K, V, dY, dm, dtype, causal, chunk, qk_scale, prep, dQ, dK, dV, ws);
  return backward_t<__nv_bfloat16>(ctx, Q, K, V, dY, dm, dtype, causal, chunk, qk_scale, prep, dQ, dK, dV, ws);
}
