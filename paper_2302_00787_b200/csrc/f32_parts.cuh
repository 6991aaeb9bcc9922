// Block products that the fp32-precision attention and its backward pass share (mma3.cuh): sums over tokens, their running
// sums over chunks, masked in-chunk scores.
#pragma once
#include "mma3.cuh"

namespace {

constexpr int NTH = 256;

// Chunk length of the causal form inside the kernels: their tiles are 128 tokens, and the result does not depend on it.
int inner_chunk(int chunk) { return chunk == 256 ? 256 : 128; }

// Column tile of [V | 1]: 64 value columns (all of them when dv <= 64) and the ones column's block of 16.  Local column
// c < wt is value column v0 + c; c = wt is the ones column.  In scratch a row of [V | 1] sums is NP = dv + 16 floats.
struct ColTile {
  int v0, wt;
  __device__ __forceinline__ ColTile(int dv, int tile) : v0(tile * 64), wt(dv < 64 ? dv : 64) {}
  __device__ __forceinline__ int nt() const { return wt + 16; }
  // position in a row of dv + 16
  __device__ __forceinline__ int at(int dv, int c) const { return c < wt ? v0 + c : dv + (c - wt); }
};

// ---- out[slot][m][n] (+)= sum_{j in slice} F[j][m] R[j][n] ----------------------------------
// FROM_G = false: F = phi(K), R = [V | 1] (S^T [V | 1]);  true: F = phi(Q), R = G (rows of dv + 16, the backward pass).
template <typename T, bool FROM_G>
__global__ void __launch_bounds__(mma3::THREADS, 2)
state_kernel(const float* __restrict__ F, const T* __restrict__ V, TensorAddr av, const float* __restrict__ G, int H, int L, int M,
             int dv, int slice_len, int nslices, int per_slice_out, float* __restrict__ out, int flip, int* __restrict__ status) {
  fs_grid_dependency_wait();
  const int zi = mma3::unit_of(flip);
  extern __shared__ uint8_t smem[];
  const int bh = zi / nslices, sl = zi % nslices, b = bh / H, h = bh % H;
  const int m0 = blockIdx.x * mma3::ROWS, NP = dv + 16;
  const int j0 = sl * slice_len, j1 = min(L, j0 + slice_len);
  if (j0 >= j1) return;
  const ColTile ct(dv, blockIdx.y);
  mma3::Block blk;
  blk.begin(smem, ct.nt(), j1 - j0, status);
  const float* P = F + ((int64_t)bh * L + j0) * M + m0;
  const float* Gb = FROM_G ? G + ((int64_t)bh * L + j0) * NP : nullptr;
  const T* Vb = V + b * av.sb + h * av.sh + (int64_t)j0 * av.sl;
  constexpr int VP = FROM_G ? 3 : mma3::PartsOf<T>::N;
  blk.template segment<false, 3, false, VP>(
      j1 - j0, [&](int r, int k, mma3::Piece<3>& p) { if (m0 + r < M) p.load(P + (int64_t)k * M + r); else p.zero(); },
      [&](int c, int k, mma3::Piece<VP>& p) {
        if constexpr (FROM_G) {
          p.load(Gb + (int64_t)k * NP + ct.at(dv, c));
        } else {
          if (c < ct.wt) p.load(Vb + (int64_t)k * av.sl + ct.v0 + c);
          else if (c == ct.wt) p.unit();
          else p.zero();
        }
      });
  blk.finish();
  float* O = out + (int64_t)(per_slice_out ? zi : bh) * M * NP;
  blk.rows([&](int r, int c, float4 v) {
    if (m0 + r >= M || (c >= ct.wt && blockIdx.y > 0)) return;        // the ones block is written by the first tile
    float4* dst = reinterpret_cast<float4*>(O + (int64_t)(m0 + r) * NP + ct.at(dv, c));
    if (per_slice_out) *dst = v;
    else atomicAdd(dst, v);
  });
  blk.end();
}

// ---- exclusive running sum over the chunks, forwards (earlier chunks) or backwards (later chunks) ------
__global__ void __launch_bounds__(NTH)
prefix_kernel(float* __restrict__ st, int nchunks, int64_t elems, int reverse, int flip) {
  fs_grid_dependency_wait();
  const int bh = flip ? gridDim.y - 1 - blockIdx.y : blockIdx.y;
  float* base = st + (int64_t)bh * nchunks * elems;
  for (int64_t e = blockIdx.x * (int64_t)NTH + threadIdx.x; e < elems; e += (int64_t)gridDim.x * NTH) {
    float run = 0.f;
    // eight chunks at a time: the loads are issued together, then the running sums are stored
    for (int c0 = 0; c0 < nchunks; c0 += 8) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; u++) {
        const int c = reverse ? nchunks - 1 - (c0 + u) : c0 + u;
        v[u] = c0 + u < nchunks ? base[c * elems + e] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; u++) {
        const int c = reverse ? nchunks - 1 - (c0 + u) : c0 + u;
        if (c0 + u < nchunks) base[c * elems + e] = run;
        run += v[u];
      }
    }
  }
}

// Columns of a tile of a product over M features (mma3.cuh: LONG_K).
__host__ __device__ inline int tile_columns(int columns, int M) { return M > mma3::LONG_K && columns > 64 ? 64 : columns; }

// ---- masked in-chunk scores: sc[bh, c][i][j] = (j <= i) phiQ_i . phiK_j; tiles above the diagonal are neither written nor read
__global__ void __launch_bounds__(mma3::THREADS, 2)
scores_kernel(const float* __restrict__ phiQ, const float* __restrict__ phiK, int L, int M, int C, int nchunks,
              float* __restrict__ sc, int flip, int* __restrict__ status) {
  fs_grid_dependency_wait();
  const int zi = mma3::unit_of(flip);
  extern __shared__ uint8_t smem[];
  const int bh = zi / nchunks, c = zi % nchunks;
  const int cols = tile_columns(mma3::ROWS, M), i0 = blockIdx.x * mma3::ROWS, j0 = blockIdx.y * cols;
  if (j0 >= i0 + mma3::ROWS) return;
  mma3::Block blk;
  blk.begin(smem, cols, M, status);
  const int rows = min(C, L - c * C);                                  // the last chunk may be short
  const float* PQ = phiQ + ((int64_t)bh * L + (int64_t)c * C) * M;
  const float* PK = phiK + ((int64_t)bh * L + (int64_t)c * C) * M;
  blk.template segment<true, 3, true, 3>(
      M, [&](int r, int k, mma3::Piece<3>& p) { if (i0 + r < rows) p.load(PQ + (int64_t)(i0 + r) * M + k); else p.zero(); },
      [&](int n, int k, mma3::Piece<3>& p) { if (j0 + n < rows) p.load(PK + (int64_t)(j0 + n) * M + k); else p.zero(); });
  blk.finish();
  float* S = sc + (int64_t)zi * C * C;
  blk.rows([&](int r, int n, float4 v) {
    const int i = i0 + r, j = j0 + n;
    if (j + 1 > i) v.y = 0.f;
    if (j + 2 > i) v.z = 0.f;
    if (j + 3 > i) v.w = 0.f;
    if (j > i) v.x = 0.f;
    *reinterpret_cast<float4*>(S + (int64_t)i * C + j) = v;
  });
  blk.end();
}

__device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v) {
  *reinterpret_cast<uint2*>(p) = make_uint2(tc::pack_bf16(v.x, v.y), tc::pack_bf16(v.z, v.w));
}

}  // namespace
