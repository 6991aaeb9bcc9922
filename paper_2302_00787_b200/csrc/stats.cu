// Set statistics of Theorems 4.2 and 4.3: M1 = L^-1 sum x x^T, M2 = L^-1 sum y y^T,
// mu4 = mean x, mu5 = mean y.
//
// One thread block accumulates the Gram matrix of a slice of tokens of one
// (batch, head, side): products in fp32 over 64 tokens, then folded into fp64
// registers; slices are combined with fp64 atomics.  Tokens are read in 16-byte pieces: base and strides are multiples of 16 bytes
// (the entry points refuse others).
#include "common.cuh"

namespace {

// A thread has R x R products of one token after the other (rows and columns in pieces of four, one 16-byte load each);
// the (D / R)^2 threads that cover the matrix form a group, and the groups of a block share out the tokens of a tile.  The next tile's loads
// are in flight under this one's products.  (A matrix over the whole block at every d, 2 x 2 products at d = 32 for four
// loads, a tile of 32 tokens at a time and its loads waited for: 24 us for 2 x 32 x 1501 tokens.)
constexpr int ST_THREADS = 256;
template <int D> struct StGeo {
  static constexpr int R = D == 128 ? 8 : 4, TPG = (D / R) * (D / R), NG = ST_THREADS / TPG, TT = 4096 / D;      // tokens per tile
  static constexpr int FLUSH = 64 / (TT / NG);       // tiles between fp32 -> fp64 folds: 64 tokens of a thread
  static constexpr int LD = D + 4;
};

// the tile's values that this thread brings: 16-byte pieces
template <typename T, int D> struct StTile {
  static constexpr int E = 16 / sizeof(T), N = 4096 / E / ST_THREADS;
  uint4 r[N];
  __device__ __forceinline__ void load(const T* X, int64_t sl, int rows, int tid) {
#pragma unroll
    for (int u = 0; u < N; u++) {
      const int e = (tid + u * ST_THREADS) * E, t = e / D, c = e % D;
      r[u] = t < rows ? *reinterpret_cast<const uint4*>(X + (int64_t)t * sl + c) : make_uint4(0u, 0u, 0u, 0u);
    }
  }
  __device__ __forceinline__ void store(float* xs, float scale, int tid, bool& bad) const {
#pragma unroll
    for (int u = 0; u < N; u++) {
      const int e = (tid + u * ST_THREADS) * E, t = e / D, c = e % D;
      const uint32_t w[4] = {r[u].x, r[u].y, r[u].z, r[u].w};
      float v[E];
#pragma unroll
      for (int j = 0; j < E; j++) {
        v[j] = scale * (sizeof(T) == 4 ? __uint_as_float(w[j]) : __uint_as_float(j & 1 ? w[j / 2] & 0xffff0000u : w[j / 2] << 16));
        bad |= !isfinite(v[j]);
      }
#pragma unroll
      for (int j = 0; j < E; j += 4) *reinterpret_cast<float4*>(xs + t * StGeo<D>::LD + c + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    }
  }
};

template <typename T, int D>
__global__ void __launch_bounds__(ST_THREADS)
stats_kernel(const T* __restrict__ Q, const T* __restrict__ K, TensorAddr aq, TensorAddr ak, int H, int Lq, int Lk,
             int pool, int Bpool, float qk_scale, int tokens_per_split, double* __restrict__ stats,
             int* __restrict__ status) {
  using G = StGeo<D>;
  constexpr int R = G::R, NG = G::NG, TT = G::TT, LD = G::LD, SUB = ST_THREADS / D;
  __shared__ __align__(16) float xs[TT * LD];
  __shared__ double sums[NG > 1 ? D * D : 1], cols[ST_THREADS];
  const int side = blockIdx.z;           // 0: queries, 1: keys
  const int bh = blockIdx.y;
  const int b = bh / H, h = bh % H;
  const int L = side ? Lk : Lq;
  const TensorAddr ad = side ? ak : aq;
  const T* X = (side ? K : Q) + b * ad.sb + h * ad.sh;
  const int t0 = blockIdx.x * tokens_per_split;
  const int t1 = min(L, t0 + tokens_per_split);
  if (t0 >= t1) return;
  const int g = pool == FSHARP_POOL_PER_BH ? bh : h;
  const int tid = threadIdx.x, grp = tid / G::TPG, tx = tid % G::TPG % (D / R), ty = tid % G::TPG / (D / R);
  // row / column of the thread's products: pieces of four, D / 2 apart where there are two
  const auto at = [](int i, int x) { return (i & 3) + 4 * x + (i >> 2) * (D / 2); };

  float acc[R][R];
  double accd[R][R];
#pragma unroll
  for (int i = 0; i < R; i++)
#pragma unroll
    for (int j = 0; j < R; j++) { acc[i][j] = 0.f; accd[i][j] = 0.0; }
  float colacc = 0.f;                    // column tid % D over every SUB-th token
  double colaccd = 0.0;
  bool bad = false;
  int since = 0;
  StTile<T, D> tile;
  tile.load(X + (int64_t)t0 * ad.sl, ad.sl, t1 - t0, tid);
  for (int tb = t0; tb < t1; tb += TT) {
    tile.store(xs, qk_scale, tid, bad);
    __syncthreads();
    if (tb + TT < t1) tile.load(X + (int64_t)(tb + TT) * ad.sl, ad.sl, t1 - tb - TT, tid);
    const int n = min(TT, t1 - tb);      // (rows up to the tile's end are zeros)
#pragma unroll 4
    for (int t = grp; t < n; t += NG) {
      float a[R], bb[R];
#pragma unroll
      for (int i = 0; i < R; i += 4) {
        const float4 u = *reinterpret_cast<const float4*>(xs + t * LD + at(i, ty)), v = *reinterpret_cast<const float4*>(xs + t * LD + at(i, tx));
        a[i] = u.x; a[i + 1] = u.y; a[i + 2] = u.z; a[i + 3] = u.w;
        bb[i] = v.x; bb[i + 1] = v.y; bb[i + 2] = v.z; bb[i + 3] = v.w;
      }
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) acc[i][j] = fmaf(a[i], bb[j], acc[i][j]);
    }
#pragma unroll 4
    for (int t = tid / D; t < n; t += SUB) colacc += xs[t * LD + tid % D];
    __syncthreads();
    if (++since == G::FLUSH) {
      since = 0;
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) { accd[i][j] += (double)acc[i][j]; acc[i][j] = 0.f; }
      colaccd += (double)colacc;
      colacc = 0.f;
    }
  }
  const double inv = 1.0 / ((double)L * (double)Bpool);
  StatsLayout sl{D};
  double* out = stats + (size_t)g * sl.total();
  double* Mo = out + sl.M(side + 1);
  cols[tid] = colaccd + (double)colacc;
  if (NG > 1) {
    for (int k = 0; k < NG; k++) {
      if (grp == k)
#pragma unroll
        for (int i = 0; i < R; i++)
#pragma unroll
          for (int j = 0; j < R; j++) {
            double* s = &sums[at(i, ty) * D + at(j, tx)];
            *s = (k ? *s : 0.0) + (accd[i][j] + (double)acc[i][j]);
          }
      __syncthreads();
    }
    for (int e = tid; e < D * D; e += ST_THREADS) atomicAdd(&Mo[e], sums[e] * inv);
  } else {
    __syncthreads();
    // four lanes exchange their pieces of four columns, so that an instruction's atomics fill 32-byte sectors (2 x 4096 tokens, d = 128, 128
    // tokens per block: 36.4 us without, 27.6 so)
    const int t = tx & 3;
#pragma unroll
    for (int i = 0; i < R; i++)
#pragma unroll
      for (int p = 0; p < R; p += 4) {
        double v[4];
#pragma unroll
        for (int j = 0; j < 4; j++) v[j] = (accd[i][p + j] + (double)acc[i][p + j]) * inv;
#pragma unroll
        for (int o = 1; o < 4; o *= 2)
#pragma unroll
          for (int j = 0; j < 4; j++)
            if (!(j & o)) {
              const double got = __shfl_xor_sync(0xffffffffu, t & o ? v[j] : v[j | o], o);
              if (t & o) v[j] = got; else v[j | o] = got;
            }
#pragma unroll
        for (int j = 0; j < 4; j++) atomicAdd(&Mo[(size_t)at(i, ty) * D + at(p, (tx & ~3) + j) + t], v[j]);
      }
  }
  if (tid < D) {
    double c = 0.0;
#pragma unroll
    for (int k = 0; k < SUB; k++) c += cols[k * D + tid];
    atomicAdd(&out[sl.mu(side + 4) + tid], c * inv);
  }
  if (bad) atomicExch(status, FSHARP_E_NONFINITE);
}

template <typename T>
int launch_stats(fsharp_ctx* ctx, const void* Q, const void* K, const fsharp_dims* dm, float qk_scale,
                 double* stats) {
  const int BH = dm->B * dm->H;
  const int Lmax = dm->Lq > dm->Lk ? dm->Lq : dm->Lk;
  // The split with the least work on the fullest SM, over the blocks that have tokens.  A block's start, its fold and its atomics cost as much as
  // some 600 tokens at d = 16, 200, 100 and 70 at d = 32, 64 and 128; d = 128: one block on an SM at a time, else two, which together take
  // one and a half times as long as one (chosen over 230 shapes and their splits).  (As many blocks as
  // are resident for two sequences of the longer length, rounded down: 75 x 1024 tokens, d = 64, 83.5 us, 71 for four blocks per SM's worth before the
  // tokens were shared out, 60 so; 2 x 512 queries and 8192 keys, d = 128, 49, 36 and 31; 40 x 4096, d = 128, 490, 597 and 313.)
  const int64_t start = 64 + 140000 / (dm->d * dm->d);
  const int most = (Lmax + 127) / 128 < 4 * ctx->sm_count ? (Lmax + 127) / 128 : 4 * ctx->sm_count;
  int nsplit = 1, tps = 0;
  int64_t least = 0;
  for (int n = 1; n <= most; n++) {
    const int t = ((Lmax + n - 1) / n + 31) / 32 * 32;
    if ((Lmax + t - 1) / t != n) continue;
    const int64_t blocks = (int64_t)BH * ((dm->Lq + t - 1) / t + (dm->Lk + t - 1) / t), per = (blocks + ctx->sm_count - 1) / ctx->sm_count;
    const int64_t cost = (dm->d == 128 ? 2 * per : 3 * (per / 2) + 2 * (per % 2)) * (t + start);
    if (tps == 0 || cost < least) { least = cost; nsplit = n; tps = t; }
  }
  dim3 grid(nsplit, BH, 2);
  TensorAddr aq = fs_addr(dm->q_stride, dm->H, dm->Lq, dm->d);
  TensorAddr ak = fs_addr(dm->k_stride, dm->H, dm->Lk, dm->d);
  const int Bpool = dm->pool == FSHARP_POOL_PER_BH ? 1 : dm->B;
#define FS_ST(DD)                                                                                           \
  stats_kernel<T, DD><<<grid, ST_THREADS, 0, ctx->stream>>>((const T*)Q, (const T*)K, aq, ak, dm->H, dm->Lq, \
                                                            dm->Lk, dm->pool, Bpool, qk_scale, tps, stats,   \
                                                            ctx->d_status)
  FS_TIME_BEGIN(ctx, FS_K_STATS);
  switch (dm->d) {
    case 16: FS_ST(16); break;
    case 32: FS_ST(32); break;
    case 64: FS_ST(64); break;
    case 128: FS_ST(128); break;
    default: return FSHARP_E_SHAPE;
  }
#undef FS_ST
  FS_TIME_END(ctx);
  FS_LAUNCH_CHECK(ctx);
  return FSHARP_OK;
}

}  // namespace

int fs_run_stats(fsharp_ctx* ctx, const void* Q, const void* K, const fsharp_dims* dm, int dtype,
                 float qk_scale, double* stats) {
  const int G = fs_groups(dm);
  FS_CUDA_OK(cudaMemsetAsync(stats, 0, (size_t)G * StatsLayout{dm->d}.total() * sizeof(double), ctx->stream));
  if (dm->Lq == 0 && dm->Lk == 0) return FSHARP_OK;
  if (ctx->impl != FSHARP_IMPL_SIMT && fs_tc_stats_supported(Q, K, dm, dtype)) return fs_tc_stats(ctx, Q, K, dm, qk_scale, stats);
  if (dtype == FSHARP_F32) return launch_stats<float>(ctx, Q, K, dm, qk_scale, stats);
  return launch_stats<__nv_bfloat16>(ctx, Q, K, dm, qk_scale, stats);
}
