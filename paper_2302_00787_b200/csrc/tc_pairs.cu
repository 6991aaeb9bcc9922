// Kernel estimates of (x, y) pairs over R feature draws (Section 2.1: Khat = sum_m P_m S_m) on the tensor cores at fp32
// precision (three-part bf16 operands, split3.cuh).
//
// With [x | y] as one row of 2 d values and [W1_m | W2_m] as one row per (draw, feature), the exponent of a summand is
// one dot product of length 2 d, so the batch is a [pairs x 2 d] x [2 d x R M] product whose epilogue takes exponentials
// and sums them per draw.  The fp32 kernel it replaces did the two products on the fp32 cores, rebuilt x^T C x for every
// draw and re-read W for every 64 pairs: 290 ms for 2^20 pairs, d = M = 64, R = 32, dense C.
//
// Block (one per SM, persistent) = tile of 128 pairs at a time.  Its 256 epilogue threads split the pairs' 2 d values
// into the three parts: h and m as swizzled shared-memory operands, l as a tensor-memory operand (it meets only the h
// part of W, and with it in shared memory d = 128 would not fit).  The parts of [W1 | W2] are written once per call as
// operand images (pair_images_kernel) and stream through a ring of bulk copies, 64 values of K at a time; every block
// reads all of them once per 128 pairs (L2).  Six MMAs per 16 values of K.  Two accumulators, one per warpgroup of the
// epilogue: while one warpgroup takes the exponentials of its tile the other's is multiplied.  A tile of columns holds
// whole draws (M <= 128) or one draw takes several tiles of the same warpgroup, so the sum over features stays in one
// thread.  The quadratic terms x^T C x are products with C as further columns, once per tile of pairs.
// The tensor core truncates the accumulator at every MMA, by up to one unit in the last place of its value at that
// point: the five products with m or l parts (2^-8 of the result and less) are therefore accumulated first and the h h
// products last, so that only the last 2 d / 16 steps round at the size of the result (mean error of an estimate at
// d = 64: 5.3e-6 with the products in any order, 0.9e-6 so, 0.8e-6 for the fp32 kernel).
// What those steps lose on average of a sum is put back as a factor on W and C (lost()): the mean error of the estimates was
// 0.40, 0.45, 1.25, 1.95 units of 2^-23 of the exponents' products at d = 16, 32, 64, 128 (PosRF, GERF and ADERF; all of one sign).
// Relative error of the estimates for points of norm 2, without it / with it / fp32 multiply-adds: d = M = 64, ADERF 2.3e-6 /
// 0.9e-6 / 1.2e-6; d = 128, M = 256, GERF 5.1e-6 / 2.2e-6 / 1.8e-6, SDERF, whose products are nearly all of one sign and lose
// more, 5.7e-6 / 2.4e-6 / 0.8e-6.  (Two accumulators for the h h products at d = 128: SDERF 2.3e-6, and 13 % longer.)
// Bound: tensor pipe (d = 64: 48 MMAs of N = 128 per tile, 3.1 k cycles, against 1.5 k issue cycles of exponentials per
// warpgroup).
#include "common.cuh"
#include "split3.cuh"
#include "tc_layout.cuh"

using namespace tc;
using namespace tcl;

namespace {

constexpr int PT_EPI = 256, PT_WARP_LOAD = 8, PT_WARP_MMA = 9, PT_THREADS = 320;
constexpr uint32_t PT_ACC = 128;                        // columns of one accumulator
constexpr uint32_t PT_LCOL = 2 * PT_ACC;                // first column of the l parts
constexpr uint32_t PT_TMEM = 512;
constexpr int PT_MAX_STAGES = 4;

// Geometry of one call, shared by the host, the image kernel and the main kernel.
struct PairGeom {
  int d, M, R;
  int nks;        // K slices of 64 values
  int kstep;      // MMA steps of 16 values per slice
  int J;          // column tiles per unit
  int dpu;        // draws per unit
  int NT;         // columns of a feature tile
  int nunits;
  int NQ, nqt;    // columns and number of the tiles that carry C
  int stages;
  __host__ __device__ uint32_t slice_bytes(int n) const { return 3u * (uint32_t)n * 128u; }
  __host__ __device__ size_t quad_tile(int q) const { return (size_t)q * nks * slice_bytes(NQ); }
  __host__ __device__ size_t feat_tile(int t) const { return quad_tile(nqt) + (size_t)t * nks * slice_bytes(NT); }
  __host__ __device__ uint32_t stage_bytes() const { return slice_bytes(NT > NQ ? NT : NQ); }
};

PairGeom pair_geom(int d, int M, int R) {
  PairGeom g{};
  g.d = d; g.M = M; g.R = R;
  const int K = 2 * d;
  g.nks = (K + 63) / 64;
  g.kstep = K < 64 ? K / 16 : 4;
  if (M <= 128) {
    g.J = 1;
    g.dpu = 128 / M;
    if (g.dpu > R) g.dpu = R;
    g.NT = g.dpu * M;
  } else {
    g.J = (M + 127) / 128;
    g.dpu = 1;
    g.NT = ((M + g.J - 1) / g.J + 15) / 16 * 16;
  }
  g.nunits = (R + g.dpu - 1) / g.dpu;
  g.NQ = K < 128 ? K : 128;
  g.nqt = K / g.NQ;
  const size_t room = 232448 - 1024 - 2048 - (size_t)g.nks * 2 * TILE_BYTES;
  g.stages = (int)(room / g.stage_bytes());
  if (g.stages > PT_MAX_STAGES) g.stages = PT_MAX_STAGES;
  return g;
}

// mean loss, relative, of a sum over n steps
__device__ __forceinline__ float lost(int n) { return (n <= 4 ? 0.4f : n <= 8 ? 1.25f : 1.95f) * 1.1920929e-7f; }

// One thread = 8 values of K of one column of one tile: three parts into the images (rows of 128 bytes, 128-byte swizzle).
__global__ void __launch_bounds__(256)
pair_images_kernel(PairGeom g, const float* __restrict__ prep, uint8_t* __restrict__ img, float* __restrict__ a2) {
  fs_grid_dependency_wait();
  PrepLayout pr{g.d, g.M};
  const int ntiles = g.nqt + g.nunits * g.J;
  const int nmax = g.NT > g.NQ ? g.NT : g.NQ;
  const int chunks = g.nks * 8;
  const size_t total = (size_t)ntiles * nmax * chunks;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % chunks), n = (int)(e / chunks % nmax), t = (int)(e / chunks / nmax);
    const bool quad = t < g.nqt;
    const int N = quad ? g.NQ : g.NT;
    if (n >= N) continue;
    const int k0 = c * 8;                       // first of this thread's values of K
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; j++) v[j] = 0.f;
    const int side = k0 < g.d ? 0 : 1, kk = k0 - side * g.d;
    if (k0 < 2 * g.d) {
      if (quad) {
        const int col = t * g.NQ + n;           // column of [C1 | C2], block diagonal
        if ((col < g.d) == (side == 0)) {
          const float* Cm = prep + (size_t)side * pr.total() + pr.Cmat();
          const int j2 = col - side * g.d;
#pragma unroll
          for (int j = 0; j < 8; j++) v[j] = fmaf(Cm[(kk + j) * g.d + j2], lost(g.d / 16), Cm[(kk + j) * g.d + j2]);
        }
      } else {
        const int u = (t - g.nqt) / g.J, jt = (t - g.nqt) % g.J;
        const int draw = u * g.dpu + (g.J == 1 ? n / g.M : 0), m = g.J == 1 ? n % g.M : jt * g.NT + n;
        if (draw < g.R && m < g.M) {
          const float* W = prep + ((size_t)draw * 2 + side) * pr.total() + pr.W() + (size_t)m * g.d + kk;
#pragma unroll
          for (int j = 0; j < 8; j++) v[j] = fmaf(W[j], lost(g.d / 8), W[j]);
          if (c == 0) a2[(size_t)(t - g.nqt) * g.NT + n] = 2.f * prep[(size_t)draw * 2 * pr.total() + pr.a() + m];
        } else if (c == 0) {
          a2[(size_t)(t - g.nqt) * g.NT + n] = 0.f;
        }
      }
    }
    uint4 h, mm, l;
    split3::split8(v, h, mm, l);
    uint8_t* base = img + (quad ? g.quad_tile(t) : g.feat_tile(t - g.nqt)) + (size_t)(c >> 3) * g.slice_bytes(N);
    const uint32_t off = (uint32_t)n * 128u + (uint32_t)(((c & 7) ^ (n & 7)) << 4);
    *reinterpret_cast<uint4*>(base + off) = h;
    *reinterpret_cast<uint4*>(base + (size_t)N * 128 + off) = mm;
    *reinterpret_cast<uint4*>(base + (size_t)2 * N * 128 + off) = l;
  }
}

struct PtMisc {
  uint64_t full[PT_MAX_STAGES], empty[PT_MAX_STAGES], a_full, t_full[2], t_free[2];
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(PtMisc) <= 512, "misc block");

// The order in which the column tiles of an item (units u0 .. u1-1) go through the accumulators: units in pairs, one per
// warpgroup, their tiles alternating.  f(unit, tile in unit, warpgroup) is called in that order until it returns false.
template <class F>
__device__ __forceinline__ void for_tiles(const PairGeom& g, int u0, int u1, F f) {
  for (int u = u0; u < u1; u += 2)
    for (int j = 0; j < g.J; j++)
      for (int w = 0; w < 2 && u + w < u1; w++)
        if (!f(u + w, j, w)) return;
}

// four consecutive values; rows of a caller's array need not start on a 16-byte boundary
__device__ __forceinline__ float4 load4(const float* p, bool vec) {
  if (vec) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], p[1], p[2], p[3]);
}

template <int D>
__global__ void __launch_bounds__(PT_THREADS, 1)
tc_pairs_kernel(PairGeom g, const float* __restrict__ X, const float* __restrict__ Y, int64_t np, const float* __restrict__ prep,
                const uint8_t* __restrict__ img, const float* __restrict__ a2, int usplit, int units_per_split, int nitems,
                float* __restrict__ est, int* __restrict__ status) {
  fs_grid_dependency_wait();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  constexpr int NKS = (2 * D + 63) / 64;
  constexpr bool KEEP = NKS <= 2;                  // the ring holds a whole tile: its slices are used twice
  constexpr uint32_t A_BYTES = NKS * 2 * TILE_BYTES;                     // [slice][h, m][128 rows x 128 bytes]
  uint8_t* sA = sm;
  uint8_t* sB = sm + A_BYTES;
  const uint32_t stage_bytes = g.stage_bytes();
  float* c_s = reinterpret_cast<float*>(sB + (size_t)g.stages * stage_bytes);     // [2][128] quadratic terms of x and of y
  PtMisc* misc = reinterpret_cast<PtMisc*>(c_s + 256);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abortp = &misc->abort_flag;
  PrepLayout pr{D, g.M};
  const float* scal1 = prep + pr.scal();
  const float* scal2 = prep + pr.total() + pr.scal();
  const bool scalar = scal1[PS_CSCALAR] != 0.f && scal2[PS_CSCALAR] != 0.f;
  const int nqt = scalar ? 0 : g.nqt;

  if (threadIdx.x == 0) {
    for (int i = 0; i < PT_MAX_STAGES; i++) { mbar_init(&misc->full[i], 1); mbar_init(&misc->empty[i], 1); }
    mbar_init(&misc->a_full, PT_EPI / 32);
    for (int i = 0; i < 2; i++) { mbar_init(&misc->t_full[i], 1); mbar_init(&misc->t_free[i], 4); }
    misc->abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == PT_WARP_MMA) {
    tmem_alloc(&misc->tmem_base, PT_TMEM);
    tmem_relinquish();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = misc->tmem_base;

  if (warp == PT_WARP_LOAD) {
    if (lane == 0) {
      int n = 0;                                     // slices issued
      bool ok = true;
      auto load_tile = [&](const uint8_t* src, uint32_t bytes) {
        for (int s = 0; s < (KEEP ? NKS : 2 * NKS) && ok; s++, n++) {
          const int st = n % g.stages;
          ok = mbar_wait(&misc->empty[st], ((n / g.stages) & 1) ^ 1, abortp, status);
          if (!ok) break;
          const uint32_t take = s < NKS ? bytes : bytes / 3;      // second pass: the h parts alone
          mbar_expect_tx(&misc->full[st], take);
          bulk_load(sB + (size_t)st * stage_bytes, src + (size_t)(s % NKS) * bytes, take, &misc->full[st]);
        }
        return ok;
      };
      for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
        const int u0 = item % usplit * units_per_split, u1 = min(g.nunits, u0 + units_per_split);
        for (int q = 0; q < nqt && ok; q++) load_tile(img + g.quad_tile(q), g.slice_bytes(g.NQ));
        if (ok) for_tiles(g, u0, u1, [&](int u, int j, int) { return load_tile(img + g.feat_tile(u * g.J + j), g.slice_bytes(g.NT)); });
      }
      // no copy of this block may still be in flight when it exits
      for (int i = max(0, n - g.stages); i < n; i++) mbar_wait(&misc->full[i % g.stages], (i / g.stages) & 1, abortp, status, false);
    }
  } else if (warp == PT_WARP_MMA) {
    // the whole warp walks the schedule, one elected lane issues
    int n = 0, used[2] = {0, 0}, it = 0;
    bool ok = true;
    const uint64_t dA0 = smem_desc(smem_u32(sA), 16, 1024, SWZ_128B), dB0 = smem_desc(smem_u32(sB), 16, 1024, SWZ_128B);
    const uint32_t ah = (uint32_t)(dA0 >> 32), bh = (uint32_t)(dB0 >> 32);
    auto tile = [&](int N, int w) {
      ok = __all_sync(0xffffffffu, mbar_wait(&misc->t_free[w], (used[w] & 1) ^ 1, abortp, status));
      if (!ok) return false;
      used[w]++;
      const uint32_t idesc = idesc_bf16(128, N, 0, 0), acc = tmem + w * PT_ACC;
      const int n0 = n;
      const uint32_t part = (uint32_t)N * 8;         // 128 N bytes in 16-byte units
      for (int q = 0; q < 2 * NKS; q++) {            // pass 0: the five small products; pass 1: h h
        const int pass = q >= NKS ? 1 : 0, s = q - pass * NKS;
        const bool fresh = pass == 0 || !KEEP;       // a slice that was just loaded
        const int idx = KEEP ? n0 + s : n0 + q, st = idx % g.stages;
        if (fresh) {
          ok = __all_sync(0xffffffffu, mbar_wait(&misc->full[st], (idx / g.stages) & 1, abortp, status));
          if (!ok) return false;
          n++;
        }
        tcgen05_fence_after();
        uint32_t al = (uint32_t)dA0 + s * (2 * TILE_BYTES / 16), bl = (uint32_t)dB0 + st * (stage_bytes / 16);
        opaque(al); opaque(bl);
        const uint32_t lcol = tmem + PT_LCOL + s * 32;
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < 4; k++) {
            if (k < g.kstep) {
              const uint32_t a_h = al + 2 * k, a_m = a_h + TILE_BYTES / 16, b_h = bl + 2 * k, b_m = b_h + part, b_l = b_m + part;
              if (pass == 0) {
                mma_bf16_ta_lh(acc, lcol + 8 * k, b_h, bh, idesc, (s | k) ? 1u : 0u);
                mma_bf16_lh(acc, a_h, ah, b_l, bh, idesc, 1u);
                mma_bf16_lh(acc, a_m, ah, b_m, bh, idesc, 1u);
                mma_bf16_lh(acc, a_m, ah, b_h, bh, idesc, 1u);
                mma_bf16_lh(acc, a_h, ah, b_m, bh, idesc, 1u);
              } else {
                mma_bf16_lh(acc, a_h, ah, b_h, bh, idesc, 1u);
              }
            }
          }
          if (pass == 1 || !KEEP) mma_commit(&misc->empty[st]);
          if (q == 2 * NKS - 1) mma_commit(&misc->t_full[w]);
        }
        __syncwarp();
      }
      return true;
    };
    for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x, it++) {
      const int u0 = item % usplit * units_per_split, u1 = min(g.nunits, u0 + units_per_split);
      ok = __all_sync(0xffffffffu, mbar_wait(&misc->a_full, it & 1, abortp, status));
      if (!ok) break;
      tcgen05_fence_after();
      for (int q = 0; q < nqt && ok; q++) tile(g.NQ, 0);
      if (ok) for_tiles(g, u0, u1, [&](int, int, int w) { return tile(g.NT, w); });
    }
  } else {
    // Epilogue warpgroups; thread = pair.  A wait that runs out leaves the results undefined (the status word says so)
    // and the thread goes on, so that all 256 threads keep meeting at the named barriers.
    const int w = threadIdx.x >> 7, row = threadIdx.x & 127;
    const uint32_t lanes = tmem + ((uint32_t)(row & ~31) << 16);
    const float bias2 = 2.f * scal1[PS_BIAS];
    const bool vec = ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15) == 0;
    int used = 0;
    for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
      const int64_t p = (int64_t)(item / usplit) * TILE + row;
      const int u0 = item % usplit * units_per_split, u1 = min(g.nunits, u0 + units_per_split);
      // operand parts of this tile: warpgroup 0 takes x, warpgroup 1 takes y
      named_bar_sync(1, PT_EPI);                     // the previous tile's products have been read by both warpgroups
      {
        const float* src = (w ? Y : X) + p * D;
        float sq[4] = {};
#pragma unroll
        for (int c0 = 0; c0 < D / 8; c0 += 2) {      // 16 values per step: eight columns of l parts
          uint32_t lreg[8];
#pragma unroll
          for (int cc = 0; cc < 2; cc++) {
            const int c = c0 + cc;
            float v[8] = {};
            if (p < np) {
              const float4 v0 = load4(src + 8 * c, vec), v1 = load4(src + 8 * c + 4, vec);
              v[0] = v0.x; v[1] = v0.y; v[2] = v0.z; v[3] = v0.w; v[4] = v1.x; v[5] = v1.y; v[6] = v1.z; v[7] = v1.w;
            }
#pragma unroll
            for (int j = 0; j < 8; j++) sq[j & 3] = fmaf(v[j], v[j], sq[j & 3]);
            uint4 h, m, l;
            split3::split8(v, h, m, l);
            const int kc = w * (D / 8) + c;          // 16-byte piece along K
            uint8_t* dst = sA + (size_t)(kc >> 3) * 2 * TILE_BYTES + row * 128 + (((kc & 7) ^ (row & 7)) << 4);
            *reinterpret_cast<uint4*>(dst) = h;
            *reinterpret_cast<uint4*>(dst + TILE_BYTES) = m;
            lreg[4 * cc] = l.x; lreg[4 * cc + 1] = l.y; lreg[4 * cc + 2] = l.z; lreg[4 * cc + 3] = l.w;
          }
          tmem_st8(lanes + PT_LCOL + (w * (D / 8) + c0) * 4, lreg);
        }
        if (nqt == 0) c_s[w * 128 + row] = ((sq[0] + sq[1]) + (sq[2] + sq[3])) * (w ? scal2 : scal1)[PS_CGAMMA];
        tmem_wait_st();
        fence_proxy_async_smem();
        tcgen05_fence_before();
        mbar_arrive_warp(&misc->a_full, lane);
      }
      if (w == 0) {
        float q01[2] = {0.f, 0.f};
        for (int q = 0; q < nqt; q++) {
          mbar_wait(&misc->t_full[0], used & 1, abortp, status);
          used++;
          __syncwarp();
          tcgen05_fence_after();
          for (int c = 0; c < g.NQ / 16; c++) {
            uint32_t t[16];
            tmem_ld16(lanes + c * 16, t);
            tmem_wait_ld();
            const int col = q * g.NQ + c * 16, s = col < D ? 0 : 1;
            if (p < np) {
              const float* src = (s ? Y : X) + p * D + col - s * D;
              float sum = 0.f;
#pragma unroll
              for (int j = 0; j < 16; j += 4) {
                const float4 v = load4(src + j, vec);
                sum = fmaf(__uint_as_float(t[j]), v.x, sum);
                sum = fmaf(__uint_as_float(t[j + 1]), v.y, sum);
                sum = fmaf(__uint_as_float(t[j + 2]), v.z, sum);
                sum = fmaf(__uint_as_float(t[j + 3]), v.w, sum);
              }
              q01[s] += sum;
            }
          }
          tcgen05_fence_before();
          mbar_arrive_warp(&misc->t_free[0], lane);
        }
        if (nqt) { c_s[row] = q01[0]; c_s[128 + row] = q01[1]; }
      }
      named_bar_sync(1, PT_EPI);
      const float base = bias2 + c_s[row] + c_s[128 + row];
      float sum = 0.f;
      for_tiles(g, u0, u1, [&](int u, int j, int tw) {
        if (tw != w) return true;
        mbar_wait(&misc->t_full[w], used & 1, abortp, status);
        used++;
        __syncwarp();
        tcgen05_fence_after();
        const float* at = a2 + (size_t)(u * g.J + j) * g.NT;
        const int cols = g.J == 1 ? g.NT : min(g.NT, g.M - j * g.NT);
        int left = g.J == 1 ? g.M : g.M - j * g.NT;   // columns of the running draw from this tile's position on
        int draw = u * g.dpu;
        for (int c = 0; c < cols; c += 16) {
          uint32_t t[16];
          tmem_ld16(lanes + w * PT_ACC + c, t);
          float am[16];
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(at + c + i));
            am[i] = v.x; am[i + 1] = v.y; am[i + 2] = v.z; am[i + 3] = v.w;
          }
          tmem_wait_ld();
          float s0 = 0.f, s1 = 0.f;
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            s0 += expf(__uint_as_float(t[i]) + (base + am[i]));
            s1 += expf(__uint_as_float(t[i + 1]) + (base + am[i + 1]));
          }
          sum += s0 + s1;
          left -= 16;
          if (left == 0) {
            if (p < np && draw < g.R) est[(int64_t)draw * np + p] = sum;
            sum = 0.f;
            draw++;
            left = g.M;
          }
        }
        tcgen05_fence_before();
        mbar_arrive_warp(&misc->t_free[w], lane);
        return true;
      });
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == PT_WARP_MMA) {
    tcgen05_fence_after();
    tmem_dealloc(tmem, PT_TMEM);
  }
}

}  // namespace

size_t fs_tc_pairs_scratch_bytes(int d, int M, int R) {
  const PairGeom g = pair_geom(d, M, R);
  return ws_round(g.feat_tile(g.nunits * g.J)) + ws_round((size_t)g.nunits * g.J * g.NT * 4);
}

// est [R][np] from X, Y [np][d] and the prep blocks of the R draws
int fs_tc_pairs(fsharp_ctx* ctx, const float* X, const float* Y, int64_t np, int d, int M, int R, const float* prep, float* est,
                WsAlloc* ws) {
  const PairGeom g = pair_geom(d, M, R);
  uint8_t* img = ws->take<uint8_t>(g.feat_tile(g.nunits * g.J));
  float* a2 = ws->take<float>((size_t)g.nunits * g.J * g.NT);
  const int64_t ptiles = (np + TILE - 1) / TILE;
  // few tiles of pairs: the draws are divided as well, so that every SM has an item
  int usplit = (int)((ctx->sm_count + ptiles - 1) / ptiles);
  if (usplit > g.nunits) usplit = g.nunits;
  if (usplit < 1) usplit = 1;
  const int ups = (g.nunits + usplit - 1) / usplit;
  usplit = (g.nunits + ups - 1) / ups;
  if (ptiles * usplit > 2147483647LL) return FSHARP_E_SHAPE;
  const int nitems = (int)(ptiles * usplit);
  const size_t nthr = (size_t)(g.nqt + g.nunits * g.J) * (g.NT > g.NQ ? g.NT : g.NQ) * g.nks * 8;
  FS_TIME_BEGIN(ctx, FS_K_PAIR_IMAGES);
  (void)fs_launch_chained(pair_images_kernel, dim3((unsigned)((nthr + 255) / 256)), dim3(256), 0, ctx->stream, g, prep, img, a2);
  FS_TIME_END(ctx);
  FS_LAUNCH_CHECK(ctx);
  const int grid = nitems < ctx->sm_count ? nitems : ctx->sm_count;
  const size_t smem = 1024 + (size_t)g.nks * 2 * TILE_BYTES + (size_t)g.stages * g.stage_bytes() + 1024 + sizeof(PtMisc);
#define FS_TCP(DD)                                                                                                       \
  do {                                                                                                                   \
    FS_CUDA_OK(fs_allow_smem(tc_pairs_kernel<DD>));                                                                       \
    FS_TIME_BEGIN(ctx, FS_K_PAIRS);                                                                                       \
    (void)fs_launch_chained(tc_pairs_kernel<DD>, grid, dim3(PT_THREADS), smem, ctx->stream, g, X, Y, np, prep, img, a2, usplit, ups, nitems, est,    \
                                                                 ctx->d_status);                                         \
    FS_TIME_END(ctx);                                                                                                     \
  } while (0)
  switch (d) {
    case 16: FS_TCP(16); break;
    case 32: FS_TCP(32); break;
    case 64: FS_TCP(64); break;
    case 128: FS_TCP(128); break;
    default: return FSHARP_E_SHAPE;
  }
#undef FS_TCP
  FS_LAUNCH_CHECK(ctx);
  return FSHARP_OK;
}
