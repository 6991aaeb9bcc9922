// Attention at fp32 precision: features from feat3.cu, the linear-attention contraction (Sections 2.1 / 2.2), bidirectional and
// causal-chunked, on the tensor cores with three-part bf16 operands (mma3.cuh); and the chain of bf16 kernels for d = dv = 128.
// Used for fp32 inputs, for shapes the fused tensor-core kernels do not take, and on request (FSHARP_IMPL_SIMT: the name is older
// than the kernels).
//
// Scratch (from the context workspace): the two feature matrices, the per-token
// quadratic term, S^T [V | 1] (per (batch, head); per chunk when causal) and, when
// causal, the masked in-chunk score blocks.
#include "common.cuh"
#include "feat3.cuh"
#include "f32_parts.cuh"

namespace {

// ---- Y = num / den -------------------------------------------------------------------
// Bidirectional: [num | den] = phiQ (S^T [V | 1]).  Causal: per chunk, phiQ_c times the
// prefix state plus the masked scores times [V_c | 1].
template <typename T>
__global__ void __launch_bounds__(mma3::THREADS, 2)
out_kernel(const float* __restrict__ phiQ, const float* __restrict__ KV, const float* __restrict__ sc,
           const T* __restrict__ V, TensorAddr av, T* __restrict__ Y, TensorAddr ay, int H, int L, int M, int dv,
           int causal, int C, int nchunks, const float* __restrict__ lsq, const float* __restrict__ lsk, int flip,
           int* __restrict__ status) {
  fs_grid_dependency_wait();
  // lsq != nullptr: the unnormalised operator Khat C of Section 2.1 is wanted: row i of the numerator times
  // exp(lsq[i] + lsk[bh]), the shifts that the feature kernels took out of phi(Q) and phi(K), without their factors 2^LIFT (taken
  // off the sums, not off exp(), which may be next to the smallest number as it is)
  extern __shared__ uint8_t smem[];
  __shared__ float inv_s[mma3::ROWS];
  const int bh = mma3::unit_of(flip), b = bh / H, h = bh % H, NP = dv + 16;
  const int i0 = blockIdx.x * mma3::ROWS;
  const ColTile ct(dv, blockIdx.y);
  mma3::Block blk;
  blk.begin(smem, ct.nt(), M + (causal ? C : 0), status);
  const float* PQ = phiQ + ((int64_t)bh * L + i0) * M;
  const int chunk = causal ? i0 / C : 0;
  const float* S = KV + (int64_t)(causal ? bh * nchunks + chunk : bh) * M * NP;
  const T* Vb = V + b * av.sb + h * av.sh;
  blk.template segment<true, 3, false, 3>(
      M, [&](int r, int k, mma3::Piece<3>& p) { if (i0 + r < L) p.load(PQ + (int64_t)r * M + k); else p.zero(); },
      [&](int c, int k, mma3::Piece<3>& p) { p.load(S + (int64_t)k * NP + ct.at(dv, c)); });
  if (causal) {
    const int ic = i0 - chunk * C;                    // row offset inside the chunk; keys beyond the tile are masked
    const float* SC = sc + (((int64_t)bh * nchunks + chunk) * C + ic) * C;
    const T* Vc = Vb + (int64_t)chunk * C * av.sl;
    const int keys = min(ic + mma3::ROWS, L - chunk * C);
    constexpr int VP = mma3::PartsOf<T>::N;
    // (the score tiles are complete to 128 columns: with `keys` short of that the V rows beyond it count as zero)
    blk.template segment<true, 3, false, VP>(
        (keys + 7) & ~7, [&](int r, int k, mma3::Piece<3>& p) { p.load(SC + (int64_t)r * C + k); },
        [&](int c, int k, mma3::Piece<VP>& p) {
          if (k >= keys) p.zero();
          else if (c < ct.wt) p.load(Vc + (int64_t)k * av.sl + ct.v0 + c);
          else if (c == ct.wt) p.unit();
          else p.zero();
        });
  }
  blk.finish();
  if (threadIdx.x < mma3::ROWS) {
    const float den = blk.column(ct.wt);
    const int64_t i = i0 + (int)threadIdx.x;
    float inv = 0.f;
    if (i < L) {
      if (lsq != nullptr) {
        inv = expf(lsq[(int64_t)bh * L + i] + lsk[bh]);
      } else {
        if (!(den > 0.f) || !isfinite(den)) atomicExch(status, FSHARP_E_NONFINITE);
        inv = 1.f / den;
      }
    }
    inv_s[threadIdx.x] = inv;
  }
  __syncthreads();
  const float unlift = lsq != nullptr ? 1.f / (float)(1ull << 2 * feat3::LIFT) : 1.f;
  T* Yb = Y + b * ay.sb + h * ay.sh + (int64_t)i0 * ay.sl;
  blk.rows([&](int r, int c, float4 v) {
    if (i0 + r >= L || c >= ct.wt) return;
    const float inv = inv_s[r];
    store4(Yb + (int64_t)r * ay.sl + ct.v0 + c, make_float4(unlift * v.x * inv, unlift * v.y * inv, unlift * v.z * inv, unlift * v.w * inv));
  });
  blk.end();
}

template <typename T>
int attend_t(fsharp_ctx* ctx, const void* Q, const void* K, const void* V, const fsharp_dims* dm, int causal,
             int chunk, float qk_scale, const float* prep, void* Y, WsAlloc* ws, bool unnormalised) {
  const int B = dm->B, H = dm->H, BH = B * H, Lq = dm->Lq, Lk = dm->Lk, d = dm->d, dv = dm->dv, M = dm->M;
  const int NP = dv + 16, ctiles = (dv + 63) / 64;
  TensorAddr aq = fs_addr(dm->q_stride, H, Lq, d), ak = fs_addr(dm->k_stride, H, Lk, d);
  TensorAddr av = fs_addr(dm->v_stride, H, Lk, dv), ay = fs_addr(dm->y_stride, H, Lq, dv);
  // causal, bf16 tensors, d = dv = 128: scores, per-chunk sums and query side from bf16 features
  const bool tc = causal && !unnormalised && sizeof(T) == 2 && d == 128 && ctx->impl != FSHARP_IMPL_SIMT &&
                  fs_tc_kv128_supported(V, av, dv, M, chunk) && fs_tc_out128_supported(Y, ay);
  float* phiQ = tc ? nullptr : ws->take<float>((size_t)BH * Lq * M);
  float* phiK = tc ? nullptr : ws->take<float>((size_t)BH * Lk * M);
  __nv_bfloat16* phiQ16 = tc ? ws->take<__nv_bfloat16>((size_t)BH * Lq * M) : nullptr;
  __nv_bfloat16* phiK16 = tc ? ws->take<__nv_bfloat16>((size_t)BH * Lk * M) : nullptr;
  float* rowc = ws->take<float>((size_t)BH * Lk);
  unsigned* gmax = ws->take<unsigned>((size_t)BH);
  float* rowcq = ws->take<float>((size_t)BH * Lq);
  float* lsq = ws->take<float>((size_t)BH * Lq);
  float* lsk = ws->take<float>((size_t)BH);
  uint8_t* img = ws->take<uint8_t>(feat3::image_bytes(fs_groups(dm), d, M, 2));
  const feat3::Task tasks[2] = {{K, ak, Lk, 2, FSHARP_STAB_GROUP, rowc, gmax, phiK, phiK16, lsk, feat3::LIFT},
                                {Q, aq, Lq, 1, FSHARP_STAB_ROW, rowcq, nullptr, phiQ, phiQ16, lsq, feat3::LIFT}};
  float* KV = causal ? nullptr : ws->take<float>((size_t)BH * M * NP);
  FS_TRY(feat3::run(ctx, tasks, 2, sizeof(T) == 2 ? FSHARP_BF16 : FSHARP_F32, B, H, d, M, dm->pool, prep, qk_scale, img, KV,
                    causal ? 0 : (size_t)BH * M * NP));
  const dim3 gout((Lq + mma3::ROWS - 1) / mma3::ROWS, ctiles, BH);
  const dim3 gkv((M + mma3::ROWS - 1) / mma3::ROWS, ctiles, 1);
  if (!causal) {
    int slen = 0;
    const int nsl = fs_token_slices(ctx, BH * gkv.x * gkv.y, BH, Lk, &slen);
    FS_TRY(mma3::launch(ctx, FS_K_KV, state_kernel<T, false>, dim3(gkv.x, gkv.y, BH * nsl), phiK, (const T*)V, av, nullptr, H, Lk, M, dv, slen, nsl, 0,
                        KV, 0, ctx->d_status));
    FS_TRY(mma3::launch(ctx, FS_K_OUT, out_kernel<T>, gout, phiQ, KV, nullptr, (const T*)V, av, (T*)Y, ay, H, Lq, M, dv, 0, 0, 1,
                        unnormalised ? lsq : nullptr, lsk, 1, ctx->d_status));
    return FSHARP_OK;
  }
  if (tc) {
    const int C = chunk, nch = Lq / C;
    const int slots = fs_tc_kv128_slots(ctx, BH, M, nch);
    const int64_t elems = (int64_t)M * (dv + 1);
    float* tot = ws->take<float>((size_t)BH * slots * elems);
    __nv_bfloat16* st16 = ws->take<__nv_bfloat16>((size_t)BH * nch * M * dv);
    __nv_bfloat16* z16 = ws->take<__nv_bfloat16>((size_t)BH * nch * M);
    if (slots > 1) {
      FS_TRY(fs_tc_kv128(ctx, phiK16, V, av, B, H, Lk, M, C, tot, nullptr, nullptr));
      FS_TIME_BEGIN(ctx, FS_K_PREFIX);
      (void)fs_launch_chained(prefix_kernel, dim3((unsigned)((elems + NTH - 1) / NTH), BH), dim3(NTH), 0, ctx->stream, tot, slots, elems, 0, 0);
      FS_TIME_END(ctx);
      FS_LAUNCH_CHECK(ctx);
    }
    FS_TRY(fs_tc_kv128(ctx, phiK16, V, av, B, H, Lk, M, C, tot, st16, z16));
    return fs_tc_out128(ctx, phiQ16, phiK16, st16, z16, V, av, Y, ay, B, H, Lq, M, C);
  }
  const int C = inner_chunk(chunk), nch = (Lq + C - 1) / C;
  const int64_t elems = (int64_t)M * NP;
  float* st = ws->take<float>((size_t)BH * nch * elems);
  float* sc = ws->take<float>((size_t)BH * nch * C * C);
  FS_TRY(mma3::launch(ctx, FS_K_KV, state_kernel<T, false>, dim3(gkv.x, gkv.y, BH * nch), phiK, (const T*)V, av, nullptr, H, Lk, M, dv, C, nch, 1, st, 0,
                      ctx->d_status));
  FS_TIME_BEGIN(ctx, FS_K_PREFIX);
  (void)fs_launch_chained(prefix_kernel, dim3((unsigned)((elems + NTH - 1) / NTH), BH), dim3(NTH), 0, ctx->stream, st, nch, elems, 0, 1);
  FS_TIME_END(ctx);
  FS_LAUNCH_CHECK(ctx);
  FS_TRY(mma3::launch(ctx, FS_K_SCORES, scores_kernel, dim3(C / mma3::ROWS, C / tile_columns(mma3::ROWS, M), BH * nch), phiQ, phiK, Lq, M, C, nch, sc, 1,
                      ctx->d_status));
  return mma3::launch(ctx, FS_K_OUT, out_kernel<T>, gout, phiQ, st, sc, (const T*)V, av, (T*)Y, ay, H, Lq, M, dv, 1, C, nch, nullptr,
                      nullptr, 0, ctx->d_status);
}

}  // namespace

int fs_simt_featurize(fsharp_ctx* ctx, const void* X, int dtype, TensorAddr ax, int B, int H, int L, int d,
                      int M, int pool, const float* prep, int side, float qk_scale, int stab,
                      float* rowc, unsigned* gmax, float* phi, float* logscale, uint8_t* img) {
  const feat3::Task task{X, ax, L, side, stab, rowc, gmax, phi, nullptr, logscale, 0};
  return feat3::run(ctx, &task, 1, dtype, B, H, d, M, pool, prep, qk_scale, img);
}

size_t fs_simt_attend_scratch_bytes(const fsharp_ctx* ctx, const fsharp_dims* dm, int causal, int chunk) {
  const size_t BH = (size_t)dm->B * dm->H, NP = dm->dv + 16;
  const size_t shifts = ws_round(BH * dm->Lk * 4) + 2 * ws_round(BH * 4) + 2 * ws_round(BH * dm->Lq * 4) +
                        feat3::image_bytes(fs_groups(dm), dm->d, dm->M, 2);
  size_t b = ws_round(BH * dm->Lq * dm->M * 4) + ws_round(BH * dm->Lk * dm->M * 4) + shifts;
  if (!causal) {
    b += ws_round(BH * dm->M * NP * 4);
  } else {
    const size_t C = inner_chunk(chunk), nch = (dm->Lq + C - 1) / C;
    b += ws_round(BH * nch * dm->M * NP * 4) + ws_round(BH * nch * C * C * 4);
    // the chain on bf16 features: half the bytes for the features, running sums in bf16, no scores
    if (dm->d == 128 && dm->dv == 128 && dm->M % 128 == 0 && (chunk == 128 || chunk == 256)) {
      const size_t t = ws_round(BH * dm->Lq * dm->M * 2) + ws_round(BH * dm->Lk * dm->M * 2) + shifts +
                       ws_round(BH * fs_tc_kv128_slots(ctx, (int)BH, dm->M, (int)nch) * dm->M * 129 * 4) + ws_round(BH * nch * dm->M * 128 * 2) +
                       ws_round(BH * nch * dm->M * 2);
      if (t > b) b = t;
    }
  }
  return b;
}

int fs_simt_attend(fsharp_ctx* ctx, const void* Q, const void* K, const void* V, const fsharp_dims* dm,
                   int dtype, int causal, int chunk, float qk_scale, const float* prep, void* Y, WsAlloc* ws) {
  if (dtype == FSHARP_F32) return attend_t<float>(ctx, Q, K, V, dm, causal, chunk, qk_scale, prep, Y, ws, false);
  return attend_t<__nv_bfloat16>(ctx, Q, K, V, dm, causal, chunk, qk_scale, prep, Y, ws, false);
}

// The unnormalised operator Khat C (Section 2.1): the bidirectional pipeline with the shifts carried to the output.
int fs_simt_kernel_apply(fsharp_ctx* ctx, const void* X, const void* Yset, const void* Cmat, const fsharp_dims* dm,
                         int dtype, float qk_scale, const float* prep, void* out, WsAlloc* ws) {
  if (dtype == FSHARP_F32) return attend_t<float>(ctx, X, Yset, Cmat, dm, 0, 0, qk_scale, prep, out, ws, true);
  return attend_t<__nv_bfloat16>(ctx, X, Yset, Cmat, dm, 0, 0, qk_scale, prep, out, ws, true);
}
