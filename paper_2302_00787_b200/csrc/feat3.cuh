// Features at fp32 precision on the tensor cores (feat3.cu): one or two token sets per launch.
#pragma once
#include "common.cuh"

namespace feat3 {

struct Task {
  const void* X;          // tokens, strides ax (elements)
  TensorAddr ax;
  int L, side, stab;
  float* rowc;            // [B*H][L] scratch: the x^T C x terms
  unsigned* gmax;         // [B*H] scratch, FSHARP_STAB_GROUP
  float* phi;             // [B*H][L][M], or
  __nv_bfloat16* phi16;   // the same rounded to bf16 (bf16 tokens with d = 128 only; phi is then not written, and the shifts
                          // are those of a maximum taken from the leading parts of W)
  float* logscale;        // as fsharp_featurize; may be null (FSHARP_STAB_ROW: only when needs_logscale() says so)
};

// Features of a block: all of M when M <= this, so that a row's largest exponent is known inside the block.
inline bool needs_logscale(int d, int M, int stab) { return stab == FSHARP_STAB_ROW && M > (d == 128 ? 128 : 256); }

// Scratch for the operand images of W.
size_t image_bytes(int groups, int d, int M, int ntasks);

// Images of W (img, 16-byte aligned; nullptr: the blocks convert W themselves), quadratic terms, largest exponents where a
// shift needs them, then the features of all tasks.  Two tasks are of different sides.
int run(fsharp_ctx* ctx, const Task* tasks, int ntasks, int dtype, int B, int H, int d, int M, int pool, const float* prep,
        float qk_scale, uint8_t* img);

}  // namespace feat3
