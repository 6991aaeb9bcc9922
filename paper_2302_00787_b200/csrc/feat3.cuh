// Features at fp32 precision on the tensor cores (feat3.cu): one or two token sets per launch.
#pragma once
#include "common.cuh"

namespace feat3 {

// Features that stay inside the library (attention, its gradients, the kernel operator) carry a factor 2^LIFT against shifted ones:
// three bf16 parts hold all 24 bits of a value only above 2^-109 (split3.cuh), fp32 multiply-adds held them down to 2^-126,
// and a causal query may see nothing but keys that lie far below the sequence's largest.  It cancels wherever shifts do; what
// it costs is the top of the range: a product of both sides overflows 2^32 earlier.
constexpr int LIFT = 16;

struct Task {
  const void* X;          // tokens, strides ax (elements)
  TensorAddr ax;
  int L, side, stab;
  float* rowc;            // [B*H][L] scratch: the x^T C x terms
  unsigned* gmax;         // [B*H] scratch, FSHARP_STAB_GROUP
  float* phi;             // [B*H][L][M], or
  __nv_bfloat16* phi16;   // the same rounded to bf16 (bf16 tokens with d = 128 only; phi is then not written, and a group's shift
                          // is that of a maximum taken from the leading parts of W)
  float* logscale;        // as fsharp_featurize (the shift alone, whatever the lift); may be null where M fits one block of features
  int lift;               // 0 or LIFT: features times 2^lift (FSHARP_STAB_ROW and _GROUP)
};

// Scratch for the operand images of W (0: none are kept).
size_t image_bytes(int groups, int d, int M, int ntasks);

// Images of W (img, 16-byte aligned; nullptr: the blocks convert W themselves), quadratic terms, largest exponents where a
// shift needs them, then the features of all tasks.  Two tasks are of different sides.  zero (16-byte aligned, a multiple of four
// floats): cleared on the way, for sums that later kernels of the chain add up (a memset between them would end the chain of
// programmatic dependents).
int run(fsharp_ctx* ctx, const Task* tasks, int ntasks, int dtype, int B, int H, int d, int M, int pool, const float* prep,
        float qk_scale, uint8_t* img, float* zero = nullptr, size_t zero_floats = 0);

}  // namespace feat3
