// fp32 operands on the bf16 tensor cores without loss: x = h + m + l with h = bf16(x), m = bf16(x - h),
// l = bf16(x - h - m).  The two differences are exact in fp32 and the three parts carry 8 significant bits each, so
// h + m + l holds all 24 bits of x (while the parts stay above the smallest bf16, i.e. for |x| > 2^-109; features inside the library
// are lifted for it, feat3.cuh; infinities give NaN).  A product of
// two fp32 operands is the sum of the six part products hh + hm + mh + mm + hl + lh; what is left out (ml, lm, ll) is
// below 2^-24 of |x||y|, the rounding of one fp32 multiply-add.  Where one operand is a bf16 tensor its value is its h
// part and three products (hh, mh, lh) are exact.  Every part product is exact in the fp32 accumulator's adder tree.
#pragma once
#include "tc_common.cuh"

namespace split3 {

// (h, m, l) parts of a pair of values, packed (first value in the low half)
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = tc::pack_bf16(x0, x1);
  const float r0 = x0 - __uint_as_float(h << 16), r1 = x1 - __uint_as_float(h & 0xffff0000u);
  m = tc::pack_bf16(r0, r1);
  l = tc::pack_bf16(r0 - __uint_as_float(m << 16), r1 - __uint_as_float(m & 0xffff0000u));
}
// eight consecutive values -> three 16-byte pieces
__device__ __forceinline__ void split8(const float (&x)[8], uint4& h, uint4& m, uint4& l) {
  split_pair(x[0], x[1], h.x, m.x, l.x);
  split_pair(x[2], x[3], h.y, m.y, l.y);
  split_pair(x[4], x[5], h.z, m.z, l.z);
  split_pair(x[6], x[7], h.w, m.w, l.w);
}

}  // namespace split3
