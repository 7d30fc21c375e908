// Arithmetic of the streaming passes (per-tensor cast, penalty and gradient) on register vectors, shared by the kernels
// of their own and by the warps that do such work beside a grouped GEMM.  Not part of the public ABI.
#pragma once

#include "common.cuh"

namespace tweo_detail {

struct QTensor {
  const uint16_t* x;
  uint8_t* q;
  int64_t n;
  float* scale;
  float* scale_inv;
  float* amax;
  int32_t fmt;
  int32_t mode;
};

// 16 elements: two 16-byte loads -> one 16-byte store.  SAT counts elements whose scaled value
// exceeds the format's range, AMAX folds |x| into the running maximum m2.  NaN inputs come out of the
// converter as the code 0x7F (see cvt_fp8x2).
template <int FMT, bool SAT, bool AMAX>
__device__ __forceinline__ uint4 cast16(const uint4 a, const uint4 b, float scale, uint32_t& sat, float& m0, float& m1) {
  const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  uint32_t c[8];
  const float fmax = FMT == TWEO_E4M3 ? kE4M3Max : kE5M2Max;
  const uint64_t ss = pack_f32x2(scale, scale);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    float lo, hi;
    unpack_f32x2(mul_f32x2(bf16x2_to_f32x2(w[j]), ss), lo, hi);   // one packed multiply, each lane rounded once
    if (SAT) sat += (fabsf(lo) > fmax) + (fabsf(hi) > fmax);
    c[j] = cvt_fp8x2<FMT>(lo, hi);
    if (AMAX) absmax_f32(m0, m1, w[j]);
  }
  return make_uint4(c[0] | (c[1] << 16), c[2] | (c[3] << 16), c[4] | (c[5] << 16), c[6] | (c[7] << 16));
}

// One 16-byte vector (8 bf16) of the penalty at p = 4: packed binary32 pairs -- s = a*a is exact (8-bit significands), a^3 = s*a
// too (24 bits), so g = fl32(k * a^3) rounds once; the a^4 terms are folded into the running pair `acc2` by a
// fused multiply-add (acc2 += s*s), which the caller empties into its binary64 sum after at most 16 terms per lane.
template <bool GRAD>
__device__ __forceinline__ void penalty4_vec(const uint4 v, float k, uint64_t& acc2, uint64_t (&g2)[4]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  const uint64_t kk = pack_f32x2(k, k);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint64_t a2 = bf16x2_to_f32x2(w[j]);
    const uint64_t s2 = mul_f32x2(a2, a2);
    acc2 = fma_f32x2(s2, s2, acc2);
    if (GRAD) g2[j] = mul_f32x2(kk, mul_f32x2(s2, a2));
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
  return v;
}

}  // namespace tweo_detail
