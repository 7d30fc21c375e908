// Symmetric AbsMax b-bit quantisation (Eq. 4): s = max|X| + eps, X_q = round(X / s * Q_b),
// Q_b = 2^(b-1) - 1, with one s per tensor or per row (per output channel of a weight, per
// token of an activation), computed now or given (static).  Codes are int8 (b = 6 uses the
// same container).  Everything is binary32, each operation rounded once; Eq. 4's X / s * Q_b is
// evaluated as X * (Q_b / s), one division per scale and one multiplication per element:
//   s = fl32(amax + eps);  c = fl32(Q_b / s);  q = clamp(rne_int(fl32(x * c)), -Q_b, Q_b);  NaN -> 0.
// HBM-bound streaming kernels: 16-byte loads of 8 bf16, 16-byte stores of 16 codes.
//   per row   : one CTA per row.  Rows of up to 8192 aligned elements stay in registers between the maximum and
//               the cast (absmax_rows_reg_kernel); others are read twice, the second time from L1/L2.
//   per tensor: kernel 1 writes per-CTA maxima to workspace slots, kernel 2 reduces them in
//               every CTA and casts (no atomics, no reset kernel); static s skips kernel 1.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"

namespace {

using namespace tweo_detail;

constexpr int kThreads = 256;
constexpr int kMaxSlots = 2048;

__device__ __forceinline__ uint32_t cta_max_bits(uint32_t m, uint32_t* part) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) m = max(m, part[w]);
  return m;
}

// c = fl32(Q / s)
__device__ __forceinline__ int quant1(float x, float c, float Q) {
  const int r = __float2int_rn(__fmul_rn(x, c));  // ties to even; NaN -> 0; saturates
  const int q = (int)Q;
  return max(-q, min(q, r));
}

// 16 bf16 (two 16-byte vectors) -> 16 int8 codes
__device__ __forceinline__ uint4 quant16(const uint4 a, const uint4 b, float c, float Q) {
  const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  uint32_t pk[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int q0 = quant1(bf16lo_to_f32(w[2 * j]), c, Q), q1 = quant1(bf16hi_to_f32(w[2 * j]), c, Q);
    const int q2 = quant1(bf16lo_to_f32(w[2 * j + 1]), c, Q), q3 = quant1(bf16hi_to_f32(w[2 * j + 1]), c, Q);
    pk[j] = (uint32_t)(q0 & 0xFF) | ((uint32_t)(q1 & 0xFF) << 8) | ((uint32_t)(q2 & 0xFF) << 16) |
           ((uint32_t)(q3 & 0xFF) << 24);
  }
  return make_uint4(pk[0], pk[1], pk[2], pk[3]);
}

// maximum of |x| over [x, x+n) by this CTA's threads (packed lanes, see absmax_bits)
__device__ __forceinline__ uint32_t span_absmax(const uint16_t* x, int64_t n, int64_t first_vec, int64_t vec_stride) {
  uint32_t m2 = 0;
  const bool vec_ok = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
  const int64_t nvec = vec_ok ? (n >> 3) : 0;
  const uint4* xv = reinterpret_cast<const uint4*>(x);
  for (int64_t i = first_vec; i < nvec; i += vec_stride) {
    const uint4 v = __ldg(xv + i);
    m2 = absmax_bits(m2, v.x);
    m2 = absmax_bits(m2, v.y);
    m2 = absmax_bits(m2, v.z);
    m2 = absmax_bits(m2, v.w);
  }
  for (int64_t i = (nvec << 3) + first_vec; i < n; i += vec_stride) m2 = absmax_bits(m2, (uint32_t)x[i]);
  return m2;
}

__device__ __forceinline__ void span_quantize(const uint16_t* x, int8_t* q, int64_t n, float s, float Q,
                                              int64_t first, int64_t stride) {
  const float c = __fdiv_rn(Q, s);
  const bool vec_ok = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(q)) & 15u) == 0;
  const int64_t n16 = vec_ok ? (n >> 4) : 0;
  const uint4* xv = reinterpret_cast<const uint4*>(x);
  uint4* qv = reinterpret_cast<uint4*>(q);
  for (int64_t i = first; i < n16; i += 2 * stride) {  // two groups of 16 per iteration: four loads in flight
    const int64_t i1 = i + stride;
    const uint4 a0 = __ldcs(xv + 2 * i), b0 = __ldcs(xv + 2 * i + 1);
    uint4 a1 = a0, b1 = b0;
    if (i1 < n16) {
      a1 = __ldcs(xv + 2 * i1);
      b1 = __ldcs(xv + 2 * i1 + 1);
    }
    __stcs(qv + i, quant16(a0, b0, c, Q));
    if (i1 < n16) __stcs(qv + i1, quant16(a1, b1, c, Q));
  }
  for (int64_t i = (n16 << 4) + first; i < n; i += stride)
    q[i] = (int8_t)quant1(bf16lo_to_f32((uint32_t)x[i]), c, Q);
}

// one scale per row
template <bool GIVEN>
__global__ void __launch_bounds__(kThreads)
absmax_rows_kernel(const uint16_t* x, int64_t rows, int64_t cols, int64_t ldx, float eps, float Q, float* s_out,
                   int8_t* q, int64_t ldq) {
  __shared__ uint32_t part[kThreads / 32];
  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
    const uint16_t* xr = x + r * ldx;
    float s;
    if (GIVEN) {
      s = __ldg(s_out + r);
    } else {
      const uint32_t m = cta_max_bits(absmax_fold(span_absmax(xr, cols, threadIdx.x, kThreads)), part);
      s = __fadd_rn(__uint_as_float(m << 16), eps);
      if (threadIdx.x == 0) s_out[r] = s;
    }
    span_quantize(xr, q + r * ldq, cols, s, Q, threadIdx.x, kThreads);
  }
}

// The same with the row held in registers: VPT vectors of 8 elements per thread (thread-interleaved), the block sized
// to the row.  One read of x, and no conversion instruction: the unit that converts to integers does 16 a clock, 1.8 us
// for 8 M elements.  With a finite row maximum no |x c| exceeds Q_b by more than one rounding, so the nearest integer
// is read off the sum fl32(x c) + 1.5 2^23, whose low byte is the code (the addition rounds to nearest-even, as the
// conversion does); rows with a NaN, an infinity or an infinite c take the converting path.  Launched in a chain, like
// the residual addition below.  The per-token pass (quantise, integer linear, quantise, add) at 1999 tokens and
// [4096x4096] went from 66.9 to 57.1 us with both, at 8192 tokens and [3072x5120] from 193.1 to 168.4.
constexpr uint32_t kRoundMagicBits = 0x4B400000u;   // 1.5 * 2^23
constexpr int64_t kRegRowCols = 8192;

// Low bytes of four such sums -> one word of codes.
__device__ __forceinline__ uint32_t pack_low_bytes(float a, float b, float c, float d) {
  const uint32_t ab = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x0040);
  const uint32_t cd = __byte_perm(__float_as_uint(c), __float_as_uint(d), 0x0040);
  return __byte_perm(ab, cd, 0x5410);
}
// four values (two pairs) times c, rounded to the nearest integers -> four codes.  Scalar instructions: a packed product
// followed by a packed addition comes out of the assembler as one fused operation, which rounds differently at ties.
__device__ __forceinline__ uint32_t quant4_magic(uint64_t v01, uint64_t v23, float c) {
  const float magic = __uint_as_float(kRoundMagicBits);
  float v[4];
  unpack_f32x2(v01, v[0], v[1]);
  unpack_f32x2(v23, v[2], v[3]);
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __fadd_rn(__fmul_rn(v[i], c), magic);
  return pack_low_bytes(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ uint32_t quant4_slow(const uint32_t w0, const uint32_t w1, float c, float Q) {
  return (uint32_t)(quant1(bf16lo_to_f32(w0), c, Q) & 0xFF) | ((uint32_t)(quant1(bf16hi_to_f32(w0), c, Q) & 0xFF) << 8) |
         ((uint32_t)(quant1(bf16lo_to_f32(w1), c, Q) & 0xFF) << 16) | ((uint32_t)(quant1(bf16hi_to_f32(w1), c, Q) & 0xFF) << 24);
}
// the maximum of m over the CTA (any number of warps up to 8)
__device__ __forceinline__ uint32_t block_max_bits(uint32_t m, uint32_t* part) {
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
  __syncthreads();
  const int warps = blockDim.x >> 5;
  for (int w = 0; w < warps; ++w) m = max(m, part[w]);
  return m;
}

template <int VPT>
__global__ void __launch_bounds__(kThreads)
absmax_rows_reg_kernel(const uint16_t* x, int64_t rows, int64_t cols, int64_t ldx, float eps, float Q, float* s_out, int8_t* q, int64_t ldq) {
  __shared__ uint32_t part[kThreads / 32], part2[kThreads / 32];
  chain_wait();   // and no chain_release(): it costs each CTA about 1 ns (16384 rows of 768: 9.8 us without, 17.6 with it)
  const int nvec = (int)(cols >> 3);
  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {   // one turn, unless there are more rows than a grid has CTAs
  if (r != blockIdx.x) __syncthreads();                      // part[] may still be read from the turn before
  const uint4* xv = reinterpret_cast<const uint4*>(x + r * ldx);
  uint4 v[VPT];
  uint32_t m2 = 0;   // two lanes: the largest sign-stripped patterns, NaN patterns included
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int idx = threadIdx.x + i * blockDim.x;
    v[i] = idx < nvec ? __ldg(xv + idx) : make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    m2 = __vmaxu2(m2, v[i].x & 0x7FFF7FFFu);
    m2 = __vmaxu2(m2, v[i].y & 0x7FFF7FFFu);
    m2 = __vmaxu2(m2, v[i].z & 0x7FFF7FFFu);
    m2 = __vmaxu2(m2, v[i].w & 0x7FFF7FFFu);
  }
  uint32_t m = block_max_bits(absmax_fold(m2), part);
  const bool finite = m < 0x7F80u;   // uniform over the CTA, as all that follows from m
  if (!finite) {                     // NaN patterns do not count
    m2 = 0;
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      m2 = absmax_bits(m2, v[i].x);
      m2 = absmax_bits(m2, v[i].y);
      m2 = absmax_bits(m2, v[i].z);
      m2 = absmax_bits(m2, v[i].w);
    }
    m = block_max_bits(absmax_fold(m2), part2);
  }
  const float s = __fadd_rn(__uint_as_float(m << 16), eps);
  if (threadIdx.x == 0) s_out[r] = s;
  const float c = __fdiv_rn(Q, s);
  uint2* qv = reinterpret_cast<uint2*>(q + r * ldq);
  if (finite && c < __int_as_float(0x7F800000)) {
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      const int idx = threadIdx.x + i * blockDim.x;
      if (idx < nvec)
        qv[idx] = make_uint2(quant4_magic(bf16x2_to_f32x2(v[i].x), bf16x2_to_f32x2(v[i].y), c),
                             quant4_magic(bf16x2_to_f32x2(v[i].z), bf16x2_to_f32x2(v[i].w), c));
    }
  } else {
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      const int idx = threadIdx.x + i * blockDim.x;
      if (idx < nvec) qv[idx] = make_uint2(quant4_slow(v[i].x, v[i].y, c, Q), quant4_slow(v[i].z, v[i].w, c, Q));
    }
  }
  }
}

// Threads per CTA for a row of `nvec` vectors, `vpt` per thread: whole warps.
int row_threads(int64_t nvec, int vpt) { return (int)(((nvec + vpt - 1) / vpt + 31) / 32 * 32); }

cudaError_t launch_rows_reg(const uint16_t* x, int64_t rows, int64_t cols, int64_t ldx, float eps, float Q, float* s, int8_t* q,
                            int64_t ldq, cudaStream_t st) {
  const int64_t nvec = cols >> 3;
  const dim3 grid((unsigned)std::min<int64_t>(rows, INT32_MAX));
  if (nvec <= kThreads)
    return launch_chain(absmax_rows_reg_kernel<1>, grid, dim3(row_threads(nvec, 1)), 0, st, 0, x, rows, cols, ldx, eps, Q, s, q, ldq);
  if (nvec <= 2 * kThreads)
    return launch_chain(absmax_rows_reg_kernel<2>, grid, dim3(row_threads(nvec, 2)), 0, st, 0, x, rows, cols, ldx, eps, Q, s, q, ldq);
  return launch_chain(absmax_rows_reg_kernel<4>, grid, dim3(row_threads(nvec, 4)), 0, st, 0, x, rows, cols, ldx, eps, Q, s, q, ldq);
}

// one scale for the whole (contiguous) tensor: per-CTA maxima ...
__global__ void __launch_bounds__(kThreads) absmax_slots_kernel(const uint16_t* x, int64_t n, uint32_t* slots) {
  __shared__ uint32_t part[kThreads / 32];
  const uint32_t m = cta_max_bits(
      absmax_fold(span_absmax(x, n, (int64_t)blockIdx.x * kThreads + threadIdx.x, (int64_t)gridDim.x * kThreads)), part);
  if (threadIdx.x == 0) slots[blockIdx.x] = m;
}

// ... then every CTA reduces them itself and casts its share
template <bool GIVEN>
__global__ void __launch_bounds__(kThreads)
absmax_tensor_kernel(const uint16_t* x, int64_t n, float eps, float Q, float* s_io, const uint32_t* slots, int n_slots,
                     int8_t* q) {
  __shared__ uint32_t part[kThreads / 32];
  float s;
  if (GIVEN) {
    s = __ldg(s_io);
  } else {
    uint32_t m = 0;
    for (int k = threadIdx.x; k < n_slots; k += kThreads) m = max(m, __ldcg(slots + k));
    m = cta_max_bits(m, part);
    s = __fadd_rn(__uint_as_float(m << 16), eps);
    if (blockIdx.x == 0 && threadIdx.x == 0) *s_io = s;
  }
  span_quantize(x, q, n, s, Q, (int64_t)blockIdx.x * kThreads + threadIdx.x, (int64_t)gridDim.x * kThreads);
}

int grid_cap(int64_t want, int per_sm) {
  return balanced_grid(want, (int64_t)sm_count() * per_sm);
}

}  // namespace

namespace tweo_detail {
size_t absmax_workspace_bytes() { return (size_t)kMaxSlots * sizeof(uint32_t); }
}

extern "C" tweo_status_t tweo_absmax_quantize(const uint16_t* x, int64_t rows, int64_t cols, int64_t ldx, int32_t bits,
                                              int32_t granularity, int32_t mode, float eps, float* s, int8_t* q,
                                              int64_t ldq, void* ws, size_t ws_bytes, void* stream) {
  TWEO_LOG_CALL("tweo_absmax_quantize " "rows=%lld cols=%lld ldx=%lld bits=%d", (long long)rows,(long long)cols,(long long)ldx,bits);
  if (rows < 0 || cols < 0 || !s) return TWEO_ERR_INVALID_ARG;
  if (bits < 2 || bits > 8) return TWEO_ERR_INVALID_ARG;
  if (granularity != TWEO_GRAN_TENSOR && granularity != TWEO_GRAN_ROW) return TWEO_ERR_INVALID_ARG;
  if (mode != TWEO_SCALE_CURRENT && mode != TWEO_SCALE_GIVEN) return TWEO_ERR_INVALID_ARG;
  if (!(eps >= 0.0f)) return TWEO_ERR_INVALID_ARG;
  if (rows * cols > 0 && (!x || !q || ldx < cols || ldq < cols)) return TWEO_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const float Q = (float)((1 << (bits - 1)) - 1);
  const bool given = mode == TWEO_SCALE_GIVEN;
  if (granularity == TWEO_GRAN_ROW) {
    if (rows == 0) return TWEO_OK;
    if (!given && cols >= 8 && cols <= kRegRowCols && !(cols & 7) && !(ldx & 7) && !(ldq & 7) && aligned16(x) &&
        !(reinterpret_cast<uintptr_t>(q) & 7u)) {
      TWEO_CUDA_TRY(launch_rows_reg(x, rows, cols, ldx, eps, Q, s, q, ldq, st));
      count_launch();
      return check_launch("absmax_rows_reg_kernel");
    }
    const int grid = grid_cap(rows, 8);
    if (given) absmax_rows_kernel<true><<<grid, kThreads, 0, st>>>(x, rows, cols, ldx, eps, Q, s, q, ldq);
    else absmax_rows_kernel<false><<<grid, kThreads, 0, st>>>(x, rows, cols, ldx, eps, Q, s, q, ldq);
    count_launch();
    return check_launch("absmax_rows_kernel");
  }
  if (rows > 1 && (ldx != cols || ldq != cols)) return TWEO_ERR_UNSUPPORTED_SHAPE;  // one scale: dense tensor
  const int64_t n = rows * cols;
  uint32_t* slots = reinterpret_cast<uint32_t*>(ws);
  int n_slots = 0;
  if (!given) {
    if (!ws || ws_bytes < absmax_workspace_bytes()) return TWEO_ERR_WORKSPACE_TOO_SMALL;
    if (!aligned16(ws)) return TWEO_ERR_ALIGNMENT;
    n_slots = grid_cap(((n >> 3) + kThreads * 4 - 1) / (kThreads * 4), 8);
    if (n_slots > kMaxSlots) n_slots = kMaxSlots;
    absmax_slots_kernel<<<n_slots, kThreads, 0, st>>>(x, n, slots);
    count_launch();
  }
  const int grid = grid_cap(((n >> 4) + kThreads * 2 - 1) / (kThreads * 2), 8);
  if (given) absmax_tensor_kernel<true><<<grid, kThreads, 0, st>>>(x, n, eps, Q, s, slots, n_slots, q);
  else absmax_tensor_kernel<false><<<grid, kThreads, 0, st>>>(x, n, eps, Q, s, slots, n_slots, q);
  count_launch();
  return check_launch("absmax_tensor_kernel");
}

// ------------------------------------------------------------------ 8-bit residual stream (Sec. 4.4)
// yq = clamp(rne_int(xq * (sx / sy) + fq * (sf / sy))): Eq. 4 dequantise, add, Eq. 4 quantise with Q_b
// cancelled.  2 bytes read and 1 written per element, 16 codes per 16-byte vector, four vectors of each
// input in flight per thread; one product, one fused multiply-add and three conversions per element.
namespace {

__device__ __forceinline__ float code_to_f32(uint32_t w, int e) { return (float)(int)(int8_t)(w >> (8 * e)); }

__device__ __forceinline__ int add1_q8(float x, float f, float a, float b, int q) {
  const int r = __float2int_rn(__fmaf_rn(f, b, __fmul_rn(x, a)));  // ties to even; NaN -> 0; saturates
  return max(-q, min(q, r));
}

__device__ __forceinline__ uint32_t add4_q8(uint32_t xw, uint32_t fw, float a, float b, int q) {
  uint32_t out = 0u;
#pragma unroll
  for (int e = 0; e < 4; ++e) out |= ((uint32_t)add1_q8(code_to_f32(xw, e), code_to_f32(fw, e), a, b, q) & 0xFFu) << (8 * e);
  return out;
}

__global__ void __launch_bounds__(256) residual_add_q8_kernel(const int8_t* xq, const int8_t* fq,  // yq may alias either
                                                              int8_t* yq, int64_t n, float Q,
                                                              const float* __restrict__ sx, const float* __restrict__ sf,
                                                              const float* __restrict__ sy) {
  const float a = __fdiv_rn(__ldg(sx), __ldg(sy)), b = __fdiv_rn(__ldg(sf), __ldg(sy));
  const int q = (int)Q;
  const int64_t nvec = n >> 4;
  const uint4* xv = reinterpret_cast<const uint4*>(xq);
  const uint4* fv = reinterpret_cast<const uint4*>(fq);
  uint4* yv = reinterpret_cast<uint4*>(yq);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + 3 * stride < nvec; i += 4 * stride) {
    uint4 va[4], vb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      va[u] = __ldcs(xv + i + u * stride);
      vb[u] = __ldcs(fv + i + u * stride);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      __stcs(yv + i + u * stride, make_uint4(add4_q8(va[u].x, vb[u].x, a, b, q), add4_q8(va[u].y, vb[u].y, a, b, q),
                                             add4_q8(va[u].z, vb[u].z, a, b, q), add4_q8(va[u].w, vb[u].w, a, b, q)));
  }
  for (; i < nvec; i += stride) {
    const uint4 va = __ldcs(xv + i), vb = __ldcs(fv + i);
    __stcs(yv + i, make_uint4(add4_q8(va.x, vb.x, a, b, q), add4_q8(va.y, vb.y, a, b, q),
                              add4_q8(va.z, vb.z, a, b, q), add4_q8(va.w, vb.w, a, b, q)));
  }
  // ragged tail (n % 16 codes) by the first threads of the grid
  const int64_t t = (nvec << 4) + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) {
    yq[t] = (int8_t)add1_q8((float)xq[t], (float)fq[t], a, b, q);
  }
}

}  // namespace

extern "C" tweo_status_t tweo_residual_add_q8(const int8_t* xq, const float* sx, const int8_t* fq, const float* sf,
                                              int64_t n, int32_t bits, const float* sy, int8_t* yq, void* stream) {
  TWEO_LOG_CALL("tweo_residual_add_q8 " "n=%lld bits=%d", (long long)n,bits);
  if (n < 0 || bits < 2 || bits > 8 || !sx || !sf || !sy) return TWEO_ERR_INVALID_ARG;
  if (n == 0) return TWEO_OK;
  if (!xq || !fq || !yq) return TWEO_ERR_INVALID_ARG;
  if (!tweo_detail::aligned16(xq) || !tweo_detail::aligned16(fq) || !tweo_detail::aligned16(yq)) return TWEO_ERR_ALIGNMENT;
  const float Q = (float)((1 << (bits - 1)) - 1);
  const int64_t nvec = n >> 4;
  const int64_t want = (nvec + 4 * 256 - 1) / (4 * 256);
  const int grid = tweo_detail::balanced_grid(want, (int64_t)tweo_detail::sm_count() * 8);
  residual_add_q8_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(xq, fq, yq, n, Q, sx, sf, sy);
  tweo_detail::count_launch();
  return tweo_detail::check_launch("residual_add_q8_kernel");
}

// ------------------------------------------------------------------ per-token 8-bit residual stream (Sec. 4.4)
// One CTA per row, the block sized to the row, or one warp (the launcher says where): VPT 16-byte vectors of each input per
// thread, the dequantised sums formed
// once and held in registers, their maximum found by shuffles and one barrier, the codes of the sum written in the same
// pass: 2 bytes read and 1 written per element plus three scales per row.  Converting instructions (bytes to binary32 and
// back) go through a unit that does 16 a clock per SM, five of them per element bounded an earlier form of one warp per
// row (9.5 us at [1999x4096], and a row's work behind one warp: 4.4 us at 16 rows).  Instead a byte becomes binary32 by
// placing it in the mantissa of 2^23 and subtracting, and the code is the low byte of fl32(y c) + 1.5 2^23 (see
// absmax_rows_reg_kernel); rows whose scales are not far from overflow take the converting path.
namespace {

struct RowAddArgs {
  const int8_t* xq;
  const int8_t* fq;
  int8_t* yq;
  const float* sx;
  const float* sf;
  float* sy;
  int64_t rows;
  int32_t cols;
  float Q, eps;
};

// codes of word w (int8) -> two binary32 pairs, exact: 2^23 + (code + 128), minus 2^23 + 128
__device__ __forceinline__ void codes_to_f32x2(uint32_t w, uint64_t& p01, uint64_t& p23) {
  const uint32_t u = w ^ 0x80808080u;
  const uint64_t bias = splat_f32x2(-8388736.0f);
  p01 = add_f32x2(pack_f32x2(__uint_as_float(__byte_perm(u, 0x4B000000u, 0x7440)),
                             __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7441))), bias);
  p23 = add_f32x2(pack_f32x2(__uint_as_float(__byte_perm(u, 0x4B000000u, 0x7442)),
                             __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7443))), bias);
}

// WARP: a warp per row, eight rows per CTA (short rows); otherwise the CTA per row.
template <int VPT, bool WARP>
__global__ void __launch_bounds__(256) residual_add_q8_rows_kernel(const RowAddArgs a) {
  __shared__ float part[8];
  if (gridDim.x <= 148) chain_release();   // it costs each CTA about 1 ns ([16384x256] 9.9 -> 17.4 us): not with more CTAs than SMs
  chain_wait();
  const int nvec = a.cols >> 4;
  const int tid = WARP ? threadIdx.x & 31 : threadIdx.x, threads = WARP ? 32 : blockDim.x;
  const int64_t first = WARP ? (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5) : blockIdx.x;
  const int64_t step = WARP ? (int64_t)gridDim.x * 8 : gridDim.x;
  for (int64_t row = first; row < a.rows; row += step) {   // one turn, as in absmax_rows_reg_kernel
  if (!WARP && row != first) __syncthreads();
  const uint4* xv = reinterpret_cast<const uint4*>(a.xq + row * a.cols);
  const uint4* fv = reinterpret_cast<const uint4*>(a.fq + row * a.cols);
  uint4 vx[VPT], vf[VPT];
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int idx = tid + i * threads;
    vx[i] = idx < nvec ? __ldcs(xv + idx) : make_uint4(0u, 0u, 0u, 0u);
    vf[i] = idx < nvec ? __ldcs(fv + idx) : make_uint4(0u, 0u, 0u, 0u);
  }
  const float cx = __fdiv_rn(__ldg(a.sx + row), a.Q), cf = __fdiv_rn(__ldg(a.sf + row), a.Q);
  const uint64_t cx2 = splat_f32x2(cx), cf2 = splat_f32x2(cf);
  uint64_t y[VPT][8];
  float amax = 0.0f;  // padding lanes hold zero codes: their sum is 0 (or, like any NaN, does not count)
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const uint32_t wx[4] = {vx[i].x, vx[i].y, vx[i].z, vx[i].w};
    const uint32_t wf[4] = {vf[i].x, vf[i].y, vf[i].z, vf[i].w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      uint64_t x01, x23, f01, f23;
      codes_to_f32x2(wx[k], x01, x23);
      codes_to_f32x2(wf[k], f01, f23);
      y[i][2 * k] = fma_f32x2(f01, cf2, mul_f32x2(x01, cx2));
      y[i][2 * k + 1] = fma_f32x2(f23, cf2, mul_f32x2(x23, cx2));
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      float lo, hi;
      unpack_f32x2(y[i][k], lo, hi);
      amax = fmaxf(amax, fmaxf(fabsf(lo), fabsf(hi)));
    }
  }
  amax = warp_max(amax);
  if (!WARP) {
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = amax;
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) amax = fmaxf(amax, part[w]);
  }
  const float s = __fadd_rn(amax, a.eps);
  const float c = __fdiv_rn(a.Q, s);
  if (tid == 0) a.sy[row] = s;
  // no sum of the row can have been infinite or NaN, and Q / s is finite: |y c| stays within one rounding of Q
  const bool plain = (fabsf(cx) + fabsf(cf)) * 256.0f < 3.0e38f && c < __int_as_float(0x7F800000);
  uint4* yv = reinterpret_cast<uint4*>(a.yq + row * a.cols);
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int idx = tid + i * threads;
    uint32_t o4[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (plain) {
        o4[k] = quant4_magic(y[i][2 * k], y[i][2 * k + 1], c);
      } else {
        float v[4];
        unpack_f32x2(y[i][2 * k], v[0], v[1]);
        unpack_f32x2(y[i][2 * k + 1], v[2], v[3]);
        o4[k] = 0u;
#pragma unroll
        for (int e = 0; e < 4; ++e) o4[k] |= ((uint32_t)quant1(v[e], c, a.Q) & 0xFFu) << (8 * e);
      }
    }
    if (idx < nvec) __stcs(yv + idx, make_uint4(o4[0], o4[1], o4[2], o4[3]));
  }
  }
}

}  // namespace

extern "C" tweo_status_t tweo_residual_add_q8_rows(const int8_t* xq, const float* sx, const int8_t* fq, const float* sf,
                                                   int64_t rows, int64_t cols, int32_t bits, float eps, int8_t* yq,
                                                   float* sy, void* stream) {
  TWEO_LOG_CALL("tweo_residual_add_q8_rows " "rows=%lld cols=%lld bits=%d eps=%g", (long long)rows,(long long)cols,bits,(double)eps);
  if (rows < 0 || cols < 1 || bits < 2 || bits > 8 || !(eps >= 0.0f)) return TWEO_ERR_INVALID_ARG;
  if ((cols & 15) || cols > 8192) return TWEO_ERR_UNSUPPORTED_SHAPE;
  if (rows == 0) return TWEO_OK;
  if (!xq || !fq || !yq || !sx || !sf || !sy) return TWEO_ERR_INVALID_ARG;
  if (!tweo_detail::aligned16(xq) || !tweo_detail::aligned16(fq) || !tweo_detail::aligned16(yq)) return TWEO_ERR_ALIGNMENT;
  RowAddArgs a;
  a.xq = xq;
  a.fq = fq;
  a.yq = yq;
  a.sx = sx;
  a.sf = sf;
  a.sy = sy;
  a.rows = rows;
  a.cols = (int32_t)cols;
  a.Q = (float)((1 << (bits - 1)) - 1);
  a.eps = eps;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t nvec = cols >> 4;
  const dim3 grid((unsigned)std::min<int64_t>(rows, INT32_MAX)), grid8((unsigned)std::min<int64_t>((rows + 7) / 8, INT32_MAX));
  cudaError_t e;
  // A warp per row where a row gives it one vector per lane, or two and there are rows for every SM's warps: with a CTA per
  // row the start of the CTAs bounds many short rows.  Microseconds, CTA per row / warp per row: [16x512] 1.6 / 1.5,
  // [16384x256] 9.9 / 6.0, [131072x64] 68.8 / 38.5, [131072x512] 69.2 / 45.3; two vectors [16x1024] 1.6 / 1.8,
  // [512x768] 1.8 / 2.0, [2048x768] 2.7 / 2.4, [16384x1024] 11.3 / 9.6; four [16384x2048] 21.4 / 21.5.
  if (nvec <= 32)
    e = tweo_detail::launch_chain(residual_add_q8_rows_kernel<1, true>, grid8, dim3(256), 0, st, 0, a);
  else if (nvec <= 64 && rows >= 2048)
    e = tweo_detail::launch_chain(residual_add_q8_rows_kernel<2, true>, grid8, dim3(256), 0, st, 0, a);
  else if (nvec <= 256)
    e = tweo_detail::launch_chain(residual_add_q8_rows_kernel<1, false>, grid, dim3(row_threads(nvec, 1)), 0, st, 0, a);
  else
    e = tweo_detail::launch_chain(residual_add_q8_rows_kernel<2, false>, grid, dim3(row_threads(nvec, 2)), 0, st, 0, a);
  if (e != cudaSuccess) return tweo_detail::cuda_fail(e, "residual_add_q8_rows_kernel");
  tweo_detail::count_launch();
  return TWEO_OK;
}
