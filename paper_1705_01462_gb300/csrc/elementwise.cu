// The non-contraction steps of a chained quantized ResNet forward (Section 4: activations
// stay 8-bit DFP codes between layers): max pooling of codes and the residual addition.
//
// Max pooling of unsigned codes is exact in the code domain (one shared scale, and the
// codes of post-ReLU activations are >= 0, so padding never wins).  The residual addition
// v = a * 2^Ea + b * 2^Eb is computed in fp32 (each product is exact; the sum is rounded
// once) and either stored as fp32 or requantized at a given scale 2^Eo with the rule of
// the activation quantizer (u8: negative sums become 0, the ReLU after the addition).
#include <cstdint>

#include "fgq_device.cuh"

namespace fgq {
namespace {

// One thread per V words (4 channels each) of one output pixel, per-byte maxima with vmaxu4; V = 4
// (16-byte loads) where C % 16 == 0 and both pointers are 16-byte aligned, else V = 1.  3x3/2 over
// 112 x 112 x 64 at batch 64: 45 us with V = 1, 21 with V = 4.
template <int V>
__global__ void __launch_bounds__(256) maxpool_u8_kernel(const uint8_t* __restrict__ in, int B, int H, int W, int C,
                                                         int R, int stride, int pad, int Ho, int Wo,
                                                         uint8_t* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int CV = C / (4 * V);
  if (i >= (int64_t)B * Ho * Wo * CV) return;
  const int cv = (int)(i % CV);
  int64_t r = i / CV;
  const int wo = (int)(r % Wo);
  r /= Wo;
  const int ho = (int)(r % Ho);
  const int b = (int)(r / Ho);
  uint32_t m[V] = {};
  for (int dr = 0; dr < R; ++dr) {
    const int h = ho * stride - pad + dr;
    if (h < 0 || h >= H) continue;
    for (int ds = 0; ds < R; ++ds) {
      const int w = wo * stride - pad + ds;
      if (w < 0 || w >= W) continue;
      const uint8_t* p = in + (((int64_t)b * H + h) * W + w) * C;
      if constexpr (V == 4) {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(p) + cv);
        m[0] = __vmaxu4(m[0], x.x);
        m[1] = __vmaxu4(m[1], x.y);
        m[2] = __vmaxu4(m[2], x.z);
        m[3] = __vmaxu4(m[3], x.w);
      } else {
        m[0] = __vmaxu4(m[0], __ldg(reinterpret_cast<const uint32_t*>(p) + cv));
      }
    }
  }
  if constexpr (V == 4) reinterpret_cast<uint4*>(out)[i] = make_uint4(m[0], m[1], m[2], m[3]);
  else reinterpret_cast<uint32_t*>(out)[i] = m[0];
}

__device__ __forceinline__ float add_value(uint8_t a, int a_signed, float sa, uint8_t b, int b_signed, float sb) {
  const float va = a_signed ? (float)(int8_t)a : (float)a, vb = b_signed ? (float)(int8_t)b : (float)b;
  return __fadd_rn(__fmul_rn(va, sa), __fmul_rn(vb, sb));
}

// The four codes of a word as floats: 2^23 + code assembled by byte permutes (signed codes biased to
// unsigned first), less the bias, exact and without integer conversions.
__device__ __forceinline__ void word_values(uint32_t w, uint32_t flip, float bias, float (&v)[4]) {
  w ^= flip;
  v[0] = __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7540)) - bias;
  v[1] = __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7541)) - bias;
  v[2] = __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7542)) - bias;
  v[3] = __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7543)) - bias;
}
// rq_code of four values in a word: the saturating packs clamp to the type's range.
__device__ __forceinline__ uint32_t rq_word(const float (&v)[4], const RqMul& r, int is_signed) {
  int x[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) x[e] = __float2int_rn(v[e] * r.m1 * r.m2);
  uint32_t hi, q;
  if (is_signed) {
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(x[3]), "r"(x[2]));
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(q) : "r"(x[1]), "r"(x[0]), "r"(hi));
  } else {
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(x[3]), "r"(x[2]));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(q) : "r"(x[1]), "r"(x[0]), "r"(hi));
  }
  return q;
}

// n16 pieces of 16 codes by 16-byte loads and stores (all pointers 16-byte aligned), the rest -- all
// codes, where a pointer is not aligned -- one by one.  Bound: the bytes (two codes read, one written).
// One code per thread and step, with integer conversions and clamps: 79 us for 51 M codes to codes (154 MB,
// 23 us) and 21 for 13 M; this form 32 and 10 (pieces without the word conversions: 57 and 17).
__global__ void __launch_bounds__(256) add_codes_kernel(const uint8_t* __restrict__ a, int a_signed,
                                                        const float* __restrict__ a_scale,
                                                        const uint8_t* __restrict__ b, int b_signed,
                                                        const float* __restrict__ b_scale, int64_t n, int64_t n16,
                                                        float* __restrict__ out, uint8_t* __restrict__ out_q,
                                                        const float* __restrict__ out_scale, int o_signed) {
  const float sa = __ldg(a_scale), sb = __ldg(b_scale);
  RqMul rq;
  if (out_q) rq = rq_mul(out_scale, o_signed);
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  const uint32_t fa = a_signed ? 0x80808080u : 0u, fb = b_signed ? 0x80808080u : 0u;
  const float ba = a_signed ? 8388736.0f : 8388608.0f, bb = b_signed ? 8388736.0f : 8388608.0f;  // 2^23 (+ 128)
  for (int64_t i = tid; i < n16; i += step) {
    const uint4 va = __ldg(reinterpret_cast<const uint4*>(a) + i), vb = __ldg(reinterpret_cast<const uint4*>(b) + i);
    const uint32_t wa[4] = {va.x, va.y, va.z, va.w}, wb[4] = {vb.x, vb.y, vb.z, vb.w};
    uint32_t q[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      float v[4], x[4], y[4];
      word_values(wa[w], fa, ba, x);
      word_values(wb[w], fb, bb, y);
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = __fadd_rn(__fmul_rn(x[e], sa), __fmul_rn(y[e], sb));
      if (out_q) q[w] = rq_word(v, rq, o_signed);
      else reinterpret_cast<float4*>(out)[4 * i + w] = make_float4(v[0], v[1], v[2], v[3]);
    }
    if (out_q) reinterpret_cast<uint4*>(out_q)[i] = make_uint4(q[0], q[1], q[2], q[3]);
  }
  for (int64_t i = 16 * n16 + tid; i < n; i += step) {
    const float v = add_value(__ldg(a + i), a_signed, sa, __ldg(b + i), b_signed, sb);
    if (out_q)
      out_q[i] = rq_code(v, rq);
    else
      out[i] = v;
  }
}

}  // namespace

fgq_status launch_maxpool_u8(const uint8_t* in, int B, int H, int W, int C, int R, int stride, int pad, uint8_t* out,
                             cudaStream_t s) {
  const int Ho = (H + 2 * pad - R) / stride + 1, Wo = (W + 2 * pad - R) / stride + 1;
  const bool wide = C % 16 == 0 && ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
  const int64_t n = (int64_t)B * Ho * Wo * (C / (wide ? 16 : 4));
  const unsigned blocks = (unsigned)((n + 255) / 256);
  if (wide)
    maxpool_u8_kernel<4><<<blocks, 256, 0, s>>>(in, B, H, W, C, R, stride, pad, Ho, Wo, out);
  else
    maxpool_u8_kernel<1><<<blocks, 256, 0, s>>>(in, B, H, W, C, R, stride, pad, Ho, Wo, out);
  return after_launch();
}

fgq_status launch_add_codes(const uint8_t* a, int a_signed, const float* a_scale, const uint8_t* b, int b_signed,
                            const float* b_scale, int64_t n, float* out, uint8_t* out_q, const float* out_scale,
                            int o_signed, cudaStream_t s) {
  const int sms = device_sms();
  const uintptr_t bits = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) |
                         reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(out_q);
  const int64_t n16 = (bits & 15) ? 0 : n / 16;
  const int64_t want = ((n16 ? n16 : n) + 255) / 256;
  const int blocks = (int)(want < 8 * sms ? (want > 0 ? want : 1) : 8 * sms);
  add_codes_kernel<<<blocks, 256, 0, s>>>(a, a_signed, a_scale, b, b_signed, b_scale, n, n16, out, out_q, out_scale,
                                          o_signed);
  return after_launch();
}

}  // namespace fgq
