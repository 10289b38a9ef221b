// Dynamic-fixed-point activation quantization (Section 4: activations are quantized to 8
// or 4 bits before each convolution, with one shared exponent per tensor).
//
//   E   = smallest integer with max * 2^-E <= qmax (max = max|x|, or max(x, 0) for the
//         unsigned types), 0 when max = 0, clamped to [-149, 127];
//   q_i = clamp(round_half_even(x_i * 2^-E), qmin, qmax),   scale = 2^E.
//
// x * 2^-E is exact in fp32 whenever the result is at least 2^-126 (a power-of-two
// scaling), and a product below that rounds to the integer 0 whichever way it is rounded,
// so the codes are exact.  When 2^-E exceeds the fp32 range the scaling is applied as two
// exact factors.
//
// Pass 1 (derived scale only): per-block maxima of the magnitude bit patterns (non-negative
// floats order like their bits) into the caller's workspace.  Pass 2: every block reduces
// the block maxima, derives E, and quantizes a grid-stride share of 16-element chunks.
#include <climits>
#include <cstdint>
#include <cstring>
#include <mutex>

#include "fgq_device.cuh"

namespace fgq {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ uint32_t mag_bits(float x, bool is_unsigned) {
  const uint32_t b = __float_as_uint(x);
  if (is_unsigned) return (b >> 31) ? 0u : b;  // negative (and -0) count as 0
  return b & 0x7fffffffu;
}

// float4 loads with an L2 eviction-priority hint: pass 1 marks the input evict-last so that
// as much of it as fits is still in L2 when pass 2 reads it (evict-first: not needed again).
__device__ __forceinline__ float4 ld_f4_policy(const float4* p, uint64_t pol) {
  float4 v;
  asm volatile("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

__global__ void __launch_bounds__(kThreads) qa_max_kernel(const float* __restrict__ x, size_t n, int is_unsigned,
                                                          uint32_t* __restrict__ partials, unsigned int* err) {
  uint32_t mx = 0;
  bool bad = false;
  const size_t n4 = n / 4;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t nth = (size_t)gridDim.x * blockDim.x;
  const uint64_t keep = policy_evict_last();
  for (size_t i = tid; i < n4; i += nth) {
    const float4 f = ld_f4_policy(x4 + i, keep);
    const float e[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      bad |= (__float_as_uint(e[j]) & 0x7fffffffu) >= 0x7f800000u;
      mx = max(mx, mag_bits(e[j], is_unsigned));
    }
  }
  for (size_t i = n4 * 4 + tid; i < n; i += nth) {
    const float e = __ldg(x + i);
    bad |= (__float_as_uint(e) & 0x7fffffffu) >= 0x7f800000u;
    mx = max(mx, mag_bits(e, is_unsigned));
  }
  __shared__ uint32_t red[kThreads / 32];
  mx = __reduce_max_sync(FULL_MASK, mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  if (__syncthreads_or(bad) && threadIdx.x == 0) record_error(err, FGQ_ERR_NONFINITE);
  if (threadIdx.x == 0) {
    uint32_t m = 0;
    for (int i = 0; i < kThreads / 32; ++i) m = max(m, red[i]);
    partials[blockIdx.x] = m;
  }
}

__device__ __forceinline__ int dfp_exponent(uint32_t mbits, int qmax) {
  if (mbits == 0 || mbits >= 0x7f800000u) return 0;
  // mbits = 1.f 2^e against qmax = 1.q 2^k: E = e - k, one more where 1.f exceeds 1.q (in fp64 every
  // fp32 magnitude is normal)
  const uint64_t b = (uint64_t)__double_as_longlong((double)__uint_as_float(mbits));
  const uint64_t frac = ((uint64_t)1 << 52) - 1;
  const int k = 31 - __clz(qmax);
  const int E = (int)(b >> 52) - 1023 - k + ((b & frac) > (((uint64_t)qmax << (52 - k)) & frac) ? 1 : 0);
  return max(-149, min(127, E));
}

template <int TYPE>
struct QTraits;
template <> struct QTraits<FGQ_U8> { static constexpr int qmin = 0, qmax = 255, bits = 8; };
template <> struct QTraits<FGQ_S8> { static constexpr int qmin = -128, qmax = 127, bits = 8; };
template <> struct QTraits<FGQ_U4> { static constexpr int qmin = 0, qmax = 15, bits = 4; };
template <> struct QTraits<FGQ_S4> { static constexpr int qmin = -8, qmax = 7, bits = 4; };

// Four codes of an 8-bit type in a word: conversions, then saturating packs (the int32 conversion
// saturates and takes NaN to 0, as in qcode).  ONE: mul2 is 1.
template <int TYPE, bool ONE>
__device__ __forceinline__ uint32_t qword(const float4& f, float mul1, float mul2) {
  static_assert(QTraits<TYPE>::bits == 8, "8-bit codes");
  const int a = __float2int_rn(ONE ? f.x * mul1 : f.x * mul1 * mul2);
  const int b = __float2int_rn(ONE ? f.y * mul1 : f.y * mul1 * mul2);
  const int c = __float2int_rn(ONE ? f.z * mul1 : f.z * mul1 * mul2);
  const int d = __float2int_rn(ONE ? f.w * mul1 : f.w * mul1 * mul2);
  uint32_t hi, r;
  if (TYPE == FGQ_U8) {
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(d), "r"(c));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(b), "r"(a), "r"(hi));
  } else {
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(d), "r"(c));
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(b), "r"(a), "r"(hi));
  }
  return r;
}

template <int TYPE>
__device__ __forceinline__ uint32_t qcode(float x, float mul1, float mul2) {
  using T = QTraits<TYPE>;
  int r = __float2int_rn(x * mul1 * mul2);
  r = max(T::qmin, min(T::qmax, r));
  return (uint32_t)r & ((1u << T::bits) - 1u);
}

template <int TYPE>
__global__ void __launch_bounds__(kThreads) qa_quant_kernel(const float* __restrict__ x, size_t n,
                                                            const uint32_t* __restrict__ partials, int nparts,
                                                            int E_given, uint8_t* __restrict__ q,
                                                            float* __restrict__ scale_out) {
  using T = QTraits<TYPE>;
  __shared__ int sE;
  __shared__ uint32_t red[kThreads / 32];
  int E = E_given;
  if (partials != nullptr) {
    uint32_t mx = 0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) mx = max(mx, partials[i]);
    mx = __reduce_max_sync(FULL_MASK, mx);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t m = 0;
      for (int i = 0; i < kThreads / 32; ++i) m = max(m, red[i]);
      sE = dfp_exponent(m, T::qmax);
    }
    __syncthreads();
    E = sE;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && scale_out != nullptr) *scale_out = pow2f(E);
  const float mul1 = (-E <= 127) ? pow2f(-E) : pow2f(64);
  const float mul2 = (-E <= 127) ? 1.0f : pow2f(-E - 64);

  const size_t n16 = n / 16;
  const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t nth = (size_t)gridDim.x * blockDim.x;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  const uint64_t drop = policy_evict_first();
  // chunks in reverse of pass 1's order: the part of x pass 1 read last is the part most
  // likely still in L2
  for (size_t c0 = tid; c0 < n16; c0 += nth) {
    const size_t c = n16 - 1 - c0;
    float e[16];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 f = ld_f4_policy(x4 + 4 * c + j, drop);
      e[4 * j] = f.x; e[4 * j + 1] = f.y; e[4 * j + 2] = f.z; e[4 * j + 3] = f.w;
    }
    if (T::bits == 8) {
      uint4 o;
      uint32_t wv[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        wv[j] = qcode<TYPE>(e[4 * j], mul1, mul2) | (qcode<TYPE>(e[4 * j + 1], mul1, mul2) << 8) |
                (qcode<TYPE>(e[4 * j + 2], mul1, mul2) << 16) | (qcode<TYPE>(e[4 * j + 3], mul1, mul2) << 24);
      }
      o.x = wv[0]; o.y = wv[1]; o.z = wv[2]; o.w = wv[3];
      reinterpret_cast<uint4*>(q)[c] = o;
    } else {
      uint32_t wv[2] = {0u, 0u};
#pragma unroll
      for (int j = 0; j < 16; ++j) wv[j / 8] |= qcode<TYPE>(e[j], mul1, mul2) << (4 * (j % 8));
      reinterpret_cast<uint2*>(q)[c] = make_uint2(wv[0], wv[1]);
    }
  }
  if (tid == 0) {  // ragged tail of fewer than 16 elements
    for (size_t i = n16 * 16; i < n; ++i) {
      const uint32_t code = qcode<TYPE>(x[i], mul1, mul2);
      if (T::bits == 8) {
        q[i] = (uint8_t)code;
      } else if ((i & 1) == 0) {
        q[i / 2] = (uint8_t)code;  // the high nibble of an odd tail stays 0
      } else {
        q[i / 2] = (uint8_t)(q[i / 2] | (code << 4));
      }
    }
  }
}

int max_blocks(size_t n) {
  const size_t need = (n / 16 + kThreads - 1) / kThreads;
  const size_t cap = (size_t)device_sms() * 8;
  return (int)(need < 1 ? 1 : (need < cap ? need : cap));
}

}  // namespace

namespace {

// Fixed-point alphas (Section 4): one warp per filter row; the row's DFP exponent from its
// maximum (the activation quantizer's rule, unsigned 8- or 4-bit), then the codes (4-bit:
// two per byte, element 2i in the low nibble) and the row scale 2^E.  A row holding
// NaN/Inf gets zero codes and scale 0 and records FGQ_ERR_NONFINITE.
template <int TYPE>
__global__ void __launch_bounds__(256) quantize_alpha_kernel(const float* __restrict__ alpha, int M, int ng,
                                                            uint8_t* __restrict__ aq, float* __restrict__ ascale,
                                                            unsigned int* err) {
  using T = QTraits<TYPE>;
  const int m = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (m >= M) return;
  const float* row = alpha + (int64_t)m * ng;
  uint32_t mx = 0;
  bool bad = false;
  for (int g = lane; g < ng; g += 32) {
    const float v = __ldg(row + g);
    bad |= (__float_as_uint(v) & 0x7fffffffu) >= 0x7f800000u;
    mx = max(mx, mag_bits(v, true));
  }
  mx = __reduce_max_sync(FULL_MASK, mx);
  bad = __any_sync(FULL_MASK, bad);
  const int rb = T::bits == 8 ? ng : (ng + 1) / 2;  // code bytes per row
  uint8_t* out = aq + (int64_t)m * rb;
  if (bad) {
    if (lane == 0) {
      record_error(err, FGQ_ERR_NONFINITE);
      ascale[m] = 0.0f;
    }
    for (int i = lane; i < rb; i += 32) out[i] = 0;
    return;
  }
  const int E = dfp_exponent(mx, T::qmax);
  const float mul1 = (-E <= 127) ? pow2f(-E) : pow2f(64);
  const float mul2 = (-E <= 127) ? 1.0f : pow2f(-E - 64);
  if (lane == 0) ascale[m] = pow2f(E);
  for (int i = lane; i < rb; i += 32) {
    if (T::bits == 8) {
      out[i] = (uint8_t)qcode<TYPE>(__ldg(row + i), mul1, mul2);
    } else {
      const uint32_t lo = qcode<TYPE>(__ldg(row + 2 * i), mul1, mul2);
      const uint32_t hi = 2 * i + 1 < ng ? qcode<TYPE>(__ldg(row + 2 * i + 1), mul1, mul2) : 0u;
      out[i] = (uint8_t)(lo | (hi << 4));
    }
  }
}

// alpha' = a * scale per row (exact in fp32), for the paths that take fp32 alphas.
__global__ void __launch_bounds__(256) dequantize_alpha_kernel(const uint8_t* __restrict__ aq, int bits, int M, int ng,
                                                              const float* __restrict__ ascale,
                                                              float* __restrict__ alpha) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)M * ng) return;
  const int m = (int)(i / ng), g = (int)(i - (int64_t)m * ng);
  uint32_t a;
  if (bits == 8) {
    a = __ldg(aq + i);
  } else {
    const uint8_t b = __ldg(aq + (int64_t)m * ((ng + 1) / 2) + g / 2);
    a = (g & 1) ? (b >> 4) : (b & 0xfu);
  }
  alpha[i] = (float)a * __ldg(ascale + m);
}

}  // namespace

fgq_status launch_quantize_alpha(const float* alpha, int M, int ng, int bits, uint8_t* aq, float* ascale,
                                 unsigned int* err, cudaStream_t s) {
  const unsigned blocks = (unsigned)((M + 7) / 8);
  if (bits == 8)
    quantize_alpha_kernel<FGQ_U8><<<blocks, 256, 0, s>>>(alpha, M, ng, aq, ascale, err);
  else
    quantize_alpha_kernel<FGQ_U4><<<blocks, 256, 0, s>>>(alpha, M, ng, aq, ascale, err);
  return after_launch();
}

fgq_status launch_dequantize_alpha(const uint8_t* aq, int bits, int M, int ng, const float* ascale, float* alpha,
                                   cudaStream_t s) {
  const int64_t n = (int64_t)M * ng;
  dequantize_alpha_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(aq, bits, M, ng, ascale, alpha);
  return after_launch();
}

size_t quantize_workspace_bytes(size_t n) {
  if (n == 0) return 0;
  return sizeof(uint32_t) * (size_t)max_blocks(n);
}

fgq_status launch_quantize(const float* x, size_t n, int type, int E_given, bool derive, void* q,
                           float* scale_out, uint32_t* partials, unsigned int* err, cudaStream_t s) {
  const int blocks = max_blocks(n);
  if (derive) {
    qa_max_kernel<<<blocks, kThreads, 0, s>>>(x, n, (type == FGQ_U8 || type == FGQ_U4) ? 1 : 0, partials, err);
    fgq_status st = after_launch();
    if (st != FGQ_OK) return st;
  } else {
    partials = nullptr;
  }
  uint8_t* qb = static_cast<uint8_t*>(q);
  switch (type) {
    case FGQ_U8: qa_quant_kernel<FGQ_U8><<<blocks, kThreads, 0, s>>>(x, n, partials, blocks, E_given, qb, scale_out); break;
    case FGQ_S8: qa_quant_kernel<FGQ_S8><<<blocks, kThreads, 0, s>>>(x, n, partials, blocks, E_given, qb, scale_out); break;
    case FGQ_U4: qa_quant_kernel<FGQ_U4><<<blocks, kThreads, 0, s>>>(x, n, partials, blocks, E_given, qb, scale_out); break;
    case FGQ_S4: qa_quant_kernel<FGQ_S4><<<blocks, kThreads, 0, s>>>(x, n, partials, blocks, E_given, qb, scale_out); break;
    default: return FGQ_ERR_ARG;
  }
  return after_launch();
}

}  // namespace fgq

// ----------------------------------------------------------------------------------------
// fgq_quantize_act_batch: the same quantization for many tensors (the inputs of a network's
// layers) in one cooperative launch.  The tensors are cut into items of kBatchElems consecutive
// elements, and taken in order in chunks of about kBatchChunkBytes of fp32 input.  The items of all
// passes form one list -- pass 1 (the maximum) of chunk k, then pass 2 (the codes) of chunk k - 1 --
// that the resident blocks work off in order, block b taking items b, b + grid, ...: pass 2 reads
// from the L2 what pass 1 brought there shortly before, beside the HBM reads of the next chunk.
//
// A tensor's word holds its largest exponent so far, in an order-preserving code (the exponent of the
// maximum is the maximum of the items' exponents), above the count of its items that pass 1 has
// finished.  A pass 2 item waits until that count is complete; the items that it waits for precede it
// in the list and wait for nothing, and all blocks are resident, so every wait ends (and is bounded
// in time all the same: FGQ_ERR_TIMEOUT).
//
// Bound: one read of the inputs and one write of the codes (31 tensors, 162 M elements: 810 MB, 120
// us).  That batch took 250 us as one launch per 48 MB chunk (15 launches of 17 us) and takes 199 a
// call: 24 to 40 MB chunks, 64 or 128 KB items and 5 to 8 blocks per SM all give 195 to 200 (what is
// left is the host's part of a call), items of 32 KB 226 (an item's maximum is then one batch of
// loads, and a reduction and an atomic with nothing in flight).
namespace fgq {
namespace {

constexpr int kBatchThreads = 256;
constexpr int kBatchBlocks = 5;                        // resident blocks per SM
constexpr int kBatchElems = 16384;                     // elements per item (64 KB of fp32)
constexpr size_t kBatchChunkBytes = (size_t)24 << 20;  // two chunks and their codes stay in the L2
constexpr int kBatchCountBits = 23;                    // of a tensor's word; its exponent code above
constexpr uint32_t kBatchBadCode = 511;                // a NaN or infinity: exponent 0, and above all others
constexpr uint64_t kBatchTimeoutNs = 2000000000ull;

struct QTensor {
  const float* x;
  uint8_t* q;
  float* scale;
  unsigned int* word;
  int64_t n;
  int type;
  int items;
};

// Items first, first + 1, ... (up to the next segment's first): pass 1 or 2 of one tensor.
struct QSegment {
  int first;
  int16_t tensor;
  int16_t pass;
};

template <int MAXT>
struct QBatch {
  QTensor t[MAXT];
  QSegment seg[2 * MAXT];
  int nseg;
  int items;
  uint64_t timeout_ns;
};

__device__ __forceinline__ uint32_t exponent_code(uint32_t mbits, int qmax) {
  return mbits == 0 ? 0u : (mbits >= 0x7f800000u ? kBatchBadCode : (uint32_t)(dfp_exponent(mbits, qmax) + 150));
}
__device__ __forceinline__ int code_exponent(uint32_t code) {
  return code == 0 || code == kBatchBadCode ? 0 : (int)code - 150;
}
__device__ __forceinline__ uint32_t load_acquire(const unsigned int* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void qab_max_item(const QTensor& T, int item, uint32_t* red, unsigned int* err) {
  const int64_t e0 = (int64_t)item * kBatchElems;
  const int64_t e1 = e0 + kBatchElems < T.n ? e0 + kBatchElems : T.n;
  const bool is_unsigned = T.type == FGQ_U8 || T.type == FGQ_U4;
  // mag: the largest magnitude pattern (NaN and infinities above all finite ones); pos: the largest
  // pattern as a signed integer, so that negative floats count as 0 for the unsigned types
  uint32_t mag = 0;
  int pos = 0;
  auto take = [&](float e) {
    mag = max(mag, __float_as_uint(e) & 0x7fffffffu);
    pos = max(pos, __float_as_int(e));
  };
  const float4* x4 = reinterpret_cast<const float4*>(T.x + e0);  // e0 is a multiple of 4: aligned
  const int n4 = (int)((e1 - e0) / 4);
  const uint64_t keep = policy_evict_last();
  constexpr int U = 8;  // independent 16-byte loads in flight per thread
  int i = threadIdx.x;
  for (; i + (U - 1) * kBatchThreads < n4; i += U * kBatchThreads) {
    float4 f[U];
#pragma unroll
    for (int u = 0; u < U; ++u) f[u] = ld_f4_policy(x4 + i + u * kBatchThreads, keep);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      take(f[u].x);
      take(f[u].y);
      take(f[u].z);
      take(f[u].w);
    }
  }
  for (; i < n4; i += kBatchThreads) {
    const float4 f = ld_f4_policy(x4 + i, keep);
    take(f.x);
    take(f.y);
    take(f.z);
    take(f.w);
  }
  for (int64_t j = e0 + (int64_t)n4 * 4 + threadIdx.x; j < e1; j += kBatchThreads) take(__ldg(T.x + j));
  uint32_t mx = is_unsigned ? (uint32_t)pos : mag;
  const bool bad = mag >= 0x7f800000u;
  mx = __reduce_max_sync(FULL_MASK, mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  if (__syncthreads_or(bad) && threadIdx.x == 0) record_error(err, FGQ_ERR_NONFINITE);
  if (threadIdx.x == 0) {
    uint32_t m = 0;
    for (int i = 0; i < kBatchThreads / 32; ++i) m = max(m, red[i]);
    const int qmax = T.type == FGQ_U8 ? 255 : (T.type == FGQ_S8 ? 127 : (T.type == FGQ_U4 ? 15 : 7));
    const uint32_t code = exponent_code(m, qmax);
    uint32_t w = *reinterpret_cast<volatile unsigned int*>(T.word);
    while (code > w >> kBatchCountBits) {  // raise the exponent and count in one step
      const uint32_t old = atomicCAS(T.word, w, (code << kBatchCountBits) | ((w & ((1u << kBatchCountBits) - 1u)) + 1u));
      if (old == w) return;
      w = old;
    }
    atomicAdd(T.word, 1u);  // (a word's exponent never falls)
  }
}

// Four consecutive codes per thread and step: a warp loads 512 consecutive bytes and stores 128 (or 64).
template <int TYPE, bool ONE>
__device__ __forceinline__ void qab_quant_quads(const float4* x4, uint8_t* q, int n4, float mul1, float mul2) {
  using Tr = QTraits<TYPE>;
  const uint64_t drop = policy_evict_first();
  auto put = [&](int i, const float4& f) {
    if constexpr (Tr::bits == 8)
      reinterpret_cast<uint32_t*>(q)[i] = qword<TYPE, ONE>(f, mul1, mul2);
    else
      reinterpret_cast<uint16_t*>(q)[i] =
          (uint16_t)(qcode<TYPE>(f.x, mul1, mul2) | (qcode<TYPE>(f.y, mul1, mul2) << 4) |
                     (qcode<TYPE>(f.z, mul1, mul2) << 8) | (qcode<TYPE>(f.w, mul1, mul2) << 12));
  };
  constexpr int U = 8;
  int i = threadIdx.x;
  for (; i + (U - 1) * kBatchThreads < n4; i += U * kBatchThreads) {
    float4 f[U];
#pragma unroll
    for (int u = 0; u < U; ++u) f[u] = ld_f4_policy(x4 + i + u * kBatchThreads, drop);
#pragma unroll
    for (int u = 0; u < U; ++u) put(i + u * kBatchThreads, f[u]);
  }
  for (; i < n4; i += kBatchThreads) put(i, ld_f4_policy(x4 + i, drop));
}

template <int TYPE>
__device__ __forceinline__ void qab_quant_range(const QTensor& T, int64_t e0, int64_t e1, bool write_scale, int E) {
  using Tr = QTraits<TYPE>;
  if (write_scale && threadIdx.x == 0) *T.scale = pow2f(E);
  const float mul1 = (-E <= 127) ? pow2f(-E) : pow2f(64);
  const float mul2 = (-E <= 127) ? 1.0f : pow2f(-E - 64);
  const int n4 = (int)((e1 - e0) / 4);
  const float4* x4 = reinterpret_cast<const float4*>(T.x + e0);
  uint8_t* q = T.q + (Tr::bits == 8 ? e0 : e0 / 2);
  if (-E <= 127) qab_quant_quads<TYPE, true>(x4, q, n4, mul1, mul2);
  else qab_quant_quads<TYPE, false>(x4, q, n4, mul1, mul2);
  if (threadIdx.x == 0) {  // the tensor's ragged tail (last block only): fewer than 4 elements
    for (int64_t i = e0 + (int64_t)n4 * 4; i < e1; ++i) {
      const uint32_t code = qcode<TYPE>(T.x[i], mul1, mul2);
      if (Tr::bits == 8) {
        T.q[i] = (uint8_t)code;
      } else if ((i & 1) == 0) {
        T.q[i / 2] = (uint8_t)code;  // the high nibble of an odd tail stays 0
      } else {
        T.q[i / 2] = (uint8_t)(T.q[i / 2] | (code << 4));
      }
    }
  }
}

__device__ __forceinline__ void qab_quant_item(const QTensor& T, int item, int E) {
  const int64_t e0 = (int64_t)item * kBatchElems;
  const int64_t e1 = e0 + kBatchElems < T.n ? e0 + kBatchElems : T.n;
  switch (T.type) {
    case FGQ_U8: qab_quant_range<FGQ_U8>(T, e0, e1, item == 0, E); break;
    case FGQ_S8: qab_quant_range<FGQ_S8>(T, e0, e1, item == 0, E); break;
    case FGQ_U4: qab_quant_range<FGQ_U4>(T, e0, e1, item == 0, E); break;
    default: qab_quant_range<FGQ_S4>(T, e0, e1, item == 0, E); break;
  }
}

template <int MAXT>
__global__ void __launch_bounds__(kBatchThreads, kBatchBlocks) qab_kernel(const __grid_constant__ QBatch<MAXT> p,
                                                                        unsigned int* err) {
  __shared__ uint32_t red[2][kBatchThreads / 32];  // alternating: an item's is read while the next is reduced
  __shared__ int sE[2];
  int b = 0, cur = -1, E = 0;
  for (int i = blockIdx.x; i < p.items; i += gridDim.x) {
    int lo = 0, hi = p.nseg - 1;
    while (lo < hi) {  // the last segment that starts at or before i
      const int mid = (lo + hi + 1) >> 1;
      if (p.seg[mid].first <= i) lo = mid;
      else hi = mid - 1;
    }
    const QTensor& T = p.t[p.seg[lo].tensor];
    const int item = i - p.seg[lo].first;
    if (p.seg[lo].pass == 1) {
      qab_max_item(T, item, red[b], err);
      b ^= 1;
    } else {
      if (p.seg[lo].tensor != cur) {  // the same tensor as before: its exponent is known
        bool late = false;
        if (threadIdx.x == 0) {
          const uint32_t mask = (1u << kBatchCountBits) - 1u;
          uint32_t w;
          uint64_t t0 = 0;
          while (((w = load_acquire(T.word)) & mask) != (uint32_t)T.items) {
            uint64_t now;
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now));
            if (t0 == 0) t0 = now;
            if (now - t0 > p.timeout_ns) {
              record_error(err, FGQ_ERR_TIMEOUT);
              late = true;
              break;
            }
            __nanosleep(100);
          }
          sE[b] = code_exponent(w >> kBatchCountBits);
        }
        if (__syncthreads_or(late)) return;
        E = sE[b];
        b ^= 1;
        cur = p.seg[lo].tensor;
      }
      qab_quant_item(T, item, E);
    }
  }
}

template <int MAXT>
fgq_status launch_qab(int n, const float* const* x, const size_t* nelem, const int* type, void* const* q,
                      float* const* scale_out, unsigned int* words, unsigned int* err, cudaStream_t s) {
  QBatch<MAXT> p;
  memset(&p, 0, sizeof p);
  int nt = 0;
  for (int i = 0; i < n; ++i) {
    if (nelem[i] == 0) continue;
    const int64_t items = ((int64_t)nelem[i] + kBatchElems - 1) / kBatchElems;
    if (items >= (int64_t)1 << kBatchCountBits) return FGQ_ERR_UNSUPPORTED;  // 256 GB of input
    QTensor& T = p.t[nt++];
    T.x = x[i];
    T.q = static_cast<uint8_t*>(q[i]);
    T.scale = scale_out[i];
    T.word = words + i;
    T.n = (int64_t)nelem[i];
    T.type = type[i];
    T.items = (int)items;
  }
  if (nt == 0) return FGQ_OK;
  int64_t total = 0;
  auto add = [&](int t0, int t1, int pass) {
    for (int t = t0; t < t1; ++t) {
      p.seg[p.nseg].first = (int)total;
      p.seg[p.nseg].tensor = (int16_t)t;
      p.seg[p.nseg++].pass = (int16_t)pass;
      total += p.t[t].items;
    }
  };
  int prev = 0;  // first tensor of the chunk that waits for pass 2
  for (int t = 0; t < nt;) {
    // a chunk: consecutive tensors up to kBatchChunkBytes of input (at least one tensor)
    int end = t;
    size_t bytes = 0;
    while (end < nt && (end == t || bytes + (size_t)p.t[end].n * sizeof(float) <= kBatchChunkBytes))
      bytes += (size_t)p.t[end++].n * sizeof(float);
    add(t, end, 1);
    add(prev, t, 2);
    prev = t;
    t = end;
  }
  add(prev, nt, 2);
  if (total > INT32_MAX / 2) return FGQ_ERR_UNSUPPORTED;
  p.items = (int)total;
  const int64_t lim_us = debug_wait_limit_us();
  p.timeout_ns = lim_us < 0 ? kBatchTimeoutNs : (uint64_t)lim_us * 1000u;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kBatchThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // A context that holds a part of the SMs (a partition of the device) cannot keep the whole grid
  // resident: fewer blocks, down to one, do the same items.
  const int64_t cap = (int64_t)device_sms() * kBatchBlocks, resident = debug_resident_blocks();
  for (int64_t grid = total < cap ? total : cap;; grid = (grid + 1) / 2) {
    cfg.gridDim = dim3((unsigned)grid);
    const cudaError_t e = resident >= 0 && grid > resident ? cudaErrorCooperativeLaunchTooLarge
                                                           : cudaLaunchKernelEx(&cfg, qab_kernel<MAXT>, p, err);
    if (e != cudaErrorCooperativeLaunchTooLarge || grid == 1) return after_launch(e);
    cudaGetLastError();
  }
}

}  // namespace

size_t quantize_batch_workspace_bytes(int n) { return n > 0 ? sizeof(unsigned int) * (size_t)n : 0; }

fgq_status launch_quantize_batch(int n, const float* const* x, const size_t* nelem, const int* type, void* const* q,
                                 float* const* scale_out, unsigned int* words, unsigned int* err, cudaStream_t s) {
  if (cudaMemsetAsync(words, 0, sizeof(unsigned int) * (size_t)n, s) != cudaSuccess) return FGQ_ERR_CUDA;
  return n <= 32 ? launch_qab<32>(n, x, nelem, type, q, scale_out, words, err, s)
                 : launch_qab<FGQ_QUANTIZE_BATCH_MAX>(n, x, nelem, type, q, scale_out, words, err, s);
}

}  // namespace fgq

// ----------------------------------------------------------------------------------------
// fgq_quantize_act_noalloc: the derived-scale quantizer for callers that cannot allocate
// device memory.  Some hosts own every device allocation themselves (a framework's memory
// pool with a fixed budget, a plugin that only receives pre-allocated tensors) or cannot
// afford cudaMalloc/cudaFree on the inference path (cudaFree synchronizes the device, and a
// fresh allocation can stall or fail under memory pressure).  For them the per-block maxima
// of pass 1 live in this file-scope device array instead of a caller-provided workspace.
//
// The array is a host-side stand-in in host code, not a device address, so its address is
// obtained once per device with cudaGetSymbolAddress (with that device current) and passed
// to the kernels.  That set-up happens in the first call on each device, which should
// therefore come before any stream capture.  Every GPU that loads the library keeps the
// array (16 KB) until exit.  All calls share it: each call fully rewrites the slots it uses
// before reading them, so nothing needs clearing, but calls that overlap on the GPU (in
// different streams, or from different threads) race on it and must be serialized.
namespace fgq {
namespace {

constexpr int kNoallocScratchWords = 4096;  // maximum number of pass-1 blocks
static __device__ __align__(256) uint32_t g_noalloc_scratch[kNoallocScratchWords];

constexpr int kNoallocMaxDevices = 64;
uint32_t* g_noalloc_ptr[kNoallocMaxDevices];
std::mutex g_noalloc_mu;

// Device address of the scratch array on the current device (nullptr on failure).
uint32_t* noalloc_scratch() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoallocMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) return nullptr;
    g_noalloc_ptr[dev] = static_cast<uint32_t*>(p);
  }
  return g_noalloc_ptr[dev];
}

}  // namespace
}  // namespace fgq

extern "C" fgq_status fgq_quantize_act_noalloc(const float* x, size_t n, fgq_act_type type, float scale_in,
                                               void* q, float* scale_out, cudaStream_t stream) {
  using namespace fgq;
  if (type != FGQ_U8 && type != FGQ_S8 && type != FGQ_U4 && type != FGQ_S4) return FGQ_ERR_ARG;
  int E = 0;
  const bool derive = !(scale_in > 0.0f);
  if (!derive) {  // a given scale must be a power of two 2^E (subnormal ones included)
    uint32_t b;
    memcpy(&b, &scale_in, sizeof b);
    const uint32_t ex = b >> 23, man = b & 0x7fffffu;
    if (ex == 255) return FGQ_ERR_ARG;
    if (ex > 0) {
      if (man != 0) return FGQ_ERR_ARG;
      E = (int)ex - 127;
    } else {
      if (man & (man - 1)) return FGQ_ERR_ARG;
      E = -149 + (31 - __builtin_clz(man));
    }
  }
  if (n == 0) return FGQ_OK;
  if (!x || !q || (derive && !scale_out)) return FGQ_ERR_ARG;
  if ((reinterpret_cast<uintptr_t>(x) & 15) || (reinterpret_cast<uintptr_t>(q) & 15) ||
      (scale_out && (reinterpret_cast<uintptr_t>(scale_out) & 3)))
    return FGQ_ERR_ALIGN;
  uint32_t* scratch = nullptr;
  if (derive) {
    if (quantize_workspace_bytes(n) > sizeof(uint32_t) * (size_t)kNoallocScratchWords) return FGQ_ERR_UNSUPPORTED;
    scratch = noalloc_scratch();
    if (!scratch) return FGQ_ERR_CUDA;
  }
  return launch_quantize(x, n, type, E, derive, q, scale_out, scratch, device_error_word(), stream);
}
