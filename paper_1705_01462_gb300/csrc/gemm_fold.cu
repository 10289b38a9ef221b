// Tensor-core (tcgen05) grouped ternary contraction with the group scales folded into the
// weights, for groups smaller than an MMA K-tile (G = 4, 8, 16, 32) and for G = 64 where the channels
// do not fill the K-tiles of the per-group kernel.
//
// Eq. 2 is one dense contraction, y[p][m] = s_x sum_k A[m][k] q[p][k] with A = alpha(m, k / G)
// t[m][k], if it can be summed without losing what the 32-bit group accumulators of Section 4
// keep.  Here it can, because the folded weights are integers on a common grid: the reduction
// is cut into units of about 256 elements and whole groups (plan_units), and in each unit row m is
// scaled by a power of two 2^e that puts its largest alpha into [2^10, 2^11) ([2^9, 2^10) at G = 64);
// with v = alpha 2^e and d = 12 (11 at G = 64),
//     hi = round(v),   lo = round((v - hi) 2^d),
// fp16 numbers of magnitude at most 2^(d - 1) on a grid of 2^-f (and of their own ulp).
//
// f = 0, integers, where a group may reach over several MMA steps (G >= 32, or channels that are no
// multiple of G).  Products with 8-bit codes are integers, and so are their sums, exact in the fp32
// accumulator below 2^24, in any order, whatever cancels.  What an accumulator holds of whole
// groups is bounded by their own |alpha s|, what it holds of a group half summed by 2^23 (32
// products of 255 with 2^10 at G = 64, 16 with 2^11 at G = 32), however much of that the other half
// takes back: a prefix that passes 2^24 has more than 2^23 from S = s_x sum_g |alpha_g s_g| in it, and
// rounding it costs at most 2^-22 of S in each of a unit's 16 to 32 accumulations.
//
// f = 6 where every group lies inside one MMA step of 16 elements: the accumulator then holds whole
// groups only, and a step adds its 16 products and the accumulator without loss between 2^19, the
// largest, and 2^-8 (found exact on this chip, and tested down to 2^-6 of products next to
// cancelling ones of 2^19; a narrower sum would lose what a large group leaves behind).  Alphas down to
// 2^-7 of the largest then keep 22 bits in one pair.
//
// What the pair (hi, lo) leaves out of an alpha at f = 0 is at most 2^-(d + 1) of v's unit: 2^-13, or
// 2^-24 of the unit's largest alpha, but more of a smaller one.  A unit in which some alpha of the
// tile's 64 filters loses more than pair_tolerance of itself gets a second pair, the next two digits of
// the same rule, contracted in a pass of its own over the unit: 47 bits of the largest alpha in all (43
// at G = 64), every bit of alphas down to 2^-23 (2^-19) of it and 18 bits down to 2^-29 (2^-25).
// The tolerance keeps the output's error no larger than that of fp32 alphas on exact group sums,
// also where a row's large alphas meet inactive channels.  Gaussian weights: no unit at f = 6 where a
// filter has 20 groups more than three per unit, else all; at G = 32 and 64 nearly all.
// (Integers in one pair, and a third part only from alphas 64 times below the largest on, erred by
// 2.6e-6 where dp4a errs by 4.4e-7: one large alpha in 256 elements with zero activations, the others
// 45 times smaller.  Integers for all G, in two pairs wherever the tolerance asks, at G = 4 everywhere,
// took 48 us for the first call below and 366 for the fourth.)
// Against S the error is below 16 2^-22 (accumulations of four K-tiles) + 2^-20 (alphas of one pair) +
// n_units 2^-24 for each pair (fp32 adds): 1e-5 up to 88 units of one pair or 52 of two, if every rounding
// goes the same way; measured it is 1e-7.
//
// hi and lo are two rows of the same MMA operand: a tile is 64 filters x up to 256 positions,
// 128 operand rows (rows 32 q + i and 32 q + 16 + i: hi and lo of filter 16 q + i), so that one
// epilogue warp reads both parts of its 16 filters (adding them across lanes by shuffles cost
// more than the rest of the tile end).  The MMA work is
// twice the dense contraction's for each pair.  (A block-diagonal operand with a row per group slot,
// used at G = 4 before, did eight times the dense work, drained TMEM every K-tile and wrote 16 bytes of
// operand per weight.  A call before and now, us: 3x3 128 -> 128 on 28 x 28, batch 64, G = 4: 82 and
// 33; 3x3 256 -> 256 on 14 x 14, batch 64, G = 8 (dp4a before): 236 and 32, and with two pairs, G = 32,
// 179 and 54; 5x5 with 2 x 48 channels on 27 x 27, batch 256, G = 4 (dp4a before): 2661 and 207, with two
// pairs, G = 64, 1742 and 366; GEMM 4096 x 9216, P = 256, G = 4: 555 and 89.)
// Bound: the tensor pipe for long reductions (512 clk per 64 x 256 x 64 K-tile pair), the stores
// of the tile end for short ones.
//
// Both operands are prepared once per call by one launch (prep_fold_kernel): the folded weights
// as ready 16 KB K-tile images (128-byte swizzle, fetched by one bulk copy each), the
// activations as fp16 with each conv group's channels padded to a multiple of 64.  The producer
// and the MMA issuer run their loops warp-uniformly and issue from an elected lane: with the
// loop inside a single divergent lane every TMA and MMA instruction cost about 100 clk to
// issue (four MMAs 386 clk and a K-tile's loads 625 clk, against the 512 clk the tensor pipe
// needs for the K-tile).
//
// Warp roles (352 threads, one CTA per SM, persistent over tiles):
//   warps 0-7  epilogue: warp w reads the operand rows of 16 filters (TMEM lanes 32 (w % 4) ..) for
//              the positions of half w / 4, adds each drained unit's hi + 2^-12 lo, scaled by the
//              row's 2^-e, into fp32 registers, and at tile end stores y or its codes;
//   warps 8, 9 MMA issue (warp 8 also allocates TMEM), the units in turn: four M = 128 MMAs per
//              K-tile into the unit's accumulator, a commit per K-tile frees its stage, one per
//              unit hands it over;
//   warp 10    producer: per K-tile one bulk copy (weights) and one TMA box (activations: 2D
//              rows, or an im2col box of the tile's positions at the K-tile's filter tap).
// Every mbarrier wait is bounded in time; on expiry the kernel records FGQ_ERR_TIMEOUT, every
// role leaves its loop (the epilogue uniformly), issued copies and MMAs are waited for, and
// TMEM is freed.
#include <cuda_fp16.h>

#include <cmath>
#include <cstdint>
#include <cstring>

#include "operand_prep.cuh"
#include "tc_common.cuh"

namespace fgq {
namespace {

using tc::make_map_2d;
using tc::make_map_im2col;

constexpr int TF_ROWS = 128;      // MMA M
constexpr int TF_FM = 64;         // filters per tile (two operand rows each)
constexpr int TF_KT = 64;         // reduction elements per K-tile: 4 MMAs
constexpr int TF_DIGIT = 12;      // bits of an alpha's part: integers up to 2048.  11 at G = 64, so that half a
                                  // group, 32 products of 255 with the largest alpha, is 2^23 there too
constexpr int TF_FRAC = 6;        // fractional bits of a part where groups lie inside MMA steps
constexpr int TF_UNIT = 4;        // K-tiles per unit (one TMEM accumulation) where its groups allow it,
constexpr int TF_MAX_UNIT = 8;    // and at most (plan_units)
constexpr int TF_MAX_BN = 256;    // positions per tile (MMA N), a multiple of 64
constexpr int TF_MAX_NST = 8;     // operand ring depth, at most (as many stages as fit)
constexpr int TF_EPI_WARPS = 8;
constexpr int TF_MMA_WARP = 8;    // warps 8 and 9
constexpr int TF_PROD_WARP = 10;
constexpr int TF_THREADS = 32 * (TF_PROD_WARP + 1);
constexpr int TF_COLS = TF_MAX_BN / 4;  // positions per epilogue thread, at most
constexpr uint64_t TF_TIMEOUT_NS = 1000000000ull;  // 1 s per wait
constexpr uint32_t TF_DRAIN_LIMIT = 1u << 20;      // polls of the final drains (never shortened)
constexpr uint32_t BAR_EPIF = 2;

constexpr int TF_A = TF_ROWS * TF_KT * 2;      // 16 KB; a stage adds bn * 128 bytes of activations
constexpr int TF_RING = 196608;                // 4 stages at bn = 256, 8 at bn <= 64
constexpr int TF_SHORT = 4;                    // K-tiles up to which a tile has four output boxes per warp
                                               // (K = 64, 64 -> 256 channels on 56 x 56, batch 64: 51 us
                                               // against 69 us with two)
constexpr int TF_BOX_POS = 32;                 // positions per output box
constexpr int TF_BOX = TF_BOX_POS * 16 * 4;    // 2 KB: fp32 [32 positions][16 filters]
// Two output boxes per epilogue warp behind the ring -- or, for tiles of few K-tiles, whose time
// goes into the stores, four (a whole tile at bn = 256): a ring one stage shorter.
constexpr int TF_OUT = 2 * TF_EPI_WARPS * TF_BOX;
constexpr int TF_SMEM = 1024 + TF_RING + TF_OUT + 8 * (2 * TF_MAX_NST + 7) + 16;
static_assert(TF_SMEM <= 232448, "shared memory budget");

struct FoldArgs {
  CUtensorMap act_map;   // fp16 activations: 2D [positions][Ca] or im2col, box 64 channels x bn positions
  CUtensorMap out_map;   // out_tma: outputs [P][M] (fp32 or codes), box {16 filters, 32 positions}
  const uint8_t* a_op;   // weight K-tile images [tile][nunits][uk + ux] of TF_A bytes
  const uint8_t* a_ext;  // the second pairs, same layout (written where ext is set)
  const float* rs;       // 2^-e [tile][nunits][TF_FM]
  const uint8_t* ext;    // [tile][nunits]
  const float* act_scale;
  float* out;
  unsigned int* err;
  Geom g;
  int cpad;                     // channels per conv group in the padded activations
  int bn, nst;                  // positions per tile, ring depth
  int obufs;                    // output boxes per epilogue warp: 2 or 4
  float lo_scale, ext_scale;    // 2^-dbits, 2^-(2 dbits)
  int mtiles, ntiles, ktiles, nunits;
  int uk, ux;                   // K-tiles from a unit's start to the next one's, and past that (plan_units)
  int out_tma;
  uint64_t timeout_ns;
};

// Tile t: weight tile gm = gi mtiles + mt (filters gi Mg + 64 mt ..), positions p0 ...  Weight
// tiles of one position tile are consecutive, so CTAs running at the same time share
// activation boxes in L2.
__device__ __forceinline__ void fold_tile(const FoldArgs& a, int t, int& gm, int& pt) {
  const int per_p = a.g.groups * a.mtiles;
  pt = t / per_p;
  gm = t - pt * per_p;
}

// ---------------------------------------------------------------------------- preparation

// What one launch prepares.  Blocks [0, fold_blocks): the weight images of one (weight tile,
// unit), K-tiles split nsub ways over blocks; the others: activations to fp16.
struct PrepFold {
  const uint32_t* codes;
  const float* alpha;
  uint8_t* a_op;
  uint8_t* a_ext;
  float* rs;
  uint8_t* ext;
  int wrow, ng, gshift;  // G = 1 << gshift
  int dbits, fbits;      // bits of a part; fractional bits
  int Mg, Cg, cpad, mtiles, ktiles, nunits, uk, ux, nsub, fold_blocks;
  float tol;             // share of an alpha that one pair of parts may leave out
  int quads;             // Cg % 4 == 0: 4 elements from a multiple of 4 lie in one tap and one group
  int padded;            // activations need the padded expansion
  int fast8;             // ... of 8-bit codes in aligned runs of 8 (Cg and C multiples of 8)
  int sC, sgroups;       // source channels, conv groups (padded expansion)
  int64_t npix;          // pixels of the expanded activations
};

constexpr int PF_GPU = TF_UNIT * TF_KT / 4 + 2;  // groups of a unit, at most 65, and a pad word

__device__ __forceinline__ uint32_t h2u(float v) { return (uint32_t)__half_as_ushort(__float2half_rn(v)); }

// Padded expansion: 8 channels (16 bytes of fp16) of one pixel and conv group per step.
__device__ __forceinline__ int64_t src_pixel(const prep::ActSrc& s, int64_t pix) {
  if (!s.strided) return pix;
  const int wo = (int)(pix % s.Wo);
  const int64_t q = pix / s.Wo;
  return ((q / s.Ho) * s.H + (q % s.Ho) * s.stride) * s.W + (int64_t)wo * s.stride;
}

// Aligned 8-bit codes: four source loads in flight per thread; the (pixel, chunk) pair of the
// next step is advanced without a division.
__device__ __forceinline__ void expand_padded8(const PrepFold& f, const prep::ActSrc& s, int64_t first, int64_t step,
                                               uint4* out) {
  const int cpp = f.cpad / 8;            // chunks per pixel and group
  const int cpr = cpp * f.sgroups;       // chunks per pixel
  const uint32_t flip = s.sgn ? 0x80808080u : 0u, bias = s.sgn ? 0x64806480u : 0x64006400u;
  const int64_t n = f.npix * cpr, dpix = step / cpr;
  const int dc = (int)(step - dpix * cpr);
  int64_t pix = first / cpr;
  int c = (int)(first - pix * cpr);
  for (int64_t i = first; i < n; i += 4 * step) {
    uint2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[u] = make_uint2(0u, 0u);
      const int gi = c / cpp, c0 = (c - gi * cpp) * 8;
      if (i + u * step < n && c0 < f.Cg)
        v[u] = __ldg(reinterpret_cast<const uint2*>(s.act + src_pixel(s, pix) * f.sC + gi * f.Cg + c0));
      pix += dpix;
      c += dc;
      if (c >= cpr) {
        c -= cpr;
        ++pix;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (i + u * step < n)
        out[i + u * step] = make_uint4(tc::u8pair_to_h2(v[u].x ^ flip, 0x4140, bias), tc::u8pair_to_h2(v[u].x ^ flip, 0x4342, bias),
                                       tc::u8pair_to_h2(v[u].y ^ flip, 0x4140, bias), tc::u8pair_to_h2(v[u].y ^ flip, 0x4342, bias));
    }
  }
}

// Any channel counts, 8- or 4-bit codes: element by element.
__device__ __forceinline__ void expand_padded(const PrepFold& f, const prep::ActSrc& s, int64_t first, int64_t step,
                                              uint4* out) {
  const int cpp = f.cpad / 8;  // chunks per pixel and group
  const int64_t n = f.npix * f.sgroups * cpp;
  for (int64_t i = first; i < n; i += step) {
    const int64_t pg = i / cpp;
    const int c0 = (int)(i - pg * cpp) * 8;
    const int64_t pix = pg / f.sgroups;
    const int gi = (int)(pg - pix * f.sgroups);
    const int64_t e0 = src_pixel(s, pix) * f.sC + (int64_t)gi * f.Cg + c0;
    uint32_t h[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      int x = 0;
      if (c0 + e < f.Cg) {
        const int64_t el = e0 + e;
        if (s.abits == 8) {
          const uint8_t b = __ldg(s.act + el);
          x = s.sgn ? (int)(int8_t)b : (int)b;
        } else {
          x = (__ldg(s.act + (el >> 1)) >> (4 * (int)(el & 1))) & 15;
          if (s.sgn) x = (x ^ 8) - 8;
        }
      }
      h[e] = h2u((float)x);
    }
    out[i] = make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
  }
}

// The fp16 number next to v on a grid of 1 / frac, which is finer than fp16 itself from 1024 / frac on.
__device__ __forceinline__ __half grid_half(float v, float frac, float unfrac) {
  return __float2half_rn(fabsf(v) < 1024.0f * unfrac ? rintf(v * frac) * unfrac : v);
}

// The two parts of a scaled alpha, fp16 bits of hi and (above) lo; v becomes what they leave, times
// digit^2: the next pair's v.
__device__ __forceinline__ uint32_t split2(float& v, float digit, float frac, float unfrac) {
  const __half h = grid_half(v, frac, unfrac);
  const float r1 = (v - __half2float(h)) * digit;
  const __half l = grid_half(r1, frac, unfrac);
  v = (r1 - __half2float(l)) * digit;
  return (uint32_t)__half_as_ushort(h) | (uint32_t)__half_as_ushort(l) << 16;
}

// The fp16 pair (x, x) with the signs and zeros of two codes (4 bits: 00 = 0, 01 = +1, 11 = -1).
__device__ __forceinline__ uint32_t code_pair(uint32_t c, uint32_t x) {
  const uint32_t nz = ((c & 1u) | ((c & 4u) << 14)) * 0xffffu;
  const uint32_t sg = ((c & 2u) << 14) | ((c & 8u) << 28);
  return ((x * 0x10001u) ^ sg) & nz;
}

// Four blocks per SM: without that bound 74 registers and three, GEMM 4096 x 9216 51 us instead of 46.
__global__ void __launch_bounds__(256, 4) prep_fold_kernel(const __grid_constant__ PrepFold f,
                                                        const __grid_constant__ prep::ActSrc src, uint4* __restrict__ x16) {
  __shared__ uint32_t al[TF_FM][PF_GPU + 1];  // a pair of parts of each of the unit's alphas (split2)
  pdl_wait();
  pdl_trigger();
  if ((int)blockIdx.x >= f.fold_blocks) {
    const int64_t nb = (int64_t)gridDim.x - f.fold_blocks;
    const int64_t first = ((int64_t)blockIdx.x - f.fold_blocks) * blockDim.x + threadIdx.x;
    if (f.fast8) expand_padded8(f, src, first, nb * blockDim.x, x16);
    else if (f.padded) expand_padded(f, src, first, nb * blockDim.x, x16);
    else prep::act_expand<false>(src, first, nb * blockDim.x, x16);
    return;
  }
  const int sub = (int)blockIdx.x % f.nsub;
  const int tu = (int)blockIdx.x / f.nsub;
  const int tile = tu / f.nunits, u = tu - tile * f.nunits;
  const int gi = tile / f.mtiles, mt = tile - gi * f.mtiles;
  const int kt0 = u * f.uk;
  // the unit's groups [g0, g1): those that begin in its own uk K-tiles.  The last may run into the
  // K-tiles after them (ux), whose other groups are left to the next unit.
  auto real = [&](int kt) {  // real reduction elements ahead of K-tile kt
    const int tap = kt * TF_KT / f.cpad;
    return tap * f.Cg + (kt * TF_KT - tap * f.cpad);
  };
  const int ge = (1 << f.gshift) - 1;
  const int g0 = (real(kt0) + ge) >> f.gshift;
  const int g1 = kt0 + f.uk < f.ktiles ? (real(kt0 + f.uk) + ge) >> f.gshift : f.ng;
  const int kt1 = kt0 + f.uk + f.ux < f.ktiles ? kt0 + f.uk + f.ux : f.ktiles;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float digit = (float)(1 << f.dbits);
  const float frac = (float)(1 << f.fbits), unfrac = 1.0f / frac;
  const float tol = f.tol * digit * digit;
  bool wide = false;  // some alpha needs the second pair
  float v[TF_FM / 8][3];  // 8 filters per warp, every load in flight at once
#pragma unroll
  for (int i = 0; i < TF_FM / 8; ++i) {
    const int local = mt * TF_FM + (TF_FM / 8) * warp + i;
    const float* ar = f.alpha + ((int64_t)gi * f.Mg + (local < f.Mg ? local : 0)) * f.ng;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int gg = g0 + lane + 32 * j;
      v[i][j] = local < f.Mg && gg < g1 ? __ldg(ar + gg) : 0.0f;
    }
  }
#pragma unroll
  for (int i = 0; i < TF_FM / 8; ++i) {
    const int fl = (TF_FM / 8) * warp + i;
    uint32_t mx = 0;  // the largest magnitude's bits: above infinity's if one is a NaN
#pragma unroll
    for (int j = 0; j < 3; ++j) mx = max(mx, __float_as_uint(v[i][j]) & 0x7fffffffu);
    mx = __reduce_max_sync(FULL_MASK, mx);
    // 2^e puts the largest alpha into [digit / 4, digit / 2); e is kept where 2^e and 2^-e are normal
    int e = 0;
    if (mx < 0x7f800000u) {
      if (mx != 0) e = f.dbits - 2 - ilogbf(__uint_as_float(mx));
      e = e < -120 ? -120 : (e > 120 ? 120 : e);
    } else {
      // An infinite alpha: a number that both pairs hold a share of, at a row scale of infinity; the others
      // zero.  The unit gives infinity where its codes' sum is not zero, else NaN, as infinity times
      // the group sum does.  A NaN: a row scale of NaN.
#pragma unroll
      for (int j = 0; j < 3; ++j)
        v[i][j] = (__float_as_uint(v[i][j]) & 0x7fffffffu) == 0x7f800000u ? copysignf(0x1.000002p-1f, v[i][j]) : 0.0f;
    }
    const float mul = pow2f(e);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float x = v[i][j] * mul;  // exact: a power of two
      v[i][j] = x;
      const uint32_t parts = split2(v[i][j], digit, frac, unfrac);  // leaves the rest in v
      if (fabsf(v[i][j]) > tol * fabsf(x)) wide = true;
      if (lane + 32 * j < PF_GPU) al[fl][lane + 32 * j] = parts;
    }
    if (sub == 0 && lane == 0)
      f.rs[((int64_t)tile * f.nunits + u) * TF_FM + fl] = mx < 0x7f800000u ? pow2f(-e) : __uint_as_float(mx);
  }
  const bool ext = __syncthreads_or(wide);
  if (sub == 0 && threadIdx.x == 0) f.ext[(int64_t)tile * f.nunits + u] = ext ? 1 : 0;

  for (int pair = 0;; ++pair) {
    // 16-byte chunks of the images: chunk c (8 elements) of the operand rows of filter fl
    for (int kt = kt0 + sub; kt < kt1; kt += f.nsub) {
      const int tap = kt * TF_KT / f.cpad, cb = kt * TF_KT - tap * f.cpad;
      uint8_t* img = (pair ? f.a_ext : f.a_op) + (((int64_t)tile * f.nunits + u) * (f.uk + f.ux) + (kt - kt0)) * TF_A;
#pragma unroll
      for (int it = 0; it < TF_FM * 8 / 256; ++it) {
        const int idx = (int)threadIdx.x + 256 * it;
        const int fl = idx >> 3, c = idx & 7;
        const int local = mt * TF_FM + fl;
        const int ch = cb + 8 * c;  // channel of the chunk's first element
        const int nv = local < f.Mg ? f.Cg - ch : 0;  // real elements from here on
        const int k = tap * f.Cg + ch;
        uint32_t cw = 0u;
        if (nv > 0) {
          const uint32_t* cr = f.codes + ((int64_t)gi * f.Mg + local) * f.wrow + (k >> 4);
          const uint32_t lo = __ldg(cr);
          const uint32_t hi = (k & 15) > 8 && (k >> 4) + 1 < f.wrow ? __ldg(cr + 1) : 0u;
          cw = __funnelshift_r(lo, hi, 2 * (k & 15));
          cw &= nv < 8 ? (1u << (2 * nv)) - 1u : 0xffffu;
        }
        uint32_t p0[4], p1[4];
        if (f.quads) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int gr = ((k + 4 * q) >> f.gshift) - g0;
            const uint32_t c4 = (uint32_t)gr < (uint32_t)(g1 - g0) ? (cw >> (8 * q)) & 0xffu : 0u;
            const uint32_t x = c4 ? al[fl][gr] : 0u;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const uint32_t c2 = (c4 >> (4 * h)) & 15u;
              p0[2 * q + h] = code_pair(c2, x & 0xffffu);
              p1[2 * q + h] = code_pair(c2, x >> 16);
            }
          }
        } else {
#pragma unroll
          for (int e2 = 0; e2 < 4; ++e2) {
            p0[e2] = p1[e2] = 0u;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int e = 2 * e2 + h;
              const uint32_t t = (cw >> (2 * e)) & 3u;  // 00 = 0, 01 = +1, 11 = -1
              const int gr = ((k + e) >> f.gshift) - g0;
              if (t && (uint32_t)gr < (uint32_t)(g1 - g0)) {
                const uint32_t x = al[fl][gr] ^ (t == 3u ? 0x80008000u : 0u);
                p0[e2] |= (x & 0xffffu) << (16 * h);
                p1[e2] |= (x >> 16) << (16 * h);
              }
            }
          }
        }
        const int r0 = ((fl >> 4) << 5) + (fl & 15);  // operand row of hi; lo is 16 below
        const int o0 = r0 * 128 + ((c ^ (r0 & 7)) << 4);
        const int o1 = o0 + 16 * 128;  // (r0 + 16) & 7 == r0 & 7
        *reinterpret_cast<uint4*>(img + o0) = make_uint4(p0[0], p0[1], p0[2], p0[3]);
        *reinterpret_cast<uint4*>(img + o1) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
      }
    }
    if (pair || !ext) return;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TF_FM / 8; ++i) {
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (lane + 32 * j < PF_GPU) al[(TF_FM / 8) * warp + i][lane + 32 * j] = split2(v[i][j], digit, frac, unfrac);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------- contraction

// RQ: the output is requantized codes (a kernel of its own: the epilogue is one long unrolled
// block, and with both forms in it instruction fetch held it up).
template <bool TMAP, bool RQ>
__global__ void __launch_bounds__(TF_THREADS, 1) fold_contract_kernel(const __grid_constant__ FoldArgs a) {
  extern __shared__ uint8_t smem_rawf[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_rawf) + 1023) & ~uintptr_t(1023));
  uint8_t* obox = smem + TF_RING + TF_OUT - TF_EPI_WARPS * a.obufs * TF_BOX;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + TF_RING + TF_OUT);
  uint64_t* empty = full + TF_MAX_NST;
  uint64_t* acc_full = empty + TF_MAX_NST;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* turn = acc_empty + 2;
  uint64_t* drain_bar = turn + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // warp-uniform
  const int lane = threadIdx.x & 31;
  const Geom& g = a.g;
  const uint64_t tmo = a.timeout_ns;
  const int nst = a.nst;
  const uint32_t stage = (uint32_t)(TF_A + a.bn * TF_KT * 2);  // bytes of a stage

  if (threadIdx.x == 0) {
    for (int i = 0; i < nst; ++i) {
      mbar_init(&full[i], 1);   // the producer's expect_tx, then the copies' bytes
      mbar_init(&empty[i], 1);  // the commit after the K-tile's MMAs
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], TF_EPI_WARPS);
      mbar_init(&turn[i], 1);
    }
    mbar_init(drain_bar, 2);  // one commit per MMA issuer
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == TF_MMA_WARP) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // the prologue above overlapped the previous kernel; global memory only from here on
  pdl_wait();
  pdl_trigger();

  auto fail = [&]() {
    *abort_flag = 1;
    record_error(a.err, FGQ_ERR_TIMEOUT);
  };

  if (warp == TF_PROD_WARP) {
    // -------------------------------------------------------------- producer
    const uint32_t sbase = smem_u32(smem);
    int s = 0;
    uint32_t ph = 1;  // parity of the stage's previous release; the first round passes at once
    int issued = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
      int gm, pt;
      fold_tile(a, t, gm, pt);
      const uint8_t* xp = a.ext + (int64_t)gm * a.nunits;
      int next_ext = __ldg(xp);  // the unit's mark, loaded one unit ahead
      const int cb = (gm / a.mtiles) * a.cpad;  // the conv group's first channel
      const int p0 = pt * a.bn;
      int n0 = 0, h0 = 0, w0 = 0;  // im2col: the tile's first window origin (input pixel coordinates)
      if (!TMAP) {
        const int wo = p0 % g.Wo;
        const int q = p0 / g.Wo;
        n0 = q / g.Ho;
        h0 = (q - n0 * g.Ho) * g.stride - g.pad;
        w0 = wo * g.stride - g.pad;
      }
      int tr = 0, ts = 0, tc0 = 0;
      int ntr = 0, nts = 0, ntc = 0;  // where the next unit begins
      for (int u = 0, kt0 = 0; u < a.nunits && ok; ++u, kt0 += a.uk) {
        const int nk = a.ktiles - kt0 < a.uk + a.ux ? a.ktiles - kt0 : a.uk + a.ux;
        const int passes = 1 + next_ext;
        if (u + 1 < a.nunits) next_ext = __ldg(xp + u + 1);
        const int utr = ntr, uts = nts, utc = ntc;
        for (int pass = 0; pass < passes && ok; ++pass) {
          const uint8_t* asrc = (pass ? a.a_ext : a.a_op) + ((int64_t)gm * a.nunits + u) * (a.uk + a.ux) * TF_A;
          tr = utr;
          ts = uts;
          tc0 = utc;
          for (int j = 0; j < nk; ++j, asrc += TF_A) {
            if (!mbar_wait_warp(&empty[s], ph, tmo, abort_flag)) {
              ok = false;
              break;
            }
            if (elect_one()) {
              const uint32_t sa = sbase + (uint32_t)s * stage;
              mbar_arrive_expect_tx(&full[s], stage);
              bulk_load(sa, asrc, TF_A, &full[s]);
              if (TMAP)
                tma_load_2d(sa + TF_A, &a.act_map, cb + tc0, p0, &full[s]);
              else
                tma_load_im2col_4d(sa + TF_A, &a.act_map, cb + tc0, w0, h0, n0, (uint16_t)ts, (uint16_t)tr, &full[s]);
            }
            __syncwarp();
            ++issued;
            if (++s == nst) {
              s = 0;
              ph ^= 1u;
            }
            tc0 += TF_KT;
            if (tc0 == a.cpad) {
              tc0 = 0;
              if (++ts == g.S) {
                ts = 0;
                ++tr;
              }
            }
            if (j == a.uk - 1) {
              ntr = tr;
              nts = ts;
              ntc = tc0;
            }
          }
        }
      }
    }
    if (!ok && !*abort_flag) fail();
    // loads the MMA issuers may not have consumed: the last nst issued, one per stage, each the
    // latest phase of its stage's barrier; none may outlive the CTA
    for (int j = issued - nst < 0 ? 0 : issued - nst; j < issued; ++j)
      mbar_wait_bounded(&full[j % nst], (j / nst) & 1, TF_DRAIN_LIMIT);
  } else if (warp >= TF_MMA_WARP) {
    // -------------------------------------------------------------- MMA issuers
    // Two warps, one per accumulator, take the units in turn: what one spends between units on
    // barriers overlaps the other's MMAs.  A unit begins when the other issuer has issued the one
    // before it (turn): the ring's barriers are then never more than one phase ahead of a wait.
    const int b = warp - TF_MMA_WARP;
    const uint32_t idesc = idesc_f16_f32(TF_ROWS, a.bn);
    const uint64_t ad0 = sdesc_k_sw128(smem_u32(smem)), bd0 = sdesc_k_sw128(smem_u32(smem) + TF_A);
    const uint32_t d = tmem + (uint32_t)(b * TF_MAX_BN);
    int s = 0, uc = 0;  // the ring position and the CTA's unit count
    uint32_t ph = 0, aph = 1, tph = b == 0 ? 1u : 0u;
    bool ok = true;
    for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
      int gm, pt;
      fold_tile(a, t, gm, pt);
      const uint8_t* xp = a.ext + (int64_t)gm * a.nunits;
      int next_ext = __ldg(xp);  // the unit's mark, loaded one unit ahead
      for (int u = 0, kt0 = 0; u < a.nunits && ok; ++u, kt0 += a.uk) {
        const int nk = a.ktiles - kt0 < a.uk + a.ux ? a.ktiles - kt0 : a.uk + a.ux;
        const int passes = 1 + next_ext;
        if (u + 1 < a.nunits) next_ext = __ldg(xp + u + 1);
        for (int pass = 0; pass < passes; ++pass, ++uc) {
          if ((uc & 1) != b) {  // the other issuer's unit
            for (s += nk; s >= nst; s -= nst) ph ^= 1u;
            continue;
          }
          if (!mbar_wait_warp(&acc_empty[b], aph, tmo, abort_flag) || !mbar_wait_warp(&turn[b], tph, tmo, abort_flag)) {
            ok = false;
            break;
          }
          aph ^= 1u;
          tph ^= 1u;
          for (int j = 0; j < nk; ++j) {
            if (!mbar_wait_warp(&full[s], ph, tmo, abort_flag)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (elect_one()) {
              const uint64_t off = (uint64_t)(((uint32_t)s * stage) >> 4);
#pragma unroll
              for (int k = 0; k < TF_KT / 16; ++k)  // advance 16 fp16 (32 bytes) along K
                mma_f16(d, ad0 + off + 2 * k, bd0 + off + 2 * k, idesc, (j | k) != 0 ? 1u : 0u);
              mma_commit(&empty[s]);
              if (j == nk - 1) {
                mma_commit(&acc_full[b]);
                mbar_arrive(&turn[b ^ 1]);
              }
            }
            __syncwarp();
            if (++s == nst) {
              s = 0;
              ph ^= 1u;
            }
          }
          if (!ok) break;
        }
      }
    }
    if (!ok && !*abort_flag) fail();
    // every MMA issued by both warps is complete once the drain barrier flips
    if (elect_one()) mma_commit(drain_bar);
    __syncwarp();
    mbar_wait_bounded(drain_bar, 0, TF_DRAIN_LIMIT);
  } else {
    // -------------------------------------------------------------- epilogue
    // Warp (quarter, half): 16 filters, bn / 2 positions.  A TMEM load of 16 lanes x 2 column runs
    // gives threads 0-15 the even and threads 16-31 the odd runs of 16 positions of the same
    // operand rows, so that each thread reads a filter's hi and lo itself.
    const int quarter = warp & 3, half = warp >> 2;
    const int fl = 16 * quarter + (lane & 15);  // filter of the tile
    const int hcols = a.bn / 2;                 // positions of this warp (a multiple of 32)
    const uint32_t tbase = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(hcols * half);
    const float sx = __ldg(a.act_scale), lo_scale = a.lo_scale;
    int b = 0, obuf = 0;
    uint32_t fph = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
      int gm, pt;
      fold_tile(a, t, gm, pt);
      const int gi = gm / a.mtiles;
      const int local = (gm - gi * a.mtiles) * TF_FM + fl;
      const int m = gi * g.Mg + local;
      const bool mok = local < g.Mg;
      const float* rsp = a.rs + (int64_t)gm * a.nunits * TF_FM + fl;
      const uint8_t* xp = a.ext + (int64_t)gm * a.nunits;
      float next_r = __ldg(rsp);  // the unit's row scale and mark, loaded one unit ahead
      int next_ext = __ldg(xp);
      float acc[TF_COLS];  // run j, position i: 16 j + i
#pragma unroll
      for (int i = 0; i < TF_COLS; ++i) acc[i] = 0.0f;
      for (int u = 0; u < a.nunits; ++u) {
        const float r0 = next_r;
        const int passes = 1 + next_ext;
        if (u + 1 < a.nunits) {
          next_r = __ldg(rsp + (int64_t)(u + 1) * TF_FM);
          next_ext = __ldg(xp + u + 1);
        }
        for (int pass = 0; pass < passes; ++pass) {
          if (!ok) continue;  // after a failed wait: run out the tile, then leave with the others
          const float r = pass ? r0 * a.ext_scale : r0;  // the second pair, below the first
          if (!mbar_wait_warp(&acc_full[b], fph, tmo, abort_flag)) {
            ok = false;
            continue;
          }
          tc_fence_after();
          const uint32_t ta = tbase + (uint32_t)(b * TF_MAX_BN);
#pragma unroll
          for (int j = 0; j < TF_COLS / 16; ++j) {
            if (32 * j < hcols) {
              uint32_t dh[16], dl[16];
              tmem_ld16x2(ta + 32 * j, dh);
              tmem_ld16x2(ta + 32 * j + (16u << 16), dl);
              tmem_ld_wait_regs16(dh);
              reg_fence16(dl);
#pragma unroll
              for (int i = 0; i < 16; ++i)
                acc[16 * j + i] =
                    fmaf(r, fmaf(lo_scale, __uint_as_float(dl[i]), __uint_as_float(dh[i])), acc[16 * j + i]);
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[b]);  // every column of the unit is in registers
          b ^= 1;
          if (b == 0) fph ^= 1u;
        }
      }
      if (!ok && !*abort_flag) fail();
      if (named_bar_or(BAR_EPIF, 32 * TF_EPI_WARPS, !ok)) break;  // leave together
      const int pw = pt * a.bn + hcols * half;  // the warp's first position
      RqMul rq;
      if (RQ) rq = rq_mul(g.rq_scale, g.rq_signed);
      if (a.out_tma) {
        // boxes of 32 positions x 16 filters through the warp's own buffers (no barrier with other
        // warps); positions past P and filters past M are clipped by the map
        if (local - (lane & 15) < g.Mg) {  // some of the warp's filters exist
          const int obufs = a.obufs;
          uint8_t* const ob0 = obox + obufs * warp * TF_BOX;
#pragma unroll
          for (int j = 0; j < TF_COLS / 16; ++j) {
            if (32 * j < hcols) {
              if (lane == 0) {  // the buffer's previous box has been read out
                if (obufs == 4) bulk_wait_read<3>();
                else bulk_wait_read<1>();
              }
              __syncwarp();
              uint8_t* ob = ob0 + obuf * TF_BOX;
              const int o0 = 16 * (lane & 16) + (lane & 15);  // row 0 or 16 of the box, the thread's filter
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float y = sx * acc[16 * j + i];
                if (RQ) ob[o0 + 16 * i] = rq_code(y, rq);  // fused requantization: 8-bit codes
                else reinterpret_cast<float*>(ob)[o0 + 16 * i] = y;
              }
              fence_proxy_async_smem();
              __syncwarp();
              if (lane == 0) {
                if (pw + 32 * j < g.P) tma_store_2d(&a.out_map, m, pw + 32 * j, smem_u32(ob));
                bulk_commit();
              }
              if (++obuf == obufs) obuf = 0;
            }
          }
        }
      } else if (mok) {
        const int64_t pb = (int64_t)pw + (lane & 16);
#pragma unroll
        for (int j = 0; j < TF_COLS / 16; ++j) {
          if (32 * j < hcols) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int64_t p = pb + 32 * j + i;
              if (p < g.P) {
                if (RQ) g.rq_out[p * g.M + m] = rq_code(sx * acc[16 * j + i], rq);
                else a.out[p * g.M + m] = sx * acc[16 * j + i];
              }
            }
          }
        }
      }
    }
    if (lane == 0) bulk_wait_all();  // this thread's TMA stores are complete
  }

  tc_fence_before();
  __syncthreads();
  if (warp == TF_MMA_WARP) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <bool TMAP, bool RQ>
fgq_status launch_fold(const FoldArgs& args, int grid, cudaStream_t s) {
  if (!tc::smem_attr_once<fold_contract_kernel<TMAP, RQ>>(TF_SMEM)) return FGQ_ERR_CUDA;
  return after_launch(launch_pdl(fold_contract_kernel<TMAP, RQ>, dim3(grid), dim3(TF_THREADS), TF_SMEM, s, args));
}

// Whether every group lies inside one 16-element slice of a K-tile (one MMA step).
bool in_slices(const Geom& g) { return g.G <= 16 && (g.Cg % g.G == 0 || g.R * g.S == 1); }

// The share of an alpha that its first pair of parts may leave out before the unit takes the second
// pair: so much that the output's error, with the fp32 adds of the units beside it, is no larger than
// that of fp32 alphas on exact group sums added in fp32 (the dp4a kernel), whichever alphas the
// activations leave active.  Measured, root mean square against 64 bits: n fp32 adds err by
// 1.75e-8 sqrt(n) for dp4a's groups (72 1.41e-7, 288 3.0e-7, 576 4.3e-7) and 2.8e-8 sqrt(n) for the units'
// (9 8.5e-8); a share that is uniform up to tol adds tol / sqrt(3).  G = 4 keeps 22 bits, as the
// split per group slot that ran it before, and every G 20 (the 1e-5 of S above).
float pair_tolerance(const Geom& g, int nunits) {
  const double spare = g.ng - 3.0 * nunits;
  const double tol = spare > 0.0 ? 2.7e-8 * sqrt(spare) : 0.0;
  return g.G == 4 ? 0x1p-22f : (float)(tol < 0x1p-20 ? tol : 0x1p-20);
}

// Positions per tile: the size that makes the persistent grid's last wave cheap.  A K-tile
// takes 2 bn clk of the tensor pipe (at least about 400 clk of issue), a tile's drain and
// stores about 10 bn + 600 clk, which overlap the next tile's MMAs.
int choose_bn(int64_t P, int wtiles, int ktiles, int sms) {
  int best = 64;
  double best_t = 1e30;
  for (const int bn : {256, 192, 128, 64}) {
    const int64_t tiles = (int64_t)wtiles * ((P + bn - 1) / bn);
    const int64_t waves = (tiles + sms - 1) / sms;
    const double mma = (double)ktiles * (2 * bn > 400 ? 2 * bn : 400), epi = 10.0 * bn + 600.0;
    const double t = (double)waves * (mma > epi ? mma : epi) + epi;
    if (t < best_t * 0.99) {
      best_t = t;
      best = bn;
    }
  }
  return best;
}

// Units of a reduction: uk K-tiles each, and ux more where a unit's last group runs past them (a K-tile
// starts inside a group where a tap's channels are no multiple of G: 3x3 over 72 channels at G = 32).  Every
// group is summed in one unit: its halves in two would carry two roundings and two scales of its alpha,
// as large as the halves themselves where these cancel.  Four K-tiles where that fits, else the number
// up to eight that takes the fewest K-tiles in all; false where none fits.
bool plan_units(const Geom& g, int kpt, int ktiles, int& uk, int& ux) {
  int best = INT32_MAX;
  for (int n = TF_UNIT; n <= TF_MAX_UNIT; ++n) {
    if (n != TF_UNIT && n * TF_KT / g.G + 1 >= PF_GPU) break;
    int x = 0, tiles = 0;
    for (int kt = n; g.Cg % g.G != 0 && kt < ktiles; kt += n) {
      int rem = (g.G - (kt / kpt * g.Cg + kt % kpt * TF_KT) % g.G) % g.G, t = 0;
      for (; rem > 0 && kt + t < ktiles; ++t) {
        const int c = g.Cg - (kt + t) % kpt * TF_KT;
        rem -= c < TF_KT ? c : TF_KT;
      }
      if (t > x) x = t;
    }
    if (n + x > TF_MAX_UNIT) continue;
    for (int kt = 0; kt < ktiles; kt += n) tiles += ktiles - kt < n + x ? ktiles - kt : n + x;
    if (tiles < best) {
      best = tiles;
      uk = n;
      ux = x;
    }
    if (x == 0) break;  // (a larger unit takes no fewer K-tiles)
  }
  return best < INT32_MAX;
}

int fold_ktiles_per_tap(const Geom& g) { return (g.Cg + TF_KT - 1) / TF_KT; }

}  // namespace

bool fold_supports(const Geom& g) {
  if (g.G < 4 || g.G > 64 || (g.G & (g.G - 1)) != 0) return false;
  int uk, ux;
  const int kpt = fold_ktiles_per_tap(g);
  if (!plan_units(g, kpt, g.R * g.S * kpt, uk, ux)) return false;
  if (g.P >= (int64_t)1 << 31) return false;  // positions decoded in 32 bits
  if (tc::encode_tiled() == nullptr) return false;
  return tc::act_pointwise(g) || (tc::encode_im2col() != nullptr && tc::im2col_fits(g.R, g.S, g.stride, g.pad));
}

fgq_status launch_fold_contract(const void* act, const Geom& g, const uint32_t* codes, const float* alpha,
                                const float* act_scale, float* out, unsigned int* err, cudaStream_t s,
                                bool& no_scratch) {
  if (!fold_supports(g)) return FGQ_ERR_UNSUPPORTED;
  FoldArgs a;
  memset(&a, 0, sizeof a);
  a.act_scale = act_scale;
  a.out = out;
  a.err = err;
  a.g = g;
  a.cpad = fold_ktiles_per_tap(g) * TF_KT;
  a.ktiles = g.R * g.S * (a.cpad / TF_KT);
  if (!plan_units(g, a.cpad / TF_KT, a.ktiles, a.uk, a.ux)) return FGQ_ERR_UNSUPPORTED;
  a.nunits = (a.ktiles + a.uk - 1) / a.uk;
  a.mtiles = (g.Mg + TF_FM - 1) / TF_FM;
  const int wtiles = g.groups * a.mtiles;
  const int sms = device_sms();
  a.bn = choose_bn(g.P, wtiles, a.ktiles, sms);
  const int stage = TF_A + a.bn * TF_KT * 2;
  a.obufs = a.ktiles <= TF_SHORT ? 4 : 2;
  a.nst = (TF_RING + TF_OUT - TF_EPI_WARPS * a.obufs * TF_BOX) / stage;
  if (a.nst > TF_MAX_NST) a.nst = TF_MAX_NST;
  const int64_t ntiles = (int64_t)wtiles * ((g.P + a.bn - 1) / a.bn);
  if (ntiles > INT32_MAX) return FGQ_ERR_UNSUPPORTED;
  a.ntiles = (int)ntiles;
  // a test may shorten the waits (debug_wait_limit_us), never the final drains
  const int64_t lim_us = debug_wait_limit_us();
  a.timeout_ns = lim_us < 0 ? TF_TIMEOUT_NS : (uint64_t)lim_us * 1000u;

  // one temporary from the stream-ordered pool: weight images, second pairs, row scales, marks,
  // fp16 activations
  const bool pointwise = tc::act_pointwise(g);
  const int64_t npix = pointwise && g.stride > 1 ? g.P : (int64_t)g.B * g.H * g.W;
  const int64_t ca = (int64_t)g.groups * a.cpad;
  const size_t a_bytes = (size_t)wtiles * a.nunits * (a.uk + a.ux) * TF_A;
  const size_t rs_bytes = ((size_t)wtiles * a.nunits * TF_FM * 4 + 255) / 256 * 256;
  const size_t ext_bytes = ((size_t)wtiles * a.nunits + 255) / 256 * 256;
  const size_t x_bytes = (size_t)npix * ca * 2;
  void* tmp = scratch_alloc(2 * a_bytes + rs_bytes + ext_bytes + x_bytes, s);
  no_scratch = !tmp;
  if (!tmp) return FGQ_ERR_CUDA;
  uint8_t* base = static_cast<uint8_t*>(tmp);
  PrepFold f;
  memset(&f, 0, sizeof f);
  f.codes = codes;
  f.alpha = alpha;
  f.a_op = base;
  f.a_ext = base + a_bytes;
  f.rs = reinterpret_cast<float*>(base + 2 * a_bytes);
  f.ext = base + 2 * a_bytes + rs_bytes;
  uint8_t* x16 = base + 2 * a_bytes + rs_bytes + ext_bytes;
  f.wrow = g.wrow;
  f.ng = g.ng;
  f.gshift = 31 - __builtin_clz((unsigned)g.G);
  f.dbits = g.G > 32 ? TF_DIGIT - 1 : TF_DIGIT;
  f.fbits = in_slices(g) ? TF_FRAC : 0;
  a.lo_scale = 1.0f / (float)(1 << f.dbits);
  a.ext_scale = a.lo_scale * a.lo_scale;
  f.Mg = g.Mg;
  f.Cg = g.Cg;
  f.cpad = a.cpad;
  f.mtiles = a.mtiles;
  f.ktiles = a.ktiles;
  f.nunits = a.nunits;
  f.uk = a.uk;
  f.ux = a.ux;
  f.nsub = wtiles * a.nunits >= 2 * sms ? 1 : TF_UNIT;
  f.tol = pair_tolerance(g, a.nunits);
  f.quads = g.Cg % 4 == 0 ? 1 : 0;
  f.padded = (a.cpad != g.Cg || g.C % 16 != 0) ? 1 : 0;
  f.fast8 = f.padded && g.Cg % 8 == 0 && g.C % 8 == 0 && (g.act_type == FGQ_U8 || g.act_type == FGQ_S8) ? 1 : 0;
  f.sC = g.C;
  f.sgroups = g.groups;
  f.npix = npix;
  f.fold_blocks = wtiles * a.nunits * f.nsub;
  const prep::ActSrc src = prep::act_src(act, g);
  const int xb = prep::blocks_for(f.padded ? npix * ca / 8 : src.nchunks);
  fgq_status st = after_launch(launch_pdl(prep_fold_kernel, dim3(f.fold_blocks + xb), dim3(256), 0, s, f, src,
                                          reinterpret_cast<uint4*>(x16)));
  a.a_op = f.a_op;
  a.a_ext = f.a_ext;
  a.rs = f.rs;
  a.ext = f.ext;
  if (st == FGQ_OK) {
    const bool map_ok =
        pointwise ? make_map_2d(&a.act_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, x16, (uint64_t)ca, (uint64_t)npix,
                                (uint64_t)ca * 2, TF_KT, (uint32_t)a.bn, CU_TENSOR_MAP_SWIZZLE_128B)
                  : make_map_im2col(&a.act_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, x16, (uint64_t)ca, 2, g.B, g.H, g.W,
                                    g.R, g.S, g.stride, g.pad, TF_KT, (uint32_t)a.bn, CU_TENSOR_MAP_SWIZZLE_128B);
    if (!map_ok) st = FGQ_ERR_CUDA;
  }
  // output boxes by TMA store: 16-byte row pitch, and no box that reaches into another conv group
  if (st == FGQ_OK && (g.groups == 1 || g.Mg % 16 == 0)) {
    if (g.rq_out)
      a.out_tma = g.M % 16 == 0 && (reinterpret_cast<uintptr_t>(g.rq_out) & 15) == 0 &&
                  make_map_2d(&a.out_map, CU_TENSOR_MAP_DATA_TYPE_UINT8, g.rq_out, (uint64_t)g.M, (uint64_t)g.P,
                              (uint64_t)g.M, 16, TF_BOX_POS, CU_TENSOR_MAP_SWIZZLE_NONE);
    else
      a.out_tma = g.M % 4 == 0 && make_map_2d(&a.out_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, out, (uint64_t)g.M,
                                              (uint64_t)g.P, (uint64_t)g.M * 4, 16, TF_BOX_POS,
                                              CU_TENSOR_MAP_SWIZZLE_NONE);
  }
  if (st == FGQ_OK) {
    const int grid = a.ntiles < sms ? a.ntiles : sms;
    if (g.rq_out) st = pointwise ? launch_fold<true, true>(a, grid, s) : launch_fold<false, true>(a, grid, s);
    else st = pointwise ? launch_fold<true, false>(a, grid, s) : launch_fold<false, false>(a, grid, s);
  }
  // the temporary returns to the pool once the work queued on s before this point is done
  if (cudaFreeAsync(tmp, s) != cudaSuccess && st == FGQ_OK) st = FGQ_ERR_CUDA;
  return st;
}

}  // namespace fgq
