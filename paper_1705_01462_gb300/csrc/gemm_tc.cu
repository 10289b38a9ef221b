// Tensor-core (tcgen05) grouped ternary contraction for G in {64, 128}, and the
// bounded-wait self test.
//
// Math (Eq. 2 with the 32-bit group accumulators of Section 4): per output filter m,
// position p and group g of G consecutive reduction elements, s[m][g][p] is an exact
// integer; y[p][m] = s_x * sum_g alpha[m][g] * s[m][g][p].  sm_103a has no integer
// tcgen05 MMA, so the group sums run as fp16 MMAs on exact integers: codes {-1, 0, +1}
// and 8-bit (or 4-bit) activations are exact in fp16, products are exact, and a group's
// fp32 accumulation stays an exact integer (|s| <= 128 * 255 < 2^24).  The K-tile of the
// MMA chain is 64 and aligned to the group, so after a group's MMAs the TMEM accumulator
// holds exactly s[m][g][p] for a 128-filter x up-to-256-position tile; the epilogue multiplies
// it by alpha[m][g] and adds it into an fp32 register accumulator (one multiply per group,
// Section 4.1).  Two or more TMEM buffers let the MMAs of the next groups run while group g
// drains.  The group-sums variant (SUMS) stores each drained accumulator as the int32
// s[m][g][p] instead (the exact integers themselves, for verification).
//
// Both operands reach shared memory by TMA, already as MMA operands: the codes are expanded
// to {0, +1, -1} and the activations to their integer values once per call (stream-ordered
// temporaries written by one launch, prep64_kernel), fp16 for 8-bit activations and e4m3
// (kind::f8f6f4) for 4-bit ones, so every K-tile is two box loads into one ring stage and
// no thread converts operands inside the contraction.  An activation is read by R * S filter
// taps and M / 128 filter tiles; converting it once instead of at every use takes the
// conversion off the MMA's path.
//
// Warp roles (384 threads, one CTA per SM, persistent over tiles):
//   warps 0-7  epilogue: warp w reads TMEM lanes 32*(w%4).. (filter rows) and the positions of half
//              w/4 of the drained buffer in 32-column tcgen05.ld, adds alpha * s into 128 fp32
//              registers and frees the buffer.  At tile end it stores boxes of 16 positions x 32
//              filters through its own buffers by TMA (or directly), requantized when asked.
//              The drain bounds this kernel: about 1040 clk per group of 256 positions against 512 of
//              MMAs.  Its registers come from a setmaxnreg split.
//   warps 8, 9 the MMA issuers (warp 8 also allocates TMEM), the groups in turn into the 512 / bn
//              accumulators in turn: 4 tcgen05.mma (M = 128, K = 16) per K-tile, a commit per K-tile
//              that frees its stage and one per group; while one waits for its accumulator, the
//              other's MMAs keep the tensor pipe busy.  Each waits for every
//              K-tile's operands, its own or not, and a stage is refilled only when both have:
//              no wait is ever more than one phase behind its barrier.
//   warp 10    the producer: per K-tile, the ternary box (64 reduction elements x 128 filters) and
//              the activation box (64 channels x the tile's positions) into one ring stage: a 2D
//              box of consecutive input rows when the im2col rows are input rows (1x1 stride-1
//              convolutions, GEMMs), otherwise an im2col box (the output positions' pixels at the
//              K-tile's filter tap, zeros in the padding).
// The loops of warps 8-10 are warp-uniform and an elected lane issues (from a single divergent
// lane each TMA or MMA instruction took about 100 clk).
// Every mbarrier wait is bounded in time; on expiry the kernel records FGQ_ERR_TIMEOUT, each role
// leaves its loop (uniformly within the epilogue, which uses named barriers), in-flight
// copies and MMAs are waited for, and TMEM is freed.
#include <cstdint>
#include <cstring>

#include "operand_prep.cuh"
#include "tc_common.cuh"

namespace fgq {
namespace {

using tc::encode_im2col;
using tc::encode_tiled;
using tc::im2col_fits;
using tc::make_map_2d;
using tc::make_map_im2col;

constexpr int TC_BM = 128;        // filters per tile (MMA M, TMEM lanes)
constexpr int TC_MAX_BN = 256;    // positions per tile (MMA N), a multiple of 64
constexpr int TC_KT = 64;         // reduction elements per K-tile
constexpr int TC_TMEM_COLS = 512; // all of TMEM: 512 / bn accumulator buffers, 2 to TC_MAX_NACC
constexpr int TC_MAX_NACC = 8;
constexpr int TC_ISSUERS = 2;
constexpr int TC_EPI_WARPS = 8;
constexpr int TC_MMA_WARP = TC_EPI_WARPS;       // warps 8 and 9: MMA issuers of even and odd groups
constexpr int TC_PROD_WARP = TC_EPI_WARPS + 2;  // warp 10 streams both operands; warp 11 idles
constexpr int TC_THREADS = 384;                 // three warpgroups of 168 registers a thread at launch, split
constexpr int TC_EPI_REGS = 224;                // into 224 for the epilogue's two
constexpr int TC_CTL_REGS = 56;                 // and 56 for warps 8-11
static_assert(256 * TC_EPI_REGS + 128 * TC_CTL_REGS <= TC_THREADS * 168, "register split");
constexpr int TC_EPI_COLS = TC_MAX_BN / 2;         // positions per epilogue thread, at most
constexpr uint64_t TC_TIMEOUT_NS = 1000000000ull;  // 1 s per wait
constexpr uint32_t TC_DRAIN_LIMIT = 1u << 20;      // polls of the final drains (never shortened)
constexpr uint32_t BAR_EPI = 2;                    // named barrier of the epilogue threads

constexpr int OUT_POS = 16;                      // positions per output box
constexpr int OUT_BOX = OUT_POS * 32 * 4;        // 2 KB: fp32 [16 positions][32 filters]
constexpr int TC_MAX_NST = 8;                    // operand ring depth, at most (as many stages as fit)
constexpr int TC_RING = 196608;                  // 4 stages of fp16 operands at bn = 256, 8 of e4m3
// Output boxes per epilogue warp behind the ring, twice as many for tiles of few K-tiles.
constexpr int TC_OBUFS = 2;
constexpr int TC_OUT = TC_OBUFS * TC_EPI_WARPS * OUT_BOX;
constexpr int TC_SHORT = 4;
constexpr int TC_SMEM = 1024 + TC_RING + TC_OUT + 8 * (2 * TC_MAX_NST + 2 * TC_MAX_NACC + 1) + 16;
static_assert(TC_SMEM <= 232448, "shared memory budget");

// Operand plan of a variant.  fp16 operands (8-bit activations): 128-byte rows of 64
// elements, 128-byte swizzle, 4 MMAs of K = 16 per K-tile.  e4m3 operands (4-bit
// activations, F8): every 4-bit value and every code is exact in e4m3, so the K-tile is
// 64-byte rows with the 64-byte swizzle and 2 MMAs of K = 32 (kind::f8f6f4) -- half the bytes
// per K-tile in HBM, L2 and shared memory, twice the ring depth.
template <bool F8>
struct TcCfg {
  static constexpr int ES = F8 ? 1 : 2;              // bytes per operand element
  static constexpr int A_TILE = TC_BM * TC_KT * ES;  // ternary operand; the activations take bn * 64 * ES
};

struct TcArgs {
  CUtensorMap a16_map;    // expanded codes [M][Kp] (fp16, or e4m3 for F8), box {64, 128 rows}
  CUtensorMap act_map;    // expanded activations: act_tma: 2D [positions][C], box {64, bn rows}; otherwise
                          // the im2col map of the NHWC tensor, bn pixels x 64 channels
  CUtensorMap out_map;    // outputs [P][M] (fp32 or codes), box {32 filters, 16 positions}; if out_tma
  const float* alpha_t;   // alphas transposed, [ng][M]: a warp's 32 filters read one line per group
  const float* act_scale;
  float* out;
  int32_t* sums;    // SUMS: int32 group sums [M][ng][P]
  unsigned int* err;
  Geom g;
  int mtiles;       // filter tiles per conv group
  int ntiles;       // work items: groups * mtiles * ptiles tiles, each split into ksplit group ranges
  int ktiles;       // K-tiles of a whole tile (= ng * G / 64)
  int ksplit;       // group ranges per tile (1: whole tiles; > 1: partial sums added into the output)
  int gpk;          // groups per range
  int kt_per_group; // G / 64
  int act_tma;      // 2D activation map (one row per output position); else im2col map
  int out_tma;      // output boxes by TMA store
  int bn, nst;      // positions per tile, ring depth
  int nacc;         // TMEM accumulator buffers of bn columns
  int obufs;        // output boxes per epilogue warp: 2 or 4
  uint64_t timeout_ns;
};

// Work item w: tile w / ksplit, groups [g0, g1) of range w % ksplit.  Tiles are numbered
// with the filter tiles of one position tile consecutive, so that CTAs running at the same
// time share activation boxes in L2.
__device__ __forceinline__ void item_coords(const TcArgs& a, int w, int& gi, int& m0, int64_t& p0, int& g0, int& g1) {
  const int tile = w / a.ksplit;
  const int ks = w - tile * a.ksplit;
  const int per_p = a.g.groups * a.mtiles;
  const int pt = tile / per_p;
  const int r = tile - pt * per_p;
  gi = r / a.mtiles;
  const int mt = r - gi * a.mtiles;
  m0 = gi * a.g.Mg + mt * TC_BM;
  p0 = (int64_t)pt * a.bn;
  g0 = ks * a.gpk;
  g1 = g0 + a.gpk < a.g.ng ? g0 + a.gpk : a.g.ng;
}

// One launch prepares both operands of a call: blocks [0, code_blocks) expand the ternary codes
// (one 16-code word per thread and step) and transpose the alphas ([M][ng] -> [ng][M]: read by rows
// in the epilogue, a group's alphas of 32 filters took 32 cache lines per warp and bounded the
// kernel), the others the activations (16 elements per thread and step); fp16 operands, or
// e4m3 for 4-bit activations (F8).
template <bool F8>
__global__ void __launch_bounds__(256) prep64_kernel(const uint32_t* __restrict__ codes, int64_t nwords,
                                                     uint4* __restrict__ a_op, const float* __restrict__ alpha, int M,
                                                     int ng, float* __restrict__ alpha_t, const prep::ActSrc src,
                                                     uint4* __restrict__ x_op, int code_blocks) {
  pdl_wait();
  pdl_trigger();
  if ((int)blockIdx.x < code_blocks) {
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)code_blocks * blockDim.x;
    for (int64_t i = first; i < nwords; i += step) {
      if (F8) prep::codes_e4m3(codes, i, a_op);
      else prep::codes_f16(codes, i, a_op);
    }
    if (alpha) {
      for (int64_t i = first; i < (int64_t)M * ng; i += step) {
        const int64_t gr = i / M;
        alpha_t[i] = __ldg(alpha + (i - gr * M) * ng + gr);
      }
    }
  } else {
    const int64_t nb = (int64_t)gridDim.x - code_blocks;
    prep::act_expand<F8>(src, ((int64_t)blockIdx.x - code_blocks) * blockDim.x + threadIdx.x, nb * blockDim.x, x_op);
  }
}

// TMAP: the layer's im2col rows are contiguous input rows (2D box loads); otherwise the
// activation boxes come from an im2col map (one load per K-tile: the tile's output positions at
// one filter tap and 64 channels, padding read as zeros).  OUT: 0 fp32, 1 requantized codes, 2
// int32 group sums (kernels of their own, so that each epilogue's unrolled code stays short).
template <bool TMAP, int OUT, bool F8>
__global__ void __launch_bounds__(TC_THREADS, 1) tc_contract_kernel(const __grid_constant__ TcArgs a) {
  constexpr int ES = TcCfg<F8>::ES;
  constexpr int A_TILE = TcCfg<F8>::A_TILE;
  constexpr bool SUMS = OUT == 2, RQ = OUT == 1;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* obox = smem + TC_RING + TC_OUT - TC_EPI_WARPS * a.obufs * OUT_BOX;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + TC_RING + TC_OUT);  // stage loaded (both boxes' bytes)
  uint64_t* empty = full + TC_MAX_NST;                                    // stage free (its MMAs are complete)
  uint64_t* acc_full = empty + TC_MAX_NST;
  uint64_t* acc_empty = acc_full + TC_MAX_NACC;
  uint64_t* drain_bar = acc_empty + TC_MAX_NACC;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // warp-uniform
  const int lane = threadIdx.x & 31;
  const Geom& g = a.g;
  const uint64_t tmo = a.timeout_ns;
  const int nst = a.nst, nacc = a.nacc;
  const uint32_t stage = (uint32_t)(A_TILE + a.bn * TC_KT * ES);

  if (threadIdx.x == 0) {
    for (int i = 0; i < nst; ++i) {
      mbar_init(&full[i], 1);   // the producer's expect_tx, then the two boxes' bytes
      mbar_init(&empty[i], 2);  // the commit after the K-tile's MMAs, and the other issuer's arrival
    }
    for (int i = 0; i < nacc; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], TC_EPI_WARPS);  // one arrival per epilogue warp
    }
    mbar_init(drain_bar, TC_ISSUERS);  // one commit per MMA issuer
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == TC_MMA_WARP) {
    tmem_alloc(tmem_slot, TC_TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // the prologue above overlapped the previous kernel; global memory only from here on
  pdl_wait();
  pdl_trigger();
  const int my_tiles = (a.ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;

  auto fail = [&]() {
    *abort_flag = 1;
    record_error(a.err, FGQ_ERR_TIMEOUT);
  };

  if (warp >= TC_EPI_WARPS) {
    setmaxnreg_dec<TC_CTL_REGS>();
    if (warp == TC_PROD_WARP) {
      // ---------------------------------------------------------------- producer
      const uint32_t sbase = smem_u32(smem);
      const int kpt = g.Cg / TC_KT;  // K-tiles per filter tap
      int issued = 0;                // K-tiles issued by this CTA
      int s = 0;
      uint32_t ph = 1;  // parity of the stage's previous release; the first round passes at once
      bool ok = true;
      for (int tl = 0; tl < my_tiles && ok; ++tl) {
        int gi, m0, g0, g1;
        int64_t p0;
        item_coords(a, (int)blockIdx.x + tl * (int)gridDim.x, gi, m0, p0, g0, g1);
        int n0 = 0, h0 = 0, w0 = 0;  // im2col: the tile's first window origin (input pixel coordinates)
        if (!TMAP) {
          const int pp = (int)p0;  // < P < 2^31
          const int wo = pp % g.Wo;
          const int q = pp / g.Wo;
          n0 = q / g.Ho;
          h0 = (q - n0 * g.Ho) * g.stride - g.pad;
          w0 = wo * g.stride - g.pad;
        }
        // the range's first K-tile and its filter tap (tr, ts) and channel offset tc0, which
        // then advance incrementally
        const int kt0 = g0 * a.kt_per_group, kt1 = g1 * a.kt_per_group;
        int tc0 = (kt0 % kpt) * TC_KT, ts = (kt0 / kpt) % g.S, tr = (kt0 / kpt) / g.S;
        const int cb = gi * g.Cg;  // a multiple of 64 (128-byte aligned in fp16)
        for (int kt = kt0; kt < kt1; ++kt) {
          if (!mbar_wait_warp(&empty[s], ph, tmo, abort_flag)) {
            ok = false;
            break;
          }
          if (elect_one()) {
            const uint32_t sa = sbase + (uint32_t)s * stage;
            mbar_arrive_expect_tx(&full[s], stage);
            tma_load_2d(sa, &a.a16_map, kt * TC_KT, m0, &full[s]);
            if (TMAP)
              tma_load_2d(sa + A_TILE, &a.act_map, cb + tc0, (int)p0, &full[s]);
            else
              tma_load_im2col_4d(sa + A_TILE, &a.act_map, cb + tc0, w0, h0, n0, (uint16_t)ts, (uint16_t)tr, &full[s]);
          }
          __syncwarp();
          ++issued;
          if (++s == nst) {
            s = 0;
            ph ^= 1u;
          }
          tc0 += TC_KT;
          if (tc0 == g.Cg) {
            tc0 = 0;
            if (++ts == g.S) {
              ts = 0;
              ++tr;
            }
          }
        }
      }
      if (!ok && !*abort_flag) fail();
      // loads the MMA issuers may not have consumed: the last nst issued, one per stage, each the
      // latest phase of its stage's barrier; none may outlive the CTA
      for (int j = issued - nst < 0 ? 0 : issued - nst; j < issued; ++j)
        mbar_wait_bounded(&full[j % nst], (j / nst) & 1, TC_DRAIN_LIMIT);
    } else if (warp == TC_MMA_WARP || warp == TC_MMA_WARP + 1) {
      // ---------------------------------------------------------------- MMA issuers
      const int b = warp - TC_MMA_WARP;  // parity of the groups this warp issues
      const uint32_t idesc = idesc_f16_f32(TC_BM, a.bn);
      const uint64_t ad0 = F8 ? sdesc_k_sw64(smem_u32(smem)) : sdesc_k_sw128(smem_u32(smem));
      const uint64_t bd0 = F8 ? sdesc_k_sw64(smem_u32(smem) + A_TILE) : sdesc_k_sw128(smem_u32(smem) + A_TILE);
      int s = 0, gc = 0, ab = 0;  // ring position, group count, accumulator of group gc
      uint32_t ph = 0, aph = 1;
      bool ok = true;
      for (int tl = 0; tl < my_tiles && ok; ++tl) {
        int gi_, m0_, g0, g1;
        int64_t p0_;
        item_coords(a, (int)blockIdx.x + tl * (int)gridDim.x, gi_, m0_, p0_, g0, g1);
        for (int grp = g0; grp < g1 && ok; ++grp, ++gc) {
          const bool mine = (gc & 1) == b;
          if (mine && !mbar_wait_warp(&acc_empty[ab], aph, tmo, abort_flag)) {
            ok = false;
            break;
          }
          const uint32_t d = tmem + (uint32_t)(ab * a.bn);
          for (int sub = 0; sub < a.kt_per_group; ++sub) {
            if (!mbar_wait_warp(&full[s], ph, tmo, abort_flag)) {
              ok = false;
              break;
            }
            if (mine) {
              tc_fence_after();
              if (elect_one()) {
                const uint64_t off = (uint64_t)(((uint32_t)s * stage) >> 4);
                if constexpr (F8) {
#pragma unroll
                  for (int k = 0; k < TC_KT / 32; ++k)  // advance 32 e4m3 (32 bytes) along K
                    mma_e4m3(d, ad0 + off + 2 * k, bd0 + off + 2 * k, idesc, (sub | k) != 0 ? 1u : 0u);
                } else {
#pragma unroll
                  for (int k = 0; k < TC_KT / 16; ++k)  // advance 16 fp16 (32 bytes) along K
                    mma_f16(d, ad0 + off + 2 * k, bd0 + off + 2 * k, idesc, (sub | k) != 0 ? 1u : 0u);
                }
                mma_commit(&empty[s]);
                if (sub == a.kt_per_group - 1) mma_commit(&acc_full[ab]);
              }
            } else if (elect_one()) {
              mbar_arrive(&empty[s]);
            }
            __syncwarp();
            if (++s == nst) {
              s = 0;
              ph ^= 1u;
            }
          }
          if (++ab == nacc) {
            ab = 0;
            aph ^= 1u;
          }
        }
      }
      if (!ok && !*abort_flag) fail();
      // all MMAs issued by both warps are complete once the drain barrier flips
      if (elect_one()) mma_commit(drain_bar);
      __syncwarp();
      mbar_wait_bounded(drain_bar, 0, TC_DRAIN_LIMIT);
    }
  } else {
    setmaxnreg_inc<TC_EPI_REGS>();
    // ---------------------------------------------------------------- epilogue
    // At tile end the finished sums go back into the buffer just drained and a rolled loop stores
    // them: each CTA runs the tile end a few times only, so its code is fetched cold -- about 6 us
    // of a call for 13 KB of unrolled stores (3x3 256 -> 256 on 14 x 14, batch 128).
    const int quarter = warp & 3, part = warp >> 2;
    const int t = 32 * quarter + lane;  // TMEM lane = filter row of the tile
    const int hcols = a.bn / 2;  // positions of this warp (a multiple of 32)
    const uint32_t tbase = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(hcols * part);
    const float sx = SUMS ? 0.0f : __ldg(a.act_scale);
    const uint32_t bar_full = smem_u32(acc_full), bar_empty = smem_u32(acc_empty);
    int b = 0, obuf = 0;
    uint32_t fph = 0;
    bool ok = true;
    for (int tl = 0; tl < my_tiles; ++tl) {
      int gi, m0, g0, g1;
      int64_t p0;
      item_coords(a, (int)blockIdx.x + tl * (int)gridDim.x, gi, m0, p0, g0, g1);
      const int m = m0 + t;
      const int mend = gi * g.Mg + g.Mg;  // the conv group's filters end here
      const bool mok = m < mend;
      const int64_t pbase = p0 + hcols * part;
      const float* acol = SUMS ? nullptr : a.alpha_t + (int64_t)g0 * g.M + (mok ? m : 0);
      float acc[TC_EPI_COLS];
      if (!SUMS) {
#pragma unroll
        for (int j = 0; j < TC_EPI_COLS; ++j) acc[j] = 0.0f;
      }
      float al_next = SUMS ? 0.0f : __ldg(acol);  // (filters past M: sums that nobody stores)
      uint32_t ta = tbase;
      for (int grp = g0; grp < g1; ++grp) {
        const float al = al_next;  // alpha of this group, loaded one group ahead
        if (!SUMS && grp + 1 < g1) al_next = __ldg(acol += g.M);
        if (!mbar_wait_warp(bar_full + 8u * (uint32_t)b, fph, tmo, abort_flag)) {
          ok = false;  // leave with the others below
          break;
        }
        tc_fence_after();
        ta = tbase + (uint32_t)(b * a.bn);
        if (SUMS) {
          // the exact group sums of positions pbase + j, filter m: s[m][grp][p]
          int32_t* srow = a.sums + ((int64_t)(mok ? m : 0) * g.ng + grp) * g.P;
#pragma unroll 1
          for (int c = 0; 16 * c < hcols; ++c) {
            uint32_t r16[16];
            tmem_ld16(ta + 16 * c, r16);
            tmem_ld_wait_regs16(r16);
            if (mok) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const int64_t p = pbase + 16 * c + j;
                if (p < g.P) srow[p] = __float2int_rn(__uint_as_float(r16[j]));
              }
            }
          }
        } else {
#pragma unroll
          for (int c = 0; c < TC_EPI_COLS / 32; ++c) {
            if (32 * c < hcols) {
              uint32_t r[32];
              tmem_ld32(ta + 32 * c, r);
              tmem_ld_wait_regs(r);
#pragma unroll
              for (int j = 0; j < 32; j += 2)
                ffma2(acc[32 * c + j], acc[32 * c + j + 1], __uint_as_float(r[j]), __uint_as_float(r[j + 1]), al);
            }
          }
        }
        if (SUMS || grp + 1 < g1) {  // the tile's last buffer is freed after the stores
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_empty + 8u * (uint32_t)b);  // the buffer is free once the values are in registers
          if (++b == nacc) {
            b = 0;
            fph ^= 1u;
          }
        }
      }
      if (!ok && !*abort_flag) fail();
      if (named_bar_or(BAR_EPI, 32 * TC_EPI_WARPS, !ok)) break;  // leave together
      if (SUMS) continue;  // the group sums are stored already
#pragma unroll
      for (int c = 0; c < TC_EPI_COLS / 16; ++c)
        if (16 * c < hcols) tmem_st16(ta + 16 * c, acc + 16 * c);
      tmem_st_wait();
      RqMul rq;
      if (RQ) rq = rq_mul(g.rq_scale, g.rq_signed);
      const bool wok = m0 + 32 * quarter < mend;  // some of the warp's filters exist
      uint8_t* const ob0 = obox + a.obufs * warp * OUT_BOX;
#pragma unroll 1
      for (int c = 0; 16 * c < hcols; ++c) {
        uint32_t v[16];
        tmem_ld16(ta + 16 * c, v);
        tmem_ld_wait_regs16(v);
        if (a.out_tma) {
          // a box of 16 positions x 32 filters through the warp's own buffers; positions past P and
          // filters past M are clipped by the tensor map
          if (lane == 0) {  // the buffer's previous box has been read out
            if (a.obufs == TC_OBUFS) bulk_wait_read<TC_OBUFS - 1>();
            else bulk_wait_read<2 * TC_OBUFS - 1>();
          }
          __syncwarp();
          uint8_t* ob = ob0 + obuf * OUT_BOX;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float y = sx * __uint_as_float(v[j]);
            if (RQ) ob[32 * j + lane] = rq_code(y, rq);  // fused requantization: 8-bit codes
            else reinterpret_cast<float*>(ob)[32 * j + lane] = y;
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            const int pb = (int)pbase + 16 * c;
            if (wok && pb < g.P) {
              if (!RQ && a.ksplit > 1)  // a group range's partial sums: added into the (zeroed) output
                tma_reduce_add_2d(&a.out_map, m, pb, smem_u32(ob));
              else
                tma_store_2d(&a.out_map, m, pb, smem_u32(ob));
            }
            bulk_commit();
          }
          if (++obuf == a.obufs) obuf = 0;
        } else if (mok) {
          // the warp's 32 lanes are 32 consecutive filters
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int64_t p = pbase + 16 * c + j;
            if (p < g.P) {
              const float y = sx * __uint_as_float(v[j]);
              if (RQ) g.rq_out[p * g.M + m] = rq_code(y, rq);
              else if (a.ksplit > 1) atomicAdd(a.out + p * g.M + m, y);
              else a.out[p * g.M + m] = y;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_empty + 8u * (uint32_t)b);
      if (++b == nacc) {
        b = 0;
        fph ^= 1u;
      }
    }
    if (lane == 0) bulk_wait_all();  // this thread's TMA stores are complete
  }

  tc_fence_before();
  __syncthreads();
  if (warp == TC_MMA_WARP) {
    tc_fence_after();
    tmem_dealloc(tmem, TC_TMEM_COLS);
  }
}

template <bool TMAP, int OUT, bool F8>
fgq_status launch_tc(const TcArgs& args, int grid, cudaStream_t s) {
  if (!tc::smem_attr_once<tc_contract_kernel<TMAP, OUT, F8>>(TC_SMEM)) return FGQ_ERR_CUDA;
  return after_launch(launch_pdl(tc_contract_kernel<TMAP, OUT, F8>, dim3(grid), dim3(TC_THREADS), TC_SMEM, s, args));
}

template <bool F8>
fgq_status launch_tc_variant(const TcArgs& a, int grid, cudaStream_t s) {
  if (a.sums) return a.act_tma ? launch_tc<true, 2, F8>(a, grid, s) : launch_tc<false, 2, F8>(a, grid, s);
  if (a.g.rq_out) return a.act_tma ? launch_tc<true, 1, F8>(a, grid, s) : launch_tc<false, 1, F8>(a, grid, s);
  return a.act_tma ? launch_tc<true, 0, F8>(a, grid, s) : launch_tc<false, 0, F8>(a, grid, s);
}

// One block waits on an mbarrier that nothing arrives on; every wait is bounded, so the
// kernel always returns and records FGQ_ERR_TIMEOUT.
__global__ void wait_timeout_selftest_kernel(uint32_t max_iter, unsigned int* err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  const bool ok = mbar_wait_bounded(&bar, 0, max_iter);
  if (!ok && threadIdx.x == 0) record_error(err, FGQ_ERR_TIMEOUT);
}

// One warp waits on one barrier for two phases at once: the even lanes' phase is complete, the odd
// lanes' never will be.  A wait that the lanes decide together expires for all of them.
__global__ void wait_warp_selftest_kernel(uint64_t limit_ns, unsigned int* err) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  const bool ok = mbar_wait_warp(&bar, (threadIdx.x & 1) ^ 1, limit_ns, &abort_flag);
  const uint32_t passed = __ballot_sync(0xffffffffu, ok);
  if (threadIdx.x == 0) record_error(err, passed == 0 ? FGQ_ERR_TIMEOUT : FGQ_ERR_UNSUPPORTED);
}

}  // namespace

namespace tc {

bool act_pointwise(const Geom& g) { return g.R == 1 && g.S == 1 && g.pad == 0; }

int64_t act16_elems(const Geom& g) {
  return act_pointwise(g) && g.stride > 1 ? g.P * g.C : (int64_t)g.B * g.H * g.W * g.C;
}

bool act16_map(CUtensorMap* m, const void* x16, const Geom& g, uint32_t pixels) {
  if (act_pointwise(g))
    return make_map_2d(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, x16, (uint64_t)g.C, (uint64_t)(act16_elems(g) / g.C),
                       (uint64_t)g.C * 2, 64, pixels, CU_TENSOR_MAP_SWIZZLE_128B);
  return make_map_im2col(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, x16, (uint64_t)g.C, 2, g.B, g.H, g.W, g.R, g.S, g.stride,
                         g.pad, 64, pixels, CU_TENSOR_MAP_SWIZZLE_128B);
}

bool act16_supported(const Geom& g) {
  if (g.C % 16 != 0 || g.Cg % 64 != 0) return false;
  if (encode_tiled() == nullptr) return false;
  return act_pointwise(g) || (encode_im2col() != nullptr && im2col_fits(g.R, g.S, g.stride, g.pad));
}

}  // namespace tc

using tc::act_pointwise;

bool tc_supports(const Geom& g) {
  if (g.G != 64 && g.G != 128) return false;
  if (g.P >= (int64_t)1 << 31) return false;  // positions decoded in 32 bits
  // every K-tile inside one filter tap (conv) or row (GEMM); 16-element expansion chunks;
  // activation boxes by 2D or im2col maps
  return tc::act16_supported(g);
}

namespace {

// Positions per tile and group ranges per tile, by estimated time in clk.  A group costs its drain
// about 700 + 1.3 bn (measured: 128 positions 870, 192 960, 256 1040; the instructions around the
// 64 to 128 multiplies of a thread weigh most), a K-tile the tensor pipe 2 bn (fp16) or bn (e4m3);
// a tile's stores take about 10 bn + 600, overlapped with the next tile's K-tiles.
// Where tiles are fewer than SMs and the reduction is long (at least
// 64 K-tiles: 4096 products per output), each tile's groups may be split into ranges of at least
// two groups whose partial sums are added into the zeroed output (fp32 adds in L2): that costs the
// zeroing launch and an add per output and range.  Outputs that are requantized or group sums keep
// whole tiles.
void plan_tiles(TcArgs& a, const Geom& g, bool f8, int sms, bool may_split) {
  const int wtiles = g.groups * a.mtiles;
  const int64_t tiles256 = (int64_t)wtiles * ((g.P + TC_MAX_BN - 1) / TC_MAX_BN);
  const int kmax = may_split && a.ktiles >= 64 && tiles256 < sms ? debug_max_ksplit() : 1;
  double best = 1e30;
  int ksplit = 1;
  for (const int bn : {256, 192, 128, 64}) {
    const int64_t tiles = (int64_t)wtiles * ((g.P + bn - 1) / bn);
    if (bn < TC_MAX_BN && tiles > INT32_MAX / 8) break;
    const double drain = (700.0 + 1.3 * bn) / a.kt_per_group, mma = f8 ? bn : 2.1 * bn;
    const double kt = mma > drain ? (mma > 320.0 ? mma : 320.0) : (drain > 320.0 ? drain : 320.0);
    for (int k = 1; k <= kmax && (k == 1 || k <= g.ng / 2); ++k) {
      const int64_t items = tiles * k, waves = (items + sms - 1) / sms;
      const double body = (double)((g.ng + k - 1) / k) * a.kt_per_group * kt, epi = 10.0 * bn + 600.0;
      double t = (double)waves * (body > epi ? body : epi) + epi;
      if (k > 1) t += 4000.0 + (double)g.P * g.M * 4.0 * (1.0 + k) / 2500.0;
      if (t < best * 0.98) {
        best = t;
        a.bn = bn;
        ksplit = k;
      }
    }
  }
  a.gpk = (g.ng + ksplit - 1) / ksplit;
  a.ksplit = (g.ng + a.gpk - 1) / a.gpk;  // every range non-empty
  a.ntiles = (int)(wtiles * ((g.P + a.bn - 1) / a.bn) * a.ksplit);
}

}  // namespace

namespace {

// Ring depth, accumulators, output boxes and wait limit once the tile size is known.
void finish_plan(TcArgs& a, int row) {  // row: operand bytes per row of a K-tile
  const int stage = (TC_BM + a.bn) * row;
  a.obufs = a.ktiles <= TC_SHORT ? 2 * TC_OBUFS : TC_OBUFS;
  a.nacc = TC_TMEM_COLS / a.bn;
  a.nst = (TC_RING + TC_OUT - TC_EPI_WARPS * a.obufs * OUT_BOX) / stage;
  if (a.nst > TC_MAX_NST) a.nst = TC_MAX_NST;
  // a test may shorten the waits (debug_wait_limit_us), never the final drains
  const int64_t lim_us = debug_wait_limit_us();
  a.timeout_ns = lim_us < 0 ? TC_TIMEOUT_NS : (uint64_t)lim_us * 1000u;
}

// Output boxes by TMA store: 16-byte row pitch, and no box that reaches into another conv group.
void plan_out_map(TcArgs& a, float* out) {
  const Geom& g = a.g;
  if (a.sums || (g.groups != 1 && g.Mg % 32 != 0)) return;
  if (g.rq_out)
    a.out_tma = g.M % 16 == 0 && (reinterpret_cast<uintptr_t>(g.rq_out) & 15) == 0 &&
                make_map_2d(&a.out_map, CU_TENSOR_MAP_DATA_TYPE_UINT8, g.rq_out, (uint64_t)g.M, (uint64_t)g.P,
                            (uint64_t)g.M, 32, OUT_POS, CU_TENSOR_MAP_SWIZZLE_NONE);
  else
    a.out_tma = g.M % 4 == 0 && make_map_2d(&a.out_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, out, (uint64_t)g.M,
                                            (uint64_t)g.P, (uint64_t)g.M * 4, 32, OUT_POS, CU_TENSOR_MAP_SWIZZLE_NONE);
}

}  // namespace

fgq_status launch_tc_contract(const void* act, const Geom& g, const uint32_t* codes, const float* alpha,
                              const float* act_scale, float* out, int32_t* sums, unsigned int* err,
                              cudaStream_t s) {
  if (!tc_supports(g)) return FGQ_ERR_UNSUPPORTED;
  TcArgs a;
  memset(&a, 0, sizeof a);
  a.act_scale = act_scale;
  a.out = out;
  a.sums = sums;
  a.err = err;
  a.g = g;
  a.mtiles = (g.Mg + TC_BM - 1) / TC_BM;
  a.kt_per_group = g.G / TC_KT;
  a.ktiles = g.ng * a.kt_per_group;
  const int sms = device_sms();
  // 4-bit activations run on e4m3 operands (exact), 8-bit ones on fp16 (exact)
  const bool f8 = g.act_type == FGQ_U4 || g.act_type == FGQ_S4;
  const int es = f8 ? 1 : 2;
  plan_tiles(a, g, f8, sms, sums == nullptr && !g.rq_out);
  note_ksplit(a.ksplit);
  finish_plan(a, TC_KT * es);
  // one temporary from the stream-ordered pool: the codes expanded [M][Kp] (Kp = 16 wrow), the
  // activations expanded NHWC (a strided 1x1 convolution: only the pixels it reads, [P][C]) and the
  // transposed alphas
  const int64_t nwords = (int64_t)g.M * g.wrow;
  const int64_t nact = tc::act16_elems(g);
  const size_t a_bytes = ((size_t)nwords * 16 * es + 255) / 256 * 256, x_bytes = ((size_t)nact * es + 255) / 256 * 256;
  void* a16 = scratch_alloc(a_bytes + x_bytes + (alpha ? sizeof(float) * (size_t)g.M * g.ng : 0), s);
  if (!a16) return FGQ_ERR_CUDA;
  void* x16 = static_cast<uint8_t*>(a16) + a_bytes;
  float* alpha_t = reinterpret_cast<float*>(static_cast<uint8_t*>(x16) + x_bytes);
  a.alpha_t = alpha_t;
  // both operands in one launch, the blocks split by the two jobs' sizes
  const prep::ActSrc src = prep::act_src(act, g);
  const int cb = prep::blocks_for(nwords), xb = prep::blocks_for(src.nchunks);
  fgq_status st = after_launch(
      f8 ? launch_pdl(prep64_kernel<true>, dim3(cb + xb), dim3(256), 0, s, codes, nwords, static_cast<uint4*>(a16),
                      alpha, g.M, g.ng, alpha_t, src, static_cast<uint4*>(x16), cb)
         : launch_pdl(prep64_kernel<false>, dim3(cb + xb), dim3(256), 0, s, codes, nwords, static_cast<uint4*>(a16),
                      alpha, g.M, g.ng, alpha_t, src, static_cast<uint4*>(x16), cb));
  const CUtensorMapDataType dt = f8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  const CUtensorMapSwizzle sw = f8 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B;
  if (st == FGQ_OK && !make_map_2d(&a.a16_map, dt, a16, (uint64_t)g.wrow * 16, (uint64_t)g.M,
                                   (uint64_t)g.wrow * 16 * es, TC_KT, TC_BM, sw))
    st = FGQ_ERR_CUDA;
  a.act_tma = act_pointwise(g) ? 1 : 0;
  bool act_ok = true;
  if (st == FGQ_OK) {
    if (!f8)
      act_ok = tc::act16_map(&a.act_map, x16, g, (uint32_t)a.bn);
    else if (a.act_tma)
      act_ok = make_map_2d(&a.act_map, dt, x16, (uint64_t)g.C, (uint64_t)(nact / g.C), (uint64_t)g.C, TC_KT,
                           (uint32_t)a.bn, sw);
    else
      act_ok = make_map_im2col(&a.act_map, dt, x16, (uint64_t)g.C, 1, g.B, g.H, g.W, g.R, g.S, g.stride, g.pad, TC_KT,
                               (uint32_t)a.bn, sw);
  }
  if (!act_ok) st = FGQ_ERR_CUDA;
  if (st == FGQ_OK) plan_out_map(a, out);
  if (st == FGQ_OK && a.ksplit > 1 && cudaMemsetAsync(out, 0, (size_t)g.P * g.M * sizeof(float), s) != cudaSuccess)
    st = FGQ_ERR_CUDA;
  const int grid = a.ntiles < sms ? a.ntiles : sms;
  if (st == FGQ_OK) st = f8 ? launch_tc_variant<true>(a, grid, s) : launch_tc_variant<false>(a, grid, s);
  // the temporary returns to the pool once the work queued on s before this point is done
  if (cudaFreeAsync(a16, s) != cudaSuccess && st == FGQ_OK) st = FGQ_ERR_CUDA;
  return st;
}

// The same kernel as one dense contraction per output: the whole reduction is a single group whose
// scale is the filter's row scale, so TMEM sums across all K-tiles and is drained once per tile.
namespace {

void dense_plan(TcArgs& a, const Geom& g, int ktiles, const float* rs, const float* act_scale, float* out,
                unsigned int* err) {
  memset(&a, 0, sizeof a);
  a.alpha_t = rs;
  a.act_scale = act_scale;
  a.out = out;
  a.err = err;
  a.g = g;
  a.g.ng = 1;
  a.mtiles = (g.Mg + TC_BM - 1) / TC_BM;
  a.kt_per_group = a.ktiles = ktiles;
}

}  // namespace

bool tc_rows_supports(const Geom& g) {
  return (g.act_type == FGQ_U8 || g.act_type == FGQ_S8) && g.P < (int64_t)1 << 31 && tc::act16_supported(g);
}

size_t tc_rows_act_bytes(const Geom& g) { return (size_t)tc::act16_elems(g) * 2; }

fgq_status launch_tc_rows(const void* act, void* x16, const Geom& g, const void* a16, const float* rs,
                          const float* act_scale, float* out, unsigned int* err, cudaStream_t s) {
  if (!tc_rows_supports(g)) return FGQ_ERR_UNSUPPORTED;
  TcArgs a;
  dense_plan(a, g, g.Kred / TC_KT, rs, act_scale, out, err);
  const int sms = device_sms();
  plan_tiles(a, a.g, false, sms, false);
  finish_plan(a, TC_KT * 2);
  const prep::ActSrc src = prep::act_src(act, g);
  fgq_status st = after_launch(launch_pdl(prep64_kernel<false>, dim3(prep::blocks_for(src.nchunks)), dim3(256), 0, s,
                                          static_cast<const uint32_t*>(nullptr), (int64_t)0, static_cast<uint4*>(nullptr),
                                          static_cast<const float*>(nullptr), 0, 0, static_cast<float*>(nullptr), src,
                                          static_cast<uint4*>(x16), 0));
  if (st != FGQ_OK) return st;
  if (!make_map_2d(&a.a16_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, a16, (uint64_t)g.Kp, (uint64_t)g.M, (uint64_t)g.Kp * 2,
                   TC_KT, TC_BM, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !tc::act16_map(&a.act_map, x16, g, (uint32_t)a.bn))
    return FGQ_ERR_CUDA;
  a.act_tma = act_pointwise(g) ? 1 : 0;
  plan_out_map(a, out);
  return launch_tc_variant<false>(a, a.ntiles < sms ? a.ntiles : sms, s);
}

fgq_status launch_wait_timeout_selftest(uint32_t max_iter, unsigned int* err, cudaStream_t s) {
  wait_timeout_selftest_kernel<<<1, 32, 0, s>>>(max_iter, err);
  return after_launch();
}

fgq_status launch_wait_warp_selftest(uint64_t limit_ns, unsigned int* err, cudaStream_t s) {
  wait_warp_selftest_kernel<<<1, 32, 0, s>>>(limit_ns, err);
  return after_launch();
}

}  // namespace fgq
