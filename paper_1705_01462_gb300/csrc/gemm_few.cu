// Dense 8-bit-weight convolutions of few channels (a network's first layer): tensor-core (tcgen05)
// contraction that reads its windows straight out of shared memory.
//
// With at most 8 channels a position's window is R short runs of S taps, and an im2col copy of it
// holds every input value up to R S / stride^2 times.  Here each CTA converts the input rows of its
// tile once, to fp16 with Cp = 4 or 8 channels a pixel, and the MMAs read the overlapping windows
// where they lie: the activation operand is K-major without swizzle, whose core matrix is 8 rows of
// 16 bytes at a row pitch of 16 bytes, and output positions are exactly one 16-byte piece apart once
// the pieces of a row are dealt into u = stride Cp / 8 planes (piece c in plane c % u at index c / u).
// Filter row kr and the pieces j, j + 1 of a run are then one MMA of K = 16 whose descriptor starts
// at that row and piece; nothing is copied per tap.
//
// Tile: up to 256 positions (MMA N) of bh output rows, x 128 operand rows (MMA M).  Rows of a tile
// lie pitch pieces apart, so N runs over the spare columns between them, which nobody reads.  With at
// most 64 filters the operand rows are two copies of the filters, the second shifted by the stride:
// one MMA computes output rows 2 v and 2 v + 1 (pr = 2), Rv = R + stride filter rows instead of 2 R.
// The input rows lie by phase (row % sv, sv = pr stride), so that successive output rows are the same
// distance apart for every filter row.
//
// Sums: products of two 8-bit integers, at most 514 per output: every partial sum is below 2^24 and
// exact in the fp32 accumulator; y = (s_x wscale[m]) sum, or its requantized code.
//
// Warps (one CTA per SM, a contiguous range of tiles each):
//   0-7   epilogue: TMEM lanes 32 (w % 4) .., 16 positions at a time: scale, box in shared memory,
//         TMA store (or direct stores where rows of the output are no multiple of 16 bytes);
//   8-23  convert the input rows, eight warps for each of two stages;
//   24    TMEM allocation and MMA issue.  Two accumulators of 256 columns.
// The weights are expanded into shared memory once per CTA; there is no temporary and one launch.
//
// Bound: the fp32 output (7x7/2 over 224 x 224 x 3, 64 filters, batch 64: 206 MB, 30 us of writes).
// That call takes 53 us, 45 us of them with nothing but the stores left in; im2col rows and a GEMM over
// them took 155.  Eight converting warps instead of sixteen: 67 us (under a full write load the loads
// take microseconds, so two tiles' loads have to be in flight).  The same windows by 5D tensor maps of
// overlapping positions, 64 bytes a row: 126 us.  MMAs on the unswizzled operand take about 140 clk at
// N = 240 (120 from a swizzled tile), which the stores hide.
// Other shapes, before and after: 11x11/4 over 227 x 227 x 3, 96 filters, batch 256, 409 and 181 us;
// 3x3 over 32 x 32 x 3, batch 256, 66 and 21; 3x3 over 250 x 250 x 4, 512 filters, batch 8, 254 and 171;
// 7x7/2 at batch 1 30 and 15.
// Every wait is bounded in time; on expiry the kernel records FGQ_ERR_TIMEOUT, each role leaves its
// loop, MMAs and stores in flight are waited for, and TMEM is freed.
#include <cuda_fp16.h>

#include <cstdint>
#include <cstring>

#include "tc_common.cuh"

namespace fgq {
namespace {

constexpr int FW_EPI_WARPS = 8;
constexpr int FW_CONV_WARPS = 16;    // two groups, one per stage
constexpr int FW_GROUP_WARPS = FW_CONV_WARPS / 2;
constexpr int FW_MMA_WARP = FW_EPI_WARPS + FW_CONV_WARPS;
constexpr int FW_THREADS = 32 * (FW_MMA_WARP + 1);
constexpr int FW_MAX_N = 256;        // columns per accumulator
constexpr int FW_NACC = 2;
constexpr int FW_NST = 2;            // stages of input rows
constexpr int FW_OBUFS = 4;          // output boxes per epilogue warp, or 2 where that makes room for rows
constexpr int FW_OBOX = 16 * 32 * 4; // fp32 [16 positions][32 filters]
constexpr int FW_MAX_ROWS = 128;     // input rows of a tile
constexpr int FW_BARS = 8 * (2 * FW_NST + 2 * FW_NACC + 2) + 16 + 4 * FW_MAX_ROWS;
constexpr int FW_SMEM = 232448;      // shared memory of a block, at most
constexpr int FW_MAX_PIECES = 16;    // 16-byte pieces of a run
constexpr uint64_t FW_TIMEOUT_NS = 1000000000ull;
constexpr uint32_t FW_DRAIN_LIMIT = 1u << 20;

struct FewArgs {
  CUtensorMap out_map;  // outputs [B Ho][Wo][M], box {32 filters, 16 positions, 1 row}; if out_tma
  const uint8_t* act;
  const int8_t* wq;
  const float* wscale;
  const float* act_scale;
  float* out;
  unsigned int* err;
  Geom g;
  int u, nch;           // planes; pieces of a run (even)
  int pl, pitch;        // pieces of a row per plane; the same with the spare columns
  int pr, fb;           // output rows per operand copy; filters per tile (128 / pr)
  int sv, Rv;           // input rows between virtual output rows (pr output rows each); their filter rows
  int bh, nh;           // virtual output rows per tile; rows per phase
  int n;                // MMA N
  int tpi, tiles, per;  // tiles per image, tiles, tiles per CTA
  int arows;            // operand rows kept in shared memory (those past the filters are never read out)
  int a_bytes, stage;
  int obufs;            // output boxes per epilogue warp: 4 or 2
  int out_tma;
  uint64_t timeout_ns;
  uint8_t ord[FW_MAX_PIECES];       // piece of the run at K position e (plane by plane)
  uint32_t koff[FW_MAX_PIECES / 2]; // of each pair of pieces: byte offset of the first,
  uint32_t klbo[FW_MAX_PIECES / 2]; // and of the second from it
};

// Eight input bytes (zero where ok is false) as fp16 integers.
template <int CP>
__device__ __forceinline__ uint4 piece_f16(const uint8_t* row, int px, int W, int C, bool rowok, uint32_t flip,
                                           uint32_t bias) {
  uint32_t b[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int p = px + e / CP, c = e % CP;
    const bool in = rowok && (uint32_t)p < (uint32_t)W;
    b[e] = in && (c == 0 || c < C) ? (uint32_t)__ldg(row + p * C + c) : 0u;
  }
  const uint32_t lo = (b[0] | b[1] << 8 | b[2] << 16 | b[3] << 24) ^ flip;
  const uint32_t hi = (b[4] | b[5] << 8 | b[6] << 16 | b[7] << 24) ^ flip;
  return make_uint4(tc::u8pair_to_h2(lo, 0x4140, bias), tc::u8pair_to_h2(lo, 0x4342, bias),
                    tc::u8pair_to_h2(hi, 0x4140, bias), tc::u8pair_to_h2(hi, 0x4342, bias));
}

template <int CP, bool RQ, int OBUFS>
__global__ void __launch_bounds__(FW_THREADS, 1) few_kernel(const __grid_constant__ FewArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* obox = smem + a.a_bytes;
  uint8_t* stages = obox + FW_EPI_WARPS * OBUFS * FW_OBOX;
  uint64_t* full = reinterpret_cast<uint64_t*>(stages + FW_NST * a.stage);
  uint64_t* empty = full + FW_NST;
  uint64_t* acc_full = empty + FW_NST;
  uint64_t* acc_empty = acc_full + FW_NACC;
  uint64_t* drain_bar = acc_empty + FW_NACC;
  uint64_t* a_full = drain_bar + 1;  // weights in place
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(a_full + 1);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  uint32_t* row_at = tmem_slot + 4;  // first piece of input row i of a stage

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // warp-uniform
  const int lane = threadIdx.x & 31;
  const Geom& g = a.g;
  const uint64_t tmo = a.timeout_ns;
  const int m0 = (int)blockIdx.y * a.fb;

  if (threadIdx.x == 0) {
    for (int i = 0; i < FW_NST; ++i) {
      mbar_init(&full[i], FW_GROUP_WARPS);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < FW_NACC; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], FW_EPI_WARPS);
    }
    mbar_init(drain_bar, 1);
    mbar_init(a_full, FW_EPI_WARPS);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == FW_MMA_WARP) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  const int rows = (a.bh - 1) * a.sv + a.Rv;
  for (int i = threadIdx.x; i < rows; i += FW_THREADS) row_at[i] = (uint32_t)((i % a.sv) * a.nh + i / a.sv) * (uint32_t)a.pitch;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // the prologue above overlapped the previous kernel; global memory only from here on
  pdl_wait();
  pdl_trigger();
  const uint32_t tmem = *tmem_slot;
  const int t0 = (int)blockIdx.x * a.per;
  const int my_tiles = a.tiles - t0 < a.per ? a.tiles - t0 : a.per;  // (none: <= 0)

  auto fail = [&]() {
    *abort_flag = 1;
    record_error(a.err, FGQ_ERR_TIMEOUT);
  };

  if (warp == FW_MMA_WARP) {
    // ------------------------------------------------------------------ MMA issue
    const uint32_t idesc = idesc_f16_f32(128, a.n);
    const uint64_t ad0 = sdesc_k_sw32(smem_u32(smem));
    const uint32_t ablk = (uint32_t)a.arows * 32u >> 4;
    const uint32_t rowb = (uint32_t)a.pitch * 16u;
    bool ok = my_tiles <= 0 || mbar_wait_warp(a_full, 0, tmo, abort_flag);
    for (int tl = 0; tl < my_tiles && ok; ++tl) {
      const int s = tl & 1;
      const uint32_t ph = (uint32_t)(tl >> 1) & 1u;
      if (!mbar_wait_warp(&acc_empty[s], ph ^ 1u, tmo, abort_flag) || !mbar_wait_warp(&full[s], ph, tmo, abort_flag)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t base = smem_u32(stages) + (uint32_t)(s * a.stage);
      uint64_t ad = ad0;
      int f = 0, hi = 0;  // phase and row of filter row kr
      for (int kr = 0; kr < a.Rv; ++kr) {
        const uint32_t rb = base + (uint32_t)(f * a.nh + hi) * rowb;
        for (int i = 0; i < a.nch / 2; ++i, ad += ablk) {
          const uint64_t bd = sdesc_k_plain(rb + a.koff[i], a.klbo[i], 128);
          if (elect_one()) mma_f16(tmem + (uint32_t)(s * FW_MAX_N), ad, bd, idesc, (kr | i) != 0 ? 1u : 0u);
          __syncwarp();
        }
        if (++f == a.sv) {
          f = 0;
          ++hi;
        }
      }
      if (elect_one()) {
        mma_commit(&empty[s]);
        mma_commit(&acc_full[s]);
      }
      __syncwarp();
    }
    if (!ok && !*abort_flag) fail();
    if (elect_one()) mma_commit(drain_bar);
    __syncwarp();
    mbar_wait_bounded(drain_bar, 0, FW_DRAIN_LIMIT);
  } else if (warp >= FW_EPI_WARPS) {
    // ------------------------------------------------------------------ input rows
    const int group = (warp - FW_EPI_WARPS) / FW_GROUP_WARPS;
    const int tid = (int)threadIdx.x - 32 * (FW_EPI_WARPS + group * FW_GROUP_WARPS);
    const uint32_t flip = g.act_type == FGQ_S8 ? 0x80808080u : 0u, bias = flip ? 0x64806480u : 0x64006400u;
    const int cpr = a.u * a.pl;                                // pieces of a row
    const uint32_t plane = (uint32_t)(a.sv * a.nh * a.pitch);  // of a plane of a stage
    constexpr int STEP = 32 * FW_GROUP_WARPS, U = 6;
    // pieces tid, tid + STEP, ... of the tile's rows x cpr
    const int i0 = tid / cpr, c00 = tid - i0 * cpr, di = STEP / cpr, dc = STEP - di * cpr;
    bool ok = true;
    for (int tl = group; tl < my_tiles; tl += 2) {
      const int s = group;
      const int tile = t0 + tl, b = tile / a.tpi, v0 = (tile - b * a.tpi) * a.bh;
      const int h0 = v0 * a.sv - g.pad;
      const uint8_t* img = a.act + (int64_t)b * g.H * g.W * g.C;
      uint4* st = reinterpret_cast<uint4*>(stages + s * a.stage);
      int i = i0, c = c00;
      bool free = false;
      while (i < rows || !free) {  // U pieces at a time, their loads ahead of the wait for the stage
        uint4 x[U];
        uint32_t at[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const int h = h0 + i;
          const bool in = i < rows, rowok = in && h >= 0 && h < g.H;
          x[k] = piece_f16<CP>(img + (int64_t)(rowok ? h : 0) * g.W * g.C, c * (8 / CP) - g.pad, g.W, g.C, rowok, flip, bias);
          at[k] = !in ? 0xffffffffu
                      : row_at[i] + (a.u == 1 ? (uint32_t)c : (uint32_t)(c % a.u) * plane + (uint32_t)(c / a.u));
          c += dc;
          i += di;
          if (c >= cpr) {
            c -= cpr;
            ++i;
          }
        }
        if (!free) {
          ok = mbar_wait_warp(&empty[s], ((uint32_t)(tl >> 1) & 1u) ^ 1u, tmo, abort_flag);
          free = true;
          if (!ok) break;
        }
#pragma unroll
        for (int k = 0; k < U; ++k)
          if (at[k] != 0xffffffffu) st[at[k]] = x[k];
      }
      if (!__all_sync(0xffffffffu, ok)) {
        ok = false;
        break;
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
    }
    if (!ok && !*abort_flag) fail();
  } else {
    // ------------------------------------------------------------------ epilogue
    const int quarter = warp & 3, part = warp >> 2;
    const int lrow = 32 * quarter;                // operand row of lane 0
    const int sub = lrow >= a.fb ? 1 : 0;         // output row of the virtual row
    const int mw = m0 + lrow - sub * a.fb, m = mw + lane;
    const uint32_t tbase = tmem + ((uint32_t)lrow << 16);
    // the weights: piece ord[e] of filter row kr as 16 bytes of block (kr nch + e) / 2, which holds
    // arows operand rows of 32 bytes (two pieces) in the 32-byte swizzle
#pragma unroll 4
    for (int i = threadIdx.x; i < a.Rv * a.nch * a.arows; i += 32 * FW_EPI_WARPS) {
      const int ke = i / a.arows, row = i - ke * a.arows;
      const int kr = ke / a.nch, j = a.ord[ke - kr * a.nch];
      const int sb = row >= a.fb ? 1 : 0, mm = m0 + row - sb * a.fb, r = kr - sb * g.stride;
      const bool rok = mm < g.M && r >= 0 && r < g.R;
      const int8_t* wrow = a.wq + (rok ? ((int64_t)mm * g.R + r) * g.S * g.C : 0);
      int q[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int x = 8 * j + e, sx = x / CP, c = x % CP;
        q[e] = rok && sx < g.S && c < g.C ? (int)__ldg(wrow + sx * g.C + c) : 0;
      }
      uint32_t v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        v[e] = (uint32_t)__half_as_ushort(__int2half_rn(q[2 * e])) | (uint32_t)__half_as_ushort(__int2half_rn(q[2 * e + 1])) << 16;
      reinterpret_cast<uint4*>(smem)[(ke >> 1) * a.arows * 2 + row * 2 + ((ke ^ (row >> 2)) & 1)] = make_uint4(v[0], v[1], v[2], v[3]);
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(a_full);
    const float sc = m < g.M ? __ldg(a.act_scale) * __ldg(a.wscale + m) : 0.0f;
    RqMul rq;
    if (RQ) rq = rq_mul(g.rq_scale, g.rq_signed);
    const int bpr = (g.Wo + 15) / 16, nb = a.bh * bpr;  // blocks of 16 positions: per row, per tile
    uint8_t* const ob0 = obox + OBUFS * warp * FW_OBOX;
    int obuf = 0;
    bool ok = true;
    for (int tl = 0; tl < my_tiles; ++tl) {
      const int s = tl & 1;
      if (!mbar_wait_warp(&acc_full[s], (uint32_t)(tl >> 1) & 1u, tmo, abort_flag)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const int tile = t0 + tl, b = tile / a.tpi, v0 = (tile - b * a.tpi) * a.bh;
      int j = part / bpr, blk = part - j * bpr;
#pragma unroll 1
      for (int k = part; k < nb; k += 2) {
        const int ho = (v0 + j) * a.pr + sub;
        const int wo = 16 * blk;
        const bool live = ho < g.Ho && mw < g.M;  // warp-uniform
        if (live) {
          uint32_t v[16];
          tmem_ld16(tbase + (uint32_t)(s * FW_MAX_N + j * a.pitch + wo), v);
          tmem_ld_wait_regs16(v);
          const int row = b * g.Ho + ho;
          if (a.out_tma) {  // positions past Wo and filters past M are clipped by the tensor map
            if (lane == 0) bulk_wait_read<OBUFS - 1>();  // the buffer's previous box has been read out
            __syncwarp();
            uint8_t* ob = ob0 + obuf * FW_OBOX;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const float y = sc * __uint_as_float(v[e]);
              if (RQ) ob[32 * e + lane] = rq_code(y, rq);
              else reinterpret_cast<float*>(ob)[32 * e + lane] = y;
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
              tma_store_3d(&a.out_map, mw, wo, row, smem_u32(ob));
              bulk_commit();
            }
            obuf = (obuf + 1) & (OBUFS - 1);
          } else if (m < g.M) {
            const int64_t o = ((int64_t)row * g.Wo + wo) * g.M + m;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              if (wo + e < g.Wo) {
                const float y = sc * __uint_as_float(v[e]);
                if (RQ) g.rq_out[o + (int64_t)e * g.M] = rq_code(y, rq);
                else a.out[o + (int64_t)e * g.M] = y;
              }
            }
          }
        }
        blk += 2;
        while (blk >= bpr && j < a.bh) {
          blk -= bpr;
          ++j;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[s]);
    }
    if (!ok && !*abort_flag) fail();
    if (lane == 0) bulk_wait_all();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == FW_MMA_WARP) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// Layout and tiles of a shape; false where it does not fit.
bool plan_few(const Geom& g, FewArgs& a, int sms) {
  if (g.act_type != FGQ_U8 && g.act_type != FGQ_S8) return false;
  if (g.groups != 1 || g.C > 8 || g.Kred > 514 || g.Wo > FW_MAX_N || g.P >= (int64_t)1 << 31) return false;
  if (g.stride > 64 || g.pad > 1024 || g.M > 65535) return false;
  const int Cp = g.C <= 4 && g.stride % 2 == 0 ? 4 : 8;
  a.u = g.stride * Cp / 8;
  a.nch = (g.S * Cp + 15) / 16 * 2;
  if (a.nch > FW_MAX_PIECES) return false;
  const int maxidx = (a.nch - 1) / a.u;
  a.pl = g.Wo + maxidx;
  a.pitch = (a.pl + 15) / 16 * 16;
  const int wo16 = (g.Wo + 15) / 16 * 16;
  double best = 1e30;
  // two output rows per MMA where the filters leave half of its rows free and the operand fits
  for (int pr = g.M <= 64 && g.Ho > 1 ? 2 : 1; pr >= 1; --pr) {
    const int fb = 128 / pr, sv = pr * g.stride, Rv = g.R + (pr - 1) * g.stride;
    const int vrows = (g.Ho + pr - 1) / pr, mtiles = (g.M + fb - 1) / fb;
    const int arows = pr == 2 || g.M >= 128 ? 128 : (g.M + 7) / 8 * 8;
    const int a_bytes = (Rv * a.nch * arows * 16 + 1023) / 1024 * 1024;
    for (int obufs = FW_OBUFS; obufs >= 2; obufs /= 2) {
      const int fixed = 1024 + a_bytes + FW_EPI_WARPS * obufs * FW_OBOX + FW_BARS;
      for (int bh = 1; bh <= vrows; ++bh) {
        const int n = (bh - 1) * a.pitch + wo16;
        if (n > FW_MAX_N || (bh - 1) * sv + Rv > FW_MAX_ROWS) break;
        const int nh = bh + (Rv - 1) / sv;
        const int64_t stage = ((int64_t)a.u * sv * nh * a.pitch * 16 + 256 + 127) / 128 * 128;
        if (fixed + FW_NST * stage > FW_SMEM) break;
        const int tpi = (vrows + bh - 1) / bh;
        const int64_t tiles = (int64_t)g.B * tpi;
        if (tiles > INT32_MAX / 2) continue;
        const int gx = sms / mtiles > 1 ? sms / mtiles : 1, per = (int)((tiles + gx - 1) / gx);
        // clk per tile: MMAs of n / 2 (at least 64), boxes of 16 positions, 16-byte pieces converted
        const double mma = Rv * a.nch / 2 * (n > 128 ? n / 2.0 : 64.0);
        const double epi = (obufs == 2 ? 125.0 : 100.0) * bh * ((g.Wo + 15) / 16);
        const double conv = 1.2 * ((bh - 1) * sv + Rv) * a.u * a.pl;
        const double body = mma > epi ? (mma > conv ? mma : conv) : (epi > conv ? epi : conv);
        const double t = per * (body + 200.0) + body;
        if (t < best) {
          best = t;
          a.pr = pr;
          a.fb = fb;
          a.sv = sv;
          a.Rv = Rv;
          a.bh = bh;
          a.nh = nh;
          a.n = n;
          a.tpi = tpi;
          a.tiles = (int)tiles;
          a.per = per;
          a.arows = arows;
          a.a_bytes = a_bytes;
          a.stage = (int)stage;
          a.obufs = obufs;
        }
      }
    }
  }
  return best < 1e30;
}

template <int CP, bool RQ, int OBUFS>
fgq_status launch_few_kernel(const FewArgs& a, dim3 grid, int smem, cudaStream_t s) {
  if (!tc::smem_attr_once<few_kernel<CP, RQ, OBUFS>>(FW_SMEM)) return FGQ_ERR_CUDA;
  return after_launch(launch_pdl(few_kernel<CP, RQ, OBUFS>, grid, dim3(FW_THREADS), smem, s, a));
}

template <int CP>
fgq_status launch_few_cp(const FewArgs& a, dim3 grid, int smem, cudaStream_t s) {
  if (a.obufs == FW_OBUFS)
    return a.g.rq_out ? launch_few_kernel<CP, true, FW_OBUFS>(a, grid, smem, s)
                      : launch_few_kernel<CP, false, FW_OBUFS>(a, grid, smem, s);
  return a.g.rq_out ? launch_few_kernel<CP, true, 2>(a, grid, smem, s) : launch_few_kernel<CP, false, 2>(a, grid, smem, s);
}

}  // namespace

bool few_supports(const Geom& g) {
  FewArgs a;
  return tc::encode_tiled() != nullptr && plan_few(g, a, device_sms());
}

fgq_status launch_few(const void* act, const Geom& g, const int8_t* wq, const float* wscale, const float* act_scale,
                      float* out, unsigned int* err, cudaStream_t s) {
  FewArgs a;
  memset(&a, 0, sizeof a);
  if (!plan_few(g, a, device_sms())) return FGQ_ERR_UNSUPPORTED;
  a.act = static_cast<const uint8_t*>(act);
  a.wq = wq;
  a.wscale = wscale;
  a.act_scale = act_scale;
  a.out = out;
  a.err = err;
  a.g = g;
  // a run's pieces plane by plane, and where each pair of them starts
  const uint32_t plane = (uint32_t)(a.sv * a.nh * a.pitch);
  uint32_t off[FW_MAX_PIECES];
  int e = 0;
  for (int q = 0; q < a.u && q < a.nch; ++q)
    for (int j = q; j < a.nch; j += a.u) {
      a.ord[e] = (uint8_t)j;
      off[e++] = ((uint32_t)q * plane + (uint32_t)(j / a.u)) * 16u;
    }
  for (int i = 0; i < a.nch / 2; ++i) {
    a.koff[i] = off[2 * i];
    a.klbo[i] = off[2 * i + 1] - off[2 * i];
  }
  // a test may shorten the waits (debug_wait_limit_us), never the final drains
  const int64_t lim_us = debug_wait_limit_us();
  a.timeout_ns = lim_us < 0 ? FW_TIMEOUT_NS : (uint64_t)lim_us * 1000u;
  const size_t es = g.rq_out ? 1 : 4;
  void* y = g.rq_out ? static_cast<void*>(g.rq_out) : static_cast<void*>(out);
  if ((size_t)g.M * es % 16 == 0 && (reinterpret_cast<uintptr_t>(y) & 15) == 0) {
    const cuuint64_t dims[3] = {(cuuint64_t)g.M, (cuuint64_t)g.Wo, (cuuint64_t)g.B * g.Ho};
    const cuuint64_t strides[2] = {(cuuint64_t)g.M * es, (cuuint64_t)g.Wo * g.M * es};
    const cuuint32_t box[3] = {32, 16, 1}, estr[3] = {1, 1, 1};
    a.out_tma = tc::encode_tiled()(&a.out_map, g.rq_out ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                                   3, y, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                   CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  }
  const dim3 grid((unsigned)((a.tiles + a.per - 1) / a.per), (unsigned)((g.M + a.fb - 1) / a.fb));
  const int smem = 1024 + a.a_bytes + FW_EPI_WARPS * a.obufs * FW_OBOX + FW_NST * a.stage + FW_BARS;
  const bool four = g.stride % 2 == 0 && g.C <= 4;
  return four ? launch_few_cp<4>(a, grid, smem, s) : launch_few_cp<8>(a, grid, smem, s);
}

}  // namespace fgq
