// Tensor-core (tcgen05) group sums for G = 4: the 32-bit group accumulators of Section 4
// themselves, s[m][g][p] = sum over a group of 4 reduction elements of t q, as int32.  (The fp32
// outputs of G = 4 come from the folded kernel, gemm_fold.cu.)
//
// A dense MMA would sum across groups, so each K = 16 MMA step (4 groups) uses a block-diagonal
// ternary operand A' of 128 rows: row 4 m' + j holds filter m' of the tile (32 filters) only
// in the 4 columns of group slot j (zeros elsewhere), and D[4 m' + j][p] of one MMA
// (M = 128, N = 256, K = 16) is exactly the sum of group 4 step + j.  A' depends only on the
// weights, so it is built once per call in fp16 {0, +1, -1}; the activations are the plain
// dense operand, expanded to fp16 once per call (one launch, prep4_kernel, prepares both) and
// loaded by TMA (2D rows or im2col boxes).
//
// Tile: 32 filters x 256 positions; K-tile 64 (16 groups, 4 steps); TMEM: two 256-column
// accumulators.
// Warp roles (352 threads, one CTA per SM, persistent over tiles):
//   warps 0-7  epilogue: warp w reads TMEM lanes 32 (w % 4) .. (filter rows x slots) and the
//              128 positions of half w / 4 in 16-column loads, frees the buffer, and stores the
//              values as int32;
//   warps 8, 9 the MMA issuers (one thread each; warp 8 also allocates TMEM): alternate steps
//              into their own accumulator, so one thread's barrier waits overlap the other's
//              MMAs;
//   warp 10    the producer (one thread): per K-tile, the A' box (64 reduction elements x 128
//              rows) and the activation box (64 channels x 256 positions) into one ring stage.
// A stage is released by the epilogue when it sees the K-tile's last accumulator commit, so
// no commit is spent on the stages.  Every mbarrier wait is bounded in time; on expiry the
// kernel records FGQ_ERR_TIMEOUT, each role leaves its loop (uniformly within the epilogue,
// which uses named barriers), in-flight copies and MMAs are waited for, and TMEM is freed.
#include <cstdint>
#include <cstring>

#include "operand_prep.cuh"
#include "tc_common.cuh"

namespace fgq {
namespace {

using tc::encode_tiled;
using tc::make_map_2d;

constexpr int T4_FM = 32;       // filters per tile
constexpr int T4_ROWS = 128;    // MMA M: 4 slots x 32 filters, row 4 m' + j
constexpr int T4_BN = 256;      // positions per tile (MMA N)
constexpr int T4_KT = 64;       // reduction elements per K-tile: 16 groups, 4 MMA steps
constexpr int T4_NACC = 2;      // TMEM accumulators of 256 columns
constexpr int T4_EPI_WARPS = 8;
constexpr int T4_MMA_WARP = 8;  // warps 8 and 9
constexpr int T4_PROD_WARP = 10;
constexpr int T4_THREADS = 32 * (T4_PROD_WARP + 1);
constexpr int T4_TMEM_COLS = T4_NACC * T4_BN;
constexpr int T4_EPI_COLS = T4_BN / 2;             // positions per epilogue thread
constexpr uint64_t T4_TIMEOUT_NS = 1000000000ull;  // 1 s per wait
constexpr uint32_t T4_DRAIN_LIMIT = 1u << 20;      // polls of the final drains (never shortened)
constexpr uint32_t BAR_EPI4 = 2;

constexpr int A_TILE4 = T4_ROWS * T4_KT * 2;  // 16 KB fp16 block-diagonal operand
constexpr int B_TILE4 = T4_BN * T4_KT * 2;    // 32 KB fp16 activations

constexpr int T4_STAGE = A_TILE4 + B_TILE4;
constexpr int T4_NST = 4;
constexpr int T4_SMEM = 1024 + T4_NST * T4_STAGE + 8 * (2 * T4_NST + 2 * T4_NACC + 1) + 16;
static_assert(T4_SMEM <= 232448, "shared memory budget");
static_assert(A_TILE4 % 1024 == 0 && B_TILE4 % 1024 == 0, "stage alignment");

struct T4Args {
  CUtensorMap a_map;    // fp16 A' [(groups * mtiles) * 128 rows][Kp], box {64, 128}, 128B swizzle
  CUtensorMap act_map;  // fp16 activations: 2D [positions][C] or im2col, box 64 channels x 256 positions
  int32_t* sums;        // int32 group sums [M][ng][P]
  unsigned int* err;
  Geom g;
  int mtiles, ptiles, ntiles, ktiles;  // mtiles: 32-filter tiles per conv group
  uint64_t timeout_ns;
};

// Tiles are numbered with the filter tiles of one position tile consecutive, so that
// CTAs running at the same time share activation boxes in L2.
__device__ __forceinline__ void tile_coords4(const T4Args& a, int tile, int& gi, int& mt, int64_t& p0) {
  const int per_p = a.g.groups * a.mtiles;
  const int pt = tile / per_p;
  const int r = tile - pt * per_p;
  gi = r / a.mtiles;
  mt = r - gi * a.mtiles;
  p0 = (int64_t)pt * T4_BN;
}

// One launch prepares both operands of a call.  Blocks [0, fold_blocks) build the
// block-diagonal ternary operand A' straight from the 2-bit codes, one block per 32-filter
// tile and slice of the reduction axis: row 4 m' + j of tile (gi, mt) holds, for filter
// gi Mg + mt 32 + m', the codes (fp16 {0, +1, -1}) of the groups whose index is j modulo 4 (slot j
// of every K = 16 step) and zeros elsewhere.  One thread per 16-byte chunk of A' (8 elements = 2
// groups, at most one of them in the row's slot).  The other blocks expand the activations
// to fp16.
constexpr int PREP4_CHUNKS = 8;  // 16-byte chunks of a row per fold block (64 elements)

__global__ void __launch_bounds__(256) prep4_kernel(const uint32_t* __restrict__ codes, int wrow, int ng, int Kp,
                                                    int Mg, int mtiles, int ksplit, uint4* __restrict__ a0,
                                                    int fold_blocks, const prep::ActSrc src, uint4* __restrict__ x16) {
  pdl_wait();
  pdl_trigger();
  if ((int)blockIdx.x >= fold_blocks) {
    const int64_t nb = (int64_t)gridDim.x - fold_blocks;
    prep::act_expand<false>(src, ((int64_t)blockIdx.x - fold_blocks) * blockDim.x + threadIdx.x, nb * blockDim.x, x16);
    return;
  }
  const int tile = (int)blockIdx.x / ksplit, ks = (int)blockIdx.x - tile * ksplit;
  const int gi = tile / mtiles, mt = tile - gi * mtiles;
  const int cpr = Kp / 8;  // chunks per row
  const int c0 = ks * PREP4_CHUNKS;
  const int nc = (cpr - c0) < PREP4_CHUNKS ? (cpr - c0) : PREP4_CHUNKS;
  for (int it = threadIdx.x; it < T4_ROWS * nc; it += blockDim.x) {
    const int rr = it / nc, c = c0 + (it - rr * nc);
    const int mp = rr >> 2, j = rr & 3;
    const int local = mt * T4_FM + mp;
    uint32_t h[4] = {0u, 0u, 0u, 0u};
    // group 2c occupies halves 0-3 of the chunk, group 2c + 1 halves 4-7; slot = group % 4
    const int grp = ((2 * c) & 3) == j ? 2 * c : (((2 * c + 1) & 3) == j ? 2 * c + 1 : -1);
    if (local < Mg && grp >= 0 && grp < ng) {
      const int64_t m = (int64_t)gi * Mg + local;
      const int k0 = 4 * grp;  // the group's 4 codes lie in one word, bits 2 (k0 % 16) ..
      const uint32_t cw = (__ldg(codes + m * wrow + k0 / 16) >> (2 * (k0 % 16))) & 0xffu;
      uint32_t e4[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t t = (cw >> (2 * e)) & 3u;  // 00 = 0, 01 = +1, 11 = -1
        e4[e] = t == 1u ? 0x3C00u : (t == 3u ? 0xBC00u : 0u);
      }
      // the group fills 32-bit words 0-1 of the chunk (group 2c) or 2-3 (group 2c + 1)
      const bool first = grp == 2 * c;
      const uint32_t p0 = e4[0] | (e4[1] << 16), p1 = e4[2] | (e4[3] << 16);
      h[0] = first ? p0 : 0u;
      h[1] = first ? p1 : 0u;
      h[2] = first ? 0u : p0;
      h[3] = first ? 0u : p1;
    }
    a0[((int64_t)tile * T4_ROWS + rr) * cpr + c] = make_uint4(h[0], h[1], h[2], h[3]);
  }
}

template <bool TMAP>
__global__ void __launch_bounds__(T4_THREADS, 1) tc4_sums_kernel(const __grid_constant__ T4Args a) {
  constexpr int NST = T4_NST;
  extern __shared__ uint8_t smem_raw4[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw4) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + NST * T4_STAGE);
  uint64_t* full = bars;
  uint64_t* empty = bars + NST;
  uint64_t* acc_full = empty + NST;
  uint64_t* acc_empty = acc_full + T4_NACC;
  uint64_t* drain_bar = acc_empty + T4_NACC;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const Geom& g = a.g;
  const uint64_t tmo = a.timeout_ns;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NST; ++i) {
      mbar_init(&full[i], 1);   // the producer's expect_tx, then the boxes' bytes
      mbar_init(&empty[i], 1);  // released by the epilogue (the K-tile's MMAs completed)
    }
    for (int i = 0; i < T4_NACC; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], T4_EPI_WARPS);
    }
    mbar_init(drain_bar, T4_NACC);  // one commit per MMA issuer
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == T4_MMA_WARP) {
    tmem_alloc(tmem_slot, T4_TMEM_COLS);
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
  const int units_per_tile = 4 * a.ktiles;  // drains (MMA steps) per tile

  auto fail = [&]() {
    *abort_flag = 1;
    record_error(a.err, FGQ_ERR_TIMEOUT);
  };

  // ------------------------------------------------------------------ producer
  if (warp == T4_PROD_WARP && lane == 0) {
    const int total = my_tiles * a.ktiles;
    int gi = 0, mt = 0, tr = 0, ts = 0, tc0 = 0, kt = 0, tl = 0;
    int64_t p0 = 0;
    int n0 = 0, h0 = 0, w0 = 0;  // im2col: the tile's first window origin (input pixel coordinates)
    int issued = 0;
    bool ok = true;
    for (int j = 0; j < total; ++j) {
      if (kt == 0) {
        tile_coords4(a, (int)blockIdx.x + tl * (int)gridDim.x, gi, mt, p0);
        tr = ts = tc0 = 0;
        if (!TMAP) {
          const int pp = (int)p0;  // < P < 2^31
          const int wo = pp % g.Wo;
          const int q = pp / g.Wo;
          n0 = q / g.Ho;
          h0 = (q - n0 * g.Ho) * g.stride - g.pad;
          w0 = wo * g.stride - g.pad;
        }
      }
      const int s = j % NST;
      if (j >= NST && !mbar_wait_timed(&empty[s], ((j / NST) & 1) ^ 1, tmo, abort_flag, 64)) {
        ok = false;
        break;
      }
      uint8_t* sa = smem + s * T4_STAGE;
      const int arow = (gi * a.mtiles + mt) * T4_ROWS;
      const int ch = gi * g.Cg + tc0;  // a multiple of 64 (128-byte aligned in fp16)
      mbar_arrive_expect_tx(&full[s], T4_STAGE);
      tma_load_2d(smem_u32(sa), &a.a_map, kt * T4_KT, arow, &full[s]);
      uint8_t* sb = sa + A_TILE4;
      if (TMAP)
        tma_load_2d(smem_u32(sb), &a.act_map, ch, (int)p0, &full[s]);
      else
        tma_load_im2col_4d(smem_u32(sb), &a.act_map, ch, w0, h0, n0, (uint16_t)ts, (uint16_t)tr, &full[s]);
      issued = j + 1;
      tc0 += T4_KT;
      if (tc0 == g.Cg) {
        tc0 = 0;
        if (++ts == g.S) {
          ts = 0;
          ++tr;
        }
      }
      if (++kt == a.ktiles) {
        kt = 0;
        ++tl;
      }
    }
    if (!ok && !*abort_flag) fail();
    // loads the MMA issuers may not have consumed: the last NST issued, one per stage, each
    // the latest phase of its stage's barrier; none may outlive the CTA
    for (int j = issued - NST < 0 ? 0 : issued - NST; j < issued; ++j)
      mbar_wait_bounded(&full[j % NST], (j / NST) & 1, T4_DRAIN_LIMIT);
  }

  // ------------------------------------------------------------------ MMA issuers
  if ((warp == T4_MMA_WARP || warp == T4_MMA_WARP + 1) && lane == 0) {
    const int b = warp - T4_MMA_WARP;  // this thread's accumulator: the units of its parity
    const uint32_t idesc = idesc_f16_f32(T4_ROWS, T4_BN);
    const int total = my_tiles * units_per_tile;
    const uint32_t d = tmem + (uint32_t)(b * T4_BN);
    bool ok = true;
    for (int u = b; u < total && ok; u += 2) {
      if (!mbar_wait_timed(&acc_empty[b], ((u >> 1) & 1) ^ 1, tmo, abort_flag, 0)) {
        ok = false;
        break;
      }
      const int kt = u >> 2;  // the CTA's K-tile sequence number
      const int s = kt % NST;
      if (!mbar_wait_timed(&full[s], (kt / NST) & 1, tmo, abort_flag, 0)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t abase = smem_u32(smem + s * T4_STAGE);
      const uint64_t bd = sdesc_k_sw128(abase + A_TILE4);
      const int st = u & 3;  // one step: the exact sums of its 4 groups
      mma_f16(d, sdesc_k_sw128(abase) + 2 * st, bd + 2 * st, idesc, 0u);
      mma_commit(&acc_full[b]);
    }
    if (!ok && !*abort_flag) fail();
    // all MMAs issued by both threads are complete once the drain barrier flips
    mma_commit(drain_bar);
    mbar_wait_bounded(drain_bar, 0, T4_DRAIN_LIMIT);
  }

  // ------------------------------------------------------------------ epilogue
  if (warp < T4_EPI_WARPS) {
    const int quarter = warp & 3, half = warp >> 2;
    const int mp = 8 * quarter + (lane >> 2);  // filter of the tile
    const int j = lane & 3;                    // group slot of this TMEM lane
    const uint32_t tbase = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(T4_EPI_COLS * half);
    const bool leader = threadIdx.x == 0;
    int u = 0;  // drain units of this CTA so far
    bool ok = true;
    for (int tl = 0; tl < my_tiles; ++tl) {
      int gi, mt;
      int64_t p0;
      tile_coords4(a, (int)blockIdx.x + tl * (int)gridDim.x, gi, mt, p0);
      const int local = mt * T4_FM + mp;
      const int m = gi * g.Mg + local;
      const bool mok = local < g.Mg;
      const int64_t pbase = p0 + T4_EPI_COLS * half;
      for (int k = 0; k < units_per_tile; ++k, ++u) {
        if (!ok) continue;
        const int b = u & 1;
        if (!mbar_wait_warp(&acc_full[b], (u >> 1) & 1, tmo, abort_flag)) {
          ok = false;
          continue;
        }
        if (leader && (u & 3) == 3) mbar_arrive(&empty[(u >> 2) % NST]);  // the K-tile's MMAs have completed: refill its stage
        tc_fence_after();
        const uint32_t ta = tbase + (uint32_t)(b * T4_BN);
        // exact sums of group 16 kt + 4 step + j, filter m, positions pbase + i
        const int grp = 16 * (k >> 2) + 4 * (k & 3) + j;
        int32_t* srow = a.sums + ((int64_t)(mok ? m : 0) * g.ng + (grp < g.ng ? grp : 0)) * g.P;
#pragma unroll
        for (int c = 0; c < T4_EPI_COLS / 16; ++c) {
          uint32_t r[16];
          tmem_ld16(ta + 16 * c, r);
          tmem_ld_wait_regs16(r);
          if (c == T4_EPI_COLS / 16 - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[b]);
          }
          if (mok && grp < g.ng) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int64_t p = pbase + 16 * c + i;
              if (p < g.P) srow[p] = __float2int_rn(__uint_as_float(r[i]));
            }
          }
        }
      }
      if (!ok && !*abort_flag) fail();
      if (named_bar_or(BAR_EPI4, 32 * T4_EPI_WARPS, !ok)) break;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == T4_MMA_WARP) {
    tc_fence_after();
    tmem_dealloc(tmem, T4_TMEM_COLS);
  }
}

template <bool TMAP>
fgq_status launch_tc4(const T4Args& args, int grid, cudaStream_t s) {
  if (!tc::smem_attr_once<tc4_sums_kernel<TMAP>>(T4_SMEM)) return FGQ_ERR_CUDA;
  return after_launch(launch_pdl(tc4_sums_kernel<TMAP>, dim3(grid), dim3(T4_THREADS), T4_SMEM, s, args));
}

}  // namespace

bool tc4_supports(const Geom& g) {
  if (g.G != 4) return false;
  if (g.P >= (int64_t)1 << 31) return false;  // positions decoded in 32 bits
  // every K-tile inside one filter tap (conv) or row (GEMM); activation boxes by 2D or
  // im2col maps of the fp16 copy
  return tc::act16_supported(g);
}

fgq_status launch_tc4_sums(const void* act, const Geom& g, const uint32_t* codes, int32_t* sums, unsigned int* err,
                           cudaStream_t s) {
  if (!tc4_supports(g)) return FGQ_ERR_UNSUPPORTED;
  T4Args a;
  memset(&a, 0, sizeof a);
  a.sums = sums;
  a.err = err;
  a.g = g;
  a.mtiles = (g.Mg + T4_FM - 1) / T4_FM;
  a.ptiles = (int)((g.P + T4_BN - 1) / T4_BN);
  a.ktiles = g.Kp / T4_KT;
  a.ntiles = g.groups * a.mtiles * a.ptiles;
  // a test may shorten the waits (debug_wait_limit_us), never the final drains
  const int64_t lim_us = debug_wait_limit_us();
  a.timeout_ns = lim_us < 0 ? T4_TIMEOUT_NS : (uint64_t)lim_us * 1000u;

  // one temporary from the stream-ordered pool: the block-diagonal ternary operand A' and the
  // activations in fp16
  const int64_t arows = (int64_t)g.groups * a.mtiles * T4_ROWS;
  const size_t diag_bytes = (size_t)arows * g.Kp * 2;
  const size_t x16_bytes = (size_t)tc::act16_elems(g) * 2;
  void* tmp = scratch_alloc(diag_bytes + x16_bytes, s);
  if (!tmp) return FGQ_ERR_CUDA;
  uint8_t* diag = static_cast<uint8_t*>(tmp);
  uint8_t* x16 = diag + diag_bytes;
  const int ksplit = (g.Kp / 8 + PREP4_CHUNKS - 1) / PREP4_CHUNKS;
  const int fold_blocks = g.groups * a.mtiles * ksplit;
  const prep::ActSrc src = prep::act_src(act, g);
  const int xb = prep::blocks_for(src.nchunks);
  fgq_status st = after_launch(launch_pdl(prep4_kernel, dim3(fold_blocks + xb), dim3(256), 0, s, codes, g.wrow, g.ng,
                                          g.Kp, g.Mg, a.mtiles, ksplit, reinterpret_cast<uint4*>(diag), fold_blocks,
                                          src, reinterpret_cast<uint4*>(x16)));
  if (st == FGQ_OK && !make_map_2d(&a.a_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, diag, (uint64_t)g.Kp, (uint64_t)arows,
                                   (uint64_t)g.Kp * 2, T4_KT, T4_ROWS, CU_TENSOR_MAP_SWIZZLE_128B))
    st = FGQ_ERR_CUDA;
  if (st == FGQ_OK && !tc::act16_map(&a.act_map, x16, g, T4_BN)) st = FGQ_ERR_CUDA;
  if (st == FGQ_OK) {
    const int sms = device_sms();
    const int grid = a.ntiles < sms ? a.ntiles : sms;
    st = tc::act_pointwise(g) ? launch_tc4<true>(a, grid, s) : launch_tc4<false>(a, grid, s);
  }
  // the temporary returns to the pool once the work queued on s before this point is done
  if (cudaFreeAsync(tmp, s) != cudaSuccess && st == FGQ_OK) st = FGQ_ERR_CUDA;
  return st;
}

}  // namespace fgq
