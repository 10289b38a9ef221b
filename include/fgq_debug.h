/*
 * fgq_debug.h -- test and benchmark controls of libfgq (not needed to use the library).
 *
 * Each control is per host thread: it affects only the calls that thread makes, so a
 * test or benchmark that sets one cannot change the kernels another thread's calls run.
 * Paper counterpart: none.
 */
#ifndef FGQ_DEBUG_H_
#define FGQ_DEBUG_H_

#include <stdint.h>

#include "fgq.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Contraction kernel families (see fgq_set_path / fgq_last_path). */
typedef enum {
  FGQ_PATH_AUTO = 0,   /* choose per shape: the few-row path for small GEMMs; with
                          fixed-point alphas the dense tensor-core path where it applies;
                          else the tensor cores where the shape is covered (G < 64, and G = 64
                          on channels that are no multiple of 64 with 18 groups or more, only
                          with at least 64 filters and 16 channels per conv group, and not the
                          smallest layers), else the CUDA cores */
  FGQ_PATH_SIMT = 1,   /* CUDA-core path: dp4a group sums, one FMA per group */
  FGQ_PATH_TC = 2,     /* tensor-core path (tcgen05): G in {64, 128} with K-tiles aligned to
                          the group; smaller G with the alphas folded into the weights on a
                          common grid per about 256 reduction elements (one or two pairs of
                          fp16 parts).  Forced: G in {4, 64, 128} with Cg a multiple of 64; the
                          automatic choice also takes it for G = 8, 16, 32 and other channel
                          counts */
  FGQ_PATH_GEMV = 3,   /* few-row path for GEMMs with P <= 8 (8-bit activations, Kred a
                          multiple of 16, G >= 4): one warp per filter row streams the
                          weights once; the automatic choice for such calls */
  FGQ_PATH_DENSE = 4   /* dense tensor-core path (tcgen05, any G, 8-bit activations, Cg a
                          multiple of 64): the alphas are folded into fp16 weights
                          alpha(m, k / G) * t[m][k] built per call, and one dense
                          contraction replaces the per-group multiplies.  Fixed-point alphas
                          fold into integer weights |a t| <= 255: the automatic choice for
                          fgq_gemm_qa / fgq_conv2d_qa (bounds in fgq.h).  With fp32 alphas
                          forcing this path returns FGQ_ERR_UNSUPPORTED unless
                          fgq_debug_allow_split_fold(1) was called on the thread: the alphas
                          are then split per filter row into two fp16 parts after scaling the
                          row's largest alpha into [2^14, 2^15), about 22 bits of alpha, and
                          the fp32 accumulator rounds once per 16 reduction elements -- a
                          numerical ablation of folding, outside the fgq_gemm tolerance. */
} fgq_path;

/*
 * Restricts this thread's contraction calls to one kernel family (FGQ_PATH_AUTO restores
 * the default per-shape choice).  A forced path that cannot run a shape makes the call
 * return FGQ_ERR_UNSUPPORTED.  Returns the previous setting, or -1 for an unknown path.
 */
int fgq_set_path(int path);

/* The kernel family (fgq_path) the most recent contraction call on this host thread used. */
int fgq_last_path(void);

/*
 * Shortens every mbarrier wait of the tensor-core contraction kernels launched by this
 * thread, and the wait for a tensor's maximum in fgq_quantize_act_batch, to about `us`
 * microseconds (us < 0 restores the kernels' own limits of one and two seconds per wait), so that a test can make a wait run out on purpose: the kernel then
 * records FGQ_ERR_TIMEOUT, each role leaves its loop, and the kernel waits -- with its
 * normal limits, which this setting never shortens -- for the copies and MMAs it issued,
 * frees its tensor memory and returns.  Returns the previous setting.
 */
int64_t fgq_debug_set_wait_limit_us(int64_t us);

/*
 * Makes this thread's requests for per-call temporaries of more than `bytes` bytes fail as they do on
 * a device without memory (bytes < 0, the default: none); returns the previous setting.
 */
int64_t fgq_debug_set_scratch_limit(int64_t bytes);

/*
 * Makes this thread's cooperative launches of more than `blocks` blocks (fgq_quantize_act_batch) fail as
 * they do in a context that can keep no more resident (blocks < 0, the default: none); returns the
 * previous setting.
 */
int64_t fgq_debug_set_resident_blocks(int64_t blocks);

/*
 * Lets FGQ_PATH_DENSE run calls with fp32 alphas on this thread through the split-fp16
 * ablation (allow != 0), outside the fgq_gemm tolerance; 0 restores FGQ_ERR_UNSUPPORTED.
 * Returns the previous setting.
 */
int fgq_debug_allow_split_fold(int allow);

/*
 * Remembered per thread and returned by the next call; no kernel depends on it (the CTA-pair
 * form of the G = 4 kernel that it used to select is gone: every contraction kernel runs on
 * single CTAs).  Returns the previous setting.
 */
int fgq_debug_cta_pairs(int on);

/*
 * At most k (1 .. 8, clamped) group ranges per output tile in this thread's G >= 64
 * tensor-core calls; returns the previous limit (default 8).  A layer with fewer output tiles
 * than SMs splits each tile's groups into ranges and adds the ranges' partial sums into the
 * output: the same sum in another fp32 rounding order, and with more than two ranges not
 * bit-reproducible from run to run.  k = 1 keeps whole tiles (one rounding order, the one
 * the fused requantizing entries use).
 */
int fgq_debug_max_ksplit(int k);

/* Group ranges per tile of this thread's last G >= 64 tensor-core call (1: whole tiles). */
int fgq_debug_last_ksplit(void);

/*
 * Self test of the wait that the warps of the tensor-core kernels share: the lanes of one warp wait,
 * for at most limit_us microseconds, on phases of which half are complete and half never will be.
 * Records FGQ_ERR_TIMEOUT if the wait expired for every lane, as it must (lanes that part here would
 * part ahead of warp-collective instructions), FGQ_ERR_UNSUPPORTED otherwise; read the result with
 * fgq_stream_status().
 */
fgq_status fgq_debug_selftest_warp_wait(uint32_t limit_us, cudaStream_t stream);

/*
 * The CUDA runtime error (a cudaError_t value) behind the last FGQ_ERR_CUDA that a kernel
 * launch of this thread returned, 0 if none; reading it clears it.  `name` receives the
 * runtime's name of that error (at most `len` bytes including the terminator) when non-null.
 */
int fgq_debug_last_cuda_error(char* name, size_t len);

#ifdef __cplusplus
}
#endif

#endif /* FGQ_DEBUG_H_ */
