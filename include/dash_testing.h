/*
 * dash_testing.h -- test hooks of the halted-prefill library (libdash.so).
 *
 * Not part of the product interface (dash.h): entry points that exist so that a test can drive
 * the library into a corner its normal inputs never reach.  Conventions as in dash.h (device
 * pointers, `stream` is a cudaStream_t passed as void*, int status returned).
 */
#ifndef DASH_TESTING_H_
#define DASH_TESTING_H_

#include <stddef.h>
#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

/* dash_compact (dash.h; the single-pass compaction of Sec. 3.4 / Alg. 1 "gathering tokens") on its
 * look-back path, whatever the size, with a stall planted: the tile ticket starts at 1, so no CTA
 * ever takes tile 0, and tile 1 looks back at a state word that nobody publishes.  Every device-side
 * wait of the library is bounded: after `spin_limit` polls (1 .. 2^22) the waiting tile gives up,
 * sets DASH_ERR_TIMEOUT in the device status word (dash_check_status returns it once and clears it),
 * takes 0 as its base and publishes, so that every later tile finishes and the kernel returns.
 * No row tensors are moved; idx_out [n], cu_out [S+1], n_out_dev as in dash_compact (their contents
 * are unspecified after a timeout; everything written stays inside the buffers).  n >= 64.
 * ws: dash_workspace_bytes(DASH_WS_COMPACT, n, S, ...). */
int dash_testing_compact_stalled(const uint8_t* mask, int64_t n, const int32_t* cu_in, int S,
                                 int32_t* idx_out, int32_t* cu_out, int32_t* n_out_dev,
                                 uint32_t spin_limit, void* ws, size_t ws_bytes, void* stream);

/* Into how many shares a block step deals out the K steps (64 deep) of a bf16 projection C[n, N] = A[n, K] W[K, N] on the
 * current device, 0: none, the projection runs in whole tiles (256 x 256).  A share runs through ceil(N / 256) * ceil(K / 64) /
 * shares steps, tile after tile along N, for every row of tiles.  Pure host function. */
int dash_testing_gemm_groups(int64_t n, int64_t N, int64_t K);

/* C [n, N] = A [n, K] W [K, N], bf16, contiguous, in tiles cut along K as a block step cuts them (DASH_ERR_UNSUPPORTED where dash_testing_gemm_groups is 0).
 * ws: the arrival counters -- 32-bit words, one per tile, CTA of the pair and epilogue warp, tile 0 first, 74 x 4 x 16 of them on 148 SMs --, then the
 * partial tiles, 512 KB per share and row of tiles.  The counters are cleared on `stream` first, as a step does.
 * stall = 1: the first counter then starts at 1, so that the pair that takes itself for the last one of rows 64 .. 95, columns 0 .. 127 waits for parts that
 * do not add up: after `spin_limit` polls (1 .. 2^22) it gives up, sets DASH_ERR_TIMEOUT in the device status word, leaves these rows and columns
 * of C unwritten and the counter as it is, and the kernel returns. */
int dash_testing_gemm_cut(const void* A, const void* W, void* C, int64_t n, int64_t N, int64_t K, int stall, uint32_t spin_limit,
                          void* ws, size_t ws_bytes, void* stream);

/* Shared memory of a CTA of the decoding kernel for heads of D (-1: no such kernel).  Pure host function. */
int dash_testing_decode_smem_bytes(int D);

#ifdef __cplusplus
}
#endif
#endif /* DASH_TESTING_H_ */
