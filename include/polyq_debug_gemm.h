/*
 * polyq_debug_gemm.h - the debug build's calls (see polyq_debug.h) that tests
 * use to know and to choose the prefill GEMM's kernel.
 */
#ifndef POLYQ_DEBUG_GEMM_H
#define POLYQ_DEBUG_GEMM_H

#include <stddef.h>
#include <stdint.h>

#include "polyq.h"

#ifdef __cplusplus
extern "C" {
#endif

/* polyq_linear_gemm with the kernel of a given token tile (32, 64, 128, 256 or
 * 512; 0: the one that the library would take).  M rounded up to the tile must
 * not exceed what the workspace of M is laid out for: the library's own tile
 * for M, a narrower one, or any for M > 256 (else POLYQ_EINVAL).  w_out as for
 * polyq_debug_gemm_weights, or NULL. */
int polyq_debug_linear_gemm(const polyq_dev_layer* layer, const void* X, int64_t M, float* Y,
                            void* workspace, size_t workspace_bytes, int tokens, uint16_t* w_out,
                            void* stream);

/* What polyq_linear_gemm launches for M tokens on the current device. */
typedef struct {
  int32_t tokens;   /* token tile of the kernel */
  int32_t pairs;    /* pairs of SMs that it runs on */
  int32_t ksplit;   /* ranges of a uniform split of K (1: none) */
  int32_t streamk;  /* 1: units shared along K by equal shares of K tiles */
  int64_t whole;    /* with streamk: units that one pair computes alone before */
} polyq_gemm_choice;
int polyq_debug_gemm_choice(const polyq_dev_layer* layer, int64_t M, polyq_gemm_choice* choice);

#ifdef __cplusplus
}
#endif
#endif /* POLYQ_DEBUG_GEMM_H */
