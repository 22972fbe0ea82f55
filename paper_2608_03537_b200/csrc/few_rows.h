// The fused kinds behind a GEMM of FEW ROWS (a decoding step, a small batch, the scores of a few heads): plan and launch.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "host_common.h"

namespace comfuse {

// How one call is cut (mt = 0: the call does not take this form).
struct FewRowsPlan {
  int mt = 0;         // rows per work item: the N dimension of the UMMA (16, 32 or 64)
  int nt = 0;         // 128-column tiles of the row per CTA (1 or 2)
  int ct = 0;         // CTAs that share a row's columns
  int ks = 0;         // CTAs that share the contraction of one column range; the cluster has ct * ks CTAs
  int nblocks = 1;    // 256-column blocks of the two-kernel form
  bool wide = false;  // two-kernel form: x leaves as fp16 with the blocks' statistics, the finishing kernel normalises it
};

struct FewRowsParams {
  int M, N, K, batch;
  int ct, ks, nblocks, groups;  // groups = row groups of mt rows
  float alpha, eps;
  int b_nk, wide, post_relu, no_activation;
  int causal;             // softmax kind
  float softcap;          // softmax kind, 0 = none
  const uint16_t* mask;   // softmax kind: additive [M, N] mask shared by the batches, or null
  const uint16_t* bias;
  const uint16_t* gamma;
  const uint16_t* beta;
  const uint16_t* residual;
  long long ldr, batch_stride_r;
  uint16_t* Y;
  long long ldy, batch_stride_y;
  float* row_max;
  int* row_argmax;
  float2* wide_partials;
  unsigned int* status;
  unsigned long long timeout_ns;
};

// `wide_block`: column block width of the two-kernel form the call would take otherwise (0: the row stays on chip).
// `ld_rows`, `ld_weights`: leading dimensions of the activations and of the weights; `b_nk`: weights stored [N, K].
FewRowsPlan few_rows_plan(int epi, int batch, int M, int N, int K, int wide_block, long long ld_rows, long long ld_weights, bool b_nk, const DeviceInfo& dev);
// tmW: the weights in boxes of 64 x 64 elements (either storage order); tmX: the rows in boxes of 64 elements x mt rows.
cudaError_t launch_few_rows(int epi, const FewRowsPlan& plan, const CUtensorMap& tmW, const CUtensorMap& tmX, FewRowsParams p,
                            cudaStream_t stream);

}  // namespace comfuse
