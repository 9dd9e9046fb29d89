// Internal interface of the tensor-core contraction used by the weight-gradient, input-gradient
// and Monte-Carlo entry points.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/bsp.h"

namespace bsp {

enum { EPI_STORE_F32 = 0, EPI_STORE_BF16 = 1, EPI_MC = 2, EPI_SPLIT = 3, EPI_MOMENTS = 4 };

// C[b][M][ldc] = alpha * A[M][K] * B[b][N][K]^T, alpha = (1/sa) * (1/sb); operands K-major.
// EPI_MC: S1 += C - ref, S2 += (C - ref)^2 for every batch in order (single [M][ldc] buffers).
// EPI_SPLIT: the result as two bf16 terms side by side, split[M][2 N] = hi | lo, besides C when given;
// with ref also the terms of ref - C below each other, diff[2 M][N].
// EPI_MOMENTS: S1 += f C, S2 += f C^2 with f = moment_scale, or without the sums so far (moment_first).
struct GemmArgs {
  int64_t M = 0, N = 0, K = 0;
  int nb = 1;
  bool fp8 = true;
  int a_fmt = 0, b_fmt = 0;            // bsp_format_t of A and B when fp8
  const void* A = nullptr;
  const void* B = nullptr;
  bool a_mn = false, b_mn = false;     // operand stored [K][M] / [K][N] (pitch lda / ldb) instead
  int64_t lda = 0, ldb = 0;            // row pitch in elements
  int64_t b_batch_stride = 0;          // elements between batches of B
  float sa = 1.f, sb = 1.f;
  const float* sa_dev = nullptr;
  const float* sb_dev = nullptr;
  int mode = EPI_STORE_F32;
  void* C = nullptr;
  int64_t ldc = 0;
  const float* ref = nullptr;
  float* S1 = nullptr;
  float* S2 = nullptr;
  uint16_t* split = nullptr;
  uint16_t* diff = nullptr;
  float moment_scale = 1.f;
  bool moment_first = false;
  bool mc_first = false;               // EPI_MC: the sums start here (S1 and S2 need not be cleared)
  float* split_ws = nullptr;           // EPI_MC: room for split ranges of draws (gemm_mc_split_bytes), or none
  size_t split_ws_bytes = 0;
  bsp_diag_t* diag = nullptr;
};

int gemm_run(const GemmArgs& g, cudaStream_t st);

// Workspace with which an EPI_MC contraction of nb draws can split the draws of its last wave of tiles.
size_t gemm_mc_split_bytes(int64_t M, int64_t N, int64_t K, bool fp8, int nb);
// bsp_linear_wgrad_mc with such a workspace; first: the sums start with these draws.
int linear_wgrad_mc_run(int64_t T, int64_t O, int64_t C, const uint8_t* dy_codes_t, bsp_quant_t q_dy,
                        const uint8_t* x_t_draws, bsp_quant_t q_x, int64_t ld_t, int n_draws, const float* g_ref, float* S1,
                        float* S2, bool first, float* split_ws, size_t split_ws_bytes, bsp_diag_t* diag, void* stream);

}  // namespace bsp
