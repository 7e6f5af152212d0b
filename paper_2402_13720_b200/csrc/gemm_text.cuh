// The weight GEMMs of a long block of known text (up to OURO_TEXT_ROWS rows): gemm_text.cu.
#pragma once

#include <cuda.h>

#include "ouro_internal.h"
#include "attn_fold.cuh"
#include "row_ops.cuh"

enum { TEXT_QKV = 0, TEXT_RESIDUAL = 1, TEXT_SWIGLU = 2 };

struct TextGemm {
  CUtensorMap a;                // activations [OURO_TEXT_ROWS][K], box 128 x 64
  CUtensorMap w[3];             // weight matrices stacked along the output dimension (q|k|v), or gate and up; box 64 x 64
  int w_tiles[3], w_rows[3];    // their tiles of 128 rows (gate and up: 64 of each) and their rows
  int w_count;
  int mode;
  int tiles, kb;                // all tiles, k-blocks of 64
  int t0, per;                  // where the decoding launches cut these tiles along K (ws::cut)
  int rows;
  // TEXT_QKV
  const int32_t *pos;
  const float *cos_t, *sin_t;
  __nv_bfloat16 *q_out, *k_out, *v_out;
  int head_dim, dq, dkv, L;
  // TEXT_RESIDUAL
  float *x;                     // [rows][ldx]
  int ldx;
  const __nv_bfloat16 *gain;
  __nv_bfloat16 *xb;
  float *ss_out;                // [tiles][OURO_TEXT_ROWS]
  // TEXT_SWIGLU
  __nv_bfloat16 *act;           // [rows][w_rows[0]]
  // RMSNorm of the activations (NULL: none)
  const float *ss_in;
  int ss_tiles;
  float ss_inv_d, eps;
  int *status;
  // filled in by the launch
  int units, token_tiles;
};

int text_gemm_setup();
void launch_text_gemm(TextGemm &g, int sms, cudaStream_t s);
void launch_text_embed(const rowops::Embed &e, int sms, cudaStream_t s);
void launch_text_fold(const fold::Params &f, int sms, cudaStream_t s);
