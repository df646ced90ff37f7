// LSTM training and inference kernels with the products on the tensor cores
// (weights as their BF16 copies, FP32 activations and gradients as exact sums
// of three BF16 parts).
#pragma once
#include "rpod_internal.cuh"

namespace rpod {

// One cell of a forward phase: z = x W_x^T + h_prev W_h^T + b, gates, c, h.
struct LstmFwdCell {
  const float* x;               // B x Il
  const float* hprev;           // B x H (null: zero)
  const float* cprev;           // B x H (null: zero)
  const __nv_bfloat16* Wx;      // 4H x Il
  const __nv_bfloat16* Wh;      // 4H x H
  const float* bias;            // 4H
  float *c, *h, *gates;         // B x H, B x H, B x 4H
  float* xd;                    // masked h for the layer above (null: no dropout)
  unsigned char* keep;          // its keep bits
  int Il;
  uint64_t drop_layer;          // the layer above, and the first element's index t B H
  int64_t drop_e0;
};
struct LstmFwd {
  LstmFwdCell cell[8];
  int cells, B, H;
  uint64_t drop_seed, drop_pass, drop_thr;
  float drop_scale;
};

// One cell of a backward phase: dh = sum over the segments A W (A B x K, W K x
// H row-major; the first is masked by `keep` when not null), then the gate
// gradients in place of the gates.
struct LstmBwdCell {
  const float* A[2];
  const __nv_bfloat16* W[2];
  int K[2];                     // 0: no segment; lda = K
  const unsigned char* keep;    // of segment 0
  const float *c, *cprev;       // cprev null: zero
  float *gates, *dc;            // gates in, dz out; dc in (unless first) and out
  int first;                    // dc starts from zero
};
struct LstmBwd {
  LstmBwdCell cell[8];
  int cells, B, H;
  float drop_scale;
};

// out (M x N row-major) = sum_k A[k lda + i] X[k ldx + j]; rows of X below
// `zero` count as zero.
struct LstmGradEntry {
  const float *A, *X;
  float* out;
  int64_t K;
  int lda, ldx, M, N, zero, tile0;
};
struct LstmGrad {
  LstmGradEntry e[17];
  int entries, tiles;
};

// out[c] = sum_i in[i N + c]
struct LstmSumEntry {
  const float* in;
  float* out;
  int64_t rows;
  int N, block0;
};
struct LstmSums {
  LstmSumEntry e[9];
  int entries, blocks;
  const double* lpart;          // loss shares of the head, summed into *loss
  int nlpart;
  double lcount;
  float* loss;
};

cudaError_t lstm_fwd_phase(cudaStream_t st, const LstmFwd& a);
cudaError_t lstm_bwd_phase(cudaStream_t st, const LstmBwd& a);
cudaError_t lstm_weight_grads(cudaStream_t st, LstmGrad& a);
cudaError_t lstm_sums(cudaStream_t st, LstmSums& a);
// y = h W_y^T + b_y; with a target dy = 2 (y - t) / (B O) and the shares of
// sum (y - t)^2 (one per eight rows).
int lstm_head_blocks(int B);
cudaError_t lstm_head(cudaStream_t st, int B, int O, int H, const float* h, const __nv_bfloat16* Wy,
                      const float* by, float* y, const float* tgt, float* dy, double* lpart);

}  // namespace rpod
