// LSTM training and inference kernels with the products on the tensor cores
// (weights as their BF16 copies, FP32 activations and gradients as exact sums
// of three BF16 parts).
#pragma once
#include "rpod_internal.cuh"

namespace rpod {

// An FP32 matrix as three BF16 ones (parts of every value, summing to it
// exactly), row-major; ld a multiple of 8, so every row starts on 16 bytes.
struct Parts {
  __nv_bfloat16* p;    // null: no matrix
  int64_t plane;       // elements from one part to the next
  int ld;
  __host__ __device__ Parts rows(int64_t r) const { return {p + r * ld, plane, ld}; }
};
inline int parts_ld(int cols) { return (cols + 7) / 8 * 8; }

// One cell of a forward phase: z = x W_x^T + h_prev W_h^T + b, gates, c, h.
struct LstmFwdCell {
  Parts x, hprev;               // B x Il, B x H (hprev null: zero)
  const float* cprev;           // B x H (null: zero)
  const __nv_bfloat16* Wx;      // 4H x Il
  const __nv_bfloat16* Wh;      // 4H x H
  const float* bias;            // 4H
  float *c, *gates;             // B x H, B x 4H
  Parts h;                      // B x H
  float* hf;                    // h in FP32 (null: not needed)
  Parts xd;                     // masked h for the layer above (null: no dropout)
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
// gradients dz.
struct LstmBwdCell {
  Parts A[2];
  const __nv_bfloat16* W[2];
  int K[2];                     // 0: no segment
  const unsigned char* keep;    // of segment 0
  const float *c, *cprev;       // cprev null: zero
  const float* gates;
  float* dc;                    // in (unless first) and out
  Parts dz;                     // B x 4H
  int first;                    // dc starts from zero
};
struct LstmBwd {
  LstmBwdCell cell[8];
  int cells, B, H;
  float drop_scale;
};

// out (M x N row-major) = sum_k A(k, i) X(k - shift, j), k < K; rows k < shift
// count as zero.
struct LstmGradEntry {
  Parts A, X;
  float* out;
  int64_t K;
  int M, N, shift, tile0;
};
struct LstmGrad {
  LstmGradEntry e[17];
  int entries, tiles;
};

// out[c] = sum_i in(i, c)
struct LstmSumEntry {
  Parts in;
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

// Parts of the windows, time-major: row t B + b from X[b sb + t st + k].
cudaError_t lstm_input_parts(cudaStream_t st, int B, int T, int I, const float* X, int64_t sb, int64_t stt,
                             Parts out);
cudaError_t lstm_fwd_phase(cudaStream_t st, const LstmFwd& a);
cudaError_t lstm_bwd_phase(cudaStream_t st, const LstmBwd& a);
cudaError_t lstm_weight_grads(cudaStream_t st, LstmGrad& a);
cudaError_t lstm_sums(cudaStream_t st, LstmSums& a);
// y = h W_y^T + b_y; with a target dy = 2 (y - t) / (B O) and the shares of
// sum (y - t)^2 (one per eight rows).
int lstm_head_blocks(int B);
cudaError_t lstm_head(cudaStream_t st, int B, int O, int H, const float* h, const __nv_bfloat16* Wy,
                      const float* by, float* y, const float* tgt, Parts dy, double* lpart);

}  // namespace rpod
