// LSTM cells (Sec. 4.3, Table tab:hyperparam) with the products on the tensor
// cores, one launch per anti-diagonal of layer x time.
//
// Cell (l, t) needs (l, t - 1) and (l - 1, t), so the cells with equal l + t run
// in one launch: L + T - 1 launches forward and as many backward, each with
// the whole product of its cells (input and recurrent, or the gradients from
// the layer above and from the next step) and the pointwise part as its
// epilogue.  The weight gradients of all layers are one launch, the bias
// gradients and the loss another.
//
// Arithmetic: FP32 activations and gradients are split exactly into three
// BF16 parts; times the BF16 weights that is three products, and six (those
// above 2^-26) for the FP32 x FP32 weight gradients.  The tensor core does not
// round its sums to nearest, so its accumulators (one for the products of the
// leading parts, one for the small ones) take 64 values of k and are then
// added to FP32 sums.
//
// A CTA has eight warps in WM x WN x WK: 16 batch rows each in m, WK shares of
// every 64 values of k.  Tiles are staged in shared memory (FP32 values split
// on the way, the next tile's loads in flight during the products) with rows
// of 144 bytes, so that ldmatrix touches every bank once.
//
// Bound: batch 512, 2 x 256: the mma.sync rate and the staging; small
// networks: launch latency.  Measured: LSTM_FIGURE
#include <algorithm>

#include "rpod_lstm_mma.cuh"

namespace rpod {
namespace {

constexpr int kLd = 72;  // bf16 per staged row: 64 values and 16 bytes

__device__ __forceinline__ float sigm_m(float x) { return 1.f / (1.f + __expf(-x)); }

// a = a1 + a2 + a3 for two values, packed as bf16 pairs (low half a)
__device__ __forceinline__ void parts3(float a, float b, uint32_t (&p)[3]) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  p[0] = __byte_perm(ua, ub, 0x7632);
  const float ra = a - __uint_as_float(ua & 0xffff0000u), rb = b - __uint_as_float(ub & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p[1]) : "f"(rb), "f"(ra));
  const float qa = ra - __uint_as_float(p[1] << 16), qb = rb - __uint_as_float(p[1] & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p[2]) : "f"(qb), "f"(qa));
}
__device__ __forceinline__ void ldm4(uint32_t (&r)[4], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldm4t(uint32_t (&r)[4], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Sums of a warp's 16 x 32 tile: FP32 sums of finished chunks, and the chunk in
// the tensor core (leading and small products).
struct Acc {
  float sum[4][4], hi[4][4], lo[4][4];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) sum[n][i] = hi[n][i] = lo[n][i] = 0.f;
  }
  __device__ __forceinline__ void flush() {
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        sum[n][i] += lo[n][i];
        sum[n][i] += hi[n][i];
        hi[n][i] = lo[n][i] = 0.f;
      }
  }
};

// The shares of the WK warps of a tile added into the first one's sums.
template <int TILES, int WK>
__device__ __forceinline__ void share_sum(Acc& acc, float* red, int tile, int wk, int lane) {
  if (WK == 1) return;
  __syncthreads();  // the staged tiles are free
  if (wk > 0) {
    float* d = red + ((size_t)((wk - 1) * TILES + tile) * 16) * 32 + lane;
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) d[(n * 4 + i) * 32] = acc.sum[n][i];
  }
  __syncthreads();
  if (wk == 0)
    for (int k = 0; k < WK - 1; ++k) {
      const float* d = red + ((size_t)(k * TILES + tile) * 16) * 32 + lane;
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc.sum[n][i] += d[(n * 4 + i) * 32];
    }
}

__device__ __forceinline__ uint32_t bf16_pair(const __nv_bfloat16* p, bool two, bool vec) {
  if (vec) return *(const uint32_t*)p;
  const uint32_t a = *(const uint16_t*)p;
  return two ? a | ((uint32_t)((const uint16_t*)p)[1] << 16) : a;
}

// ---- forward phase: blockIdx (batch tile, unit tile, cell)
template <int WM, int WN, int WK>
__global__ void __launch_bounds__(256) k_cell_fwd(const __grid_constant__ LstmFwd a) {
  constexpr int BM = 16 * WM, UN = 8 * WN, BR = 4 * UN;
  constexpr int NA = BM * 32 / 256, NB = BR * 32 / 256;  // pairs of a chunk per thread
  static_assert(WM * WN * WK == 8, "eight warps");
  __shared__ __align__(16) __nv_bfloat16 As[3][BM][kLd];
  __shared__ __align__(16) __nv_bfloat16 Bs[BR][kLd];
  __shared__ float red[WK > 1 ? (WK - 1) * WM * WN * 512 : 1];
  const LstmFwdCell& C = a.cell[blockIdx.z];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wk = warp % WK, wn = (warp / WK) % WN, wm = warp / (WK * WN);
  const int b0 = blockIdx.x * BM, u0 = blockIdx.y * UN;
  const int B = a.B, H = a.H;
  const int n0 = (C.Il + 63) / 64, nch = n0 + (C.hprev ? (H + 63) / 64 : 0);
  float2 ra[NA];
  uint32_t rb[NB];
  auto fetch = [&](int ch) {
    const bool first = ch < n0;
    const int K = first ? C.Il : H, k0 = (first ? ch : ch - n0) * 64;
    const float* A = first ? C.x : C.hprev;
    const __nv_bfloat16* W = first ? C.Wx : C.Wh;
    const bool even = (K & 1) == 0;
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int p = tid + 256 * i, r = b0 + (p >> 5), k = k0 + 2 * (p & 31);
      ra[i] = make_float2(0.f, 0.f);
      if (r < B && k < K) {
        const float* s = A + (int64_t)r * K + k;
        if (even) ra[i] = *(const float2*)s;
        else {
          ra[i].x = s[0];
          if (k + 1 < K) ra[i].y = s[1];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int p = tid + 256 * i, r = p >> 5, k = k0 + 2 * (p & 31);
      const int u = u0 + (r >> 5) * 8 + (r & 7), q = (r >> 3) & 3;  // row (group, gate, unit)
      rb[i] = (u < H && k < K) ? bf16_pair(W + ((int64_t)q * H + u) * K + k, k + 1 < K, even) : 0u;
    }
  };
  Acc acc;
  acc.clear();
  fetch(0);
  for (int ch = 0; ch < nch; ++ch) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int p = tid + 256 * i, r = p >> 5, k = 2 * (p & 31);
      uint32_t w[3];
      parts3(ra[i].x, ra[i].y, w);
#pragma unroll
      for (int q = 0; q < 3; ++q) *(uint32_t*)&As[q][r][k] = w[q];
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int p = tid + 256 * i;
      *(uint32_t*)&Bs[p >> 5][2 * (p & 31)] = rb[i];
    }
    __syncthreads();
    if (ch + 1 < nch) fetch(ch + 1);
    const int mat = lane >> 3, i8 = lane & 7;
#pragma unroll
    for (int ks = wk; ks < 4; ks += WK) {
      const int k = ks * 16;
      uint32_t fa[3][4], fb[2][4];
#pragma unroll
      for (int q = 0; q < 3; ++q) ldm4(fa[q], &As[q][wm * 16 + (mat & 1) * 8 + i8][k + (mat >> 1) * 8]);
#pragma unroll
      for (int h = 0; h < 2; ++h) ldm4(fb[h], &Bs[wn * 32 + h * 16 + (mat >> 1) * 8 + i8][k + (mat & 1) * 8]);
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const uint32_t x0 = fb[n >> 1][(n & 1) * 2], x1 = fb[n >> 1][(n & 1) * 2 + 1];
        mma16816(acc.lo[n], fa[2], x0, x1);
        mma16816(acc.lo[n], fa[1], x0, x1);
        mma16816(acc.hi[n], fa[0], x0, x1);
      }
    }
    acc.flush();
    __syncthreads();
  }
  share_sum<WM * WN, WK>(acc, red, wm * WN + wn, wk, lane);
  if (wk > 0) return;
  // n-tile q is gate q of this warp's eight units
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int b = b0 + wm * 16 + (lane >> 2) + (i >> 1) * 8, u = u0 + wn * 8 + 2 * (lane & 3) + (i & 1);
    if (b >= B || u >= H) continue;
    const int64_t e = (int64_t)b * H + u;
    float* g = C.gates + (int64_t)b * 4 * H + u;
    const float ig = sigm_m(acc.sum[0][i] + C.bias[u]), fg = sigm_m(acc.sum[1][i] + C.bias[H + u]);
    const float gg = tanhf(acc.sum[2][i] + C.bias[2 * H + u]), og = sigm_m(acc.sum[3][i] + C.bias[3 * H + u]);
    const float c = (C.cprev ? fg * C.cprev[e] : 0.f) + ig * gg;
    const float h = og * tanhf(c);
    C.c[e] = c;
    C.h[e] = h;
    g[0] = ig;
    g[H] = fg;
    g[2 * (int64_t)H] = gg;
    g[3 * (int64_t)H] = og;
    if (C.xd) {
      // the dropout mask of the layer above (see rpod_lstm_set_dropout)
      const int64_t de = C.drop_e0 + e;
      uint64_t w[4] = {(uint64_t)(de >> 2), C.drop_layer, a.drop_pass, 0ull};
      philox4x64_10(w, a.drop_seed, 1ull);
      const uint64_t x = (de & 2) ? ((de & 1) ? w[3] : w[2]) : ((de & 1) ? w[1] : w[0]);
      const bool keep = (x >> 11) >= a.drop_thr;
      C.xd[e] = keep ? h * a.drop_scale : 0.f;
      C.keep[e] = keep;
    }
  }
}

// ---- backward phase: blockIdx (batch tile, unit tile of 32 WN, cell)
template <int WM, int WN, int WK>
__global__ void __launch_bounds__(256) k_cell_bwd(const __grid_constant__ LstmBwd a) {
  constexpr int BM = 16 * WM, UN = 32 * WN, LB = UN + 8;
  constexpr int NA = BM * 32 / 256, NB = 64 * (UN / 2) / 256;
  static_assert(WM * WN * WK == 8, "eight warps");
  __shared__ __align__(16) __nv_bfloat16 As[3][BM][kLd];
  __shared__ __align__(16) __nv_bfloat16 Bs[64][LB];
  __shared__ float red[WK > 1 ? (WK - 1) * WM * WN * 512 : 1];
  const LstmBwdCell& C = a.cell[blockIdx.z];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wk = warp % WK, wn = (warp / WK) % WN, wm = warp / (WK * WN);
  const int b0 = blockIdx.x * BM, u0 = blockIdx.y * UN;
  const int B = a.B, H = a.H;
  const int n0 = (C.K[0] + 63) / 64, nch = n0 + (C.K[1] + 63) / 64;
  float2 ra[NA];
  uint32_t rb[NB];
  auto fetch = [&](int ch) {
    const int sg = ch < n0 ? 0 : 1;
    const int K = C.K[sg], k0 = (sg ? ch - n0 : ch) * 64;
    const float* A = C.A[sg];
    const __nv_bfloat16* W = C.W[sg];
    const bool even = (K & 1) == 0, heven = (H & 1) == 0;
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int p = tid + 256 * i, r = b0 + (p >> 5), k = k0 + 2 * (p & 31);
      ra[i] = make_float2(0.f, 0.f);
      if (r < B && k < K) {
        const float* s = A + (int64_t)r * K + k;
        if (even) ra[i] = *(const float2*)s;
        else {
          ra[i].x = s[0];
          if (k + 1 < K) ra[i].y = s[1];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int p = tid + 256 * i, k = k0 + p / (UN / 2), u = u0 + 2 * (p % (UN / 2));
      rb[i] = (u < H && k < K) ? bf16_pair(W + (int64_t)k * H + u, u + 1 < H, heven) : 0u;
    }
  };
  Acc acc;
  acc.clear();
  if (nch > 0) fetch(0);
  for (int ch = 0; ch < nch; ++ch) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int p = tid + 256 * i, r = p >> 5, k = 2 * (p & 31);
      uint32_t w[3];
      parts3(ra[i].x, ra[i].y, w);
#pragma unroll
      for (int q = 0; q < 3; ++q) *(uint32_t*)&As[q][r][k] = w[q];
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int p = tid + 256 * i;
      *(uint32_t*)&Bs[p / (UN / 2)][2 * (p % (UN / 2))] = rb[i];
    }
    __syncthreads();
    if (ch + 1 < nch) fetch(ch + 1);
    const int mat = lane >> 3, i8 = lane & 7;
#pragma unroll
    for (int ks = wk; ks < 4; ks += WK) {
      const int k = ks * 16;
      uint32_t fa[3][4], fb[2][4];
#pragma unroll
      for (int q = 0; q < 3; ++q) ldm4(fa[q], &As[q][wm * 16 + (mat & 1) * 8 + i8][k + (mat >> 1) * 8]);
#pragma unroll
      for (int h = 0; h < 2; ++h) ldm4t(fb[h], &Bs[k + (mat & 1) * 8 + i8][wn * 32 + h * 16 + (mat >> 1) * 8]);
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const uint32_t x0 = fb[n >> 1][(n & 1) * 2], x1 = fb[n >> 1][(n & 1) * 2 + 1];
        mma16816(acc.lo[n], fa[2], x0, x1);
        mma16816(acc.lo[n], fa[1], x0, x1);
        mma16816(acc.hi[n], fa[0], x0, x1);
      }
    }
    acc.flush();
    __syncthreads();
    if (ch == n0 - 1 && C.keep) {
      // what came through the dropout of the layer above
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int b = b0 + wm * 16 + (lane >> 2) + (i >> 1) * 8;
          const int u = u0 + wn * 32 + n * 8 + 2 * (lane & 3) + (i & 1);
          const bool keep = b < B && u < H && C.keep[(int64_t)b * H + u];
          acc.sum[n][i] = keep ? acc.sum[n][i] * a.drop_scale : 0.f;
        }
    }
  }
  share_sum<WM * WN, WK>(acc, red, wm * WN + wn, wk, lane);
  if (wk > 0) return;
#pragma unroll
  for (int n = 0; n < 4; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int b = b0 + wm * 16 + (lane >> 2) + (i >> 1) * 8;
      const int u = u0 + wn * 32 + n * 8 + 2 * (lane & 3) + (i & 1);
      if (b >= B || u >= H) continue;
      const int64_t e = (int64_t)b * H + u;
      float* g = C.gates + (int64_t)b * 4 * H + u;
      const float ig = g[0], fg = g[H], gg = g[2 * (int64_t)H], og = g[3 * (int64_t)H];
      const float dh = acc.sum[n][i];
      const float tc = tanhf(C.c[e]);
      const float d_o = dh * tc;
      const float dcv = (C.first ? 0.f : C.dc[e]) + dh * og * (1.f - tc * tc);
      const float di = dcv * gg, dg = dcv * ig, df = C.cprev ? dcv * C.cprev[e] : 0.f;
      C.dc[e] = dcv * fg;
      g[0] = di * ig * (1.f - ig);
      g[H] = df * fg * (1.f - fg);
      g[2 * (int64_t)H] = dg * (1.f - gg * gg);
      g[3 * (int64_t)H] = d_o * og * (1.f - og);
    }
}

// ---- weight gradients: a 64 x 64 tile of one entry per CTA, warps 4 x 2
__global__ void __launch_bounds__(256) k_weight_grads(const __grid_constant__ LstmGrad a) {
  extern __shared__ __align__(16) __nv_bfloat16 sm[];
  typedef __nv_bfloat16 Tile[64][kLd];
  Tile* As = (Tile*)sm;         // [3][64 k][64 m]
  Tile* Xs = As + 3;            // [3][64 k][64 n]
  int ei = 0;
  while (ei + 1 < a.entries && (int)blockIdx.x >= a.e[ei + 1].tile0) ++ei;
  const LstmGradEntry& E = a.e[ei];
  const int nt = (E.N + 63) / 64, tile = blockIdx.x - E.tile0;
  const int m0 = (tile / nt) * 64, c0 = (tile % nt) * 64;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wm = warp >> 1, wn = warp & 1;
  const bool ea = (E.lda & 1) == 0, ex = (E.ldx & 1) == 0;
  float2 ra[8], rx[8];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int p = tid + 256 * i, c = 2 * (p & 31);
      const int64_t k = k0 + (p >> 5);
      ra[i] = rx[i] = make_float2(0.f, 0.f);
      if (k >= E.K) continue;
      if (m0 + c < E.M) {
        const float* s = E.A + k * E.lda + m0 + c;
        if (ea && m0 + c + 1 < E.M) ra[i] = *(const float2*)s;
        else {
          ra[i].x = s[0];
          if (m0 + c + 1 < E.M) ra[i].y = s[1];
        }
      }
      if (c0 + c < E.N && k >= E.zero) {
        const float* s = E.X + k * E.ldx + c0 + c;
        if (ex && c0 + c + 1 < E.N) rx[i] = *(const float2*)s;
        else {
          rx[i].x = s[0];
          if (c0 + c + 1 < E.N) rx[i].y = s[1];
        }
      }
    }
  };
  Acc acc;
  acc.clear();
  fetch(0);
  for (int64_t k0 = 0; k0 < E.K; k0 += 64) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int p = tid + 256 * i, r = p >> 5, c = 2 * (p & 31);
      uint32_t w[3];
      parts3(ra[i].x, ra[i].y, w);
#pragma unroll
      for (int q = 0; q < 3; ++q) *(uint32_t*)&As[q][r][c] = w[q];
      parts3(rx[i].x, rx[i].y, w);
#pragma unroll
      for (int q = 0; q < 3; ++q) *(uint32_t*)&Xs[q][r][c] = w[q];
    }
    __syncthreads();
    if (k0 + 64 < E.K) fetch(k0 + 64);
    const int mat = lane >> 3, i8 = lane & 7;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const int k = ks * 16;
      uint32_t fa[3][4];
#pragma unroll
      for (int q = 0; q < 3; ++q) ldm4t(fa[q], &As[q][k + (mat >> 1) * 8 + i8][wm * 16 + (mat & 1) * 8]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t fx[3][4];
#pragma unroll
        for (int q = 0; q < 3; ++q) ldm4t(fx[q], &Xs[q][k + (mat & 1) * 8 + i8][wn * 32 + h * 16 + (mat >> 1) * 8]);
#pragma unroll
        for (int n2 = 0; n2 < 2; ++n2) {
          const int n = 2 * h + n2, j = 2 * n2;
          mma16816(acc.lo[n], fa[2], fx[0][j], fx[0][j + 1]);
          mma16816(acc.lo[n], fa[0], fx[2][j], fx[2][j + 1]);
          mma16816(acc.lo[n], fa[1], fx[1][j], fx[1][j + 1]);
          mma16816(acc.lo[n], fa[1], fx[0][j], fx[0][j + 1]);
          mma16816(acc.lo[n], fa[0], fx[1][j], fx[1][j + 1]);
          mma16816(acc.hi[n], fa[0], fx[0][j], fx[0][j + 1]);
        }
      }
    }
    acc.flush();
    __syncthreads();
  }
#pragma unroll
  for (int n = 0; n < 4; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = m0 + wm * 16 + (lane >> 2) + (i >> 1) * 8;
      const int c = c0 + wn * 32 + n * 8 + 2 * (lane & 3) + (i & 1);
      if (r < E.M && c < E.N) E.out[(int64_t)r * E.N + c] = acc.sum[n][i];
    }
}

// ---- column sums (32 columns per block, 32 slices of rows, compensated FP32
// sums combined in FP64) and, in the last block, the loss
__global__ void __launch_bounds__(1024) k_lstm_sums(const __grid_constant__ LstmSums a) {
  __shared__ double part[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if ((int)blockIdx.x == a.blocks) {
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int i = 0; i < a.nlpart; ++i) s += a.lpart[i];
      *a.loss = (float)(s / a.lcount);
    }
    return;
  }
  int ei = 0;
  while (ei + 1 < a.entries && (int)blockIdx.x >= a.e[ei + 1].block0) ++ei;
  const LstmSumEntry& E = a.e[ei];
  const int c = (blockIdx.x - E.block0) * 32 + tx;
  float s = 0.f, err = 0.f;
  if (c < E.N) {
#pragma unroll 8
    for (int64_t i = ty; i < E.rows; i += 32) {
      const float x = E.in[i * E.N + c], t = s + x, bp = t - s;
      err += (s - (t - bp)) + (x - bp);
      s = t;
    }
  }
  part[ty][tx] = (double)s + (double)err;
  __syncthreads();
  if (ty == 0 && c < E.N) {
    double t = 0.0;
    for (int k = 0; k < 32; ++k) t += part[k][tx];
    E.out[c] = (float)t;
  }
}

// ---- head: a warp per batch row, lanes over the hidden units
constexpr int kHeadRows = 8;
__global__ void __launch_bounds__(kHeadRows * 32)
k_head(int B, int O, int H, const float* __restrict__ h, const __nv_bfloat16* __restrict__ Wy,
       const float* __restrict__ by, float* __restrict__ y, const float* __restrict__ tgt,
       float* __restrict__ dy, double* __restrict__ lpart) {
  __shared__ double red[kHeadRows];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * kHeadRows + warp;
  double s = 0.0;
  if (b < B) {
    const float* hb = h + (int64_t)b * H;
    for (int o0 = 0; o0 < O; o0 += 8) {
      float v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = 0.f;
      for (int k = lane; k < H; k += 32) {
        const float x = hb[k];
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (o0 + j < O) v[j] = fmaf(__bfloat162float(Wy[(int64_t)(o0 + j) * H + k]), x, v[j]);
      }
      // transposing butterfly: lane group lane >> 2 ends with output j
#pragma unroll
      for (int n = 4, m = 16; n >= 1; n >>= 1, m >>= 1)
#pragma unroll
        for (int i = 0; i < n; ++i) {
          const bool up = (lane & m) != 0;
          const float got = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + n], m);
          v[i] = (up ? v[i + n] : v[i]) + got;
        }
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
      const int o = o0 + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
      if ((lane & 3) == 0 && o < O) {
        const float z = v[0] + by[o];
        y[(int64_t)b * O + o] = z;
        if (tgt) {
          const float d = z - tgt[(int64_t)b * O + o];
          dy[(int64_t)b * O + o] = 2.f / ((float)B * (float)O) * d;
          s += (double)d * d;
        }
      }
    }
  }
  if (!tgt) return;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) red[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < kHeadRows; ++k) t += red[k];
    lpart[blockIdx.x] = t;
  }
}

}  // namespace

// Up to 32 rows a batch tile of 16 with four shares of k (more CTAs, each chunk
// of k one step per warp); above, tiles of 64 rows.
cudaError_t lstm_fwd_phase(cudaStream_t st, const LstmFwd& a) {
  if (a.B <= 32)
    k_cell_fwd<1, 2, 4><<<dim3((a.B + 15) / 16, (a.H + 15) / 16, a.cells), 256, 0, st>>>(a);
  else
    k_cell_fwd<4, 2, 1><<<dim3((a.B + 63) / 64, (a.H + 15) / 16, a.cells), 256, 0, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

cudaError_t lstm_bwd_phase(cudaStream_t st, const LstmBwd& a) {
  if (a.B <= 32)
    k_cell_bwd<1, 1, 8><<<dim3((a.B + 15) / 16, (a.H + 31) / 32, a.cells), 256, 0, st>>>(a);
  else
    k_cell_bwd<4, 1, 2><<<dim3((a.B + 63) / 64, (a.H + 31) / 32, a.cells), 256, 0, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

cudaError_t lstm_weight_grads(cudaStream_t st, LstmGrad& a) {
  a.tiles = 0;
  for (int i = 0; i < a.entries; ++i) {
    a.e[i].tile0 = a.tiles;
    a.tiles += ((a.e[i].M + 63) / 64) * ((a.e[i].N + 63) / 64);
  }
  const int smem = 6 * 64 * kLd * 2;
  const cudaError_t e = cudaFuncSetAttribute(k_weight_grads, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  k_weight_grads<<<a.tiles, 256, smem, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

cudaError_t lstm_sums(cudaStream_t st, LstmSums& a) {
  a.blocks = 0;
  for (int i = 0; i < a.entries; ++i) {
    a.e[i].block0 = a.blocks;
    a.blocks += (a.e[i].N + 31) / 32;
  }
  k_lstm_sums<<<a.blocks + 1, 1024, 0, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

int lstm_head_blocks(int B) { return (B + kHeadRows - 1) / kHeadRows; }

cudaError_t lstm_head(cudaStream_t st, int B, int O, int H, const float* h, const __nv_bfloat16* Wy,
                      const float* by, float* y, const float* tgt, float* dy, double* lpart) {
  k_head<<<lstm_head_blocks(B), kHeadRows * 32, 0, st>>>(B, O, H, h, Wy, by, y, tgt, dy, lpart);
  note_launch();
  return cudaGetLastError();
}

}  // namespace rpod
