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
// BF16 parts; times the BF16 weights that is three products, and six for the
// FP32 x FP32 weight gradients (the three left out are at most 2^-23, 2^-23 and
// 2^-32 of a product, about 2^-26 with random signs).  The tensor core does not
// round its sums to nearest, so its accumulators (one for the products of the
// leading parts, one for the small ones) take 64 values of k and are then
// added to FP32 sums.
//
// A CTA has eight warps in WM x WN x WK: 16 batch rows each in m, WK shares of
// every 64 values of k.  Every activation and gradient is kept as its three
// parts, written once by the kernel that computes it (splitting in the readers
// was repeated by every CTA of a row and took more issue slots than the
// products), and staged by 16-byte cp.async two chunks ahead, in rows of 144
// bytes, so that ldmatrix touches every bank once.
//
// Bound: batch 512, 2 x 256: staging from L2 and the mma.sync rate (about 1000
// multiply-adds a clock and SM, a quarter of it for FP32 x FP32); small
// networks: launch latency.  Measured, loss and gradients at 2 x 256, window 10,
// batch 512: 685 us, 743 with each phase launched after the previous one's end (of
// these 11 forward phases 188, 11 backward ones 230, the weight gradients 239),
// 4045 us with FP32 products and about 100 launches; a training step at 3 x 50,
// batch 16: 157 us (1570 us).
#include <cooperative_groups.h>
#include <float.h>
#include <math.h>

#include <algorithm>
#include <utility>

#include "rpod_lstm_mma.cuh"

namespace rpod {
namespace {

constexpr int kLd = 72;  // bf16 per staged row: 64 values and 16 bytes

__device__ __forceinline__ float sigm_m(float x) { return 1.f / (1.f + __expf(-x)); }

// a = a1 + a2 + a3 for two values, packed as bf16 pairs (low half a).  INF: an
// infinity is (a, 0, 0).  The difference to its first part would be NaN, and
// with it every sum that the infinity alone leaves infinite (a window with an
// infinite entry saturates its gates, as with FP32 products).  Only what comes
// from outside can be infinite while the rest stays finite: inputs and targets.
template <bool INF>
__device__ __forceinline__ void parts3(float a, float b, uint32_t (&p)[3]) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  p[0] = __byte_perm(ua, ub, 0x7632);
  const float ra = INF && fabsf(a) == INFINITY ? 0.f : a - __uint_as_float(ua & 0xffff0000u);
  const float rb = INF && fabsf(b) == INFINITY ? 0.f : b - __uint_as_float(ub & 0xffff0000u);
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
  // The same with the rounding error of each sum (Knuth's TwoSum) kept with the
  // small products, for the weight gradients' many chunks: with plain sums the 80
  // of window 10, batch 512 left 1.3e-7 of error against 64 bits, now 1.1e-7, that
  // of FP32 products.  finish() adds what is left.
  __device__ __forceinline__ void flush_exact() {
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float s = sum[n][i], y = hi[n][i] + lo[n][i], t = s + y, b = t - s;
        lo[n][i] = (s - (t - b)) + (y - b);
        sum[n][i] = t;
        hi[n][i] = 0.f;
      }
  }
  __device__ __forceinline__ void finish() {
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) sum[n][i] += lo[n][i];
  }
};

// 16 x 32 x 16: FP32 operand in three parts times BF16, n-tile n's two registers
// in fb[n / 2]
__device__ __forceinline__ void products(Acc& acc, const uint32_t (&fa)[3][4], const uint32_t (&fb)[2][4]) {
#pragma unroll
  for (int n = 0; n < 4; ++n) mma16816(acc.lo[n], fa[2], fb[n >> 1][(n & 1) * 2], fb[n >> 1][(n & 1) * 2 + 1]);
#pragma unroll
  for (int n = 0; n < 4; ++n) mma16816(acc.hi[n], fa[0], fb[n >> 1][(n & 1) * 2], fb[n >> 1][(n & 1) * 2 + 1]);
#pragma unroll
  for (int n = 0; n < 4; ++n) mma16816(acc.lo[n], fa[1], fb[n >> 1][(n & 1) * 2], fb[n >> 1][(n & 1) * 2 + 1]);
}

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

// Two neighbours of a weight row; EVEN: every row length is even, so a pair is
// whole and aligned (`two` is read otherwise).  The choice is made at compile
// time: with a branch per pair the loads of a chunk took about 1000 clocks to
// issue.
template <bool EVEN>
__device__ __forceinline__ uint32_t ld_pair(const __nv_bfloat16* p, bool in, bool two) {
  uint32_t v = 0u;
  if (in) {
    if (EVEN) v = *(const uint32_t*)p;
    else {
      v = *(const uint16_t*)p;
      if (two) v |= (uint32_t)((const uint16_t*)p)[1] << 16;
    }
  }
  return v;
}
// 16 bytes to shared memory, of which `n` from memory and the rest zero.
__device__ __forceinline__ void cp16(__nv_bfloat16* dst, const __nv_bfloat16* src, int n) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// Rows [r0, r0 + ROWS) and columns [c0, c0 + 64) of a matrix's parts into
// dst[part][row][kLd]; zero outside of rows x cols.
template <int ROWS>
__device__ __forceinline__ void stage_parts(__nv_bfloat16* dst, const Parts& P, int64_t r0, int64_t rlo,
                                            int64_t rhi, int c0, int cols) {
  constexpr int N = 3 * ROWS * 8;  // pieces of 8 values
#pragma unroll
  for (int i = 0; i < (N + 255) / 256; ++i) {
    const int e = threadIdx.x + 256 * i;
    if (N % 256 != 0 && e >= N) break;
    const int c = (e & 7) * 8, r = (e >> 3) % ROWS, q = (e >> 3) / ROWS;
    const int64_t row = r0 + r;
    const int left = (cols - c0 - c) * 2;
    const bool in = row >= rlo && row < rhi && left > 0;
    cp16(dst + (q * ROWS + r) * kLd + c, in ? P.p + q * P.plane + row * P.ld + c0 + c : P.p,
         in ? (left < 16 ? left : 16) : 0);
  }
}
// the parts of a pair of neighbours (column even)
template <bool INF = false>
__device__ __forceinline__ void store_pair(const Parts& P, int64_t row, int col, float a, float b) {
  uint32_t w[3];
  parts3<INF>(a, b, w);
#pragma unroll
  for (int q = 0; q < 3; ++q) *(uint32_t*)(P.p + q * P.plane + row * P.ld + col) = w[q];
}
template <bool INF = false>
__device__ __forceinline__ void store_one(const Parts& P, int64_t row, int col, float a) {
  uint32_t w[3];
  parts3<INF>(a, 0.f, w);
#pragma unroll
  for (int q = 0; q < 3; ++q) *(uint16_t*)(P.p + q * P.plane + row * P.ld + col) = (uint16_t)w[q];
}

// ---- forward phase: blockIdx (batch tile, unit tile, cell)
template <int BM, int BR>
struct FwdStage {
  __nv_bfloat16 A[3][3][BM][kLd];  // [stage][part]
  __nv_bfloat16 B[2][BR][kLd];
};
template <int WM, int WN, int WK, bool EVEN>
__global__ void __launch_bounds__(256, 2) k_cell_fwd(const __grid_constant__ LstmFwd a) {
  constexpr int BM = 16 * WM, UN = 8 * WN, BR = 4 * UN;
  constexpr int NB = BR * 32 / 256;  // weight pairs of a chunk per thread
  static_assert(WM * WN * WK == 8, "eight warps");
  extern __shared__ __align__(16) uint8_t sm[];
  FwdStage<BM, BR>& S = *(FwdStage<BM, BR>*)sm;
  float* const red = (float*)sm;  // after the products
  const LstmFwdCell& C = a.cell[blockIdx.z];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wk = warp % WK, wn = (warp / WK) % WN, wm = warp / (WK * WN);
  const int b0 = blockIdx.x * BM, u0 = blockIdx.y * UN;
  const int B = a.B, H = a.H, Il = C.Il;
  const Parts x = C.x, hp = C.hprev;
  const __nv_bfloat16 *const Wx = C.Wx, *const Wh = C.Wh;
  const int n0 = (Il + 63) / 64, nch = n0 + (hp.p ? (H + 63) / 64 : 0);
  auto load_a = [&](int ch) {
    const bool first = ch < n0;
    if (ch < nch)
      stage_parts<BM>(&S.A[ch % 3][0][0][0], first ? x : hp, b0, 0, B, (first ? ch : ch - n0) * 64, first ? Il : H);
    cp_commit();
  };
  auto load_w = [&](int ch, uint32_t (&rb)[NB]) {
    if (ch >= nch) return;
    const bool first = ch < n0;
    const int K = first ? Il : H, k = (first ? ch : ch - n0) * 64 + 2 * lane;
    // staged row 8 i + warp: unit group i / 4, gate i % 4, unit `warp`
    const __nv_bfloat16* pw = (first ? Wx : Wh) + (int64_t)(u0 + warp) * K + k;
#pragma unroll
    for (int i = 0; i < NB; ++i)
      rb[i] = ld_pair<EVEN>(pw + (int64_t)((i & 3) * H + (i >> 2) * 8) * K,
                            k < K && u0 + (i >> 2) * 8 + warp < H, k + 1 < K);
  };
  pdl_trigger();
  uint32_t rb0[NB], rb1[NB];
  load_w(0, rb0);  // the weights are older than this pass
  load_w(1, rb1);
  // what the epilogue reads: rows (lane >> 2) + 8 h, units 2 (lane & 3) + j
  const int eb = b0 + wm * 16 + (lane >> 2), eu = u0 + wn * 8 + 2 * (lane & 3);
  float bias[4][2], cp[2][2];
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) bias[q][j] = eu + j < H ? C.bias[q * H + eu + j] : 0.f;
  pdl_wait();
  load_a(0);
  load_a(1);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      cp[h][j] = (C.cprev && eb + 8 * h < B && eu + j < H) ? C.cprev[(int64_t)(eb + 8 * h) * H + eu + j] : 0.f;
  }
  Acc acc;
  acc.clear();
  auto chunk = [&](int ch, uint32_t (&rb)[NB], __nv_bfloat16 (&Bs)[BR][kLd]) {
#pragma unroll
    for (int i = 0; i < NB; ++i) *(uint32_t*)&Bs[8 * i + warp][2 * lane] = rb[i];
    cp_wait<1>();
    __syncthreads();
    load_a(ch + 2);
    load_w(ch + 2, rb);
    const int mat = lane >> 3, i8 = lane & 7;
    auto& As = S.A[ch % 3];
#pragma unroll
    for (int ks = wk; ks < 4; ks += WK) {
      const int k = ks * 16;
      uint32_t fa[3][4], fb[2][4];
#pragma unroll
      for (int q = 0; q < 3; ++q) ldm4(fa[q], &As[q][wm * 16 + (mat & 1) * 8 + i8][k + (mat >> 1) * 8]);
#pragma unroll
      for (int h = 0; h < 2; ++h) ldm4(fb[h], &Bs[wn * 32 + h * 16 + (mat >> 1) * 8 + i8][k + (mat & 1) * 8]);
      products(acc, fa, fb);
    }
    acc.flush();
  };
  for (int ch = 0; ch < nch; ch += 2) {
    chunk(ch, rb0, S.B[0]);
    if (ch + 1 < nch) chunk(ch + 1, rb1, S.B[1]);
  }
  cp_wait<0>();
  share_sum<WM * WN, WK>(acc, red, wm * WN + wn, wk, lane);
  if (wk > 0) return;
  // n-tile q is gate q of this warp's eight units
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int b = eb + 8 * h;
    if (b >= B || eu >= H) continue;
    float hv[2], hd[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int i = 2 * h + j, u = eu + j;
      hv[j] = hd[j] = 0.f;
      if (u >= H) continue;
      const int64_t e = (int64_t)b * H + u;
      const float ig = sigm_m(acc.sum[0][i] + bias[0][j]), fg = sigm_m(acc.sum[1][i] + bias[1][j]);
      const float gg = tanhf(acc.sum[2][i] + bias[2][j]), og = sigm_m(acc.sum[3][i] + bias[3][j]);
      const float c = fg * cp[h][j] + ig * gg;
      hv[j] = og * tanhf(c);
      float* g = C.gates + (int64_t)b * 4 * H + u;
      C.c[e] = c;
      g[0] = ig;
      g[H] = fg;
      g[2 * (int64_t)H] = gg;
      g[3 * (int64_t)H] = og;
      if (C.hf) C.hf[e] = hv[j];
      if (C.xd.p) {
        // the dropout mask of the layer above (see rpod_lstm_set_dropout)
        const int64_t de = C.drop_e0 + e;
        uint64_t w[4] = {(uint64_t)(de >> 2), C.drop_layer, a.drop_pass, 0ull};
        philox4x64_10(w, a.drop_seed, 1ull);
        const uint64_t r = (de & 2) ? ((de & 1) ? w[3] : w[2]) : ((de & 1) ? w[1] : w[0]);
        const bool keep = (r >> 11) >= a.drop_thr;
        hd[j] = keep ? hv[j] * a.drop_scale : 0.f;
        C.keep[e] = keep;
      }
    }
    store_pair(C.h, b, eu, hv[0], hv[1]);
    if (C.xd.p) store_pair(C.xd, b, eu, hd[0], hd[1]);
  }
}

// ---- backward phase: blockIdx (batch tile, unit tile of 32 WN, cell and half)
template <int BM, int UN>
struct BwdStage {
  __nv_bfloat16 A[3][3][BM][kLd];  // [stage][part]
  __nv_bfloat16 B[2][64][UN + 8];
};
template <int WM, int WN, int WK, bool EVEN>
__global__ void __launch_bounds__(256, 2) k_cell_bwd(const __grid_constant__ LstmBwd a) {
  constexpr int BM = 16 * WM, UN = 32 * WN;
  constexpr int PR = UN / 2, KR = 256 / PR;  // pairs of a weight row, rows at a time
  constexpr int NB = 64 / KR;
  static_assert(WM * WN * WK == 8, "eight warps");
  extern __shared__ __align__(16) uint8_t sm[];
  BwdStage<BM, UN>& S = *(BwdStage<BM, UN>*)sm;
  float* const red = (float*)sm;  // after the products
  // A cluster of two CTAs shares a tile, one segment each; dh[half] takes the
  // halves' sums, and each CTA does the pointwise part of half of the rows.
  float(*const dh)[BM][UN] = (float(*)[BM][UN])(sm + sizeof(BwdStage<BM, UN>));
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int sg = (int)cl.block_rank();
  auto started = cl.barrier_arrive();
  const LstmBwdCell& C = a.cell[blockIdx.z >> 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wk = warp % WK, wn = (warp / WK) % WN, wm = warp / (WK * WN);
  const int b0 = blockIdx.x * BM, u0 = blockIdx.y * UN;
  const int B = a.B, H = a.H;
  const int K = C.K[sg], nch = (K + 63) / 64;
  const Parts A = C.A[sg];
  const __nv_bfloat16* const W = C.W[sg];
  const int bk = tid / PR, bu = 2 * (tid % PR);
  auto load_a = [&](int ch) {
    if (ch < nch) stage_parts<BM>(&S.A[ch % 3][0][0][0], A, b0, 0, B, ch * 64, K);
    cp_commit();
  };
  auto load_w = [&](int ch, uint32_t (&rb)[NB]) {
    if (ch >= nch) return;
    const int kw = ch * 64 + bk;
    const __nv_bfloat16* pw = W + (int64_t)kw * H + u0 + bu;
#pragma unroll
    for (int i = 0; i < NB; ++i)
      rb[i] = ld_pair<EVEN>(pw + i * KR * H, u0 + bu < H && kw + i * KR < K, u0 + bu + 1 < H);
  };
  pdl_trigger();
  uint32_t rb0[NB], rb1[NB];
  load_w(0, rb0);  // the weights are older than this pass
  load_w(1, rb1);
  pdl_wait();
  load_a(0);
  load_a(1);
  Acc acc;
  acc.clear();
  auto chunk = [&](int ch, uint32_t (&rb)[NB], __nv_bfloat16 (&Bs)[64][UN + 8]) {
#pragma unroll
    for (int i = 0; i < NB; ++i) *(uint32_t*)&Bs[bk + i * KR][bu] = rb[i];
    cp_wait<1>();
    __syncthreads();
    load_a(ch + 2);
    load_w(ch + 2, rb);
    const int mat = lane >> 3, i8 = lane & 7;
    auto& As = S.A[ch % 3];
#pragma unroll
    for (int ks = wk; ks < 4; ks += WK) {
      const int k = ks * 16;
      uint32_t fa[3][4], fb[2][4];
#pragma unroll
      for (int q = 0; q < 3; ++q) ldm4(fa[q], &As[q][wm * 16 + (mat & 1) * 8 + i8][k + (mat >> 1) * 8]);
#pragma unroll
      for (int h = 0; h < 2; ++h) ldm4t(fb[h], &Bs[k + (mat & 1) * 8 + i8][wn * 32 + h * 16 + (mat >> 1) * 8]);
      products(acc, fa, fb);
    }
    acc.flush();
  };
  for (int ch = 0; ch < nch; ch += 2) {
    chunk(ch, rb0, S.B[0]);
    if (ch + 1 < nch) chunk(ch + 1, rb1, S.B[1]);
  }
  cp_wait<0>();
  share_sum<WM * WN, WK>(acc, red, wm * WN + wn, wk, lane);
  cl.barrier_wait(std::move(started));
  if (wk == 0) {
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const int r = wm * 16 + (lane >> 2) + (i >> 1) * 8;
      // rows of the lower half to CTA 0, of the upper half to CTA 1
      float(*const to)[BM][UN] = (float(*)[BM][UN])cl.map_shared_rank((float*)dh, r >= BM / 2 ? 1 : 0);
#pragma unroll
      for (int n = 0; n < 4; ++n)
        *(float2*)&to[sg][r][wn * 32 + n * 8 + 2 * (lane & 3)] = make_float2(acc.sum[n][i], acc.sum[n][i + 1]);
    }
  }
  cl.sync();
  // pointwise: each thread takes pairs of neighbouring units, all loads first
  constexpr int NP = BM / 2 * PR / 256 > 0 ? BM / 2 * PR / 256 : 1;
  float gt[NP][4][2], cc[NP][2], cq[NP][2], dcv[NP][2];
  bool kp[NP][2];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int e = tid + 256 * p, r = sg * (BM / 2) + e / PR, b = b0 + r, u = u0 + 2 * (e % PR);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const bool in = e < BM / 2 * PR && b < B && u + j < H;
      const int64_t x = (int64_t)b * H + u + j;
#pragma unroll
      for (int q = 0; q < 4; ++q) gt[p][q][j] = in ? C.gates[(int64_t)b * 4 * H + q * H + u + j] : 0.f;
      cc[p][j] = in ? C.c[x] : 0.f;
      cq[p][j] = in && C.cprev ? C.cprev[x] : 0.f;
      dcv[p][j] = in && !C.first ? C.dc[x] : 0.f;
      kp[p][j] = in && (!C.keep || C.keep[x]);
    }
  }
  const float scale = C.keep ? a.drop_scale : 1.f;
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int e = tid + 256 * p, r = sg * (BM / 2) + e / PR, b = b0 + r, u = u0 + 2 * (e % PR);
    if (e >= BM / 2 * PR || b >= B || u >= H) continue;
    float dz[4][2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      // the first segment came through the dropout of the layer above
      const float from = kp[p][j] ? dh[0][r][2 * (e % PR) + j] * scale : 0.f;
      const float d = from + dh[1][r][2 * (e % PR) + j];
      const float ig = gt[p][0][j], fg = gt[p][1][j], gg = gt[p][2][j], og = gt[p][3][j];
      const float tc = tanhf(cc[p][j]);
      const float d_o = d * tc, dv = dcv[p][j] + d * og * (1.f - tc * tc);
      const float di = dv * gg, dg = dv * ig, df = dv * cq[p][j];
      if (u + j < H) C.dc[(int64_t)b * H + u + j] = dv * fg;
      dz[0][j] = di * ig * (1.f - ig);
      dz[1][j] = df * fg * (1.f - fg);
      dz[2][j] = dg * (1.f - gg * gg);
      dz[3][j] = d_o * og * (1.f - og);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (EVEN) store_pair(C.dz, b, q * H + u, dz[q][0], dz[q][1]);
      else {
        store_one(C.dz, b, q * H + u, dz[q][0]);
        if (u + 1 < H) store_one(C.dz, b, q * H + u + 1, dz[q][1]);
      }
    }
  }
}

// ---- weight gradients: a 64 x 64 tile of one entry per CTA, warps 4 x 2
struct GradStage {
  __nv_bfloat16 A[3][64][kLd], X[3][64][kLd];  // [part][k][m or n]
};
__global__ void __launch_bounds__(256, 2) k_weight_grads(const __grid_constant__ LstmGrad a) {
  extern __shared__ __align__(16) uint8_t sm[];
  GradStage* const stg = (GradStage*)sm;
  pdl_trigger();
  int ei = 0;
  while (ei + 1 < a.entries && (int)blockIdx.x >= a.e[ei + 1].tile0) ++ei;
  const LstmGradEntry& E = a.e[ei];
  const int nt = (E.N + 63) / 64, tile = blockIdx.x - E.tile0;
  const int m0 = (tile / nt) * 64, c0 = (tile % nt) * 64;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wm = warp >> 1, wn = warp & 1;
  const int M = E.M, N = E.N, shift = E.shift;
  const int64_t K = E.K;
  const Parts A = E.A, X = E.X;
  auto load = [&](int64_t k0, GradStage& S) {
    if (k0 < K) {
      stage_parts<64>(&S.A[0][0][0], A, k0, 0, K, m0, M);
      stage_parts<64>(&S.X[0][0][0], X, k0 - shift, 0, K - shift, c0, N);
    }
    cp_commit();
  };
  Acc acc;
  acc.clear();
  pdl_wait();
  load(0, stg[0]);
  for (int64_t k0 = 0; k0 < K; k0 += 64) {
    GradStage& S = stg[(k0 >> 6) & 1];
    cp_wait<0>();
    __syncthreads();  // this stage is in, and every warp is done with the other
    load(k0 + 64, stg[((k0 >> 6) & 1) ^ 1]);
    const int mat = lane >> 3, i8 = lane & 7;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const int k = ks * 16;
      uint32_t fa[3][4];
#pragma unroll
      for (int q = 0; q < 3; ++q) ldm4t(fa[q], &S.A[q][k + (mat >> 1) * 8 + i8][wm * 16 + (mat & 1) * 8]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t fx[3][4];
#pragma unroll
        for (int q = 0; q < 3; ++q) ldm4t(fx[q], &S.X[q][k + (mat & 1) * 8 + i8][wn * 32 + h * 16 + (mat >> 1) * 8]);
        // parts (of A, of X), the small products and the leading one in turn
        const int pa[6] = {2, 0, 0, 1, 1, 0}, px[6] = {0, 0, 2, 1, 0, 1};
#pragma unroll
        for (int t = 0; t < 6; ++t)
#pragma unroll
          for (int n2 = 0; n2 < 2; ++n2)
            mma16816(t == 1 ? acc.hi[2 * h + n2] : acc.lo[2 * h + n2], fa[pa[t]], fx[px[t]][2 * n2],
                     fx[px[t]][2 * n2 + 1]);
      }
    }
    acc.flush_exact();
  }
  acc.finish();
#pragma unroll
  for (int n = 0; n < 4; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = m0 + wm * 16 + (lane >> 2) + (i >> 1) * 8;
      const int c = c0 + wn * 32 + n * 8 + 2 * (lane & 3) + (i & 1);
      if (r < M && c < N) E.out[(int64_t)r * N + c] = acc.sum[n][i];
    }
}

// ---- column sums and, in one more cluster, the loss: 64 columns per cluster of
// four CTAs, pairs of neighbours per lane, 128 slices of rows; compensated FP32
// sums (Knuth's TwoSum) combined in FP64
constexpr int kSumSplit = 4;
__global__ void __cluster_dims__(1, kSumSplit, 1) __launch_bounds__(1024) k_lstm_sums(const __grid_constant__ LstmSums a) {
  __shared__ double part[32][65];
  __shared__ double tot[64];
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  pdl_trigger();
  pdl_wait();
  const int lane = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if ((int)blockIdx.x == a.blocks) {
    if (threadIdx.x == 0 && blockIdx.y == 0) {
      double s = 0.0;
      for (int i = 0; i < a.nlpart; ++i) s += a.lpart[i];
      *a.loss = (float)(s / a.lcount);
    }
    return;
  }
  int ei = 0;
  while (ei + 1 < a.entries && (int)blockIdx.x >= a.e[ei + 1].block0) ++ei;
  const LstmSumEntry& E = a.e[ei];
  const int c0 = (blockIdx.x - E.block0) * 64, c = c0 + 2 * lane;
  float s[2] = {0.f, 0.f}, err[2] = {0.f, 0.f};
  if (c < E.N) {
    const __nv_bfloat16* in = E.in.p + c;
    const int64_t plane = E.in.plane, ld = E.in.ld;
#pragma unroll 4
    for (int64_t i = blockIdx.y * 32 + ty; i < E.rows; i += 32 * kSumSplit) {
      uint32_t w[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) w[q] = *(const uint32_t*)(in + q * plane + i * ld);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        // the parts add up exactly
        auto val = [&](uint32_t v) { return __uint_as_float(j ? v & 0xffff0000u : v << 16); };
        const float x = (val(w[0]) + val(w[1])) + val(w[2]);
        const float t = s[j] + x, bp = t - s[j];
        err[j] += (s[j] - (t - bp)) + (x - bp);
        s[j] = t;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j)  // an infinite sum has no error term (TwoSum's is NaN)
    part[ty][2 * lane + j] = (double)s[j] + (fabsf(s[j]) <= FLT_MAX ? (double)err[j] : 0.0);
  __syncthreads();
  if (threadIdx.x < 64) {
    double t = 0.0;
    for (int k = 0; k < 32; ++k) t += part[k][threadIdx.x];
    tot[threadIdx.x] = t;
  }
  cl.sync();
  if (blockIdx.y == 0 && threadIdx.x < 64 && c0 + (int)threadIdx.x < E.N) {
    double t = 0.0;
    for (int r = 0; r < kSumSplit; ++r) t += cl.map_shared_rank(tot, r)[threadIdx.x];
    E.out[c0 + threadIdx.x] = (float)t;
  }
  cl.sync();  // nobody leaves before its sums were read
}

// ---- parts of the windows
__global__ void k_input_parts(int B, int T, int I, const float* __restrict__ X, int64_t sb, int64_t stt, Parts out) {
  pdl_trigger();
  const int64_t row = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row >= (int64_t)T * B) return;
  const float* x = X + (row % B) * sb + (row / B) * stt;
  for (int k = 2 * (threadIdx.x & 31); k < I; k += 64)
    store_pair<true>(out, row, k, x[k], k + 1 < I ? x[k + 1] : 0.f);
}

// ---- head: a warp per batch row, lanes over the hidden units
constexpr int kHeadRows = 8;
__global__ void __launch_bounds__(kHeadRows * 32)
k_head(int B, int O, int H, const float* __restrict__ h, const __nv_bfloat16* __restrict__ Wy,
       const float* __restrict__ by, float* __restrict__ y, const float* __restrict__ tgt,
       const Parts dy, double* __restrict__ lpart) {
  pdl_trigger();
  pdl_wait();
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
#pragma unroll 4
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
          store_one<true>(dy, b, o, 2.f / ((float)B * (float)O) * d);
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

namespace {
template <int WM, int WN, int WK, bool EVEN>
cudaError_t fwd_launch(cudaStream_t st, const LstmFwd& a) {
  constexpr int BM = 16 * WM, UN = 8 * WN;
  constexpr int smem = (int)sizeof(FwdStage<BM, 4 * UN>);
  static_assert(smem >= (WK - 1) * WM * WN * 2048, "the shares fit");
  cudaError_t e = cudaFuncSetAttribute(k_cell_fwd<WM, WN, WK, EVEN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(st, dim3((a.B + BM - 1) / BM, (a.H + UN - 1) / UN, a.cells), 256, smem,
                    k_cell_fwd<WM, WN, WK, EVEN>, a);
}
template <int WM, int WN, int WK, bool EVEN>
cudaError_t bwd_launch(cudaStream_t st, const LstmBwd& a) {
  constexpr int BM = 16 * WM, UN = 32 * WN;
  constexpr int smem = (int)sizeof(BwdStage<BM, UN>) + 2 * BM * UN * 4;
  static_assert(smem >= (WK - 1) * WM * WN * 2048, "the shares fit");
  cudaError_t e = cudaFuncSetAttribute(k_cell_bwd<WM, WN, WK, EVEN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.B + BM - 1) / BM, (a.H + UN - 1) / UN, 2 * a.cells);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 2;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_pdl
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, k_cell_bwd<WM, WN, WK, EVEN>, a);
  note_launch();
  return e == cudaSuccess ? cudaGetLastError() : e;
}
}  // namespace

// Up to 32 rows, batch tiles of 16 and shares of k within a chunk (one step per
// warp, so that a small network's few CTAs have short chains); above, 64 rows.
// Measured at 2 x 256, window 10, loss and gradients in 16-row and in 64-row
// tiles: 32 rows 264 and 350 us, 64 rows 305 and 388, 128 rows 344 and 430; 3 x 50: 162
// and 191, 167 and 208, 216 and 234.  So up to 128 rows the line lies too low.
cudaError_t lstm_fwd_phase(cudaStream_t st, const LstmFwd& a) {
  bool even = (a.H & 1) == 0;
  for (int i = 0; i < a.cells; ++i) even = even && (a.cell[i].Il & 1) == 0;
  if (even) return a.B <= 32 ? fwd_launch<1, 2, 4, true>(st, a) : fwd_launch<4, 2, 1, true>(st, a);
  return a.B <= 32 ? fwd_launch<1, 2, 4, false>(st, a) : fwd_launch<4, 2, 1, false>(st, a);
}
cudaError_t lstm_bwd_phase(cudaStream_t st, const LstmBwd& a) {
  const bool even = (a.H & 1) == 0;
  if (even) return a.B <= 32 ? bwd_launch<1, 2, 4, true>(st, a) : bwd_launch<4, 1, 2, true>(st, a);
  return a.B <= 32 ? bwd_launch<1, 2, 4, false>(st, a) : bwd_launch<4, 1, 2, false>(st, a);
}

cudaError_t lstm_weight_grads(cudaStream_t st, LstmGrad& a) {
  a.tiles = 0;
  for (int i = 0; i < a.entries; ++i) {
    a.e[i].tile0 = a.tiles;
    a.tiles += ((a.e[i].M + 63) / 64) * ((a.e[i].N + 63) / 64);
  }
  const int smem = 2 * (int)sizeof(GradStage);
  const cudaError_t e = cudaFuncSetAttribute(k_weight_grads, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(st, a.tiles, 256, smem, k_weight_grads, a);
}

cudaError_t lstm_sums(cudaStream_t st, LstmSums& a) {
  a.blocks = 0;
  for (int i = 0; i < a.entries; ++i) {
    a.e[i].block0 = a.blocks;
    a.blocks += (a.e[i].N + 63) / 64;
  }
  return launch_pdl(st, dim3(a.blocks + 1, kSumSplit), 1024, 0, k_lstm_sums, a);
}

cudaError_t lstm_input_parts(cudaStream_t st, int B, int T, int I, const float* X, int64_t sb, int64_t stt,
                             Parts out) {
  k_input_parts<<<(unsigned)(((int64_t)T * B + 7) / 8), 256, 0, st>>>(B, T, I, X, sb, stt, out);
  note_launch();
  return cudaGetLastError();
}

int lstm_head_blocks(int B) { return (B + kHeadRows - 1) / kHeadRows; }

cudaError_t lstm_head(cudaStream_t st, int B, int O, int H, const float* h, const __nv_bfloat16* Wy,
                      const float* by, float* y, const float* tgt, Parts dy, double* lpart) {
  return launch_pdl(st, lstm_head_blocks(B), kHeadRows * 32, 0, k_head, B, O, H, h, Wy, by, y, tgt, dy, lpart);
}

}  // namespace rpod
