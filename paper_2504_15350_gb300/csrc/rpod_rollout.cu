// LSTM rollout kernels (the online stage of Sec. 4.3): autoregressive
// prediction of `steps` coefficient vectors in one launch.  The pipelined kernel
// over a cluster per sample is the second half of this file; first the
// persistent cooperative kernel, for what it does not fit or takes longer for.
//
// The network maps a window of T rows [mu, alpha] to the next alpha, with
// zero initial states for every window, so each prediction runs L x T cells.
// One CTA owns U consecutive hidden units of every layer: the 4U gate rows
// of W_x and W_h (widened to FP32 from the weights the products read), the
// biases, and the cell states of its units stay in shared memory for the
// whole rollout.  Cell (l, t) needs h(l, t - 1) and h(l - 1, t), so the cells
// of one anti-diagonal l + t run in the same phase: L + T - 1 phases per
// prediction, each ended by a grid barrier, then the linear head (rows of
// W_y spread over the CTAs) writes the prediction into a ring buffer of
// window rows, which replaces the oldest row, and a last barrier.
//
// Grid barrier: a monotonic arrival counter in the workspace; a CTA arrives
// (after a device-scope fence) and its first thread waits for the count of
// the barrier with a 2 s %globaltimer limit.  A wait that runs out records
// ST_TIMEOUT, raises an abort word that every waiting CTA checks, and the
// kernel returns; nothing waits without a limit.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "rpod_internal.cuh"

namespace rpod {
namespace {

constexpr uint64_t kBarrierTimeoutNs = 2000000000ull;

__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier number k (0, 1, 2, ...) over gridDim.x CTAs: false when a
// wait ran out (here or in another CTA).
__device__ bool grid_sync(unsigned* count, unsigned k, volatile int* abort_word, unsigned* status,
                          uint64_t limit_ns, bool arrive = true) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    __threadfence();
    if (arrive) atomicAdd(count, 1u);
    const unsigned target = (k + 1) * gridDim.x;
    const uint64_t t0 = gtimer();
    while (*(volatile unsigned*)count < target) {
      if (*abort_word) {
        ok = 0;
        break;
      }
      if (gtimer() - t0 > limit_ns) {
        atomicOr(status, ST_TIMEOUT);
        *abort_word = 1;
        ok = 0;
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

__device__ __forceinline__ float sigm_r(float x) { return 1.f / (1.f + __expf(-x)); }
__device__ __forceinline__ float wld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ float wld(const float* p) { return *p; }

struct RollArgs {
  int I, H, L, O, T, B, d, U, steps;
  const float* theta;          // FP32 parameters (biases, and weights when TW = float)
  const void* wbf;             // weight copies the products read (BF16) or theta
  int64_t off_w[4][3];         // per layer: W_x, W_h, b offsets into the flat vector
  int64_t off_wy, off_by;
  float* ring;                 // T x B x I window rows (ring buffer), time-major
  float* hbuf;                 // L x T x B x H hidden states of the current window
  float* out;                  // B x steps x O predictions
  unsigned* count;             // barrier arrivals (zeroed by the host)
  int* abort_word;
  unsigned* status;
};

// Dynamic shared memory per CTA: for every layer the 4U gate rows of
// [W_x | W_h] (K_l = I_l + H floats, stride K_l + 1), 4U biases, U x B cell
// states; the gathered inputs [x | h_prev] of the phase's cells (B x (I + H)
// per cell, two cells at most in flight per layer) reuse one staging area
// per layer; the gate pre-activations (4U x B per layer); W_y rows of the
// outputs this CTA computes.
__host__ __device__ inline size_t roll_smem_floats(int I, int H, int L, int O, int B, int U, int G) {
  size_t f = 0;
  for (int l = 0; l < L; ++l) {
    const int K = (l == 0 ? I : H) + H;
    f += (size_t)4 * U * (K + 1) + 4 * U + (size_t)U * B + (size_t)B * (K + 1) + (size_t)4 * U * B;
  }
  const int rows = (O + G - 1) / G;
  f += (size_t)rows * H + rows;
  return f;
}

template <typename TW>
__global__ void __launch_bounds__(512, 1) k_rollout(RollArgs a) {
  extern __shared__ float sm[];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int I = a.I, H = a.H, L = a.L, O = a.O, T = a.T, B = a.B, U = a.U;
  const int G = gridDim.x, cta = blockIdx.x;
  const int u0 = cta * U;
  const TW* W = (const TW*)a.wbf;
  // ---- carve shared memory and load this CTA's rows once
  float* Wl[4];
  float* bl[4];
  float* cl[4];
  float* xl[4];
  float* zl[4];
  float* p = sm;
  for (int l = 0; l < L; ++l) {
    const int Il = l == 0 ? I : H, K = Il + H;
    Wl[l] = p; p += (size_t)4 * U * (K + 1);
    bl[l] = p; p += 4 * U;
    cl[l] = p; p += (size_t)U * B;
    xl[l] = p; p += (size_t)B * (K + 1);  // rows padded: samples of one warp on distinct banks
    zl[l] = p; p += (size_t)4 * U * B;
    for (int e = tid; e < 4 * U * K; e += nt) {
      const int r = e / K, k = e % K;
      const int g = r / U, u = u0 + r % U;
      const int64_t row = (int64_t)g * H + u;
      Wl[l][r * (K + 1) + k] = k < Il ? wld(W + a.off_w[l][0] + row * Il + k)
                                      : wld(W + a.off_w[l][1] + row * H + (k - Il));
    }
    for (int r = tid; r < 4 * U; r += nt) bl[l][r] = a.theta[a.off_w[l][2] + (r / U) * H + u0 + r % U];
  }
  const int yrows = (O + G - 1) / G;
  float* Wy = p; p += (size_t)yrows * H;
  float* byl = p;
  for (int e = tid; e < yrows * H; e += nt) {
    const int r = e / H, k = e % H, o = cta + r * G;
    Wy[e] = o < O ? wld(W + a.off_wy + (int64_t)o * H + k) : 0.f;
  }
  for (int r = tid; r < yrows; r += nt) {
    const int o = cta + r * G;
    byl[r] = o < O ? a.theta[a.off_by + o] : 0.f;
  }
  __syncthreads();

  unsigned bar = 0;
  const volatile int* abort_word = a.abort_word;
  for (int s = 0; s < a.steps; ++s) {
    // the window of this prediction: ring rows (s + t) mod T, t = 0..T-1
    for (int ph = 0; ph < L + T - 1; ++ph) {
      if (*abort_word) return;
      // gather the inputs of this phase's cells (l, t = ph - l): x, h_prev
      for (int l = 0; l < L; ++l) {
        const int t = ph - l;
        if (t < 0 || t >= T) continue;
        const int Il = l == 0 ? I : H, K = Il + H;
        const float* xin = l == 0 ? a.ring + (size_t)((s + t) % T) * B * I
                                  : a.hbuf + ((size_t)(l - 1) * T + t) * B * H;
        const float* hprev = t > 0 ? a.hbuf + ((size_t)l * T + t - 1) * B * H : nullptr;
        // x (B x Il) and h_prev (B x H) are contiguous in global memory: four
        // independent loads in flight per thread, then the padded stores
        for (int e0 = 0; e0 < B * Il; e0 += 4 * nt) {
          float v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int e = e0 + j * nt + tid;
            v[j] = e < B * Il ? __ldcg(xin + e) : 0.f;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int e = e0 + j * nt + tid;
            if (e < B * Il) xl[l][(e / Il) * (K + 1) + e % Il] = v[j];
          }
        }
        for (int e0 = 0; e0 < B * H; e0 += 4 * nt) {
          float v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int e = e0 + j * nt + tid;
            v[j] = (e < B * H && hprev) ? __ldcg(hprev + e) : 0.f;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int e = e0 + j * nt + tid;
            if (e < B * H) xl[l][(e / H) * (K + 1) + Il + e % H] = v[j];
          }
        }
        if (t == 0)
          for (int e = tid; e < U * B; e += nt) cl[l][e] = 0.f;
      }
      __syncthreads();
      // gate pre-activations: 4U rows x B samples, 4 threads per dot product
      for (int l = 0; l < L; ++l) {
        const int t = ph - l;
        if (t < 0 || t >= T) continue;
        const int Il = l == 0 ? I : H, K = Il + H;
        const int ndot = 4 * U * B;
        for (int q0 = 0; q0 < ndot * 4; q0 += nt) {
          const int q = q0 + tid;
          const int dot = q >> 2, part = q & 3;
          float acc = 0.f;
          if (dot < ndot) {
            const int r = dot / B, b = dot % B;
            const float* w = Wl[l] + (size_t)r * (K + 1);
            const float* x = xl[l] + (size_t)b * (K + 1);
            float acc2 = 0.f;
            int k = part;
            for (; k + 4 < K; k += 8) {
              acc = fmaf(w[k], x[k], acc);
              acc2 = fmaf(w[k + 4], x[k + 4], acc2);
            }
            if (k < K) acc = fmaf(w[k], x[k], acc);
            acc += acc2;
          }
          acc += __shfl_xor_sync(0xffffffffu, acc, 1);
          acc += __shfl_xor_sync(0xffffffffu, acc, 2);
          if (dot < ndot && part == 0) zl[l][dot] = acc + bl[l][dot / B];
        }
      }
      __syncthreads();
      // cell updates of this CTA's units; h to the window's state buffer
      for (int l = 0; l < L; ++l) {
        const int t = ph - l;
        if (t < 0 || t >= T) continue;
        float* hout = a.hbuf + ((size_t)l * T + t) * B * H;
        for (int e = tid; e < U * B; e += nt) {
          const int uu = e / B, b = e % B;
          const float zi = zl[l][(0 * U + uu) * B + b], zf = zl[l][(1 * U + uu) * B + b];
          const float zg = zl[l][(2 * U + uu) * B + b], zo = zl[l][(3 * U + uu) * B + b];
          const float c = sigm_r(zf) * cl[l][e] + sigm_r(zi) * tanhf(zg);
          cl[l][e] = c;
          hout[(size_t)b * H + u0 + uu] = sigm_r(zo) * tanhf(c);
        }
      }
      if (!grid_sync(a.count, bar++, a.abort_word, a.status, kBarrierTimeoutNs)) return;
    }
    // head on the top layer's last state: this CTA's outputs o = cta + r G;
    // the prediction replaces the oldest ring row (s mod T), the parameters
    // of the newest row carry over
    const float* hT = a.hbuf + ((size_t)(L - 1) * T + T - 1) * B * H;
    float* newrow = a.ring + (size_t)(s % T) * B * I;
    const float* lastrow = a.ring + (size_t)((s + T - 1) % T) * B * I;
    for (int e = tid / 32; e < yrows * B; e += nt / 32) {
      const int r = e / B, b = e % B, o = cta + r * G;
      float acc = 0.f;
      for (int k = tid & 31; k < H; k += 32) acc = fmaf(Wy[r * H + k], __ldcg(hT + (size_t)b * H + k), acc);
      for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
      if ((tid & 31) == 0 && o < O) {
        const float y = acc + byl[r];
        newrow[(size_t)b * I + a.d + o] = y;
        a.out[((size_t)b * a.steps + s) * O + o] = y;
      }
    }
    if (cta == 0)
      for (int e = tid; e < B * a.d; e += nt) {
        const int b = e / a.d, k = e % a.d;
        newrow[(size_t)b * I + k] = __ldcg(lastrow + (size_t)b * I + k);
      }
    if (!grid_sync(a.count, bar++, a.abort_word, a.status, kBarrierTimeoutNs)) return;
  }
}

// ---- pipelined rollout over a thread-block cluster ------------------------
// Every prediction runs the whole window from zero states, but the windows of
// consecutive predictions share all rows but one: when row r becomes known,
// the T windows that contain it can all advance by one time step.  So instead
// of T + L - 1 dependent phases per prediction there are L: layer 0 of all T
// windows on row r, layer 1 on their new h_0, ..., then the head on the one
// window that row r completes, which gives row r + 1.  The work per
// prediction is the same (T steps of L cells), its dependent chain is T times
// shorter, and a product has T columns instead of one.
//
// Samples never interact, so one cluster of CS CTAs owns one sample (clusters
// beyond the GPU's capacity run later; nothing waits across clusters).  A CTA
// owns U hidden units of every layer: their 4U gate rows of W_x and W_h stay
// in shared memory, in the type the products read (half the shared memory of
// widened copies for BF16), and multiply the cluster's h (k-major, the T
// windows' values contiguous) with packed FP32 pairs of windows: a thread
// holds two gate rows x T sums of one k-slice, so an inner step is one 4-byte
// weight load and T/4 broadcast 16-byte loads of h for T packed FMAs.  New h
// values go to every CTA of the cluster as bulk copies between shared memories
// that complete on the receiver's mbarrier; the wait for them comes after the
// next phase's recurrent product, which needs only the previous row.  The head
// is split over the units: each CTA sends its share of the O outputs with its
// h, and every CTA adds the CS shares itself.
//
// Bound: the FP32 pipes (3 products of 4U x T x H per row and CTA) and the
// phase latency (partial sums over the k-slices, gates, exchange).  Measured
// at 2 x 256, window 10, 8 samples, 500 steps: 4.1 ms; the kernel with
// T + L - 1 grid barriers per prediction above takes 68.4 ms.  Every wave of
// clusters loads the weights and runs the window first, so many samples over
// few steps take the per-step kernels (rollout_pipelined's limit).
constexpr int kPipeThreads = 384;
constexpr size_t kPipeSmemMax = (size_t)226 * 1024;

struct PipeArgs {
  int I, H, L, O, T, d, U, CS, steps;
  int SL, threads;             // k-slices, threads that multiply (SL x 2U)
  const float* theta;
  const void* w;               // weights in the products' type
  int64_t off_w[4][3];
  int64_t off_wy, off_by;
  const float* window;         // B x T x I
  float* out;                  // B x steps x O
  unsigned* status;
};

__host__ __device__ inline int even_up(int x) { return (x + 1) & ~1; }

// Shared memory of one CTA; ws: bytes of a stored weight.
__host__ __device__ inline size_t pipe_smem_bytes(int I, int H, int L, int O, int U, int CS, int Tp,
                                                  int SL, size_t ws) {
  const size_t R = 4 * (size_t)U;
  size_t w = (size_t)O * U;
  for (int l = 0; l < L; ++l) w += R * (size_t)(even_up(l == 0 ? I : H) + even_up(H));
  size_t f = (size_t)2 * L * CS * U * Tp;        // h, two buffers per layer
  f += (size_t)2 * CS * ((O + 3) & ~3);          // head shares
  f += (size_t)SL * R * Tp;                      // partial sums
  f += (size_t)L * R + (size_t)L * U * Tp;       // biases, cell states
  f += (size_t)even_up(I) + O;
  return f * 4 + ((w * ws + 15) & ~(size_t)15) + 64;
}

__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float2 wpair(const __nv_bfloat16* p) {
  return __bfloat1622float2(*(const __nv_bfloat162*)p);
}
__device__ __forceinline__ float2 wpair(const float* p) { return *(const float2*)p; }

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// bytes (a multiple of 16) from this CTA's shared memory to another's; the
// writes were made visible to the async proxy before
__device__ __forceinline__ void send_block(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "r"(src), "r"(bytes), "r"(mbar)
      : "memory");
}
// Bounded wait for a phase of the exchange; false when 2 s passed.
__device__ __forceinline__ bool exch_wait(uint32_t mbar, uint32_t parity) {
  uint32_t ok = 0;
  const uint64_t t0 = gtimer();
  while (true) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (gtimer() - t0 > kBarrierTimeoutNs) return false;
  }
}

// acc += W(k, rows) h(k, windows) for k in [k0, k1) (k0 even, k1 - k0 even):
// W k-major with R rows (this thread's two at W), h k-major with 2 NP windows.
template <typename TW, int NP>
__device__ __forceinline__ void pipe_prod(const TW* W, int R, const float* h, int k0, int k1,
                                          uint64_t (&acc)[2][NP]) {
#pragma unroll 4
  for (int k = k0; k < k1; k += 2) {
    const float2 wa = wpair(W + k * R), wb = wpair(W + (k + 1) * R);
    const ulonglong2* hp = (const ulonglong2*)(h + k * (2 * NP));
    uint64_t hv[2 * NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const ulonglong2 v = hp[i];
      hv[2 * i] = v.x;
      hv[2 * i + 1] = v.y;
    }
    const uint64_t a0 = pack2(wa.x, wa.x), a1 = pack2(wa.y, wa.y);
    const uint64_t b0 = pack2(wb.x, wb.x), b1 = pack2(wb.y, wb.y);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      acc[0][i] = fma2(a0, hv[i], acc[0][i]);
      acc[1][i] = fma2(a1, hv[i], acc[1][i]);
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      acc[0][i] = fma2(b0, hv[NP + i], acc[0][i]);
      acc[1][i] = fma2(b1, hv[NP + i], acc[1][i]);
    }
  }
}

template <typename TW, int NP>
__global__ void __launch_bounds__(kPipeThreads, 1) k_rollout_pipe(const __grid_constant__ PipeArgs a) {
  namespace cg = cooperative_groups;
  constexpr int Tp = 2 * NP, NT = kPipeThreads;
  extern __shared__ __align__(16) float sm[];
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ volatile int s_dead;
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int I = a.I, H = a.H, L = a.L, O = a.O, T = a.T, U = a.U, CS = a.CS, SL = a.SL;
  const int rank = (int)cl.block_rank(), b = blockIdx.x / CS;
  const int u0 = rank * U, R = 4 * U, Hr = CS * U;
  const int Ip = even_up(I), Hp = even_up(H), Op = (O + 3) & ~3;
  // ---- shared memory (16-byte pieces first: h, head shares, weights)
  float* hs = sm;                                   // [L][2][Hr][Tp]
  float* yp = hs + (size_t)2 * L * Hr * Tp;         // [2][CS][Op]
  float* part = yp + (size_t)2 * CS * Op;           // [SL][R][Tp], gate row r = 4 u + gate
  float* bias = part + (size_t)SL * R * Tp;         // [L][R]
  float* cst = bias + (size_t)L * R;                // [L][U][Tp]
  float* xs = cst + (size_t)L * U * Tp;             // [Ip]
  float* by = xs + Ip;                              // [O]
  TW* wsm = (TW*)(sm + (((by + O - sm) + 3) & ~(ptrdiff_t)3));
  TW* wy;                                           // [O][U]
  const TW* W = (const TW*)a.w;
  {
    TW* p = wsm;
    for (int l = 0; l < L; ++l) {
      const int Il = l == 0 ? I : H, Ilp = even_up(Il);
      for (int pi = 0; pi < 2; ++pi) {  // W_x, then W_h
        const int K = pi ? H : Il, Kp = pi ? Hp : Ilp;
        const TW* src = W + a.off_w[l][pi];
        // read along k (contiguous), write k-major
        for (int e = tid; e < R * Kp; e += NT) {
          const int r = e / Kp, k = e % Kp, u = u0 + (r >> 2);
          p[k * R + r] = (k < K && u < H) ? src[((int64_t)(r & 3) * H + u) * K + k] : TW(0.f);
        }
        p += (size_t)R * Kp;
      }
      for (int r = tid; r < R; r += NT) {
        const int u = u0 + (r >> 2);
        bias[l * R + r] = u < H ? a.theta[a.off_w[l][2] + (int64_t)(r & 3) * H + u] : 0.f;
      }
    }
    wy = p;
    for (int e = tid; e < O * U; e += NT) {
      const int o = e / U, u = u0 + e % U;
      wy[e] = u < H ? W[a.off_wy + (int64_t)o * H + u] : TW(0.f);
    }
    for (int e = tid; e < O; e += NT) by[e] = a.theta[a.off_by + e];
    for (int e = tid; e < 2 * L * Hr * Tp; e += NT) hs[e] = 0.f;
    for (int e = tid; e < L * U * Tp; e += NT) cst[e] = 0.f;
    for (int e = tid; e < Ip; e += NT) xs[e] = 0.f;
  }
  const uint32_t mb = smem_u32(mbar);
  if (tid == 0) {
    for (int i = 0; i < 2; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb + 8 * i) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_dead = 0;
  }
  // this thread's two gate rows and its k-slice
  const bool live = tid < a.threads;
  const int slice = tid / (2 * U), row = 2 * (tid % (2 * U));
  auto span = [&](int Kp, int& k0, int& k1) {
    const int c = 2 * ((Kp / 2 + SL - 1) / SL);
    k0 = slice * c < Kp ? slice * c : Kp;
    k1 = k0 + c < Kp ? k0 + c : Kp;
  };
  int hk0, hk1, xk0, xk1;
  span(Hp, hk0, hk1);
  span(Ip, xk0, xk1);
  cl.sync();

  int g = 0;                     // exchanges started
  const int rows = T + a.steps;  // the last one only takes the last prediction
  bool dead = false;
  for (int r = 0; r < rows && !dead; ++r) {
    const int buf = r & 1, z = r % T;
    const bool last = r == rows - 1;
    const TW* wl = wsm;
    for (int l = 0; l < L; ++l) {
      const int Ilp = l == 0 ? Ip : Hp;
      const TW* Wx = wl;
      const TW* Wh = wl + (size_t)R * Ilp;
      wl = Wh + (size_t)R * Hp;
      float* hl = hs + (size_t)(2 * l) * Hr * Tp;
      auto arrived = [&]() {
        if (g > 0 && !exch_wait(mb + 8 * ((g - 1) & 1), ((g - 1) >> 1) & 1)) {
          atomicOr(a.status, ST_TIMEOUT);
          s_dead = 1;
        }
      };
      // a single layer's own h is what the exchange in flight brings
      if (L == 1) arrived();
      uint64_t acc[2][NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) acc[0][i] = acc[1][i] = 0ull;
      if (live && !last) {
        pipe_prod<TW, NP>(Wh + row, R, hl + (size_t)(buf ^ 1) * Hr * Tp, hk0, hk1, acc);
        // the window that starts with this row starts from h = 0
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            float v0, v1;
            unpack2(acc[q][i], v0, v1);
            acc[q][i] = pack2(2 * i == z ? 0.f : v0, 2 * i + 1 == z ? 0.f : v1);
          }
      }
      if (L > 1) arrived();
      if (l == 0) {
        // row r of the sequence: the given window, then the predictions (the
        // parameters of the newest given row carry over)
        if (r < T) {
          for (int k = tid; k < I; k += NT) xs[k] = a.window[((int64_t)b * T + r) * I + k];
        } else {
          const float* ys = yp + (size_t)(buf ^ 1) * CS * Op;
          for (int e0 = 0; e0 < 4 * Op; e0 += NT) {  // four lanes per output
            const int e = e0 + tid, o = e >> 2;
            float y = 0.f;
            if (o < O) {
#pragma unroll 4
              for (int c = e & 3; c < CS; c += 4) y += ys[c * Op + o];
            }
            y += __shfl_xor_sync(0xffffffffu, y, 1);
            y += __shfl_xor_sync(0xffffffffu, y, 2);
            if ((e & 3) == 0 && o < O) {
              y += by[o];
              xs[a.d + o] = y;
              if (rank == 0) a.out[((int64_t)b * a.steps + (r - T)) * O + o] = y;
            }
          }
        }
        if (last) break;
        __syncthreads();
        if (live) {
          // the row is the same for all windows
          float x0 = 0.f, x1 = 0.f;
#pragma unroll 4
          for (int k = xk0; k < xk1; ++k) {
            const float2 w = wpair(Wx + k * R + row);
            x0 = fmaf(w.x, xs[k], x0);
            x1 = fmaf(w.y, xs[k], x1);
          }
          const uint64_t p0 = pack2(x0, x0), p1 = pack2(x1, x1);
#pragma unroll
          for (int i = 0; i < NP; ++i) {
            acc[0][i] = add2(acc[0][i], p0);
            acc[1][i] = add2(acc[1][i], p1);
          }
        }
      } else if (live) {
        pipe_prod<TW, NP>(Wx + row, R, hs + (size_t)(2 * (l - 1) + buf) * Hr * Tp, hk0, hk1, acc);
      }
      if (live) {
        uint64_t* d0 = (uint64_t*)(part + (slice * R + row) * Tp);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          d0[i] = acc[0][i];
          d0[NP + i] = acc[1][i];
        }
      }
      __syncthreads();
      if (s_dead) {  // uniform: set before the barrier
        dead = true;
        break;
      }
      // sums over the k-slices, four values per thread, into the first slice
      float* hnew = hl + (size_t)buf * Hr * Tp + (size_t)u0 * Tp;
      for (int e = tid; e < U * Tp; e += NT) {
        float4* p4 = (float4*)part + e;
        float4 v = p4[0];
#pragma unroll 8
        for (int s = 1; s < SL; ++s) {
          const float4 t = p4[s * U * Tp];
          v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
        }
        p4[0] = v;
      }
      __syncthreads();
      // gates and cell update of this CTA's units
      for (int cell = tid; cell < U * Tp; cell += NT) {
        const int u = cell / Tp, w = cell % Tp;
        const float* ps = part + 4 * u * Tp + w;
        const float* bs = bias + l * R + 4 * u;
        const float gi = sigm_r(ps[0] + bs[0]), gf = sigm_r(ps[Tp] + bs[1]);
        const float gg = tanhf(ps[2 * Tp] + bs[2]), go = sigm_r(ps[3 * Tp] + bs[3]);
        float* cp = cst + l * U * Tp + cell;
        const float c = gf * (w == z ? 0.f : *cp) + gi * gg;
        *cp = c;
        hnew[cell] = go * tanhf(c);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      const uint32_t bar = mb + 8 * (g & 1);
      const bool top = l == L - 1;
      if (tid == 0)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                     "r"((uint32_t)((CS - 1) * (U * Tp + (top ? Op : 0)) * 4))
                     : "memory");
      float* yo = yp + ((size_t)buf * CS + rank) * Op;
      if (top) {
        // this CTA's share of the head for the window that ends with row r,
        // four lanes per output
        const float* hw = hnew + (r + 1) % T;  // its slot
        for (int e0 = 0; e0 < 4 * Op; e0 += NT) {
          const int e = e0 + tid, o = e >> 2;
          float v = 0.f;
          if (o < O) {
#pragma unroll 4
            for (int u = e & 3; u < U; u += 4) v = fmaf(wld(wy + o * U + u), hw[u * Tp], v);
          }
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          v += __shfl_xor_sync(0xffffffffu, v, 2);
          if ((e & 3) == 0 && o < Op) yo[o] = v;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
      }
      // this CTA's block of h and head share to every other CTA of the cluster
      // (bulk copies: per-lane asynchronous stores spent about 2000 clocks of
      // the receivers' shared memory on mbarrier updates per phase)
      for (int c = 1 + warp; c < CS && lane == 0; c += NT / 32) {
        const int dst = rank + c < CS ? rank + c : rank + c - CS;
        const uint32_t rbar = cluster_addr(bar, dst);
        if (top) send_block(cluster_addr(smem_u32(yo), dst), smem_u32(yo), Op * 4, rbar);
        send_block(cluster_addr(smem_u32(hnew), dst), smem_u32(hnew), U * Tp * 4, rbar);
      }
      ++g;
    }
  }
  cl.sync();  // nothing is sent to a CTA that has left
}

// Self-test of the grid barrier's limit: CTA 0 never arrives, so the wait
// of every CTA runs out and records the timeout.  Its words live here (the
// library allocates nothing): [0] arrivals, [1] abort word, [2] status.
__device__ unsigned g_selftest_words[4];

__global__ void k_grid_sync_selftest(uint64_t limit_ns) {
  grid_sync(&g_selftest_words[0], 0, (int*)&g_selftest_words[1], &g_selftest_words[2], limit_ns,
            blockIdx.x != 0);
}

}  // namespace

int rollout_units(int H, int sms) {
  // the fewest units per CTA that keep the grid within 64 CTAs and one CTA
  // per SM (every barrier waits for all CTAs' arrivals)
  const int cap = sms < 64 ? sms : 64;
  for (int U = 1; U <= H; ++U)
    if (H % U == 0 && H / U <= cap) return U;
  return H;
}

size_t rollout_smem_bytes(int I, int H, int L, int O, int B, int U) {
  return sizeof(float) * roll_smem_floats(I, H, L, O, B, U, H / U);
}

cudaError_t rollout_persistent(cudaStream_t st, bool bf16_weights, int I, int H, int L, int O, int T,
                               int B, int d, int steps, const float* theta, const void* wbf,
                               const int64_t (*off_w)[3], int64_t off_wy, int64_t off_by,
                               float* ring, float* hbuf, float* out, unsigned* count,
                               int* abort_word, unsigned* status, int sms) {
  RollArgs a;
  a.I = I; a.H = H; a.L = L; a.O = O; a.T = T; a.B = B; a.d = d; a.steps = steps;
  a.U = rollout_units(H, sms);
  a.theta = theta;
  a.wbf = wbf;
  for (int l = 0; l < L; ++l)
    for (int j = 0; j < 3; ++j) a.off_w[l][j] = off_w[l][j];
  a.off_wy = off_wy;
  a.off_by = off_by;
  a.ring = ring;
  a.hbuf = hbuf;
  a.out = out;
  a.count = count;
  a.abort_word = abort_word;
  a.status = status;
  const size_t smem = rollout_smem_bytes(I, H, L, O, B, a.U);
  const dim3 grid((unsigned)(H / a.U)), block(512);
  void* args[] = {&a};
  const void* fn = bf16_weights ? (const void*)k_rollout<__nv_bfloat16> : (const void*)k_rollout<float>;
  if (smem > kRollSmemMax) return cudaErrorCooperativeLaunchTooLarge;
  // the kernel's largest size, not this network's: see pipe_launch
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRollSmemMax);
  if (e == cudaSuccess) e = cudaLaunchCooperativeKernel(fn, grid, block, args, smem, st);
  note_launch();
  return e;
}

namespace {

// One cluster per sample: the launch, or with `active` only how many clusters
// run at once (nothing enqueued).  The attributes are the kernel's on this
// device, for every thread: always set to the same values, so that no thread
// lowers them between another's call and its launch.
template <typename TW, int NP>
cudaError_t pipe_launch(cudaStream_t st, const PipeArgs& a, int B, size_t smem, int* active) {
  auto fn = k_rollout_pipe<TW, NP>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPipeSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(B * a.CS));
  cfg.blockDim = dim3(kPipeThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)a.CS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (active) return cudaOccupancyMaxActiveClusters(active, fn, &cfg);
  return cudaLaunchKernelEx(&cfg, fn, a);
}

template <typename TW>
cudaError_t pipe_np(cudaStream_t st, const PipeArgs& a, int B, int np, size_t smem, int* active) {
  switch (np) {
    case 2: return pipe_launch<TW, 2>(st, a, B, smem, active);
    case 4: return pipe_launch<TW, 4>(st, a, B, smem, active);
    case 5: return pipe_launch<TW, 5>(st, a, B, smem, active);
    case 6: return pipe_launch<TW, 6>(st, a, B, smem, active);
    default: return pipe_launch<TW, 8>(st, a, B, smem, active);
  }
}

// How many clusters of a shape run at once on the current device, kept for the
// last 64 shapes asked for: a query takes about 2 us, the six of a call as long
// as a whole prediction of a small network.
template <typename TW>
int pipe_active(const PipeArgs& a, int np, size_t smem) {
  struct Entry {
    int dev, np, cs, active;
    size_t smem;
  };
  static std::mutex lock;
  static Entry known[64];
  static unsigned count = 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> hold(lock);
  for (unsigned i = 0; i < count && i < 64; ++i) {
    const Entry& k = known[i];
    if (k.dev == dev && k.np == np && k.cs == a.CS && k.smem == smem) return k.active;
  }
  int n = 0;
  if (pipe_np<TW>(nullptr, a, 1, np, smem, &n) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  known[count++ % 64] = {dev, np, a.CS, n, smem};
  return n;
}

}  // namespace

cudaError_t rollout_pipelined(cudaStream_t st, bool bf16_weights, int I, int H, int L, int O, int T,
                              int B, int d, int steps, const float* theta, const void* wbf,
                              const int64_t (*off_w)[3], int64_t off_wy, int64_t off_by,
                              const float* window, float* out, unsigned* status, double limit_us) {
  if (L > 4 || T > 16) return cudaErrorInvalidConfiguration;
  const int np = T <= 4 ? 2 : (T <= 8 ? 4 : (T <= 10 ? 5 : (T <= 12 ? 6 : 8)));
  const size_t wsz = bf16_weights ? 2 : 4;
  PipeArgs a;
  a.I = I; a.H = H; a.L = L; a.O = O; a.T = T; a.d = d; a.steps = steps;
  a.theta = theta;
  a.w = wbf;
  for (int l = 0; l < L; ++l)
    for (int j = 0; j < 3; ++j) a.off_w[l][j] = off_w[l][j];
  a.off_wy = off_wy;
  a.off_by = off_by;
  a.window = window;
  a.out = out;
  a.status = status;
  // Cluster size: the waves that the B clusters need at that size times one
  // row's time, its products at the FP32 rate plus a fixed latency per layer
  // (partial sums, gates, exchange: about 1500 clocks).  Sizes above 8 are
  // the non-portable ones; at 2 x 256 seven clusters of 16 run at once, or
  // eight of 12, so 8 samples take 12 (one wave).
  auto shape = [&](int CS) {
    a.CS = CS;
    a.U = even_up((H + CS - 1) / CS);
    a.SL = std::min(kPipeThreads / (2 * a.U), std::max(1, std::min(16, H / 8)));
    a.threads = a.SL * 2 * a.U;
    return a.SL < 1 ? (size_t)-1 : pipe_smem_bytes(I, H, L, O, a.U, CS, 2 * np, a.SL, wsz);
  };
  // Whole call in us, measured at seven networks (20 to 256 units, windows of 4
  // to 16), 1 to 4096 samples, 1 to 200 steps, BF16 and FP32 weights: each wave
  // loads the weights (0.56 us per 1000 of a CTA) and runs T + steps rows of L
  // phases and the products; within a fifth of the measured times.
  auto call_us = [&](int waves) {
    double weights = 0.0;
    for (int l = 0; l < L; ++l) weights += 4.0 * a.U * ((l == 0 ? I : H) + H);
    const double products = 4.0 * a.U * 2 * np * (2.0 * L - 1.0) * H / 128.0;  // clocks
    const double row = 0.6 + 1.45 * L + 1.9 * products / 2030.0 + 0.2 * L * std::max(0, 2 * np - 12);
    return 25.0 + waves * (4.0 + 0.56e-3 * weights + (T + steps) * row);
  };
  // no cluster size can do better than all samples at once on the fewest units
  shape(16);
  if (call_us(1) > limit_us) return cudaErrorInvalidConfiguration;
  int pick = 0, waves = 1;
  double best = 0.0;
  for (int CS : {16, 12, 8, 4, 2, 1}) {
    const size_t smem = shape(CS);
    if (smem > kPipeSmemMax || (CS > 1 && H < 2 * CS)) continue;
    const int active = bf16_weights ? pipe_active<__nv_bfloat16>(a, np, smem)
                                    : pipe_active<float>(a, np, smem);
    if (active < 1) continue;
    const double products = 4.0 * a.U * 2 * np * (2.0 * L - 1.0) * H / 128.0;
    const int w = (B + active - 1) / active;
    const double cost = (double)w * (1.5 * products + 1500.0 * L);
    if (!pick || cost < best) {
      pick = CS;
      best = cost;
      waves = w;
    }
  }
  if (!pick) return cudaErrorInvalidConfiguration;
  const size_t smem = shape(pick);
  if (call_us(waves) > limit_us) return cudaErrorInvalidConfiguration;
  const cudaError_t e = bf16_weights ? pipe_np<__nv_bfloat16>(st, a, B, np, smem, nullptr)
                                     : pipe_np<float>(st, a, B, np, smem, nullptr);
  if (e == cudaSuccess) note_launch();
  return e;
}

// Runs the self-test kernel and returns the status word it left (after
// synchronising the stream).
cudaError_t grid_sync_selftest(cudaStream_t st, double seconds, unsigned* status_out) {
  const unsigned zero[4] = {0u, 0u, 0u, 0u};
  cudaError_t e = cudaMemcpyToSymbolAsync(g_selftest_words, zero, sizeof(zero), 0,
                                          cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e;
  uint64_t limit = (uint64_t)(seconds * 1e9);
  void* args[] = {&limit};
  e = cudaLaunchCooperativeKernel((void*)k_grid_sync_selftest, dim3(2), dim3(32), args, 0, st);
  note_launch();
  if (e != cudaSuccess) return e;
  unsigned w[4];
  e = cudaMemcpyFromSymbolAsync(w, g_selftest_words, sizeof(w), 0, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  *status_out = w[2];
  return e;
}

}  // namespace rpod
