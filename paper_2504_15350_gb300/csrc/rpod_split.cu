// FP32 products with a skinny operand on the bf16 tensor cores: the passes
// over S of the plain FP32 form (S Lambda, S^T Q, S Z, Q^T S of Alg. 1,
// Sec. 4.2), its CholeskyQR applies and lift, the FP16 form's refinement pass
// and the projection of FP32 snapshots.
//
//   D(i, c) = sum_k A(i, k) B(k, c),  i < M, c < N <= 128, k < K
//
// Every FP32 value is split into three bf16 parts x = x1 + x2 + x3 (x1 the
// upper 16 bits, x2 the rest rounded to nearest, x3 what remains: 8 + 8 + 8
// significant bits), exactly for |x| above 2^-110 (below, x3 leaves bf16's
// range: an error of at most 2^-134), and the six products
//   a3 b1, a1 b3, a2 b2, a2 b1, a1 b2, a1 b1
// are accumulated.  Of the three dropped, a2 b3 and a3 b2 are at most 2^-23 of a
// b each, since a truncated x1 leaves up to 2^-7 of x to x2 and 2^-16 to x3, and
// about 2^-26 with random signs, below the rounding of one FP32 product (2^-24);
// a3 b3 is at most 2^-32.  An infinity becomes inf + NaN: what it reaches is NaN,
// as in the kernel this replaces.  The tensor
// core's own FP32 accumulation does not round to nearest, so an accumulator
// takes the products of 64 values of k only (the small ones first) and is
// then added to FP32 sums in registers.  Measured against 64 bits, products of
// random values are off by 0.9 (K = 10) to 1.6 (K = 300) times 2^-24 of the
// result's norm, those of the FP32 FMA kernel this replaces by 1.1 to 5.2.
//
// One CTA per SM walks over work items (a tile of 128 rows of D, a range of
// k).  Per 64 values of k:
//   warp 0       TMA of the raw FP32 tile of A (32 KB) into a ring
//   warp 18      TMA of B's three planes (split once by k_split3) into a ring
//   warps 2-9    two groups of four: a thread owns one row of the tile, splits
//                its 64 values and stores the packed parts to TMEM (tcgen05.st)
//   warp 1       24 MMAs, A from TMEM, B from shared memory, into one of two
//                accumulators
//   warps 10-17  add the finished accumulator to their FP32 sums (one TMEM
//                lane quarter and half of the columns each); at the end of an
//                item they store its tile
// A takes its parts through TMEM, so that neither converted tiles nor the
// skinny side's re-reads load the shared memory, which a 128 x 128 MMA with
// both operands there would saturate.  An A that TMA cannot address (base or
// leading dimension not a multiple of 16 bytes) is staged by 4-byte cp.async
// from warps 0, 19 and 20 instead.
//
// Bound: 6 bf16 products per value, so at N = 128 the tensor cores need as
// long for a tile as HBM (1536 clocks per 32 KB at 4096 FMA a clock and SM);
// at N = 64 HBM alone.  Measured (kernel alone, products of 1.05 GB, 155 us of
// HBM): S^T Q at 65536 x 4000, l = 120, 245 us and S Z 267 us (1640 and 1600 us on
// the FP32 pipes); at 4096 x 64000, l = 60, 205 and 170 us (1400 and 6600 us, the
// latter on 32 CTAs).
#include <algorithm>
#include <mutex>

#include "rpod_ptx.cuh"
#include "rpod_split.cuh"

namespace rpod {
namespace tc {

template <int NT>
struct SplitSmem {
  static constexpr int RS = NT == 128 ? 2 : (NT == 96 ? 3 : 4);  // raw slots
  static constexpr int BS = NT == 32 ? 4 : 3;                    // B stages
  static constexpr uint32_t RAW = 32768;
  static constexpr uint32_t PLANE = NT * 128;
  static constexpr uint32_t BST = 3 * PLANE;
  static constexpr uint32_t BARS = RS * RAW + BS * BST;
  static constexpr size_t TOTAL = 1024 + (size_t)BARS + 256;
};

// x = x1 + x2 + x3 for two values; parts packed as bf16 pairs (low half a)
__device__ __forceinline__ void split3(float a, float b, uint32_t& p1, uint32_t& p2, uint32_t& p3) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  p1 = __byte_perm(ua, ub, 0x7632);
  const float ra = a - __uint_as_float(ua & 0xffff0000u), rb = b - __uint_as_float(ub & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p2) : "f"(rb), "f"(ra));
  const float qa = ra - __uint_as_float(p2 << 16), qb = rb - __uint_as_float(p2 & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p3) : "f"(qb), "f"(qa));
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// A from TMEM (a: its first column), B from shared memory
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"(acc));
}

struct SplitArgs {
  const float* A;
  int64_t lda, M, K;
  int N, kbs, kb_per;            // k-blocks of 64 in all and per item
  int64_t tiles, items;
  float* out;                    // out[z * osplit + i * di + c * dj]
  int64_t di, dj, osplit;
  unsigned* status;
  int check;                     // flag non-finite values of A
};

// KC: A(i, k) = A[k + i lda] (k contiguous), else A[i + k lda].  TMA: tmA
// describes A as it lies in memory (box {32, 128} swizzled when KC, else
// {128, 64} plain); tmB the planes, K x 3 N.
template <int NT, bool KC, bool TMA>
__global__ void __launch_bounds__(TMA ? 608 : 672, 1)
k_split_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
             const __grid_constant__ SplitArgs g) {
  using L = SplitSmem<NT>;
  constexpr int RS = L::RS, BS = L::BS;
  constexpr int NH = NT / 2;      // columns of one drain warp
  constexpr uint32_t TA = 256;    // first TMEM column of A's parts: 2 stages x 3 x 32
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem1024(smem_raw);
  uint8_t* bsm = smem + RS * L::RAW;
  uint64_t* rfull = (uint64_t*)(smem + L::BARS);
  uint64_t* rempty = rfull + RS;
  uint64_t* bfull = rempty + RS;
  uint64_t* bempty = bfull + BS;
  uint64_t* aready = bempty + BS;  // [2] parts of a k-block are in TMEM
  uint64_t* mdone = aready + 2;    // [2] its MMAs are done: parts free, sums ready
  uint64_t* dempty = mdone + 2;    // [2] accumulator read
  uint32_t* tslot = (uint32_t*)(dempty + 2);
  volatile int* abort_flag = (volatile int*)(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < RS; ++s) {
      mbar_init(&rfull[s], TMA ? 1 : 96);
      mbar_init(&rempty[s], 4);
    }
    for (int s = 0; s < BS; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bempty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&aready[s], 4);
      mbar_init(&mdone[s], 1);
      mbar_init(&dempty[s], 8);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc(tslot, 512);
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = *tslot;

  // Every role walks over the same items and counts k-blocks in `it`.
  if (warp == 0 && TMA) {
    if (elect_one()) {
      int it = 0;
      bool go = true;
      for (int64_t w = blockIdx.x; w < g.items && go; w += gridDim.x) {
        const int i0 = (int)(w % g.tiles) * 128, kb0 = (int)(w / g.tiles) * g.kb_per;
        const int kb1 = min(kb0 + g.kb_per, g.kbs);
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
          const int s = it % RS;
          const uint32_t ph = (uint32_t)(it / RS) & 1u;
          if (it >= RS && !mbar_wait(&rempty[s], ph ^ 1u, abort_flag)) { go = false; break; }
          uint8_t* dst = smem + s * L::RAW;
          mbar_expect_tx(&rfull[s], L::RAW);
          if (KC) {
            tma_load_2d(dst, &tmA, &rfull[s], kb * 64, i0);
            tma_load_2d(dst + 16384, &tmA, &rfull[s], kb * 64 + 32, i0);
          } else {
            tma_load_2d(dst, &tmA, &rfull[s], i0, kb * 64);
          }
        }
      }
      if (*abort_flag)
        for (int j = it > RS ? it - RS : 0; j < it; ++j)
          mbar_wait_drain(&rfull[j % RS], (uint32_t)(j / RS) & 1u);
    }
  } else if (warp == 18) {
    if (elect_one()) {
      int it = 0;
      bool go = true;
      for (int64_t w = blockIdx.x; w < g.items && go; w += gridDim.x) {
        const int kb0 = (int)(w / g.tiles) * g.kb_per, kb1 = min(kb0 + g.kb_per, g.kbs);
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
          const int s = it % BS;
          const uint32_t ph = (uint32_t)(it / BS) & 1u;
          if (it >= BS && !mbar_wait(&bempty[s], ph ^ 1u, abort_flag)) { go = false; break; }
          mbar_expect_tx(&bfull[s], L::BST);
#pragma unroll
          for (int p = 0; p < 3; ++p)
            tma_load_2d(bsm + s * L::BST + p * L::PLANE, &tmB, &bfull[s], kb * 64, p * g.N);
        }
      }
      if (*abort_flag)
        for (int j = it > BS ? it - BS : 0; j < it; ++j)
          mbar_wait_drain(&bfull[j % BS], (uint32_t)(j / BS) & 1u);
    }
  } else if (warp == 1) {
    if (elect_one()) {
      constexpr uint32_t id = idesc(1, false, 128, NT);
      int it = 0;
      bool go = true;
      for (int64_t w = blockIdx.x; w < g.items && go; w += gridDim.x) {
        const int kb0 = (int)(w / g.tiles) * g.kb_per, kb1 = min(kb0 + g.kb_per, g.kbs);
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
          const int s = it & 1, bs = it % BS;
          const uint32_t ph = (uint32_t)(it >> 1) & 1u;
          if (!mbar_wait(&aready[s], ph, abort_flag) ||
              !mbar_wait(&bfull[bs], (uint32_t)(it / BS) & 1u, abort_flag) ||
              (it >= 2 && !mbar_wait(&dempty[s], ph ^ 1u, abort_flag))) {
            go = false;
            break;
          }
          tc_after();
          const uint32_t d = tmem + (uint32_t)(s * NT), a = tmem + TA + (uint32_t)(s * 96);
          const uint32_t b = su32(bsm + bs * L::BST);
          // (part of A, part of B), the smallest products first
          const int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
          for (int t = 0; t < 6; ++t)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_ts(d, a + (uint32_t)(pa[t] * 32 + kk * 8),
                     sdesc(b + (uint32_t)pb[t] * L::PLANE + 32 * kk, 16, 1024), id,
                     (t > 0 || kk > 0) ? 1u : 0u);
          mma_commit(&bempty[bs]);
          mma_commit(&mdone[s]);
        }
      }
      // MMAs in flight end before TMEM is released
      for (int j = it > 2 ? it - 2 : 0; j < it; ++j)
        mbar_wait_drain(&mdone[j & 1], (uint32_t)(j >> 1) & 1u);
    }
  } else if (warp >= 2 && warp < 10) {
    const int grp = (warp - 2) >> 2, row = (warp & 3) * 32 + lane;
    const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + TA + (uint32_t)(grp * 96);
    uint32_t top = 0;
    int it = 0;
    bool go = true;
    for (int64_t w = blockIdx.x; w < g.items && go; w += gridDim.x) {
      const int kb0 = (int)(w / g.tiles) * g.kb_per, kb1 = min(kb0 + g.kb_per, g.kbs);
      for (int kb = kb0; kb < kb1; ++kb, ++it) {
        if ((it & 1) != grp) continue;
        const int s = it % RS;
        // the parts' stage first: its last MMAs come after those of k-block
        // it - 3, the last one in this raw slot when RS is 3, so the slot's
        // barrier cannot be a whole phase behind the parity waited for
        bool ok = it < 2 || mbar_wait(&mdone[grp], ((uint32_t)(it >> 1) & 1u) ^ 1u, abort_flag);
        if (ok) ok = mbar_wait(&rfull[s], (uint32_t)(it / RS) & 1u, abort_flag);
        if (!__all_sync(0xffffffffu, ok)) { go = false; break; }
        tc_after();
        const uint8_t* raw = smem + s * L::RAW;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float x[16];
          if (KC) {
            const uint8_t* rp = raw + (c >> 1) * 16384 + row * 128;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float4 v = *(const float4*)(rp + ((((c & 1) * 4 + u) ^ (row & 7)) << 4));
              x[4 * u] = v.x; x[4 * u + 1] = v.y; x[4 * u + 2] = v.z; x[4 * u + 3] = v.w;
            }
          } else {
            const float* rp = (const float*)raw + c * 16 * 128 + row;
#pragma unroll
            for (int u = 0; u < 16; ++u) x[u] = rp[u * 128];
          }
          if (g.check) {
#pragma unroll
            for (int u = 0; u < 16; ++u) top = max(top, __float_as_uint(x[u]) & 0x7fffffffu);
          }
          uint32_t p1[8], p2[8], p3[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) split3(x[2 * u], x[2 * u + 1], p1[u], p2[u], p3[u]);
          tmem_st8(ta + (uint32_t)(c * 8), p1);
          tmem_st8(ta + (uint32_t)(32 + c * 8), p2);
          tmem_st8(ta + (uint32_t)(64 + c * 8), p3);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&rempty[s]);
          mbar_arrive(&aready[grp]);
        }
      }
    }
    if (g.check && top >= 0x7f800000u) atomicOr(g.status, ST_NONFINITE);
  } else if (warp >= 10 && warp < 18) {
    const int q = warp & 3, half = (warp - 10) >> 2;
    const uint32_t td = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * NH);
    int it = 0;
    bool go = true;
    for (int64_t w = blockIdx.x; w < g.items && go; w += gridDim.x) {
      const int64_t z = w / g.tiles;
      const int kb0 = (int)z * g.kb_per, kb1 = min(kb0 + g.kb_per, g.kbs);
      float acc[NH];
#pragma unroll
      for (int i = 0; i < NH; ++i) acc[i] = 0.f;
      for (int kb = kb0; kb < kb1; ++kb, ++it) {
        const int s = it & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(&mdone[s], (uint32_t)(it >> 1) & 1u, abort_flag))) {
          go = false;
          break;
        }
        tc_after();
#pragma unroll
        for (int c = 0; c < NH; c += 16) {
          float v[16];
          tmem_ld16(td + (uint32_t)(s * NT + c), v);
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[c + i] += v[i];
        }
        tc_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&dempty[s]);
      }
      const int64_t i = (w % g.tiles) * 128 + q * 32 + lane;
      if (go && i < g.M) {
        float* o = g.out + z * g.osplit + i * g.di + (int64_t)half * NH * g.dj;
#pragma unroll
        for (int c = 0; c < NH; ++c)
          if (half * NH + c < g.N) o[c * g.dj] = acc[c];
      }
    }
  } else if (!TMA && (warp == 0 || warp >= 19)) {
    // Three warps, each a line of the tile (!KC: 128 rows of one k; KC: 64 k of
    // one row) in turn.  A whole tile takes the loop without conditions, whose
    // 32 copies in flight per lane hide the loads' latency: with a condition and
    // an index computation per copy, about five were in flight, and a k-block took
    // 8.7 us (!KC) or 4.2 us; now 1.1 us.  S^T Q and S Z of 65537 x 4000 by
    // 128: 428 and 390 us (FP32 FMAs 1950 us).
    const int w3 = warp == 0 ? 0 : warp - 18;
    constexpr int LN = KC ? 128 : 64, PER = KC ? 2 : 4;  // lines, 32-value pieces of one
    int it = 0;
    bool go = true;
    for (int64_t w = blockIdx.x; w < g.items && go; w += gridDim.x) {
      const int64_t i0 = (w % g.tiles) * 128;
      const int kb0 = (int)(w / g.tiles) * g.kb_per, kb1 = min(kb0 + g.kb_per, g.kbs);
      for (int kb = kb0; kb < kb1; ++kb, ++it) {
        const int s = it % RS;
        if (it >= RS && !mbar_wait(&rempty[s], ((uint32_t)(it / RS) & 1u) ^ 1u, abort_flag)) {
          go = false;
          break;
        }
        const int64_t k0 = (int64_t)kb * 64, l0 = KC ? i0 : k0, c0 = KC ? k0 : i0;
        const int nl = (int)min((int64_t)LN, (KC ? g.M : g.K) - l0);  // lines inside A
        const int nc = (int)min((int64_t)(32 * PER), (KC ? g.K : g.M) - c0) - lane;  // a line's values from here on
        const uint32_t dst = su32(smem + s * L::RAW);
        const float* src = g.A + c0 + lane + (l0 + w3) * g.lda;
        auto at = [&](int ln, int h) {  // byte offset in the slot
          return KC ? (uint32_t)(h * 16384 + ln * 128 + (((lane >> 2) ^ (ln & 7)) << 4) + (lane & 3) * 4)
                    : (uint32_t)(ln * 512 + (32 * h + lane) * 4);
        };
        if (nl == LN && nc + lane == 32 * PER) {
#pragma unroll 8
          for (int ln = w3; ln < LN; ln += 3, src += 3 * g.lda) {
#pragma unroll
            for (int h = 0; h < PER; ++h)
              asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + at(ln, h)), "l"(src + 32 * h)
                           : "memory");
          }
        } else {
          for (int ln = w3; ln < LN; ln += 3, src += 3 * g.lda) {
#pragma unroll
            for (int h = 0; h < PER; ++h) {
              const bool in = ln < nl && 32 * h < nc;
              asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + at(ln, h)),
                           "l"(in ? src + 32 * h : g.A), "r"(in ? 4 : 0)
                           : "memory");
            }
          }
        }
        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(su32(&rfull[s])) : "memory");
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  __syncwarp();
  if (threadIdx.x == 0 && *abort_flag) atomicOr(g.status, ST_TIMEOUT);
  tc_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// Planes of B: P[p (N ldp) + c ldp + k] = part p of B[k + c ldb], two values
// per thread.
__global__ void __launch_bounds__(256)
k_split3(int64_t K, const float* __restrict__ B, int64_t ldb, uint32_t* __restrict__ P, int64_t ldp,
         int64_t plane) {
  const int64_t k = 2 * ((int64_t)blockIdx.x * 256 + threadIdx.x);
  if (k >= K) return;
  const float* b = B + k + (int64_t)blockIdx.y * ldb;
  const float x = b[0], y = k + 1 < K ? b[1] : 0.f;
  uint32_t p1, p2, p3;
  split3(x, y, p1, p2, p3);
  uint32_t* o = P + (k + (int64_t)blockIdx.y * ldp) / 2;
  o[0] = p1;
  o[plane / 2] = p2;
  o[plane] = p3;
}

template <int NT, bool KC, bool TMA>
static void split_launch(cudaStream_t st, unsigned grid, const CUtensorMap& ta, const CUtensorMap& tb,
                         const SplitArgs& g) {
  static std::once_flag once;
  std::call_once(once, [] {
    cudaFuncSetAttribute(k_split_gemm<NT, KC, TMA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)SplitSmem<NT>::TOTAL);
  });
  k_split_gemm<NT, KC, TMA><<<grid, TMA ? 608 : 672, SplitSmem<NT>::TOTAL, st>>>(ta, tb, g);
}

template <bool KC, bool TMA>
static void split_launch_n(cudaStream_t st, unsigned grid, const CUtensorMap& ta,
                           const CUtensorMap& tb, const SplitArgs& g) {
  if (g.N <= 32) split_launch<32, KC, TMA>(st, grid, ta, tb, g);
  else if (g.N <= 64) split_launch<64, KC, TMA>(st, grid, ta, tb, g);
  else if (g.N <= 96) split_launch<96, KC, TMA>(st, grid, ta, tb, g);
  else split_launch<128, KC, TMA>(st, grid, ta, tb, g);
}

}  // namespace tc

size_t split_plane_bytes(int64_t K, int N) {
  return (size_t)6 * (size_t)((K + 63) / 64 * 64) * (size_t)N;
}

int split_count(int64_t M, int64_t K, int N, size_t max_elems) {
  const int64_t tiles = (M + 127) / 128, kbs = (K + 63) / 64, sms = split_sm_count();
  int best = 1;
  double cost = 0.0;
  for (int s = 1; s <= 64 && s <= kbs; ++s) {
    if (s > 1 && (size_t)s * (size_t)M * (size_t)N > max_elems) break;
    const int64_t per = (kbs + s - 1) / s;
    const int64_t waves = (tiles * s + sms - 1) / sms;
    // in k-block times (about 0.5 us): the busiest CTA's k-blocks, one per
    // item for its start and store, and the partial sums' traffic
    const double c = (double)(waves * (per + 1)) +
                     (s > 1 ? 6.0 + (double)s * (double)M * (double)N * 8.0 / 2.5e6 : 0.0);
    if (s == 1 || c < cost) {
      best = s;
      cost = c;
    }
  }
  return best;
}

int split_sm_count() {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
    return v;
  cudaGetLastError();
  return 152;
}

int split_gemm(cudaStream_t st, bool kc, int64_t M, int N, int64_t K, const float* A, int64_t lda,
               const float* B, int64_t ldb, float* D, int64_t di, int64_t dj, void* planes, float* part,
               size_t part_elems, int pct, unsigned* status, bool check) {
  if (N < 1 || N > 128 || M < 1 || K < 1) return RPOD_ERR_INVALID_ARG;
  const int64_t ldp = (K + 63) / 64 * 64;
  tc::SplitArgs g;
  g.A = A; g.lda = lda; g.M = M; g.K = K; g.N = N;
  g.kbs = (int)(ldp / 64);
  g.tiles = (M + 127) / 128;
  int s = split_count(M, K, N, part ? part_elems : 0);
  if (pct != 100) s = std::max(1, std::min((int)((int64_t)s * pct / 100), s));
  g.kb_per = (g.kbs + s - 1) / s;
  s = (g.kbs + g.kb_per - 1) / g.kb_per;
  g.items = g.tiles * s;
  g.out = s > 1 ? part : D;
  g.di = s > 1 ? 1 : di;
  g.dj = s > 1 ? M : dj;
  g.osplit = s > 1 ? M * N : 0;
  g.status = status;
  g.check = check ? 1 : 0;
  CUtensorMap ta, tb;
  const int nt = N <= 32 ? 32 : (N <= 64 ? 64 : (N <= 96 ? 96 : 128));
  if (int rc = make_map(&tb, planes, RPOD_BF16, K, 3 * (int64_t)N, ldp, 64, nt)) return rc;
  int rc = kc ? make_map(&ta, A, RPOD_F32, K, M, lda, 32, 128)
              : make_map(&ta, A, RPOD_F32, M, K, lda, 128, 64, false);
  if (rc == RPOD_ERR_CUDA) return rc;
  const bool tma = rc == RPOD_OK;
  if (!tma) ta = tb;  // not read
  dim3 sg((unsigned)((K + 511) / 512), (unsigned)N);
  tc::k_split3<<<sg, 256, 0, st>>>(K, B, ldb, (uint32_t*)planes, ldp, (int64_t)N * ldp);
  note_launch();
  const unsigned grid = (unsigned)std::min<int64_t>(g.items, split_sm_count());
  if (kc) {
    if (tma) tc::split_launch_n<true, true>(st, grid, ta, tb, g);
    else tc::split_launch_n<true, false>(st, grid, ta, tb, g);
  } else {
    if (tma) tc::split_launch_n<false, true>(st, grid, ta, tb, g);
    else tc::split_launch_n<false, false>(st, grid, ta, tb, g);
  }
  note_launch();
  if (cudaGetLastError() != cudaSuccess) return RPOD_ERR_CUDA;
  if (s > 1 && reduce_splits<float, float>(st, M, N, s, part, D, di, dj) != cudaSuccess) return RPOD_ERR_CUDA;
  return RPOD_OK;
}

}  // namespace rpod
