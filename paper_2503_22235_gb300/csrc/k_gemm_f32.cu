// FP32 linear layers on the tensor cores: out = epilogue(A[M, K] . W[N, K]^T + bias)
// with FP32 operands, FP32 accuracy and FP32 accumulation.
//
// Each operand value is split into three bf16 numbers, a = a1 + a2 + a3, by
// rounding to nearest and taking the remainder twice. The split is exact: a
// float has 24 significant bits, every remainder is a float, and the last one
// has at most 8 bits left. A product is then the six bf16 products a1 b1,
// a1 b2, a2 b1, a1 b3, a2 b2, a3 b1, each exact in the tensor core; the ones
// left out (a2 b3, a3 b2, a3 b3) are below 2^-25 of a b with either sign,
// under half a unit in the last place of the product. The tensor core's FP32
// accumulator runs over 64 values of k only, smallest products of all 64
// first, so that sums at full size meet at most four of its additions (it
// truncates); these partial sums are added in registers, rounding to nearest.
// Relative L2 error against float64, a chain of K FP32 FMAs and here:
// K = 128 2.1e-7 and 8.3e-8, K = 768 5.0e-7 and 1.0e-7, K = 3072 9.9e-7 and
// 1.5e-7; with one accumulator over 64 k in the order the slabs arrive,
// K = 128 had 3.1e-7.
//
// Persistent, one CTA per SM; a slab is 32 values of k, an accumulator two
// slabs:
//   splitting  (four warps, eight when W is split here too) read the slab's
//              rows of A from shared memory (tensor copies, 128-byte swizzle)
//              and write the three planes of A to tensor memory; W's planes
//              lie in shared memory, 64-byte swizzle
//   one warp issues the 12 tcgen05.mma of a slab (A from tensor memory, W
//              from shared memory; M = 128, N = BN, K = 16)
//   one thread issues the tensor copies of A's slabs and W's planes
//   summing    (eight warps) add a finished accumulator to their register
//              sums; at the end of a tile bias, erf GELU, and the tile leaves
//              by tensor copies (tensor reductions for the residual add)
// What bounds it: at M = N = 128 an MMA with both operands in shared memory
// reads 8 KB in 64 clocks, the whole 128 bytes a clock, and every other use of
// shared memory then stalls it: with A's planes there the same pipeline ran a
// slab in 1750 clocks, with A in tensor memory in about 1050 (768 are MMA
// time). Wider tiles do not fit the register sums (64 a thread here).
// Weights that come ready as planes save the CTA two thirds of the splitting:
// M = 145800, N = 768, K = 3072 took 4.8 ms with W split inside, 2.70 ms with
// planes (2.38 with the converged MMA warp below), 13.5 ms as FP32 FMAs on CUDA
// cores: 51 TFLOP/s, now 289.
// M = 20475, N = 1536, K = 384 with GELU: 559 us before, 149 so; M = 4608,
// N = 512, K = 128 with GELU: 22.5 and 15.2 us. The loop that issues the MMAs
// inside one lane's branch left the tensor pipe idle between slabs; walked by
// the whole warp, one elected lane issuing: 149 -> 136 us, a block of 145,800
// tokens (C = 768) 13.41 -> 12.51 ms, both the same within 1 % with the look for
// small operands below.
//
// NaN and infinity: a non-finite operand (or one that rounds up to infinity)
// makes its second plane NaN, so every sum it enters comes out NaN. Sums that
// are not finite are recomputed by the chain of FP32 FMAs.
// Small operands: the tensor core takes bf16 subnormals as zero, so an operand
// may lose up to 2^-125 of itself (below 2^-110 its last planes, below 2^-126
// all), and a product up to 2^-126. Where neither the row of A nor W has an
// operand below 2^-48 (but zeros) nothing of that kind reaches 2^-25 of a
// product. Else a sum of K products is off by at most K 2^-125 (max|w| + 3),
// and K 2^-125 max|a| more where W has one: sums below 2^25 times that, zeros
// included, are recomputed too. Ordinary sums are far above, whatever the
// operands, so the epilogue compares first (with 2^30 for max|a|; a row that
// passes it, which matters where W has small ones, is marked as it is split)
// and looks for small operands in the row of A only where a sum is below. Where
// it finds none (zero columns of W, zero rows), the splitting tests every
// operand from then on, which costs 2 to 4 % (72,900 x 768 x 768: 350 us, 415
// with a zero column, 610 with a look at every such row). W's range comes from
// the pre-pass, or from the splitting here.
//
// Every wait is bounded in time; on a timeout the CTA records WM_ERR_TIMEOUT,
// its MMAs are drained, TMEM is freed and it returns.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "tc_gemm.cuh"

namespace wm {
namespace f32tc {

using namespace ptx;
using namespace tc;

constexpr int BM = 128, BK = 32;        // rows of A per tile, k per slab
constexpr int GROUP = 2;                // slabs per accumulator
constexpr int ROW = 2 * BK;             // bytes of a W plane's row
constexpr int NA = 4, NST = 4;          // slabs of A in shared memory; of W planes and of A planes (tensor memory)
constexpr int A_BYTES = BM * BK * 4;    // a slab of A, fp32, 128-byte swizzle
constexpr int A_COLS = 3 * BK / 2;      // tensor-memory columns of a slab's A planes (two k a column)
constexpr uint32_t T_A = 256;           // they follow the accumulators

template <int BN, bool PRE>
struct Cfg {
  // splitting warps: four for A alone, eight for A and W; then eight that sum, one that issues MMAs, one for copies
  static constexpr int CONV = PRE ? 4 : 8, EPI = CONV, MMA_WARP = CONV + 8, TMA_WARP = CONV + 9;
  static constexpr int THREADS = 32 * (CONV + 10);
  static constexpr int PLANE = BN * ROW, STAGE = 3 * PLANE;
  static constexpr int OFF_A = NST * STAGE;            // A slabs
  static constexpr int OFF_OUT = OFF_A + NA * A_BYTES; // 32 x 32 output chunks, two per epilogue warp
  static constexpr int SMEM = OFF_OUT + 16 * 4096 + 1024;   // + alignment slack
  static constexpr int NACC = 256 / BN;                // accumulators
};
static_assert(T_A + NST * A_COLS <= 512, "tensor memory");
static_assert(GROUP == 2 && NST >= 3, "the MMA loop takes the slabs of an accumulator two by two");

// Shared-memory matrix descriptor: K-major, 64-byte swizzle (16-byte unit u of
// row r at u ^ ((r >> 1) & 3)), rows of 64 bytes, 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&p);
}
// (x0, x1) -> packed bf16 pair, and the exact remainders
__device__ __forceinline__ uint32_t split2(float& x0, float& x1) {
  const uint32_t p = bf16x2(x0, x1);
  sub_f2(x0, x1, x0, x1, pack_f2(__uint_as_float(p << 16), __uint_as_float(p & 0xffff0000u)));
  return p;
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }

// Element (r, c) of a 32 x 32 staging tile (128-byte swizzle, as the output's tensor map has it).
__device__ __forceinline__ float* stage_at(uint8_t* stg, int r, int c) {
  return reinterpret_cast<float*>(stg + r * 128 + (((c >> 2) ^ (r & 7)) << 4) + (c & 3) * 4);
}

constexpr float kSmall = 3.552713679e-15f, kLarge = 1073741824.f;   // 2^-48, 2^30
constexpr float kMaxFloat = 3.402823466e38f;

// What operands span: the largest magnitude, and the smallest but zero (twice
// its bits, less one). An infinity makes every sum it enters NaN: it counts for
// no maximum.
struct Range {
  float hi = 0.f;
  uint32_t lo = 0xffffffffu;
  template <int N>
  __device__ __forceinline__ void add(const float (&x)[N]) {
    float m = 0.f;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      m = fmaxf(m, fabsf(x[j]));
      lo = __viaddmin_u32(__float_as_uint(x[j]) << 1, 0xffffffffu, lo);
    }
    if (m <= kMaxFloat) hi = fmaxf(hi, m);
  }
  // as one word: the magnitude, and the sign bit where one but zero is small
  __device__ __forceinline__ uint32_t word() const {
    return __float_as_uint(hi) | (lo < (__float_as_uint(kSmall) << 1) - 1u ? 0x80000000u : 0u);
  }
};
__device__ __forceinline__ uint32_t range_merge(uint32_t a, uint32_t b) {
  return max(a & 0x7fffffffu, b & 0x7fffffffu) | ((a | b) & 0x80000000u);
}
__device__ __forceinline__ uint32_t range_of_warp(uint32_t a) {
  return __reduce_max_sync(0xffffffffu, a & 0x7fffffffu) | (__reduce_or_sync(0xffffffffu, a) & 0x80000000u);
}

// Sums below this are recomputed, by the ranges of A's row (its magnitude at most a_hi) and of W.
__device__ __forceinline__ float doubt_below(float a_hi, uint32_t w, int K) {
  if (w == 0u) return 0.f;   // W is zero
  return (float)K * 3.155443621e-30f *   // 2^-98
         (1.f + __uint_as_float(w & 0x7fffffffu) + ((w >> 31) != 0u ? a_hi : 0.f));
}
__device__ __forceinline__ bool doubtful(float y, float below) {
  return !(fabsf(y) >= below) || !(fabsf(y) <= kMaxFloat);
}

// The threshold of this lane's row of A (from row0 on), for the rows in `look`;
// w: W's range.
__device__ __forceinline__ float look_at_rows(const float* A, int row0, int K, uint32_t look, uint32_t w) {
  const int lane = threadIdx.x & 31;
  float below = 0.f;
  for (; look != 0u; look &= look - 1u) {
    const int r = __ffs(look) - 1;
    const float* a = A + (size_t)(row0 + r) * K;
    Range ra;
#pragma unroll 8
    for (int k = lane; k < K; k += 32) {
      const float x[1] = {__ldg(a + k)};
      ra.add(x);
    }
    const uint32_t range = range_of_warp(ra.word());
    if (lane == r && ((range | w) >> 31) != 0u) below = doubt_below(__uint_as_float(range & 0x7fffffffu), w, K);
  }
  return below;
}

// A staged chunk (rows row0 .., columns n ..) with sums that are not finite or
// below `first`: each lane's row, in doubt below `below` or, in the rows `look`,
// below what the row of A says, by the plain chain of FP32 FMAs. Returns
// whether the look was in vain.
__device__ __noinline__ bool recompute(uint8_t* stg, const float* A, const float* W, int row0, int M, int n, int N,
                                       int K, uint32_t look, float below, uint32_t w) {
  const int lane = threadIdx.x & 31;
  const float looked = look_at_rows(A, row0, K, look, w);
  const bool vain = look != 0u && (w >> 31) == 0u && !__any_sync(0xffffffffu, looked > 0.f);
  if ((look >> lane) & 1u) below = looked;
  if (row0 + lane >= M) return vain;
  const float* a = A + (size_t)(row0 + lane) * K;
#pragma unroll 1
  for (int e = 0; e < 32 && n + e < N; ++e) {
    float* y = stage_at(stg, lane, e);
    if (!doubtful(*y, below)) continue;
    const float* wn = W + (size_t)(n + e) * K;
    float s = 0.f;
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
      s = fmaf(a[k], wn[k], s);
      if (s != s) break;   // NaN stays NaN
    }
    *y = s;
  }
  return vain;
}

// Tensor-core product with A from tensor memory (lane = row, two k a column).
__device__ __forceinline__ void umma_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// TMA_A: A arrives by tensor copies (tmA; K % 4 == 0, 16-byte aligned), else by
// plain loads of each thread's row. PRE: W's planes come ready from global
// memory by tensor copies (tmW), else W is split here like A; VEC_W: by
// 128-bit loads.
template <int BN, bool TMA_A, bool PRE, bool VEC_W>
__global__ void __launch_bounds__(Cfg<BN, PRE>::THREADS, 1)
    gemm_f32_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW,
                       const __grid_constant__ CUtensorMap tmC, const float* __restrict__ A, const float* __restrict__ W,
                       const float* __restrict__ bias,
                       float* out, int M, int N, int K, int epi, int tma_out, const uint32_t* __restrict__ w_ranges,
                       int num_ranges, int* __restrict__ status) {
  using CF = Cfg<BN, PRE>;
  constexpr int NACC = CF::NACC, CONV = CF::CONV;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t a_full[NA], a_empty[NA], planes_full[NST], planes_empty[NST];
  __shared__ __align__(8) uint64_t accf_bar[NACC], acce_bar[NACC], drain_bar;
  // Whether a row of the tile held an operand above 2^30 (where W has small ones) or a small one (from the tile a_from
  // of each splitting warp on, once a_watch asks for it), and the range of W by splitting warp; over all tiles so
  // far: the splitting runs ahead, so they may hold more than the tile at hand, never less
  __shared__ volatile uint32_t w_range[CONV];
  __shared__ volatile uint8_t a_large[BM], a_small[BM];
  __shared__ volatile int a_watch, a_from[CONV];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int num_n = (N + BN - 1) / BN;
  const int num_tiles = ((M + BM - 1) / BM) * num_n;
  const int nk = (K + BK - 1) / BK;

  if (tid == 0) {
    for (int s = 0; s < NA; ++s) {
      mbar_init(&a_full[s], 1);
      mbar_init(&a_empty[s], CONV);
    }
    for (int s = 0; s < NST; ++s) {
      mbar_init(&planes_full[s], CONV + (PRE ? 1 : 0));
      mbar_init(&planes_empty[s], 1);
    }
    for (int b = 0; b < NACC; ++b) {
      mbar_init(&accf_bar[b], 1);
      mbar_init(&acce_bar[b], 8);
    }
    mbar_init(&drain_bar, 1);
    abort_flag = 0;
    a_watch = 0;
    for (int i = 0; i < CONV; ++i) {
      w_range[i] = 0u;
      a_from[i] = 0x7fffffff;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (tid < BM) a_large[tid] = a_small[tid] = 0;
  uint32_t rw = 0u;   // range of W: all of it, where the pre-pass took it, else what this warp has split or seen split
  if constexpr (PRE) {
    for (int i = lane; i < num_ranges; i += 32) rw = range_merge(rw, __ldg(w_ranges + i));
    rw = range_of_warp(rw);
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp < CONV) {
    // ------------------------------------------------------- split into planes
    // A: this thread's row and KT of the slab's 32 k; W (not PRE): float4 q of rows r0 + 32 i
    constexpr int KT = 4 * CONV == 16 ? 32 : 16, LDW = PRE ? 0 : BN / 32;
    const int row = 32 * (warp & 3) + lane, hk = warp >> 2;
    const uint32_t ta = tmem + T_A + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(KT / 2 * hk);
    const int r0 = tid >> 3, q = tid & 7;
    // 8 bytes at 16-byte unit q / 2 of row r0 of a W plane (+ 32 i rows: the same swizzle)
    const uint32_t soff = (uint32_t)(r0 * ROW + (((q >> 1) ^ ((r0 >> 1) & 3)) << 4) + (q & 1) * 8);
    float4 v[PRE ? 1 : LDW];
    auto load_w = [&](int i, int n0, int k0) -> float4 {
      const int k = k0 + 4 * q, n = n0 + 32 * i + r0;
      const float* p = W + (size_t)n * K + k;
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
      if (n < N) {
        if constexpr (VEC_W) {
          if (k < K) t = __ldg(reinterpret_cast<const float4*>(p));
        } else {
          if (k < K) t.x = __ldg(p);
          if (k + 1 < K) t.y = __ldg(p + 1);
          if (k + 2 < K) t.z = __ldg(p + 2);
          if (k + 3 < K) t.w = __ldg(p + 3);
        }
      }
      return t;
    };
    if constexpr (!PRE) {
#pragma unroll
      for (int i = 0; i < LDW; ++i) v[i] = load_w(i, ((int)blockIdx.x % num_n) * BN, 0);
    }
    int stage = 0, ia = 0;
    uint32_t phase = 0, aphase = 0;
    bool ok = true, watch = (rw >> 31) != 0u;   // test the operands of A
    if (watch && lane == 0) a_from[warp] = 0;
    Range w_split;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
      const int m = (tile / num_n) * BM + row;
      if (PRE && !watch && __any_sync(0xffffffffu, a_watch != 0)) {
        watch = true;
        if (lane == 0) a_from[warp] = tile;
      }
      // (two loops: a branch in the one held up every slab, 3 % of a projection of 145,800 x 768 x 768)
      auto slabs = [&](auto tag) {
        constexpr bool kWatch = PRE && decltype(tag)::value;
        for (int kb = 0; kb < nk; ++kb) {
          float x[KT];
          if constexpr (TMA_A) {
            ok = __all_sync(0xffffffffu, mbar_wait(&a_full[ia], aphase, &abort_flag));
            if (!ok) return;
            const uint8_t* src = smem + CF::OFF_A + ia * A_BYTES + row * 128;
#pragma unroll
            for (int j = 0; j < KT / 4; ++j) {
              const float4 t = *reinterpret_cast<const float4*>(src + (((KT / 4 * hk + j) ^ (row & 7)) << 4));
              x[4 * j] = t.x; x[4 * j + 1] = t.y; x[4 * j + 2] = t.z; x[4 * j + 3] = t.w;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&a_empty[ia]);
            if (++ia == NA) {
              ia = 0;
              aphase ^= 1u;
            }
          } else {
            const int k0 = kb * BK + KT * hk;
            const float* p = A + (size_t)m * K + k0;
#pragma unroll
            for (int j = 0; j < KT; ++j) x[j] = m < M && k0 + j < K ? __ldg(p + j) : 0.f;
          }
          if constexpr (kWatch) {
            Range r;
            r.add(x);
            if (r.hi > kLarge) a_large[row] = 1;
            if ((r.word() >> 31) != 0u) a_small[row] = 1;
          }
          ok = __all_sync(0xffffffffu, mbar_wait(&planes_empty[stage], phase ^ 1u, &abort_flag));
          if (!ok) return;
          tc_fence_after();
#pragma unroll
          for (int pl = 0; pl < 3; ++pl)
#pragma unroll
            for (int h = 0; h < KT; h += 16) {
              uint32_t w[8];
#pragma unroll
              for (int j = 0; j < 8; ++j)
                w[j] = pl < 2 ? split2(x[h + 2 * j], x[h + 2 * j + 1]) : bf16x2(x[h + 2 * j], x[h + 2 * j + 1]);
              tmem_st8(ta + (uint32_t)(stage * A_COLS + pl * (BK / 2) + h / 2), w);
            }
          if constexpr (!PRE) {
            // the slab after this one
            const bool last = kb + 1 == nk;
            const int lt = last ? tile + (int)gridDim.x : tile;
            uint8_t* st = smem + stage * CF::STAGE + soff;
#pragma unroll
            for (int i = 0; i < LDW; ++i) {
              float4 y = v[i];
              const float y4[4] = {y.x, y.y, y.z, y.w};
              w_split.add(y4);
              if (lt < num_tiles) v[i] = load_w(i, (lt % num_n) * BN, last ? 0 : (kb + 1) * BK);
              uint8_t* d = st + i * 32 * ROW;
#pragma unroll
              for (int pl = 0; pl < 3; ++pl)
                *reinterpret_cast<uint2*>(d + pl * CF::PLANE) = pl < 2 ? make_uint2(split2(y.x, y.y), split2(y.z, y.w))
                                                                       : make_uint2(bf16x2(y.x, y.y), bf16x2(y.z, y.w));
            }
            if (last) {
              const uint32_t range = range_of_warp(w_split.word());
              if (lane == 0) w_range[warp] = range;
            }
            fence_async_smem();
          }
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&planes_full[stage]);
          if (++stage == NST) {
            stage = 0;
            phase ^= 1u;
          }
        }
      };
      if (PRE && watch) slabs(std::true_type{});
      else slabs(std::false_type{});
    }
    if (!ok) {
      abort_flag = 1;
      atomicExch(status, (int)WM_ERR_TIMEOUT);
    }
  } else if (warp == CF::TMA_WARP) {
    if ((TMA_A || PRE) && lane == 0) {
      // ------------------------------------ tensor copies: A slabs, W's planes
      int stage = 0, ia = 0, issued = 0;
      uint32_t phase = 0, aphase = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
        for (int kb = 0; kb < nk && ok; ++kb) {
          if constexpr (TMA_A) {
            ok = mbar_wait(&a_empty[ia], aphase ^ 1u, &abort_flag);
            if (!ok) break;
            mbar_expect_tx(&a_full[ia], A_BYTES);
            asm volatile(
                "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
                "%4}], [%2];" ::"r"(sbase + CF::OFF_A + ia * A_BYTES),
                "l"((uint64_t)&tmA), "r"(smem_u32(&a_full[ia])), "r"(kb * BK), "r"((tile / num_n) * BM)
                : "memory");
            issued = 1;
            if (++ia == NA) {
              ia = 0;
              aphase ^= 1u;
            }
          }
          if constexpr (PRE) {
            ok = mbar_wait(&planes_empty[stage], phase ^ 1u, &abort_flag);
            if (!ok) break;
            mbar_expect_tx(&planes_full[stage], CF::STAGE);
            asm volatile(
                "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
                "%5}], [%2];" ::"r"(sbase + stage * CF::STAGE),
                "l"((uint64_t)&tmW), "r"(smem_u32(&planes_full[stage])), "r"(kb * BK), "r"((tile % num_n) * BN), "r"(0)
                : "memory");
            issued = 1;
            if (++stage == NST) {
              stage = 0;
              phase ^= 1u;
            }
          }
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicExch(status, (int)WM_ERR_TIMEOUT);
        // give the copies in flight a fixed 50 us to land
        const unsigned long long t0 = globaltimer();
        while (issued && globaltimer() - t0 < 50000ull) {
        }
      }
    }
  } else if (warp == CF::MMA_WARP) {
    {
      // ---------------------------------------------------------- MMA issue
      // (the whole warp walks the loop, one elected lane issues)
      const bool leader = elect_one();
      auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
        return __all_sync(0xffffffffu, mbar_wait(bar, parity, &abort_flag));
      };
      constexpr uint32_t idesc = idesc_bf16(BM, BN);
      int stage = 0, buf = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true, ready = false;
      // products whose planes sum to 2 (smallest), 1 or 0 of the slab at stage st, into accumulator buf
      auto issue = [&](int st, int sum, uint32_t accumulate) {
        const uint32_t sb = sbase + st * CF::STAGE, ta = tmem + T_A + (uint32_t)(st * A_COLS);
#pragma unroll
        for (int pa = 0; pa < 3; ++pa) {
          if (pa > sum) break;
          const uint64_t bd = sw64_desc(sb + (sum - pa) * CF::PLANE);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            umma_ta(tmem + (uint32_t)(buf * BN), ta + (uint32_t)(pa * (BK / 2) + 8 * k), bd + (uint64_t)(2 * k), idesc,
                    accumulate);
            accumulate = 1u;
          }
        }
      };
      for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
        for (int kb = 0; kb < nk; kb += GROUP) {
          const bool two = kb + 1 < nk;   // slabs of this accumulator
          const int s0 = stage, s1 = stage + 1 == NST ? 0 : stage + 1, s2 = (stage + (two ? 2 : 1)) % NST;
          const uint32_t ph1 = s1 < s0 ? phase ^ 1u : phase, ph2 = s2 <= s0 ? phase ^ 1u : phase;
          ok = wait(&acce_bar[buf], acc_phase ^ 1u) && (ready || wait(&planes_full[s0], phase));
          if (!ok) break;
          tc_fence_after();
          if (leader) issue(s0, 2, 0u);
          if (two) {
            ok = wait(&planes_full[s1], ph1);
            if (!ok) break;
            tc_fence_after();
            if (leader) issue(s1, 2, 1u);
          }
          if (leader) {
            issue(s0, 1, 1u);
            if (two) issue(s1, 1, 1u);
          }
          // while the tensor core works: are the next accumulator's first planes there?
          ready = __all_sync(0xffffffffu, mbar_test(smem_u32(&planes_full[s2]), ph2));
          if (leader) {
            issue(s0, 0, 1u);
            umma_commit(&planes_empty[s0]);
            if (two) {
              issue(s1, 0, 1u);
              umma_commit(&planes_empty[s1]);
            }
            umma_commit(&accf_bar[buf]);
          }
          stage = s2;
          phase = ph2;
          if (++buf == NACC) {
            buf = 0;
            acc_phase ^= 1u;
          }
        }
      }
      if (!ok && leader) {
        abort_flag = 1;
        atomicExch(status, (int)WM_ERR_TIMEOUT);
        umma_commit(&drain_bar);   // every MMA issued above has finished
        volatile int never = 0;
        mbar_wait(&drain_bar, 0, &never);
      }
    }
  } else {
    // ------------------------------------------------------- sums, epilogue
    constexpr int HC = BN / 2;                    // columns of this warp
    const int quarter = warp & 3, half = (warp - CF::EPI) >> 2;
    const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * HC);
    int buf = 0;
    uint32_t phase = 0;
    bool ok = true;
    uint8_t* stg0 = smem + CF::OFF_OUT + (warp - CF::EPI) * 8192;   // 16-byte unit u of row r at u ^ (r & 7)
    uint32_t staged = 0;   // chunks staged so far (all tiles; a ragged tile may skip its second)
    float acc[HC];
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
#pragma unroll
      for (int j = 0; j < HC; ++j) acc[j] = 0.f;
      for (int kb = 0; kb < nk; kb += GROUP) {
        if (!mbar_wait(&accf_bar[buf], phase, &abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
        __syncwarp();
#pragma unroll
        for (int c = 0; c < HC; c += 16) {
          uint32_t t[16];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
              : "=r"(t[0]), "=r"(t[1]), "=r"(t[2]), "=r"(t[3]), "=r"(t[4]), "=r"(t[5]), "=r"(t[6]), "=r"(t[7]),
                "=r"(t[8]), "=r"(t[9]), "=r"(t[10]), "=r"(t[11]), "=r"(t[12]), "=r"(t[13]), "=r"(t[14]), "=r"(t[15])
              : "r"(tbase + (uint32_t)(buf * BN + c)));
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 16; j += 2)
            add_f2(acc[c + j], acc[c + j + 1], acc[c + j], acc[c + j + 1], __uint_as_float(t[j]),
                   __uint_as_float(t[j + 1]));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce_bar[buf]);
        if (++buf == NACC) {
          buf = 0;
          phase ^= 1u;
        }
      }
      if (!ok) break;
      const int row0 = (tile / num_n) * BM + quarter * 32, n0 = (tile % num_n) * BN + half * HC;
      if (row0 >= M) continue;
      if constexpr (!PRE) {
#pragma unroll
        for (int i = 0; i < CONV; ++i) rw = range_merge(rw, w_range[i]);
      }
      // sums below `first` may need recomputing
      const bool w_small = (rw >> 31) != 0u;
      float first = doubt_below(kLarge, rw, K);
      if (w_small && (!PRE || a_large[quarter * 32 + lane] != 0)) first = INFINITY;
      // 32 columns at a time, through the two staging tiles in turn
#pragma unroll
      for (int c = 0; c < HC; c += 32) {
        const int n = n0 + c;
        if (n >= N) continue;
        uint8_t* stg = stg0 + (staged & 1u) * 4096;
        ++staged;
        // the copy that last used this staging tile, the one before the newest, has read it
        if (tma_out && lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        __syncwarp();
        // (a product with zero is NaN where the sum is not finite)
        float z[4] = {}, least[2] = {INFINITY, INFINITY};
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          fma_f2(z[0], z[1], acc[c + j], acc[c + j + 1], 0ull, pack_f2(z[0], z[1]));
          fma_f2(z[2], z[3], acc[c + j + 2], acc[c + j + 3], 0ull, pack_f2(z[2], z[3]));
          least[0] = fminf(fminf(least[0], fabsf(acc[c + j])), fabsf(acc[c + j + 1]));
          least[1] = fminf(fminf(least[1], fabsf(acc[c + j + 2])), fabsf(acc[c + j + 3]));
        }
        if (n + 32 > N) {   // columns past N are zeros
          least[0] = least[1] = INFINITY;
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (n + j < N) least[0] = fminf(least[0], fabsf(acc[c + j]));
        }
        const bool low = row0 + lane < M && fminf(least[0], least[1]) < first;
        if (__any_sync(0xffffffffu, low || (z[0] + z[1]) + (z[2] + z[3]) != 0.f)) {
#pragma unroll
          for (int j = 0; j < 32; ++j) *stage_at(stg, lane, j) = acc[c + j];
          uint32_t look = __ballot_sync(0xffffffffu, low);
          float below = 0.f;
          if (PRE && !w_small && tile >= a_from[quarter]) {   // known from the splitting
            look = 0u;
            if (a_small[quarter * 32 + lane] != 0) below = first;
          }
          if (recompute(stg, A, W, row0, M, n, N, K, look, below, rw)) a_watch = 1;
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[c + j] = *stage_at(stg, lane, j);
        }
        const float bl = bias && n + lane < N ? __ldg(bias + n + lane) : 0.f;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          float y[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            y[e] = acc[c + j + e] + __shfl_sync(0xffffffffu, bl, j + e);
            if (epi == EPI_GELU) y[e] = gelu(y[e]);
          }
          *reinterpret_cast<float4*>(stage_at(stg, lane, j)) = make_float4(y[0], y[1], y[2], y[3]);
        }
        if (tma_out) {
          fence_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (epi == EPI_RESID_F32)
              asm volatile(
                  "cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                      (uint64_t)&tmC),
                  "r"(smem_u32(stg)), "r"(n), "r"(row0)
                  : "memory");
            else
              asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                               (uint64_t)&tmC),
                           "r"(smem_u32(stg)), "r"(n), "r"(row0)
                           : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        } else {
          // rows that a tensor copy cannot address (N % 4 != 0, unaligned output)
          __syncwarp();
          if (n + lane < N)
            for (int r = 0; r < 32 && row0 + r < M; ++r) {
              float* o = out + (size_t)(row0 + r) * N + n + lane;
              const float y = *stage_at(stg, r, lane);
              *o = epi == EPI_RESID_F32 ? *o + y : y;
            }
        }
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (!ok) {
      abort_flag = 1;
      atomicExch(status, (int)WM_ERR_TIMEOUT);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

constexpr int kSplitThreads = 512, kMaxSplitBlocks = 256;
int split_blocks(int N, int Kp) {
  return (int)std::min<long>(((long)N * (Kp / 2) + kSplitThreads - 1) / kSplitThreads, kMaxSplitBlocks);
}

// W [N, K] as three planes [3][N][Kp] (Kp: K rounded up to a slab, zeros past
// K), then each block's range of W.
__global__ void __launch_bounds__(kSplitThreads)
    split_planes_kernel(const float* __restrict__ W, __nv_bfloat16* __restrict__ P, int N, int K, int Kp) {
  __shared__ uint32_t part[kSplitThreads / 32];
  const long total = (long)N * (Kp / 2), plane = (long)N * Kp;
  Range r;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const int n = (int)(i / (Kp / 2)), k = 2 * (int)(i - (long)n * (Kp / 2));
    float x0 = k < K ? W[(size_t)n * K + k] : 0.f, x1 = k + 1 < K ? W[(size_t)n * K + k + 1] : 0.f;
    const float x[2] = {x0, x1};
    r.add(x);
    uint32_t* o = reinterpret_cast<uint32_t*>(P + (size_t)n * Kp + k);
    o[0] = split2(x0, x1);
    o[plane / 2] = split2(x0, x1);
    o[plane] = bf16x2(x0, x1);
  }
  const uint32_t range = range_of_warp(r.word());
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = range;
  __syncthreads();
  if (threadIdx.x < 32) {
    const uint32_t all = range_of_warp(part[threadIdx.x & (kSplitThreads / 32 - 1)]);
    if (threadIdx.x == 0) reinterpret_cast<uint32_t*>(P + 3 * plane)[blockIdx.x] = all;
  }
}

template <int BN, bool TMA_A, bool PRE, bool VEC_W>
wm_status launch_one(const CUtensorMap& tmA, const CUtensorMap& tmW, const float* A, const float* W,
                     const __nv_bfloat16* planes, const float* bias, float* out, int M, int N, int K, int epi,
                     cudaStream_t s) {
  const long tiles = (long)((M + BM - 1) / BM) * ((N + BN - 1) / BN);
  if (tiles > (1L << 30)) return fail(WM_ERR_INVALID_ARG, "too many FP32 GEMM tiles");
  const int grid = (int)std::min<long>(tiles, num_sms());
  CUtensorMap tmC{};
  const int tma_out = make_tmap_out(&tmC, out, (uint64_t)M, (uint64_t)N, true);   // false: unaligned rows
  const int Kp = f32_plane_k(K);
  const uint32_t* ranges = PRE ? reinterpret_cast<const uint32_t*>(planes + (size_t)3 * N * Kp) : nullptr;
  gemm_f32_tc_kernel<BN, TMA_A, PRE, VEC_W><<<grid, Cfg<BN, PRE>::THREADS, Cfg<BN, PRE>::SMEM, s>>>(
      tmA, tmW, tmC, A, W, bias, out, M, N, K, epi, tma_out, ranges, PRE ? split_blocks(N, Kp) : 0,
      device_status_word());
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

template <int BN>
wm_status launch_bn(const float* A, const float* W, const __nv_bfloat16* planes, const float* bias, float* out, int M,
                    int N, int K, int epi, cudaStream_t s) {
  CUtensorMap tmA{}, tmW{};
  const bool tma_a = K % 4 == 0 && make_tmap_f32(&tmA, A, (uint64_t)M, (uint64_t)K, BM);
  if (planes && !make_tmap_planes(&tmW, planes, (uint64_t)N, (uint64_t)f32_plane_k(K), BN))
    return fail(WM_ERR_CUDA, "cuTensorMapEncodeTiled failed for the split weights");
  if (planes)
    return tma_a ? launch_one<BN, true, true, false>(tmA, tmW, A, W, planes, bias, out, M, N, K, epi, s)
                 : launch_one<BN, false, true, false>(tmA, tmW, A, W, planes, bias, out, M, N, K, epi, s);
  const bool vec_w = K % 4 == 0 && (uintptr_t)W % 16 == 0;
  if (tma_a && vec_w) return launch_one<BN, true, false, true>(tmA, tmW, A, W, planes, bias, out, M, N, K, epi, s);
  return launch_one<BN, false, false, false>(tmA, tmW, A, W, planes, bias, out, M, N, K, epi, s);
}

template <int BN, bool TMA_A, bool PRE, bool VEC_W>
wm_status set_attr() {
  WM_CUDA(cudaFuncSetAttribute(gemm_f32_tc_kernel<BN, TMA_A, PRE, VEC_W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               Cfg<BN, PRE>::SMEM));
  return WM_OK;
}
template <int BN>
wm_status set_attrs() {
  wm_status st = set_attr<BN, true, true, false>();
  if (st == WM_OK) st = set_attr<BN, false, true, false>();
  if (st == WM_OK) st = set_attr<BN, true, false, true>();
  if (st == WM_OK) st = set_attr<BN, false, false, false>();
  return st;
}

}  // namespace f32tc

wm_status prepare_gemm_f32() {
  wm_status st = f32tc::set_attrs<64>();
  if (st == WM_OK) st = f32tc::set_attrs<128>();
  return st;
}

int f32_plane_k(int K) { return (K + f32tc::BK - 1) / f32tc::BK * f32tc::BK; }
size_t f32_planes_size(int N, int K) {
  return (size_t)3 * N * f32_plane_k(K) + f32tc::kMaxSplitBlocks * sizeof(uint32_t) / sizeof(__nv_bfloat16);
}

wm_status launch_split_planes(const float* W, __nv_bfloat16* planes, int N, int K, cudaStream_t s) {
  const int Kp = f32_plane_k(K);
  f32tc::split_planes_kernel<<<f32tc::split_blocks(N, Kp), f32tc::kSplitThreads, 0, s>>>(W, planes, N, K, Kp);
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

wm_status launch_gemm_f32(const float* A, const float* W, const __nv_bfloat16* planes, const float* bias, float* out,
                          int M, int N, int K, int epi, cudaStream_t s) {
  if (M <= 0 || N <= 0) return WM_OK;
  // Tile width: the fewest clocks over the waves of a persistent grid. A slab
  // of 64 or 128 columns takes about 840 or 1130 clocks (shared memory at 128
  // bytes a clock).
  const long rows = (M + f32tc::BM - 1) / f32tc::BM;
  const long w64 = (rows * ((N + 63) / 64) + num_sms() - 1) / num_sms() * 840;
  const long w128 = (rows * ((N + 127) / 128) + num_sms() - 1) / num_sms() * 1130;
  return w128 <= w64 ? f32tc::launch_bn<128>(A, W, planes, bias, out, M, N, K, epi, s)
                     : f32tc::launch_bn<64>(A, W, planes, bias, out, M, N, K, epi, s);
}

// Planes for one call come from a stream-ordered pool of this library (kept up
// to 64 MB, so that a loop of calls allocates once).
static cudaMemPool_t planes_pool() {
  static std::mutex mu;
  static cudaMemPool_t pools[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lk(mu);
  if (!pools[dev]) {
    cudaMemPoolProps pr{};
    pr.allocType = cudaMemAllocationTypePinned;
    pr.location.type = cudaMemLocationTypeDevice;
    pr.location.id = dev;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = 64ull << 20;
    if (cudaMemPoolCreate(&pool, &pr) == cudaSuccess) {
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
      pools[dev] = pool;
    } else {
      cudaGetLastError();
    }
  }
  return pools[dev];
}

wm_status launch_linear_f32(const float* A, const float* W, const float* bias, float* out, int M, int N, int K, int epi,
                            cudaStream_t s) {
  if (M <= 0 || N <= 0) return WM_OK;
  // Splitting W beforehand costs a launch and a pass over W (about 4 us) and
  // takes a slab from ~1700 to ~1050 clocks: worth it from about 16 slabs per
  // CTA (M = 4608, N = 128, K = 512: 21 us both ways; M = 1024, K = 128: 11
  // against 13 us; M = 2000, N = K = 768: 37 against 29 us). Inside a stream
  // capture, or without memory, W is split in the GEMM itself.
  const long rows = (M + f32tc::BM - 1) / f32tc::BM, nk = (K + f32tc::BK - 1) / f32tc::BK;
  const long waves = (rows * ((N + 127) / 128) + num_sms() - 1) / num_sms();
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  void* planes = nullptr;
  if (waves * nk > 16 && cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
    cudaMemPool_t pool = planes_pool();
    const size_t bytes = f32_planes_size(N, K) * sizeof(__nv_bfloat16);
    if (!pool || cudaMallocFromPoolAsync(&planes, bytes, pool, s) != cudaSuccess) {
      cudaGetLastError();
      planes = nullptr;
    }
  }
  if (!planes) return launch_gemm_f32(A, W, nullptr, bias, out, M, N, K, epi, s);
  wm_status st = launch_split_planes(W, (__nv_bfloat16*)planes, N, K, s);
  if (st == WM_OK) st = launch_gemm_f32(A, W, (const __nv_bfloat16*)planes, bias, out, M, N, K, epi, s);
  const cudaError_t e = cudaFreeAsync(planes, s);
  if (st == WM_OK && e != cudaSuccess) st = cuda_fail(e, "cudaFreeAsync");
  return st;
}

}  // namespace wm
