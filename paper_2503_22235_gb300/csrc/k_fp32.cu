// Plain FP32 path: LayerNorm and 3D neighborhood attention on CUDA cores
// (strict FP32 FMA; the linear layers are in k_gemm_f32.cu), so that a block
// matches the float64 oracle to ~1e-6 relative L2.
#include <cuda_fp8.h>

#include <algorithm>

#include "wm_internal.cuh"

namespace wm {

// ------------------------------------------------------------ LayerNorm ----
// One warp per row. Mean and biased variance over C in FP32 (two passes over
// the row held in registers when C is a multiple of 128 and <= 1024).

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename OutT>
__device__ __forceinline__ void store_val(OutT* p, float v);
template <>
__device__ __forceinline__ void store_val<float>(float* p, float v) { *p = v; }
template <>
__device__ __forceinline__ void store_val<__nv_bfloat16>(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

template <typename OutT, int V4>  // V4 float4 per lane, C = 128 * V4
__global__ void ln_rows_reg(const float* __restrict__ x, const float* __restrict__ g, const float* __restrict__ b,
                            OutT* __restrict__ out, int M, float eps) {
  const int C = 128 * V4;
  const int lane = threadIdx.x & 31;
  const long row = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= M) return;
  const float4* xr = reinterpret_cast<const float4*>(x + row * C);
  float4 v[V4];
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < V4; ++i) {
    v[i] = xr[lane + 32 * i];
    s += (v[i].x + v[i].y) + (v[i].z + v[i].w);
  }
  const float mean = warp_sum(s) / C;
  float q = 0.f;
#pragma unroll
  for (int i = 0; i < V4; ++i) {
    float a = v[i].x - mean, bb = v[i].y - mean, c = v[i].z - mean, d = v[i].w - mean;
    q += (a * a + bb * bb) + (c * c + d * d);
  }
  const float rstd = rsqrtf(warp_sum(q) / C + eps);
  const float4* g4 = reinterpret_cast<const float4*>(g);
  const float4* b4 = reinterpret_cast<const float4*>(b);
  OutT* orow = out + row * C;
#pragma unroll
  for (int i = 0; i < V4; ++i) {
    const int c = 4 * (lane + 32 * i);
    float4 gg = g4[lane + 32 * i], bb = b4[lane + 32 * i];
    float r0 = (v[i].x - mean) * rstd * gg.x + bb.x;
    float r1 = (v[i].y - mean) * rstd * gg.y + bb.y;
    float r2 = (v[i].z - mean) * rstd * gg.z + bb.z;
    float r3 = (v[i].w - mean) * rstd * gg.w + bb.w;
    if constexpr (sizeof(OutT) == 4) {
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(orow) + c) = make_float4(r0, r1, r2, r3);
    } else {
      __nv_bfloat162 p0 = __floats2bfloat162_rn(r0, r1), p1 = __floats2bfloat162_rn(r2, r3);
      uint2 u;
      u.x = *reinterpret_cast<uint32_t*>(&p0);
      u.y = *reinterpret_cast<uint32_t*>(&p1);
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(orow) + c) = u;
    }
  }
}

template <typename OutT>
__global__ void ln_rows_generic(const float* __restrict__ x, const float* __restrict__ g,
                                const float* __restrict__ b, OutT* __restrict__ out, int M, int C, float eps) {
  const int lane = threadIdx.x & 31;
  const long row = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= M) return;
  const float* xr = x + row * C;
  float s = 0.f;
  for (int c = lane; c < C; c += 32) s += xr[c];
  const float mean = warp_sum(s) / C;
  float q = 0.f;
  for (int c = lane; c < C; c += 32) {
    float d = xr[c] - mean;
    q += d * d;
  }
  const float rstd = rsqrtf(warp_sum(q) / C + eps);
  for (int c = lane; c < C; c += 32) store_val(out + row * C + c, (xr[c] - mean) * rstd * g[c] + b[c]);
}

// Row statistics: one warp per row, (mean, M2) in FP32 from the row held in
// registers, plus the bf16 copy of the row.
template <int V4>
__global__ void row_stats_kernel(const float* __restrict__ x, __nv_bfloat16* __restrict__ xb, float* __restrict__ st,
                                 int M) {
  const int C = 128 * V4;
  const int lane = threadIdx.x & 31;
  const long row = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  pdl_wait();
  pdl_trigger();
  if (row >= M) return;
  const float4* xr = reinterpret_cast<const float4*>(x + row * C);
  float4 v[V4];
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < V4; ++i) {
    v[i] = xr[lane + 32 * i];
    s += (v[i].x + v[i].y) + (v[i].z + v[i].w);
  }
  const float mean = warp_sum(s) / C;
  float q = 0.f;
#pragma unroll
  for (int i = 0; i < V4; ++i) {
    float a = v[i].x - mean, bb = v[i].y - mean, c = v[i].z - mean, d = v[i].w - mean;
    q += (a * a + bb * bb) + (c * c + d * d);
    __nv_bfloat162 p0 = __floats2bfloat162_rn(v[i].x, v[i].y), p1 = __floats2bfloat162_rn(v[i].z, v[i].w);
    uint2 u;
    u.x = *reinterpret_cast<uint32_t*>(&p0);
    u.y = *reinterpret_cast<uint32_t*>(&p1);
    *reinterpret_cast<uint2*>(xb + row * C + 4 * (lane + 32 * i)) = u;
  }
  const float m2 = warp_sum(q);
  if (lane == 0) {
    st[2 * row] = mean;
    st[2 * row + 1] = m2;
  }
}

wm_status launch_row_stats(const float* x, __nv_bfloat16* xb, float* stats, int M, int C, cudaStream_t s,
                           bool pdl) {
  if (M <= 0) return WM_OK;
  const int warps = 8;
  dim3 grid((M + warps - 1) / warps), block(32 * warps);
  switch (C) {
    case 128: WM_CUDA(launch_pdl(row_stats_kernel<1>, grid, block, 0, s, pdl, x, xb, stats, M)); break;
    case 256: WM_CUDA(launch_pdl(row_stats_kernel<2>, grid, block, 0, s, pdl, x, xb, stats, M)); break;
    case 384: WM_CUDA(launch_pdl(row_stats_kernel<3>, grid, block, 0, s, pdl, x, xb, stats, M)); break;
    case 512: WM_CUDA(launch_pdl(row_stats_kernel<4>, grid, block, 0, s, pdl, x, xb, stats, M)); break;
    case 768: WM_CUDA(launch_pdl(row_stats_kernel<6>, grid, block, 0, s, pdl, x, xb, stats, M)); break;
    case 1024: WM_CUDA(launch_pdl(row_stats_kernel<8>, grid, block, 0, s, pdl, x, xb, stats, M)); break;
    default: return fail(WM_ERR_INVALID_ARG, "row statistics need C in {128, 256, 384, 512, 768, 1024}");
  }
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

// LayerNorm rows to e4m3: one warp per row, FP32 statistics as above, output
// e4m3(LN(x) * inv_scale) with round-to-nearest-even and saturation.
template <int V4>
__global__ void ln_rows_e4m3(const float* __restrict__ x, const float* __restrict__ g, const float* __restrict__ b,
                             uint8_t* __restrict__ out, int M, float eps, float inv_scale) {
  const int C = 128 * V4;
  const int lane = threadIdx.x & 31;
  const long row = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  pdl_wait();
  pdl_trigger();
  if (row >= M) return;
  const float4* xr = reinterpret_cast<const float4*>(x + row * C);
  float4 v[V4];
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < V4; ++i) {
    v[i] = xr[lane + 32 * i];
    s += (v[i].x + v[i].y) + (v[i].z + v[i].w);
  }
  const float mean = warp_sum(s) / C;
  float q = 0.f;
#pragma unroll
  for (int i = 0; i < V4; ++i) {
    float a = v[i].x - mean, bb = v[i].y - mean, c = v[i].z - mean, d = v[i].w - mean;
    q += (a * a + bb * bb) + (c * c + d * d);
  }
  const float rstd = rsqrtf(warp_sum(q) / C + eps);
  const float4* g4 = reinterpret_cast<const float4*>(g);
  const float4* b4 = reinterpret_cast<const float4*>(b);
#pragma unroll
  for (int i = 0; i < V4; ++i) {
    const int c = 4 * (lane + 32 * i);
    float4 gg = g4[lane + 32 * i], bb = b4[lane + 32 * i];
    const float r0 = ((v[i].x - mean) * rstd * gg.x + bb.x) * inv_scale;
    const float r1 = ((v[i].y - mean) * rstd * gg.y + bb.y) * inv_scale;
    const float r2 = ((v[i].z - mean) * rstd * gg.z + bb.z) * inv_scale;
    const float r3 = ((v[i].w - mean) * rstd * gg.w + bb.w) * inv_scale;
    const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(r0, r1), __NV_SATFINITE, __NV_E4M3);
    const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(r2, r3), __NV_SATFINITE, __NV_E4M3);
    *reinterpret_cast<uint32_t*>(out + row * C + c) = lo | (hi << 16);
  }
}

wm_status launch_layernorm_e4m3(const float* x, const float* g, const float* b, uint8_t* out, int M, int C,
                                float eps, float inv_scale, cudaStream_t s, bool pdl) {
  if (M <= 0) return WM_OK;
  const int warps = 8;
  dim3 grid((M + warps - 1) / warps), block(32 * warps);
  switch (C) {
    case 128: WM_CUDA(launch_pdl(ln_rows_e4m3<1>, grid, block, 0, s, pdl, x, g, b, out, M, eps, inv_scale)); break;
    case 256: WM_CUDA(launch_pdl(ln_rows_e4m3<2>, grid, block, 0, s, pdl, x, g, b, out, M, eps, inv_scale)); break;
    case 384: WM_CUDA(launch_pdl(ln_rows_e4m3<3>, grid, block, 0, s, pdl, x, g, b, out, M, eps, inv_scale)); break;
    case 512: WM_CUDA(launch_pdl(ln_rows_e4m3<4>, grid, block, 0, s, pdl, x, g, b, out, M, eps, inv_scale)); break;
    case 768: WM_CUDA(launch_pdl(ln_rows_e4m3<6>, grid, block, 0, s, pdl, x, g, b, out, M, eps, inv_scale)); break;
    case 1024: WM_CUDA(launch_pdl(ln_rows_e4m3<8>, grid, block, 0, s, pdl, x, g, b, out, M, eps, inv_scale)); break;
    default: return fail(WM_ERR_INVALID_ARG, "e4m3 LayerNorm needs C in {128, 256, 384, 512, 768, 1024}");
  }
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

wm_status launch_layernorm(const float* x, const float* g, const float* b, void* out, bool out_bf16, int M, int C,
                           float eps, cudaStream_t s) {
  if (M <= 0) return WM_OK;
  const int warps = 8;
  dim3 grid((M + warps - 1) / warps), block(32 * warps);
  const bool aligned = ((uintptr_t)x % 16 == 0) && ((uintptr_t)g % 16 == 0) && ((uintptr_t)b % 16 == 0) &&
                       ((uintptr_t)out % 16 == 0);
  const int v4 = (C % 128 == 0 && aligned) ? C / 128 : 0;
#define WM_LN_CASE(N)                                                                                          \
  case N:                                                                                                     \
    if (out_bf16)                                                                                             \
      ln_rows_reg<__nv_bfloat16, N><<<grid, block, 0, s>>>(x, g, b, (__nv_bfloat16*)out, M, eps);             \
    else                                                                                                      \
      ln_rows_reg<float, N><<<grid, block, 0, s>>>(x, g, b, (float*)out, M, eps);                             \
    break;
  switch (v4) {
    WM_LN_CASE(1)
    WM_LN_CASE(2)
    WM_LN_CASE(3)
    WM_LN_CASE(4)
    WM_LN_CASE(6)
    WM_LN_CASE(8)
    default:
      if (out_bf16)
        ln_rows_generic<__nv_bfloat16><<<grid, block, 0, s>>>(x, g, b, (__nv_bfloat16*)out, M, C, eps);
      else
        ln_rows_generic<float><<<grid, block, 0, s>>>(x, g, b, (float*)out, M, C, eps);
  }
#undef WM_LN_CASE
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

// ------------------------------------------------------- rotary embedding ----
// One thread per (token, rotation pair) of q and of k in an fp32 qkv [M, 3C].
__global__ void rope_f32_kernel(float* __restrict__ qkv, long M, const RopeArgs* __restrict__ R) {
  const int P = R->C / 2;
  const long total = M * 2 * P;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const long m = i / (2 * P);
    const int r = (int)(i % (2 * P));   // pair index over q (r < P) then k
    const int col = 2 * (r % P) + (r >= P ? R->C : 0);
    const int p = (col % R->C) % R->dh / 2;
    const int tok = (int)(m % ((long)R->D * R->H * R->W));
    const int pos[3] = {tok / (R->H * R->W), (tok / R->W) % R->H, tok % R->W};
    const int ax = p < R->n[0] ? 0 : (p < R->n[0] + R->n[1] ? 1 : 2);
    const int pm = p - (ax > 0 ? R->n[0] : 0) - (ax > 1 ? R->n[1] : 0);
    const float2 cs = R->tab[ax][pos[ax] * R->n[ax] + pm];
    float* v = qkv + m * 3L * R->C + col;
    const float a0 = v[0], a1 = v[1];
    v[0] = a0 * cs.x - a1 * cs.y;
    v[1] = a0 * cs.y + a1 * cs.x;
  }
}

wm_status launch_rope_f32(float* qkv, long M, const RopeArgs* rope_dev, const RopeArgs& rope_host, cudaStream_t s) {
  if (M <= 0) return WM_OK;
  const long total = M * rope_host.C;
  const int blocks = (int)std::min<long>((total + 255) / 256, (long)num_sms() * 16);
  rope_f32_kernel<<<blocks, 256, 0, s>>>(qkv, M, rope_dev);
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

// ------------------------------------------------- neighborhood attention ----
// One warp per (token, head). Scores for the kd*kh*kw neighbours go to shared
// memory, the softmax max and sum are warp-shuffle reductions in FP32, and the
// output channels are split across lanes.

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__global__ void na_f32_kernel(const float* __restrict__ qkv, float* __restrict__ out, int B, int D, int H, int W,
                              int C, int heads, int kd, int kh, int kw, int periodic) {
  extern __shared__ float smem[];
  const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int dh = C / heads, K = kd * kh * kw;
  float* qs = smem + warp * (K + dh);
  float* sc = qs + dh;
  const long N = (long)D * H * W;
  const long gw = (long)blockIdx.x * warps + warp;
  if (gw >= (long)B * N * heads) return;  // whole warp leaves together
  const int head = (int)(gw % heads);
  const long bt = gw / heads;
  const long t = bt % N, b = bt / N;
  const int l = (int)(t / ((long)H * W)), i = (int)((t / W) % H), j = (int)(t % W);
  const int sl = clampi(l - kd / 2, 0, D - kd), si = clampi(i - kh / 2, 0, H - kh);
  const int sj = periodic ? j - kw / 2 : clampi(j - kw / 2, 0, W - kw);
  const long C3 = 3L * C;
  const float scale = rsqrtf((float)dh);
  const float* qrow = qkv + (b * N + t) * C3 + head * dh;
  for (int c = lane; c < dh; c += 32) qs[c] = qrow[c];
  __syncwarp();

  auto key_token = [&](int kk) -> long {
    const int a = kk / (kh * kw), bb = (kk / kw) % kh, cc = kk % kw;
    int jj = sj + cc;
    if (periodic) jj = ((jj % W) + W) % W;
    return ((long)(sl + a) * H + (si + bb)) * W + jj;
  };

  float mx = -INFINITY;
  for (int kk = lane; kk < K; kk += 32) {
    const float* krow = qkv + (b * N + key_token(kk)) * C3 + C + head * dh;
    float d = 0.f;
    for (int c = 0; c < dh; ++c) d = fmaf(qs[c], krow[c], d);
    d *= scale;
    sc[kk] = d;
    mx = fmaxf(mx, d);
  }
  mx = warp_max(mx);
  float sum = 0.f;
  for (int kk = lane; kk < K; kk += 32) {
    const float e = expf(sc[kk] - mx);
    sc[kk] = e;
    sum += e;
  }
  sum = warp_sum(sum);
  __syncwarp();
  const float inv = 1.f / sum;
  float* orow = out + (b * N + t) * C + head * dh;
  for (int c = lane; c < dh; c += 32) {
    float acc = 0.f;
    for (int kk = 0; kk < K; ++kk) acc = fmaf(sc[kk], qkv[(b * N + key_token(kk)) * C3 + 2 * C + head * dh + c], acc);
    orow[c] = acc * inv;
  }
}

// Tiled FP32 attention: CTA = batch element, head, query level and an 8 x 8
// block of queries; four threads per query, each owning a quarter of the
// head's channels (a score is the quarters' dot products added with two
// shuffles).
// For every key level the CTA stages the tile's K and V halo slabs (rows of
// dh + 4 floats: 128-bit loads of consecutive keys hit distinct banks) in
// shared memory; each query walks its own window row by row with an online
// softmax (running max and sum in FP32, O rescaled once per window row).
// Strict FP32 FMA and expf throughout.
template <int DH>
__global__ void __launch_bounds__(256, 2) na_f32_tile_kernel(const float* __restrict__ qkv, float* __restrict__ out,
                                                          int B, int D, int H, int W, int C, int heads, int kd, int kh,
                                                          int kw, int periodic, int tiles_h, int tiles_w,
                                                          int* __restrict__ dstatus) {
  constexpr int TH = 8, TW = 8, TPQ = 4, HD = DH / TPQ, KS = DH + 4;   // KS: key row stride in shared memory (floats)
  constexpr int KW_MAX = 9;
  extern __shared__ __align__(16) float sm[];
  const int HR = min(TH + kh - 1, H);
  const int WC = periodic ? TW + kw - 1 : min(TW + kw - 1, W);
  float* Ks = sm;
  float* Vs = sm + HR * WC * KS;
  int t = blockIdx.x;
  const int tw = t % tiles_w;
  t /= tiles_w;
  const int th = t % tiles_h;
  t /= tiles_h;
  const int d = t % D;
  t /= D;
  const int head = t % heads, b = t / heads;
  const int h0 = th * TH, w0 = tw * TW, rh = kh / 2, rw = kw / 2;
  const int hs0 = clampi(h0 - rh, 0, H - HR);
  const int ws0 = periodic ? w0 - rw : clampi(w0 - rw, 0, W - WC);
  const int ld0 = clampi(d - kd / 2, 0, D - kd);
  const int pair = threadIdx.x / TPQ, half = threadIdx.x % TPQ;   // query of the tile, channel quarter
  const int hq = h0 + pair / TW, wq = w0 + pair % TW;
  bool valid = hq < H && wq < W;
  const int hc = min(hq, H - 1), wc = min(wq, W - 1);
  int ra = clampi(hc - rh, 0, H - kh) - hs0;                                   // window rows in the slab
  int cb = (periodic ? wc - rw : clampi(wc - rw, 0, W - kw)) - ws0;            // window columns
  // debug builds: the window lies inside the staged slab; on a failure it is
  // clamped into the slab and the query is not written
  if (!WM_DCHECK(ra >= 0 && ra + kh <= HR && cb >= 0 && cb + kw <= WC && ld0 >= 0 && ld0 + kd <= D, dstatus)) {
    ra = clampi(ra, 0, HR - kh);
    cb = clampi(cb, 0, WC - kw);
    valid = false;
  }
  const long N = (long)D * H * W, C3 = 3L * C;
  const float scale = rsqrtf((float)DH);
  float q[HD], o[HD];
  {
    const float4* qs = reinterpret_cast<const float4*>(qkv + ((long)b * N + ((long)d * H + hc) * W + wc) * C3 +
                                                       head * DH + half * HD);
#pragma unroll
    for (int i = 0; i < HD / 4; ++i) {
      const float4 v = qs[i];
      q[4 * i] = v.x; q[4 * i + 1] = v.y; q[4 * i + 2] = v.z; q[4 * i + 3] = v.w;
    }
  }
#pragma unroll
  for (int i = 0; i < HD; ++i) o[i] = 0.f;
  float m = -INFINITY, l = 0.f;
  const int slab_keys = HR * WC;
  for (int li = 0; li < kd; ++li) {
    __syncthreads();   // the previous level's slabs are no longer read
    const long lev = (long)b * D + ld0 + li;
    for (int idx = threadIdx.x; idx < 2 * slab_keys * (DH / 4); idx += blockDim.x) {
      const int kv = idx / (slab_keys * (DH / 4));
      const int rem = idx - kv * slab_keys * (DH / 4);
      const int key = rem / (DH / 4), c4 = rem - key * (DH / 4);
      const int r = key / WC, c = key - r * WC;
      int lon = ws0 + c;
      if (periodic) lon = ((lon % W) + W) % W;
      const float4 v = *reinterpret_cast<const float4*>(qkv + ((lev * H + hs0 + r) * W + lon) * C3 + (1 + kv) * C +
                                                        head * DH + 4 * c4);
      *reinterpret_cast<float4*>((kv ? Vs : Ks) + key * KS + 4 * c4) = v;
    }
    __syncthreads();
    for (int a = 0; a < kh; ++a) {
      const int row = (ra + a) * WC + cb;
      float sc[KW_MAX];
      float rmax = -INFINITY;
#pragma unroll
      for (int j = 0; j < KW_MAX; ++j) {
        if (j < kw) {
          const float4* kr = reinterpret_cast<const float4*>(Ks + (row + j) * KS + half * HD);
          float acc = 0.f;
#pragma unroll
          for (int i = 0; i < HD / 4; ++i) {
            const float4 k4 = kr[i];
            acc = fmaf(q[4 * i], k4.x, acc);
            acc = fmaf(q[4 * i + 1], k4.y, acc);
            acc = fmaf(q[4 * i + 2], k4.z, acc);
            acc = fmaf(q[4 * i + 3], k4.w, acc);
          }
          acc += __shfl_xor_sync(0xffffffffu, acc, 1);   // the other channel quarters
          acc += __shfl_xor_sync(0xffffffffu, acc, 2);
          sc[j] = acc * scale;
          rmax = fmaxf(rmax, sc[j]);
        }
      }
      if (rmax > m) {
        const float alpha = expf(m - rmax);   // 0 while m = -inf: O and l are still zero
        l *= alpha;
#pragma unroll
        for (int i = 0; i < HD; ++i) o[i] *= alpha;
        m = rmax;
      }
#pragma unroll
      for (int j = 0; j < KW_MAX; ++j) {
        if (j < kw) {
          const float p = expf(sc[j] - m);
          l += p;
          const float4* vr = reinterpret_cast<const float4*>(Vs + (row + j) * KS + half * HD);
#pragma unroll
          for (int i = 0; i < HD / 4; ++i) {
            const float4 v4 = vr[i];
            o[4 * i] = fmaf(p, v4.x, o[4 * i]);
            o[4 * i + 1] = fmaf(p, v4.y, o[4 * i + 1]);
            o[4 * i + 2] = fmaf(p, v4.z, o[4 * i + 2]);
            o[4 * i + 3] = fmaf(p, v4.w, o[4 * i + 3]);
          }
        }
      }
    }
  }
  if (!valid) return;
  const float inv = 1.f / l;
  float4* orow = reinterpret_cast<float4*>(out + ((long)b * N + ((long)d * H + hq) * W + wq) * C + head * DH +
                                           half * HD);
#pragma unroll
  for (int i = 0; i < HD / 4; ++i)
    orow[i] = make_float4(o[4 * i] * inv, o[4 * i + 1] * inv, o[4 * i + 2] * inv, o[4 * i + 3] * inv);
}

// FP32 attention with 2 x 2 blocks of queries (windows of 3, 5 or 7
// longitudes). A tile of BH x BW blocks of one (batch element, head, level)
// stages the K and V halo slab of one key level at a time in shared memory
// (cp.async). TPB threads share a block: each holds the block's four queries
// and outputs in every TPB-th float4 of the head's channels, so a K or V value
// read from shared memory serves four queries (196 of the 256 query-key pairs
// of the block's 8 x 8 keys lie in a 7 x 7 window). A key's four scores are
// summed over the block's threads by a reduce-scatter (three shuffles at
// TPB = 4) that leaves each thread the whole score of one query, its own; its
// probability goes back by three shuffles. A thread keeps the four queries in
// an order of its own, query (own ^ k) at place k, so neither step selects
// registers. The block's key rows of a level are divided between the CTA's
// two halves (the same blocks), whose softmax states are merged at the end.
// What bounds it (dh = 48, per key of a block and warp): 30 clocks of shared
// memory (six 128-bit loads of 512 bytes a warp, six shuffles) and 96 of the
// FMA lanes of one scheduler (48 f32x2, which take two clocks each); 60 % and
// 53 % busy as measured, three warps a scheduler at 168 registers not hiding
// all of the loads' and shuffles' latency. 9 x 90 x 180 x 768, 16 heads,
// window 5 x 7 x 7: 17.2 ms with one query per four threads (every K and V
// value read for one query only), 4.4 ms here.
// FP32 FMA and expf throughout. A masked key has probability zero; where its
// V is not finite that makes the output NaN, and a V above FLT_MAX / e^8 can
// overflow before the division by the sum. An output that is not finite although
// the query's own scores are is recomputed over its own window alone, with
// probabilities already divided, by the lanes of its block. 9 x 90 x 180 x 768: 4.4 ms with every token NaN or none,
// 8.1 with one in 4001 and 16.5 with one in 50, whose neighbours are recomputed
// (by one thread for each float4, whatever the scores: 380 ms with one in 4001,
// seconds with more).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// Four floats from shared memory as two f32x2 operands.
__device__ __forceinline__ void lds_f2(uint32_t addr, uint64_t& lo, uint64_t& hi) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float2 unpack2(uint64_t a) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(a));
  return f;
}

// Floats between keys in shared memory: two keys apart lands half the banks
// away, so that neighbouring blocks' 128-bit loads do not collide.
template <int DH>
struct NaBlk {
  static constexpr int TPB = DH == 64 ? 8 : 4;       // threads per block of queries
  static constexpr int NI = DH / 4 / TPB;            // float4 per thread
  static constexpr int KS = DH == 64 ? 64 : DH + 8;
  static constexpr int MAXT = DH == 48 ? 384 : 512;  // threads per CTA: 168 or 128 registers
};

// The output of one query over its own window alone, by the TPB lanes `group` of
// its block: each takes the block kernel's share of the channels of every key
// (q, key0: the query's and the batch element's K of this head; V lies C floats
// on), and a key's score is summed over the lanes. The softmax reference M and
// 1 / sum are the block kernel's. Writes the float4 of the set `bits`.
template <int DH, int KW>
__device__ __noinline__ void na_f32_query(const float* q, const float* key0, float* o, uint32_t bits, uint32_t group,
                                          int part, int H, int W, int C, int ld0, int kd, int r0, int kh, int c0,
                                          float scale, float M, float inv) {
  constexpr int TPB = NaBlk<DH>::TPB, NI = NaBlk<DH>::NI;
  float4 qv[NI], acc[NI];
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    qv[i] = *reinterpret_cast<const float4*>(q + 4 * (i * TPB + part));
    acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll 1
  for (int l = 0; l < kd; ++l)
#pragma unroll 1
    for (int r = 0; r < kh; ++r) {
      const float* row = key0 + ((long)(ld0 + l) * H + r0 + r) * W * 3 * C + 4 * part;
      const float* key[KW];
      float s[KW];
#pragma unroll
      for (int j = 0; j < KW; ++j) {
        int lon = c0 + j;
        while (lon < 0) lon += W;
        while (lon >= W) lon -= W;
        key[j] = row + (long)lon * 3 * C;
        s[j] = 0.f;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const float4 k = *reinterpret_cast<const float4*>(key[j] + 4 * i * TPB);
          s[j] = fmaf(qv[i].x, k.x, fmaf(qv[i].y, k.y, fmaf(qv[i].z, k.z, fmaf(qv[i].w, k.w, s[j]))));
        }
      }
#pragma unroll
      for (int j = 0; j < KW; ++j) {
#pragma unroll
        for (int d = 1; d < TPB; d *= 2) s[j] += __shfl_xor_sync(group, s[j], d);
        const float p = expf(s[j] * scale - M) * inv;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const float4 v = *reinterpret_cast<const float4*>(key[j] + C + 4 * i * TPB);
          acc[i].x = fmaf(p, v.x, acc[i].x);
          acc[i].y = fmaf(p, v.y, acc[i].y);
          acc[i].z = fmaf(p, v.z, acc[i].z);
          acc[i].w = fmaf(p, v.w, acc[i].w);
        }
      }
    }
#pragma unroll
  for (int i = 0; i < NI; ++i)
    if ((bits >> i) & 1u) *reinterpret_cast<float4*>(o + 4 * (i * TPB + part)) = acc[i];
}

template <int DH, int KW>
__global__ void __launch_bounds__(NaBlk<DH>::MAXT, 1)
    na_f32_block_kernel(const float* __restrict__ qkv, float* __restrict__ out, int D, int H, int W, int C, int heads,
                        int kd, int kh, int periodic, int BH, int BW, int tiles_h, int tiles_w,
                        int* __restrict__ dstatus) {
  using NB = NaBlk<DH>;
  constexpr int TPB = NB::TPB, NI = NB::NI, KS = NB::KS, NC = KW + 1, NU = DH / 4;
  extern __shared__ __align__(16) float sm[];
  const int HR = min(2 * BH + kh - 1, H);
  const int WC = periodic ? 2 * BW + KW - 1 : min(2 * BW + KW - 1, W);
  const int vs = HR * WC * KS;   // K, then V, then one more key: a block may read a column past its window
  if (threadIdx.x < KS) sm[2 * vs + threadIdx.x] = 0.f;
  int t = blockIdx.x;
  const int tw = t % tiles_w;
  t /= tiles_w;
  const int th = t % tiles_h;
  t /= tiles_h;
  const int d = t % D;
  t /= D;
  const int head = t % heads, b = t / heads;
  const int h0 = th * 2 * BH, w0 = tw * 2 * BW, rh = kh / 2, rw = KW / 2;
  const int hs0 = clampi(h0 - rh, 0, H - HR);
  const int ws0 = periodic ? w0 - rw : clampi(w0 - rw, 0, W - WC);
  const int ld0 = clampi(d - kd / 2, 0, D - kd);
  const int nthr = blockDim.x >> 1;                       // threads of a half
  const int half = threadIdx.x >= nthr ? 1 : 0, ht = threadIdx.x - half * nthr;
  const int part = ht % TPB, blk = ht / TPB;
  const int bh = h0 + 2 * (blk / BW), bw = w0 + 2 * (blk % BW);
  const int own = 2 * (part & 1) + ((part >> 1) & 1);     // this thread's query: row own / 2, column own % 2
  auto row_start = [&](int h) { return clampi(min(h, H - 1) - rh, 0, H - kh) - hs0; };
  auto col_start = [&](int w) { return (periodic ? min(w, W - 1) - rw : clampi(min(w, W - 1) - rw, 0, W - KW)) - ws0; };
  int ra = row_start(bh), cb = col_start(bw);             // the block's first key row and column
  const int dr = row_start(bh + (own >> 1)) - ra, dc = col_start(bw + (own & 1)) - cb;
  bool ok = true;
  // debug builds: the block's windows lie in the slab
  if (!WM_DCHECK(ra >= 0 && ra + dr + kh <= HR && cb >= 0 && cb + dc + KW <= WC && dr >= 0 && dr <= 1 && dc >= 0 &&
                     dc <= 1 && ld0 >= 0 && ld0 + kd <= D,
                 dstatus)) {
    ra = cb = 0;
    ok = false;
  }
  const uint32_t cmask = ((1u << KW) - 1u) << dc;
  const long N = (long)D * H * W, C3 = 3L * C;
  const float scale = rsqrtf((float)DH);
  uint64_t q[4][2 * NI], o[4][2 * NI];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int qi = own ^ k, hq = min(bh + (qi >> 1), H - 1), wq = min(bw + (qi & 1), W - 1);
    const ulonglong2* src = reinterpret_cast<const ulonglong2*>(qkv + ((long)b * N + ((long)d * H + hq) * W + wq) * C3 +
                                                                head * DH);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const ulonglong2 v = src[i * TPB + part];
      q[k][2 * i] = v.x;
      q[k][2 * i + 1] = v.y;
      o[k][2 * i] = o[k][2 * i + 1] = 0ull;
    }
  }
  float m = -3.402823466e38f, l = 0.f;
  const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(sm);
  const int rows0 = (kh + 2) / 2;                         // rows of the first half; the second has kh + 1 - rows0
  for (int li = 0; li < kd; ++li) {
    __syncthreads();   // the previous level's slabs are no longer read
    const long lev = (long)b * D + ld0 + li;
    // a thread brings one 16-byte unit of a column of K or V, row after row
    for (int idx = threadIdx.x; idx < 2 * WC * NU; idx += blockDim.x) {
      const int c2 = idx / NU, u = idx - c2 * NU, kv = c2 >= WC ? 1 : 0, c = c2 - kv * WC;
      int lon = ws0 + c;
      while (lon < 0) lon += W;
      while (lon >= W) lon -= W;
      const float* src = qkv + ((lev * H + hs0) * W + lon) * C3 + (1 + kv) * C + head * DH + 4 * u;
      uint32_t dst = smem0 + (uint32_t)(kv * vs + c * KS + 4 * u) * 4u;
#pragma unroll 4
      for (int r = 0; r < HR; ++r) {
        cp_async16(dst, src);
        src += (long)W * C3;
        dst += (uint32_t)(WC * KS) * 4u;
      }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int a_end = half ? kh + 1 : rows0;
#pragma unroll 1
    for (int a = half ? rows0 : 0; a < a_end; ++a) {
      const uint32_t krow = smem0 + (uint32_t)((min(ra + a, HR - 1) * WC + cb) * KS + 4 * part) * 4u;
      const uint32_t vrow = krow + (uint32_t)vs * 4u;
      const uint32_t cm = a >= dr && a < dr + kh ? cmask : 0u;   // columns of this thread's query
      float sc[NC], rmax = -INFINITY;
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        uint64_t s2[4];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          uint64_t k0, k1;
          lds_f2(krow + (uint32_t)(j * KS + 4 * i * TPB) * 4u, k0, k1);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            s2[k] = i == 0 ? mul2(q[k][0], k0) : fma2(q[k][2 * i], k0, s2[k]);
            s2[k] = fma2(q[k][2 * i + 1], k1, s2[k]);
          }
        }
        float f[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 u = unpack2(s2[k]);
          f[k] = u.x + u.y;
        }
        f[0] += __shfl_xor_sync(0xffffffffu, f[2], 1);
        f[1] += __shfl_xor_sync(0xffffffffu, f[3], 1);
        f[0] += __shfl_xor_sync(0xffffffffu, f[1], 2);
        if constexpr (TPB == 8) f[0] += __shfl_xor_sync(0xffffffffu, f[0], 4);
        sc[j] = (cm >> j) & 1u ? f[0] * scale : -INFINITY;
        rmax = fmaxf(rmax, sc[j]);
      }
      // The references of a block's queries move together, and only when some score
      // of the block passes its query's by more than 8 (probabilities stay below
      // e^8), so most rows rescale nothing. The vote is the block's alone: what
      // shares its warp follows from the tile, which the batch size may change.
      const uint32_t votes = __ballot_sync(0xffffffffu, rmax > m + 8.f);
      if (votes != 0u) {
        const bool moves = ((votes >> (threadIdx.x & 31 & ~(TPB - 1))) & ((1u << TPB) - 1u)) != 0u;
        const float mn = moves ? fmaxf(m, rmax) : m;
        const float a0 = moves ? expf(m - mn) : 1.f;   // 0 while m is the initial value: o and l are still zero
        l *= a0;
        m = mn;
        const float a1 = __shfl_xor_sync(0xffffffffu, a0, 2), a2 = __shfl_xor_sync(0xffffffffu, a0, 1),
                    a3 = __shfl_xor_sync(0xffffffffu, a1, 1);
        const uint64_t al[4] = {pack_f2(a0, a0), pack_f2(a1, a1), pack_f2(a2, a2), pack_f2(a3, a3)};
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int i = 0; i < 2 * NI; ++i) o[k][i] = mul2(o[k][i], al[k]);
      }
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const float p0 = expf(sc[j] - m);
        l += p0;
        const float p1 = __shfl_xor_sync(0xffffffffu, p0, 2), p2 = __shfl_xor_sync(0xffffffffu, p0, 1),
                    p3 = __shfl_xor_sync(0xffffffffu, p1, 1);
        const uint64_t pp[4] = {pack_f2(p0, p0), pack_f2(p1, p1), pack_f2(p2, p2), pack_f2(p3, p3)};
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          uint64_t v0, v1;
          lds_f2(vrow + (uint32_t)(j * KS + 4 * i * TPB) * 4u, v0, v1);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            o[k][2 * i] = fma2(pp[k], v0, o[k][2 * i]);
            o[k][2 * i + 1] = fma2(pp[k], v1, o[k][2 * i + 1]);
          }
        }
      }
    }
  }
  // the halves' softmax states, merged by the first half
  __syncthreads();
  float* xs = sm;
  if (half) {
    xs[ht] = m;
    xs[nthr + ht] = l;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int i = 0; i < 2 * NI; ++i) {
        const float2 u = unpack2(o[k][i]);
        xs[(2 + 4 * NI * k + 2 * i) * nthr + ht] = u.x;
        xs[(3 + 4 * NI * k + 2 * i) * nthr + ht] = u.y;
      }
  }
  __syncthreads();
  if (half) return;
  const float m1 = xs[ht], M = fmaxf(m, m1);
  const float e0 = expf(m - M), e1 = expf(m1 - M);
  const float inv = 1.f / (l * e0 + xs[nthr + ht] * e1);
  float f0[4], f1[4];   // weights of the two halves, divided by the sum
  f0[0] = e0 * inv;
  f1[0] = e1 * inv;
  f0[1] = __shfl_xor_sync(0xffffffffu, f0[0], 2);
  f1[1] = __shfl_xor_sync(0xffffffffu, f1[0], 2);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    f0[2 + k] = __shfl_xor_sync(0xffffffffu, f0[k], 1);
    f1[2 + k] = __shfl_xor_sync(0xffffffffu, f1[k], 1);
  }
  uint32_t bad = 0u;   // float4 i of query qi at bit qi NI + i
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int qi = own ^ k, hq = bh + (qi >> 1), wq = bw + (qi & 1);
    if (!ok || hq >= H || wq >= W) continue;
    float* orow = out + ((long)b * N + ((long)d * H + hq) * W + wq) * C + head * DH;
    const bool sound = f0[k] == f0[k] && f1[k] == f1[k];   // else a score of the query's own is NaN: so is all of it
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      float y[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 u = unpack2(o[k][2 * i + (e >> 1)]);
        y[e] = ((e & 1) ? u.y : u.x) * f0[k] + xs[(2 + 4 * NI * k + 4 * i + e) * nthr + ht] * f1[k];
        if (sound && !(fabsf(y[e]) <= 3.402823466e38f)) bad |= 1u << (qi * NI + i);
      }
      *reinterpret_cast<float4*>(orow + 4 * (i * TPB + part)) = make_float4(y[0], y[1], y[2], y[3]);
    }
  }
  if (__any_sync(0xffffffffu, bad != 0u)) {
    const int lane0 = threadIdx.x & 31 & ~(TPB - 1);   // of the block's lanes
    const uint32_t group = ((1u << TPB) - 1u) << lane0;
    uint32_t need = 0u;   // queries of the block with such a float4 in any lane
#pragma unroll
    for (int qi = 0; qi < 4; ++qi)
      need |= (__ballot_sync(0xffffffffu, ((bad >> (qi * NI)) & ((1u << NI) - 1u)) != 0u) & group) != 0u ? 1u << qi : 0u;
#pragma unroll 1
    for (; need != 0u; need &= need - 1u) {
      const int qi = __ffs(need) - 1, hq = bh + (qi >> 1), wq = bw + (qi & 1);
      const int owner = lane0 + ((qi >> 1) | ((qi & 1) << 1));
      const float Mq = __shfl_sync(group, M, owner), iq = __shfl_sync(group, inv, owner);
      const long tok = (long)b * N + ((long)d * H + hq) * W + wq;
      na_f32_query<DH, KW>(qkv + tok * C3 + head * DH, qkv + (long)b * N * C3 + C + head * DH, out + tok * C + head * DH,
                           (bad >> (qi * NI)) & ((1u << NI) - 1u), group, part, H, W, C, ld0, kd,
                           row_start(bh + (qi >> 1)) + hs0, kh, col_start(bw + (qi & 1)) + ws0, scale, Mq, iq);
    }
  }
}

// Tile of the block kernel (blocks along latitude and longitude), its shared
// memory and its CTAs; false if the shape is not its own.
static bool na_f32_block_plan(int B, int D, int H, int W, int heads, int dh, int kh, int kw, bool periodic, int* BH,
                              int* BW, size_t* smem, long* ctas) {
  if ((kw != 3 && kw != 5 && kw != 7) || (dh != 16 && dh != 32 && dh != 48 && dh != 64)) return false;
  const int wide = dh == 64 ? 4 : dh == 48 ? 6 : 8;
  const int cand[3][2] = {{8, wide}, {4, wide}, {4, dh == 64 ? 2 : 4}};
  const int tpb = dh == 64 ? 8 : 4, ks = dh == 64 ? 64 : dh + 8, maxt = dh == 48 ? 384 : 512;
  double best = 0.0;
  for (const auto& c : cand) {
    const int HR = std::min(2 * c[0] + kh - 1, H), WC = periodic ? 2 * c[1] + kw - 1 : std::min(2 * c[1] + kw - 1, W);
    const int threads = 2 * c[0] * c[1] * tpb;
    const size_t bytes = std::max(((size_t)2 * HR * WC + 1) * ks * 4, (size_t)threads / 2 * (dh / tpb * 4 + 2) * 4);
    if (bytes > 227 * 1024) continue;
    const long n = (long)((H + 2 * c[0] - 1) / (2 * c[0])) * ((W + 2 * c[1] - 1) / (2 * c[1])) * D * heads * B;
    const long per_sm = std::min<long>(maxt / threads, (227 * 1024) / (bytes + 1024));
    const long waves = (n + num_sms() * per_sm - 1) / (num_sms() * per_sm);
    // clocks of a CTA and level: its keys' FMAs, and its slab's way into shared
    // memory (64 bytes a clock), which another CTA of the SM can hide
    const double fma = (double)c[0] * c[1] * (kh + 1) * (kw + 1) * dh / 12.0, load = 2.0 * HR * WC * dh * 4 / 64;
    // fewer than 12 warps on an SM leave issue slots empty
    const double thin = std::max(1.0, 384.0 / (double)(per_sm * threads));
    const double cost = (double)waves * (per_sm > 1 ? std::max(per_sm * fma * thin, per_sm * load) : fma * thin + load);
    if (best == 0.0 || cost < best) {
      best = cost;
      *BH = c[0];
      *BW = c[1];
      *smem = bytes;
      *ctas = n;
    }
  }
  return best != 0.0;
}

template <int DH>
static wm_status launch_na_f32_block(const float* qkv, float* out, int D, int H, int W, int C, int heads, int kd,
                                     int kh, int kw, bool periodic, int BH, int BW, size_t smem, long ctas,
                                     cudaStream_t s) {
  const int tiles_h = (H + 2 * BH - 1) / (2 * BH), tiles_w = (W + 2 * BW - 1) / (2 * BW);
  const dim3 grid((unsigned)ctas), block(2 * BH * BW * NaBlk<DH>::TPB);
  auto kern = kw == 3 ? na_f32_block_kernel<DH, 3> : kw == 5 ? na_f32_block_kernel<DH, 5> : na_f32_block_kernel<DH, 7>;
  kern<<<grid, block, smem, s>>>(qkv, out, D, H, W, C, heads, kd, kh, periodic ? 1 : 0, BH, BW, tiles_h, tiles_w,
                                 device_status_word());
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

// Shared memory of the tiled FP32 attention (K and V slabs), or 0 if the
// shape does not fit it.
static size_t na_f32_tile_smem(int H, int W, int dh, int kh, int kw, bool periodic) {
  if (kw > 9 || (dh != 16 && dh != 32 && dh != 48 && dh != 64)) return 0;   // dh / 4 channels per thread in float4
  const int HR = std::min(8 + kh - 1, H), WC = periodic ? 8 + kw - 1 : std::min(8 + kw - 1, W);
  const size_t bytes = (size_t)2 * HR * WC * (dh + 4) * sizeof(float);
  return bytes <= 227 * 1024 ? bytes : 0;
}

template <int DH>
static wm_status prepare_na_f32_block() {
  WM_CUDA(cudaFuncSetAttribute(na_f32_block_kernel<DH, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  WM_CUDA(cudaFuncSetAttribute(na_f32_block_kernel<DH, 5>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  WM_CUDA(cudaFuncSetAttribute(na_f32_block_kernel<DH, 7>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  return WM_OK;
}

wm_status prepare_na_f32() {
  wm_status st = prepare_na_f32_block<16>();
  if (st == WM_OK) st = prepare_na_f32_block<32>();
  if (st == WM_OK) st = prepare_na_f32_block<48>();
  if (st == WM_OK) st = prepare_na_f32_block<64>();
  if (st != WM_OK) return st;
  WM_CUDA(cudaFuncSetAttribute(na_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  WM_CUDA(cudaFuncSetAttribute(na_f32_tile_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  WM_CUDA(cudaFuncSetAttribute(na_f32_tile_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  WM_CUDA(cudaFuncSetAttribute(na_f32_tile_kernel<48>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  WM_CUDA(cudaFuncSetAttribute(na_f32_tile_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  return WM_OK;
}

wm_status launch_na_f32(const float* qkv, float* out, int B, int D, int H, int W, int C, int heads, int kd, int kh,
                        int kw, bool periodic, cudaStream_t s) {
  const long total = (long)B * D * H * W * heads;
  if (total <= 0) return WM_OK;
  const int dh0 = C / heads;
  const bool aligned = C % 4 == 0 && ((uintptr_t)qkv & 15) == 0 && ((uintptr_t)out & 15) == 0;
  int BH = 0, BW = 0;
  size_t bsm = 0;
  long bctas = 0;
  if (aligned && na_f32_block_plan(B, D, H, W, heads, dh0, kh, kw, periodic, &BH, &BW, &bsm, &bctas)) {
    if (bctas > (1L << 31) - 1) return fail(WM_ERR_INVALID_ARG, "too many attention tiles");
    switch (dh0) {
      case 16: return launch_na_f32_block<16>(qkv, out, D, H, W, C, heads, kd, kh, kw, periodic, BH, BW, bsm, bctas, s);
      case 32: return launch_na_f32_block<32>(qkv, out, D, H, W, C, heads, kd, kh, kw, periodic, BH, BW, bsm, bctas, s);
      case 48: return launch_na_f32_block<48>(qkv, out, D, H, W, C, heads, kd, kh, kw, periodic, BH, BW, bsm, bctas, s);
      default: return launch_na_f32_block<64>(qkv, out, D, H, W, C, heads, kd, kh, kw, periodic, BH, BW, bsm, bctas, s);
    }
  }
  const size_t tsm = na_f32_tile_smem(H, W, dh0, kh, kw, periodic);
  if (tsm && aligned) {
    const int tiles_h = (H + 7) / 8, tiles_w = (W + 7) / 8;
    const long ctas = (long)tiles_h * tiles_w * D * heads * B;
    if (ctas > (1L << 31) - 1) return fail(WM_ERR_INVALID_ARG, "too many attention tiles");
    const dim3 grid((unsigned)ctas), block(256);
    const int per = periodic ? 1 : 0;
    switch (dh0) {
      case 16: na_f32_tile_kernel<16><<<grid, block, tsm, s>>>(qkv, out, B, D, H, W, C, heads, kd, kh, kw, per, tiles_h, tiles_w, device_status_word()); break;
      case 32: na_f32_tile_kernel<32><<<grid, block, tsm, s>>>(qkv, out, B, D, H, W, C, heads, kd, kh, kw, per, tiles_h, tiles_w, device_status_word()); break;
      case 48: na_f32_tile_kernel<48><<<grid, block, tsm, s>>>(qkv, out, B, D, H, W, C, heads, kd, kh, kw, per, tiles_h, tiles_w, device_status_word()); break;
      default: na_f32_tile_kernel<64><<<grid, block, tsm, s>>>(qkv, out, B, D, H, W, C, heads, kd, kh, kw, per, tiles_h, tiles_w, device_status_word()); break;
    }
    WM_CUDA(cudaGetLastError());
    return WM_OK;
  }
  // other shapes: one warp per (query, head)
  const int warps = 8;
  const int K = kd * kh * kw, dh = C / heads;
  const size_t smem = (size_t)warps * (K + dh) * sizeof(float);
  if (smem > 227 * 1024) return fail(WM_ERR_INVALID_ARG, "neighborhood window too large for the FP32 attention kernel");
  dim3 grid((unsigned)((total + warps - 1) / warps)), block(32 * warps);
  na_f32_kernel<<<grid, block, smem, s>>>(qkv, out, B, D, H, W, C, heads, kd, kh, kw, periodic ? 1 : 0);
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

}  // namespace wm
