// Bandwidth-proposal network: 32 -> 256 -> 256 -> 256 -> 6 with exact GELU,
// FP16 weights (the FP32 master copy is rounded on load) and FP32
// accumulation.  Forward, manual backward of the masked squared error, and
// AdamW, all on the device.
//
// The paper chooses bandwidths by cross-validation over candidates (Section
// 3.3); this network proposes the CV-optimal log bandwidths from a summary of
// the binned data, so that one smoothing pass (plus a CV check) can stand in
// for a grid.
//
// Parameter vector: for each layer, W (fan_in x fan_out, row-major) then b.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "fpca_internal.cuh"

namespace {

constexpr int NLAYER = 4;
__host__ __device__ constexpr int layer_in(int l) { return l == 0 ? 32 : 256; }
__host__ __device__ constexpr int layer_out(int l) { return l == 3 ? 6 : 256; }
__host__ __device__ constexpr long long layer_off(int l) {
  return l == 0 ? 0 : layer_off(l - 1) + (long long)layer_in(l - 1) * layer_out(l - 1) + layer_out(l - 1);
}
constexpr long long kParamCount = layer_off(NLAYER);

__device__ __forceinline__ float as_fp16(float w) { return __half2float(__float2half_rn(w)); }

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.3989422804014327f;
}

// ---------------------------------------------------------------------------
// The step in three launches:
//   k_mlp_weights  FP16 copies of the hidden layers' weights, and transposes of those the
//                  backward pass multiplies by; the batch's mask count, in parts;
//   k_mlp_rows     a CTA takes R rows of the batch through the whole network and back:
//                  the rows are independent between the loss and the weights, so nothing
//                  but the weights (384 KB in FP16, from L2) is read between layers;
//   k_mlp_grads    one CTA per 32 x 32 tile of every layer's weight gradient, with the
//                  bias gradients and the AdamW update of the tile's own parameters.
// What bounds it is latency: the network is 0.14 M parameters and a batch of 256 some
// 0.2 GFLOP.  As 17 launches (a GEMM of 32 x 32 tiles per product, column sums, loss, AdamW)
// the step took 229 us at a batch of 256, 19 us a GEMM; it takes 45 us.
// ---------------------------------------------------------------------------
constexpr int HID = 256;          // width of the hidden layers
constexpr int MR_WARPS = 8;       // warps of k_mlp_rows; each takes every 8th k of a product
// FP16 copies, in elements: layer 0, 1, 2 as stored (fan_in x fan_out), then the transposes
// of layers 1 and 2
__host__ __device__ constexpr int w16_off(int copy) {
  return copy == 0 ? 0 : 32 * HID + (copy - 1) * HID * HID;
}
constexpr int W16_COUNT = 32 * HID + 4 * HID * HID;

constexpr int MW_TILES = 8 + 64 + 64;
constexpr int MC_MAX = 128;        // parts of the mask count
constexpr int MC_BYTES = 256 * 32; // bytes of a part, unless that makes more than MC_MAX

// A 32 x 32 tile per block: blocks 0..7 layer 0, then 64 each for layers 1 and 2.  The blocks
// beyond MW_TILES count a part of the mask (nm bytes) each, into mcount.
__global__ void __launch_bounds__(256)
    k_mlp_weights(const float* __restrict__ th, __half* __restrict__ w16,
                  const uint8_t* __restrict__ mask, long long nm, int* __restrict__ mcount) {
  __shared__ __half t[32][33];
  if (blockIdx.x >= MW_TILES) {
    const int part = blockIdx.x - MW_TILES, parts = gridDim.x - MW_TILES;
    __shared__ int mc[8];
    int c = 0;
#pragma unroll 4
    for (long long e = part * 256 + threadIdx.x; e < nm; e += parts * 256) c += mask[e] ? 1 : 0;
    for (int q = 16; q > 0; q >>= 1) c += __shfl_xor_sync(0xffffffffu, c, q);
    if ((threadIdx.x & 31) == 0) mc[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int q = 1; q < 8; ++q) c += mc[q];
      mcount[part] = c;
    }
    return;
  }
  const int b = blockIdx.x, l = b < 8 ? 0 : b < 72 ? 1 : 2, tile = b - (l == 0 ? 0 : l == 1 ? 8 : 72);
  const int r0 = (tile / 8) * 32, c0 = (tile % 8) * 32;
  const float* W = th + layer_off(l);
  __half* out = w16 + w16_off(l);
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (int r = y; r < 32; r += 8) {
    const __half h = __float2half_rn(W[(r0 + r) * HID + c0 + x]);
    out[(r0 + r) * HID + c0 + x] = h;
    t[r][x] = h;
  }
  if (l == 0) return;
  __syncthreads();
  __half* tr = w16 + w16_off(l + 2);
  for (int r = y; r < 32; r += 8) tr[(c0 + r) * HID + r0 + x] = t[x][r];
}

// part[warp][r][n] = sum over the warp's k of x[k][r] W[k][n], W: K x 256 in FP16, x: K x R
// in shared memory.  Each lane takes 8 neighbouring n (one 128-bit load of W per k).
template <int R>
__device__ __forceinline__ void mlp_product(const __half* __restrict__ W, int K,
                                            const float* __restrict__ x, float* __restrict__ part) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  float acc[R][8];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[r][c] = 0.f;
#pragma unroll 4
  for (int k = wp; k < K; k += MR_WARPS) {
    const uint4 q = *reinterpret_cast<const uint4*>(W + (size_t)k * HID + 8 * lane);
    const uint32_t qs[4] = {q.x, q.y, q.z, q.w};
    float w[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&qs[c]));
      w[2 * c] = f.x;
      w[2 * c + 1] = f.y;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float xv = x[k * R + r];
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[r][c] = fmaf(xv, w[c], acc[r][c]);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float4* o = reinterpret_cast<float4*>(part + ((size_t)wp * R + r) * HID + 8 * lane);
    o[0] = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
    o[1] = make_float4(acc[r][4], acc[r][5], acc[r][6], acc[r][7]);
  }
}

struct MlpBuf {
  float* X;        // B x 32 copy of the input (16-byte rows)
  float* H[3];     // activations, B x 256
  float* D[3];     // gradients w.r.t. the hidden pre-activations, B x 256
  float* D3;       // gradient w.r.t. the output, B x 8 (two zero columns)
  float* losspart; // one per CTA
  int* mcount;     // observed targets, in `parts` parts
  int parts;
  __half* w16;
};

inline size_t mlp_rows_smem(int R) {
  return sizeof(float) * ((size_t)HID * R + 3 * (size_t)R * HID + (size_t)MR_WARPS * R * HID +
                          2 * (size_t)R * 8);
}

// R rows of the batch per CTA; `train`: gradients too, else the outputs go to `out`.
template <int R>
__global__ void __launch_bounds__(256)
    k_mlp_rows(int Bn, const float* __restrict__ th, const float* __restrict__ feat,
               const float* __restrict__ target, const uint8_t* __restrict__ mask, MlpBuf w,
               float* __restrict__ out, int train) {
  extern __shared__ __align__(16) float msm[];
  float* x = msm;                                  // [256][R], the current operand
  float* z = x + HID * R;                          // [3][R][256] pre-activations
  float* part = z + 3 * R * HID;                   // [warps][R][256]
  float* os = part + (size_t)MR_WARPS * R * HID;   // [R][8] outputs
  float* ds = os + R * 8;                          // [R][8] their gradients
  __shared__ int rc[8];
  __shared__ float rl[8];
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5, row0 = blockIdx.x * R;
  for (int e = t; e < 32 * R; e += 256) {
    const int r = e >> 5, k = e & 31, row = row0 + r;
    const float v = row < Bn ? feat[(size_t)row * 32 + k] : 0.f;
    x[k * R + r] = v;
    if (train && row < Bn) w.X[(size_t)row * 32 + k] = v;
  }
  __syncthreads();
  for (int l = 0; l < 3; ++l) {
    mlp_product<R>(w.w16 + w16_off(l), layer_in(l), x,
                   part);
    __syncthreads();
    const float b = th[layer_off(l) + (long long)layer_in(l) * HID + t];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float s = 0.f;
#pragma unroll
      for (int q = 0; q < MR_WARPS; ++q) s += part[((size_t)q * R + r) * HID + t];
      s += b;
      const float h = gelu(s);
      z[(l * R + r) * HID + t] = s;
      x[t * R + r] = h;
      if (train && row0 + r < Bn) w.H[l][(size_t)(row0 + r) * HID + t] = h;
    }
    __syncthreads();
  }
  const float* W3 = th + layer_off(3);
  for (int e = wp; e < R * 6; e += MR_WARPS) {  // one warp per output
    const int r = e / 6, o = e - r * 6;
    float s = 0.f;
    for (int k = lane; k < HID; k += 32) s = fmaf(x[k * R + r], as_fp16(W3[k * 6 + o]), s);
    for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
    if (lane == 0) os[r * 8 + o] = s + W3[HID * 6 + o];
  }
  __syncthreads();
  if (!train) {
    if (t < R * 6 && row0 + t / 6 < Bn) out[(size_t)row0 * 6 + t] = os[(t / 6) * 8 + t % 6];
    return;
  }
  // masked loss: its denominator is the whole batch's mask count (each CTA going through the
  // whole mask made the step quadratic in the batch: 2^20 rows 441 ms, 57 with the parts)
  int cnt = t < w.parts ? w.mcount[t] : 0;
  for (int q = 16; q > 0; q >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, q);
  if (lane == 0) rc[wp] = cnt;
  __syncthreads();
  cnt = 0;
  for (int q = 0; q < 8; ++q) cnt += rc[q];
  const float denom = fmaxf((float)cnt, 1.f);
  float ls = 0.f;
  if (t < R * 8) {
    const int r = t >> 3, o = t & 7, row = row0 + r;
    float g = 0.f;
    if (o < 6 && row < Bn && mask[(size_t)row * 6 + o]) {
      const float d = os[r * 8 + o] - target[(size_t)row * 6 + o];
      ls = d * d;
      g = 2.f * d / denom;
    }
    ds[t] = g;
    if (row < Bn) w.D3[(size_t)row0 * 8 + t] = g;
  }
  for (int q = 16; q > 0; q >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, q);
  if (lane == 0) rl[wp] = ls;
  __syncthreads();
  if (t == 0) {
    float s = 0.f;
    for (int q = 0; q < 8; ++q) s += rl[q];
    w.losspart[blockIdx.x] = s / denom;
  }
  {
    float wv[6];
#pragma unroll
    for (int o = 0; o < 6; ++o) wv[o] = as_fp16(W3[t * 6 + o]);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float s = 0.f;
#pragma unroll
      for (int o = 0; o < 6; ++o) s = fmaf(ds[r * 8 + o], wv[o], s);
      s *= gelu_grad(z[(2 * R + r) * HID + t]);
      x[t * R + r] = s;
      if (row0 + r < Bn) w.D[2][(size_t)(row0 + r) * HID + t] = s;
    }
  }
  __syncthreads();
  for (int l = 2; l >= 1; --l) {
    mlp_product<R>(w.w16 + w16_off(l + 2), HID, x, part);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float s = 0.f;
#pragma unroll
      for (int q = 0; q < MR_WARPS; ++q) s += part[((size_t)q * R + r) * HID + t];
      s *= gelu_grad(z[((l - 1) * R + r) * HID + t]);
      x[t * R + r] = s;
      if (row0 + r < Bn) w.D[l - 1][(size_t)(row0 + r) * HID + t] = s;
    }
    __syncthreads();
  }
}

// AdamW with bias correction; decoupled weight decay on every parameter.
struct AdamArgs {
  float *th, *m, *v;  // m == NULL: gradients only
  float lr, wd, bc1, bc2;
};
__device__ __forceinline__ void adamw(const AdamArgs& a, long long i, float gi) {
  const float mi = 0.9f * a.m[i] + 0.1f * gi;
  const float vi = 0.999f * a.v[i] + 0.001f * gi * gi;
  a.m[i] = mi;
  a.v[i] = vi;
  const float mh = mi / a.bc1, vh = vi / a.bc2;
  a.th[i] -= a.lr * (mh / (sqrtf(vh) + 1e-8f) + a.wd * a.th[i]);
}

// Gradient tile (32 inputs x 32 outputs) of one layer: sum over the batch of
// h[b][i] d[b][o].  Each warp sums every 8th row of the batch into the whole tile (4 x 8
// entries per lane), and the warps' tiles are added in shared memory.  Tiles: 8 of layer 0
// (blocks 0..7), 64 each of layers 1 and 2, 8 of layer 3.  A layer's first row of tiles
// also sums d over the batch, the bias gradient.  Block 0 adds up the loss.
constexpr int MG_KC = 64;   // batch rows staged per chunk
constexpr int MG_TILES = 8 + 64 + 64 + 8;
__global__ void __launch_bounds__(256)
    k_mlp_grads(int Bn, int nparts, MlpBuf w, AdamArgs ad, float* __restrict__ grad,
                float* __restrict__ loss) {
  __shared__ __align__(16) float part[8][32][32];
  float(*hs)[32] = part[0];   // [MG_KC][32] each, until the warps' tiles take their place
  float(*dsm)[32] = part[2];
  __shared__ float bpart[8][32];
  const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, wp = t >> 5;
  const int l = b < 8 ? 0 : b < 72 ? 1 : b < 136 ? 2 : 3;
  const int tile = b - (l == 0 ? 0 : l == 1 ? 8 : l == 2 ? 72 : 136);
  const int i0 = l == 0 ? 0 : l == 3 ? tile * 32 : (tile / 8) * 32;
  const int o0 = l == 3 ? 0 : (tile % 8) * 32;
  const float* H = l == 0 ? w.X : l == 1 ? w.H[0] : l == 2 ? w.H[1] : w.H[2];
  const float* D = l == 0 ? w.D[0] : l == 1 ? w.D[1] : l == 2 ? w.D[2] : w.D3;
  const int ldh = l == 0 ? 32 : HID, ldd = l == 3 ? 8 : HID;
  const bool bias = i0 == 0;
  const int li = 4 * (lane >> 2), lo = 8 * (lane & 3);
  float acc[4][8], bs[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    bs[c] = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r][c] = 0.f;
  }
  for (int k0 = 0; k0 < Bn; k0 += MG_KC) {
    __syncthreads();
    for (int e = t; e < MG_KC * 8; e += 256) {
      const int k = e >> 3, c = 4 * (e & 7), row = k0 + k;
      float4 h = make_float4(0.f, 0.f, 0.f, 0.f), d = h;
      if (row < Bn) {
        h = *reinterpret_cast<const float4*>(H + (size_t)row * ldh + i0 + c);
        if (l < 3 || c < 8) d = *reinterpret_cast<const float4*>(D + (size_t)row * ldd + o0 + c);
      }
      *reinterpret_cast<float4*>(&hs[k][c]) = h;
      *reinterpret_cast<float4*>(&dsm[k][c]) = d;
    }
    __syncthreads();
#pragma unroll
    for (int k = wp; k < MG_KC; k += 8) {
      const float4 h = *reinterpret_cast<const float4*>(&hs[k][li]);
      const float4 d0 = *reinterpret_cast<const float4*>(&dsm[k][lo]);
      const float4 d1 = *reinterpret_cast<const float4*>(&dsm[k][lo + 4]);
      const float hv[4] = {h.x, h.y, h.z, h.w};
      const float dv[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[r][c] = fmaf(hv[r], dv[c], acc[r][c]);
      if (bias)
#pragma unroll
        for (int c = 0; c < 8; ++c) bs[c] += dv[c];
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float4* o = reinterpret_cast<float4*>(&part[wp][li + r][lo]);
    o[0] = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
    o[1] = make_float4(acc[r][4], acc[r][5], acc[r][6], acc[r][7]);
  }
  if (bias && lane < 4)
#pragma unroll
    for (int c = 0; c < 8; ++c) bpart[wp][lo + c] = bs[c];
  __syncthreads();
  const int fo = layer_out(l);
  for (int e = t; e < 1024; e += 256) {
    const int i = e >> 5, o = e & 31;
    if (o0 + o >= fo) continue;
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) s += part[q][i][o];
    const long long at = layer_off(l) + (long long)(i0 + i) * fo + o0 + o;
    if (grad) grad[at] = s;
    if (ad.m) adamw(ad, at, s);
  }
  if (bias && t < 32 && o0 + t < fo) {
    float s = 0.f;
    for (int q = 0; q < 8; ++q) s += bpart[q][t];
    const long long at = layer_off(l) + (long long)layer_in(l) * fo + o0 + t;
    if (grad) grad[at] = s;
    if (ad.m) adamw(ad, at, s);
  }
  if (b == 0 && loss) {  // the CTAs' shares of the loss, in a fixed order
    float s = 0.f;
    for (int q = t; q < nparts; q += 256) s += w.losspart[q];
    for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
    __syncthreads();
    if (lane == 0) bpart[0][wp] = s;
    __syncthreads();
    if (t == 0) {
      s = 0.f;
      for (int q = 0; q < 8; ++q) s += bpart[0][q];
      *loss = s;
    }
  }
}

// Rows of the batch per CTA: as few as fill the SMs once (a product's latency is the
// weights' way from L2, whatever R), up to 8 (registers and shared memory).
int mlp_rows_per_cta(const fpca_ctx* ctx, int Bn) {
  return Bn <= 2 * ctx->num_sms ? 2 : Bn <= 4 * ctx->num_sms ? 4 : 8;
}

fpca_status mlp_buffers(fpca_ctx* ctx, int Bn, int R, int train, MlpBuf& w) {
  const size_t B = (size_t)Bn;
  size_t need = WsCarve::round(sizeof(__half) * W16_COUNT) + 4096;
  if (train)
    need += WsCarve::round(sizeof(float) * 32 * B) + 6 * WsCarve::round(sizeof(float) * HID * B) +
            WsCarve::round(sizeof(float) * 8 * B) + WsCarve::round(sizeof(float) * (B / R + 1)) +
            WsCarve::round(sizeof(int) * MC_MAX);
  void* ws = fpca_workspace(ctx, need);
  if (!ws) return fpca_fail(ctx, FPCA_E_OOM, "workspace (%zu bytes)", need);
  WsCarve c(ws);
  w = MlpBuf{};
  w.w16 = c.take<__half>(W16_COUNT);
  if (!train) return FPCA_OK;
  w.X = c.take<float>(32 * B);
  for (int l = 0; l < 3; ++l) {
    w.H[l] = c.take<float>(HID * B);
    w.D[l] = c.take<float>(HID * B);
  }
  w.D3 = c.take<float>(8 * B);
  w.losspart = c.take<float>(B / R + 1);
  w.mcount = c.take<int>(MC_MAX);
  w.parts = (int)std::min<long long>(MC_MAX, (6ll * Bn + MC_BYTES - 1) / MC_BYTES);
  return FPCA_OK;
}

template <int R>
fpca_status mlp_launch_rows(fpca_ctx* ctx, const float* th, const float* feat, const float* target,
                            const uint8_t* mask, int Bn, const MlpBuf& w, float* out, int train) {
  const size_t sm = mlp_rows_smem(R);
  cudaFuncSetAttribute(k_mlp_rows<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_mlp_rows<R><<<(Bn + R - 1) / R, 256, sm, ctx->stream>>>(Bn, th, feat, target, mask, w, out,
                                                            train);
  FPCA_LAUNCHED(ctx, "mlp_rows");
  return FPCA_OK;
}

fpca_status mlp_rows(fpca_ctx* ctx, const float* th, const float* feat, const float* target,
                     const uint8_t* mask, int Bn, int R, const MlpBuf& w, float* out, int train) {
  k_mlp_weights<<<MW_TILES + w.parts, 256, 0, ctx->stream>>>(th, w.w16, mask, 6ll * Bn, w.mcount);
  FPCA_LAUNCHED(ctx, "mlp_weights");
  if (R == 2) return mlp_launch_rows<2>(ctx, th, feat, target, mask, Bn, w, out, train);
  if (R == 4) return mlp_launch_rows<4>(ctx, th, feat, target, mask, Bn, w, out, train);
  return mlp_launch_rows<8>(ctx, th, feat, target, mask, Bn, w, out, train);
}

// splitmix64 (Steele, Lea and Flood 2014): the finaliser applied to a counter.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

// He-normal initial weights N(0, 2 / fan_in) and zero biases.  Parameter e draws
// its normal value by the Box-Muller transform of two uniforms in (0, 1] taken
// from the counter (seed, e): the result depends only on the seed.
__global__ void k_mlp_init(uint64_t seed, float* __restrict__ params) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= kParamCount) return;
  int l = 0;
  while (l + 1 < NLAYER && e >= layer_off(l + 1)) ++l;
  const long long r = e - layer_off(l);
  const int fi = layer_in(l), fo = layer_out(l);
  if (r >= (long long)fi * fo) {
    params[e] = 0.f;  // bias
    return;
  }
  const uint64_t a = splitmix64(seed * 0x2545F4914F6CDD1Dull + 2ull * (uint64_t)e);
  const uint64_t b = splitmix64(seed * 0x2545F4914F6CDD1Dull + 2ull * (uint64_t)e + 1ull);
  const double u1 = ((double)(a >> 11) + 1.0) * 0x1.0p-53;  // (0, 1]
  const double u2 = (double)(b >> 11) * 0x1.0p-53;          // [0, 1)
  const double z = sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
  params[e] = (float)(z * sqrt(2.0 / (double)fi));
}

// File layout of fpca_bw_mlp_io: magic, parameter count, the parameters, the
// 32 feature means and the 32 feature scales, all little-endian.
constexpr char kMlpMagic[8] = {'F', 'P', 'C', 'A', 'B', 'W', '0', '1'};

}  // namespace

extern "C" {

int64_t fpca_bw_param_count(void) { return kParamCount; }

fpca_status fpca_bw_mlp_init(fpca_ctx* ctx, uint64_t seed, float* params) {
  if (!ctx) return FPCA_E_INVALID_ARG;
  fpca_prof_mark(ctx);
  if (!params) return fpca_fail(ctx, FPCA_E_INVALID_ARG, "params is NULL");
  k_mlp_init<<<(int)((kParamCount + 255) / 256), 256, 0, ctx->stream>>>(seed, params);
  FPCA_LAUNCHED(ctx, "mlp_init");
  return FPCA_OK;
}

fpca_status fpca_bw_mlp_io(fpca_ctx* ctx, float* params, float* feat_mu, float* feat_sd,
                           const char* path, int save) {
  if (!ctx) return FPCA_E_INVALID_ARG;
  if (!params || !path) return fpca_fail(ctx, FPCA_E_INVALID_ARG, "params and path are required");
  if (fpca_no_capture(ctx, "fpca_bw_mlp_io") != FPCA_OK) return FPCA_E_UNSUPPORTED;
  std::vector<float> buf((size_t)kParamCount + 64, 0.f);
  const size_t nbytes = sizeof(float) * buf.size();
  if (save) {
    if (cudaStreamSynchronize(ctx->stream) != cudaSuccess)
      return fpca_check_launch(ctx, "mlp_io: stream");
    cudaError_t e = cudaMemcpy(buf.data(), params, sizeof(float) * kParamCount,
                               cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && feat_mu)
      e = cudaMemcpy(buf.data() + kParamCount, feat_mu, 32 * sizeof(float), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && feat_sd)
      e = cudaMemcpy(buf.data() + kParamCount + 32, feat_sd, 32 * sizeof(float),
                     cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return fpca_fail(ctx, FPCA_E_CUDA, "mlp_io: %s", cudaGetErrorString(e));
    FILE* f = std::fopen(path, "wb");
    if (!f) return fpca_fail(ctx, FPCA_E_INVALID_ARG, "mlp_io: cannot write %s", path);
    const int64_t count = kParamCount;
    const bool ok = std::fwrite(kMlpMagic, 1, 8, f) == 8 && std::fwrite(&count, 8, 1, f) == 1 &&
                    std::fwrite(buf.data(), 1, nbytes, f) == nbytes;
    if (std::fclose(f) != 0 || !ok)
      return fpca_fail(ctx, FPCA_E_INVALID_ARG, "mlp_io: short write to %s", path);
    return FPCA_OK;
  }
  FILE* f = std::fopen(path, "rb");
  if (!f) return fpca_fail(ctx, FPCA_E_INVALID_ARG, "mlp_io: cannot read %s", path);
  char magic[8];
  int64_t count = 0;
  const bool head = std::fread(magic, 1, 8, f) == 8 && std::fread(&count, 8, 1, f) == 1;
  const bool body = head && std::memcmp(magic, kMlpMagic, 8) == 0 && count == kParamCount &&
                    std::fread(buf.data(), 1, nbytes, f) == nbytes;
  std::fclose(f);
  if (!body)
    return fpca_fail(ctx, FPCA_E_INVALID_ARG,
                     "mlp_io: %s is not a saved network of %lld parameters", path,
                     (long long)kParamCount);
  cudaError_t e = cudaMemcpyAsync(params, buf.data(), sizeof(float) * kParamCount,
                                  cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess && feat_mu)
    e = cudaMemcpyAsync(feat_mu, buf.data() + kParamCount, 32 * sizeof(float),
                        cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess && feat_sd)
    e = cudaMemcpyAsync(feat_sd, buf.data() + kParamCount + 32, 32 * sizeof(float),
                        cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);  // buf is a host temporary
  if (e != cudaSuccess) return fpca_fail(ctx, FPCA_E_CUDA, "mlp_io: %s", cudaGetErrorString(e));
  return FPCA_OK;
}

fpca_status fpca_bw_predict(fpca_ctx* ctx, const float* params, const float* feat, int B,
                            float* out) {
  if (!ctx) return FPCA_E_INVALID_ARG;
  fpca_prof_mark(ctx);
  if (!params || !feat || !out || B < 1)
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "params, feat, out and B >= 1 are required");
  const int R = mlp_rows_per_cta(ctx, B);
  MlpBuf w;
  fpca_status s = mlp_buffers(ctx, B, R, 0, w);
  if (s != FPCA_OK) return s;
  return mlp_rows(ctx, params, feat, nullptr, nullptr, B, R, w, out, 0);
}

fpca_status fpca_bw_train_step(fpca_ctx* ctx, float* params, float* adam_m, float* adam_v,
                               int step, const float* feat, const float* target,
                               const uint8_t* tmask, int B, float lr, float wd, float* loss,
                               float* grad_out) {
  if (!ctx) return FPCA_E_INVALID_ARG;
  fpca_prof_mark(ctx);
  if (!params || !feat || !target || !tmask || B < 1)
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "params, feat, target, tmask and B >= 1 are required");
  if (step >= 1 && (!adam_m || !adam_v))
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "an update step needs the AdamW moments");
  const int R = mlp_rows_per_cta(ctx, B);
  MlpBuf w;
  fpca_status s = mlp_buffers(ctx, B, R, 1, w);
  if (s != FPCA_OK) return s;
  s = mlp_rows(ctx, params, feat, target, tmask, B, R, w, nullptr, 1);
  if (s != FPCA_OK) return s;
  AdamArgs ad{};
  if (step >= 1) {
    ad = AdamArgs{params, adam_m, adam_v, lr, wd, 1.f - powf(0.9f, (float)step),
                  1.f - powf(0.999f, (float)step)};
  }
  k_mlp_grads<<<MG_TILES, 256, 0, ctx->stream>>>(B, (B + R - 1) / R, w, ad, grad_out, loss);
  FPCA_LAUNCHED(ctx, "mlp_grads");
  return FPCA_OK;
}

}  // extern "C"
