// sgn_unet.cu - the periodic U-Net (include/sgn_unet.h) that corrects the
// GMRES starting value of sigma: any depth and widths.
//
// Training (forward, backward, Adam) runs direct convolutions on CUDA cores in
// NCHW: activations stored as T (BF16 or FP32), everything else FP32; sums over
// pixels (weight gradients, the loss) are per-block fixed-order reductions, so
// results are deterministic. Inference (sgn_unet_infer) runs the 3x3 layers
// after the first as BF16 implicit GEMMs on the tensor cores over NHWC
// activations (sgn_unet_tc.cuh).
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include <new>
#include <string>
#include <vector>

#include "sgn_unet.h"
#include "sgn_unet_tc.cuh"

namespace {

template <typename T>
__device__ __forceinline__ float ldf(const T* p);
template <>
__device__ __forceinline__ float ldf<float>(const float* p) {
  return *p;
}
template <>
__device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(*p);
}
template <typename T>
__device__ __forceinline__ T tof(float v);
template <>
__device__ __forceinline__ float tof<float>(float v) {
  return v;
}
template <>
__device__ __forceinline__ __nv_bfloat16 tof<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

// 3x3 periodic convolution. Forward (TR = false):
//   out[b][co][y][x] = bias[co] + sum_ci sum_k w[co][ci][k] in[b][ci][y+ky-1][x+kx-1]
// Transposed (TR = true, the gradient with respect to the input): the output
// channel is the forward input channel c, the input channel the forward output
// channel o, and the kernel is flipped:
//   out[b][c][y][x] = sum_o sum_k w[o][c][8-k] in[b][o][y+ky-1][x+kx-1]
// (Cw: the forward input-channel count, the row length of w.) H, W are powers
// of two >= 4; in and out have batch strides ibs, obs (elements).
//
// FP32-FMA bound in principle (44 of the 65 GFLOP of a training step of the
// 471,873-parameter network, batch 8 at 128^2). A thread keeps PX pixels x COT
// channels of sums in registers, as channel pairs for the packed FMA: with 8 x 8
// an input channel costs 288 packed FMAs (576 issue cycles of an SM quarter)
// against 27 shared loads (18 of them broadcasts of weights; 432). With 4 x 8 the
// loads cost more than the FMAs (360 against 288), with one pixel x 8 channels and
// a load per FMA they were all of it. Each stage of CCK input channels is
// fetched with every load in flight before the first is stored: a loop of
// dependent fetch-and-store pairs took 20 us a stage. Loss and gradients of one
// batch of 8 at 128^2: 11.5 -> 3.0 ms (with the weight gradients below).
// Each sum runs over (ci, ky, kx) in order, one rounded FMA at a time, whatever
// the tile: BF16 activations do not depend on it.
// Tile: TX x TY threads of PX x 1 pixels, TX = min(W / PX, 8),
// TY = min(H, 128 / TX, 16).
template <int PX>
constexpr int conv_cck() { return PX == 8 ? 4 : 8; }  // input channels per stage
// four consecutive elements as floats (VEC = false: of any address)
template <bool VEC = true>
__device__ __forceinline__ float4 load4(const float* p) {
  if constexpr (VEC) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], p[1], p[2], p[3]);
}
template <bool VEC = true>
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 r = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                     __uint_as_float(r.y & 0xffff0000u));
}
__device__ __forceinline__ void store4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void store4(__nv_bfloat16* p, float a, float b, float c, float d) {
  const __nv_bfloat162 u = __halves2bfloat162(__float2bfloat16_rn(a), __float2bfloat16_rn(b));
  const __nv_bfloat162 v = __halves2bfloat162(__float2bfloat16_rn(c), __float2bfloat16_rn(d));
  uint2 r;
  r.x = *reinterpret_cast<const unsigned*>(&u);
  r.y = *reinterpret_cast<const unsigned*>(&v);
  *reinterpret_cast<uint2*>(p) = r;
}

// Stages rows [0, nrow) of a tile: row r = (channel r / RPC, line r % RPC) at
// dst + dsto(r), tw interior pixels from element 4 on and the halo at 3 and
// tw + 4. 16-byte (8-byte) fetches, U in flight per thread; VEC = false: element by
// element, for a caller's input that starts at no 16-byte boundary.
template <int U, bool VEC, typename TI, class Src, class Dst>
__device__ __forceinline__ void stage_rows(int nrow, int ltw, int tid, int nthr, int x0, int W, Src src, Dst dst) {
  const int lv = ltw - 2, nvec = nrow << lv;  // 4-pixel vectors per row: 2^lv
  for (int base = 0; base < nvec; base += U * nthr) {
    float4 q[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + u * nthr + tid;
      if (i < nvec) q[u] = load4<VEC>(src(i >> lv) + x0 + 4 * (i & ((1 << lv) - 1)));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + u * nthr + tid;
      if (i < nvec) *reinterpret_cast<float4*>(dst(i >> lv) + 4 + 4 * (i & ((1 << lv) - 1))) = q[u];
    }
  }
  const int tw = 1 << ltw;
  for (int base = 0; base < 2 * nrow; base += 4 * nthr) {
    float q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = base + u * nthr + tid;
      if (i < 2 * nrow) q[u] = ldf(src(i >> 1) + ((x0 + ((i & 1) ? tw : -1)) & (W - 1)));
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = base + u * nthr + tid;
      if (i < 2 * nrow) dst(i >> 1)[(i & 1) ? tw + 4 : 3] = q[u];
    }
  }
}

template <typename TI, typename TO, bool TR, int COT, int PX, bool VEC>
__global__ void __launch_bounds__(128) k_conv3(const TI* __restrict__ in, size_t ibs, int Ci, TO* out, size_t obs,
                                               const float* __restrict__ w, const float* __restrict__ bias, int Cw,
                                               int H, int W, int lTX, int relu) {
  constexpr int CP = COT / 2, CCK = conv_cck<PX>(), LPX = PX == 8 ? 3 : 2;
  const int TX = 1 << lTX, TY = blockDim.x >> lTX, RPC = TY + 2;
  const int tid = threadIdx.x, tx = tid & (TX - 1), ty = tid >> lTX;
  const int ltw = lTX + LPX, tw = 1 << ltw, RS = tw + 8;
  extern __shared__ __align__(16) float csm[];
  float* tile = csm;                             // [CCK][TY + 2][RS]
  float* ws = csm + (size_t)CCK * RPC * RS;      // [CCK][9][COT]
  const int tiles_x = W / tw;
  const int x0 = (blockIdx.x % tiles_x) * tw, y0 = (blockIdx.x / tiles_x) * TY;
  const int co0 = blockIdx.y * COT, b = blockIdx.z;
  const size_t HW = (size_t)H * W;
  const TI* inb = in + (size_t)b * ibs;
  // r / RPC for r < 256, RPC in 6..18
  const unsigned inv = 65536u / (unsigned)RPC + 1u;
  float2 acc[PX][CP];
#pragma unroll
  for (int p = 0; p < PX; ++p)
#pragma unroll
    for (int c = 0; c < CP; ++c) acc[p][c] = make_float2(0.f, 0.f);
  for (int c0 = 0; c0 < Ci; c0 += CCK) {
    const int nc = min(CCK, Ci - c0);
    if (c0) __syncthreads();
    stage_rows<9, VEC, TI>(
        nc * RPC, ltw, tid, blockDim.x, x0, W,
        [&](int r) {
          const int ci = (int)((unsigned)r * inv >> 16), ly = r - ci * RPC;
          return inb + (size_t)(c0 + ci) * HW + (size_t)((y0 + ly - 1) & (H - 1)) * W;
        },
        [&](int r) { return tile + r * RS; });
    constexpr int WU = (CCK * 9 * COT + 127) / 128;
    const int nwt = nc * 9 * COT;
    for (int base = 0; base < nwt; base += WU * blockDim.x) {
      float q[WU];
      int to[WU];
#pragma unroll
      for (int u = 0; u < WU; ++u) {
        const int i = base + u * (int)blockDim.x + tid;
        // TR: w[c0 + ci][co0 + c][8 - k], c then ci outermost; else w[co0 + c][c0 + ci][k]
        const int k = i % 9, m = i / 9, ci = TR ? m / COT : m % nc, c = TR ? m % COT : m / nc;
        to[u] = (ci * 9 + k) * COT + c;
        if (i < nwt)
          q[u] = TR ? w[((size_t)(c0 + ci) * Cw + co0 + c) * 9 + (8 - k)] : w[((size_t)(co0 + c) * Ci + c0 + ci) * 9 + k];
      }
#pragma unroll
      for (int u = 0; u < WU; ++u)
        if (base + u * (int)blockDim.x + tid < nwt) ws[to[u]] = q[u];
    }
    __syncthreads();
    for (int ci = 0; ci < nc; ++ci) {
      const float* wc = ws + ci * 9 * COT;
#pragma unroll
      for (int ky = 0; ky < 3; ++ky) {
        const float* row = tile + (ci * RPC + ty + ky) * RS + 4 + PX * tx;
        float v[PX + 2];
        v[0] = row[-1];
        v[PX + 1] = row[PX];
#pragma unroll
        for (int p = 0; p < PX; p += 4) {
          const float4 q = *reinterpret_cast<const float4*>(row + p);
          v[p + 1] = q.x;
          v[p + 2] = q.y;
          v[p + 3] = q.z;
          v[p + 4] = q.w;
        }
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
          float2 wv[CP];
#pragma unroll
          for (int c = 0; c < CP; c += 2) {
            const float4 q = *reinterpret_cast<const float4*>(wc + (ky * 3 + kx) * COT + 2 * c);
            wv[c] = make_float2(q.x, q.y);
            wv[c + 1] = make_float2(q.z, q.w);
          }
#pragma unroll
          for (int p = 0; p < PX; ++p) {
            const float2 vv = make_float2(v[p + kx], v[p + kx]);
#pragma unroll
            for (int c = 0; c < CP; ++c) acc[p][c] = __ffma2_rn(wv[c], vv, acc[p][c]);
          }
        }
      }
    }
  }
  const int y = y0 + ty, x = x0 + PX * tx;
#pragma unroll
  for (int c = 0; c < COT; ++c) {
    const float bb = bias ? bias[co0 + c] : 0.f;
    float o[PX];
#pragma unroll
    for (int p = 0; p < PX; ++p) {
      o[p] = ((c & 1) ? acc[p][c >> 1].y : acc[p][c >> 1].x) + bb;
      if (relu) o[p] = fmaxf(o[p], 0.f);
    }
    TO* dst = out + (size_t)b * obs + (size_t)(co0 + c) * HW + (size_t)y * W + x;
#pragma unroll
    for (int p = 0; p < PX; p += 4) store4(dst + p, o[p], o[p + 1], o[p + 2], o[p + 3]);
  }
}

// Weight gradients dw[co][ci][k] = sum_{b,y,x} dp[b][co][y][x] in[b][ci][y+ky-1][x+kx-1]
// and db[co] = sum dp[b][co], as partial sums of a split of the pixels.
// A block takes 16 input x 32 output channels and the chunks z, z + splits, ...
// of up to 128 pixels (R rows x CW columns); a thread one input channel and 4
// output channels: 36 sums in registers, fed by 10 vector loads per 4 pixels and
// 72 packed FMAs: 71 us a layer on average in the step above. (One block per
// channel pair read every activation 9 Co times.) A chunk is summed on its own (128
// terms at most), a block adds its chunks one after another (chunks / splits of
// them: up to 219, the most at 512^2, batch 64 and 16 to 16 channels), and the blocks'
// sums go through k_part_sum. Fixed order: deterministic.
constexpr int DWPX = 128;
__host__ __device__ inline void dw_chunk(int H, int W, int* R, int* CW) {
  *CW = W < 64 ? W : 64;
  const int r = DWPX / *CW;
  *R = r < H ? r : H;
}
__host__ __device__ inline int dw_row_stride(int CW) { return CW + 8; }
// words per input channel of the staged tile, = 4 mod 32 (conflict-free 16-byte loads)
__host__ __device__ inline int dw_in_stride(int R, int CW) {
  const int n = (R + 2) * dw_row_stride(CW);
  return (n + 27) / 32 * 32 + 4;
}
template <typename TI, bool VEC>
__global__ void __launch_bounds__(128, 4) k_conv3_dw(const TI* __restrict__ in, size_t ibs, int Ci,
                                                  const float* __restrict__ dp, size_t dbs, int Co, int H, int W,
                                                  int B, float* part) {
  extern __shared__ __align__(16) float csm[];
  int R, CW;
  dw_chunk(H, W, &R, &CW);
  const int RS = dw_row_stride(CW), IS = dw_in_stride(R, CW);
  float* ti = csm;            // [16][IS]
  float* tg = csm + 16 * IS;  // [R * CW][32 + 4]
  constexpr int GS = 36;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cl = tid & 15, cg = tid >> 4;
  const int ci0 = blockIdx.x * 16, co0 = blockIdx.y * 32, splits = gridDim.z;
  const size_t HW = (size_t)H * W;
  const int cpr = W / CW, chunks = B * (H / R) * cpr;
  const int lCW = 31 - __clz(CW), nin = min(16, Ci - ci0);
  const unsigned inv = 65536u / (unsigned)(R + 2) + 1u;  // r / (R + 2), r < 16 (R + 2) <= 288
  // channels past Ci contribute zeros
  for (int i = nin * IS + tid; i < 16 * IS; i += 128) ti[i] = 0.f;
  float2 acc[9][2];
  float2 ab[2];
#pragma unroll
  for (int k = 0; k < 9; ++k) acc[k][0] = acc[k][1] = make_float2(0.f, 0.f);
  ab[0] = ab[1] = make_float2(0.f, 0.f);
  for (int ch = blockIdx.z; ch < chunks; ch += splits) {
    const int b = ch / ((H / R) * cpr), rem = ch - b * (H / R) * cpr;
    const int y0 = rem / cpr * R, x0 = (rem % cpr) * CW;
    __syncthreads();
    stage_rows<9, VEC, TI>(
        nin * (R + 2), lCW, tid, 128, x0, W,
        [&](int r) {
          const int c = (int)((unsigned)r * inv >> 16), ly = r - c * (R + 2);
          return in + (size_t)b * ibs + (size_t)(ci0 + c) * HW + (size_t)((y0 + ly - 1) & (H - 1)) * W;
        },
        [&](int r) {
          const int c = (int)((unsigned)r * inv >> 16);
          return ti + c * IS + (r - c * (R + 2)) * RS;
        });
    // lane = output channel: conflict-free transposed stores
    const int nv = R * CW / 4;
    const bool gok = co0 + lane < Co;
    const float* gsrc = dp + (size_t)b * dbs + (size_t)(gok ? co0 + lane : 0) * HW + (size_t)y0 * W + x0;
    float4 q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = 4 * u + warp;
      if (i < nv) {
        const int ly = 4 * i >> lCW;
        q[u] = gok ? load4(gsrc + (size_t)ly * W + (4 * i - (ly << lCW))) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = 4 * u + warp;
      if (i < nv) {
        float* t = tg + 4 * i * GS + lane;
        t[0] = q[u].x;
        t[GS] = q[u].y;
        t[2 * GS] = q[u].z;
        t[3 * GS] = q[u].w;
      }
    }
    __syncthreads();
    float2 s[9][2], sb[2];
#pragma unroll
    for (int k = 0; k < 9; ++k) s[k][0] = s[k][1] = make_float2(0.f, 0.f);
    sb[0] = sb[1] = make_float2(0.f, 0.f);
    for (int r = 0; r < R; ++r) {
      for (int x = 0; x < CW; x += 4) {
        float2 g[4][2];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const float4 q = *reinterpret_cast<const float4*>(tg + (r * CW + x + p) * GS + 4 * cg);
          g[p][0] = make_float2(q.x, q.y);
          g[p][1] = make_float2(q.z, q.w);
        }
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
          const float* row = ti + cl * IS + (r + ky) * RS + 4 + x;
          const float4 ra = *reinterpret_cast<const float4*>(row);
          const float v[6] = {row[-1], ra.x, ra.y, ra.z, ra.w, row[4]};
#pragma unroll
          for (int kx = 0; kx < 3; ++kx)
#pragma unroll
            for (int p = 0; p < 4; ++p) {
              const float2 vv = make_float2(v[p + kx], v[p + kx]);
              s[ky * 3 + kx][0] = __ffma2_rn(g[p][0], vv, s[ky * 3 + kx][0]);
              s[ky * 3 + kx][1] = __ffma2_rn(g[p][1], vv, s[ky * 3 + kx][1]);
            }
        }
        if (cl == 0) {
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            sb[0] = __fadd2_rn(sb[0], g[p][0]);
            sb[1] = __fadd2_rn(sb[1], g[p][1]);
          }
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      acc[k][0] = __fadd2_rn(acc[k][0], s[k][0]);
      acc[k][1] = __fadd2_rn(acc[k][1], s[k][1]);
    }
    ab[0] = __fadd2_rn(ab[0], sb[0]);
    ab[1] = __fadd2_rn(ab[1], sb[1]);
  }
  // this split's sums: [Co][Ci][9], then [Co]
  float* o = part + (size_t)blockIdx.z * ((size_t)Co * Ci * 9 + Co);
  const int ci = ci0 + cl;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int co = co0 + 4 * cg + c;
    if (co >= Co) continue;
    if (ci < Ci) {
#pragma unroll
      for (int k = 0; k < 9; ++k)
        o[((size_t)co * Ci + ci) * 9 + k] = (c & 1) ? acc[k][c >> 1].y : acc[k][c >> 1].x;
    }
    if (ci0 == 0 && cl == 0) o[(size_t)Co * Ci * 9 + co] = (c & 1) ? ab[c >> 1].y : ab[c >> 1].x;
  }
}
// blocks of pixel chunks a weight gradient is split into: about 600 blocks in all
inline int dw_splits(int Ci, int Co, int H, int W, int B) {
  int R, CW;
  dw_chunk(H, W, &R, &CW);
  const int tiles = ((Ci + 15) / 16) * ((Co + 31) / 32), chunks = B * (H / R) * (W / CW);
  const int s = (600 + tiles - 1) / tiles;
  return s < chunks ? s : chunks;
}
// out[i] = sum of the splits' partial sums: 8 threads a sum, each over every
// 8th split, then in order (32 x 8 threads)
__global__ void __launch_bounds__(256) k_part_sum(const float* __restrict__ part, int n, int splits, float* out) {
  __shared__ float red[8][32];
  const int i = blockIdx.x * 32 + threadIdx.x;
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  if (i < n) {
    int z = threadIdx.y;
    for (; z + 24 < splits; z += 32)
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] += part[(size_t)(z + 8 * u) * n + i];
    for (; z < splits; z += 8) s[0] += part[(size_t)z * n + i];
  }
  red[threadIdx.y][threadIdx.x] = (s[0] + s[1]) + (s[2] + s[3]);
  __syncthreads();
  if (threadIdx.y == 0 && i < n) {
    float t = 0.f;
#pragma unroll
    for (int z = 0; z < 8; ++z) t += red[z][threadIdx.x];
    out[i] = t;
  }
}

// Block sum of K floats in fixed order; thread 0 gets the sums in v.
template <int K>
__device__ __forceinline__ void block_sum(float (&v)[K], float* red /* K * 32 */) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k)
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  if (lane == 0)
    for (int k = 0; k < K; ++k) red[k * 32 + wid] = v[k];
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 0; k < K; ++k) {
      float t = 0.f;
      for (int i = 0; i < nw; ++i) t += red[k * 32 + i];
      v[k] = t;
    }
}

// 1x1 convolution C -> 1 (the output layer), FP32 output
template <typename T>
__global__ void k_conv1_fwd(const T* __restrict__ in, size_t ibs, int C, const float* __restrict__ w,
                            const float* __restrict__ bias, float* out, int HW, int B) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * HW) return;
  const int b = i / HW, yx = i % HW;
  float v = bias[0];
  for (int c = 0; c < C; ++c) v = fmaf(w[c], ldf(in + (size_t)b * ibs + (size_t)c * HW + yx), v);
  out[i] = v;
}

// gradients of the output layer: dw[c] = sum dout in[c], db = sum dout (block
// c < C: dw[c]; block C: db), as partial sums part[z][c] of gridDim.y ranges of
// the pixels; din[c] = w[c] dout masked by in > 0 (the ReLU of the layer before).
template <typename T>
__global__ void __launch_bounds__(256) k_conv1_dw(const T* __restrict__ in, size_t ibs, int C,
                                                  const float* __restrict__ dout, int HW, int B, float* part) {
  __shared__ float red[32];
  const int c = blockIdx.x;
  float acc[1] = {0.f};
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < B * HW; i += gridDim.y * blockDim.x) {
    const int b = i / HW, yx = i % HW;
    acc[0] += dout[i] * (c < C ? ldf(in + (size_t)b * ibs + (size_t)c * HW + yx) : 1.f);
  }
  block_sum<1>(acc, red);
  if (threadIdx.x == 0) part[(size_t)blockIdx.y * (C + 1) + c] = acc[0];
}

template <typename T>
__global__ void k_conv1_dx_relu(const T* __restrict__ act, size_t abs_, int C, const float* __restrict__ w,
                                const float* __restrict__ dout, float* din, size_t dbs, int HW, int B) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)B * C * HW) return;
  const int b = (int)(i / ((size_t)C * HW));
  const int r = (int)(i % ((size_t)C * HW)), c = r / HW, yx = r % HW;
  const float a = ldf(act + (size_t)b * abs_ + (size_t)c * HW + yx);
  din[(size_t)b * dbs + (size_t)c * HW + yx] = a > 0.f ? w[c] * dout[(size_t)b * HW + yx] : 0.f;
}

// g[b][c][i] = (g (+ extra)) * (act > 0): the ReLU backward, optionally after
// adding a second gradient (the skip connection's)
template <typename T>
__global__ void k_relu_bwd(const T* __restrict__ act, size_t abs_, float* g, size_t gbs,
                           const float* __restrict__ extra, size_t ebs, int C, int HW, int B) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)B * C * HW) return;
  const int b = (int)(i / ((size_t)C * HW));
  const size_t r = i % ((size_t)C * HW);
  float v = g[(size_t)b * gbs + r];
  if (extra) v += extra[(size_t)b * ebs + r];
  g[(size_t)b * gbs + r] = ldf(act + (size_t)b * abs_ + r) > 0.f ? v : 0.f;
}

// 2x2 average pool: out [C][H/2][W/2] from in [C][H][W]
template <typename T>
__global__ void k_pool(const T* __restrict__ in, size_t ibs, T* out, size_t obs, int C, int H, int W, int B) {
  const int h = H / 2, w = W / 2;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)B * C * h * w) return;
  const int b = (int)(i / ((size_t)C * h * w));
  const int r = (int)(i % ((size_t)C * h * w)), c = r / (h * w), yx = r % (h * w), y = yx / w, x = yx % w;
  const T* s = in + (size_t)b * ibs + (size_t)c * H * W + (size_t)(2 * y) * W + 2 * x;
  const float v = 0.25f * ((ldf(s) + ldf(s + 1)) + (ldf(s + W) + ldf(s + W + 1)));
  out[(size_t)b * obs + r] = tof<T>(v);
}
// din [C][H][W] = dout [C][H/2][W/2] / 4 at each of the four children
__global__ void k_pool_bwd(const float* __restrict__ dout, size_t obs, float* din, size_t ibs, int C, int H, int W,
                           int B) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)B * C * H * W) return;
  const int b = (int)(i / ((size_t)C * H * W));
  const int r = (int)(i % ((size_t)C * H * W)), c = r / (H * W), yx = r % (H * W), y = yx / W, x = yx % W;
  din[(size_t)b * ibs + r] = 0.25f * dout[(size_t)b * obs + (size_t)c * (H / 2) * (W / 2) + (y / 2) * (W / 2) + x / 2];
}
// nearest 2x upsample: out [C][2H][2W] from in [C][H][W]
template <typename T>
__global__ void k_up(const T* __restrict__ in, size_t ibs, T* out, size_t obs, int C, int H, int W, int B) {
  const int H2 = 2 * H, W2 = 2 * W;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)B * C * H2 * W2) return;
  const int b = (int)(i / ((size_t)C * H2 * W2));
  const int r = (int)(i % ((size_t)C * H2 * W2)), c = r / (H2 * W2), yx = r % (H2 * W2), y = yx / W2, x = yx % W2;
  out[(size_t)b * obs + r] = in[(size_t)b * ibs + (size_t)c * H * W + (y / 2) * W + x / 2];
}
// din [C][H][W] = sum of dout over the four children in [C][2H][2W]
__global__ void k_up_bwd(const float* __restrict__ dout, size_t obs, float* din, size_t ibs, int C, int H, int W,
                         int B) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)B * C * H * W) return;
  const int b = (int)(i / ((size_t)C * H * W));
  const int r = (int)(i % ((size_t)C * H * W)), c = r / (H * W), yx = r % (H * W), y = yx / W, x = yx % W;
  const float* s = dout + (size_t)b * obs + (size_t)c * 4 * H * W + (size_t)(2 * y) * (2 * W) + 2 * x;
  din[(size_t)b * ibs + r] = (s[0] + s[1]) + (s[2 * W] + s[2 * W + 1]);
}

// dout = 2 (out - target) / n; loss = sum (out - target)^2 / n: block sums in
// part, added in order by the last block to finish (ticket: zeroed, left zeroed)
constexpr int MSE_BLOCKS = 128;
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ out, const float* __restrict__ target,
                                             float* dout, int n, double* loss, double* part, unsigned* ticket) {
  __shared__ double red[32];
  __shared__ int s_last;
  double acc = 0.0;
  const float s = 2.f / (float)n;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float d = out[i] - target[i];
    dout[i] = s * d;
    acc += (double)d * d;
  }
  if (!loss) return;
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
    part[blockIdx.x] = t;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    if (s_last) *ticket = 0u;
  }
  __syncthreads();
  if (!s_last || threadIdx.x >= 32) return;
  double t = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += 32) t += __ldcg(part + i);
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (threadIdx.x == 0) *loss = t / (double)n;
}

__global__ void k_adam(float* p, const float* __restrict__ g, float* m, float* v, long long n, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

inline unsigned blocks_for(size_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

constexpr int kMaxLevels = 6;
constexpr int kConv1Splits = 16;  // ranges of pixels in the output layer's gradient

struct Layer {
  int Ci, Co, k;
  long long woff, boff;
  // tensor-core inference (3x3 layers after the first)
  int KC = 0, nkb = 0, smem = 0;
  long long ioff = -1;
  int level = 0;     // resolution level (grid side n / 2^level)
  bool row = false;  // >= 128 pixels per image: the halo-staged row kernel
};


}  // namespace

struct sgn_unet_ctx {
  int n = 0, maxB = 0, bf16 = 1;
  int D = 0, w[kMaxLevels] = {0};
  cudaStream_t stream = 0;
  std::vector<Layer> L;
  long long P = 0;
  float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
  // training activations (element type by bf16), NCHW, per level l (grid n / 2^l):
  //   A[l]   w_l channels: e_l's output (l < D-1), b0's output (l = D-1)
  //   CAT[l] w_{l+1} + w_l channels: upsampled level below, then s_l's output (l < D-1)
  //   Q[l]   w_l channels on level l+1's grid: the pooled s_l (l < D-1)
  //   U[l]   w_l channels: d_l's output (l < D-1), b1's output (l = D-1)
  void *A[kMaxLevels] = {}, *CAT[kMaxLevels] = {}, *Q[kMaxLevels] = {}, *U[kMaxLevels] = {};
  float *OUT = nullptr, *gOUT = nullptr;
  // partial sums of the weight gradients and of the loss
  float* part = nullptr;
  double* mse_part = nullptr;
  unsigned* ticket = nullptr;
  // FP32 gradients: two scratch tensors of wmax channels per level, and the
  // concatenation's gradient per level
  float *G[kMaxLevels][2] = {}, *gCAT[kMaxLevels] = {};
  // inference (NHWC BF16): e_l / b0 outputs, s_l outputs, pooled, d_l / b1 outputs
  __nv_bfloat16 *tA[kMaxLevels] = {}, *tS[kMaxLevels] = {}, *tQ[kMaxLevels] = {}, *tU[kMaxLevels] = {};
  __nv_bfloat16* wimg = nullptr;
  unet_tc::WImgTable wtab{};
  int* dev_err = nullptr;
  const float* lastIn = nullptr;
  int lastB = 0;
  std::vector<void*> allocs;
  std::string err;
};

namespace {

// parameter order: e_0, s_0, ..., e_{D-2}, s_{D-2}, b0, b1, d_{D-2}, ..., d_0, out
inline int iE(int l) { return 2 * l; }
inline int iS(int l) { return 2 * l + 1; }
inline int iB0(const sgn_unet_ctx* net) { return 2 * (net->D - 1); }
inline int iB1(const sgn_unet_ctx* net) { return 2 * (net->D - 1) + 1; }
inline int iD(const sgn_unet_ctx* net, int l) { return 2 * net->D + (net->D - 2 - l); }
inline int iOut(const sgn_unet_ctx* net) { return 3 * net->D - 1; }

struct Fail {
  sgn_status st;
};

#define UCK(...)                                                                                     \
  do {                                                                                               \
    cudaError_t e_ = (__VA_ARGS__);                                                                  \
    if (e_ != cudaSuccess) {                                                                         \
      net->err = std::string(#__VA_ARGS__) + ": " + cudaGetErrorString(e_);                          \
      throw Fail{SGN_ECUDA};                                                                         \
    }                                                                                                \
  } while (0)

void* ualloc(sgn_unet_ctx* net, size_t bytes) {
  void* p = nullptr;
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    net->err = "cudaMalloc failed";
    throw Fail{SGN_ENOMEM};
  }
  net->allocs.push_back(p);
  return p;
}

// Kaiming-uniform weights (bound sqrt(6 / fan_in)), zero biases; the output
// layer starts 10x smaller so that the first corrections are small.
void init_params(sgn_unet_ctx* net, unsigned long long seed) {
  std::vector<float> h((size_t)net->P, 0.f);
  unsigned long long s = seed ^ 0x9e3779b97f4a7c15ull;
  auto next = [&]() {  // splitmix64
    s += 0x9e3779b97f4a7c15ull;
    unsigned long long z = s;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    z ^= z >> 31;
    return (double)(z >> 11) / 9007199254740992.0;  // [0, 1)
  };
  const int out_layer = iOut(net);
  for (size_t li = 0; li < net->L.size(); ++li) {
    const Layer& l = net->L[li];
    const double fan_in = (double)l.Ci * l.k * l.k;
    const double bound = sqrt(6.0 / fan_in) * ((int)li == out_layer ? 0.1 : 1.0);
    const long long nw = (long long)l.Co * l.Ci * l.k * l.k;
    for (long long i = 0; i < nw; ++i) h[(size_t)(l.woff + i)] = (float)((2.0 * next() - 1.0) * bound);
  }
  UCK(cudaMemcpy(net->params, h.data(), sizeof(float) * (size_t)net->P, cudaMemcpyHostToDevice));
  UCK(cudaMemset(net->m, 0, sizeof(float) * (size_t)net->P));
  UCK(cudaMemset(net->v, 0, sizeof(float) * (size_t)net->P));
  UCK(cudaMemset(net->grads, 0, sizeof(float) * (size_t)net->P));
}

template <typename TI, typename TO, bool TR, bool VEC, int COT, int PX>
void conv3_tile(sgn_unet_ctx* net, const TI* in, size_t ibs, int Ci, TO* out, size_t obs, int Co, const float* w,
                const float* bias, int Cw, int H, int B, bool relu) {
  int lTX = 0;
  while (lTX < 3 && (2 * PX << lTX) <= H) ++lTX;
  const int TX = 1 << lTX;
  int TY = 128 / TX;
  TY = TY < 16 ? TY : 16;
  TY = TY < H ? TY : H;
  const dim3 grid((unsigned)((H / (PX * TX)) * (H / TY)), Co / COT, B);
  const size_t smem =
      sizeof(float) * conv_cck<PX>() * ((size_t)(TY + 2) * (PX * TX + 8) + 9 * (size_t)COT);
  k_conv3<TI, TO, TR, COT, PX, VEC><<<grid, TX * TY, smem, net->stream>>>(in, ibs, Ci, out, obs, w, bias, Cw, H, H, lTX,
                                                                    relu ? 1 : 0);
  UCK(cudaGetLastError());
}
// Ci input and Co output channels (Co a multiple of 16): 8 pixels x 8 channels
// a thread where that leaves two blocks per SM (64 x 16 pixels each), else 4 x 8
template <typename TI, typename TO, bool TR, bool VEC>
void conv3_launch(sgn_unet_ctx* net, const TI* in, size_t ibs, int Ci, TO* out, size_t obs, int Co, const float* w,
                  const float* bias, int Cw, int H, int B, bool relu) {
  if (H >= 64 && (long long)(H / 64) * (H / 16) * (Co / 8) * B >= 256)
    conv3_tile<TI, TO, TR, VEC, 8, 8>(net, in, ibs, Ci, out, obs, Co, w, bias, Cw, H, B, relu);
  else
    conv3_tile<TI, TO, TR, VEC, 8, 4>(net, in, ibs, Ci, out, obs, Co, w, bias, Cw, H, B, relu);
}
template <typename TI, typename TO, bool VEC = true>
void conv3(sgn_unet_ctx* net, const TI* in, size_t ibs, int li, TO* out, size_t obs, int H, int B, bool relu) {
  const Layer& l = net->L[li];
  conv3_launch<TI, TO, false, VEC>(net, in, ibs, l.Ci, out, obs, l.Co, net->params + l.woff, net->params + l.boff, l.Ci, H,
                              B, relu);
}
// gradient with respect to the layer input (channels Ci) from dp (channels Co)
void conv3_dx(sgn_unet_ctx* net, const float* dp, size_t dbs, int li, float* dx, size_t xbs, int H, int B) {
  const Layer& l = net->L[li];
  conv3_launch<float, float, true, true>(net, dp, dbs, l.Co, dx, xbs, l.Ci, net->params + l.woff, nullptr, l.Ci, H, B,
                                   false);
}
template <typename TI, bool VEC = true>
void conv3_dw(sgn_unet_ctx* net, const TI* in, size_t ibs, const float* dp, size_t dbs, int li, int H, int B) {
  const Layer& l = net->L[li];
  int R, CW;
  dw_chunk(H, H, &R, &CW);
  const int splits = dw_splits(l.Ci, l.Co, H, H, B), n = l.Co * l.Ci * 9 + l.Co;
  const size_t smem = sizeof(float) * (16 * (size_t)dw_in_stride(R, CW) + (size_t)R * CW * 36);
  k_conv3_dw<TI, VEC><<<dim3((l.Ci + 15) / 16, (l.Co + 31) / 32, splits), 128, smem, net->stream>>>(
      in, ibs, l.Ci, dp, dbs, l.Co, H, H, B, net->part);
  UCK(cudaGetLastError());
  k_part_sum<<<blocks_for(n, 32), dim3(32, 8), 0, net->stream>>>(net->part, n, splits, net->grads + l.woff);
  UCK(cudaGetLastError());
}
template <typename T>
void relu_bwd(sgn_unet_ctx* net, const T* act, size_t abs_, float* g, size_t gbs, const float* extra, size_t ebs,
              int C, int H, int B) {
  const size_t n = (size_t)B * C * H * H;
  k_relu_bwd<T><<<blocks_for(n), 256, 0, net->stream>>>(act, abs_, g, gbs, extra, ebs, C, H * H, B);
  UCK(cudaGetLastError());
}

// Whether the vector fetches of stage_rows may read p: a caller's input, the one
// tensor that the handle does not lay out itself, may start at any element.
inline bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

inline size_t npix(const sgn_unet_ctx* net, int l) { return (size_t)(net->n >> l) * (size_t)(net->n >> l); }

template <typename T>
void forward_impl(sgn_unet_ctx* net, const float* in, float* out, int B) {
  const int D = net->D;
  const int* w = net->w;
  // encoder
  for (int l = 0; l < D - 1; ++l) {
    const int H = net->n >> l;
    const size_t N = npix(net, l), Nq = npix(net, l + 1);
    T* A = (T*)net->A[l];
    T* S = (T*)net->CAT[l] + (size_t)w[l + 1] * N;  // s_l lives in CAT[l] after the upsampled channels
    const size_t cs = (size_t)(w[l + 1] + w[l]) * N;
    if (l == 0 && aligned16(in))
      conv3<float, T>(net, in, 4 * N, iE(0), A, (size_t)w[0] * N, H, B, true);
    else if (l == 0)
      conv3<float, T, false>(net, in, 4 * N, iE(0), A, (size_t)w[0] * N, H, B, true);
    else
      conv3<T, T>(net, (const T*)net->Q[l - 1], (size_t)w[l - 1] * N, iE(l), A, (size_t)w[l] * N, H, B, true);
    conv3<T, T>(net, A, (size_t)w[l] * N, iS(l), S, cs, H, B, true);
    k_pool<T><<<blocks_for((size_t)B * w[l] * Nq), 256, 0, net->stream>>>(S, cs, (T*)net->Q[l], (size_t)w[l] * Nq,
                                                                           w[l], H, H, B);
    UCK(cudaGetLastError());
  }
  // bottleneck
  {
    const int l = D - 1, H = net->n >> l;
    const size_t N = npix(net, l);
    conv3<T, T>(net, (const T*)net->Q[l - 1], (size_t)w[l - 1] * N, iB0(net), (T*)net->A[l], (size_t)w[l] * N, H, B,
                true);
    conv3<T, T>(net, (const T*)net->A[l], (size_t)w[l] * N, iB1(net), (T*)net->U[l], (size_t)w[l] * N, H, B, true);
  }
  // decoder
  for (int l = D - 2; l >= 0; --l) {
    const int H = net->n >> l;
    const size_t N = npix(net, l), Nb = npix(net, l + 1);
    const size_t cs = (size_t)(w[l + 1] + w[l]) * N;
    k_up<T><<<blocks_for((size_t)B * w[l + 1] * N), 256, 0, net->stream>>>(
        (const T*)net->U[l + 1], (size_t)w[l + 1] * Nb, (T*)net->CAT[l], cs, w[l + 1], H / 2, H / 2, B);
    UCK(cudaGetLastError());
    conv3<T, T>(net, (const T*)net->CAT[l], cs, iD(net, l), (T*)net->U[l], (size_t)w[l] * N, H, B, true);
  }
  const Layer& lo = net->L[iOut(net)];
  const size_t N0 = npix(net, 0);
  k_conv1_fwd<T><<<blocks_for((size_t)B * N0), 256, 0, net->stream>>>(
      (const T*)net->U[0], (size_t)w[0] * N0, w[0], net->params + lo.woff, net->params + lo.boff, net->OUT, (int)N0,
      B);
  UCK(cudaGetLastError());
  if (out) UCK(cudaMemcpyAsync(out, net->OUT, sizeof(float) * B * N0, cudaMemcpyDeviceToDevice, net->stream));
}

template <typename T>
void backward_impl(sgn_unet_ctx* net, const float* target, double* loss) {
  const int D = net->D, B = net->lastB;
  const int* w = net->w;
  const size_t N0 = npix(net, 0);
  k_mse<<<MSE_BLOCKS, 256, 0, net->stream>>>(net->OUT, target, net->gOUT, (int)(B * N0), loss, net->mse_part,
                                              net->ticket);
  UCK(cudaGetLastError());
  // output layer w_0 -> 1, then the ReLU of d_0
  const Layer& lo = net->L[iOut(net)];
  k_conv1_dw<T><<<dim3(w[0] + 1, kConv1Splits), 256, 0, net->stream>>>((const T*)net->U[0], (size_t)w[0] * N0, w[0],
                                                                       net->gOUT, (int)N0, B, net->part);
  UCK(cudaGetLastError());
  k_part_sum<<<blocks_for(w[0] + 1, 32), dim3(32, 8), 0, net->stream>>>(net->part, w[0] + 1, kConv1Splits, net->grads + lo.woff);
  UCK(cudaGetLastError());
  k_conv1_dx_relu<T><<<blocks_for((size_t)B * w[0] * N0), 256, 0, net->stream>>>(
      (const T*)net->U[0], (size_t)w[0] * N0, w[0], net->params + lo.woff, net->gOUT, net->G[0][0],
      (size_t)w[0] * N0, (int)N0, B);
  UCK(cudaGetLastError());
  // decoder, from the top level down the U: G[l][0] holds d(pre-activation of d_l)
  for (int l = 0; l < D - 1; ++l) {
    const int H = net->n >> l;
    const size_t N = npix(net, l), Nb = npix(net, l + 1);
    const size_t cs = (size_t)(w[l + 1] + w[l]) * N;
    conv3_dw<T>(net, (const T*)net->CAT[l], cs, net->G[l][0], (size_t)w[l] * N, iD(net, l), H, B);
    conv3_dx(net, net->G[l][0], (size_t)w[l] * N, iD(net, l), net->gCAT[l], cs, H, B);
    // the upsampled channels came from U[l+1] (the ReLU output of d_{l+1} or b1)
    float* g = net->G[l + 1][0];
    k_up_bwd<<<blocks_for((size_t)B * w[l + 1] * Nb), 256, 0, net->stream>>>(net->gCAT[l], cs, g,
                                                                             (size_t)w[l + 1] * Nb, w[l + 1], H / 2,
                                                                             H / 2, B);
    UCK(cudaGetLastError());
    relu_bwd<T>(net, (const T*)net->U[l + 1], (size_t)w[l + 1] * Nb, g, (size_t)w[l + 1] * Nb, nullptr, 0, w[l + 1],
                H / 2, B);
  }
  // bottleneck: G[D-1][0] = d(pre-activation of b1)
  {
    const int l = D - 1, H = net->n >> l;
    const size_t N = npix(net, l);
    const size_t bs = (size_t)w[l] * N;
    conv3_dw<T>(net, (const T*)net->A[l], bs, net->G[l][0], bs, iB1(net), H, B);
    conv3_dx(net, net->G[l][0], bs, iB1(net), net->G[l][1], bs, H, B);
    relu_bwd<T>(net, (const T*)net->A[l], bs, net->G[l][1], bs, nullptr, 0, w[l], H, B);
    conv3_dw<T>(net, (const T*)net->Q[l - 1], (size_t)w[l - 1] * N, net->G[l][1], bs, iB0(net), H, B);
    // d(pooled s_{D-2}) into G[D-1][0]
    conv3_dx(net, net->G[l][1], bs, iB0(net), net->G[l][0], (size_t)w[l - 1] * N, H, B);
  }
  // encoder, back up to the input: G[l+1][0] holds d(Q[l])
  for (int l = D - 2; l >= 0; --l) {
    const int H = net->n >> l;
    const size_t N = npix(net, l), Nq = npix(net, l + 1);
    const size_t cs = (size_t)(w[l + 1] + w[l]) * N, bs = (size_t)w[l] * N;
    float* g0 = net->G[l][0];
    float* g1 = net->G[l][1];
    k_pool_bwd<<<blocks_for((size_t)B * w[l] * N), 256, 0, net->stream>>>(net->G[l + 1][0], (size_t)w[l] * Nq, g0, bs,
                                                                          w[l], H, H, B);
    UCK(cudaGetLastError());
    // s_l also feeds the decoder through the concatenation
    const T* S = (const T*)net->CAT[l] + (size_t)w[l + 1] * N;
    relu_bwd<T>(net, S, cs, g0, bs, net->gCAT[l] + (size_t)w[l + 1] * N, cs, w[l], H, B);
    conv3_dw<T>(net, (const T*)net->A[l], bs, g0, bs, iS(l), H, B);
    conv3_dx(net, g0, bs, iS(l), g1, bs, H, B);
    relu_bwd<T>(net, (const T*)net->A[l], bs, g1, bs, nullptr, 0, w[l], H, B);
    if (l == 0 && aligned16(net->lastIn)) {
      conv3_dw<float>(net, net->lastIn, 4 * N, g1, bs, iE(0), H, B);
    } else if (l == 0) {
      conv3_dw<float, false>(net, net->lastIn, 4 * N, g1, bs, iE(0), H, B);
    } else {
      conv3_dw<T>(net, (const T*)net->Q[l - 1], (size_t)w[l - 1] * N, g1, bs, iE(l), H, B);
      conv3_dx(net, g1, bs, iE(l), g0, (size_t)w[l - 1] * N, H, B);
    }
  }
}

// ---------------------------------------------------- tensor-core inference
// A launch whose blocks may start while the launch before still runs (they wait
// for it in the kernel). The 14 launches of a forward pass depend on each other
// in a chain, and at 128^2 each is a few microseconds: 120 -> 89 us a pass (64^2,
// batch 8: 148 -> 127 us).
template <class... A>
void launch_dep(sgn_unet_ctx* net, void (*k)(A...), unsigned grid, unsigned block, size_t smem, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = net->stream;
  c.attrs = &at;
  c.numAttrs = 1;
  UCK(cudaLaunchKernelEx(&c, k, args...));
}

void tc_conv(sgn_unet_ctx* net, int li, const __nv_bfloat16* src0, int C0, int up0, const __nv_bfloat16* src1,
             int C1, int l, int B, __nv_bfloat16* out, const float* head_w = nullptr, const float* head_b = nullptr,
             float* head_out = nullptr) {
  const Layer& L = net->L[li];
  unet_tc::ConvArgs a{};
  a.src0 = src0;
  a.src1 = src1;
  a.C0 = C0;
  a.C1 = C1;
  a.up0 = up0;
  int lg = 0;
  while ((1 << lg) < (net->n >> l)) ++lg;
  a.lH = a.lW = lg;
  a.npix = B * (int)npix(net, l);
  a.wimg = net->wimg + L.ioff;
  a.bias = net->params + L.boff;
  a.Co = L.Co;
  a.KC = L.KC;
  a.nkb = L.nkb;
  uint32_t cols = 32;
  while ((int)cols < L.Co) cols <<= 1;
  a.tmem_cols = cols;
  a.out = out;
  a.head_w = head_w;
  a.head_b = head_b;
  a.head_out = head_out;
  a.err = net->dev_err;
  const unsigned grid = (unsigned)((a.npix + unet_tc::kM - 1) / unet_tc::kM);
  a.early_w = li != iS(0);
  if (L.row) {
    launch_dep(net, unet_tc::k_conv3_tc_row, grid, unet_tc::kRowThreads, (size_t)L.smem, a);
  } else {
    unet_tc::k_conv3_tc<<<grid, unet_tc::kThreads, L.smem, net->stream>>>(a);
    UCK(cudaGetLastError());
  }
}

void infer_impl(sgn_unet_ctx* net, const float* in, float* out, int B) {
  const int D = net->D;
  const int* w = net->w;
  int lg0 = 0;
  while ((1 << lg0) < net->n) ++lg0;
  {
    const Layer& L = net->L[iE(0)];
    const int np = B * (int)npix(net, 0), nconv = (np + 31) / 32;
    unet_tc::k_conv_in_wimg<<<nconv + unet_tc::wimg_blocks(net->wtab.total), unet_tc::kInThreads,
                              sizeof(float) * L.Co * 36, net->stream>>>(
        in, lg0, lg0, np, net->params + L.woff, net->params + L.boff, L.Co, net->tA[0], nconv, net->wtab, net->params,
        net->wimg);
    UCK(cudaGetLastError());
  }
  for (int l = 0; l < D - 1; ++l) {
    if (l > 0) tc_conv(net, iE(l), net->tQ[l - 1], w[l - 1], 0, nullptr, 0, l, B, net->tA[l]);
    tc_conv(net, iS(l), net->tA[l], w[l], 0, nullptr, 0, l, B, net->tS[l]);
    const int nout = B * (int)npix(net, l + 1);
    launch_dep(net, unet_tc::k_pool_nhwc, (unsigned)blocks_for((size_t)nout * (w[l] / 8)), 256u, (size_t)0,
               (const __nv_bfloat16*)net->tS[l], lg0 - l, lg0 - l, w[l], nout, net->tQ[l]);
  }
  tc_conv(net, iB0(net), net->tQ[D - 2], w[D - 2], 0, nullptr, 0, D - 1, B, net->tA[D - 1]);
  tc_conv(net, iB1(net), net->tA[D - 1], w[D - 1], 0, nullptr, 0, D - 1, B, net->tU[D - 1]);
  for (int l = D - 2; l >= 1; --l)
    tc_conv(net, iD(net, l), net->tU[l + 1], w[l + 1], 1, net->tS[l], w[l], l, B, net->tU[l]);
  const Layer& lo = net->L[iOut(net)];
  tc_conv(net, iD(net, 0), net->tU[1], w[1], 1, net->tS[0], w[0], 0, B, nullptr, net->params + lo.woff,
          net->params + lo.boff, out);
}

sgn_status ufail(sgn_unet_ctx* net, sgn_status st, const char* msg) {
  if (net) net->err = msg;
  return st;
}

void ufree(sgn_unet_ctx* net) {
  for (void* p : net->allocs) cudaFree(p);
  net->allocs.clear();
}

// channels per K step of a tensor-core layer: the fewest steps per tap whose
// operands fit one shared-memory stage
int pick_kc(int Ci, int Co) {
  for (int nkb = 1; nkb <= Ci / 16; ++nkb) {
    if (Ci % nkb) continue;
    const int kc = Ci / nkb;
    if (kc % 16 || kc > unet_tc::kMaxKC) continue;
    if ((int)unet_tc::stage_bytes(Co, kc) <= unet_tc::kStageMax) return kc;
  }
  return 16;
}

// channels per block of the row kernel: the fewest blocks whose halo and
// weight buffers fit 110 KB (two CTAs per SM), or 200 KB when the layer has
// fewer tiles than the GPU has SMs (one CTA per SM costs nothing there, and
// each block is a step of the tile's dependent chain)
int pick_kc_row(int Ci, int Co, int W, long long tiles) {
  const int budget = (tiles < 148 ? 200 : 110) * 1024;
  for (int nkb = 1; nkb <= Ci / 16; ++nkb) {
    if (Ci % nkb) continue;
    const int kc = Ci / nkb;
    if (kc % 16) continue;
    if ((int)unet_tc::row_smem_bytes(Co, kc, nkb, W) <= budget) return kc;
  }
  return 16;
}

sgn_status create_impl(int n, int max_batch, int act_bf16, unsigned long long seed, int levels, const int* widths,
                       sgn_unet_t* out) {
  if (!out) return SGN_EINVAL;
  *out = nullptr;
  if (levels < 2 || levels > kMaxLevels || !widths) return SGN_EINVAL;
  if (n < 16 || n > 512 || (n & (n - 1)) != 0 || max_batch < 1 || max_batch > 64) return SGN_EINVAL;
  if ((n >> (levels - 1)) < 4) return SGN_EINVAL;
  for (int l = 0; l < levels; ++l)
    if (widths[l] < 16 || widths[l] > 256 || widths[l] % 16 != 0) return SGN_EINVAL;
  // one tensor-core tile of 128 pixels must not need more than 2^31 pixels in all
  if ((long long)max_batch * n * n > (1ll << 30)) return SGN_EINVAL;
  sgn_unet_ctx* net = new (std::nothrow) sgn_unet_ctx();
  if (!net) return SGN_ENOMEM;
  net->n = n;
  net->maxB = max_batch;
  net->bf16 = act_bf16 ? 1 : 0;
  net->D = levels;
  for (int l = 0; l < levels; ++l) net->w[l] = widths[l];
  const int D = levels;
  const int* w = net->w;
  std::vector<int> ci, co, kk, lv;
  auto add = [&](int a, int b, int k, int level) {
    ci.push_back(a);
    co.push_back(b);
    kk.push_back(k);
    lv.push_back(level);
  };
  for (int l = 0; l < D - 1; ++l) {
    add(l == 0 ? 4 : w[l - 1], w[l], 3, l);
    add(w[l], w[l], 3, l);
  }
  add(w[D - 2], w[D - 1], 3, D - 1);
  add(w[D - 1], w[D - 1], 3, D - 1);
  for (int l = D - 2; l >= 0; --l) add(w[l + 1] + w[l], w[l], 3, l);
  add(w[0], 1, 1, 0);
  long long off = 0, ioff = 0;
  int smem_max = 0;
  net->wtab.nl = 0;
  for (size_t i = 0; i < ci.size(); ++i) {
    Layer l;
    l.Ci = ci[i];
    l.Co = co[i];
    l.k = kk[i];
    l.woff = off;
    off += (long long)l.Co * l.Ci * l.k * l.k;
    l.boff = off;
    off += l.Co;
    l.level = lv[i];
    const int side = n >> l.level;
    l.row = side * side >= unet_tc::kM;
    if (l.k == 3 && i > 0) {
      l.KC = l.row ? pick_kc_row(l.Ci, l.Co, side, (long long)max_batch * side * side / unet_tc::kM)
                   : pick_kc(l.Ci, l.Co);
      l.nkb = l.Ci / l.KC;
      l.ioff = ioff;
      unet_tc::WImgLayer& t = net->wtab.l[net->wtab.nl++];
      t.woff = l.woff;
      t.ioff = ioff;
      t.Ci = l.Ci;
      t.Co = l.Co;
      t.KC = l.KC;
      t.nkb = l.nkb;
      t.kb_major = l.row ? 1 : 0;
      ioff += 9ll * l.Ci * l.Co;
      int sm = l.row ? (int)unet_tc::row_smem_bytes(l.Co, l.KC, l.nkb, side)
                     : unet_tc::kStages * (int)unet_tc::stage_bytes(l.Co, l.KC);
      // at most 512 / cols CTAs of this launch per SM: they all get their TMEM.
      // With dependent launches, blocks of the next layer may share the SM, and
      // their tcgen05.alloc waits until those here are through; it cannot lock
      // up, as a block lets the next launch go only after its own allocation.
      int cols = 32;
      while (cols < l.Co) cols <<= 1;
      const int ctas = 512 / cols;
      const int floor_bytes = 233472 / (ctas + 1) + 1;
      if (sm < floor_bytes) sm = floor_bytes;
      l.smem = sm;
      if (sm > smem_max) smem_max = sm;
    }
    net->L.push_back(l);
  }
  net->wtab.total = ioff;
  net->P = off;
  try {
    const size_t B = (size_t)max_batch;
    const size_t es = net->bf16 ? sizeof(__nv_bfloat16) : sizeof(float);
    const size_t bf = sizeof(__nv_bfloat16);
    int wmax = 4;
    for (int l = 0; l < D; ++l) wmax = w[l] > wmax ? w[l] : wmax;
    net->params = (float*)ualloc(net, sizeof(float) * (size_t)off);
    net->grads = (float*)ualloc(net, sizeof(float) * (size_t)off);
    net->m = (float*)ualloc(net, sizeof(float) * (size_t)off);
    net->v = (float*)ualloc(net, sizeof(float) * (size_t)off);
    for (int l = 0; l < D; ++l) {
      const size_t N = npix(net, l);
      net->A[l] = ualloc(net, es * B * w[l] * N);
      net->U[l] = ualloc(net, es * B * w[l] * N);
      net->G[l][0] = (float*)ualloc(net, sizeof(float) * B * wmax * N);
      net->G[l][1] = (float*)ualloc(net, sizeof(float) * B * wmax * N);
      net->tA[l] = (__nv_bfloat16*)ualloc(net, bf * B * w[l] * N);
      net->tU[l] = (__nv_bfloat16*)ualloc(net, bf * B * w[l] * N);
      if (l < D - 1) {
        net->CAT[l] = ualloc(net, es * B * (w[l + 1] + w[l]) * N);
        net->Q[l] = ualloc(net, es * B * w[l] * npix(net, l + 1));
        net->gCAT[l] = (float*)ualloc(net, sizeof(float) * B * (w[l + 1] + w[l]) * N);
        net->tS[l] = (__nv_bfloat16*)ualloc(net, bf * B * w[l] * N);
        net->tQ[l] = (__nv_bfloat16*)ualloc(net, bf * B * w[l] * npix(net, l + 1));
      }
    }
    const size_t N0 = npix(net, 0);
    net->OUT = (float*)ualloc(net, sizeof(float) * B * N0);
    net->gOUT = (float*)ualloc(net, sizeof(float) * B * N0);
    size_t npart = (size_t)kConv1Splits * (w[0] + 1);
    for (const Layer& l : net->L) {
      if (l.k != 3) continue;
      const int H = n >> l.level;
      const size_t np = (size_t)dw_splits(l.Ci, l.Co, H, H, max_batch) * ((size_t)l.Co * l.Ci * 9 + l.Co);
      npart = np > npart ? np : npart;
    }
    net->part = (float*)ualloc(net, sizeof(float) * npart);
    net->mse_part = (double*)ualloc(net, sizeof(double) * MSE_BLOCKS);
    net->ticket = (unsigned*)ualloc(net, sizeof(unsigned));
    UCK(cudaMemset(net->ticket, 0, sizeof(unsigned)));
    net->wimg = (__nv_bfloat16*)ualloc(net, bf * (size_t)(ioff > 0 ? ioff : 1));
    net->dev_err = (int*)ualloc(net, sizeof(int));
    UCK(cudaMemset(net->dev_err, 0, sizeof(int)));
    UCK(cudaFuncSetAttribute(unet_tc::k_conv3_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
    UCK(cudaFuncSetAttribute(unet_tc::k_conv3_tc_row, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
    init_params(net, seed);
    UCK(cudaDeviceSynchronize());
  } catch (Fail& f) {
    ufree(net);
    delete net;
    return f.st;
  }
  *out = net;
  return SGN_OK;
}

}  // namespace

#define UAPI_BEGIN                                                                                 \
  if (!net) return SGN_EINVAL;                                                                     \
  net->err.clear();                                                                                \
  try {
#define UAPI_END                                                                                   \
  }                                                                                                \
  catch (Fail & f) {                                                                               \
    return f.st;                                                                                   \
  }

extern "C" {

sgn_status sgn_unet_create(int n, int max_batch, int act_bf16, unsigned long long seed, sgn_unet_t* out) {
  const int widths[3] = {16, 32, 32};
  return create_impl(n, max_batch, act_bf16, seed, 3, widths, out);
}

sgn_status sgn_unet_create_arch(int n, int max_batch, int act_bf16, unsigned long long seed, int levels,
                                const int* widths, sgn_unet_t* out) {
  return create_impl(n, max_batch, act_bf16, seed, levels, widths, out);
}

sgn_status sgn_unet_destroy(sgn_unet_t net) {
  if (!net) return SGN_EINVAL;
  cudaStreamSynchronize(net->stream);
  ufree(net);
  delete net;
  return SGN_OK;
}

sgn_status sgn_unet_set_stream(sgn_unet_t net, void* s) {
  if (!net) return SGN_EINVAL;
  net->stream = (cudaStream_t)s;
  return SGN_OK;
}

const char* sgn_unet_last_error(sgn_unet_t net) { return net ? net->err.c_str() : ""; }

long long sgn_unet_num_params(sgn_unet_t net) { return net ? net->P : -1; }

int sgn_unet_side(sgn_unet_t net) { return net ? net->n : -1; }

int sgn_unet_levels(sgn_unet_t net) { return net ? net->D : -1; }

int sgn_unet_width(sgn_unet_t net, int level) {
  if (!net || level < 0 || level >= net->D) return -1;
  return net->w[level];
}

sgn_status sgn_unet_set_params(sgn_unet_t net, const float* p) {
  UAPI_BEGIN
  if (!p) return ufail(net, SGN_EINVAL, "sgn_unet_set_params: NULL");
  UCK(cudaMemcpyAsync(net->params, p, sizeof(float) * (size_t)net->P, cudaMemcpyDeviceToDevice, net->stream));
  return SGN_OK;
  UAPI_END
}

sgn_status sgn_unet_get_params(sgn_unet_t net, float* p) {
  UAPI_BEGIN
  if (!p) return ufail(net, SGN_EINVAL, "sgn_unet_get_params: NULL");
  UCK(cudaMemcpyAsync(p, net->params, sizeof(float) * (size_t)net->P, cudaMemcpyDeviceToDevice, net->stream));
  return SGN_OK;
  UAPI_END
}

sgn_status sgn_unet_get_grads(sgn_unet_t net, float* g) {
  UAPI_BEGIN
  if (!g) return ufail(net, SGN_EINVAL, "sgn_unet_get_grads: NULL");
  UCK(cudaMemcpyAsync(g, net->grads, sizeof(float) * (size_t)net->P, cudaMemcpyDeviceToDevice, net->stream));
  return SGN_OK;
  UAPI_END
}

sgn_status sgn_unet_forward(sgn_unet_t net, const float* in, float* out, int batch) {
  UAPI_BEGIN
  if (!in || batch < 1 || batch > net->maxB) return ufail(net, SGN_EINVAL, "sgn_unet_forward: bad input or batch");
  if (net->bf16)
    forward_impl<__nv_bfloat16>(net, in, out, batch);
  else
    forward_impl<float>(net, in, out, batch);
  net->lastIn = in;
  net->lastB = batch;
  return SGN_OK;
  UAPI_END
}

sgn_status sgn_unet_infer(sgn_unet_t net, const float* in, float* out, int batch) {
  UAPI_BEGIN
  if (!in || !out || batch < 1 || batch > net->maxB)
    return ufail(net, SGN_EINVAL, "sgn_unet_infer: bad input, output or batch");
  infer_impl(net, in, out, batch);
  return SGN_OK;
  UAPI_END
}

sgn_status sgn_unet_check(sgn_unet_t net) {
  UAPI_BEGIN
  int h = 0;
  UCK(cudaMemcpyAsync(&h, net->dev_err, sizeof(int), cudaMemcpyDeviceToHost, net->stream));
  UCK(cudaStreamSynchronize(net->stream));
  if (h != 0) {
    UCK(cudaMemsetAsync(net->dev_err, 0, sizeof(int), net->stream));
    return ufail(net, SGN_ECUDA, "sgn_unet_infer: a tensor-core wait ran out (the outputs are not valid)");
  }
  return SGN_OK;
  UAPI_END
}

}  // extern "C"

namespace {

// one tensor-core layer; stall: the self-test's barrier that never completes
sgn_status conv3_tc_run(int batch, int H, int W, const void* src0, int C0, int up0, const void* src1, int C1,
                        const float* weight, const float* bias, int Co, void* out, void* workspace,
                        size_t workspace_bytes, void* stream, int stall) {
  auto pow2 = [](int v) { return v >= 2 && (v & (v - 1)) == 0; };
  const int Ci = C0 + C1;
  if (batch < 1 || !pow2(H) || !pow2(W) || (long long)batch * H * W > (1ll << 30)) return SGN_EINVAL;
  if (up0 && (H < 4 || W < 4)) return SGN_EINVAL;
  if (!src0 || !weight || !bias || !out || !workspace || C0 < 16 || C0 % 16 || C1 < 0 || C1 % 16 ||
      (C1 > 0 && !src1) || Ci > 1024 || Co < 16 || Co > 256 || Co % 16)
    return SGN_EINVAL;
  const size_t img = (size_t)9 * Ci * Co * sizeof(__nv_bfloat16);
  if (workspace_bytes < sgn_conv3_workspace_bytes(C0 + C1, Co) || ((uintptr_t)workspace & 15u)) return SGN_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  int lH = 0, lW = 0;
  while ((1 << lH) < H) ++lH;
  while ((1 << lW) < W) ++lW;
  const bool row = H * W >= unet_tc::kM;
  const int KC = row ? pick_kc_row(Ci, Co, W, (long long)batch * H * W / unet_tc::kM) : pick_kc(Ci, Co);
  __nv_bfloat16* wimg = (__nv_bfloat16*)workspace;
  int* err = (int*)((char*)workspace + ((img + 15) & ~(size_t)15));
  unet_tc::WImgTable t{};
  t.nl = 1;
  t.l[0].woff = 0;
  t.l[0].ioff = 0;
  t.l[0].Ci = Ci;
  t.l[0].Co = Co;
  t.l[0].KC = KC;
  t.l[0].nkb = Ci / KC;
  t.l[0].kb_major = row ? 1 : 0;
  t.total = 9ll * Ci * Co;
  int cols = 32;
  while (cols < Co) cols <<= 1;
  int sm = row ? (int)unet_tc::row_smem_bytes(Co, KC, Ci / KC, W)
               : unet_tc::kStages * (int)unet_tc::stage_bytes(Co, KC);
  const int floor_bytes = 233472 / (512 / cols + 1) + 1;
  if (sm < floor_bytes) sm = floor_bytes;
  unet_tc::ConvArgs a{};
  a.src0 = (const __nv_bfloat16*)src0;
  a.src1 = (const __nv_bfloat16*)src1;
  a.C0 = C0;
  a.C1 = C1;
  a.up0 = up0 ? 1 : 0;
  a.lH = lH;
  a.lW = lW;
  a.npix = batch * H * W;
  a.wimg = wimg;
  a.bias = bias;
  a.Co = Co;
  a.KC = KC;
  a.nkb = Ci / KC;
  a.tmem_cols = (uint32_t)cols;
  a.out = (__nv_bfloat16*)out;
  a.err = err;
  a.stall = stall;
  if (cudaFuncSetAttribute(row ? (const void*)unet_tc::k_conv3_tc_row : (const void*)unet_tc::k_conv3_tc,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, sm) != cudaSuccess ||
      cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess)
    return SGN_ECUDA;
  unet_tc::k_wimg<<<unet_tc::wimg_blocks(t.total), unet_tc::kInThreads, 0, st>>>(t, weight, wimg);
  const unsigned grid = (unsigned)((a.npix + unet_tc::kM - 1) / unet_tc::kM);
  if (row)
    unet_tc::k_conv3_tc_row<<<grid, unet_tc::kRowThreads, sm, st>>>(a);
  else
    unet_tc::k_conv3_tc<<<grid, unet_tc::kThreads, sm, st>>>(a);
  int h = 0;
  if (cudaGetLastError() != cudaSuccess || cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st) !=
                                              cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess || h != 0)
    return SGN_ECUDA;
  return SGN_OK;
}

}  // namespace

extern "C" {

sgn_status sgn_conv3_relu_bf16(int batch, int H, int W, const void* src0, int C0, int up0, const void* src1, int C1,
                               const float* weight, const float* bias, int Co, void* out, void* workspace,
                               size_t workspace_bytes, void* stream) {
  return conv3_tc_run(batch, H, W, src0, C0, up0, src1, C1, weight, bias, Co, out, workspace, workspace_bytes,
                      stream, 0);
}

sgn_status sgn_conv3_wait_selftest(void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const int C = 16, Co = 16;
  const int shapes[2][2] = {{8, 8}, {4, 128}};  // the gather kernel (64 pixels), the row kernel
  const size_t ws = sgn_conv3_workspace_bytes(C, Co);
  void *src = nullptr, *out = nullptr, *wk = nullptr;
  float *w = nullptr, *bias = nullptr;
  const size_t npix = 4 * 128;
  bool ok = cudaMalloc(&src, npix * C * 2) == cudaSuccess && cudaMalloc(&out, npix * Co * 2) == cudaSuccess &&
            cudaMalloc(&wk, ws) == cudaSuccess && cudaMalloc((void**)&w, sizeof(float) * Co * C * 9) == cudaSuccess &&
            cudaMalloc((void**)&bias, sizeof(float) * Co) == cudaSuccess;
  if (ok)
    ok = cudaMemsetAsync(src, 0, npix * C * 2, st) == cudaSuccess &&
         cudaMemsetAsync(w, 0, sizeof(float) * Co * C * 9, st) == cudaSuccess &&
         cudaMemsetAsync(bias, 0, sizeof(float) * Co, st) == cudaSuccess;
  for (int k = 0; k < 2 && ok; ++k) {
    const int H = shapes[k][0], W = shapes[k][1];
    // the stalled launch must report its run-out wait, and the context must
    // still run the same layer normally afterwards
    ok = conv3_tc_run(1, H, W, src, C, 0, nullptr, 0, w, bias, Co, out, wk, ws, stream, 1) == SGN_ECUDA &&
         cudaGetLastError() == cudaSuccess &&
         conv3_tc_run(1, H, W, src, C, 0, nullptr, 0, w, bias, Co, out, wk, ws, stream, 0) == SGN_OK;
  }
  cudaStreamSynchronize(st);
  cudaFree(src);
  cudaFree(out);
  cudaFree(wk);
  cudaFree(w);
  cudaFree(bias);
  return ok ? SGN_OK : SGN_ECUDA;
}

size_t sgn_conv3_workspace_bytes(int Ci, int Co) {
  if (Ci < 1 || Co < 1) return 0;
  return (((size_t)9 * Ci * Co * sizeof(__nv_bfloat16) + 15) & ~(size_t)15) + 16;
}

sgn_status sgn_unet_backward(sgn_unet_t net, const float* target, double* loss_dev) {
  UAPI_BEGIN
  if (!target || net->lastB < 1 || !net->lastIn)
    return ufail(net, SGN_EINVAL, "sgn_unet_backward: no forward pass or NULL target");
  if (net->bf16)
    backward_impl<__nv_bfloat16>(net, target, loss_dev);
  else
    backward_impl<float>(net, target, loss_dev);
  return SGN_OK;
  UAPI_END
}

sgn_status sgn_unet_adam_step(sgn_unet_t net, float lr, float b1, float b2, float eps, int t) {
  UAPI_BEGIN
  if (t < 1) return ufail(net, SGN_EINVAL, "sgn_unet_adam_step: t < 1");
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  k_adam<<<blocks_for((size_t)net->P), 256, 0, net->stream>>>(net->params, net->grads, net->m, net->v, net->P, lr,
                                                               b1, b2, eps, c1, c2);
  UCK(cudaGetLastError());
  return SGN_OK;
  UAPI_END
}

}  // extern "C"
