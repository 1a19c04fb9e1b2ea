// sgn_unet_tc.cuh - the U-Net's BF16 inference forward on the 5th-generation
// tensor cores (tcgen05), as implicit GEMMs over NHWC activations.
//
// A periodic 3x3 convolution of an NHWC tensor is, per output tile of 128
// pixels, the GEMM D[128][Co] = sum over the nine taps t of
// A_t[128][Ci] B_t[Ci][Co], where row m of A_t holds the Ci channels of the
// input pixel at (y + ty - 1, x + tx - 1) (wrapped) and B_t the weights of tap
// t. One CTA of 128 threads (256 in the row kernel, which stages its input once
// per channel block, below) computes one tile:
//   * the accumulator D lives in tensor memory (TMEM lane m = pixel m, one
//     32-bit column per output channel), allocated by warp 0;
//   * the K loop runs over (tap, channel block) steps through three
//     shared-memory stages: the weights of a step arrive by one bulk copy
//     (cp.async.bulk, the copy engine) from a pre-arranged BF16 image, issued
//     one step ahead; the 128 gathered input rows are written by the threads
//     themselves (each thread one pixel, its loads issued one step ahead;
//     wrap-around, nearest upsampling and the channel concatenation of the
//     decoder are folded into this gather);
//   * one thread issues the step's tcgen05.mma instructions (M = 128,
//     N = Co, K = 16 each) and commits them to the stage's mbarrier, which
//     frees the stage for the step three later;
//   * the epilogue reads D back with tcgen05.ld (each warp its 32 lanes),
//     adds the bias, applies the ReLU, rounds to BF16 and stores the NHWC row;
//     for the last layer it also applies the 1x1 output convolution.
// Operands are K-major without swizzling: 8 x 16-byte core matrices, the
// core matrices of one 8-row group along K LBO bytes apart and consecutive
// 8-row groups SBO bytes apart.
//
// Every wait is bounded: a wait that runs out records SGN_TC_WAIT in the
// error word, the CTA waits (bounded again) for what it still has in flight,
// frees its TMEM and returns.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace unet_tc {

constexpr int kM = 128;           // output pixels per CTA = TMEM lanes
constexpr int kThreads = 128;     // the step kernel: one thread per pixel row
constexpr int kRowThreads = 256;  // the row kernel: two threads per pixel row, each half the columns
constexpr int kStageMax = 56 * 1024;
constexpr int kMaxKC = 128;       // channels per K step at most (the gather's registers)
constexpr int kStages = 3;        // shared-memory stages of the K loop
constexpr int SGN_TC_WAIT = 1;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// tcgen05 shared-memory matrix descriptor, no swizzle: start address, the
// leading (K-direction) and stride (M/N-direction) byte offsets, all in
// 16-byte units, and the descriptor version 1 at bits 46-48.
__host__ __device__ constexpr uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16
// A and B (bits 7-9 and 10-12 = 1), both K-major, N / 8 at bits 17-22,
// M / 16 at bits 24-28.
__host__ __device__ constexpr uint32_t instr_desc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void bar_init(uint64_t* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ bool bar_try(uint64_t* b, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
// about a second at most: try_wait suspends the thread between polls
__device__ __forceinline__ bool bar_wait(uint64_t* b, unsigned parity) {
  for (int it = 0; it < (1 << 20); ++it)
    if (bar_try(b, parity)) return true;
  return false;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, uint64_t* b,
                                         unsigned extra_tx = 0) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(b)), "r"(bytes + extra_tx)
               : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(b))
               : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(dst)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void mma_bf16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         int accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* b) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_addr(b))
               : "memory");
}
// Programmatic dependent launch: what the launch before wrote is visible after
// dep_wait, and dep_go lets the next launch's blocks start their preparation.
// Each block waits before it goes on, so a launch starts only when the one two
// before it is complete. Without the launch attribute both do nothing.
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void dep_go() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
// 16 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// One convolution launch. The input channels are the concatenation of src0
// (C0 channels, read at (y >> 1, x >> 1) of an H/2 x W/2 grid when up0) and
// src1 (C1 channels, may be 0), both NHWC BF16 with their channel counts as
// row lengths.
struct ConvArgs {
  const __nv_bfloat16* src0;
  const __nv_bfloat16* src1;
  int C0, C1, up0;
  int lH, lW;   // log2 of the output grid (= src1's grid)
  int npix;     // B H W output pixels
  const __nv_bfloat16* wimg;  // [9 * nkb][KC / 8][Co / 8][8][8] BF16 (core-matrix image of each step)
  const float* bias;          // [Co]
  int Co, KC, nkb;
  uint32_t tmem_cols;         // power of two >= max(32, Co)
  __nv_bfloat16* out;         // NHWC [npix][Co], or null with a head
  const float* head_w;        // optional 1x1 head Co -> 1: weights [Co], bias [1]
  const float* head_b;
  float* head_out;            // [npix] FP32
  int* err;
  int early_w;                // the weight image is complete two launches before this one
  int stall;                  // self-test only: arm step 0's weight barrier for 16 bytes more
                              // than its copy delivers, so that its waits run out
};

// bytes of one K step's operands in shared memory (A rows, then B)
__host__ __device__ constexpr uint32_t a_bytes(int KC) { return (uint32_t)kM * KC * 2u; }
__host__ __device__ constexpr uint32_t b_bytes(int Co, int KC) { return (uint32_t)Co * KC * 2u; }
__host__ __device__ constexpr uint32_t stage_bytes(int Co, int KC) { return a_bytes(KC) + b_bytes(Co, KC); }

// Bias and head weights of a layer, staged in shared memory while the first
// operands are on their way: read in the epilogue they were a chain of loads
// from L2, 1200 to 3500 cycles of a tile's 9 to 30 thousand.
struct __align__(16) Consts {
  float bias[256], head[256];
};
__device__ __forceinline__ void load_consts(const ConvArgs& p, Consts& k, int tid, int nt) {
  for (int i = tid; i < p.Co; i += nt) {
    k.bias[i] = __ldg(p.bias + i);
    if (p.head_w) k.head[i] = __ldg(p.head_w + i);
  }
}

// The epilogue of both kernels, after the last MMA completed: this thread's
// TMEM lane (its pixel) read back 16 columns at a time, bias, ReLU, BF16
// store of the NHWC row; with a head, the 1x1 output convolution of the BF16
// values in FP32. A warp reads the 32 lanes of its index modulo 4; of nw > 4
// warps, those of one lane quarter share its columns in turn - not with a
// head, whose sum over the columns stays one chain of one thread. Every thread
// of the CTA calls it (tcgen05.ld is warp-wide); valid: whether the pixel
// exists (a ragged last tile).
__device__ __forceinline__ void tc_epilogue(const ConvArgs& p, const Consts& k, uint32_t tmem, int warp, int nw,
                                            int pix, bool valid) {
  tc_fence_after();
  const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const int step = p.head_w ? 1 : nw >> 2;
  if (p.head_w && warp >= 4) return;
  float head = 0.f;
  for (int q = warp >> 2; q < p.Co / 16; q += step) {
    float v[16];
    tmem_ld16(lane_addr + (uint32_t)(q * 16), v);
    __align__(16) __nv_bfloat16 o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float a = fmaxf(v[i] + k.bias[q * 16 + i], 0.f);
      o[i] = __float2bfloat16_rn(a);
      if (p.head_w) head = fmaf(k.head[q * 16 + i], __bfloat162float(o[i]), head);
    }
    if (valid && p.out) {
      uint4* dst = reinterpret_cast<uint4*>(p.out + (size_t)pix * p.Co + q * 16);
      dst[0] = reinterpret_cast<const uint4*>(o)[0];
      dst[1] = reinterpret_cast<const uint4*>(o)[1];
    }
  }
  if (valid && p.head_w) p.head_out[pix] = head + __ldg(p.head_b);
}

__global__ void __launch_bounds__(kThreads) k_conv3_tc(ConvArgs p) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t bar_w[kStages], bar_mma[kStages];
  __shared__ uint32_t tmem_slot;
  __shared__ Consts consts;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int KC = p.KC, Co = p.Co;
  const uint32_t abytes = a_bytes(KC), sbytes = stage_bytes(Co, KC);
  const uint32_t sm0 = smem_addr(sm);

  if (warp == 0) tmem_alloc(&tmem_slot, p.tmem_cols);
  if (tid == 32) {
    for (int i = 0; i < kStages; ++i) {
      bar_init(&bar_w[i], 1);
      bar_init(&bar_mma[i], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  // this thread's pixel: row m = tid of the tile
  const int pix = blockIdx.x * kM + tid;
  const bool valid = pix < p.npix;
  const int W = 1 << p.lW, H = 1 << p.lH;
  const int x = pix & (W - 1), y = (pix >> p.lW) & (H - 1), b = pix >> (p.lW + p.lH);
  const uint32_t idesc = instr_desc_bf16(kM, Co);
  const int nsteps = 9 * p.nkb;

  // this thread's gathered row of one K step: KC / 8 16-byte chunks, loaded
  // one step ahead so that the loads of step s + 1 are in flight while the
  // MMAs of step s are issued and the next buffer is waited for
  uint4 row[kMaxKC / 8];
  auto gather = [&](int step) {
    const int tap = step / p.nkb, kb = step - tap * p.nkb;
    const int yy = (y + tap / 3 - 1) & (H - 1), xx = (x + tap % 3 - 1) & (W - 1);
    const uint4* r0 = reinterpret_cast<const uint4*>(
        p.up0 ? p.src0 + ((((size_t)b << (p.lH + p.lW - 2)) + ((size_t)(yy >> 1) << (p.lW - 1)) + (xx >> 1)) * p.C0)
              : p.src0 + ((((size_t)b << (p.lH + p.lW)) + ((size_t)yy << p.lW) + xx) * p.C0));
    const uint4* r1 = p.src1 ? reinterpret_cast<const uint4*>(
                                   p.src1 + ((((size_t)b << (p.lH + p.lW)) + ((size_t)yy << p.lW) + xx) * p.C1))
                             : r0;
#pragma unroll
    for (int c = 0; c < kMaxKC / 8; ++c) {
      const int ch = kb * KC + 8 * c;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (valid && c < KC / 8) v = ch < p.C0 ? __ldg(r0 + (ch >> 3)) : __ldg(r1 + ((ch - p.C0) >> 3));
      row[c] = v;
    }
  };

  bool ok = true;
  int issued = -1;     // last step whose MMAs were committed (thread 0)
  int copied = -1;     // last step whose weight copy was issued (thread 0)
  int copy_done = -1;  // last step whose weight copy was seen complete (thread 0)
  // step s uses stage s % kStages; its k-th use is phase k of the stage's barriers
  auto stage_of = [](int st) { return st % kStages; };
  auto parity_of = [](int st) { return (unsigned)((st / kStages) & 1); };
  if (tid == 0) {
    bulk_g2s(sm + abytes, p.wimg, b_bytes(Co, KC), &bar_w[0], p.stall ? 16u : 0u);
    copied = 0;
  }
  gather(0);
  load_consts(p, consts, tid, kThreads);
  for (int s = 0; s < nsteps; ++s) {
    const int buf = stage_of(s);
    // the MMAs of step s - 2 (and so of every earlier step) are done: stage
    // (s + 1) % 3 - last used by step s - 2 - takes step s + 1's weights,
    // stage s % 3 - last used by step s - 3 - step s's rows
    if (s >= 2 && !bar_wait(&bar_mma[stage_of(s - 2)], parity_of(s - 2))) ok = false;
    if (__syncthreads_or(ok ? 0 : 1)) {
      ok = false;
      break;
    }
    unsigned char* A = sm + buf * sbytes;
    if (tid == 0 && s + 1 < nsteps) {
      bulk_g2s(sm + stage_of(s + 1) * sbytes + abytes, p.wimg + (size_t)(s + 1) * Co * KC, b_bytes(Co, KC),
               &bar_w[stage_of(s + 1)]);
      copied = s + 1;
    }
    // A row m = the KC channels [kb KC, (kb + 1) KC) of the tap's pixel
    unsigned char* arow = A + (tid >> 3) * 128 + (tid & 7) * 16;
#pragma unroll
    for (int c = 0; c < kMaxKC / 8; ++c)
      if (c < KC / 8) *reinterpret_cast<uint4*>(arow + (size_t)c * (kM / 8) * 128) = row[c];
    if (s + 1 < nsteps) gather(s + 1);
    fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      if (!bar_wait(&bar_w[buf], parity_of(s))) {
        ok = false;
      } else {
        copy_done = s;
        tc_fence_after();
        const uint32_t a0 = sm0 + buf * sbytes, b0 = a0 + abytes;
#pragma unroll 1
        for (int j = 0; j < KC / 16; ++j) {
          const uint64_t ad = smem_desc(a0 + (uint32_t)j * 2u * (kM / 8) * 128u, (kM / 8) * 128u, 128u);
          const uint64_t bd = smem_desc(b0 + (uint32_t)j * 2u * (uint32_t)(Co / 8) * 128u, (uint32_t)(Co / 8) * 128u,
                                        128u);
          mma_bf16(tmem, ad, bd, idesc, (s > 0 || j > 0) ? 1 : 0);
        }
        mma_commit(&bar_mma[buf]);
        issued = s;
      }
    }
  }
  if (ok) {
    const int last = nsteps - 1;
    if (!bar_wait(&bar_mma[stage_of(last)], parity_of(last))) ok = false;
  }
  ok = __syncthreads_and(ok ? 1 : 0) != 0;
  if (ok) {
    tc_epilogue(p, consts, tmem, warp, kThreads / 32, pix, valid);
  } else if (tid == 0) {
    atomicOr(p.err, SGN_TC_WAIT);
    // let what this CTA still has in flight finish before its memory goes
    if (issued >= 0) bar_wait(&bar_mma[stage_of(issued)], parity_of(issued));
    for (int c = copy_done + 1; c <= copied; ++c) bar_wait(&bar_w[stage_of(c)], parity_of(c));
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, p.tmem_cols);
}

}  // namespace unet_tc

namespace unet_tc {

constexpr int kInThreads = 128;

// 2x2 average pool of an NHWC BF16 tensor on a 2^lH x 2^lW grid (C channels,
// a multiple of 8): one thread per output pixel and 8-channel group, summed in
// FP32 as (a + b) + (c + d) over the rows 2y, 2y + 1.
__global__ void k_pool_nhwc(const __nv_bfloat16* in, int lH, int lW, int C, int nout,
                            __nv_bfloat16* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int groups = C >> 3;
  dep_wait();
  dep_go();
  if (i >= nout * groups) return;
  const int g = i % groups, op = i / groups;
  const int W2 = 1 << (lW - 1), H2 = 1 << (lH - 1);
  const int ox = op & (W2 - 1), oy = (op >> (lW - 1)) & (H2 - 1), b = op >> (lH + lW - 2);
  const size_t base = ((((size_t)b << (lH + lW)) + ((size_t)(2 * oy) << lW) + 2 * ox) * C) + g * 8;
  const size_t row = (size_t)C << lW;
  __align__(16) __nv_bfloat16 v[4][8];
  *reinterpret_cast<uint4*>(v[0]) = *reinterpret_cast<const uint4*>(in + base);
  *reinterpret_cast<uint4*>(v[1]) = *reinterpret_cast<const uint4*>(in + base + C);
  *reinterpret_cast<uint4*>(v[2]) = *reinterpret_cast<const uint4*>(in + base + row);
  *reinterpret_cast<uint4*>(v[3]) = *reinterpret_cast<const uint4*>(in + base + row + C);
  __align__(16) __nv_bfloat16 o[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float s = (__bfloat162float(v[0][j]) + __bfloat162float(v[1][j])) +
                    (__bfloat162float(v[2][j]) + __bfloat162float(v[3][j]));
    o[j] = __float2bfloat16_rn(0.25f * s);
  }
  *reinterpret_cast<uint4*>(out + (size_t)op * C + g * 8) = *reinterpret_cast<const uint4*>(o);
}

// BF16 core-matrix images of the 3x3 layers' FP32 weights [Co][Ci][3][3]:
// for step s = tap nkb + kb (kb 9 + tap with kb_major), element (co, k)
// (input channel kb KC + k) at s Co KC + ((k / 8) (Co / 8) + co / 8) 64 +
// (co % 8) 8 + k % 8.
constexpr int kMaxImgLayers = 16;
struct WImgLayer {
  long long woff, ioff;  // FP32 weight offset in the parameters, element offset in the image
  int Ci, Co, KC, nkb;
  int kb_major;          // step order kb 9 + tap (the row kernel) instead of tap nkb + kb
};
struct WImgTable {
  int nl;
  WImgLayer l[kMaxImgLayers];
  long long total;
};

// One thread per 8 input channels of one (co, tap), the taps of neighbouring
// threads: the loads of nine threads are consecutive, and each stores 16 bytes.
__device__ __forceinline__ void wimg_body(const WImgTable& t, int blk, const float* __restrict__ params,
                                          __nv_bfloat16* img) {
  const int i = (blk * kInThreads + (int)threadIdx.x) * 8;
  if (i >= (int)t.total) return;
  int li = 0;
  while (li + 1 < t.nl && i >= (int)t.l[li + 1].ioff) ++li;
  const WImgLayer L = t.l[li];
  const int r = (i - (int)L.ioff) >> 3, tap = r % 9, cc = r / 9, g8 = L.Ci >> 3;
  const int co = cc / g8, g = cc - co * g8;
  const float* w = params + L.woff + ((long long)co * L.Ci + g * 8) * 9 + tap;
  float v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = __ldg(w + k * 9);
  const int c8 = L.KC >> 3, kb = g / c8, c = g - kb * c8;
  const int step = L.kb_major ? kb * 9 + tap : tap * L.nkb + kb;
  __align__(16) __nv_bfloat16 o[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) o[k] = __float2bfloat16_rn(v[k]);
  *reinterpret_cast<uint4*>(img + L.ioff + (long long)step * L.Co * L.KC + (c * (L.Co >> 3) + (co >> 3)) * 64 +
                            (co & 7) * 8) = *reinterpret_cast<const uint4*>(o);
}
__host__ __device__ constexpr int wimg_blocks(long long total) {
  return (int)((total / 8 + kInThreads - 1) / kInThreads);
}

__global__ void __launch_bounds__(kInThreads) k_wimg(WImgTable t, const float* __restrict__ params,
                                                     __nv_bfloat16* img) {
  wimg_body(t, blockIdx.x, params, img);
}

// The first layer (4 FP32 NCHW input channels -> Co, ReLU) on CUDA cores: its
// K = 36 is too short for the tensor cores. A warp computes 32 pixels of 8
// output channels at a time, one pixel a thread; weights [Co][4][3][3] in
// shared memory, read as vectors of four that the warp shares, and eight
// independent sums a thread.
__device__ __forceinline__ void conv_in_body(float4* ws, int blk, const float* __restrict__ x, int lH, int lW,
                                             int npix, const float* __restrict__ w, const float* __restrict__ bias,
                                             int Co, __nv_bfloat16* out) {
  float* wf = reinterpret_cast<float*>(ws);
  for (int i = threadIdx.x; i < Co * 36; i += kInThreads) wf[i] = __ldg(w + i);
  const int pix = blk * 32 + (threadIdx.x & 31);
  const int pq = pix < npix ? pix : npix - 1;
  const int W = 1 << lW, H = 1 << lH;
  const int xq = pq & (W - 1), yq = (pq >> lW) & (H - 1), b = pq >> (lH + lW);
  float in[36];
#pragma unroll
  for (int ci = 0; ci < 4; ++ci)
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const int yy = (yq + t / 3 - 1) & (H - 1), xx = (xq + t % 3 - 1) & (W - 1);
      in[ci * 9 + t] = __ldg(x + (((size_t)(b * 4 + ci)) << (lH + lW)) + ((size_t)yy << lW) + xx);
    }
  __syncthreads();
  for (int c8 = threadIdx.x >> 5; c8 < Co / 8; c8 += kInThreads / 32) {
    float acc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 v = ws[(c8 * 8 + j) * 9 + k];
        acc[j] = fmaf(v.x, in[4 * k], acc[j]);
        acc[j] = fmaf(v.y, in[4 * k + 1], acc[j]);
        acc[j] = fmaf(v.z, in[4 * k + 2], acc[j]);
        acc[j] = fmaf(v.w, in[4 * k + 3], acc[j]);
      }
    __align__(16) __nv_bfloat16 o[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) o[j] = __float2bfloat16_rn(fmaxf(acc[j] + __ldg(bias + c8 * 8 + j), 0.f));
    if (pix < npix) *reinterpret_cast<uint4*>(out + (size_t)pix * Co + c8 * 8) = *reinterpret_cast<const uint4*>(o);
  }
}

// The first launch of a forward pass: the first layer by the blocks below
// nconv, the weight images of the other layers, which it does not need, by the
// rest. Both are short and latency-bound, 8.5 and 5.7 us as two launches (one
// thread per pixel and all channels, one per image element) at 128^2.
__global__ void __launch_bounds__(kInThreads) k_conv_in_wimg(const float* __restrict__ x, int lH, int lW, int npix,
                                                             const float* __restrict__ w,
                                                             const float* __restrict__ bias, int Co,
                                                             __nv_bfloat16* out, int nconv, WImgTable t,
                                                             const float* __restrict__ params, __nv_bfloat16* img) {
  extern __shared__ float4 ws[];  // Co * 9
  dep_go();
  if ((int)blockIdx.x < nconv)
    conv_in_body(ws, blockIdx.x, x, lH, lW, npix, w, bias, Co, out);
  else
    wimg_body(t, blockIdx.x - nconv, params, img);
}

}  // namespace unet_tc

namespace unet_tc {

// Grids whose rows hold at least 128 pixels: a tile is 128 consecutive pixels
// of one row, and the input it needs - rows y-1..y+1, columns x0-1..x0+128
// (wrapped) - is staged once per channel block into shared memory as a halo
// [KC/8 chunks][3 x 130 positions][8 channels]. The A operand of tap (dy, dx)
// is then that buffer itself: its 128 rows are the 128 consecutive positions
// from (dy + 1) 130 + dx + 1 on, 16 bytes apart, i.e. a descriptor with
// SBO = 128 and LBO = the chunk stride, started at that offset. The nine
// taps' weights of a channel block arrive by one bulk copy (the image is in
// channel-block-major order for these layers); halo and weights are
// double-buffered across channel blocks, the next block's loaded while the
// current block's MMAs run, and one thread issues a block's 9 KC/16 MMAs back
// to back with one commit.
//
// Rows of fewer than 128 pixels (W < 128, at least 128 pixels per image): a
// tile is the 128 / W whole rows y0.. of one image, and the halo holds three
// copies of rows y0-1 .. y0+128/W, copy kx shifted by kx - 1 columns (wrapped)
// and stored with row stride exactly W. Output pixel m of the tile then reads
// tap (ky, kx) at position m + ky W of copy kx: again 128 consecutive 16-byte
// positions, one descriptor per tap.
//
// At batch 1 a layer has 2 to 128 tiles, and a tile is one serial chain: halo
// copies, MMA issue, epilogue. At 128^2 (471,873 parameters) a channel block of
// 32 copies its halo in 2400 to 3400 cycles (38 per warp copy of 512 bytes, the
// rate of these copies), is issued in 1050 to 1130, and the epilogue takes 700
// to 1900. Kept: 256 threads, division-free copies, unrolled issue, staged
// constants, dependent launches: 201 -> 85 us a pass, 2.10 -> 1.46 ms at 256^2
// and batch 32. Tensor pipe 9 to 15% active on the large grids.
constexpr int kHaloPos = 3 * (kM + 2);
// positions per chunk of one halo copy, and the copies
__host__ __device__ constexpr int halo_pos(int W) { return W >= kM ? kHaloPos : kM + 2 * W; }
__host__ __device__ constexpr int halo_copies(int W) { return W >= kM ? 1 : 3; }
// positions from one chunk of a copy to the next: as many as put the chunks
// that eight lanes write together (load_block) into different banks, 2 modulo
// 8 for four chunks of two pixels, 4 modulo 8 for two chunks of four
__host__ __device__ constexpr int halo_stride(int KC, int W) {
  return (halo_pos(W) & ~7) + (KC % 32 ? 4 : 2) + ((halo_pos(W) & 7) > (KC % 32 ? 4 : 2) ? 8 : 0);
}
__host__ __device__ constexpr uint32_t halo_bytes(int KC, int W) {
  return (uint32_t)halo_copies(W) * halo_stride(KC, W) * KC * 2u;
}
// one buffer of halo + weights per channel block in flight (two when there
// are several blocks)
__host__ __device__ constexpr uint32_t row_smem_bytes(int Co, int KC, int nkb, int W) {
  return (nkb > 1 ? 2u : 1u) * (halo_bytes(KC, W) + 9u * b_bytes(Co, KC));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
  return e != 0;
}
// The MMAs of one channel block: tap (ky, kx), K step j read A at
// kx kx' + ky ky' + j aj and B at (tap KC/16 + j) bj from the block's first
// descriptors, in units of 16 bytes (the address is a descriptor's low field
// and stays below its 14 bits, so an offset is one addition).
struct TapSteps {
  uint64_t a, b;
  uint32_t kx, ky, aj, bj;
};
template <int NJ>
__device__ __forceinline__ void issue_taps(uint32_t tmem, const TapSteps& t, uint32_t idesc, int nj, bool acc) {
  const int n = NJ ? NJ : nj;
#pragma unroll
  for (int tap = 0; tap < 9; ++tap) {
    uint64_t a = t.a + (uint32_t)((tap % 3) * t.kx + (tap / 3) * t.ky), b = t.b + (uint32_t)(tap * n) * t.bj;
#pragma unroll
    for (int j = 0; j < n; ++j) {
      mma_bf16(tmem, a, b, idesc, (tap > 0 || j > 0 || acc) ? 1 : 0);
      a += t.aj;
      b += t.bj;
    }
  }
}
// Unrolled for the usual channel counts: with loops over the taps and steps,
// the one issuing thread needed 98 cycles an MMA and 195 a tap, more than the
// tensor core.
__device__ __forceinline__ void issue_block(uint32_t tmem, const TapSteps& t, uint32_t idesc, int nj, bool acc) {
  switch (nj) {
    case 1: return issue_taps<1>(tmem, t, idesc, nj, acc);
    case 2: return issue_taps<2>(tmem, t, idesc, nj, acc);
    case 3: return issue_taps<3>(tmem, t, idesc, nj, acc);
    case 4: return issue_taps<4>(tmem, t, idesc, nj, acc);
    case 6: return issue_taps<6>(tmem, t, idesc, nj, acc);
    default: return issue_taps<0>(tmem, t, idesc, nj, acc);
  }
}

__global__ void __launch_bounds__(kRowThreads) k_conv3_tc_row(ConvArgs p) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t bar_w[2], bar_mma[2];
  __shared__ uint32_t tmem_slot;
  __shared__ Consts consts;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
  const int KC = p.KC, Co = p.Co, nkb = p.nkb;
  const int W = 1 << p.lW, H = 1 << p.lH;
  const bool wide = W >= kM;
  const int P = halo_stride(KC, W);  // positions between the chunks of a halo copy
  const uint32_t hbytes = halo_bytes(KC, W), wbytes = 9u * b_bytes(Co, KC), bufbytes = hbytes + wbytes;
  const uint32_t sm0 = smem_addr(sm);

  if (warp == 0) tmem_alloc(&tmem_slot, p.tmem_cols);
  if (tid == 32) {
    for (int i = 0; i < 2; ++i) {
      bar_init(&bar_w[i], 1);
      bar_init(&bar_mma[i], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  const int tile = blockIdx.x;
  int x0, y, b;  // wide: the tile's row y and first column x0; narrow: its first row y
  if (wide) {
    const int tiles_row = W >> 7;
    x0 = (tile % tiles_row) << 7;
    y = (tile / tiles_row) & (H - 1);
    b = tile / (tiles_row << p.lH);
  } else {
    const int rows = kM >> p.lW, tiles_img = H / rows;
    x0 = 0;
    y = (tile % tiles_img) * rows;
    b = tile / tiles_img;
  }
  const int pix = tile * kM + (tid & (kM - 1));
  const uint32_t idesc = instr_desc_bf16(kM, Co);

  // channel block kb's halo and its nine taps' weights (one bulk copy, thread
  // 0) into buffer bf. A warp copies 4 channel chunks of 8 consecutive pixels
  // at a time (2 of 16 where KC is no multiple of 32), the chunks fastest:
  // eight lanes, which the load unit takes together, read 2 (4) lines and
  // write 8 banks groups. With all chunks of one pixel, or one chunk of eight
  // pixels, the same copies made the 128^2 pass 128 us instead of 120.
  // One address serves a pixel's chunks and, in narrow grids, all three copies.
  const int chunks = KC >> 3;
  const int lq = (chunks & 3) ? 1 : 2;  // log2 of the chunks a warp takes side by side
  const int lpx = (tid & 31) >> lq, lc = tid & ((1 << lq) - 1);
  auto load_weights = [&](int kb, int bf) {
    bulk_g2s(sm + (size_t)bf * bufbytes + hbytes, p.wimg + (size_t)kb * 9 * Co * KC, wbytes, &bar_w[bf],
             (p.stall && kb == 0) ? 16u : 0u);
  };
  auto load_block = [&](int kb, int bf) {
    unsigned char* dst = sm + (size_t)bf * bufbytes;
    if (tid == 0 && kb > 0) load_weights(kb, bf);
    const int up = p.up0 ? 1 : 0, ch0 = kb * KC + 8 * lc;
    const __nv_bfloat16* s0 = p.src0 + ((size_t)b << (p.lH + p.lW - 2 * up)) * p.C0 + ch0;
    const __nv_bfloat16* s1 = p.src1 + ((size_t)b << (p.lH + p.lW)) * p.C1 + (ch0 - p.C0);
    const uint32_t d0 = smem_addr(dst) + (uint32_t)lc * P * 16u;
    const uint32_t cp = (uint32_t)chunks * P * 16u;  // bytes between the copies
    const int n = halo_pos(W);
#pragma unroll 2
    for (int q = warp * (32 >> lq) + lpx; q < n; q += (kRowThreads / 32) * (32 >> lq)) {
      int r, gx;
      if (wide) {
        r = (q >= kM + 2) + (q >= 2 * (kM + 2));
        gx = (x0 + q - r * (kM + 2) - 1) & (W - 1);
      } else {
        r = q >> p.lW;
        gx = q & (W - 1);
      }
      const int gy = (y + r - 1) & (H - 1);
      const __nv_bfloat16* g0 = s0 + (size_t)(((gy >> up) << (p.lW - up)) + (gx >> up)) * p.C0;
      const __nv_bfloat16* g1 = s1 + (size_t)((gy << p.lW) + gx) * p.C1;
      const uint32_t d = d0 + (wide ? (uint32_t)q : (uint32_t)r << p.lW) * 16u;
      for (int c = 0; c < chunks; c += 1 << lq) {
        const __nv_bfloat16* g = (ch0 + 8 * c < p.C0 ? g0 : g1) + 8 * c;
        const uint32_t dc = d + (uint32_t)c * P * 16u;
        if (wide) {
          cp_async16(dc, g);
        } else {
#pragma unroll
          for (int kx = 0; kx < 3; ++kx) cp_async16(dc + kx * cp + (uint32_t)((gx + 1 - kx) & (W - 1)) * 16u, g);
        }
      }
    }
  };
  // block kb uses buffer kb & 1; its k-th use is phase k of that buffer's barriers
  auto parity_of = [](int kb) { return (unsigned)((kb >> 1) & 1); };

  // A parity wait tells a phase only from the one before it, so every wait
  // on an mbarrier here is made by warp 0, which sees every commit and every
  // copy in order; the other warps learn the outcome through the block votes.
  bool ok = true;
  int issued = -1, mma_seen = -1, copied = 0, copy_done = -1;
  // Until the launch before is complete: what does not depend on it, which
  // hides the barriers' and the tensor memory's set-up, the constants and, where
  // the image is that old, the first weights behind its tail.
  float kb0 = 0.f, kh0 = 0.f;  // a thread's bias and head weight (Co is at most its 256 threads), stored below
  if (tid < Co) {
    kb0 = __ldg(p.bias + tid);
    if (p.head_w) kh0 = __ldg(p.head_w + tid);
  }
  if (tid == 0 && p.early_w) {
    asm volatile("fence.proxy.async.global;\n" ::: "memory");
    load_weights(0, 0);
  }
  dep_wait();
  dep_go();
  if (tid == 0 && !p.early_w) load_weights(0, 0);
  load_block(0, 0);
  cp_async_commit();
  if (tid < Co) {
    consts.bias[tid] = kb0;
    consts.head[tid] = kh0;
  }
  for (int kb = 0; kb < nkb; ++kb) {
    const int bf = kb & 1;
    const bool pre = kb + 1 < nkb;
    // buffer bf ^ 1 was block kb - 1's: its MMAs must be done
    if (warp == 0 && pre && kb >= 1) {
      if (bar_wait(&bar_mma[(kb - 1) & 1], parity_of(kb - 1)))
        mma_seen = kb - 1;
      else
        ok = false;
    }
    if (__syncthreads_or(ok ? 0 : 1)) {
      ok = false;
      break;
    }
    if (pre) {
      load_block(kb + 1, bf ^ 1);
      copied = kb + 1;
    }
    cp_async_commit();
    cp_async_wait1();
    fence_async_smem();
    __syncthreads();
    if (warp == 0) {
      if (!__all_sync(0xffffffffu, bar_wait(&bar_w[bf], parity_of(kb)))) {
        ok = false;
      } else {
        copy_done = kb;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t hbase = sm0 + (uint32_t)bf * bufbytes;
          const uint32_t cstride = (uint32_t)P * 16u;  // bytes between chunks of a copy (LBO)
          TapSteps t;
          t.a = smem_desc(hbase, cstride, 128u);
          t.b = smem_desc(hbase + hbytes, (uint32_t)(Co / 8) * 128u, 128u);
          t.kx = wide ? 1u : (uint32_t)(chunks * P);
          t.ky = wide ? (uint32_t)(kM + 2) : (uint32_t)W;
          t.aj = 2u * P;
          t.bj = 2u * Co;
          issue_block(tmem, t, idesc, KC >> 4, kb > 0);
          mma_commit(&bar_mma[bf]);
        }
        __syncwarp();
        issued = kb;
      }
    }
  }
  // the last block's commit (the one before it was seen before its buffer was refilled)
  if (ok && warp == 0) {
    if (bar_wait(&bar_mma[(nkb - 1) & 1], parity_of(nkb - 1)))
      mma_seen = nkb - 1;
    else
      ok = false;
  }
  ok = __syncthreads_and(ok ? 1 : 0) != 0;
  if (ok) {
    tc_epilogue(p, consts, tmem, warp, kRowThreads / 32, pix, true);
  } else if (tid == 0) {
    atomicOr(p.err, SGN_TC_WAIT);
    // drain in order what this CTA still has in flight
    for (int k = mma_seen + 1; k <= issued; ++k)
      if (!bar_wait(&bar_mma[k & 1], parity_of(k))) break;
    for (int k = copy_done + 1; k <= copied; ++k) bar_wait(&bar_w[k & 1], parity_of(k));
  }
  cp_async_wait0();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, p.tmem_cols);
}

}  // namespace unet_tc
