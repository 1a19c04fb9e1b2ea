// fixed.cuh - block fixed-point arithmetic for the FP64 transforms.
//
// A GB300 issues one FP64 warp instruction per 77 cycles of an SM quarter
// (FP32: one per cycle, a 64-bit integer addition one per 2 cycles: a probe of
// independent chains), so an FP64 FFT is bound by its additions. Inside a
// transform every value shares one scale, which is what an integer is good
// at: the transforms of the FP64 passes run on 64-bit integers v * 2^-s with
// one s per transform, and FP64 stays the format in memory. Per complex element
// of a 2048-point transform that is about 270 issue cycles against 2700.
//
// Scale. With L1 = sum |z_j| over the transform's inputs, no intermediate of
// any FFT of them exceeds L1 (each is a sum of inputs with unit factors) and
// the butterflies' sums of two components stay below sqrt(2) L1. L1 is bounded
// from above with integers (a maximum of the exponents, then a sum of truncated
// magnitudes + 1: the order of the additions cannot change it, so the scale
// does not depend on the block shape) and s is the largest with
// L1 2^s <= 2^60.7 (the sum of the twiddle product's four cross terms then stays
// below 2^63).
// From 512 points on the first two stages run at a finer scale, at which
// 64 max|z| (all two radix-8 stages can grow to) fits, and from 1024 on the
// third at one for 512 max|z|; rounded shifts between them come down to s.
// Rounding noise grows by the root of the length that is left, and that is 64
// and 512 times shorter behind the shifts. Error against quad precision,
// relative 2-norm, for random and for 1 + localized inputs: 2048 points 5.4e-17
// and 6.0e-17 (the FP64 radix-8 FFT: 2.1e-16 and 1.9e-16), 4096 points 7.5e-17
// and 8.0e-17 (2.4e-16 and 1.9e-16); spectra of one dominant mode and white ones
// through the inverse, 1024 to 4096 points: 1.1e-16 to 1.6e-16 (2.1e-16). Below 512
// points there is one scale, and the noise is not smaller than at 2048: random
// inputs of 256 x 1024, both passes, 1.6e-16.
//
// Infinities and NaN: a transform whose inputs hold one returns all NaN.
// Magnitudes below 2^-1022 count as zero.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fft_core.cuh"

namespace sgn {

struct fx {
  long long v;
};
typedef unsigned long long u64;
__host__ __device__ __forceinline__ fx operator+(fx a, fx b) { return fx{(long long)((u64)a.v + (u64)b.v)}; }
__host__ __device__ __forceinline__ fx operator-(fx a, fx b) { return fx{(long long)((u64)a.v - (u64)b.v)}; }
__host__ __device__ __forceinline__ fx operator-(fx a) { return fx{(long long)(0ull - (u64)a.v)}; }

// 32-bit signed limbs of a 64-bit integer: h 2^32 + l
struct fxl {
  int h, l;
};
// limbs of 2v (|v| < 2^62): products with Q63 factors then need no final shift
__device__ __forceinline__ fxl limbs2(fx a) {
  const u64 d = 2ull * (u64)a.v;
  const int l = (int)(unsigned)d;
  return fxl{(int)(unsigned)(d >> 32) - (l >> 31), l};
}
// 32 x 32 -> 64 bits, kept apart from the additions by the asm: fused into
// 64-bit multiply-adds the same products take twice the issue cycles
__device__ __forceinline__ long long mul_wide(int a, int b) {
  long long r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}

// a b + c d for a, c limbs2 of data and b, d limbs of Q63 factors, rounded; the
// low x low products (below half a unit) are left out. 69 issue cycles per
// complex product; 92 with the cross products' upper halves from mad.hi, 132
// as a chain of 64-bit multiply-adds.
__device__ __forceinline__ fx dot2(fxl a, fxl b, fxl c, fxl d) {
  const long long x =
      (mul_wide(a.l, b.h) + mul_wide(c.l, d.h)) + (mul_wide(a.h, b.l) + mul_wide(c.h, d.l)) + 0x80000000ll;
  return fx{mul_wide(a.h, b.h) + mul_wide(c.h, d.h) + (long long)(int)(x >> 32)};
}
// v c, |v| < 2^62, c = limbs of a Q63 factor
__device__ __forceinline__ fx mul_q(fx a, fxl c) {
  const fxl l = limbs2(a);
  const long long x = mul_wide(l.l, c.h) + mul_wide(l.h, c.l) + 0x80000000ll;
  return fx{mul_wide(l.h, c.h) + (long long)(int)(x >> 32)};
}
// v / sqrt 2
__device__ __forceinline__ fx mul_rsqrt2(fx a) { return mul_q(a, fxl{0x5a82799a, -51432894}); }

// A twiddle factor W is stored as (-Re W, Im W) in Q63 limbs (h << 32 | l):
// +1 has no Q63 form, and the factors of the stages (exponents jm r below R Ns)
// take Re W = +1 and Im W = -1, but never the opposite signs.
__device__ __forceinline__ fxl tw_limbs(fx w) { return fxl{(int)(w.v >> 32), (int)(unsigned)(u64)w.v}; }

// (limbs are never negated: -(-2^31) has no limb; the value is, before the split)
template <>
__device__ __forceinline__ cpx<fx> cmul(cpx<fx> a, cpx<fx> w) {
  const fxl nx = tw_limbs(w.x), ny = tw_limbs(w.y);
  const fxl ax = limbs2(a.x), ay = limbs2(a.y), may = limbs2(-a.y);
  cpx<fx> r;
  r.x = -dot2(ax, nx, ay, ny);
  r.y = dot2(ax, ny, may, nx);
  return r;
}
// a * conj(w)
template <>
__device__ __forceinline__ cpx<fx> cmulc(cpx<fx> a, cpx<fx> w) {
  const fxl nx = tw_limbs(w.x), ny = tw_limbs(w.y);
  const fxl ax = limbs2(a.x), ay = limbs2(a.y), max_ = limbs2(-a.x);
  cpx<fx> r;
  r.x = dot2(max_, nx, ay, ny);
  r.y = -dot2(ax, ny, ay, nx);
  return r;
}
template <>
__device__ __forceinline__ cpx<fx> ldg(const cpx<fx>* p) {
  const longlong2 v = __ldg(reinterpret_cast<const longlong2*>(p));
  return mk(fx{v.x}, fx{v.y});
}
// 16-byte elements: the double-float layout (XOR within groups of 8, no padding)
template <>
__device__ __forceinline__ int sidx<fx>(int p, int lcs) {
  return (p ^ ((p >> 3) & 7)) << lcs;
}
template <>
struct unpadded_smem<fx> {
  static constexpr bool value = true;
};

// 8-point DFT in place (see fft_core.cuh)
template <bool INV>
__device__ __forceinline__ void bfly8(cpx<fx>* x) {
  cpx<fx> a0 = x[0] + x[4], a1 = x[1] + x[5], a2 = x[2] + x[6], a3 = x[3] + x[7];
  cpx<fx> b0 = x[0] - x[4], b1 = x[1] - x[5], b2 = x[2] - x[6], b3 = x[3] - x[7];
  if (!INV) {
    b1 = mk(mul_rsqrt2(b1.x + b1.y), mul_rsqrt2(b1.y - b1.x));
    b2 = mul_mi(b2);
    b3 = mk(mul_rsqrt2(b3.y - b3.x), mul_rsqrt2(-(b3.x + b3.y)));
  } else {
    b1 = mk(mul_rsqrt2(b1.x - b1.y), mul_rsqrt2(b1.x + b1.y));
    b2 = mul_i(b2);
    b3 = mk(mul_rsqrt2(-(b3.x + b3.y)), mul_rsqrt2(b3.x - b3.y));
  }
  bfly4<INV>(a0, a1, a2, a3);
  bfly4<INV>(b0, b1, b2, b3);
  x[0] = a0; x[2] = a1; x[4] = a2; x[6] = a3;
  x[1] = b0; x[3] = b1; x[5] = b2; x[7] = b3;
}

// a 2^-s rounded to nearest, halves to even (1 <= s <= 63, |a| < 2^62). FP64 inputs
// have so few bits below the unit that halves are common, and a transform adds up
// what always goes one way: with halves rounded up, the mean of 1024 x 8 random
// values was off by 21 times the error of its other coefficients, and column
// transforms of 1024 left a positive error of 9e-16 at x = 0 of every row; with
// the matvec's sums rounded down, L[sigma] on 8 x 1024 was off by 10 times its
// other errors at (0, 0).
__device__ __forceinline__ fx shr_round(fx a, int s) {
  const unsigned odd = (unsigned)((u64)a.v >> s) & 1u;
  return fx{(long long)((u64)a.v + ((1ull << (s - 1)) - 1ull) + (u64)odd) >> s};
}
// the same for any s >= 1, and for any s >= 0
__device__ __forceinline__ fx fx_sar1(fx a, int s) { return shr_round(a, s < 63 ? s : 63); }
__device__ __forceinline__ fx fx_sar(fx a, int s) { return s > 0 ? fx_sar1(a, s) : a; }

// Transform of length 2^lN held in v: fft_regs for fx. sh, sh2: the rounded
// shifts after the second and the third stage. One copy of the radix-8 stage.
template <bool INV>
__device__ __forceinline__ void fft_fx(cpx<fx> (&v)[8], cpx<fx>* sm, const cpx<fx>* __restrict__ tw, int t, int lN,
                                       int lcs, int plan, int sh, int sh2) {
  const int T_ = 1 << (lN - 3);
  const int n8 = lN / 3, rem = lN - 3 * n8;
  const bool first_small = plan && rem;
  // the stage of lNs reads its rows at 2^lNs - 8 of the plan's table (plan 1:
  // 2^lNs - 2^rem past entry N)
  const cpx<fx>* twp = first_small ? tw + (1 << lN) + 8 - (1 << rem) : tw;
  const int stages = n8 + (rem ? 1 : 0);
  int lNs = 0;
#pragma unroll 1
  for (int st = 0; st < stages; ++st) {
    const bool last = st == stages - 1;
    const int Ns = 1 << lNs;
    const bool small = rem && (first_small ? st == 0 : last);
    if (!small) {
      const int jm = t & (Ns - 1);
      if (lNs > 0) {
        const cpx<fx>* tws = twp + (Ns - 8) + jm;
#pragma unroll
        for (int r = 1; r < 8; ++r) {
          const cpx<fx> w = ldg(tws + (r - 1) * Ns);
          v[r] = INV ? cmulc(v[r], w) : cmul(v[r], w);
        }
      }
      bfly8<INV>(v);
      if (!last) {
        const int base = ((t >> lNs) << (lNs + 3)) + jm;
#pragma unroll
        for (int r = 0; r < 8; ++r) sm[sidx<fx>(base + r * Ns, lcs)] = v[r];
      }
      lNs += 3;
    } else if (rem == 2) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int j = t + q * T_, jm = j & (Ns - 1);
        if (lNs > 0) {
          const cpx<fx>* tws = twp + (Ns - 8) + jm;
#pragma unroll
          for (int r = 1; r < 4; ++r) {
            const cpx<fx> w = ldg(tws + (r - 1) * Ns);
            v[q + 2 * r] = INV ? cmulc(v[q + 2 * r], w) : cmul(v[q + 2 * r], w);
          }
        }
        bfly4<INV>(v[q], v[q + 2], v[q + 4], v[q + 6]);
        if (!last) {
          const int base = ((j >> lNs) << (lNs + 2)) + jm;
#pragma unroll
          for (int r = 0; r < 4; ++r) sm[sidx<fx>(base + r * Ns, lcs)] = v[q + 2 * r];
        }
      }
      lNs += 2;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = t + q * T_, jm = j & (Ns - 1);
        if (lNs > 0) {
          const cpx<fx> w = ldg(twp + (Ns - 8) + jm);
          v[q + 4] = INV ? cmulc(v[q + 4], w) : cmul(v[q + 4], w);
        }
        bfly2<INV>(v[q], v[q + 4]);
        if (!last) {
          const int base = ((j >> lNs) << (lNs + 1)) + jm;
#pragma unroll
          for (int r = 0; r < 2; ++r) sm[sidx<fx>(base + r * Ns, lcs)] = v[q + 4 * r];
        }
      }
      lNs += 1;
    }
    if (!last) {
      __syncthreads();
      load_slots(v, sm, t, T_, lcs);
      __syncthreads();
      if (st == 1 || st == 2) {
        const int d = st == 1 ? sh : sh2;
        if (d > 0) {
#pragma unroll
          for (int s = 0; s < 8; ++s) v[s] = mk(shr_round(v[s].x, d), shr_round(v[s].y, d));
        }
      }
    }
  }
}

// ----------------------------------------------------------- FP64 <-> fixed

// hi word of |x|: exponent in bits 30..20, monotonic in |x|
__device__ __forceinline__ unsigned abs_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// 0 x: zero, but an infinity or NaN stays one. What a derivative multiplies by
// m = 0 takes no part in its scale: the mean of a large value with small variations
// would set it (whole numbers of 18 bits at 1024 x 256: error of the x-derivative
// 1.6e-14 without a mean; on one of 2^30, 7.9e-13 when it counted and 2.7e-14 now;
// FP64 radix-8: 5.3e-14 on both).
__device__ __forceinline__ double fx_times0(double x) { return abs_hi(x) < 0x7ff00000u ? 0.0 : x; }

// truncated magnitude in units of 2^(E - 1043)
__device__ __forceinline__ unsigned fx_mag(unsigned hi, int E) {
  const int s = E - (int)(hi >> 20);
  return ((hi & 0xfffffu) | 0x100000u) >> (s < 31 ? s : 31);
}
// upper bound of |(a, b)| from truncated magnitudes of one unit
__device__ __forceinline__ unsigned fx_modulus(unsigned a, unsigned b) {
  const unsigned mx = a > b ? a : b, mn = a > b ? b : a;
  return mx + ((mn * 27u) >> 6) + 3u;  // max + 0.422 min >= the modulus
}

// Scale of one transform: inputs are converted with r0 (see fx_from), the
// shifts of fft_fx, results are v * 2^q.
struct FxScale {
  int r0, sh, sh2, q;
  bool bad;  // an infinity or NaN among the inputs
};

// largest k with B 2^k <= 2^60.7 (0xcfe00000 / 2^32 < 2^-0.3)
__device__ __forceinline__ int fx_room(unsigned B) {
  const int b = 32 - __clz((int)B);
  return (B << (32 - b)) <= 0xcfe00000u ? 61 - b : 60 - b;
}
// log2 scales of stages 1 and 2 (k1), of stage 3 (k3) and of the rest (k2) for
// the bounds L of the sum and M of the largest of the moduli (M < 2^23)
struct FxSteps {
  int k1, k2, k3;
};
__device__ __forceinline__ FxSteps fx_steps(unsigned L, unsigned M, int lN) {
  FxSteps r;
  r.k2 = r.k3 = r.k1 = fx_room(L);
  if (lN >= 10) r.k3 = max(r.k2, fx_room(min(512u * M, L)));
  r.k1 = r.k3;
  if (lN >= 9) r.k1 = max(r.k3, fx_room(min(64u * M, L)));
  return r;
}
// E: largest exponent field, L: bound of the sum of moduli and M: of the
// largest modulus, both in units of 2^(E - ue)
__device__ __forceinline__ FxScale fx_scale(int E, unsigned L, unsigned M, int ue, int lN) {
  FxScale r;
  r.bad = E == 0x7ff;
  const FxSteps st = fx_steps(L > 0u ? L : 1u, M, lN);
  r.sh = st.k1 - st.k3;
  r.sh2 = st.k3 - st.k2;
  r.r0 = 46 - st.k1 + E;
  r.q = E - ue - st.k2;
  return r;
}
// x at the scale r0, rounded; DER: m x with an integer 0 <= m < 2048, mm = m << 21
template <bool DER>
__device__ __forceinline__ fx fx_from(double x, int r0, unsigned mm) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned mh = 0x80000000u | ((hi & 0xfffffu) << 11) | (lo >> 21), ml = lo << 11;
  u64 M = ((u64)mh << 32) | ml;
  if (DER) M = (u64)mh * mm + __umulhi(ml, mm);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const int r = r0 - e;
  u64 u;
  if (DER && r <= 0)
    u = M << (-r & 63);
  else
    u = ((M >> ((r - 1) & 63)) + 1ull) >> 1;
  if (e == 0 || r > 64) u = 0ull;
  const u64 sg = (u64)(long long)((int)hi >> 31);
  return fx{(long long)((u ^ sg) - sg)};
}
// v 2^q in FP64, rounded to nearest (underflow to zero, overflow to infinity)
__device__ __forceinline__ double fx_to(fx a, int q) {
  const u64 sg = (u64)(a.v >> 63);
  const u64 u = ((u64)a.v ^ sg) - sg;
  const int n = __clzll((long long)u);
  const u64 w = u << (n & 63);
  const int ef = 1085 - n + q;  // exponent field less one
  u64 b = (w >> 11) + ((w >> 10) & 1ull) + ((u64)(unsigned)ef << 52);
  if ((unsigned)ef >= 2046u) b = ef < 0 ? 0ull : 0x7ff0000000000000ull;
  if (u == 0ull) b = 0ull;
  return __longlong_as_double((long long)(b | (sg << 63)));
}
// c = (h 2^32 + l) 2^-63 2^(e - 1021); zero and subnormal c give zero limbs
__device__ __forceinline__ fxl fx_mant(double c, int* e) {
  const unsigned hi = (unsigned)__double2hiint(c), lo = (unsigned)__double2loint(c);
  const int ex = (int)((hi >> 20) & 0x7ffu);
  const u64 mt = ((u64)(0x20000000u | ((hi & 0xfffffu) << 9) | (lo >> 23)) << 32) | (lo << 9);
  const u64 sg = (u64)(long long)((int)hi >> 31);
  const u64 ms = (mt ^ sg) - sg;
  fxl m;
  m.l = (int)(unsigned)ms;
  m.h = (int)(unsigned)(ms >> 32) - (m.l >> 31);
  if (ex == 0) m.h = m.l = 0;
  *e = ex;
  return m;
}
// x 2^e for a finite x whose result is normal (or x = 0)
__device__ __forceinline__ double scale_exp(double x, int e) {
  return (abs_hi(x) >> 20) == 0u ? 0.0 : __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}

// ------------------------------------------------------------ twiddle table
// W_4096^k = exp(-2 pi i k / 4096) as the product of W^(64 a) and W^b (a, b <
// 64; Q62 constants from 60-digit arithmetic): every length's factors on the
// host and on the device from 128 constants.
struct FxTw {
  long long c, s;
};
// on the host static, or each call would copy its 1 KB to the stack (55 ns an entry of a solver's tables, 0.2 ms at
// 1024 x 256); device functions cannot have static variables of this kind
#ifdef __CUDA_ARCH__
#define FX_TABLE constexpr
#else
#define FX_TABLE static constexpr
#endif
__host__ __device__ inline FxTw fx_tw_hi(int a) {
  FX_TABLE FxTw t[64] = {
      {4611686018427387904ll, 0ll}, {4589479489746651964ll, -452024275624069880ll},
      {4523073764714963030ll, -899695310372275547ll}, {4413108366765438139ll, -1338701787458110889ll},
      {4260642322793532497ll, -1764815834521887442ll}, {4067143964149113252ll, -2173933740352748318ll},
      {3834476785802888710ll, -2562115475870945497ll}, {3564881499871150442ll, -2925622638761716784ll},
      {3260954456333195553ll, -3260954456333195553ll}, {2925622638761716784ll, -3564881499871150442ll},
      {2562115475870945497ll, -3834476785802888710ll}, {2173933740352748318ll, -4067143964149113252ll},
      {1764815834521887442ll, -4260642322793532497ll}, {1338701787458110889ll, -4413108366765438139ll},
      {899695310372275547ll, -4523073764714963030ll}, {452024275624069880ll, -4589479489746651964ll},
      {0ll, -4611686018427387904ll}, {-452024275624069880ll, -4589479489746651964ll},
      {-899695310372275547ll, -4523073764714963030ll}, {-1338701787458110889ll, -4413108366765438139ll},
      {-1764815834521887442ll, -4260642322793532497ll}, {-2173933740352748318ll, -4067143964149113252ll},
      {-2562115475870945497ll, -3834476785802888710ll}, {-2925622638761716784ll, -3564881499871150442ll},
      {-3260954456333195553ll, -3260954456333195553ll}, {-3564881499871150442ll, -2925622638761716784ll},
      {-3834476785802888710ll, -2562115475870945497ll}, {-4067143964149113252ll, -2173933740352748318ll},
      {-4260642322793532497ll, -1764815834521887442ll}, {-4413108366765438139ll, -1338701787458110889ll},
      {-4523073764714963030ll, -899695310372275547ll}, {-4589479489746651964ll, -452024275624069880ll},
      {-4611686018427387904ll, 0ll}, {-4589479489746651964ll, 452024275624069880ll},
      {-4523073764714963030ll, 899695310372275547ll}, {-4413108366765438139ll, 1338701787458110889ll},
      {-4260642322793532497ll, 1764815834521887442ll}, {-4067143964149113252ll, 2173933740352748318ll},
      {-3834476785802888710ll, 2562115475870945497ll}, {-3564881499871150442ll, 2925622638761716784ll},
      {-3260954456333195553ll, 3260954456333195553ll}, {-2925622638761716784ll, 3564881499871150442ll},
      {-2562115475870945497ll, 3834476785802888710ll}, {-2173933740352748318ll, 4067143964149113252ll},
      {-1764815834521887442ll, 4260642322793532497ll}, {-1338701787458110889ll, 4413108366765438139ll},
      {-899695310372275547ll, 4523073764714963030ll}, {-452024275624069880ll, 4589479489746651964ll},
      {0ll, 4611686018427387904ll}, {452024275624069880ll, 4589479489746651964ll},
      {899695310372275547ll, 4523073764714963030ll}, {1338701787458110889ll, 4413108366765438139ll},
      {1764815834521887442ll, 4260642322793532497ll}, {2173933740352748318ll, 4067143964149113252ll},
      {2562115475870945497ll, 3834476785802888710ll}, {2925622638761716784ll, 3564881499871150442ll},
      {3260954456333195553ll, 3260954456333195553ll}, {3564881499871150442ll, 2925622638761716784ll},
      {3834476785802888710ll, 2562115475870945497ll}, {4067143964149113252ll, 2173933740352748318ll},
      {4260642322793532497ll, 1764815834521887442ll}, {4413108366765438139ll, 1338701787458110889ll},
      {4523073764714963030ll, 899695310372275547ll}, {4589479489746651964ll, 452024275624069880ll},
  };
  return t[a];
}
__host__ __device__ inline FxTw fx_tw_lo(int b) {
  FX_TABLE FxTw t[64] = {
      {4611686018427387904ll, 0ll}, {4611680592556051597ll, -7074234977634094ll},
      {4611664314954810277ll, -14148453308909941ll}, {4611637185661966712ll, -21222638347508465ll},
      {4611599204741358747ll, -28296773447188932ll}, {4611550372282359158ll, -35370841961828118ll},
      {4611490688399875439ll, -42444827245459479ll}, {4611420153234349529ll, -49518712652312324ll},
      {4611338766951757487ll, -56592481536850979ll}, {4611246529743609097ll, -63666117253813961ll},
      {4611143441826947420ll, -70739603158253140ll}, {4611029503444348282ll, -77812922605572913ll},
      {4610904714863919703ll, -84886058951569363ll}, {4610769076379301266ll, -91958995552469432ll},
      {4610622588309663429ll, -99031715764970078ll}, {4610465250999706769ll, -106104202946277443ll},
      {4610297064819661174ll, -113176440454146016ll}, {4610118030165284974ll, -120248411646917787ll},
      {4609928147457864002ll, -127320099883561417ll}, {4609727417144210613ll, -134391488523711385ll},
      {4609515839696662623ll, -141462560927707152ll}, {4609293415613082204ll, -148533300456632313ll},
      {4609060145416854711ll, -155603690472353751ll}, {4608816029656887448ll, -162673714337560785ll},
      {4608561068907608378ll, -169743355415804323ll}, {4608295263768964774ll, -176812597071536008ll},
      {4608018614866421802ll, -183881422670147362ll}, {4607731122850961054ll, -190949815578008931ll},
      {4607432788399079011ll, -198017759162509421ll}, {4607123612212785457ll, -205085236792094843ll},
      {4606803595019601825ll, -212152231836307643ll}, {4606472737572559481ll, -219218727665825837ll},
      {4606131040650197959ll, -226284707652502141ll}, {4605778505056563124ll, -233350155169403100ll},
      {4605415131621205279ll, -240415053590848213ll}, {4605040921199177221ll, -247479386292449050ll},
      {4604655874671032219ll, -254543136651148378ll}, {4604259992942821947ll, -261606288045259271ll},
      {4603853276946094353ll, -268668823854504225ll}, {4603435727637891464ll, -275730727460054268ll},
      {4603007346000747137ll, -282791982244568062ll}, {4602568133042684743ll, -289852571592231009ll},
      {4602118089797214799ll, -296912478888794348ll}, {4601657217323332534ll, -303971687521614251ll},
      {4601185516705515398ll, -311030180879690912ll}, {4600702989053720509ll, -318087942353707635ll},
      {4600209635503382042ll, -325144955336069920ll}, {4599705457215408556ll, -332201203220944539ll},
      {4599190455376180266ll, -339256669404298611ll}, {4598664631197546246ll, -346311337283938677ll},
      {4598127985916821581ll, -353365190259549761ll}, {4597580520796784455ll, -360418211732734437ll},
      {4597022237125673177ll, -367470385107051883ll}, {4596453136217183155ll, -374521693788056937ll},
      {4595873219410463798ll, -381572121183339143ll}, {4595282488070115371ll, -388621650702561795ll},
      {4594680943586185780ll, -395670265757500976ll}, {4594068587374167303ll, -402717949762084594ll},
      {4593445420874993257ll, -409764686132431407ll}, {4592811445555034612ll, -416810458286890046ll},
      {4592166662906096533ll, -423855249646078038ll}, {4591511074445414878ll, -430899043632920815ll},
      {4590844681715652623ll, -437941823672690722ll}, {4590167486284896230ll, -444983573193046019ll},
  };
  return t[b];
}
#undef FX_TABLE
__host__ __device__ inline long long fx_pack_q63(long long q62) {
  // 2 q62 as limbs; the constants' extremes are -2^62 (exactly -1) and below +2^62
  const long long w = (long long)((u64)q62 * 2ull);
  const long long h = (long long)((u64)w + 0x80000000ull) >> 32;
  return (long long)(((u64)h << 32) | (u64)(unsigned)w);
}
// (-Re, Im) limbs of W_N^k, N = 2^lN <= 4096
__host__ __device__ inline cpx<fx> fx_twiddle(int k, int lN) {
  const int i = (k << (12 - lN)) & 4095;
  const FxTw a = fx_tw_hi(i >> 6), b = fx_tw_lo(i & 63);
  const __int128 rnd = (__int128)1 << 61;
  const long long c = (long long)(((__int128)a.c * b.c - (__int128)a.s * b.s + rnd) >> 62);
  const long long s = (long long)(((__int128)a.c * b.s + (__int128)a.s * b.c + rnd) >> 62);
  cpx<fx> r;
  r.x.v = fx_pack_q63(-c);
  r.y.v = fx_pack_q63(s);
  return r;
}

}  // namespace sgn
