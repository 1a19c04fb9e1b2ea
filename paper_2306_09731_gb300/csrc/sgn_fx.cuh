// sgn_fx.cuh - the FP64 transform passes on 64-bit fixed point (fixed.cuh).
//
// The same passes as sgn_spectral.cuh's templates, with FP64 spectra and fields
// in memory and block fixed-point transforms: x-passes over row pairs, y-passes
// over column tiles. Each transform finds its scale from its own inputs (a
// row pair or a column, as far as the rounding errors of an FP64 transform
// spread too).
#pragma once
#include "fixed.cuh"
#include "sgn_internal.h"

namespace sgn {

// The threads of one transform inside a block: t of T_, group g of G; the
// group's lanes in a warp differ in the bits lo..hi/2 of the lane.
constexpr int kFxSlots = 24;  // reduction slots per group at most

struct FxGrp {
  int t, g, G, lo, hi;
  unsigned mask;
  bool lead;
  unsigned* red;  // G words per slot, zeroed at the kernel's start
};
__device__ __forceinline__ FxGrp fx_group(int t, int g, int G, int lo, int hi, unsigned* red) {
  FxGrp q;
  q.t = t;
  q.g = g;
  q.G = G;
  q.lo = lo;
  q.hi = hi < 32 ? hi : 32;
  if (q.hi > (int)blockDim.x) q.hi = (int)blockDim.x;
  q.mask = blockDim.x >= 32 ? 0xffffffffu : ((1u << blockDim.x) - 1u);
  q.lead = q.hi <= q.lo || ((threadIdx.x & 31) & (q.hi - 1) & ~(q.lo - 1)) == 0;
  q.red = red;
  return q;
}
__device__ __forceinline__ void fx_red_zero(unsigned* red, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) red[i] = 0u;
  __syncthreads();
}
// contributes v to the group's slot; the slot is complete after a barrier
__device__ __forceinline__ void grp_max(const FxGrp& q, int slot, unsigned v) {
  for (int o = q.lo; o < q.hi; o <<= 1) {
    const unsigned w = __shfl_xor_sync(q.mask, v, o);
    v = w > v ? w : v;
  }
  if (q.lead) atomicMax(q.red + slot * q.G + q.g, v);
}
__device__ __forceinline__ void grp_add(const FxGrp& q, int slot, unsigned v) {
  for (int o = q.lo; o < q.hi; o <<= 1) v += __shfl_xor_sync(q.mask, v, o);
  if (q.lead) atomicAdd(q.red + slot * q.G + q.g, v);
}
__device__ __forceinline__ unsigned grp_get(const FxGrp& q, int slot) { return q.red[slot * q.G + q.g]; }

// The scale of the complex inputs (x, y)[8] of an inverse transform (two slots),
// and their conversion. DER: each is multiplied by i mi(s), |mi| < 2048.
template <bool DER, class M>
__device__ __forceinline__ FxScale fx_load8(const FxGrp& g, int slot, double (&x)[8], double (&y)[8], int lN, M mi,
                                            cpx<fx> (&v)[8]) {
  if (DER) {
#pragma unroll
    for (int s = 0; s < 8; ++s)
      if (mi(s) == 0) {
        x[s] = fx_times0(x[s]);
        y[s] = fx_times0(y[s]);
      }
  }
  unsigned mx = 0u;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const unsigned a = abs_hi(x[s]), b = abs_hi(y[s]), c = a > b ? a : b;
    mx = c > mx ? c : mx;
  }
  grp_max(g, slot, mx);
  __syncthreads();
  const unsigned Mh = grp_get(g, slot);
  const int E = (int)(Mh >> 20);
  unsigned sum = 0u;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const unsigned m = fx_modulus(fx_mag(abs_hi(x[s]), E), fx_mag(abs_hi(y[s]), E));
    if (DER) {
      const int k = mi(s);
      sum += (((m >> 2) * (unsigned)(k < 0 ? -k : k)) >> 12) + 1u;
    } else {
      sum += (m >> 3) + 1u;
    }
  }
  grp_add(g, slot + 1, sum);
  __syncthreads();
  const unsigned L = grp_get(g, slot + 1);
  const unsigned m21 = fx_modulus(((Mh & 0xfffffu) | 0x100000u) + 1u, ((Mh & 0xfffffu) | 0x100000u) + 1u);
  const FxScale sc = DER ? fx_scale(E, L, (((m21 >> 2) * (1u << (lN - 1))) >> 12) + 1u, 1029, lN)
                         : fx_scale(E, L, (m21 >> 3) + 1u, 1040, lN);
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    if (DER) {
      // times i m: (-m y, m x)
      const int k = mi(s);
      const unsigned mm = (unsigned)(k < 0 ? -k : k) << 21;
      const fx a = fx_from<true>(x[s], sc.r0, mm), b = fx_from<true>(y[s], sc.r0, mm);
      v[s] = k < 0 ? mk(b, -a) : mk(-b, a);
    } else {
      v[s] = mk(fx_from<false>(x[s], sc.r0, 0u), fx_from<false>(y[s], sc.r0, 0u));
    }
  }
  return sc;
}

__device__ __forceinline__ u64 fx_abs(fx a) { return (u64)(a.v ^ (a.v >> 63)); }

// The same for a forward transform, of field values: relative to the value c at
// the transform's first point where that makes the sum of moduli smaller. Small
// variations around a large value (a depth of 1 + small) then get the scale of
// the variations; the transform of c, N c at index 0, is added by the caller
// in FP64 (*c, zero if nothing was taken off). FP64 butterflies have the same
// property by themselves, as the differences of neighbouring values are exact.
// Four slots and one element of shared memory per group (first).
__device__ __forceinline__ FxScale fx_load8_fwd(const FxGrp& g, int slot, const double (&x)[8], const double (&y)[8],
                                                int lN, cpx<double>* first, cpx<fx> (&v)[8], cpx<double>* c) {
  unsigned mx = 0u;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const unsigned a = abs_hi(x[s]), b = abs_hi(y[s]), d = a > b ? a : b;
    mx = d > mx ? d : mx;
  }
  grp_max(g, slot, mx);
  if (g.t == 0) *first = mk(x[0], y[0]);
  __syncthreads();
  const int E = (int)(grp_get(g, slot) >> 20);
  // |v| < 2^60: 1.f 2^(E - 1023) goes to 1.f 2^59
  const int r0 = 4 + E;
  const cpx<double> z0 = *first;
  const cpx<fx> f0 = mk(fx_from<false>(z0.x, r0, 0u), fx_from<false>(z0.y, r0, 0u));
  unsigned sv = 0u, sd = 0u;
  u64 md = 0ull;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    v[s] = mk(fx_from<false>(x[s], r0, 0u), fx_from<false>(y[s], r0, 0u));
    sv += fx_modulus((unsigned)(fx_abs(v[s].x) >> 42), (unsigned)(fx_abs(v[s].y) >> 42));
    const u64 a = fx_abs(v[s].x - f0.x), b = fx_abs(v[s].y - f0.y), d = a > b ? a : b;
    md = d > md ? d : md;
  }
  grp_add(g, slot + 1, sv);
  grp_max(g, slot + 2, (unsigned)(md >> 30));
  __syncthreads();
  // |v - f0| < 2^(30 + b); moduli in units of 2^(12 + b)
  const int b = 32 - __clz((int)grp_get(g, slot + 2));
#pragma unroll
  for (int s = 0; s < 8; ++s)
    sd += fx_modulus((unsigned)(fx_abs(v[s].x - f0.x) >> (12 + b)), (unsigned)(fx_abs(v[s].y - f0.y) >> (12 + b)));
  grp_add(g, slot + 3, sd);
  __syncthreads();
  const unsigned Lv = grp_get(g, slot + 1), Ld = grp_get(g, slot + 3);
  // both sums in units of 2^42, rounded up
  const bool centre = (b <= 30 ? (Ld >> (30 - b)) + 1u : 0xffffffffu) < Lv;
  const unsigned L = centre ? Ld : Lv;
  const int u = centre ? 12 + b : 42;
  const FxSteps k = fx_steps(L, 372800u, lN);  // a modulus is at most 1.4219 * 2^18 + 3 units
  const int sl = k.k1 - u;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    if (centre) v[s] = v[s] - f0;
    if (sl >= 0)
      v[s] = mk(fx{(long long)((u64)v[s].x.v << sl)}, fx{(long long)((u64)v[s].y.v << sl)});
    else
      v[s] = mk(shr_round(v[s].x, -sl), shr_round(v[s].y, -sl));
  }
  FxScale sc;
  sc.bad = E == 0x7ff;
  sc.r0 = r0;
  sc.sh = k.k1 - k.k3;
  sc.sh2 = k.k3 - k.k2;
  sc.q = E - 1082 + u - k.k2;  // v 2^(E - 1082) before the shift
  *c = centre ? mk(fx_to(f0.x, E - 1082), fx_to(f0.y, E - 1082)) : mk(0.0, 0.0);
  return sc;
}

// What a thread adds to the sum of moduli of the packed spectrum (fx_load_packed),
// every entry counted twice (k and N - k): entries k = t + s T_ of both rows, and
// on t = 0 the real ones at N/2.
template <bool DER>
__device__ __forceinline__ unsigned fx_packed_sum(const cpx<double> (&A)[4], const cpx<double> (&B)[4], double an,
                                                  double bn, int E, int t, int T_) {
  unsigned sum = 0u;
  if (!DER && t == 0) sum = ((fx_mag(abs_hi(an), E) + fx_mag(abs_hi(bn), E)) >> 3) + 2u;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const unsigned m = fx_modulus(fx_mag(abs_hi(A[s].x), E), fx_mag(abs_hi(A[s].y), E)) +
                       fx_modulus(fx_mag(abs_hi(B[s].x), E), fx_mag(abs_hi(B[s].y), E));
    if (DER)
      sum += (((m >> 3) * (unsigned)(t + s * T_)) >> 10) + 2u;
    else
      sum += (m >> 2) + 2u;
  }
  return sum;
}
// the conversion: Z[k] kept, Z[N - k] and Z[N/2] handed over in sm
template <bool DER>
__device__ __forceinline__ void fx_packed_from(const cpx<double> (&A)[4], const cpx<double> (&B)[4], double an,
                                               double bn, int r0, int t, int lN, cpx<fx>* sm, cpx<fx> (&v)[8]) {
  const int N = 1 << lN, T_ = N >> 3, half = N >> 1;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int k = t + s * T_;
    const unsigned mm = (unsigned)k << 21;
    cpx<fx> a = mk(fx_from<DER>(A[s].x, r0, mm), fx_from<DER>(A[s].y, r0, mm));
    cpx<fx> b = mk(fx_from<DER>(B[s].x, r0, mm), fx_from<DER>(B[s].y, r0, mm));
    if (DER) {
      a = mul_i(a);
      b = mul_i(b);
    }
    v[s] = mk(a.x - b.y, a.y + b.x);
    if (k > 0) sm[sidx<fx>(N - k, 0)] = mk(a.x + b.y, b.x - a.y);
  }
  if (t == 0)
    sm[sidx<fx>(half, 0)] = DER ? mk(fx{0}, fx{0}) : mk(fx_from<false>(an, r0, 0u), fx_from<false>(bn, r0, 0u));
}

// The packed spectrum of two real rows from their half spectra S0, S1 (see
// load_packed): a thread converts the entries k = t + s T_ < N/2 of both rows
// once, keeps Z[k] = A + i B and hands Z[N - k] = conj(A) + i conj(B) over in sm
// (free on entry and on exit). der: times i m (the factor 2 pi/Lx is left out).
// der may differ between the groups of a block: every barrier is outside its
// branches. (Where the whole block takes one form, fx_load_packed_all has the two
// as constants: 80 registers against 102 in k_fx_c2r.)
__device__ __forceinline__ FxScale fx_load_packed(const FxGrp& g, int slot, const cpx<double>* S0,
                                                  const cpx<double>* S1, int lN, bool der, cpx<fx>* sm,
                                                  cpx<fx> (&v)[8]) {
  const int N = 1 << lN, T_ = N >> 3, half = N >> 1, t = g.t;
  cpx<double> A[4], B[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const double2 a = *reinterpret_cast<const double2*>(S0 + t + s * T_);
    const double2 b = *reinterpret_cast<const double2*>(S1 + t + s * T_);
    A[s] = mk(a.x, a.y);
    B[s] = mk(b.x, b.y);
  }
  double an = 0.0, bn = 0.0;  // the real entries at N/2 (their i m multiple is zero)
  if (t == 0) {
    A[0].y = 0.0;
    B[0].y = 0.0;
    if (der) {
      A[0].x = fx_times0(A[0].x);
      B[0].x = fx_times0(B[0].x);
    } else {
      an = S0[half].x;
      bn = S1[half].x;
    }
  }
  unsigned mx = abs_hi(an) > abs_hi(bn) ? abs_hi(an) : abs_hi(bn);
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const unsigned a = abs_hi(A[s].x), b = abs_hi(A[s].y), c = abs_hi(B[s].x), d = abs_hi(B[s].y);
    const unsigned e = a > b ? a : b, f = c > d ? c : d, h = e > f ? e : f;
    mx = h > mx ? h : mx;
  }
  grp_max(g, slot, mx);
  __syncthreads();
  const unsigned Mh = grp_get(g, slot);
  const int E = (int)(Mh >> 20);
  grp_add(g, slot + 1, der ? fx_packed_sum<true>(A, B, an, bn, E, t, T_) : fx_packed_sum<false>(A, B, an, bn, E, t, T_));
  __syncthreads();
  const unsigned L = grp_get(g, slot + 1);
  // |Z| <= |A| + |B|
  const unsigned m21 = 2u * fx_modulus(((Mh & 0xfffffu) | 0x100000u) + 1u, ((Mh & 0xfffffu) | 0x100000u) + 1u);
  const FxScale sc = fx_scale(E, L, der ? (((m21 >> 3) * (unsigned)half) >> 11) + 1u : (m21 >> 3) + 1u,
                              der ? 1029 : 1040, lN);
  if (der)
    fx_packed_from<true>(A, B, an, bn, sc.r0, t, lN, sm, v);
  else
    fx_packed_from<false>(A, B, an, bn, sc.r0, t, lN, sm, v);
  __syncthreads();
#pragma unroll
  for (int s = 4; s < 8; ++s) v[s] = sm[sidx<fx>(t + s * T_, 0)];
  __syncthreads();
  return sc;
}

// the same with der equal across the block
__device__ __forceinline__ FxScale fx_load_packed_all(const FxGrp& g, int slot, const cpx<double>* S0,
                                                      const cpx<double>* S1, int lN, bool der, cpx<fx>* sm,
                                                      cpx<fx> (&v)[8]) {
  return der ? fx_load_packed(g, slot, S0, S1, lN, true, sm, v) : fx_load_packed(g, slot, S0, S1, lN, false, sm, v);
}

// After a forward transform of z = f0 + i f1: 2 F0[k], 2 F1[k] for the thread's
// k = t + s T_ (s < 4, and k = N/2 on t = 0). Leaves sm in use.
__device__ __forceinline__ void fx_split(const cpx<fx> (&v)[8], cpx<fx>* sm, int t, int lN, cpx<fx> (&f0)[5],
                                         cpx<fx> (&f1)[5]) {
  const int N = 1 << lN, T_ = N >> 3;
  store_slots(v, sm, t, T_, 0);
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const cpx<fx> P = v[s], Q = conjg(sm[sidx<fx>((N - t - s * T_) & (N - 1), 0)]);
    f0[s] = P + Q;
    f1[s] = mul_mi(P - Q);
  }
}
__device__ __forceinline__ bool fx_owns(int s, int t) { return s < 4 || t == 0; }

__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }
__device__ __forceinline__ cpx<double> fx_out(cpx<fx> z, int q, bool bad) {
  return bad ? mk(fx_nan(), fx_nan()) : mk(fx_to(z.x, q), fx_to(z.y, q));
}

// ---------------------------------------------------------------- x-passes
// (phases > 1: that many groups of threads per row pair, group ph of them)
struct FxXLay {
  int t, grp, ph, P, lN, N, T_;
  size_t y0, y1;
  bool valid;
};
template <int LN>
__device__ __forceinline__ FxXLay fx_xlay(const Geom& G, int phases = 1) {
  FxXLay L;
  L.lN = LN > 0 ? LN : G.lNx;
  L.N = 1 << L.lN;
  L.T_ = L.N >> 3;
  L.P = (blockDim.x >> (L.lN - 3)) / phases;
  L.grp = threadIdx.x >> (L.lN - 3);
  L.ph = phases > 1 ? L.grp / L.P : 0;
  L.grp -= L.ph * L.P;
  L.t = threadIdx.x & (L.T_ - 1);
  int pair = blockIdx.x * L.P + L.grp;
  L.valid = pair < (G.Ny >> 1);
  if (!L.valid) pair = (G.Ny >> 1) - 1;
  L.y0 = 2 * (size_t)pair;
  L.y1 = L.y0 + 1;
  return L;
}
// shared memory of an x-pass: P transform buffers, the extra elements, then
// the reduction slots
__device__ __forceinline__ unsigned* fx_xred(const FxXLay& L, int extra, cpx<fx>** sm) {
  extern __shared__ __align__(16) unsigned char smraw[];
  cpx<fx>* b = reinterpret_cast<cpx<fx>*>(smraw);
  *sm = b + (size_t)L.grp * L.N;
  return reinterpret_cast<unsigned*>(b + (size_t)L.P * (L.N + extra));
}

// the elements of fx_load8_fwd's first points, behind the reduction slots
__device__ __forceinline__ cpx<double>* fx_first(unsigned* red, int G, int g) {
  return reinterpret_cast<cpx<double>*>(red + kFxSlots * G) + g;
}

template <int LN>
constexpr int fx_threads() { return LN == 12 ? 512 : 256; }

struct FxR2CArgs {
  const double* f[4];
  cpx<double>* out[4];
};
template <int LN>
__global__ void __launch_bounds__(fx_threads<LN>()) k_fx_r2c(Geom G, const cpx<fx>* __restrict__ tw, FxR2CArgs a) {
  const FxXLay L = fx_xlay<LN>(G);
  cpx<fx>* sm;
  unsigned* red = fx_xred(L, 0, &sm);
  const FxGrp g = fx_group(L.t, L.grp, L.P, 1, L.T_, red);
  const double* f = a.f[blockIdx.y];
  double x[8], y[8];
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    x[s] = f[L.y0 * L.N + L.t + s * L.T_];
    y[s] = f[L.y1 * L.N + L.t + s * L.T_];
  }
  fx_red_zero(red, 4 * L.P);
  cpx<fx> v[8];
  cpx<double> c;
  const FxScale sc = fx_load8_fwd(g, 0, x, y, L.lN, fx_first(red, L.P, L.grp), v, &c);
  fft_fx<false>(v, sm, tw, L.t, L.lN, 0, 0, sc.sh, sc.sh2);
  cpx<fx> f0[5], f1[5];
  fx_split(v, sm, L.t, L.lN, f0, f1);
  if (!L.valid) return;
  cpx<double>* o = a.out[blockIdx.y];
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    if (!fx_owns(s, L.t)) continue;
    const int k = L.t + s * L.T_;
    cpx<double> z0 = fx_out(f0[s], sc.q - 1, sc.bad), z1 = fx_out(f1[s], sc.q - 1, sc.bad);
    if (k == 0) {
      z0.x += (double)L.N * c.x;
      z1.x += (double)L.N * c.y;
    }
    o[L.y0 * G.ldS + k] = z0;
    o[L.y1 * G.ldS + k] = z1;
  }
}

struct FxC2RArgs {
  const cpx<double>* in[4];
  double* out[4];
  int deriv[4];
};
// lscale: the output is divided by 2^lscale; alpha = 2 pi / Lx (derivatives)
template <int LN>
__global__ void __launch_bounds__(fx_threads<LN>()) k_fx_c2r(Geom G, const cpx<fx>* __restrict__ tw, FxC2RArgs a,
                                                            int lscale, double alpha) {
  const FxXLay L = fx_xlay<LN>(G);
  cpx<fx>* sm;
  unsigned* red = fx_xred(L, 0, &sm);
  const FxGrp g = fx_group(L.t, L.grp, L.P, 1, L.T_, red);
  const int fi = blockIdx.y;
  const bool der = a.deriv[fi] != 0;
  const cpx<double>* in = a.in[fi];
  fx_red_zero(red, 2 * L.P);
  cpx<fx> v[8];
  const FxScale sc = fx_load_packed_all(g, 0, in + L.y0 * G.ldS, in + L.y1 * G.ldS, L.lN, der, sm, v);
  fft_fx<true>(v, sm, tw, L.t, L.lN, 0, 0, sc.sh, sc.sh2);
  if (!L.valid) return;
  double* o = a.out[fi];
  int q = sc.q - lscale;
  fxl am{0, 0};
  if (der) {
    int e;
    am = fx_mant(alpha, &e);
    q += e - 1021;
  }
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int x = L.t + s * L.T_;
    if (der) v[s] = mk(mul_q(v[s].x, am), mul_q(v[s].y, am));
    const cpx<double> z = fx_out(v[s], q, sc.bad);
    o[L.y0 * L.N + x] = z.x;
    o[L.y1 * L.N + x] = z.y;
  }
}

// coefficients from the y-inverse of h_hat (see k_coef_x)
template <int LN>
__global__ void __launch_bounds__(fx_threads<LN>()) k_fx_coef_x(Geom G, const cpx<fx>* __restrict__ tw,
                                                               const cpx<double>* Hy, double* h, double* cr,
                                                               double* cc, int* flags, CoefCopy cp) {
  const FxXLay L = fx_xlay<LN>(G);
  cpx<fx>* sm;
  unsigned* red = fx_xred(L, 0, &sm);
  const FxGrp g = fx_group(L.t, L.grp, L.P, 1, L.T_, red);
  fx_red_zero(red, 2 * L.P);
  cpx<fx> v[8];
  const FxScale sc =
      fx_load_packed(g, 0, Hy + L.y0 * G.ldS, Hy + L.y1 * G.ldS, L.lN, false, sm, v);
  fft_fx<true>(v, sm, tw, L.t, L.lN, 0, 0, sc.sh, sc.sh2);
  if (!L.valid) return;
  const double invN = 1.0 / (double)G.nphys();
  const int q = sc.q - G.lNx - G.lNy;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int x = L.t + s * L.T_;
    const cpx<double> z = fx_out(v[s], q, sc.bad);
    coef_point<double>(z.x, invN, h, cr, cc, L.y0 * L.N + x, flags, cp);
    coef_point<double>(z.y, invN, h, cr, cc, L.y1 * L.N + x, flags, cp);
  }
}

// The matvec's x-pass (see k_mv_x). S, Sy: y-inverses of sigma_hat and of
// i m_y sigma_hat (without the factor 2 pi/Ly); writes Cout = a - i kx bx and
// Byout = by (of Sy as it is). k2 = (2 pi/Lx) kx per half-spectrum column: the
// derivative of phase 1 leaves 2 pi/Lx out and the combination puts both in.
// The three phases (a, bx, by: an inverse transform, a product and a forward
// one each) run one after the other, or, with PAR, at the same time in three
// groups of threads of the block: a small grid has fewer row pairs than the GPU
// has room for, and a pass then lasts as long as its chain of transforms
// (256 x 16: 35.5 -> 18.7 us; 1024 x 256: 40.7 -> 26.9). At 2048^2 the groups' buffers would halve the row pairs
// that an SM holds.
template <int LN, bool PAR>
__global__ void __launch_bounds__(PAR ? 384 : fx_threads<LN>(), PAR || LN == 12 ? 1 : 2) k_fx_mv_x(
    Geom G, const cpx<fx>* __restrict__ tw, const double* __restrict__ k2, const cpx<double>* S,
    const cpx<double>* Sy, const double* __restrict__ cr, const double* __restrict__ cc, cpx<double>* Cout,
    cpx<double>* Byout, int plan) {
  const int phases = PAR ? 3 : 1;
  const FxXLay L = fx_xlay<LN>(G, phases);
  const int t = L.t, T_ = L.T_, lN = L.lN;
  extern __shared__ __align__(16) unsigned char smraw[];
  // a transform buffer per group, the stash of a per row pair, the slots
  cpx<fx>* sm = reinterpret_cast<cpx<fx>*>(smraw) + (size_t)(L.ph * L.P + L.grp) * L.N;
  cpx<fx>* stash = reinterpret_cast<cpx<fx>*>(smraw) + (size_t)phases * L.P * L.N;
  unsigned* red = reinterpret_cast<unsigned*>(stash + (size_t)L.P * 10 * T_);
  stash += (size_t)L.grp * 10 * T_;
  const FxGrp g = fx_group(t, L.ph * L.P + L.grp, phases * L.P, 1, T_, red);
  // a's scale and whether its row pair holds an infinity or NaN
  int* qa_s = reinterpret_cast<int*>(red + kFxSlots * phases * L.P) + 2 * L.grp;
  fx_red_zero(red, 15 * phases * L.P);
  const size_t o0 = L.y0 * G.ldS, o1 = L.y1 * G.ldS, p0 = L.y0 * L.N + t, p1 = L.y1 * L.N + t;
#pragma unroll 1
  for (int it = 0; it < (PAR ? 1 : 3); ++it) {
    const int ph = PAR ? L.ph : it, slot = PAR ? 0 : 5 * it;
    const cpx<double>* in = ph == 2 ? Sy : S;
    const double* __restrict__ cf = ph == 0 ? cc : cr;
    // the largest coefficient of the row pair (complete after the barriers below)
    unsigned cm = 0u;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const unsigned a = abs_hi(cf[p0 + s * T_]), b = abs_hi(cf[p1 + s * T_]), c = a > b ? a : b;
      cm = c > cm ? c : cm;
    }
    grp_max(g, slot + 4, cm);
    cpx<fx> v[8];
    const FxScale sc = PAR ? fx_load_packed(g, slot, in + o0, in + o1, lN, ph == 1, sm, v)
                           : fx_load_packed_all(g, slot, in + o0, in + o1, lN, ph == 1, sm, v);
    const int Ec = (int)(grp_get(g, slot + 4) >> 20);
    const bool bad = sc.bad || Ec == 0x7ff;
    fft_fx<true>(v, sm, tw, t, lN, 0, plan, sc.sh, sc.sh2);
    // products with the coefficients, aligned to the largest one's exponent
    unsigned mx = 0u;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      int e0, e1;
      const fxl c0 = fx_mant(cf[p0 + s * T_], &e0), c1 = fx_mant(cf[p1 + s * T_], &e1);
      v[s] = mk(fx_sar(mul_q(v[s].x, c0), Ec - e0), fx_sar(mul_q(v[s].y, c1), Ec - e1));
      const unsigned a = (unsigned)(fx_abs(v[s].x) >> 32), b = (unsigned)(fx_abs(v[s].y) >> 32);
      const unsigned c = a > b ? a : b;
      mx = c > mx ? c : mx;
    }
    grp_max(g, slot + 2, mx);
    __syncthreads();
    // |components| < 2^(32 + b); moduli in units of 2^(14 + b)
    const int b = 32 - __clz((int)grp_get(g, slot + 2));
    unsigned sum = 0u;
#pragma unroll
    for (int s = 0; s < 8; ++s)
      sum += fx_modulus((unsigned)(fx_abs(v[s].x) >> (14 + b)), (unsigned)(fx_abs(v[s].y) >> (14 + b)));
    grp_add(g, slot + 3, sum);
    __syncthreads();
    // (a modulus is at most 1.4219 * 2^18 + 3)
    const FxSteps k = fx_steps(grp_get(g, slot + 3), 372800u, lN);
    const int sl = k.k1 - 14 - b;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      if (sl >= 0)
        v[s] = mk(fx{(long long)((u64)v[s].x.v << sl)}, fx{(long long)((u64)v[s].y.v << sl)});
      else
        v[s] = mk(shr_round(v[s].x, -sl), shr_round(v[s].y, -sl));
    }
    // value = v 2^(q + Ec - 1021) before the shift
    const int q = sc.q + Ec - 1021 - (k.k2 - 14 - b);
    fft_fx<false>(v, sm, tw, t, lN, 0, plan, k.k1 - k.k3, k.k3 - k.k2);
    cpx<fx> b0[5], b1[5];
    fx_split(v, sm, t, lN, b0, b1);
    if (ph == 0) {
      if (t == 0) {
        qa_s[0] = q;
        qa_s[1] = bad ? 1 : 0;
      }
#pragma unroll
      for (int s = 0; s < 5; ++s) {
        stash[(2 * s) * T_ + t] = b0[s];
        stash[(2 * s + 1) * T_ + t] = b1[s];
      }
    }
    __syncthreads();
    if (ph > 0) {
      const int qa = qa_s[0];
      const bool nan = bad || (ph == 1 && qa_s[1] != 0);
#pragma unroll
      for (int s = 0; s < 5; ++s) {
        if (!fx_owns(s, t) || !L.valid) continue;
        const int kc = t + s * T_;
        if (ph == 1) {
          // a - i kap b, aligned to the larger of the two scales plus one bit
          int ek;
          const fxl km = fx_mant(__ldg(k2 + kc), &ek);
          const int qb = q + ek - 1021, qc = (qa > qb ? qa : qb) + 1;
          const cpx<fx> a0 = stash[(2 * s) * T_ + t], a1 = stash[(2 * s + 1) * T_ + t];
          const int sa = qc - qa, sb = qc - qb;
          cpx<fx> z;
          z.x = fx_sar1(a0.x, sa) + fx_sar1(mul_q(b0[s].y, km), sb);
          z.y = fx_sar1(a0.y, sa) - fx_sar1(mul_q(b0[s].x, km), sb);
          Cout[o0 + kc] = fx_out(z, qc, nan);
          z.x = fx_sar1(a1.x, sa) + fx_sar1(mul_q(b1[s].y, km), sb);
          z.y = fx_sar1(a1.y, sa) - fx_sar1(mul_q(b1[s].x, km), sb);
          Cout[o1 + kc] = fx_out(z, qc, nan);
        } else {
          Byout[o0 + kc] = fx_out(b0[s], q, nan);
          Byout[o1 + kc] = fx_out(b1[s], q, nan);
        }
      }
    }
  }
}

// The RHS's x-pass (see k_rhs_x), its pointwise part in FP64. alx, aly: 2 pi /
// Lx, Ly. PAR: the five inverse transforms run side by side in five groups of
// threads, then three of them take F, q_x and q_y (grids with few row pairs, see
// k_fx_mv_x: 256 x 16 66 -> 31 us, 1024 x 256 85 -> 53).
template <int LN, bool PAR>
__global__ void __launch_bounds__(PAR ? 640 : fx_threads<LN>(), PAR || LN == 12 ? 1 : 2) k_fx_rhs_x(
    Geom G, const cpx<fx>* __restrict__ tw, const double* __restrict__ kx, const cpx<double>* Vx,
    const cpx<double>* Vy, const cpx<double>* S, const cpx<double>* Sy, const double* __restrict__ hh,
    const double* __restrict__ cr, double grav, double alx, double aly, cpx<double>* Cq, cpx<double>* Qy,
    cpx<double>* Fh, int plan) {
  const FxXLay L = fx_xlay<LN>(G, PAR ? 5 : 1);
  const int t = L.t, T_ = L.T_, lN = L.lN, N = L.N;
  extern __shared__ __align__(16) unsigned char smraw[];
  if constexpr (PAR) {
    const int ng = 5 * L.P, gi = L.ph * L.P + L.grp, ln = G.lNx + G.lNy;
    cpx<fx>* sm = reinterpret_cast<cpx<fx>*>(smraw) + (size_t)gi * N;
    cpx<double>* phys = reinterpret_cast<cpx<double>*>(smraw) + (size_t)ng * N;
    unsigned* red = reinterpret_cast<unsigned*>(phys + (size_t)ng * N);
    const FxGrp g = fx_group(t, gi, ng, 1, T_, red);
    fx_red_zero(red, 6 * ng);
    const size_t o0 = L.y0 * G.ldS, o1 = L.y1 * G.ldS, p0 = L.y0 * N + t, p1 = L.y1 * N + t;
    cpx<fx> v[8];
    // group 0: i kx sigma_hat, 1: Sy = i m_y sigma_hat, 2: sigma_hat, 3: vx, 4: vy
    {
      const int i = L.ph;
      const cpx<double>* in = i == 1 ? Sy : (i == 3 ? Vx : (i == 4 ? Vy : S));
      const FxScale sc = fx_load_packed(g, 0, in + o0, in + o1, lN, i == 0, sm, v);
      fft_fx<true>(v, sm, tw, t, lN, 0, plan, sc.sh, sc.sh2);
      const double al = i == 0 ? alx : aly;
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        cpx<double> z = fx_out(v[s], sc.q - ln, sc.bad);
        if (i < 2) z = mk(al * z.x, al * z.y);
        phys[(size_t)gi * N + t + s * T_] = z;
      }
    }
    __syncthreads();
    const int j = L.ph;  // 0: F, 1: q_x, 2: q_y; 3 and 4 only keep the barriers
    double f0[8], f1[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      f0[s] = f1[s] = 0.0;
      if (j > 2) continue;
      const cpx<double>* z = phys + (size_t)L.grp * N + t + s * T_;
      const size_t gs = (size_t)L.P * N;
      const cpx<double> vx = z[3 * gs], vy = z[4 * gs];
      const double a0 = hh[p0 + s * T_], a1 = hh[p1 + s * T_];  // h - 1
      if (j == 0) {
        const cpx<double> sx = z[0], sy = z[gs], sg = z[2 * gs];
        const double r0 = scale_exp(cr[p0 + s * T_], ln + 1), r1 = scale_exp(cr[p1 + s * T_], ln + 1);
        const double q0 = sg.x * r0 * r0, q1 = sg.y * r1 * r1;
        f0[s] = -0.5 * r0 * r0 * (sx.x * sx.x + sy.x * sy.x) - 4.5 * q0 * q0 + 0.5 * vx.x * vx.x +
                (0.5 * vy.x * vy.x + grav * a0);
        f1[s] = -0.5 * r1 * r1 * (sx.y * sx.y + sy.y * sy.y) - 4.5 * q1 * q1 + 0.5 * vx.y * vx.y +
                (0.5 * vy.y * vy.y + grav * a1);
      } else {
        const cpx<double> d = z[(j - 1) * gs], u = j == 1 ? vx : vy;
        f0[s] = (u.x + a0 * u.x) - d.x;
        f1[s] = (u.y + a1 * u.y) - d.y;
      }
    }
    cpx<double> c;
    const FxScale sc = fx_load8_fwd(g, 2, f0, f1, lN, fx_first(red, ng, gi), v, &c);
    fft_fx<false>(v, sm, tw, t, lN, 0, plan, sc.sh, sc.sh2);
    cpx<fx> h0[5], h1[5];
    fx_split(v, sm, t, lN, h0, h1);
    if (j < 3 && L.valid) {
#pragma unroll
      for (int s = 0; s < 5; ++s) {
        if (!fx_owns(s, t)) continue;
        const int k = t + s * T_;
        if (j == 1) {
          int e;
          const fxl km = fx_mant(__ldg(kx + k), &e);
          const int q = sc.q - 1 + e - 1021;
          Cq[o0 + k] = fx_out(mk(mul_q(h0[s].y, km), -mul_q(h0[s].x, km)), q, sc.bad);
          Cq[o1 + k] = fx_out(mk(mul_q(h1[s].y, km), -mul_q(h1[s].x, km)), q, sc.bad);
        } else {
          cpx<double>* o = j == 0 ? Fh : Qy;
          cpx<double> z0 = fx_out(h0[s], sc.q - 1, sc.bad), z1 = fx_out(h1[s], sc.q - 1, sc.bad);
          if (k == 0) {
            z0.x += (double)N * c.x;
            z1.x += (double)N * c.y;
          }
          o[o0 + k] = z0;
          o[o1 + k] = z1;
        }
      }
    }
    return;
  }
  cpx<fx>* sm;
  unsigned* red = fx_xred(L, 2 * N, &sm);
  // the accumulators of q_x, q_y: the thread's own slots
  cpx<double>* acc = reinterpret_cast<cpx<double>*>(smraw) + (size_t)L.P * N + (size_t)L.grp * 2 * N;
  const FxGrp g = fx_group(t, L.grp, L.P, 1, T_, red);
  fx_red_zero(red, 22 * L.P);
  const size_t o0 = L.y0 * G.ldS, o1 = L.y1 * G.ldS, p0 = L.y0 * N + t, p1 = L.y1 * N + t;
  const int ln = G.lNx + G.lNy;
  double F0[8], F1[8];
  // inputs: 0 i kx sigma_hat, 1 Sy = i m_y sigma_hat, 2 sigma_hat, 3 vx, 4 vy
#pragma unroll 1
  for (int i = 0; i < 5; ++i) {
    const cpx<double>* in = i == 1 ? Sy : (i == 3 ? Vx : (i == 4 ? Vy : S));
    cpx<fx> v[8];
    const FxScale sc = fx_load_packed_all(g, 2 * i, in + o0, in + o1, lN, i == 0, sm, v);
    fft_fx<true>(v, sm, tw, t, lN, 0, plan, sc.sh, sc.sh2);
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      cpx<double>* qx = acc + (size_t)s * T_ + t;
      cpx<double>* qy = acc + (size_t)(8 + s) * T_ + t;
      const cpx<double> z = fx_out(v[s], sc.q - ln, sc.bad);
      if (i == 0) {
        *qx = mk(-alx * z.x, -alx * z.y);  // -sigma_x
      } else if (i == 1) {
        const double r0 = scale_exp(cr[p0 + s * T_], ln + 1), r1 = scale_exp(cr[p1 + s * T_], ln + 1);
        const double z0 = aly * z.x, z1 = aly * z.y;
        const cpx<double> q = *qx;
        *qy = mk(-z0, -z1);
        F0[s] = -0.5 * r0 * r0 * (q.x * q.x + z0 * z0);
        F1[s] = -0.5 * r1 * r1 * (q.y * q.y + z1 * z1);
      } else if (i == 2) {
        const double r0 = scale_exp(cr[p0 + s * T_], ln + 1), r1 = scale_exp(cr[p1 + s * T_], ln + 1);
        const double q0 = z.x * r0 * r0, q1 = z.y * r1 * r1;
        F0[s] -= 4.5 * q0 * q0;
        F1[s] -= 4.5 * q1 * q1;
      } else {
        const double a0 = hh[p0 + s * T_], a1 = hh[p1 + s * T_];  // h - 1
        cpx<double>* q = i == 3 ? qx : qy;
        const cpx<double> w = *q;
        *q = mk(w.x + (z.x + a0 * z.x), w.y + (z.y + a1 * z.y));
        F0[s] += 0.5 * z.x * z.x;
        F1[s] += 0.5 * z.y * z.y;
        if (i == 4) {
          F0[s] += grav * a0;
          F1[s] += grav * a1;
        }
      }
    }
  }
  // the split returns twice the half spectra: one bit off the output scale
#pragma unroll 1
  for (int j = 0; j < 3; ++j) {
    if (j > 0) {
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const cpx<double> z = acc[(size_t)(8 * (j - 1) + s) * T_ + t];
        F0[s] = z.x;
        F1[s] = z.y;
      }
    }
    cpx<fx> v[8];
    cpx<double> c;
    const FxScale sc = fx_load8_fwd(g, 10 + 4 * j, F0, F1, lN, fx_first(red, L.P, L.grp), v, &c);
    fft_fx<false>(v, sm, tw, t, lN, 0, plan, sc.sh, sc.sh2);
    cpx<fx> f0[5], f1[5];
    fx_split(v, sm, t, lN, f0, f1);
#pragma unroll
    for (int s = 0; s < 5; ++s) {
      if (!fx_owns(s, t) || !L.valid) continue;
      const int k = t + s * T_;
      if (j == 1) {
        int e;
        const fxl km = fx_mant(__ldg(kx + k), &e);
        // -i kx q
        const int q = sc.q - 1 + e - 1021;
        Cq[o0 + k] = fx_out(mk(mul_q(f0[s].y, km), -mul_q(f0[s].x, km)), q, sc.bad);
        Cq[o1 + k] = fx_out(mk(mul_q(f1[s].y, km), -mul_q(f1[s].x, km)), q, sc.bad);
      } else {
        cpx<double>* o = j == 0 ? Fh : Qy;
        cpx<double> z0 = fx_out(f0[s], sc.q - 1, sc.bad), z1 = fx_out(f1[s], sc.q - 1, sc.bad);
        if (k == 0) {
          z0.x += (double)N * c.x;
          z1.x += (double)N * c.y;
        }
        o[o0 + k] = z0;
        o[o1 + k] = z1;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- y-passes
struct FxYLay {
  int t, c, lC, lN, N, T_, col;
  bool valid;
};
template <int LN>
__device__ __forceinline__ FxYLay fx_ylay(const Geom& G, int nthr, int tid) {
  FxYLay L;
  L.lN = LN > 0 ? LN : G.lNy;
  L.N = 1 << L.lN;
  L.T_ = L.N >> 3;
  L.lC = __ffs(nthr >> (L.lN - 3)) - 1;
  L.c = tid & ((1 << L.lC) - 1);
  L.t = tid >> L.lC;
  L.col = (blockIdx.x << L.lC) + L.c;
  L.valid = L.col < G.Nxh;
  if (!L.valid) L.col = G.Nxh - 1;
  return L;
}
__device__ __forceinline__ int fx_my(int row, int Ny) {
  return row < (Ny >> 1) ? row : (row == (Ny >> 1) ? 0 : row - Ny);
}

// one transform per block row (blockIdx.y picks the field), stored as it is;
// deriv: of i m_y times the input, times aly at the end when that is not 0
struct FxYArgs {
  const cpx<double>* src[4];
  cpx<double>* dst[4];
  int deriv[4];
  const int* sel;  // may be null: every src is offset by (*sel) * sel_stride
  size_t sel_stride;
};
template <bool INV, int LN>
__global__ void __launch_bounds__(fx_threads<LN>(), LN == 12 ? 1 : 2) k_fx_y(Geom G, const cpx<fx>* __restrict__ tw,
                                                                          FxYArgs a, double aly, int plan) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const FxYLay L = fx_ylay<LN>(G, blockDim.x, threadIdx.x);
  const int C = 1 << L.lC;
  cpx<fx>* smb = reinterpret_cast<cpx<fx>*>(smraw);
  unsigned* red = reinterpret_cast<unsigned*>(smb + ((size_t)L.N << L.lC));
  const FxGrp g = fx_group(L.t, L.c, C, C, 32, red);
  const int fi = blockIdx.y;
  const cpx<double>* src = a.src[fi] + (a.sel ? (size_t)(*a.sel) * a.sel_stride : 0) + L.col;
  double x[8], y[8];
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const double2 z = *reinterpret_cast<const double2*>(src + (size_t)(L.t + s * L.T_) * G.ldS);
    x[s] = z.x;
    y[s] = z.y;
  }
  fx_red_zero(red, 4 * C);
  cpx<fx> v[8];
  const bool der = a.deriv[fi] != 0;
  FxScale sc;
  cpx<double> c = mk(0.0, 0.0);
  if (!INV)
    sc = fx_load8_fwd(g, 0, x, y, L.lN, fx_first(red, C, L.c), v, &c);
  else if (der)
    sc = fx_load8<true>(g, 0, x, y, L.lN, [&](int s) { return fx_my(L.t + s * L.T_, L.N); }, v);
  else
    sc = fx_load8<false>(g, 0, x, y, L.lN, [](int) { return 0; }, v);
  fft_fx<INV>(v, smb + L.c, tw, L.t, L.lN, L.lC, plan, sc.sh, sc.sh2);
  if (!L.valid) return;
  int q = sc.q;
  const bool mul = der && aly != 0.0;
  fxl am{0, 0};
  if (mul) {
    int e;
    am = fx_mant(aly, &e);
    q += e - 1021;
  }
  cpx<double>* o = a.dst[fi] + L.col;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    if (mul) v[s] = mk(mul_q(v[s].x, am), mul_q(v[s].y, am));
    cpx<double> z = fx_out(v[s], q, sc.bad);
    if (!INV && s == 0 && L.t == 0) {
      z.x += (double)L.N * c.x;
      z.y += (double)L.N * c.y;
    }
    o[(size_t)(L.t + s * L.T_) * G.ldS] = z;
  }
}

// Forward transforms of NIN inputs combined by the epilogue: each finished
// transform but the last waits in the thread's own slots of shared memory.
// NIN = 2, the matvec: w = [M^-1] (C - i k2y By), k2 = (2 pi/Ly) ky per row.
// NIN = 3, the RHS: K = (Cq - i ky Qy, -i kx F, -i ky F), 2/3-masked if asked.
struct FxYFwdArgs {
  const cpx<double>* src[3];
  cpx<double>* dst[3];
  const double* kr;    // per row: k2y (matvec) or ky (RHS)
  const double* kx;    // per column (RHS)
  const double* minv;  // M^-1 per entry, or null (matvec)
  int dealias;
};
// PAR: the transforms run at the same time in NIN groups of threads (grids with
// few columns, see k_fx_mv_x; 1024 x 256: matvec 15.3 -> 12.4 us, RHS 20.5 ->
// 15.6), and each group writes every NIN-th of the 8 slots.
template <int NIN, int LN, bool PAR>
__global__ void __launch_bounds__(PAR ? 384 : fx_threads<LN>(), PAR || LN == 12 ? 1 : 2)
    k_fx_yfwd(Geom G, const cpx<fx>* __restrict__ tw, FxYFwdArgs a, int plan) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int phases = PAR ? NIN : 1, nthr = blockDim.x / phases;
  const int ph = PAR ? threadIdx.x / nthr : 0, tid = threadIdx.x - ph * nthr;
  const FxYLay L = fx_ylay<LN>(G, nthr, tid);
  const int C = 1 << L.lC;
  cpx<fx>* smb = reinterpret_cast<cpx<fx>*>(smraw) + ((size_t)ph * L.N << L.lC);
  cpx<fx>* stash = reinterpret_cast<cpx<fx>*>(smraw) + ((size_t)phases * L.N << L.lC);
  unsigned* red = reinterpret_cast<unsigned*>(stash + (size_t)(NIN - (PAR ? 0 : 1)) * 8 * nthr);
  const FxGrp g = fx_group(L.t, ph * C + L.c, phases * C, C, C < 32 ? 32 : C, red);
  int* q_s = reinterpret_cast<int*>(red + kFxSlots * phases * C);
  fx_red_zero(red, 2 * NIN * phases * C);
  cpx<fx> v[8];
  int q[NIN];
  bool bad = false;
#pragma unroll 1
  for (int it = 0; it < (PAR ? 1 : NIN); ++it) {
    const int i = PAR ? ph : it;
    const cpx<double>* src = (i == 0 ? a.src[0] : (i == 1 ? a.src[1] : a.src[2])) + L.col;
    double x[8], y[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const double2 z = *reinterpret_cast<const double2*>(src + (size_t)(L.t + s * L.T_) * G.ldS);
      x[s] = z.x;
      y[s] = z.y;
    }
    const FxScale sc = fx_load8<false>(g, PAR ? 0 : 2 * i, x, y, L.lN, [](int) { return 0; }, v);
    bad = bad || sc.bad;
    if (PAR) {
      if (L.t == 0) q_s[2 * (ph * C + L.c)] = sc.q, q_s[2 * (ph * C + L.c) + 1] = sc.bad ? 1 : 0;
    } else {
#pragma unroll
      for (int j = 0; j < NIN; ++j)
        if (i == j) q[j] = sc.q;
    }
    fft_fx<false>(v, smb + L.c, tw, L.t, L.lN, L.lC, plan, sc.sh, sc.sh2);
    if (PAR || i + 1 < NIN) {
#pragma unroll
      for (int s = 0; s < 8; ++s) stash[(size_t)(i * 8 + s) * nthr + tid] = v[s];
    }
  }
  if (PAR) {
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NIN; ++j) {
      q[j] = q_s[2 * (j * C + L.c)];
      bad = bad || q_s[2 * (j * C + L.c) + 1] != 0;
    }
  }
  if (!L.valid) return;
  int ekx = 0;
  fxl kxm{0, 0};
  if (NIN == 3) kxm = fx_mant(__ldg(a.kx + L.col), &ekx);
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    if (PAR && s % NIN != ph) continue;
    const int row = L.t + s * L.T_;
    const size_t e = (size_t)row * G.ldS + L.col;
    int ek;
    const fxl km = fx_mant(__ldg(a.kr + row), &ek);
    const cpx<fx> z0 = stash[(size_t)s * nthr + tid];
    const cpx<fx> z1 = NIN == 2 && !PAR ? v[s] : stash[(size_t)(8 + s) * nthr + tid];
    // z0 - i k z1, aligned to the larger of the two scales plus one bit
    const int q1 = q[1] + ek - 1021, qc = (q[0] > q1 ? q[0] : q1) + 1;
    cpx<fx> z;
    z.x = fx_sar1(z0.x, qc - q[0]) + fx_sar1(mul_q(z1.y, km), qc - q1);
    z.y = fx_sar1(z0.y, qc - q[0]) - fx_sar1(mul_q(z1.x, km), qc - q1);
    int qz = qc;
    if (NIN == 2) {
      if (a.minv) {
        int em;
        const fxl mm = fx_mant(__ldg(a.minv + e), &em);
        z = mk(mul_q(z.x, mm), mul_q(z.y, mm));
        qz += em - 1021;
      }
      a.dst[0][e] = fx_out(z, qz, bad);
    } else {
      const int my = row <= (G.Ny >> 1) ? row : G.Ny - row;
      const bool cut = a.dealias && (3 * L.col > G.Nx || 3 * my > G.Ny);
      const cpx<double> zero = mk(0.0, 0.0);
      a.dst[0][e] = cut ? zero : fx_out(z, qz, bad);
      const cpx<fx> f = PAR ? stash[(size_t)(8 * (NIN - 1) + s) * nthr + tid] : v[s];
      a.dst[1][e] = cut ? zero : fx_out(mk(mul_q(f.y, kxm), -mul_q(f.x, kxm)), q[NIN - 1] + ekx - 1021, bad);
      a.dst[2][e] = cut ? zero : fx_out(mk(mul_q(f.y, km), -mul_q(f.x, km)), q[NIN - 1] + ek - 1021, bad);
    }
  }
}

}  // namespace sgn
