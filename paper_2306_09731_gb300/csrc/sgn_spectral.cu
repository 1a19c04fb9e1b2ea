// sgn_spectral.cu - the FP64 spectral passes (the paper's method, and every
// precision's state conversions), their transforms in block fixed point
// (sgn_fx.cuh), and the host code the passes share (launch shapes, tensor
// maps); the templates of the other arithmetics are in sgn_spectral.cuh.
#define SGN_SPECTRAL_COMMON
#include "sgn_spectral.cuh"

#include "sgn_fx.cuh"

namespace sgn {

// Calls f with the compile-time length of the sizes that have one, else 0:
// 4096 points take 512 threads a transform and have their own kernels.
template <class F>
static inline void fx_ln(int lN, F&& f) {
  if (lN == 12)
    f(std::integral_constant<int, 12>());
  else
    f(std::integral_constant<int, 0>());
}

static void fx_x_config(const Geom& G, dim3& grid, dim3& block, size_t& smem, int nf, int extra_per_pair = 0,
                        int tpb = 0) {
  const int Tn = G.Nx >> 3;
  int P = builtin_pairs(G);
  if (tpb > 0 && tpb % Tn == 0) {
    const int q = tpb / Tn;
    if ((q & (q - 1)) == 0 && tpb <= (G.lNx == 12 ? 512 : 256) && q <= (G.Ny >> 1)) P = q;
  }
  block = dim3(Tn * P);
  grid = dim3((G.Ny / 2 + P - 1) / P, nf);
  smem = (size_t)P * ((size_t)(G.Nx + extra_per_pair) * sizeof(cpx<fx>) + kFxSlots * sizeof(unsigned) + sizeof(cpx<double>));
}
static void fx_y_config(const Geom& G, dim3& grid, dim3& block, size_t& smem, int nf, int stash = 0, int tpb = 0) {
  const int Tn = G.Ny >> 3;
  int C = builtin_cols(G, TT_F64, 1);
  if (tpb >= 32 && tpb % Tn == 0) {
    const int q = tpb / Tn;
    if ((q & (q - 1)) == 0 && q <= 64 && tpb <= (G.lNy == 12 ? 512 : 256)) C = q;
  }
  block = dim3(Tn * C);
  grid = dim3((G.Nxh + C - 1) / C, nf);
  smem = (size_t)C * ((size_t)G.Ny * (1 + stash) * sizeof(cpx<fx>) + kFxSlots * sizeof(unsigned) + sizeof(cpx<double>));
}

// Whether a pass of `blocks` blocks of `threads` threads runs its transforms side
// by side in `phases` groups (PAR, see k_fx_mv_x): the groups must be whole
// warps and fit the kernel's threads, and the GPU must have room, under two
// blocks per SM.
static bool fx_parallel(const dim3& grid, const dim3& block, int phases, int most = 384) {
  return block.x % 32 == 0 && (int)block.x * phases <= most && grid.x < kTwoPerSm;
}

template <int L>
static void fx_attrs() {
  set_smem<double>((const void*)k_fx_r2c<L>);
  set_smem<double>((const void*)k_fx_c2r<L>);
  set_smem<double>((const void*)k_fx_coef_x<L>);
  set_smem<double>((const void*)k_fx_mv_x<L, false>);
  set_smem<double>((const void*)k_fx_rhs_x<L, false>);
  set_smem<double>((const void*)k_fx_y<true, L>);
  set_smem<double>((const void*)k_fx_y<false, L>);
  set_smem<double>((const void*)k_fx_yfwd<2, L, false>);
  set_smem<double>((const void*)k_fx_yfwd<3, L, false>);
}
template <>
void init_kernel_attributes<double>() {
  fx_attrs<0>();
  fx_attrs<12>();
  set_smem<double>((const void*)k_fx_mv_x<0, true>);
  set_smem<double>((const void*)k_fx_rhs_x<0, true>);
  set_smem<double>((const void*)k_fx_yfwd<2, 0, true>);
  set_smem<double>((const void*)k_fx_yfwd<3, 0, true>);
  cudaGetLastError();
}

static const double kTwoPi = 6.283185307179586476925286766559;

template <>
cudaError_t launch_x_r2c<double>(const Geom& G, const Tables<double>& tb, const double* const* f, int nf,
                                 cpx<double>* const* out, const Exec& ex) {
  FxR2CArgs a{};
  for (int i = 0; i < nf; ++i) {
    a.f[i] = f[i];
    a.out[i] = out[i];
  }
  dim3 grid, block;
  size_t smem;
  fx_x_config(G, grid, block, smem, nf);
  ex.begin(PK_IO);
  fx_ln(G.lNx, [&](auto ln) { k_fx_r2c<decltype(ln)::value><<<grid, block, smem, ex.s>>>(G, tb.twx, a); });
  ex.end();
  return cudaGetLastError();
}

template <>
cudaError_t launch_x_c2r<double>(const Geom& G, const Tables<double>& tb, const cpx<double>* const* in,
                                 const int* deriv, int nf, double* const* out, double scale, const Exec& ex) {
  FxC2RArgs a{};
  for (int i = 0; i < nf; ++i) {
    a.in[i] = in[i];
    a.out[i] = out[i];
    a.deriv[i] = deriv ? deriv[i] : 0;
  }
  // scale is 1 / (Nx Ny): a power of two
  int e = 0;
  frexp(scale, &e);
  dim3 grid, block;
  size_t smem;
  fx_x_config(G, grid, block, smem, nf);
  ex.begin(PK_IO);
  fx_ln(G.lNx, [&](auto ln) {
    k_fx_c2r<decltype(ln)::value><<<grid, block, smem, ex.s>>>(G, tb.twx, a, 1 - e, kTwoPi / G.Lx);
  });
  ex.end();
  return cudaGetLastError();
}

// the column transforms of nf fields in one launch; aly: see k_fx_y
static void fx_y(const Geom& G, const Tables<double>& tb, bool inverse, const FxYArgs& a, int nf, double aly, int plan,
                 int tpb, int kind, const Exec& ex) {
  dim3 grid, block;
  size_t smem;
  fx_y_config(G, grid, block, smem, nf, 0, tpb);
  ex.begin(kind);
  fx_ln(G.lNy, [&](auto ln) {
    constexpr int L = decltype(ln)::value;
    if (inverse)
      k_fx_y<true, L><<<grid, block, smem, ex.s>>>(G, tb.twy, a, aly, plan);
    else
      k_fx_y<false, L><<<grid, block, smem, ex.s>>>(G, tb.twy, a, aly, plan);
  });
  ex.end();
}

template <>
cudaError_t launch_y_fft<double>(const Geom& G, const Tables<double>& tb, bool inverse, const cpx<double>* const* in,
                                 const int* deriv, int nf, cpx<double>* const* out, const Exec& ex) {
  FxYArgs a{};
  for (int i = 0; i < nf; ++i) {
    a.src[i] = in[i];
    a.dst[i] = out[i];
    a.deriv[i] = deriv ? deriv[i] : 0;
  }
  fx_y(G, tb, inverse, a, nf, kTwoPi / G.Ly, 0, 0, PK_IO, ex);
  return cudaGetLastError();
}

template <>
cudaError_t launch_coef_x<double>(const Geom& G, const Tables<double>& tb, const cpx<double>* Hy, double* h,
                                  double* cr, double* cc, int* flags, const CoefCopy& cp, const Exec& ex) {
  dim3 grid, block;
  size_t smem;
  fx_x_config(G, grid, block, smem, 1);
  ex.begin(PK_COEF);
  fx_ln(G.lNx, [&](auto ln) {
    k_fx_coef_x<decltype(ln)::value><<<grid, block, smem, ex.s>>>(G, tb.twx, Hy, h, cr, cc, flags, cp);
  });
  ex.end();
  return cudaGetLastError();
}

// the forward column transforms of NIN inputs and their epilogue
template <int NIN>
static void fx_yfwd(const Geom& G, const Tables<double>& tb, const FxYFwdArgs& a, int pass, int kind, const Exec& ex) {
  dim3 grid, block;
  size_t smem;
  const int plan = ex.plan(TT_F64, pass);
  fx_y_config(G, grid, block, smem, 1, NIN - 1, ex.tpb(TT_F64, pass));
  ex.begin(kind);
  if (fx_parallel(grid, block, NIN)) {
    // a buffer and a stash per transform, slots and scales per group
    const size_t C = block.x / (G.Ny >> 3);
    smem = NIN * C * (2 * (size_t)G.Ny * sizeof(cpx<fx>) + kFxSlots * sizeof(unsigned) + sizeof(cpx<double>));
    k_fx_yfwd<NIN, 0, true><<<grid, NIN * block.x, smem, ex.s>>>(G, tb.twy, a, plan);
  } else {
    fx_ln(G.lNy, [&](auto ln) {
      k_fx_yfwd<NIN, decltype(ln)::value, false><<<grid, block, smem, ex.s>>>(G, tb.twy, a, plan);
    });
  }
  ex.end();
}

template <>
cudaError_t launch_matvec<double>(const Geom& G, const Tables<double>& tb, const cpx<double>* sig, const double* cr,
                                  const double* cc, cpx<double>* w, cpx<double>* const* tmp, bool precond,
                                  const Exec& ex, const int* jsel, size_t jstride, const MvTma*) {
  dim3 grid, block;
  size_t smem;
  FxYArgs a{};
  a.src[0] = a.src[1] = sig;
  a.dst[0] = tmp[0];
  a.dst[1] = tmp[1];
  a.deriv[1] = 1;
  a.sel = jsel;
  a.sel_stride = jstride;
  fx_y(G, tb, true, a, 2, 0.0, ex.plan(TT_F64, TP_MV_YINV), ex.tpb(TT_F64, TP_MV_YINV), PK_MV_YINV, ex);
  fx_x_config(G, grid, block, smem, 1, 10 * (G.Nx >> 3), ex.tpb(TT_F64, TP_MV_X));
  ex.begin(PK_MV_X);
  if (fx_parallel(grid, block, 3)) {
    const int P = (int)block.x / (G.Nx >> 3);
    smem += (size_t)2 * P * (G.Nx * sizeof(cpx<fx>) + kFxSlots * sizeof(unsigned));
    k_fx_mv_x<0, true><<<grid, 3 * block.x, smem, ex.s>>>(G, tb.twx, tb.k2x, tmp[0], tmp[1], cr, cc, tmp[0], tmp[1],
                                                          ex.plan(TT_F64, TP_MV_X));
  } else {
    fx_ln(G.lNx, [&](auto ln) {
      k_fx_mv_x<decltype(ln)::value, false><<<grid, block, smem, ex.s>>>(G, tb.twx, tb.k2x, tmp[0], tmp[1], cr, cc,
                                                                         tmp[0], tmp[1], ex.plan(TT_F64, TP_MV_X));
    });
  }
  ex.end();
  FxYFwdArgs f{};
  f.src[0] = tmp[0];
  f.src[1] = tmp[1];
  f.dst[0] = w;
  f.kr = tb.k2y;
  f.minv = precond ? tb.minv : nullptr;
  fx_yfwd<2>(G, tb, f, TP_MV_YFWD, PK_MV_YFWD, ex);
  return cudaGetLastError();
}

template <>
cudaError_t launch_rhs<double, double>(const Geom& G, const Tables<double>& tb, const Tables<double>& tbs,
                                       cpx<double>* const* U, const cpx<double>* sig, const double* h,
                                       const double* cr, cpx<double>* const* tmp, cpx<double>* const* Un,
                                       cpx<double>* const* Unext, cpx<double>* const* acc,
                                       const cpx<double>* bcur, cpx<double>* bhat, const RkArgs& rk,
                                       const Exec& ex) {
  dim3 grid, block;
  size_t smem;
  FxYArgs a{};
  a.src[0] = U[1];
  a.src[1] = U[2];
  a.src[2] = a.src[3] = sig;
  a.deriv[3] = 1;
  for (int i = 0; i < 4; ++i) a.dst[i] = tmp[i];
  fx_y(G, tb, true, a, 4, 0.0, ex.plan(TT_F64, TP_RHS_YINV), ex.tpb(TT_F64, TP_RHS_YINV), PK_RHS_YINV, ex);
  // each block reads only its own row pair before writing it, so the outputs
  // may overwrite the inputs
  fx_x_config(G, grid, block, smem, 1, 2 * G.Nx, ex.tpb(TT_F64, TP_RHS_X));
  ex.begin(PK_RHS_X);
  const double alx = kTwoPi / G.Lx, aly = kTwoPi / G.Ly;
  const int xplan = ex.plan(TT_F64, TP_RHS_X);
  if (fx_parallel(grid, block, 5, 640)) {
    const size_t P = block.x / (G.Nx >> 3);
    smem = 5 * P * (2 * (size_t)G.Nx * sizeof(cpx<fx>) + kFxSlots * sizeof(unsigned) + sizeof(cpx<double>));
    k_fx_rhs_x<0, true><<<grid, 5 * block.x, smem, ex.s>>>(G, tb.twx, tb.kx, tmp[0], tmp[1], tmp[2], tmp[3], h, cr,
                                                           rk.g, alx, aly, tmp[0], tmp[1], tmp[2], xplan);
  } else {
    fx_ln(G.lNx, [&](auto ln) {
      k_fx_rhs_x<decltype(ln)::value, false><<<grid, block, smem, ex.s>>>(G, tb.twx, tb.kx, tmp[0], tmp[1], tmp[2],
                                                                          tmp[3], h, cr, rk.g, alx, aly, tmp[0],
                                                                          tmp[1], tmp[2], xplan);
    });
  }
  ex.end();
  FxYFwdArgs f{};
  for (int i = 0; i < 3; ++i) f.src[i] = f.dst[i] = tmp[i];
  f.kr = tb.ky;
  f.kx = tb.kx;
  f.dealias = rk.dealias;
  fx_yfwd<3>(G, tb, f, TP_RHS_YFWD, PK_RHS_YFWD, ex);
  return launch_rk_update<double, double>(G, tbs, U, sig, tmp, Un, Unext, acc, bcur, bhat, rk, ex);
}

template cudaError_t launch_coef_phys<double>(const Geom&, const double*, double*, double*, double*, int*,
                                              const CoefCopy&, const Exec&);
template cudaError_t launch_spec_div<double>(const Geom&, const Tables<double>&, const cpx<double>*,
                                             const cpx<double>*, cpx<double>*, const Exec&);
template cudaError_t launch_precond<double>(const Geom&, const Tables<double>&, const cpx<double>*, cpx<double>*,
                                            double*, const Exec&);

}  // namespace sgn
