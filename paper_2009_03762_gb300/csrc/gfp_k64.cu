// Launchers of the FP64 hot-path passes (fixed-point line transforms, gfp_fx.cuh).  Grid sizes with a
// register plan use the register kernels; every other 2^a 3^b size the shared-memory Stockham kernels.
#include <cmath>

#include "gfp_fx.cuh"

namespace gfp {

template <> bool cz_tma_ok<double>(int n3, int cols);

namespace {

constexpr int kMaxDynamic = 220 * 1024;  // below the 227 KB opt-in limit, leaving room for static shared memory

template <typename K> cudaError_t opt_in(K* kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynamic);
}

// x-lines per CTA: 3 lines T threads, at most and by default 192 (N = 256: 2 lines, 30 KB), fewer
// while the grid would leave SMs without a CTA.
template <int N> int fx_x_lines(int want, long long nlines) {
  constexpr int T = FxPlan<N>::T;
  const int most = std::min(16, 192 / (3 * T));
  if (want > 0) return std::max(1, std::min(want, most));
  int lines = std::max(1, 64 / T);
  while (lines > 1 && nlines / lines < 304) lines /= 2;
  return lines;
}

template <int N>
void launch_x(cudaStream_t s, int want, double2* spec, double* eps, const double* lam, const double* mu, const fxw* tw,
              const Dims& d, int flags, const PolarParams& pp, const SolveState* st) {
  constexpr int T = FxPlan<N>::T;
  const long long nlines = (long long)d.n2 * d.n3;
  const int lines = fx_x_lines<N>(want, nlines);
  const int threads = (3 * lines * T + 31) / 32 * 32;
  const size_t sm = sizeof(fxw) * N + sizeof(fx2) * (size_t)(threads / T) * fx_line_pitch<N>();
  pass_x_fx_kernel<N><<<(unsigned)((nlines + lines - 1) / lines), threads, sm, s>>>(spec, eps, lam, mu, tw, d, lines, flags, pp,
                                                                                 st);
}

template <int N, bool INV>
void launch_y(cudaStream_t s, int cols, double2* spec, const fxw* tw, const Dims& d, const SolveState* st, int comps) {
  const dim3 grid((d.n1h + cols - 1) / cols, d.n3, comps);
  const size_t sm = 16 * (size_t)(N + N * cols);
  const int th = cols * FxPlan<N>::T;
  if (cols == 8) pass_y_fx_kernel<N, INV, 8><<<grid, th, sm, s>>>(spec, tw, d, cols, st);
  else pass_y_fx_kernel<N, INV, 0><<<grid, th, sm, s>>>(spec, tw, d, cols, st);
}

// Parameters of the fixed-point Green step; false where the FP64 step has to run (Nyquist averaging, the paper's stopping
// rule, the other modes of the pass, or lambda_H so negative that |c| > 1).
bool fx_green_params(const GammaParams<double>& gp, int mode, FxGreen& G) {
  const double c = 0.5 * gp.c_lm / gp.c_mu;  // (lambda_H + mu_H) / (lambda_H + 2 mu_H)
  if (mode != PZ_GAMMA || gp.vprev || gp.nyq_avg || !(std::fabs(c) <= 1.0)) return false;
  const double f = -std::frexp(gp.c_mu * gp.invN, &G.ef);
  auto split = [](double x, int& h, int& l) {
    const long long q = std::llrint(std::ldexp(x, 62));
    l = (int)(unsigned)(q & 0xffffffffll);
    h = (int)((q - (long long)l) >> 32);
  };
  split(f, G.fh, G.fl);
  split(-c * f, G.ch, G.cl);
  return true;
}

template <int N>
void launch_z(cudaStream_t s, const LaunchCfg& lc, double2* spec, const fxw* tw, const Dims& d, const GammaParams<double>& gp,
              double* partials, SolveState* st, int mode) {
  const int cols = lc.z_cols, th = 3 * cols * FxPlan<N>::T;
  const dim3 grid((d.n1h + cols - 1) / cols, d.n2, 1);
  const size_t tables = 2 * sizeof(double2) * (size_t)N;
  const size_t smt = 6 * sizeof(double2) * (size_t)N * cols + tables + 128;
  if ((mode == PZ_GAMMA) && !gp.vprev && lc.z_tma && lc.ztmap && cz_tma_ok<double>(N, cols) && smt <= kMaxDynamic) {
    pass_z_fx_kernel<N, 0, true><<<grid, th, smt, s>>>(*reinterpret_cast<const CUtensorMap*>(lc.ztmap), spec, tw, d, cols, gp,
                                                       partials, st, mode, g_inject_tma_timeout);
    return;
  }
  FxGreen G;
  if (fx_green_params(gp, mode, G)) {
    const size_t smf = fx_z_smem<N>(cols);
    if (cols == 2) pass_z_fxf_kernel<N, 2><<<grid, th, smf, s>>>(spec, tw, d, cols, gp, G, partials, st);
    else if (cols == 4) pass_z_fxf_kernel<N, 4><<<grid, th, smf, s>>>(spec, tw, d, cols, gp, G, partials, st);
    else pass_z_fxf_kernel<N, 0><<<grid, th, smf, s>>>(spec, tw, d, cols, gp, G, partials, st);
    return;
  }
  const CUtensorMap none = {};
  const size_t sm = 6 * sizeof(double2) * (size_t)N * cols + tables;
  if (cols == 2) pass_z_fx_kernel<N, 2, false><<<grid, th, sm, s>>>(none, spec, tw, d, cols, gp, partials, st, mode, 0);
  else if (cols == 4) pass_z_fx_kernel<N, 4, false><<<grid, th, sm, s>>>(none, spec, tw, d, cols, gp, partials, st, mode, 0);
  else pass_z_fx_kernel<N, 0, false><<<grid, th, sm, s>>>(none, spec, tw, d, cols, gp, partials, st, mode, 0);
}

}  // namespace

template <>
cudaError_t Passes<double>::setup() {
  cudaError_t e = opt_in(pass_x_fxg_kernel);
  if (e == cudaSuccess) e = opt_in(pass_y_fxg_kernel<false>);
  if (e == cudaSuccess) e = opt_in(pass_y_fxg_kernel<true>);
  if (e == cudaSuccess) e = opt_in(pass_z_fxg_kernel<false>);
  if (e == cudaSuccess) e = opt_in(pass_z_fxg_kernel<true>);
#define GFP_SET(N)                                                    \
  if (e == cudaSuccess) e = opt_in(pass_x_fx_kernel<N>);              \
  if (e == cudaSuccess) e = opt_in(pass_y_fx_kernel<N, false, 8>);    \
  if (e == cudaSuccess) e = opt_in(pass_y_fx_kernel<N, true, 8>);     \
  if (e == cudaSuccess) e = opt_in(pass_y_fx_kernel<N, false, 0>);    \
  if (e == cudaSuccess) e = opt_in(pass_y_fx_kernel<N, true, 0>);     \
  if (e == cudaSuccess) e = opt_in(pass_z_fx_kernel<N, 0, true>);     \
  if (e == cudaSuccess) e = opt_in(pass_z_fxf_kernel<N, 0>);          \
  if (e == cudaSuccess) e = opt_in(pass_z_fxf_kernel<N, 2>);          \
  if (e == cudaSuccess) e = opt_in(pass_z_fxf_kernel<N, 4>);          \
  if (e == cudaSuccess) e = opt_in(pass_z_fx_kernel<N, 2, false>);    \
  if (e == cudaSuccess) e = opt_in(pass_z_fx_kernel<N, 4, false>);    \
  if (e == cudaSuccess) e = opt_in(pass_z_fx_kernel<N, 0, false>);
  GFP_FOR_CSIZES(GFP_SET)
#undef GFP_SET
  return e;
}

template <>
void Passes<double>::pass_x(cudaStream_t s, const LaunchCfg& lc, double2* spec, double* eps, const double* lam,
                            const double* mu, const fxw* tw, const FftPlan& plan, const Dims& d, int flags,
                            const SolveState* st, const PolarParams* ppp) {
  PolarParams pp = {};
  if (ppp) pp = *ppp;
  switch (d.n1) {
#define GFP_CASE(N) case N: launch_x<N>(s, lc.cx_lines, spec, eps, lam, mu, tw, d, flags, pp, st); return;
    GFP_FOR_CSIZES(GFP_CASE)
#undef GFP_CASE
    default: break;
  }
  const long long nlines = (long long)d.n2 * d.n3;
  const unsigned blocks = (unsigned)((nlines + lc.x_lines - 1) / lc.x_lines);
  const size_t sm = 16 * (size_t)(d.n1 + 6 * lc.x_lines * d.n1);
  pass_x_fxg_kernel<<<blocks, lc.x_threads, sm, s>>>(spec, eps, lam, mu, tw, fx_plan(plan), d, lc.x_lines, flags, pp, st);
}

template <>
void Passes<double>::pass_y(cudaStream_t s, const LaunchCfg& lc, bool inverse, double2* spec, const fxw* tw,
                            const FftPlan& plan, const Dims& d, const SolveState* st, int comps) {
  switch (d.n2) {
#define GFP_CASE(N)                                                      \
    case N:                                                              \
      if (inverse) launch_y<N, true>(s, lc.y_cols, spec, tw, d, st, comps);  \
      else launch_y<N, false>(s, lc.y_cols, spec, tw, d, st, comps);     \
      return;
    GFP_FOR_CSIZES(GFP_CASE)
#undef GFP_CASE
    default: break;
  }
  const dim3 grid((d.n1h + lc.y_cols - 1) / lc.y_cols, d.n3, comps);
  const size_t sm = 16 * (size_t)(d.n2 + 2 * lc.y_cols * d.n2);
  if (inverse) pass_y_fxg_kernel<true><<<grid, lc.y_threads, sm, s>>>(spec, tw, fx_plan(plan), d, lc.y_cols, st);
  else pass_y_fxg_kernel<false><<<grid, lc.y_threads, sm, s>>>(spec, tw, fx_plan(plan), d, lc.y_cols, st);
}

template <>
void Passes<double>::pass_z(cudaStream_t s, const LaunchCfg& lc, double2* spec, const fxw* tw, const FftPlan& plan,
                            const Dims& d, const GammaParams<double>& gp, double* partials, SolveState* st, int mode,
                            float2*) {
  switch (d.n3) {
#define GFP_CASE(N) case N: launch_z<N>(s, lc, spec, tw, d, gp, partials, st, mode); return;
    GFP_FOR_CSIZES(GFP_CASE)
#undef GFP_CASE
    default: break;
  }
  const dim3 grid((d.n1h + lc.z_cols - 1) / lc.z_cols, d.n2, 1);
  const size_t sm = 16 * (size_t)(d.n3 + 12 * lc.z_cols * d.n3);
  FxGreen G;
  if (fx_green_params(gp, mode, G))
    pass_z_fxg_kernel<true><<<grid, lc.z_threads, sm + sizeof(int) * (size_t)(d.n3 * lc.z_cols), s>>>(
        spec, tw, fx_plan(plan), d, lc.z_cols, gp, G, partials, st, mode);
  else
    pass_z_fxg_kernel<false><<<grid, lc.z_threads, sm, s>>>(spec, tw, fx_plan(plan), d, lc.z_cols, gp, G, partials, st, mode);
}

template struct Passes<double>;

// Widths of z tiles, of TMA-fed z tiles and of y tiles.
template <> bool cz_cols_ok<double>(int n3, int cols) {
  if (cols < 1) return false;
  switch (n3) {
#define GFP_CASE(N) case N: return 6 * cols * CPlan<N>::T <= 512;
    GFP_FOR_CSIZES(GFP_CASE)
#undef GFP_CASE
    default: return cols <= 64;
  }
}
template <> bool cz_tma_ok<double>(int n3, int cols) {
  switch (n3) {
#define GFP_CASE(N) case N: return cols >= 1 && 6 * cols * CPlan<N>::T <= 384;
    GFP_FOR_CSIZES(GFP_CASE)
#undef GFP_CASE
    default: return false;
  }
}
template <> int cy_cols_max<double>(int n2) {
  switch (n2) {
#define GFP_CASE(N) case N: return 512 / CPlan<N>::T;
    GFP_FOR_CSIZES(GFP_CASE)
#undef GFP_CASE
    default: return 64;
  }
}

}  // namespace gfp
