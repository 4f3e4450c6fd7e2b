// FP64 outer pass of the mixed-precision solve, evaluated in real space.
//
// After each FP32 inner solve the mixed solve needs, for its FP64 strain, the exact residual
// eta = ||T_check q^b|| / ||T_check(0)||_F and the inner iterations' source v = T_check kt (FP32).
// For every scheme the mixed solve runs (CD, ACD, AHC, AFB/R; Sec. 5.3), T_check(k) q^b(k) has the
// modulus of the transform of a difference stencil applied to the stress in real space:
//   CD    D_j f(x) = [f(x + e_j) - f(x - e_j)] / (2h)                     symbol i sin th_j
//   ACD   D_j f(x) = sum_{s,t = +-1} [f(x + e_j + s e_a + t e_b) - f(x - e_j + s e_a + t e_b)] / (8h)
//                                                                          symbol i sin th_j cos th_a cos th_b
//   AHC, AFB/R (averaged forward differences over the unit cube)
//         D_j f(x) = sum_{a,b in {0,1}} [f(x + e_j + a e_s + b e_t) - f(x + a e_s + b e_t)] / (4h)
//                    symbol e^{i phi} i 2 sin(th_j/2) cos(th_s/2) cos(th_t/2), phi = (th_1 + th_2 + th_3)/2
// with th_r = 2 pi kappa_r / n_r (the index map of eq. FieFouAppTra1D, Nyquist kappa = -n/2).  With
// r_i = sum_j D_j sigma_ij the symbol is c(k) i kt(k), |c| = 1 and common to the three components, so
// by Parseval (unnormalised forward transform) sum_k |T_check(k) kt(k)|^2 = N sum_x |r(x)|^2 and
//   eta = sqrt(N sum_x |r(x)|^2) / ||sum_x sigma(x)||_F,      v(k) = -i conj(c(k)) F[r](k).
// The residual and the mean stress are therefore FP64 sums over the stress in real space, without an
// FP64 transform, and the source comes from an FP32 transform of r: v is stored in FP32 and r carries
// its own scale, so the FP32 transform keeps v's relative accuracy.
#pragma once
#include "gfp_fxnum.cuh"

namespace gfp {

enum { RS_CD = 0, RS_ACD = 1, RS_AFD = 2 };

// Refinement step of the FP64 strain: eps += corr - mean(corr) (skipped while `gate` is done).  Bound by HBM (120 B a
// voxel) once the conversions left the FP64 pipe (2 a clock and SM): 512^3 4.89 -> 3.51 ms.
__global__ void apply_corr64_kernel(double* __restrict__ eps, const float* __restrict__ corr,
                                    const double* __restrict__ cmean, long long N, const SolveState* gate) {
  if (gate && gate->done) return;
  double cm[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) cm[c] = cmean[c];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    float f[6];
    double w[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) f[c] = corr[c * N + i];
#pragma unroll
    for (int c = 0; c < 6; ++c) w[c] = widen(f[c]);
#pragma unroll
    for (int c = 0; c < 6; ++c) eps[c * N + i] += w[c] - cm[c];
  }
}

// Tile of the real-space residual: RX x RY columns marched over RZ planes, one voxel of halo on each
// side (periodic).  A CTA has a thread per point of a halo plane and keeps one plane's stress in
// shared memory.
constexpr int kResTX = 32, kResTY = 8, kResTZ = 16;

// sigma = C : (eps - estar) (FP64), r = D^b sigma rounded to FP32 into rout [3][N], and per CTA the
// FP64 sums part[8 b + 0] = sum |r|^2 and part[8 b + 1 + c] = sum sigma_c over the CTA's voxels.
//
// Each plane is visited once and its part of the next plane's r carried on (M).  Averaged stencils (ACD; AHC and AFB/R): in a
// thread's 2x2 window on plane z, with g_ab = f(x + a, y + b, z), a, b in {-1, 1} (ACD) or {0, 1} (AFD),
//   Qx f = (g10 - g00) + (g11 - g01),  Qy f = (g01 - g00) + (g11 - g10),  P f = g00 + g01 + g10 + g11,
// and D_x f(z) = Qx f(z + lo) + Qx f(z + 1), D_y f likewise, D_z f(z) = P f(z + 1) - P f(z + lo), lo = -1 (ACD) or 0
// (AFD).  So r_1(z) = M_1(z + lo) + S_1(z + 1) with S_1 = Qx s11 + Qy s12 + P s13 and M_1 = Qx s11 + Qy s12 - P s13 (and
// likewise r_2 from s12, s22, s23 and r_3 from s13, s23, s33).  CD: r_1(z) = [dx s11 + dy s12](z) - s13(z - 1) + s13(z + 1).
//
// The stress is formed in FP64 (2 operations per clock and SM) and added in integers: 58 bits below the largest stress the
// CTA has met, rounded, so that the 24 terms of a sum and the 16 planes of a mean stay in range; the error of a term, 2^-59 of
// that stress, is below the rounding of stresses down to 1/64 of it.  The exponent only rises: what is carried is shifted where a plane
// raises it.  With sums in FP64 (18 to 60 operations a voxel) against this: AFB/R 256^3 2.16 -> 0.76 ms, 512^3 17.1 -> 5.96;
// ACD 512^3 15.1 (FP64 stress sums) -> 6.4; CD 512^3 13.0 -> 6.8.
template <int S> struct ResHalo {
  static constexpr int LO = S == RS_AFD ? 0 : 1, HX = kResTX + 1 + LO, HY = kResTY + 1 + LO;
  static constexpr int NT = (HX * HY + 31) / 32 * 32;  // a thread per point of the tile with its halo
};
template <int S, bool EST>
__global__ void __launch_bounds__(ResHalo<S>::NT) residual_fx_kernel(const double* __restrict__ eps, const double* __restrict__ lam,
                                                                     const double* __restrict__ mu,
                                                                     const double* __restrict__ estar, Dims d, double inv_h,
                                                                     float* __restrict__ rout, double* __restrict__ part,
                                                                     const SolveState* gate) {
  if (gate && gate->done) return;
  constexpr int LO = ResHalo<S>::LO, HX = ResHalo<S>::HX, HY = ResHalo<S>::HY, NO = kResTX * kResTY;
  __shared__ long long sg[6][HY * HX];
  __shared__ double red[NO / 32][8];
  __shared__ int top[2];  // largest high word of the stress, by plane parity
  const int n1 = d.n1, n2 = d.n2, n3 = d.n3;
  const long long N = d.N;
  const int x0 = blockIdx.x * kResTX, y0 = blockIdx.y * kResTY, z0 = blockIdx.z * kResTZ, t0 = threadIdx.x;
  // the point this thread loads, and the one it writes: the first NO threads' points are the tile itself, the others' its halo
  int hx, hy;
  if (t0 < NO) {
    hx = LO + t0 % kResTX;
    hy = LO + t0 / kResTX;
  } else {
    const int i = t0 - NO, rows = HY - kResTY;  // whole rows below (LO) and above, then the columns beside the tile
    if (i < rows * HX) {
      hx = i % HX;
      hy = LO && i < HX ? 0 : HY - 1;
    } else {
      const int k = i - rows * HX;
      hx = LO && k % 2 == 0 ? 0 : HX - 1;
      hy = LO + k / (1 + LO);
    }
  }
  const bool load = t0 < HX * HY, inner = t0 < NO;
  const bool col_ok = inner && x0 + hx - LO < n1 && y0 + hy - LO < n2;
  const long long off = load ? (long long)((y0 + hy - LO + n2) % n2) * n1 + (x0 + hx - LO + n1) % n1 : 0;
  const int at = hy * HX + hx;
  const int nz = min(kResTZ, n3 - z0);
  const double sc = (S == RS_AFD ? 0.25 : (S == RS_ACD ? 0.125 : 0.5)) * inv_h;
  const bool sc2 = (__double2hiint(sc) & 0xfffff) == 0 && __double2loint(sc) == 0;  // a power of two
  long long ss[6] = {};
  float rr = 0.f;
  long long M[1 + LO][3] = {};
  int hmax = 0;
  if (t0 < 2) top[t0] = 0;
  __syncthreads();
#pragma unroll 1
  for (int p = -LO; p <= nz; ++p) {  // planes z0 - LO .. z0 + nz
    const int zw = (z0 + p + n3) % n3;
    const long long v = (long long)zw * n1 * n2 + off;
    double e[6], sgm[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) e[c] = eps[c * N + v];
    const double la = lam[v], mv = mu[v];
    if (EST) {
#pragma unroll
      for (int c = 0; c < 6; ++c) e[c] -= estar[c * N + v];
    }
    const double m2 = mv + mv, ltr = la * (e[0] + e[1] + e[2]);
    int m = 0;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      sgm[c] = c < 3 ? m2 * e[c] + ltr : m2 * e[c];
      m = max(m, fx_mag(sgm[c]));
    }
    if (!load) m = 0;
    m = __reduce_max_sync(0xffffffffu, m);
    if ((t0 & 31) == 0) atomicMax(&top[p & 1], m);
    __syncthreads();  // also: the previous plane's window reads are over
    const int old = hmax;
    hmax = max(hmax, top[p & 1]);
    const FxLine L = fx_line(hmax);
    if (hmax > old && old > 0) {
      const FxLine K = fx_line(old);
      const int up = (L.e - L.off) - (K.e - K.off);
#pragma unroll
      for (int q = 0; q <= LO; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) asm("shr.s64 %0, %0, %1;" : "+l"(M[q][c]) : "r"(up));
#pragma unroll
      for (int c = 0; c < 6; ++c) asm("shr.s64 %0, %0, %1;" : "+l"(ss[c]) : "r"(up));
    }
    const bool own = col_ok && p >= 0 && p < nz;
    // (far lines apart: multiplications that are predicated off still occupy the FP64 pipe)
    if (L.far) {
#pragma unroll 1
      for (int c = 0; c < 6; ++c) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 6; ++k) s = c == k ? sgm[k] : s;
        const long long q = fx_round<58>(s * L.pin, L);
        if (load) sg[c][at] = q;
#pragma unroll
        for (int k = 0; k < 6; ++k)
          if (own && c == k) ss[k] += q;
      }
    } else {
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const long long q = fx_round<58>(sgm[c], L);
        if (load) sg[c][at] = q;
        if (own) ss[c] += q;  // at most 16 planes: 2^62
      }
    }
    if (t0 == 0) top[(p + 1) & 1] = 0;  // (its last readers passed the barrier above)
    __syncthreads();
    if (col_ok) {
      long long t[3], s[3];  // components (11, 22, 33, 23, 13, 12) = (0, 1, 2, 3, 4, 5)
      if (S == RS_CD) {
        auto dx = [&](int c) -> long long { return sg[c][at + 1] - sg[c][at - 1]; };
        auto dy = [&](int c) -> long long { return sg[c][at + HX] - sg[c][at - HX]; };
        t[0] = dx(0) + dy(5), t[1] = dx(5) + dy(1), t[2] = dx(4) + dy(3);
        s[0] = sg[4][at], s[1] = sg[3][at], s[2] = sg[2][at];
      } else {
        constexpr int W = 1 + LO;  // the window's step
        const int w0 = at - LO * (HX + 1);
        auto g = [&](int c, int a, int b) -> long long { return sg[c][w0 + W * (b * HX + a)]; };
        const long long qx11 = (g(0, 1, 0) - g(0, 0, 0)) + (g(0, 1, 1) - g(0, 0, 1));
        const long long qy22 = (g(1, 0, 1) - g(1, 0, 0)) + (g(1, 1, 1) - g(1, 1, 0));
        const long long p33 = (g(2, 0, 0) + g(2, 0, 1)) + (g(2, 1, 0) + g(2, 1, 1));
        const long long a12 = g(5, 1, 1) - g(5, 0, 0), b12 = g(5, 1, 0) - g(5, 0, 1);
        const long long u13 = g(4, 1, 0) + g(4, 1, 1), w13 = g(4, 0, 0) + g(4, 0, 1);
        const long long u23 = g(3, 0, 1) + g(3, 1, 1), w23 = g(3, 0, 0) + g(3, 1, 0);
        t[0] = qx11 + (a12 - b12), t[1] = (a12 + b12) + qy22, t[2] = (u13 - w13) + (u23 - w23);
        s[0] = u13 + w13, s[1] = u23 + w23, s[2] = p33;
      }
      if (p >= 1) {  // outputs on plane z0 + p - 1
        const long long v = (long long)(z0 + p - 1) * n1 * n2 + off;
        // value = q 2^(e - off - 1022 - 58) sc
        const int k = L.e - L.off - 1080 + ((__double2hiint(sc) >> 20) - 1023);
        const bool near = sc2 && k > -100 && k < 60;
        const float f2 = __int_as_float((k + 127) << 23);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const long long q = M[0][c] + (S == RS_CD ? s[c] : t[c] + s[c]);
          float f;
          if (near) f = __ll2float_rn(q) * f2;
          else f = (float)(scalbn((double)q, L.e - L.off - 1080) * sc);
          if (hmax >= 0x7ff00000) f = __int_as_float(0x7fc00000);
          rout[c * N + v] = f;
          rr += f * f;
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (S == RS_CD) {
          M[0][c] = t[c] - M[LO][c];
          M[LO][c] = s[c];
        } else {
          if (LO) M[0][c] = M[LO][c];
          M[LO][c] = t[c] - s[c];
        }
      }
    }
  }
  // per-CTA sums in a fixed order; the lanes' stress sums in integers, 5 bits lower (57 bits stay)
  const FxLine L = fx_line(hmax);
  double r64 = rr;
#pragma unroll
  for (int off5 = 16; off5 > 0; off5 >>= 1) r64 += __shfl_down_sync(0xffffffffu, r64, off5);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    ss[c] = (ss[c] + 16) >> 5;
#pragma unroll
    for (int off5 = 16; off5 > 0; off5 >>= 1) ss[c] += __shfl_down_sync(0xffffffffu, ss[c], off5);
  }
  if (inner && (t0 & 31) == 0) {
    red[t0 >> 5][0] = r64;
#pragma unroll
    for (int c = 0; c < 6; ++c)
      red[t0 >> 5][1 + c] = hmax >= 0x7ff00000 ? __hiloint2double(0x7ff80000, 0) : scalbn((double)ss[c], L.e - L.off - 1075);
  }
  __syncthreads();
  if (t0 < 7) {
    double sm = 0.0;
    for (int w = 0; w < NO / 32; ++w) sm += red[w][t0];
    const long long b = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    part[8 * b + t0] = sm;
  }
}

// Mean stress of an FP64 strain field with compensated summation: sigma = C : (eps - estar) per voxel.  A thread gathers
// its voxels' stresses with their rounding errors (TwoSum, every addition: sums of several voxels in plain FP64 would round alike
// wherever the stress repeats, as in layers, up to 1.4 units of 2^-53 of the mean); pairs (sum, errors) are combined the same way
// by a warp per component, per CTA into part[12 b + 2 c] and by mean_stress64_final_kernel in a fixed order.  The sum the transform
// forms at k = 0 rounds at about 1e-16 of the mean stress, which is the size of the change one voxel's modulus makes in
// the effective stiffness of a 128^3 cell; this sum keeps the rounding well below it.  FP64 operations bound it (55 a voxel):
// 256^3 1.73 ms (0.82 with groups of four in plain FP64), 32^3 23 us.
struct SumErr {
  double s, e;
  __device__ __forceinline__ void add(double x) {
    const double t = __dadd_rn(s, x), v = t - s;  // (a product x is not to be fused into the sum)
    e += (s - (t - v)) + (x - v);
    s = t;
  }
  __device__ __forceinline__ void add(const SumErr& o) {
    add(o.s);
    e += o.e;
  }
};
__device__ __forceinline__ void warp_sum(SumErr& a) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    SumErr o;
    o.s = __shfl_down_sync(0xffffffffu, a.s, off);
    o.e = __shfl_down_sync(0xffffffffu, a.e, off);
    a.add(o);
  }
}

__global__ void __launch_bounds__(256) mean_stress64_kernel(const double* __restrict__ eps, const double* __restrict__ lam,
                                                          const double* __restrict__ mu, const double* __restrict__ estar,
                                                          long long N, double* __restrict__ part) {
  __shared__ SumErr sh[6][256];
  SumErr a[6] = {};
  const long long step = (long long)gridDim.x * blockDim.x;
  for (long long v0 = blockIdx.x * (long long)blockDim.x + threadIdx.x; v0 < N; v0 += 4 * step) {
    double e[4][6], l[4], m[4];  // four voxels' loads in flight
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long v = v0 + q * step;
      const bool in = v < N;
      l[q] = in ? lam[v] : 0.0;
      m[q] = in ? mu[v] : 0.0;
#pragma unroll
      for (int c = 0; c < 6; ++c) e[q][c] = in ? eps[c * N + v] : 0.0;
      if (estar && in) {
#pragma unroll
        for (int c = 0; c < 6; ++c) e[q][c] -= estar[c * N + v];
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double m2 = 2.0 * m[q], ltr = l[q] * (e[q][0] + e[q][1] + e[q][2]);
#pragma unroll
      for (int c = 0; c < 6; ++c) a[c].add(c < 3 ? m2 * e[q][c] + ltr : m2 * e[q][c]);
    }
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) sh[c][threadIdx.x] = a[c];
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < 6) {  // a warp per component: 13 additions deep, where shuffles of all warps would add 6 x 5 times per warp
    SumErr t = sh[w][lane];
#pragma unroll
    for (int k = 1; k < 8; ++k) t.add(sh[w][lane + 32 * k]);
    warp_sum(t);
    if (lane == 0) {
      part[12 * blockIdx.x + 2 * w] = t.s;
      part[12 * blockIdx.x + 2 * w + 1] = t.e;
    }
  }
}

// Fixed-order combination of the per-CTA pairs, a warp per component: st->T0[c] = sum sigma_c (the transform at k = 0).
__global__ void mean_stress64_final_kernel(const double* __restrict__ part, int nb, SolveState* st) {
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  SumErr a = {0.0, 0.0};
  for (int b = lane; b < nb; b += 32) {
    SumErr o;
    o.s = part[12 * b + 2 * c];
    o.e = part[12 * b + 2 * c + 1];
    a.add(o);
  }
  warp_sum(a);
  if (lane == 0) st->T0[c] = a.s + a.e;
}

// Sum of the per-CTA residual sums in a fixed order: st->T0 = sum sigma (the transform at k = 0) and
// out[0] = N sum |r|^2, the spectral residual sum that reduce_eta turns into eta and the decision.
__global__ void res64_sum_kernel(const double* __restrict__ part, int np, long long N, SolveState* st,
                                 double* __restrict__ out) {
  if (st->done) return;
  __shared__ double sh[7][256];
  double q[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < np; b += blockDim.x) {
#pragma unroll
    for (int k = 0; k < 7; ++k) q[k] += part[8 * b + k];
  }
#pragma unroll
  for (int k = 0; k < 7; ++k) sh[k][threadIdx.x] = q[k];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int k = 0; k < 7; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = (double)N * sh[0][0];
    for (int c = 0; c < 6; ++c) st->T0[c] = sh[1 + c][0];
  }
}

// Forward real-to-complex transform along x1 of the three residual components r [3][N] (FP32) into
// the half spectra v [3][k3][k2][P]: `lines` consecutive x-lines per CTA (even), the same component
// of two neighbouring lines sharing one complex line (a + i b), split after the transform.
__global__ void __launch_bounds__(256) rx_kernel(const float* __restrict__ r, float2* __restrict__ v,
                                                 const float2* __restrict__ tw, FftPlan plan, Dims d, int lines,
                                                 const SolveState* gate) {
  if (gate && gate->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = d.n1, NH = n / 2 + 1, hp = lines / 2, nl = 3 * hp;
  float2* a = reinterpret_cast<float2*>(smem_raw);
  float2* b = a + nl * n;
  const long long nlines = (long long)d.n2 * d.n3;
  const long long line0 = (long long)blockIdx.x * lines;
  const FastDiv by_n(n), by_h(NH), by_hp(hp);
  for (int i = threadIdx.x; i < nl * n; i += blockDim.x) {
    const int q = by_n.div(i), e = i - q * n;
    const int c = by_hp.div(q), p2 = q - c * hp;
    const long long la = line0 + 2 * p2, lb = la + 1;
    float2 z;
    z.x = la < nlines ? r[c * d.N + la * n + e] : 0.f;
    z.y = lb < nlines ? r[c * d.N + lb * n + e] : 0.f;
    a[i] = z;
  }
  __syncthreads();
  LineLayout L{nl, 1, n, false};
  const float2* Z = fft_lines<false>(a, b, tw, plan, L);
  for (int i = threadIdx.x; i < nl * NH; i += blockDim.x) {
    const int q = by_h.div(i), k = i - q * NH;
    const int c = by_hp.div(q), p2 = q - c * hp;
    const long long la = line0 + 2 * p2, lb = la + 1;
    if (la >= nlines) continue;
    const float2 zk = Z[q * n + k], zn = Z[q * n + (k ? n - k : 0)];
    float2 A, B;
    A.x = 0.5f * (zk.x + zn.x); A.y = 0.5f * (zk.y - zn.y);
    B.x = 0.5f * (zk.y + zn.y); B.y = -0.5f * (zk.x - zn.x);
    v[c * d.S + d.xrow(la) * d.P + k] = A;
    if (lb < nlines) v[c * d.S + d.xrow(lb) * d.P + k] = B;
  }
}

// Forward transform along x3 of the three half spectra v, in place, then v <- -i conj(c(k)) v with
// c(k) = ph1[k1] ph2[k2] ph3[k3] the common phase of the stencil symbol (null tables: c = 1).  CTA =
// `cols` k1 columns of one component at fixed k2.
__global__ void __launch_bounds__(256) rz_kernel(float2* __restrict__ v, const float2* __restrict__ tw, FftPlan plan,
                                                 Dims d, int cols, const float2* __restrict__ ph1,
                                                 const float2* __restrict__ ph2, const float2* __restrict__ ph3,
                                                 const SolveState* gate) {
  if (gate && gate->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = d.n3, ls = n + 1;
  float2* a = reinterpret_cast<float2*>(smem_raw);
  float2* b = a + cols * ls;
  const int k10 = blockIdx.x * cols, k2 = blockIdx.y, c = blockIdx.z;
  float2* g = v + c * d.S + d.row(0, k2) * d.P;
  const long long zs = d.zstride();
  const FastDiv by_cols(cols);
  for (int i = threadIdx.x; i < cols * n; i += blockDim.x) {
    const int e = by_cols.div(i), l = i - e * cols;
    float2 z; z.x = 0.f; z.y = 0.f;
    if (k10 + l < d.n1h) z = g[e * zs + k10 + l];
    a[l * ls + e] = z;
  }
  __syncthreads();
  LineLayout L{cols, 1, ls, false};
  const float2* Z = fft_lines<false>(a, b, tw, plan, L);
  float2 p2; p2.x = 1.f; p2.y = 0.f;
  if (ph2) p2 = ph2[k2];
  for (int i = threadIdx.x; i < cols * n; i += blockDim.x) {
    const int e = by_cols.div(i), l = i - e * cols;
    const int k1 = k10 + l;
    if (k1 >= d.n1h) continue;
    float2 z = Z[l * ls + e];
    if (ph1) {
      float2 ph = cmul(cmul(ph1[k1], p2), ph3[e]);
      ph.y = -ph.y;  // conj(c)
      z = cmul(z, ph);
    }
    float2 o; o.x = z.y; o.y = -z.x;  // -i z
    g[e * zs + k1] = o;
  }
}

}  // namespace gfp
