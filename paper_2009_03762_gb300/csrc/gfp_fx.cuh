// FP64 line transforms in 64-bit block fixed point (sm_103a).
//
// GB300 issues 2 FP64 operations per clock and SM but about 60 64-bit integer additions or 62 32 x 32 -> 64
// multiply-adds (measured), so a transform held in 64-bit integers runs its butterflies an order of
// magnitude faster than one held in doubles: every line is scaled by its own largest exponent and enters with 60 bits
// of it (59 in the x-pass).  The fields stay doubles in memory; a pass converts a line's elements on the way in (fx_from)
// and its results on the way out (fx_to), both with integer instructions.
//
// Measured at 256^3 (FP64 butterflies -> fixed point): x-pass 4.65 -> 1.51 ms, y-pass 1.90 -> 0.53 ms, z-pass
// 5.34 -> 1.91 ms.  The passes are now bound by latency at 18 to 24 warps per SM (about 2 instructions of 4 issued per clock),
// half of the instructions being the conversions.
//
// Ranges: |re|, |im| < 2^60 at the input of a line, so that moduli stay below 2^60.5; a radix-4 layer grows
// them to 2^62.5 < 2^63, and the following layers first scale by 1/4 or 1/2 -- for free where the element takes a
// twiddle (Q62 twiddles, the product's upper 64 bits), with a rounded shift otherwise.  fx_shift counts the scaling, and
// fx_to folds it into the exponent.
//
// Precision: scaled down by S = fx_shift bits in all, a line ends in units of 2^(S - 60) of its largest element (2^(S - 59) in the
// x-pass), S within 0.3 bits of log2 n at most: 2^-54 at 256 points, 2^-52 at 512 and 729.  A line whose transform spreads over its
// elements grows by sqrt(n) and more and keeps more bits than a double; one that is a single element (the inverse
// transform of one mode) does not grow, and from 512 points on rounds like a double or up to 4 times coarser.
#pragma once
#include "gfp_fxnum.cuh"
#include "gfp_tma.cuh"

namespace gfp {

// a w / 4 (conjugate w with CONJ): the four partial products per part as 32 x 32 -> 64 multiply-adds, low x
// low dropped (below 1/4 unit).  The middle sums stay below 2^63 for |a| <= 2^62.85, |w| <= 2^62.
template <bool CONJ>
__device__ __forceinline__ fx2 fx_cmul(fx2 a, fxw w) {
  const int xl = (int)a.x, yl = (int)a.y, xh = fx_high(a.x), yh = fx_high(a.y);
  const int sh = CONJ ? -w.yh : w.yh, sl = CONJ ? -w.yl : w.yl;
  const int nh = CONJ ? w.yh : -w.yh, nl = CONJ ? w.yl : -w.yl;
  long long m = fx_mad(xh, w.xl, 0x80000000LL), p = fx_mad(xh, sl, 0x80000000LL);
  m = fx_mad(xl, w.xh, m);  p = fx_mad(xl, sh, p);
  m = fx_mad(yh, nl, m);    p = fx_mad(yh, w.xl, p);
  m = fx_mad(yl, nh, m);    p = fx_mad(yl, w.xh, p);
  fx2 r;
  r.x = fx_mad(yh, nh, fx_mad(xh, w.xh, m >> 32));
  r.y = fx_mad(yh, w.xh, fx_mad(xh, sh, p >> 32));
  return r;
}

// Shift by S bits, rounded, ties to even.  (Truncation would leave half a unit of bias on every element, and ties rounded up an
// eighth to a quarter, which the following transforms gather in a few outputs: at 256^3, with a spectrum that falls like
// 1/k^2, 18 times the rms error beside the origin.  The tie's bit costs two instructions: 256^3 iteration 4.46 -> 4.60 ms.)
template <int S>
__device__ __forceinline__ long long fx_shr(long long a) {
  return fx_add(a, ((1LL << (S - 1)) - 1) + (((unsigned)a >> S) & 1u)) >> S;
}
template <int S>
__device__ __forceinline__ fx2 fx_shr(fx2 a) {
  a.x = fx_shr<S>(a.x);
  a.y = fx_shr<S>(a.y);
  return a;
}

// a w scaled by 2^-S (S = 1 or 2).
template <bool INV, int S>
__device__ __forceinline__ fx2 fx_twiddle(fx2 a, fxw w) {
  fx2 r = fx_cmul<INV>(a, w);
  if (S == 1) { r.x = fx_add(r.x, r.x); r.y = fx_add(r.y, r.y); }
  return r;
}

// Small transforms; those of radix 6 to 16 scale by 1/4 between their two layers, radix 18 by 1/8 in all.
template <int RADIX, bool INV> struct FxDft {
  __device__ __forceinline__ static void run(fx2* v) { Dft<RADIX, INV, fx2>::run(v); }
};
template <bool INV> struct FxDft<3, INV> {
  __device__ __forceinline__ static void run(fx2* v) {
    const fx2 t = cadd(v[1], v[2]), d = mul_mi<INV>(csub(v[1], v[2]));
    const fx2 h = fx_shr<1>(t);
    const fx2 m = csub(v[0], h);
    // sqrt(3)/2 d: the constant as 2^63 sqrt(3)/2 = ch 2^32 + cl, the product's upper half doubled
    constexpr int ch = 1859775393, cl = 1630710223;
    auto mul = [&](long long a) {
      const int l = (int)a, hh = fx_high(a);
      const long long q = fx_mad(l, ch, fx_mad(hh, cl, 0x80000000LL));
      const long long r = fx_mad(hh, ch, q >> 32);
      return fx_add(r, r);
    };
    fx2 s;
    s.x = mul(d.x);
    s.y = mul(d.y);
    v[0] = cadd(v[0], t);
    v[1] = cadd(m, s);
    v[2] = csub(m, s);
  }
};
// cos and sin of pi/8 and pi/4 in Q62, split as fxw
__device__ __forceinline__ fxw fx_w16(int j, bool inv) {
  constexpr int ch[5] = {1 << 30, 992008094, 759250125, 410903207, 0};
  constexpr int cl[5] = {0, 1696238673, -25716447, -1364630830, 0};
  // cos(2 pi j / 16), sin(2 pi j / 16) for j = 0 .. 9 from the first quadrant
  const int jc = j <= 4 ? j : (j <= 8 ? 8 - j : 16 - j), js = j <= 4 ? 4 - j : (j <= 8 ? j - 4 : 12 - j);
  fxw w;
  if (j <= 4) { w.xh = ch[jc]; w.xl = cl[jc]; w.yh = ch[js]; w.yl = cl[js]; }
  else if (j <= 8) { w.xh = -ch[jc]; w.xl = -cl[jc]; w.yh = ch[js]; w.yl = cl[js]; }
  else { w.xh = -ch[j - 8]; w.xl = -cl[j - 8]; w.yh = -ch[12 - j]; w.yl = -cl[12 - j]; }
  if (!inv) { w.yh = -w.yh; w.yl = -w.yl; }
  return w;
}
template <bool INV> struct FxDft<8, INV> {
  __device__ __forceinline__ static void run(fx2* v) {
    fx2 e[4] = {v[0], v[2], v[4], v[6]};
    fx2 o[4] = {v[1], v[3], v[5], v[7]};
    Dft<4, INV, fx2>::run(e);
    Dft<4, INV, fx2>::run(o);
    o[0] = fx_shr<2>(o[0]);
    o[1] = fx_cmul<false>(o[1], fx_w16(2, INV));
    o[2] = fx_shr<2>(mul_mi<INV>(o[2]));
    o[3] = fx_cmul<false>(o[3], fx_w16(6, INV));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const fx2 s = fx_shr<2>(e[k]);
      v[k] = cadd(s, o[k]);
      v[k + 4] = csub(s, o[k]);
    }
  }
};
template <bool INV> struct FxDft<16, INV> {
  __device__ __forceinline__ static void run(fx2* v) {
    // 16 = 4 x 4 as in Dft<16>: columns p, twiddles w16^{p k1}, rows k1; in place, v[p + 4 q] and then
    // v[4 k1 + p] hold the column transforms
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      fx2 y[4] = {v[p], v[p + 4], v[p + 8], v[p + 12]};
      Dft<4, INV, fx2>::run(y);
#pragma unroll
      for (int k1 = 0; k1 < 4; ++k1) {
        const int j = p * k1;
        if (j == 0) v[p + 4 * k1] = fx_shr<2>(y[k1]);
        else if (j == 4) v[p + 4 * k1] = fx_shr<2>(mul_mi<INV>(y[k1]));
        else v[p + 4 * k1] = fx_cmul<false>(y[k1], fx_w16(j, INV));
      }
    }
    fx2 o[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      fx2 z[4] = {v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]};
      Dft<4, INV, fx2>::run(z);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) o[k1 + 4 * k2] = z[k2];
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = o[i];
  }
};

// e^{-+ 2 pi i j / 36} (Q62, split; compile-time j)
__device__ __forceinline__ fxw fx_w36(int j, bool inv) {
  constexpr long long c[10] = {4611686018427387904LL, 4541624145405292212LL, 4333567320897763126LL, 3993837246235628775LL,
                               3532756447825785444LL, 2964334632409774423LL, 2305843009213693952LL, 1577289512995517789LL,
                               800810873071977681LL,  0LL};
  auto cs = [&](int i) -> long long {
    i = (i % 36 + 36) % 36;
    return i <= 9 ? c[i] : (i <= 18 ? -c[18 - i] : (i <= 27 ? -c[i - 18] : c[36 - i]));
  };
  const long long x = cs(j), y = inv ? cs(9 - j) : -cs(9 - j);
  fxw w;
  w.xl = (int)x; w.xh = fx_high(x);
  w.yl = (int)y; w.yh = fx_high(y);
  return w;
}
// As dft_composite, with the elements scaled down by S bits between the layers.
template <int A, int B, bool INV, int S> __device__ __forceinline__ void fx_composite(fx2* v) {
  fx2 y[B][A];
#pragma unroll
  for (int p = 0; p < B; ++p) {
#pragma unroll
    for (int q = 0; q < A; ++q) y[p][q] = v[p + B * q];
    FxDft<A, INV>::run(y[p]);
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    fx2 z[B];
#pragma unroll
    for (int p = 0; p < B; ++p) {
      const int j = 36 / (A * B) * p * k1;
      if (j == 0) z[p] = fx_shr<S>(y[p][k1]);
      else if (j == 9) z[p] = fx_shr<S>(mul_mi<INV>(y[p][k1]));
      else z[p] = fx_twiddle<false, S>(y[p][k1], fx_w36(j, INV));
    }
    FxDft<B, INV>::run(z);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = z[k2];
  }
}
// (moduli from 2^60.5: radix 3 to 2^62.1, / 4, x 3 or x 2; radix 9 leaves 2^61.7, / 2, x 2)
template <bool INV> struct FxDft<6, INV> { __device__ __forceinline__ static void run(fx2* v) { fx_composite<3, 2, INV, 2>(v); } };
template <bool INV> struct FxDft<9, INV> { __device__ __forceinline__ static void run(fx2* v) { fx_composite<3, 3, INV, 2>(v); } };
template <bool INV> struct FxDft<12, INV> { __device__ __forceinline__ static void run(fx2* v) { fx_composite<4, 3, INV, 2>(v); } };
template <bool INV> struct FxDft<18, INV> { __device__ __forceinline__ static void run(fx2* v) { fx_composite<9, 2, INV, 1>(v); } };

// Register plans of the fixed-point transforms.  An element takes four registers, so a thread holds 8 of them (about 80
// registers and 24 warps per SM; 16 elements per thread took 136-176 registers and left the integer pipes waiting), and
// the T threads of a line stay within one warp (512 points: 16 elements).  At 32 and 64 points 4 elements: as many
// instructions per point, twice the threads on grids that are too small to fill the chip (32^3 iteration 51.6 -> 46.3 us).
template <int N> struct FxPlan : CPlan<N> {};
#define GFP_FXPLAN(N_, E_, NST_, R0, R1, R2)                                                        \
  template <> struct FxPlan<N_> {                                                                    \
    static constexpr int N = N_, E = E_, T = N_ / E_, NST = NST_;                                    \
    __host__ __device__ static constexpr int R(int s) { return s == 0 ? R0 : (s == 1 ? R1 : R2); }   \
    __host__ __device__ static constexpr int Ns(int s) { return s == 0 ? 1 : (s == 1 ? R0 : R0 * R1); } \
  };
GFP_FXPLAN(32, 4, 3, 4, 4, 2)
GFP_FXPLAN(64, 4, 3, 4, 4, 4)
GFP_FXPLAN(96, 12, 3, 4, 4, 6)
GFP_FXPLAN(128, 8, 3, 8, 4, 4)
GFP_FXPLAN(192, 12, 3, 12, 4, 4)
GFP_FXPLAN(256, 8, 3, 8, 8, 4)
GFP_FXPLAN(512, 16, 3, 16, 16, 2)
#undef GFP_FXPLAN
template <int N, int S> __device__ __forceinline__ int fin_idx(int t, int b, int r) {
  typedef FxPlan<N> P;
  return t + b * P::T + r * (N / P::R(S));
}
template <int N, int S> __device__ __forceinline__ int fout_idx(int t, int b, int r) {
  typedef FxPlan<N> P;
  constexpr int R = P::R(S), Ns = P::Ns(S);
  const int j = t + b * P::T;
  return (j / Ns) * Ns * R + (j % Ns) + r * Ns;
}

// Bits by which the elements of a register plan are scaled down before the stage that follows one of radix R (other
// schedules: FftPlan::post), and inside a stage of radix R.
__host__ __device__ constexpr int fx_post(int R) { return R == 8 || R == 6 || R == 2 ? 1 : 2; }
__host__ __device__ constexpr int fx_inner(int R) { return R == 18 ? 3 : (R >= 6 ? 2 : 0); }
template <int N> __host__ __device__ constexpr int fx_shift() {
  typedef FxPlan<N> P;
  int s = 0;
  for (int q = 0; q < P::NST; ++q) s += fx_inner(P::R(q)) + (q + 1 < P::NST ? fx_post(P::R(q)) : 0);
  return s;
}
inline __host__ __device__ int fx_shift(const FftPlan& p) {
  int s = 0;
  for (int q = 0; q < p.nst; ++q) s += fx_inner(p.radix[q]) + (int)(p.post >> (2 * q) & 3);
  return s;
}
// A schedule as the FP64 passes run it: merged, and scaled down before each stage by the smaller of 1 and 2 bits that keeps moduli
// below 2^62.85 (tracked in thousandths of a bit, log2 3 = 1.585).  With fx_post everywhere 729 lost 10 bits, now 8: displacements
// of a laminate 1.5 times as far off as in FP64, now 0.5; 864 lost 9, now 8.
inline FftPlan fx_plan(const FftPlan& p) {
  FftPlan m = merge_stages(p);
  int bits = 60500;
  for (int s = 0; s < m.nst; ++s) {
    const int R = m.radix[s];
    const int first = R == 2 ? 1000 : (R % 3 == 0 && R != 12 ? 1585 : 2000);  // growth by the stage's first layer
    if (s > 0) {
      const unsigned down = bits - 1000 + first <= 62850 ? 1 : 2;
      m.post |= down << (2 * (s - 1));
      bits -= 1000 * (int)down;
    }
    const int grow = R == 2 || R == 8 ? 1000 : (R == 3 || R == 12 ? 1585 : (R == 6 ? 585 : (R == 9 || R == 18 ? 1170 : 2000)));
    bits += grow;  // over the stage, less its own fx_inner
  }
  return m;
}

// ------------------------------------------------------------------------------------------------
// Register transforms (lengths with a CPlan); same element order as cfft.
// ------------------------------------------------------------------------------------------------
template <int N, int S, bool INV>
__device__ __forceinline__ void fx_stage(fx2* v, int t, const fxw* __restrict__ tw) {
  typedef FxPlan<N> P;
  constexpr int R = P::R(S), Ns = P::Ns(S), NB = P::E / R, stride = N / (Ns * R);
  constexpr int SH = S > 0 ? fx_post(P::R(S > 0 ? S - 1 : 0)) : 0;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (S > 0) {
      const int k = (t + b * P::T) % Ns;
      v[b * R] = fx_shr<SH ? SH : 1>(v[b * R]);
#pragma unroll
      for (int r = 1; r < R; ++r) v[b * R + r] = fx_twiddle<INV, SH>(v[b * R + r], tw[r * k * stride]);
    }
    FxDft<R, INV>::run(v + b * R);
  }
}
// Exchange between stages; WARP: the line's threads belong to one warp.
template <int N, int S, bool WARP, typename SL>
__device__ __forceinline__ void fx_exchange(fx2* v, SL sm, int t) {
  typedef FxPlan<N> P;
  constexpr int R = P::R(S), R1 = P::R(S + 1);
#pragma unroll
  for (int b = 0; b < P::E / R; ++b)
#pragma unroll
    for (int r = 0; r < R; ++r) sm[fout_idx<N, S>(t, b, r)] = v[b * R + r];
  if (WARP) __syncwarp(); else __syncthreads();
#pragma unroll
  for (int b = 0; b < P::E / R1; ++b)
#pragma unroll
    for (int r = 0; r < R1; ++r) v[b * R1 + r] = sm[fin_idx<N, S + 1>(t, b, r)];
  if (WARP) __syncwarp(); else __syncthreads();
}
template <int N, bool INV, bool WARP, typename SL>
__device__ __forceinline__ void fx_fft(fx2* v, SL sm, int t, const fxw* __restrict__ tw) {
  typedef FxPlan<N> P;
  fx_stage<N, 0, INV>(v, t, tw);
  if constexpr (P::NST > 1) {
    fx_exchange<N, 0, WARP>(v, sm, t);
    fx_stage<N, 1, INV>(v, t, tw);
  }
  if constexpr (P::NST > 2) {
    fx_exchange<N, 1, WARP>(v, sm, t);
    fx_stage<N, 2, INV>(v, t, tw);
  }
}

// One line's transform by the threads of several warps: registers w (doubles, first-stage order) in, doubles in last-stage
// order out; emax[line] is zero on entry.  Synchronises the CTA.
template <int N, bool INV, typename SL>
__device__ __forceinline__ void fx_tile_line(double2* w, SL sl, int t, int line, int* emax, const fxw* twl) {
  typedef FxPlan<N> P;
  atomicMax(&emax[line], fx_max<P::E>(w));
  __syncthreads();
  const FxLine L = fx_line(emax[line]);
  fx2 v[P::E];
  fx_in<60, P::E>(w, v, L);
  fx_fft<N, INV, false>(v, sl, t, twl);
  fx_out<P::E>(v, w, fx_bias<60>(L, fx_shift<N>(), 0), L);
}

__device__ __forceinline__ void fx_prefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// a / 2 without the FP64 pipe; below 2^-1021 zero
__device__ __forceinline__ double fx_half(double a) {
  const int hi = __double2hiint(a), e = hi & 0x7ff00000;
  if (e == 0x7ff00000) return a;
  return e > 0x00100000 ? __hiloint2double(hi - 0x00100000, __double2loint(a)) : 0.0;
}

// ------------------------------------------------------------------------------------------------
// pass_y: CTA = `cols` k1 columns x all n2 rows of one component at fixed k3; thread = (column, t).
// ------------------------------------------------------------------------------------------------
template <int N, bool INV, int COLS>
__global__ void __launch_bounds__(COLS > 0 ? COLS * FxPlan<N>::T : 1024) pass_y_fx_kernel(double2* __restrict__ spec, const fxw* __restrict__ tw,
                                                        Dims d, int cols_arg, const SolveState* __restrict__ st) {
  typedef FxPlan<N> P;
  const int cols = COLS > 0 ? COLS : cols_arg;
  if (st->done && !(INV && st->done == 2)) return;  // as in pass_y_c_kernel
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fxw* twl = reinterpret_cast<fxw*>(smem_raw);
  fx2* buf = reinterpret_cast<fx2*>(twl + N);
  __shared__ int emax[512];
  for (int i = threadIdx.x; i < N; i += blockDim.x) twl[i] = tw[i];
  for (int i = threadIdx.x; i < cols; i += blockDim.x) emax[i] = 0;
  const int col = threadIdx.x % cols, t = threadIdx.x / cols;
  const int k1 = blockIdx.x * cols + col;
  const bool live = k1 < d.n1h;
  double2* g = spec + blockIdx.z * d.S + d.row(blockIdx.y, 0) * d.P + k1;
  const int ys = d.ystride();
  double2 w[P::E];
#pragma unroll
  for (int b = 0; b < P::E / P::R(0); ++b)
#pragma unroll
    for (int r = 0; r < P::R(0); ++r) {
      double2 x = make_double2(0.0, 0.0);
      if (live) x = g[fin_idx<N, 0>(t, b, r) * ys];
      w[b * P::R(0) + r] = x;
    }
  __syncthreads();
  fx_tile_line<N, INV>(w, SLine<fx2, false>{buf + col, cols}, t, col, emax, twl);
  constexpr int RL = P::R(P::NST - 1);
  if (live) {
#pragma unroll
    for (int b = 0; b < P::E / RL; ++b)
#pragma unroll
      for (int r = 0; r < RL; ++r) g[fout_idx<N, P::NST - 1>(t, b, r) * ys] = w[b * RL + r];
  }
}

// ------------------------------------------------------------------------------------------------
// pass_x: CTA = `lines` x1-lines (consecutive i2 at fixed i3) x 3 component pairs; the T threads of a pair
// line belong to one warp.  A thread holds the elements x = t + T j of its line through the inverse
// transform, the update and the forward transform: only the strain's trace crosses threads.  Element j of
// the first stage is register b R0 + r with j = b + r E/R0, of the last stage's output b RL + r with
// j = b + r E/RL.  The half spectrum's two halves meet through shuffles: N - k of thread t's
// k = t + T j is element E - 1 - j of thread T - t (of t = 0: its own element E - j).  Both transforms run through one
// copy of the code (the inverse on swapped real and imaginary parts): two copies overflow the instruction cache.  What the
// update reads is prefetched into L2 during the inverse transform, and factors of two stay off the FP64 pipe (half of its
// time is busy): 256^3 1.53 -> 1.50 ms, 128^3 195 -> 186 us, 64^3 31.9 -> 30.0 us.  Four CTAs per SM at 80 registers, with up to
// 120 bytes of spills, against three at 96: 1.48 ms, 178 us, 25.5 us (1.51 ms with ties to even).
// ------------------------------------------------------------------------------------------------
template <int N> __host__ __device__ constexpr int fx_line_pitch() { return N + N / 16; }

template <int N>
__global__ void __launch_bounds__(192, FxPlan<N>::E <= 8 ? 4 : 2) pass_x_fx_kernel(double2* __restrict__ spec, double* __restrict__ eps,
                                                        const double* __restrict__ lam, const double* __restrict__ mu,
                                                        const fxw* __restrict__ tw, Dims d, int lines, int flags,
                                                        PolarParams pp, const SolveState* __restrict__ st) {
  typedef FxPlan<N> P;
  constexpr int E = P::E, T_ = P::T, EH = E / 2, R0 = P::R(0), RL = P::R(P::NST - 1), LP = fx_line_pitch<N>();
  if (st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  fxw* twl = reinterpret_cast<fxw*>(smem_raw);
  fx2* buf = reinterpret_cast<fx2*>(twl + N);  // one line of LP elements per T threads
  for (int i = threadIdx.x; i < N; i += blockDim.x) twl[i] = tw[i];
  const long long nlines = (long long)d.n2 * d.n3;
  const int t = threadIdx.x % T_, fl = threadIdx.x / T_;  // fl = pair * lines + l
  const bool in = fl < 3 * lines;
  const int p = in ? fl / lines : 2, l = in ? fl % lines : 0;
  const long long li = (long long)blockIdx.x * lines + l;
  const bool live = in && li < nlines;
  const bool zero = (flags & PX_ZERO) != 0 || st->restart;
  const bool have_delta = (flags & PX_DELTA) != 0 && !st->restart;
  const bool outmode = (flags & PX_OUTPUT) != 0, strainmode = (flags & PX_STRAIN) != 0;
  const bool polar = (flags & PX_POLAR) != 0, dres = (flags & PX_DRES) != 0;
  const int partner = (threadIdx.x & 31 & ~(T_ - 1)) | ((T_ - t) & (T_ - 1));
  const SLine<fx2, true> sl{buf + fl * LP, 1};
  // the trace's parts e11 + e22 (pair 0) and e33 (pair 1) of x-line l cross threads through the pair lines' buffers
  double* tr0 = reinterpret_cast<double*>(buf + l * LP);
  double* tr1 = reinterpret_cast<double*>(buf + (lines + l) * LP);
  double2* A = spec + (2 * p) * d.S + d.xrow(live ? li : 0) * d.P + t;
  double2* B = A + d.S;
  const long long v0 = (live ? li : 0) * N + t;
  double* ep = eps + (2 * p) * d.N + v0;
  const double E0 = p == 0 ? pp.E[0] : (p == 1 ? pp.E[2] : pp.E[4]), E1 = p == 0 ? pp.E[1] : (p == 1 ? pp.E[3] : pp.E[5]);
  if (have_delta && live) {  // what the update reads after the inverse transform, on its way into L2
    if (!zero && !outmode)  // (the output mode's eps holds three components)
      for (int i = t; i < N / 8; i += T_) fx_prefetch(eps + (2 * p + (i & 1)) * d.N + li * N + (i >> 1) * 16);
    if (p < 2)
      for (int i = t; i < N / 16; i += T_) fx_prefetch((p ? mu : lam) + li * N + i * 16);
  }
  __syncthreads();
  double2 w[E];  // elements x = t + T j: increment, strain, stress; around the spectrum: A and B at k = t + T j, j < E/2
#pragma unroll 1
  for (int ph = have_delta ? 0 : 1; ph < 2; ++ph) {
    const bool inv = ph == 0;
    double2 ny = make_double2(0.0, 0.0);  // (A, B) at N/2
    if (inv) {
#pragma unroll
      for (int j = 0; j < EH; ++j) {
        w[j] = w[EH + j] = make_double2(0.0, 0.0);
        if (live) { w[j] = A[T_ * j]; w[EH + j] = B[T_ * j]; }
      }
      if (t == 0) w[0].y = w[EH].y = 0.0;  // k = 0 is real
      if (live && t == 0) ny = make_double2(A[N / 2].x, B[N / 2].x);
    } else {
      if (!have_delta) {
#pragma unroll
        for (int j = 0; j < E; ++j) {
          w[j] = make_double2(0.0, 0.0);
          if (live) {
            if (zero) { ep[T_ * j] = 0.0; ep[d.N + T_ * j] = 0.0; }
            else w[j] = make_double2(ep[T_ * j], ep[d.N + T_ * j]);
          }
        }
      }
      if (strainmode) {
#pragma unroll
        for (int j = 0; j < E; ++j) { w[j].x = 0.5 * (w[j].x - E0); w[j].y = 0.5 * (w[j].y - E1); }
      } else {
        if (pp.estar && !polar) {
          const double* es = pp.estar + (2 * p) * d.N + v0;
#pragma unroll
          for (int j = 0; j < E; ++j)
            if (live) { w[j].x -= es[T_ * j]; w[j].y -= es[d.N + T_ * j]; }
        }
        // half the stress, mu e + (lambda / 2) tr e: the factor 2 goes into the exponent of the transform's results
        if (in && p == 0) {
#pragma unroll
          for (int j = 0; j < E; ++j) tr0[t + T_ * j] = w[j].x + w[j].y;
        } else if (in && p == 1) {
#pragma unroll
          for (int j = 0; j < E; ++j) tr1[t + T_ * j] = w[j].x;
        }
        double la[E], m[E];
#pragma unroll
        for (int j = 0; j < E; ++j) {
          m[j] = live ? mu[v0 + T_ * j] : 0.0;
          la[j] = live && p < 2 ? lam[v0 + T_ * j] : 0.0;
        }
        if (polar) {
#pragma unroll
          for (int j = 0; j < E; ++j) { m[j] -= pp.mu_h; la[j] -= pp.lam_h; }
        }
#pragma unroll
        for (int j = 0; j < E; ++j) la[j] = fx_half(la[j]);
        __syncthreads();
        if (p == 2) {
#pragma unroll
          for (int j = 0; j < E; ++j) { w[j].x *= m[j]; w[j].y *= m[j]; }
        } else {
#pragma unroll
          for (int j = 0; j < E; ++j) {
            const double ltr = la[j] * (tr0[t + T_ * j] + tr1[t + T_ * j]);
            w[j].x = m[j] * w[j].x + ltr;
            w[j].y = m[j] * w[j].y + (p == 0 ? ltr : 0.0);
          }
        }
        __syncthreads();  // the exchanges below reuse the buffers
      }
    }
    // 59 bits: the pack and the split add two elements
    int mx = max(fx_max<E>(w), max(fx_mag(ny.x), fx_mag(ny.y)));
#pragma unroll
    for (int o = 1; o < T_; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const FxLine L = fx_line(mx);
    fx2 q[E], v[E];
    if (L.far) {  // (one branch for the elements and the one at N/2)
#pragma unroll
      for (int i = 0; i < E; ++i) { w[i].x *= L.pin; w[i].y *= L.pin; }
      ny.x *= L.pin;
      ny.y *= L.pin;
    }
#pragma unroll
    for (int i = 0; i < E; ++i) { q[i].x = fx_from<59>(w[i].x, L); q[i].y = fx_from<59>(w[i].y, L); }
    if (inv) {
      // the pair's half spectra as one Hermitian-extended line: A + iB at k, conj(A) + i conj(B) at N - k
      fx2 zc[EH], nq;
      nq.x = fx_from<59>(ny.x, L);
      nq.y = fx_from<59>(ny.y, L);
#pragma unroll
      for (int j = 0; j < EH; ++j) {
        const fx2 a = q[j], b = q[EH + j];
        q[j].x = fx_sub(a.x, b.y); q[j].y = fx_add(a.y, b.x);
        zc[j].x = fx_add(a.x, b.y); zc[j].y = fx_sub(b.x, a.y);
      }
#pragma unroll
      for (int j = 0; j < EH; ++j) {
        fx2 c;
        c.x = __shfl_sync(0xffffffffu, zc[j].x, partner);
        c.y = __shfl_sync(0xffffffffu, zc[j].y, partner);
        if (t == 0) c = j + 1 < EH ? zc[j + 1] : nq;  // element E - 1 - j of t = 0 is N - (j + 1) T, or N/2
        q[E - 1 - j] = c;
      }
    }
    // the inverse transform is the forward one between swaps of the parts
#pragma unroll
    for (int j = 0; j < E; ++j) {
      fx2 c = q[j];
      if (inv) { const long long y = c.x; c.x = c.y; c.y = y; }
      v[(j % (E / R0)) * R0 + j / (E / R0)] = c;
    }
    fx_fft<N, false, true>(v, sl, t, twl);
#pragma unroll
    for (int j = 0; j < E; ++j) q[j] = v[(j % (E / RL)) * RL + j / (E / RL)];
    const int bias = fx_bias<59>(L, fx_shift<N>(), 0);
    if (inv) {
#pragma unroll
      for (int j = 0; j < E; ++j) { const long long y = q[j].x; q[j].x = q[j].y; q[j].y = y; }
    } else {
      // split Z = FFT(a + i b) of half the fields: A = Z(k) + conj Z(N - k), B = -i (Z(k) - conj Z(N - k))
      fx2 zn[EH];
#pragma unroll
      for (int j = 0; j < EH; ++j) {
        const fx2 hi = q[E - 1 - j];
        zn[j].x = __shfl_sync(0xffffffffu, hi.x, partner);
        zn[j].y = __shfl_sync(0xffffffffu, hi.y, partner);
        if (t == 0) zn[j] = q[j ? E - j : 0];
      }
      fx2 nq;
      nq.x = fx_add(q[EH].x, q[EH].x);
      nq.y = fx_add(q[EH].y, q[EH].y);
#pragma unroll
      for (int j = 0; j < EH; ++j) {
        const fx2 z = q[j];
        q[j].x = fx_add(z.x, zn[j].x); q[j].y = fx_sub(z.y, zn[j].y);
        q[EH + j].x = fx_add(z.y, zn[j].y); q[EH + j].y = fx_sub(zn[j].x, z.x);
      }
      if (t == 0) ny = make_double2(fx_to(nq.x, bias), fx_to(nq.y, bias));
    }
#pragma unroll
    for (int i = 0; i < E; ++i) w[i] = make_double2(fx_to(q[i].x, bias), fx_to(q[i].y, bias));
    if (L.far) {
#pragma unroll
      for (int i = 0; i < E; ++i) { w[i].x *= L.pout; w[i].y *= L.pout; }
      ny.x *= L.pout;
      ny.y *= L.pout;
    }
    if (inv) {
      if (outmode) {
#pragma unroll
        for (int j = 0; j < E; ++j)
          if (live && p < 2) {
            ep[T_ * j] = w[j].x;
            if (p == 0) ep[d.N + T_ * j] = w[j].y;
          }
        return;
      }
      double2 o[E];
#pragma unroll
      for (int j = 0; j < E; ++j) {
        o[j] = make_double2(0.0, 0.0);
        if (live && !zero) o[j] = make_double2(ep[T_ * j], ep[d.N + T_ * j]);
      }
      const double w0 = p == 2 ? 2.0 : 1.0, w1 = p == 0 ? 1.0 : 2.0;  // shear components count twice
      if (polar) {
        double dacc = 0.0;
#pragma unroll
        for (int j = 0; j < E; ++j) {
          w[j].x += E0;
          w[j].y += E1;
          const double fx = w[j].x - o[j].x, fy = w[j].y - o[j].y;
          dacc += w0 * fx * fx + w1 * fy * fy;
        }
        const double sum = block_sum(live ? dacc : 0.0, red);
        if (threadIdx.x == 0) pp.partials[blockIdx.x] = sum;
      } else {
        if (dres) {
          double dacc = 0.0;
#pragma unroll
          for (int j = 0; j < E; ++j) dacc += w0 * w[j].x * w[j].x + w1 * w[j].y * w[j].y;
          const double sum = block_sum(live ? dacc : 0.0, red);
          if (threadIdx.x == 0) pp.partials[blockIdx.x] = sum;
        }
#pragma unroll
        for (int j = 0; j < E; ++j) { w[j].x += o[j].x; w[j].y += o[j].y; }
      }
      if (live) {
#pragma unroll
        for (int j = 0; j < E; ++j) { ep[T_ * j] = w[j].x; ep[d.N + T_ * j] = w[j].y; }
      }
    } else if (live) {
#pragma unroll
      for (int j = 0; j < EH; ++j) { A[T_ * j] = w[j]; B[T_ * j] = w[EH + j]; }
      if (t == 0) { A[N / 2] = make_double2(ny.x, 0.0); B[N / 2] = make_double2(ny.y, 0.0); }
    }
  }
}

// ------------------------------------------------------------------------------------------------
// pass_z_gamma: CTA = `cols` k1 columns x 6 components x all n3 rows at fixed k2; a thread takes line (comp, col) and
// then (comp + 3, col).  The lines are transformed in registers, meet as doubles in a shared tile for the Green
// step and are transformed back; the tile of 4 columns of 256 takes 104 KB, so that two CTAs share an SM and
// one's FP64 Green step overlaps the other's integer transforms.  TMA: the tile arrives by one TMA load per component
// (bounded wait) instead of ordinary loads.
// ------------------------------------------------------------------------------------------------
// -Gamma0(k) / N applied to a tensor whose product with k is v: with u = a v - (b/2) k (k.v), out_ij = k_i u_j + k_j u_i
// (a = -1 / (2 mu |k|^2 N), b = -c_lm / (|k|^4 N)); 0 where k = 0.
__device__ __forceinline__ void gamma64_from_v(double2 v1, double2 v2, double2 v3, double k1, double k2, double k3,
                                               const GammaParams<double>& gp, double2 o[6]) {
  const double s = k1 * k1 + k2 * k2 + k3 * k3;
  if (s == 0.0) {
#pragma unroll
    for (int c = 0; c < 6; ++c) o[c] = make_double2(0.0, 0.0);
    return;
  }
  const double is = 1.0 / s;
  const double a = -(gp.c_mu * gp.invN) * is, hb = (0.5 * gp.c_lm * gp.invN) * is * is;
  const double gx = hb * (k1 * v1.x + k2 * v2.x + k3 * v3.x), gy = hb * (k1 * v1.y + k2 * v2.y + k3 * v3.y);
  const double2 u1 = make_double2(a * v1.x + k1 * gx, a * v1.y + k1 * gy);
  const double2 u2 = make_double2(a * v2.x + k2 * gx, a * v2.y + k2 * gy);
  const double2 u3 = make_double2(a * v3.x + k3 * gx, a * v3.y + k3 * gy);
  const double d1 = k1 + k1, d2 = k2 + k2, d3 = k3 + k3;
  o[0] = make_double2(d1 * u1.x, d1 * u1.y);
  o[1] = make_double2(d2 * u2.x, d2 * u2.y);
  o[2] = make_double2(d3 * u3.x, d3 * u3.y);
  o[3] = make_double2(k2 * u3.x + k3 * u2.x, k2 * u3.y + k3 * u2.y);
  o[4] = make_double2(k1 * u3.x + k3 * u1.x, k1 * u3.y + k3 * u1.y);
  o[5] = make_double2(k1 * u2.x + k2 * u1.x, k1 * u2.y + k2 * u1.y);
}

// Green step on a tile of all n rows x cols columns (modes as in green_tile): residual partials of the thread, T(0),
// and the increment through put(z, component, column, value) for get(z, component, column).  The z-pass is bound by
// these FP64 operations once its transforms are integer, so the wave vector's products are shared along a column.
template <typename Get, typename Put>
__device__ __forceinline__ void fx_green_points(int n, int cols, int k10, int k2, const Dims& d, const GammaParams<double>& gp,
                                                SolveState* __restrict__ st, int mode, const double2* __restrict__ ab3,
                                                double& acc, double& acc2, Get get, Put put) {
  const int nt = (int)blockDim.x / cols * cols;  // threads beyond the last whole row sit out
  if ((int)threadIdx.x >= nt) return;
  const int cc = threadIdx.x % cols, k1 = k10 + cc;
  const double2 nil = make_double2(0.0, 0.0);
  const bool dead = k1 >= d.n1h;
  const int k1s = dead ? 0 : k1;
  const bool ny1 = ((d.n1 & 1) == 0) && (2 * k1 == d.n1), ny2 = ((d.n2 & 1) == 0) && (2 * k2 == d.n2);
  const bool self1 = (k1 == 0) || ny1;
  const double a1 = gp.A[0][k1s], b1 = gp.B[0][k1s], a2 = gp.A[1][k2], b2 = gp.B[1][k2];
  const double f1 = a1 * b2, f2 = a2 * b1, f3 = b1 * b2;  // kt = (f1 b3, f2 b3, f3 a3)
  for (int z = threadIdx.x / cols; z < n; z += nt / cols) {
    double2 t[6], o[6];
    if (dead) {
#pragma unroll
      for (int c = 0; c < 6; ++c) put(z, c, cc, nil);
      continue;
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) t[c] = get(z, c, cc);
    const double2 ab = ab3 ? ab3[z] : make_double2(gp.A[2][z], gp.B[2][z]);
    const double q1 = f1 * ab.y, q2 = f2 * ab.y, q3 = f3 * ab.x;
    const long long vi = d.row(z, k2) * d.P + k1;
    if (mode == PZ_DISP) {
      disp_point<double>(t, q1, q2, q3, gp.half_shift, d, k1, k2, z, gp.invN, o);
    } else {
      if (k1 == 0 && k2 == 0 && z == 0) {
#pragma unroll
        for (int c = 0; c < 6; ++c) st->T0[c] = t[c].x;
      }
      const bool ny3 = ((n & 1) == 0) && 2 * z == n;
      double2 v1, v2, v3;
      tk_vec<double>(t, q1, q2, q3, v1, v2, v3);
      // residual: the stored point plus (for interior k1) its Hermitian partner, whose wave vector is -kt with the
      // components on Nyquist axes 2, 3 negated back
      double r2 = vnorm2(v1, v2, v3);
      if (!self1) {
        if (gp.nyq_avg && (ny2 || ny3)) r2 += tk_norm2<double>(t, q1, ny2 ? -q2 : q2, ny3 ? -q3 : q3);
        else r2 *= 2.0;
      }
      acc += r2;
      if (mode == PZ_GAMMA && gp.vprev) {
        const double c = incr_point<double>(v1, v2, v3, q1, q2, q3, gp, vi, d.S);
        acc2 += self1 ? c : 2.0 * c;
      }
      if (mode == PZ_DGO) {
        dgo_apply_point<double>(t, gp.dgo, vi, d.S, gp.invN, o);
      } else {
        gamma64_from_v(v1, v2, v3, q1, q2, q3, gp, o);
        if (gp.nyq_avg && (ny1 || ny2 || ny3)) {
          const double p1 = ny1 ? -q1 : q1, p2 = ny2 ? -q2 : q2, p3 = ny3 ? -q3 : q3;
          double2 o2[6];
          tk_vec<double>(t, p1, p2, p3, v1, v2, v3);
          gamma64_from_v(v1, v2, v3, p1, p2, p3, gp, o2);
#pragma unroll
          for (int c = 0; c < 6; ++c) o[c] = make_double2(0.5 * (o[c].x + o2[c].x), 0.5 * (o[c].y + o2[c].y));
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) put(z, c, cc, o[c]);
  }
}

// ------------------------------------------------------------------------------------------------
// The Green step in fixed point, for the schemes with one real wave vector per mode (no Nyquist averaging) and the residual
// stopping rule.  Gamma0 depends on the direction n = kt / |kt| only: with v = T n, p = n.v and
//   u_i = f v_i - c f n_i p,  c = (lambda_H + mu_H) / (lambda_H + 2 mu_H),   out_ij = n_i u_j + n_j u_i,
// out = -Gamma0 T / N up to the power of two in  -1 / (2 mu_H N) = f 2^ef, |f| in [1/2, 1).  In FP64 the step took 122
// operations per point and bound the pass at 2 per clock and SM; here 18 remain (n and the residual).  Each point
// is scaled by its own largest component, so that the products' errors (a few units of 2^-56 of |T|) stay
// below those of FP64.  Points z and N - z share n up to the sign of n3.
// ------------------------------------------------------------------------------------------------
struct FxGreen {
  int fh, fl;    // 2^62 f, split
  int ch, cl;    // -2^62 c f, split (|c| <= 1)
  int ef;
};
__device__ __forceinline__ void fx_split(long long q, int& h, int& l) { l = (int)q; h = fx_high(q); }
__device__ __forceinline__ long long fx_q62(double v) {  // 2^62 v for |v| <= 1
  const int hi = __double2hiint(v), lo = __double2loint(v), ev = (hi >> 20) & 0x7ff;
  unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)lo;
  m <<= 10;
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(1023 - ev));
  const long long s = hi >> 31;
  return (long long)((m ^ (unsigned long long)s) - (unsigned long long)s);
}
// (sum_j a_j w_j) / 4 for split a, w
__device__ __forceinline__ long long fx_dot1(int ah, int al, int wh, int wl) {
  const long long m = fx_mad(al, wh, fx_mad(ah, wl, 0x80000000LL));
  return fx_mad(ah, wh, m >> 32);
}
__device__ __forceinline__ long long fx_dot2(int ah, int al, int wh, int wl, int bh, int bl, int xh, int xl) {
  long long m = fx_mad(al, wh, fx_mad(ah, wl, 0x80000000LL));
  m = fx_mad(bl, xh, fx_mad(bh, xl, m));
  return fx_mad(bh, xh, fx_mad(ah, wh, m >> 32));
}
struct fxs { int h, l; };
__device__ __forceinline__ fxs fx_sp(long long q) { fxs r; fx_split(q, r.h, r.l); return r; }
__device__ __forceinline__ long long fx_dot3(fxs a, fxs b, fxs c, const fxs n[3]) {
  long long m = fx_mad(a.l, n[0].h, fx_mad(a.h, n[0].l, 0x80000000LL));
  m = fx_mad(b.l, n[1].h, fx_mad(b.h, n[1].l, m));
  m = fx_mad(c.l, n[2].h, fx_mad(c.h, n[2].l, m));
  return fx_mad(c.h, n[2].h, fx_mad(b.h, n[1].h, fx_mad(a.h, n[0].h, m >> 32)));
}
__device__ __forceinline__ int fx_absh(long long q) { const int h = (int)(q >> 32); return h ^ (h >> 31); }
__device__ __forceinline__ long long fx_sar(long long q, int d) { asm("shr.s64 %0, %0, %1;" : "+l"(q) : "r"(d)); return q; }
__device__ __forceinline__ long long fx_shl(long long q, int d) { return (long long)((unsigned long long)q << d); }
// q 2^-d, rounded (d >= 1).  Shifts towards minus infinity would leave half a unit of bias on every mode, which the inverse
// transforms gather at the voxels beside the origin (256^3 with a spectrum that falls like 1/k^2: 40 times the rms error there).
__device__ __forceinline__ long long fx_rsar(long long q, int d) { return fx_add(fx_sar(q, d - 1), 1) >> 1; }
// The shift that fills the word: |re|, |im| <= 2^(63 - result); 63 for zero.
__device__ __forceinline__ int fx_lead(fx2 v) { return __clzll((v.x ^ (v.x >> 63)) | (v.y ^ (v.y >> 63))) - 1; }

constexpr int kFxBad = 1 << 28;  // exponent of a line with an infinity or a NaN

// Binary exponent of the unit of a forward line's results (value = q 2^unit).
__device__ __forceinline__ int fx_unit(int hmax, int shift) {
  const FxLine L = fx_line(hmax);
  return hmax >= 0x7ff00000 ? kFxBad : hmax == 0 ? -(1 << 20) : L.e - L.off - 1022 - 60 + shift;
}

// One point: t (units U[c]) -> out, scaled so that its largest part fills 62 bits of a 64-bit integer; returns the point's
// exponent P (unit 2^(P + 10 + ef)) and adds |T kt|^2 for |kt|^2 = s to acc.
__device__ __forceinline__ int fx_green_point(const fx2 t[6], const int U[6], const fxs n[3], double s, double wgt,
                                              const FxGreen& G, double& acc, fx2 o[6]) {
  int zc[6], X = -(1 << 28);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    zc[c] = min(31, __clz(fx_absh(t[c].x) | fx_absh(t[c].y)));
    X = max(X, U[c] - zc[c]);
  }
  fxs a[6][2];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int d = X - (U[c] - zc[c]) + 2;
    a[c][0] = fx_sp(fx_rsar(fx_shl(t[c].x, zc[c] - 1), d));
    a[c][1] = fx_sp(fx_rsar(fx_shl(t[c].y, zc[c] - 1), d));
  }
  const int bias = (63 + min(max(X, -1000), 900) + 5 + 1022) << 20;  // of v, whose unit is 2^(X + 5)
  double r2 = 0.0;
  const int row[3][3] = {{0, 5, 4}, {5, 1, 3}, {4, 3, 2}};
  int m = 0;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    long long v[3];
    fxs vs[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      v[i] = fx_dot3(a[row[i][0]][q], a[row[i][1]][q], a[row[i][2]][q], n);
      vs[i] = fx_sp(v[i]);
      const double vd = fx_to(v[i], bias);
      r2 += vd * vd;
    }
    const long long p = fx_shl(fx_dot3(vs[0], vs[1], vs[2], n), 2);
    const fxs ps = fx_sp(p);
    const fxs pc = fx_sp(fx_shl(fx_dot1(ps.h, ps.l, G.ch, G.cl), 2));
    fxs u[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i] = fx_sp(fx_dot2(vs[i].h, vs[i].l, G.fh, G.fl, pc.h, pc.l, n[i].h, n[i].l));
    long long r[6];
#pragma unroll
    for (int i = 0; i < 3; ++i) r[i] = fx_shl(fx_dot1(u[i].h, u[i].l, n[i].h, n[i].l), 1);
    r[3] = fx_dot2(u[2].h, u[2].l, n[1].h, n[1].l, u[1].h, u[1].l, n[2].h, n[2].l);
    r[4] = fx_dot2(u[2].h, u[2].l, n[0].h, n[0].l, u[0].h, u[0].l, n[2].h, n[2].l);
    r[5] = fx_dot2(u[1].h, u[1].l, n[0].h, n[0].l, u[0].h, u[0].l, n[1].h, n[1].l);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      m |= fx_absh(r[c]);
      if (q == 0) o[c].x = r[c]; else o[c].y = r[c];
    }
  }
  if (X > kFxBad / 2) {
    acc = __hiloint2double(0x7ff80000, 0);
    return kFxBad;
  }
  acc += wgt * (s * r2);
  const int z = min(31, __clz(m));
#pragma unroll
  for (int c = 0; c < 6; ++c) { o[c].x = fx_shl(o[c].x, z - 1); o[c].y = fx_shl(o[c].y, z - 1); }
  return X - z;
}

// All points of a tile: get(z, c, cc) and put(z, c, cc, value) the tile's elements, unit(c, cc) a line's unit, and
// pexp(z, cc) the place of the point's exponent.
template <typename Get, typename Put, typename Unit, typename Pexp>
__device__ __forceinline__ void fx_green_fixed(int n3, int cols, int k10, int k2, const Dims& d, const GammaParams<double>& gp,
                                               const FxGreen& G, SolveState* __restrict__ st, double& acc, Get get,
                                               Put put, Unit unit, Pexp pexp) {
  const int nt = (int)blockDim.x / cols * cols;  // threads beyond the last whole row sit out
  if ((int)threadIdx.x >= nt) return;
  const int cc = threadIdx.x % cols, k1 = k10 + cc;
  if (k1 >= d.n1h) return;  // lines beyond the half spectrum are zero and their results are not written
  const bool self1 = (k1 == 0) || 2 * k1 == d.n1;
  const double a1 = gp.A[0][k1], b1 = gp.B[0][k1], a2 = gp.A[1][k2], b2 = gp.B[1][k2];
  const double f1 = a1 * b2, f2 = a2 * b1, f3 = b1 * b2;  // kt = (f1 b3, f2 b3, f3 a3)
  const double wgt = self1 ? 1.0 : 2.0;  // the stored point and its Hermitian partner
  int U[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) U[c] = unit(c, cc);
  const int half = n3 / 2;
  for (int z = threadIdx.x / cols; z <= half; z += nt / cols) {
    const double a3 = gp.A[2][z], b3 = gp.B[2][z];
    const double q1 = f1 * b3, q2 = f2 * b3, q3 = f3 * a3;
    const double s = q1 * q1 + q2 * q2 + q3 * q3;
    const double rs = s > 0.0 ? rsqrt(s) : 0.0;  // kt = 0 (k = 0 and modes without a wave vector): no increment
    const long long n3q = fx_q62(q3 * rs);
    fxs n[3] = {fx_sp(fx_q62(q1 * rs)), fx_sp(fx_q62(q2 * rs)), fx_sp(n3q)};
    const bool two = z > 0 && 2 * z != n3;  // z and n3 - z differ
#pragma unroll 1
    for (int side = 0; side <= (two ? 1 : 0); ++side) {
      const int zz = side ? n3 - z : z;
      if (side) n[2] = fx_sp(-n3q);
      fx2 t[6], o[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) t[c] = get(zz, c, cc);
      if (k1 == 0 && k2 == 0 && zz == 0) {
#pragma unroll
        for (int c = 0; c < 6; ++c) st->T0[c] = U[c] == kFxBad ? __hiloint2double(0x7ff80000, 0) : scalbn((double)t[c].x, U[c]);
      }
      pexp(zz, cc) = fx_green_point(t, U, n, s, wgt, G, acc, o);
#pragma unroll
      for (int c = 0; c < 6; ++c) put(zz, c, cc, o[c]);
    }
  }
}

// Line scale for the inverse transform, each line's own (with one scale per column of six lines, components that are small
// beside the others lost bits: 64 x 64 x 512, shear increments under an axial load, rms error 4.9e-15 of them, now 1.5e-15;
// z-pass at 256^3 1.91 -> 1.94 ms): an element o of a point with exponent P fills the word shifted left by L = fx_lead(o) and
// then has the exponent P - L; with top the line's largest, elements go in shifted right by top - (P - L) + 3 from there, in the unit 2^(top + 13 + ef).
struct FxBack {
  int bias;
  bool far;
  double pout;
};
__device__ __forceinline__ FxBack fx_back(int top, int ef, int shift) {
  FxBack B;
  int e = 63 + top + 13 + ef + shift + 1022;
  B.pout = 1.0;
  B.far = top < (1 << 27) && top > -(1 << 27) ? (unsigned)(e - 100) > 1800u : top > 0;
  if (B.far) {
    // results outside the doubles' comfortable range are formed 2^800 away and multiplied back; a line that held an
    // infinity or a NaN becomes NaN
    const bool low = e < 1000;
    const bool bad = top >= (1 << 27);
    B.pout = bad ? __hiloint2double(0x7ff80000, 0) : __hiloint2double(low ? (1023 - 800) << 20 : (1023 + 800) << 20, 0);
    e = bad ? 1000 : e + (low ? 800 : -800);
    if (e < 100) { e = 100; B.pout = 0.0; }
  }
  if (top < -(1 << 27)) e = 1000;  // no live point: zeros
  B.bias = e << 20;
  return B;
}

// The z tile in shared memory: [comp][k3][cols] (as TMA delivers it).
struct FxTile {
  double2* base;
  int cols;
  __device__ __forceinline__ double2& at(int n, int z, int c, int cc) const { return base[(c * n + z) * cols + cc]; }
  __device__ __forceinline__ double2* line(int n, int c, int cc) const { return base + c * n * cols + cc; }
  __device__ __forceinline__ int step() const { return cols; }
};

template <int N, int COLS> struct FxZBound {
  static constexpr int threads = COLS > 0 ? 3 * COLS * FxPlan<N>::T : 512;
  // registers a thread gets: about 84 for 8 elements per thread, 120 for 12, 160 for 16
  static constexpr int regs = FxPlan<N>::E <= 8 ? 84 : (FxPlan<N>::E <= 12 ? 120 : 160);
  static constexpr int most = 65536 / (threads * regs), blocks = COLS == 0 || most < 1 ? 1 : (most > 8 ? 8 : most);
};
template <int N, int COLS, bool TMA>
__global__ void __launch_bounds__(FxZBound<N, COLS>::threads, FxZBound<N, COLS>::blocks)
pass_z_fx_kernel(const __grid_constant__ CUtensorMap tmap, double2* __restrict__ spec, const fxw* __restrict__ tw, Dims d,
                 int cols_arg, GammaParams<double> gp, double* __restrict__ partials, SolveState* __restrict__ st, int mode,
                 unsigned inject_timeout) {
  typedef FxPlan<N> P;
  const int cols = COLS > 0 ? COLS : cols_arg;
  if (st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // TMA destinations must be 128-byte aligned: the region is aligned by hand (the launch adds 128 bytes)
  unsigned char* base = smem_raw + (TMA ? (128u - (smem_u32(smem_raw) & 127u)) & 127u : 0u);
  double2* buf = reinterpret_cast<double2*>(base);
  fxw* twl = reinterpret_cast<fxw*>(buf + 6 * N * cols);
  double2* ab3 = reinterpret_cast<double2*>(twl + N);
  __shared__ double red[32];
  __shared__ int emax[4][64];  // per phase; 3 cols lines
  __shared__ __align__(8) unsigned long long bars[2];
  __shared__ int abort_flag;
  const int w3 = 3 * cols;
  const int l = threadIdx.x % w3, t = threadIdx.x / w3;
  const int comp0 = l / cols, col = l % cols;
  const int k10 = blockIdx.x * cols, k2 = blockIdx.y;
  const bool live = k10 + col < d.n1h;
  if (TMA) {
    if (threadIdx.x == 0) {
      mbar_init(&bars[0], 1);
      mbar_init(&bars[1], 1);  // never arrived at (inject_timeout)
      mbar_fence_init();
      abort_flag = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      constexpr int ZB = N < 256 ? N : 256;
      mbar_expect_tx(&bars[0], (unsigned)(6 * N * cols * sizeof(double2)));
      for (int c = 0; c < 6; ++c)
        for (int z0 = 0; z0 < N; z0 += ZB) tma_load_4d(buf + (c * N + z0) * cols, &tmap, &bars[0], 2 * k10, k2, z0, c);
    }
  }
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    twl[i] = tw[i];
    ab3[i] = make_double2(gp.A[2][i], gp.B[2][i]);
  }
  for (int i = threadIdx.x; i < 4 * w3; i += blockDim.x) emax[i / w3][i % w3] = 0;
  if (TMA) {
    // inject_timeout (tests of failure detection): poll, with a short budget, a barrier nothing arrives at; the
    // tile's loads keep their true byte count, so the drain confirms that they have landed
    if (threadIdx.x == 0) {
      const bool ok = inject_timeout ? mbar_wait_bounded(&bars[1], 0, 1LL << 22) : mbar_wait_bounded(&bars[0], 0);
      if (!ok) {
        abort_flag = 1;
        atomicExch(&st->done, (int)DONE_TIMEOUT);
        mbar_wait_bounded(&bars[0], 0);  // the loads land in this CTA's shared memory: wait (bounded) for them
      }
    }
  }
  __syncthreads();
  if (TMA && abort_flag) return;
  const long long zs = d.zstride();
  constexpr int RL = P::R(P::NST - 1), R0 = P::R(0);
  // phases 0, 1: components 0-2, 3-5 forward; the Green step; phases 2, 3: back (the forward transform between swaps of
  // the parts).  One copy of the transform's code serves the four.
#pragma unroll 1
  for (int ph = 0; ph < 4; ++ph) {
    const bool inv = ph >= 2;
    const int comp = comp0 + 3 * (ph & 1);
    const FxTile tile{buf, cols};
    const SLine<double2, false> sd{tile.line(N, comp, col), tile.step()};
    const SLine<fx2, false> sl{reinterpret_cast<fx2*>(sd.base), sd.es};
    double2* g = spec + comp * d.S + d.row(0, k2) * d.P + k10 + col;
    double2 w[P::E];
#pragma unroll
    for (int b = 0; b < P::E / R0; ++b)
#pragma unroll
      for (int r = 0; r < R0; ++r) {
        const int z = fin_idx<N, 0>(t, b, r);
        double2 x = make_double2(0.0, 0.0);
        if (inv || TMA) x = sd[z];
        else if (live) x = g[z * zs];
        if (inv) { const double y = x.x; x.x = x.y; x.y = y; }
        w[b * R0 + r] = x;
      }
    fx_tile_line<N, false>(w, sl, t, l, emax[ph], twl);
    if (inv) {
#pragma unroll
      for (int b = 0; b < P::E / RL; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r) {
          const double2 x = w[b * RL + r];
          if (live) g[fout_idx<N, P::NST - 1>(t, b, r) * zs] = make_double2(x.y, x.x);
        }
    } else {
#pragma unroll
      for (int b = 0; b < P::E / RL; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r) sd[fout_idx<N, P::NST - 1>(t, b, r)] = w[b * RL + r];
    }
    if (ph == 1) {
      __syncthreads();
      double acc = 0.0, acc2 = 0.0;
      fx_green_points(N, cols, k10, k2, d, gp, st, mode, ab3, acc, acc2,
                      [&](int z, int c, int cc) { return tile.at(N, z, c, cc); },
                      [&](int z, int c, int cc, double2 o) { tile.at(N, z, c, cc) = o; });
      const int cta = blockIdx.y * gridDim.x + blockIdx.x;
      if (gp.vprev) {
        const double s2 = block_sum(acc2, red);
        if (threadIdx.x == 0) gp.cpart[cta] = s2;
        __syncthreads();
      }
      const double s = block_sum(acc, red);  // synchronises the CTA after the Green step's writes
      if (threadIdx.x == 0) partials[cta] = s;
    }
  }
}

// The z-pass with the fixed-point Green step: the tile stays in fixed point from the forward to the inverse transform.
// Shared memory: tile [6][N][cols], twiddles, point exponents [N][cols].
template <int N> __host__ __device__ constexpr size_t fx_z_smem(int cols) {
  return sizeof(fx2) * 6 * (size_t)N * cols + sizeof(fxw) * N + sizeof(int) * (size_t)N * cols;
}
template <int N, int COLS>
__global__ void __launch_bounds__(FxZBound<N, COLS>::threads, FxZBound<N, COLS>::blocks)
pass_z_fxf_kernel(double2* __restrict__ spec, const fxw* __restrict__ tw, Dims d, int cols_arg, GammaParams<double> gp,
                  FxGreen G, double* __restrict__ partials, SolveState* __restrict__ st) {
  typedef FxPlan<N> P;
  constexpr int RL = P::R(P::NST - 1), R0 = P::R(0);
  const int cols = COLS > 0 ? COLS : cols_arg;
  if (st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx2* tile = reinterpret_cast<fx2*>(smem_raw);
  fxw* twl = reinterpret_cast<fxw*>(tile + 6 * N * cols);
  int* pexp = reinterpret_cast<int*>(twl + N);
  __shared__ double red[32];
  __shared__ int emax[2][64], top[2][64];
  const int w3 = 3 * cols;
  const int l = threadIdx.x % w3, t = threadIdx.x / w3;
  const int comp0 = l / cols, col = l % cols;
  const int k10 = blockIdx.x * cols, k2 = blockIdx.y;
  const bool live = k10 + col < d.n1h;
  for (int i = threadIdx.x; i < N; i += blockDim.x) twl[i] = tw[i];
  for (int i = threadIdx.x; i < 2 * w3; i += blockDim.x) {
    emax[i / w3][i % w3] = 0;
    top[i / w3][i % w3] = -(1 << 30);
  }
  const long long zs = d.zstride();
  __syncthreads();
#pragma unroll 1
  for (int ph = 0; ph < 4; ++ph) {
    const bool inv = ph >= 2;
    const int comp = comp0 + 3 * (ph & 1);
    const SLine<fx2, false> sl{tile + comp * N * cols + col, cols};
    double2* g = spec + comp * d.S + d.row(0, k2) * d.P + k10 + col;
    fx2 v[P::E];
    FxBack back = {};
    if (!inv) {
      double2 w[P::E];
#pragma unroll
      for (int b = 0; b < P::E / R0; ++b)
#pragma unroll
        for (int r = 0; r < R0; ++r) {
          w[b * R0 + r] = make_double2(0.0, 0.0);
          if (live) w[b * R0 + r] = g[fin_idx<N, 0>(t, b, r) * zs];
        }
      atomicMax(&emax[ph][l], fx_max<P::E>(w));
      __syncthreads();
      const FxLine L = fx_line(emax[ph][l]);
      fx_in<60, P::E>(w, v, L);
    } else {
      int ex[P::E], mx = -(1 << 30);
#pragma unroll
      for (int b = 0; b < P::E / R0; ++b)
#pragma unroll
        for (int r = 0; r < R0; ++r) {
          const int i = b * R0 + r, z = fin_idx<N, 0>(t, b, r);
          const fx2 x = sl[z];
          const int lead = fx_lead(x);
          ex[i] = pexp[z * cols + col] - lead;
          mx = max(mx, ex[i]);
          v[i].x = fx_shl(x.y, lead);  // the inverse transform is the forward one between swaps of the parts
          v[i].y = fx_shl(x.x, lead);
        }
      atomicMax(&top[ph - 2][l], mx);
      __syncthreads();
      const int tc = top[ph - 2][l];
      back = fx_back(tc, G.ef, fx_shift<N>());
#pragma unroll
      for (int i = 0; i < P::E; ++i) {
        const int sh = tc - ex[i] + 3;
        v[i].x = fx_rsar(v[i].x, sh);
        v[i].y = fx_rsar(v[i].y, sh);
      }
    }
    fx_fft<N, false, false>(v, sl, t, twl);
    if (!inv) {
#pragma unroll
      for (int b = 0; b < P::E / RL; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r) sl[fout_idx<N, P::NST - 1>(t, b, r)] = v[b * RL + r];
    } else if (live) {
      double2 w[P::E];
#pragma unroll
      for (int i = 0; i < P::E; ++i) w[i] = make_double2(fx_to(v[i].y, back.bias), fx_to(v[i].x, back.bias));
      if (back.far) {
#pragma unroll
        for (int i = 0; i < P::E; ++i) { w[i].x *= back.pout; w[i].y *= back.pout; }
      }
#pragma unroll
      for (int b = 0; b < P::E / RL; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r) g[fout_idx<N, P::NST - 1>(t, b, r) * zs] = w[b * RL + r];
    }
    if (ph == 1) {
      __syncthreads();
      double acc = 0.0;
      fx_green_fixed(N, cols, k10, k2, d, gp, G, st, acc,
                     [&](int z, int c, int cc) { return tile[(c * N + z) * cols + cc]; },
                     [&](int z, int c, int cc, fx2 o) { tile[(c * N + z) * cols + cc] = o; },
                     [&](int c, int cc) { return fx_unit(emax[c >= 3][(c >= 3 ? c - 3 : c) * cols + cc], fx_shift<N>()); },
                     [&](int z, int cc) -> int& { return pexp[z * cols + cc]; });
      const double s = block_sum(acc, red);  // synchronises the CTA after the Green step's writes
      if (threadIdx.x == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Lengths 2^a 3^b without a register plan: Stockham stages in shared memory with a runtime radix schedule,
// as fft_lines, on fixed-point lines.
// ------------------------------------------------------------------------------------------------
template <int RADIX, bool INV>
__device__ __forceinline__ void fx_stage_lines(const fx2* __restrict__ src, fx2* __restrict__ dst, const fxw* __restrict__ tw,
                                               int n, int Ns, int post, LineLayout L) {
  const int nb = n / RADIX, total = L.lines * nb, tstride = n / (Ns * RADIX);
  const FastDiv by_line(L.line_fast ? L.lines : nb), by_ns(Ns);
  for (int q = threadIdx.x; q < total; q += blockDim.x) {
    const int hi = by_line.div(q), lo = q - hi * (int)by_line.d;
    const int l = L.line_fast ? lo : hi, j = L.line_fast ? hi : lo;
    const fx2* sb = src + l * L.ls;
    fx2 v[RADIX];
#pragma unroll
    for (int r = 0; r < RADIX; ++r) v[r] = sb[(j + r * nb) * L.es];
    const int jn = by_ns.div(j), k = j - jn * Ns;
    if (post) {
      v[0] = post == 1 ? fx_shr<1>(v[0]) : fx_shr<2>(v[0]);
#pragma unroll
      for (int r = 1; r < RADIX; ++r) {
        v[r] = fx_cmul<INV>(v[r], tw[r * k * tstride]);
        if (post == 1) v[r] = cadd(v[r], v[r]);
      }
    }
    FxDft<RADIX, INV>::run(v);
    fx2* db = dst + l * L.ls;
    const int o = jn * Ns * RADIX + k;
#pragma unroll
    for (int r = 0; r < RADIX; ++r) db[(o + r * Ns) * L.es] = v[r];
  }
  __syncthreads();
}

template <bool INV>
__device__ __forceinline__ fx2* fx_lines(fx2* a, fx2* b, const fxw* tw, const FftPlan& P, LineLayout L) {
  int Ns = 1, post = 0;
  fx2 *src = a, *dst = b;
#pragma unroll 1
  for (int s = 0; s < P.nst; ++s) {
    const int R = P.radix[s];
    switch (R) {
      case 2: fx_stage_lines<2, INV>(src, dst, tw, P.n, Ns, post, L); break;
      case 3: fx_stage_lines<3, INV>(src, dst, tw, P.n, Ns, post, L); break;
      case 4: fx_stage_lines<4, INV>(src, dst, tw, P.n, Ns, post, L); break;
      case 6: fx_stage_lines<6, INV>(src, dst, tw, P.n, Ns, post, L); break;
      case 8: fx_stage_lines<8, INV>(src, dst, tw, P.n, Ns, post, L); break;
      case 9: fx_stage_lines<9, INV>(src, dst, tw, P.n, Ns, post, L); break;
      case 12: fx_stage_lines<12, INV>(src, dst, tw, P.n, Ns, post, L); break;
      case 18: fx_stage_lines<18, INV>(src, dst, tw, P.n, Ns, post, L); break;
      default: fx_stage_lines<16, INV>(src, dst, tw, P.n, Ns, post, L); break;
    }
    Ns *= R;
    post = (int)(P.post >> (2 * s)) & 3;
    fx2* t = src; src = dst; dst = t;
  }
  return src;
}

// Line exponents of a tile of doubles (the caller has zeroed emax and synchronised) and the conversion in
// place to fixed point; returns synchronised.
template <int BITS>
__device__ __forceinline__ void fx_tile_in(double2* buf, int* emax, int n, LineLayout L) {
  const int per = max(1, (int)blockDim.x / L.lines);  // threads per line, each on every per-th element
  const FastDiv by_per(L.line_fast ? L.lines : per), by_n(L.line_fast ? L.lines : n);
  for (int q = threadIdx.x; q < per * L.lines; q += blockDim.x) {
    const int hi = by_per.div(q), lo = q - hi * (int)by_per.d, l = L.line_fast ? lo : hi, c = L.line_fast ? hi : lo;
    int m = 0;
    for (int e = c; e < n; e += per) {
      const double2 w = buf[l * L.ls + e * L.es];
      m = max(m, max(fx_mag(w.x), fx_mag(w.y)));
    }
    atomicMax(&emax[l], m);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < n * L.lines; q += blockDim.x) {
    const int hi = by_n.div(q), lo = q - hi * (int)by_n.d, l = L.line_fast ? lo : hi, e = L.line_fast ? hi : lo;
    const FxLine F = fx_line(emax[l]);
    double2* at = buf + l * L.ls + e * L.es;
    double2 w = *at;
    fx2 v;
    fx_in<BITS, 1>(&w, &v, F);
    *reinterpret_cast<fx2*>(at) = v;
  }
  __syncthreads();
}
__device__ __forceinline__ double2 fx_out(fx2 q, int bias, const FxLine& F) {
  double2 w;
  fx_out<1>(&q, &w, bias, F);
  return w;
}

template <bool INV>
__global__ void __launch_bounds__(512) pass_y_fxg_kernel(double2* __restrict__ spec, const fxw* __restrict__ tw, FftPlan plan,
                                                         Dims d, int cols, const SolveState* __restrict__ st) {
  if (st->done && !(INV && st->done == 2)) return;  // as in pass_y_c_kernel
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fxw* twl = reinterpret_cast<fxw*>(smem_raw);
  double2* buf = reinterpret_cast<double2*>(twl + d.n2);  // [n2][cols], two ping-pong copies
  __shared__ int emax[64];
  const int k10 = blockIdx.x * cols;
  const FastDiv by_cols(cols);
  for (int i = threadIdx.x; i < d.n2; i += blockDim.x) twl[i] = tw[i];
  for (int i = threadIdx.x; i < cols; i += blockDim.x) emax[i] = 0;
  double2* g = spec + blockIdx.z * d.S + d.row(blockIdx.y, 0) * d.P + k10;
  const long long ys = d.ystride();
  for (int i = threadIdx.x; i < d.n2 * cols; i += blockDim.x) {
    const int y = by_cols.div(i), cc = i - y * cols;
    buf[i] = k10 + cc < d.n1h ? g[y * ys + cc] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const LineLayout L{cols, cols, 1, true};
  fx_tile_in<60>(buf, emax, d.n2, L);
  const fx2* r = fx_lines<INV>(reinterpret_cast<fx2*>(buf), reinterpret_cast<fx2*>(buf + d.n2 * cols), twl, plan, L);
  const int sh = fx_shift(plan);
  for (int i = threadIdx.x; i < d.n2 * cols; i += blockDim.x) {
    const int y = by_cols.div(i), cc = i - y * cols;
    if (k10 + cc >= d.n1h) continue;
    const FxLine F = fx_line(emax[cc]);
    g[y * ys + cc] = fx_out(r[i], fx_bias<60>(F, sh, 0), F);
  }
}

__global__ void __launch_bounds__(512) pass_x_fxg_kernel(double2* __restrict__ spec, double* __restrict__ eps,
                                                         const double* __restrict__ lam, const double* __restrict__ mu,
                                                         const fxw* __restrict__ tw, FftPlan plan, Dims d, int lines, int flags,
                                                         PolarParams pp, const SolveState* __restrict__ st) {
  if (st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  __shared__ int emax[2][48];
  fxw* twl = reinterpret_cast<fxw*>(smem_raw);
  double2* bufa = reinterpret_cast<double2*>(twl + d.n1);  // [3 pairs][lines][n1], two ping-pong copies
  double2* bufb = bufa + 3 * lines * d.n1;
  const int n1 = d.n1, n1h = d.n1h, tot = 3 * lines, sh = fx_shift(plan);
  const long long nlines = (long long)d.n2 * d.n3, line0 = (long long)blockIdx.x * lines;
  const bool zero = (flags & PX_ZERO) != 0 || st->restart;
  const bool have_delta = (flags & PX_DELTA) != 0 && !st->restart;
  const bool outmode = (flags & PX_OUTPUT) != 0, strainmode = (flags & PX_STRAIN) != 0;
  const bool polar = (flags & PX_POLAR) != 0, dres = (flags & PX_DRES) != 0;
  const LineLayout L{tot, 1, n1, false};
  const FastDiv by_n(n1), by_h(n1h), by_lines(lines);
  for (int i = threadIdx.x; i < n1; i += blockDim.x) twl[i] = tw[i];
  for (int i = threadIdx.x; i < 2 * tot; i += blockDim.x) emax[i / tot][i % tot] = 0;
  fx2* inc = reinterpret_cast<fx2*>(bufa);
  if (have_delta) {
    for (int i = threadIdx.x; i < tot * n1h; i += blockDim.x) {
      const int pl = by_h.div(i), k = i - pl * n1h, p = by_lines.div(pl), l = pl - p * lines;
      const long long li = line0 + l;
      double2 z0 = make_double2(0.0, 0.0), z1 = z0;
      if (li < nlines) {
        const long long row = d.xrow(li) * d.P;
        double2 a = spec[(2 * p) * d.S + row + k], b = spec[(2 * p + 1) * d.S + row + k];
        if (k == 0 || 2 * k == n1) a.y = b.y = 0.0;
        z0 = make_double2(a.x - b.y, a.y + b.x);    // A + iB at k
        z1 = make_double2(a.x + b.y, -a.y + b.x);   // conj(A) + i conj(B) at n1 - k
      }
      double2* line = bufa + pl * n1;
      line[k] = z0;
      if (k > 0 && 2 * k != n1) line[n1 - k] = z1;
    }
    __syncthreads();
    fx_tile_in<60>(bufa, emax[0], n1, L);
    inc = fx_lines<true>(reinterpret_cast<fx2*>(bufa), reinterpret_cast<fx2*>(bufb), twl, plan, L);
  } else {
    __syncthreads();
  }
  double2* sig = reinterpret_cast<double2*>(inc);
  double dacc = 0.0;
  for (int i = threadIdx.x; i < lines * n1; i += blockDim.x) {
    const int l = by_n.div(i), x = i - l * n1;
    const long long li = line0 + l;
    if (li >= nlines) {
      for (int p = 0; p < 3; ++p) sig[(p * lines + l) * n1 + x] = make_double2(0.0, 0.0);
      continue;
    }
    const long long v = li * n1 + x;
    double e[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) e[c] = zero || outmode ? 0.0 : eps[c * d.N + v];
    if (have_delta) {
      double dd[6];
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        const FxLine F = fx_line(emax[0][p * lines + l]);
        const double2 z = fx_out(inc[(p * lines + l) * n1 + x], fx_bias<60>(F, sh, 0), F);
        dd[2 * p] = z.x;
        dd[2 * p + 1] = z.y;
      }
      if (outmode) {
#pragma unroll
        for (int c = 0; c < 3; ++c) eps[c * d.N + v] = dd[c];
        continue;
      }
      if (polar) dacc += polar_update<double>(e, dd, pp);
      else {
        if (dres) dacc += incr_norm2<double>(dd);
#pragma unroll
        for (int c = 0; c < 6; ++c) e[c] += dd[c];
      }
    }
    if (have_delta || zero) {
#pragma unroll
      for (int c = 0; c < 6; ++c) eps[c * d.N + v] = e[c];
    }
    double2 zz[3];
    if (strainmode) {
#pragma unroll
      for (int p = 0; p < 3; ++p) zz[p] = make_double2(e[2 * p] - pp.E[2 * p], e[2 * p + 1] - pp.E[2 * p + 1]);
    } else if (polar) {
      pack_stress<double>(e, lam[v] - pp.lam_h, mu[v] - pp.mu_h, zz);
    } else {
      if (pp.estar) {
#pragma unroll
        for (int c = 0; c < 6; ++c) e[c] -= pp.estar[c * d.N + v];
      }
      pack_stress<double>(e, lam[v], mu[v], zz);
    }
#pragma unroll
    for (int p = 0; p < 3; ++p) sig[(p * lines + l) * n1 + x] = zz[p];
  }
  if (outmode) return;
  if ((polar || dres) && have_delta) {
    const double sum = block_sum(dacc, red);
    if (threadIdx.x == 0) pp.partials[blockIdx.x] = sum;
  }
  __syncthreads();
  fx_tile_in<59>(sig, emax[1], n1, L);  // one bit less: the split adds two elements
  double2* other = sig == bufa ? bufb : bufa;
  const fx2* Z = fx_lines<false>(reinterpret_cast<fx2*>(sig), reinterpret_cast<fx2*>(other), twl, plan, L);
  for (int i = threadIdx.x; i < tot * n1h; i += blockDim.x) {
    const int pl = by_h.div(i), k = i - pl * n1h, p = by_lines.div(pl), l = pl - p * lines;
    const long long li = line0 + l;
    if (li >= nlines) continue;
    const FxLine F = fx_line(emax[1][pl]);
    const int bias = fx_bias<59>(F, sh, -1);
    const fx2 zk = Z[pl * n1 + k], zn = Z[pl * n1 + (k ? n1 - k : 0)];
    const long long row = d.xrow(li) * d.P;
    fx2 A, B;
    A.x = fx_add(zk.x, zn.x); A.y = fx_sub(zk.y, zn.y);
    B.x = fx_add(zk.y, zn.y); B.y = fx_sub(zn.x, zk.x);
    spec[(2 * p) * d.S + row + k] = fx_out(A, bias, F);
    spec[(2 * p + 1) * d.S + row + k] = fx_out(B, bias, F);
  }
}

// Tile [k3][6][cols] of 16-byte elements, two ping-pong copies.  FIXED: the fixed-point Green step (fx_green_fixed), the tile
// staying in fixed point between the transforms; otherwise the FP64 one, for every mode of the pass.
template <bool FIXED>
__global__ void __launch_bounds__(512) pass_z_fxg_kernel(double2* __restrict__ spec, const fxw* __restrict__ tw, FftPlan plan,
                                                         Dims d, int cols, GammaParams<double> gp, FxGreen G,
                                                         double* __restrict__ partials, SolveState* __restrict__ st, int mode) {
  if (st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = d.n3, w6 = 6 * cols, sh = fx_shift(plan);
  fxw* twl = reinterpret_cast<fxw*>(smem_raw);
  double2* buf = reinterpret_cast<double2*>(twl + n);
  double2* buf2 = buf + n * w6;
  int* pexp = reinterpret_cast<int*>(buf2 + n * w6);  // [n][cols], FIXED only
  __shared__ double red[32];
  __shared__ int emax[2][384];  // largest high words of the lines; back: FIXED their exponents
  const int k10 = blockIdx.x * cols, k2 = blockIdx.y;
  const LineLayout L{w6, w6, 1, true};
  const FastDiv by_cols(cols), by_w6(w6);
  for (int i = threadIdx.x; i < n; i += blockDim.x) twl[i] = tw[i];
  for (int i = threadIdx.x; i < w6; i += blockDim.x) {
    emax[0][i] = 0;
    emax[1][i] = FIXED ? -(1 << 30) : 0;
  }
  for (int i = threadIdx.x; i < n * w6; i += blockDim.x) {
    const int z = by_w6.div(i), line = i - z * w6, comp = by_cols.div(line), k1 = k10 + line - comp * cols;
    buf[i] = k1 < d.n1h ? spec[comp * d.S + d.row(z, k2) * d.P + k1] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  fx_tile_in<60>(buf, emax[0], n, L);
  fx2* r = fx_lines<false>(reinterpret_cast<fx2*>(buf), reinterpret_cast<fx2*>(buf2), twl, plan, L);
  double2* tile = reinterpret_cast<double2*>(r);
  double acc = 0.0, acc2 = 0.0;
  if (FIXED) {
    fx_green_fixed(n, cols, k10, k2, d, gp, G, st, acc,
                   [&](int z, int c, int cc) { return r[(z * 6 + c) * cols + cc]; },
                   [&](int z, int c, int cc, fx2 o) { r[(z * 6 + c) * cols + cc] = o; },
                   [&](int c, int cc) { return fx_unit(emax[0][c * cols + cc], sh); },
                   [&](int z, int cc) -> int& { return pexp[z * cols + cc]; });
  } else {
    fx_green_points(n, cols, k10, k2, d, gp, st, mode, nullptr, acc, acc2,
                    [&](int z, int c, int cc) {
                      const FxLine F = fx_line(emax[0][c * cols + cc]);
                      return fx_out(r[(z * 6 + c) * cols + cc], fx_bias<60>(F, sh, 0), F);
                    },
                    [&](int z, int c, int cc, double2 o) { tile[(z * 6 + c) * cols + cc] = o; });
  }
  const int cta = blockIdx.y * gridDim.x + blockIdx.x;
  if (!FIXED && gp.vprev) {
    const double s2 = block_sum(acc2, red);
    if (threadIdx.x == 0) gp.cpart[cta] = s2;
    __syncthreads();
  }
  const double s = block_sum(acc, red);  // synchronises the CTA after the Green step's writes
  if (threadIdx.x == 0) partials[cta] = s;
  if (FIXED) {
    const int per = max(1, (int)blockDim.x / w6);  // threads per line, as in fx_tile_in
    for (int q = threadIdx.x; q < per * w6; q += blockDim.x) {
      const int c = by_w6.div(q), line = q - c * w6, cc = line - by_cols.div(line) * cols;
      int m = -(1 << 30);
      for (int z = c; z < n; z += per) m = max(m, pexp[z * cols + cc] - fx_lead(r[z * w6 + line]));
      atomicMax(&emax[1][line], m);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n * w6; i += blockDim.x) {
      const int z = by_w6.div(i), line = i - z * w6, cc = line - by_cols.div(line) * cols;
      fx2 v = r[i];
      const int lead = fx_lead(v), down = emax[1][line] - (pexp[z * cols + cc] - lead) + 3;
      v.x = fx_rsar(fx_shl(v.x, lead), down);
      v.y = fx_rsar(fx_shl(v.y, lead), down);
      r[i] = v;
    }
    __syncthreads();
  } else {
    fx_tile_in<60>(tile, emax[1], n, L);
  }
  fx2* other = reinterpret_cast<fx2*>(tile == buf ? buf2 : buf);
  r = fx_lines<true>(r, other, twl, plan, L);
  for (int i = threadIdx.x; i < n * w6; i += blockDim.x) {
    const int z = by_w6.div(i), line = i - z * w6, comp = by_cols.div(line), k1 = k10 + line - comp * cols;
    if (k1 >= d.n1h) continue;
    double2 w;
    if (FIXED) {
      const FxBack B = fx_back(emax[1][line], G.ef, sh);
      w = make_double2(fx_to(r[i].x, B.bias), fx_to(r[i].y, B.bias));
      if (B.far) { w.x *= B.pout; w.y *= B.pout; }
    } else {
      const FxLine F = fx_line(emax[1][line]);
      w = fx_out(r[i], fx_bias<60>(F, sh, 0), F);
    }
    spec[comp * d.S + d.row(z, k2) * d.P + k1] = w;
  }
}

}  // namespace gfp
