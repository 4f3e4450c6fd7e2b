// 64-bit block fixed point: the number and its conversions from and to doubles (sm_103a).  gfp_fx.cuh says why and holds
// the transforms; the real-space residual of gfp_outer.cuh adds in the same form.
#pragma once
#include "gfp_kernels.cuh"

namespace gfp {

struct __align__(16) fx2 { long long x, y; };        // complex, 64-bit fixed point

__device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }
__device__ __forceinline__ long long fx_add(long long a, long long b) { return (long long)((unsigned long long)a + (unsigned long long)b); }
__device__ __forceinline__ long long fx_sub(long long a, long long b) { return (long long)((unsigned long long)a - (unsigned long long)b); }
template <> __device__ __forceinline__ fx2 cadd<fx2>(fx2 a, fx2 b) { fx2 r; r.x = fx_add(a.x, b.x); r.y = fx_add(a.y, b.y); return r; }
template <> __device__ __forceinline__ fx2 csub<fx2>(fx2 a, fx2 b) { fx2 r; r.x = fx_sub(a.x, b.x); r.y = fx_sub(a.y, b.y); return r; }

// High word of a = h 2^32 + l with the low word taken as signed.
__device__ __forceinline__ int fx_high(long long a) { return (int)(a >> 32) + (int)((unsigned)a >> 31); }

// ------------------------------------------------------------------------------------------------
// Conversions.  A line's scale comes from the largest exponent field e of its elements' high words.
// Lines with exponents outside [200, 1800] (beyond 1e-248 .. 1e234, zeros, infinities, NaN) are scaled
// by a power of two on the way in and back on the way out, and lines that hold an infinity or a NaN
// become NaN throughout (FP64 transforms spread them over the line as well).
// ------------------------------------------------------------------------------------------------
struct FxLine {
  int e;           // exponent field the line's elements are scaled to
  bool far;        // multiply by pin = 2^off before the conversion and by pout after it
  int off;
  double pin, pout;
};
__device__ __forceinline__ int fx_mag(double v) { return __double2hiint(v) & 0x7fffffff; }
__device__ __forceinline__ FxLine fx_line(int hmax) {
  FxLine L;
  L.e = hmax >> 20;
  L.far = (unsigned)(L.e - 200) > 1600u;
  L.off = 0;
  L.pin = 1.0;
  L.pout = 1.0;
  if (hmax == 0) {  // zeros (or below 2^-1042): any exponent gives zeros
    L.e = 1000;
    L.far = false;
  }
  if (L.far) {
    const bool low = L.e < 200, bad = L.e == 0x7ff;
    L.pin = __hiloint2double(low ? (1023 + 800) << 20 : (1023 - 800) << 20, 0);
    L.pout = bad ? __hiloint2double(0x7ff80000, 0) : __hiloint2double(low ? (1023 - 800) << 20 : (1023 + 800) << 20, 0);
    L.off = low ? 800 : -800;
    L.e += L.off;
  }
  return L;
}
// v 2^(BITS - 1 - (e - 1023)), truncated: |result| < 2^BITS
template <int BITS>
__device__ __forceinline__ long long fx_from(double v, const FxLine& L) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int ev = (hi >> 20) & 0x7ff;
  const unsigned mh = (hi & 0xfffff) | 0x100000;
  unsigned long long m = ((unsigned long long)mh << 32) | (unsigned)lo;
  m <<= BITS - 53;
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(L.e - ev));  // shifts beyond 63 give 0
  const long long s = hi >> 31;
  return (long long)((m ^ (unsigned long long)s) - (unsigned long long)s);
}
// The same, rounded to the nearest: for long sums, where truncation would add up
template <int BITS>
__device__ __forceinline__ long long fx_round(double v, const FxLine& L) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)lo;
  m <<= BITS + 1 - 53;
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(L.e - ((hi >> 20) & 0x7ff)));
  m = (m + 1) >> 1;
  const long long s = hi >> 31;
  return (long long)((m ^ (unsigned long long)s) - (unsigned long long)s);
}
// (double)f without the FP64 pipe: the fields shifted, denormal numbers normalised first
__device__ __forceinline__ double widen(float f) {
  const bool small = (__float_as_uint(f) & 0x7fffffffu) < 0x00800000u;
  const unsigned b = __float_as_uint(small ? f * 16777216.f : f), a = b & 0x7fffffffu;
  unsigned h = (a >> 3) + (small ? 0x38000000u - (24u << 20) : 0x38000000u);
  if (a == 0) h = 0;
  if (a >= 0x7f800000u) h += 0x38000000u;  // infinity, NaN
  return __hiloint2double((int)((b & 0x80000000u) | h), (int)(b << 29));
}
// Exponent bias of fx_to for a line that was read with BITS bits and scaled down by `shift` bits since,
// times 2^(extra).
template <int BITS>
__device__ __forceinline__ int fx_bias(const FxLine& L, int shift, int extra) {
  // value = q 2^(e - 1023 + 1 - BITS + shift + extra); a leading bit at 63 - n puts the exponent field at
  // 63 - n + e + 1 - BITS + shift + extra, less the implicit bit that the mantissa adds
  return (63 + L.e - BITS + shift + extra) << 20;
}
// Rounded to the nearest double.
__device__ __forceinline__ double fx_to(long long q, int bias) {
  const long long s = q >> 63;
  const unsigned long long u = (unsigned long long)(q ^ s) - (unsigned long long)s;
  const int n = __clzll((long long)u);
  unsigned long long m = u << (n - 1);
  m = (m + 0x200ull) >> 10;
  int hi = (int)(m >> 32) + bias - (n << 20);
  hi = u == 0 ? 0 : hi | ((int)(q >> 32) & 0x80000000);
  return __hiloint2double(hi, (int)m);
}
// K elements in and out (the multiplications of far lines are a branch of their own: predicated off, they would still
// occupy the FP64 pipe).
template <int BITS, int K>
__device__ __forceinline__ void fx_in(double2* w, fx2* v, const FxLine& L) {
  if (L.far) {
#pragma unroll
    for (int i = 0; i < K; ++i) { w[i].x *= L.pin; w[i].y *= L.pin; }
  }
#pragma unroll
  for (int i = 0; i < K; ++i) { v[i].x = fx_from<BITS>(w[i].x, L); v[i].y = fx_from<BITS>(w[i].y, L); }
}
template <int K>
__device__ __forceinline__ int fx_max(const double2* w) {
  int m = 0;
#pragma unroll
  for (int i = 0; i < K; ++i) m = max(m, max(fx_mag(w[i].x), fx_mag(w[i].y)));
  return m;
}
template <int K>
__device__ __forceinline__ void fx_out(const fx2* v, double2* w, int bias, const FxLine& L) {
#pragma unroll
  for (int i = 0; i < K; ++i) w[i] = make_double2(fx_to(v[i].x, bias), fx_to(v[i].y, bias));
  if (L.far) {
#pragma unroll
    for (int i = 0; i < K; ++i) { w[i].x *= L.pout; w[i].y *= L.pout; }
  }
}

}  // namespace gfp
