// 1D contractions of the FP64 form in integer arithmetic.
//
// GB300 executes two FP64 instructions per SM and cycle, but about 14 widening integer multiply-adds
// (32 x 32 + 64 bit), 44 64-bit additions and 64 32-bit logic operations (measured with a throughput
// probe).  The sweeps of the sum factorization only multiply data by the constant 1D tables, so a line
// can be contracted in block floating point: its values become 62-bit integers relative to the line's
// largest exponent, the table entries are 62-bit integers with one scale per operator, a product costs
// three multiply-adds of 32-bit halves, and the sums are integer additions.  The conversions between
// double and integer are shifts and masks; nothing of a line touches the FP64 pipe, which is left to the
// pointwise fluxes.
//
// Error: the inputs are cut at 2^-61 and the tables rounded at 2^-61 of their largest entry (row sum), the
// product of the two low halves (2^-60 at most) and the bits below 2^-58 of (largest input) x (row sum) are
// dropped, and the result is rounded once to 53 bits.  A chain of FP64 multiply-adds rounds every partial
// sum at 2^-53.  The result is therefore closer to the exact sum, except in entries far below the line's
// largest value, where the absolute error stays below 2^-57 of that value.  Against 128-bit arithmetic over
// random operators, lengths 2 to 23 and magnitudes spread over 1, 2^6 and 2^20: 4.7e-17 to 5.6e-17 relative
// (2-norm), the FP64 lines 8.1e-17 to 1.4e-16.
//
// Measured with the sweeps of all FP64 kernels (before -> after, per stage): TGV 64^3, k = 3: face kernel
// 30.5 -> 24.6 ms, cell kernel 32.5 -> 21.2 ms; TGV 40^3, k = 5: L(U) 55.8 -> 39.4 ms.
#pragma once
#include <cstdint>

namespace dgcns {

// The line's values as integers: value i = F[i] 2^(E - 1075 - SH), |F[i]| < 2^61, E the largest biased exponent.
// NA > 1: the element-wise sum of NA lines (SH leaves room for four).  Returns false when the line needs the
// FP64 path: infinities and NaN, values whose result could leave the normal range, and denormal values.  A line
// of zeros is F = 0 with E in range.
template <int NA>
constexpr int fx_shift() {
  static_assert(NA <= 4, "room for four inputs");
  return NA == 1 ? 8 : 6;
}
template <int NA, int D>
__host__ __device__ __forceinline__ bool fx_load(const double (&x)[NA][D], int64_t (&F)[D], int& E) {
  uint32_t m = 0, any = 0;
  uint32_t hi[NA][D], lo[NA][D];
#pragma unroll
  for (int k = 0; k < NA; ++k)
#pragma unroll
    for (int i = 0; i < D; ++i) {
      uint64_t b;
#ifdef __CUDA_ARCH__
      b = (uint64_t)__double_as_longlong(x[k][i]);
#else
      __builtin_memcpy(&b, &x[k][i], 8);
#endif
      hi[k][i] = (uint32_t)(b >> 32);
      lo[k][i] = (uint32_t)b;
      const uint32_t a = hi[k][i] & 0x7fffffffu;
      m = a > m ? a : m;
      any |= lo[k][i];
    }
  E = (int)(m >> 20);
  if (m == 0 && any == 0) E = 1023;
  if ((uint32_t)(E - 200) > 1600u) return false;
#pragma unroll
  for (int k = 0; k < NA; ++k)
#pragma unroll
    for (int i = 0; i < D; ++i) {
      // (an input of exponent 0, zero or far below the line's range, is shifted out entirely)
      int s = E - (int)((hi[k][i] >> 20) & 0x7ffu);
      s = s < 63 ? s : 63;
      const uint32_t mh = (hi[k][i] & 0xfffffu) | 0x100000u;
      const uint64_t v = ((((uint64_t)mh << 32) | lo[k][i]) << fx_shift<NA>()) >> s;
      const int64_t w = (int32_t)hi[k][i] < 0 ? -(int64_t)v : (int64_t)v;
      F[i] = k == 0 ? w : F[i] + w;
    }
  return true;
}

// a 2^(X - 1086) as a double (rounded to nearest, halves away from zero), X in the range that
// fx_load guarantees: the biased exponent of a when its leading bit is bit 63.
__host__ __device__ __forceinline__ double fx_store(int64_t a, int X) {
  const uint32_t neg = (uint32_t)((uint64_t)a >> 32) & 0x80000000u;
  uint64_t u = a < 0 ? (uint64_t)(-a) : (uint64_t)a;
  uint32_t h = (uint32_t)(u >> 32), l = (uint32_t)u;
  if (h == 0) {  // fewer than 32 significant bits
    h = l;
    l = 0;
    X -= 32;
  }
#ifdef __CUDA_ARCH__
  const int lz = __clz((int)h);
#else
  const int lz = h ? __builtin_clz(h) : 32;
#endif
  u = (((uint64_t)h << 32) | l) << lz;
  const uint64_t r = (u >> 11) + ((u >> 10) & 1u);  // 2^52 <= r <= 2^53: the carry goes into the exponent
  uint64_t b = r + ((uint64_t)(uint32_t)(X - lz - 1) << 52);
  if (h == 0) b = 0;
  b |= (uint64_t)neg << 32;
  double y;
#ifdef __CUDA_ARCH__
  y = __longlong_as_double((long long)b);
#else
  __builtin_memcpy(&y, &b, 8);
#endif
  return y;
}

// Halves of an integer, v = h 2^32 + l with l signed: |h| <= 2^30 for |v| < 2^62.
__host__ __device__ __forceinline__ void fx_split(int64_t v, int32_t& h, int32_t& l) {
  l = (int32_t)(uint32_t)(uint64_t)v;
  h = (int32_t)((uint32_t)((uint64_t)v >> 32) + ((uint32_t)(uint64_t)v >> 31));
}

// What a function that is not inlined cannot see: its pointer is to shared memory (generic loads took 5 % of the
// face kernel's time).
#ifdef __CUDA_ARCH__
#define DGCNS_SHARED(p) __builtin_assume(__isShared(p))
#else
#define DGCNS_SHARED(p)
#endif

struct FxAcc {
  int64_t hh, m;
  __host__ __device__ __forceinline__ void zero() {
    hh = 0;
    m = (int64_t)1 << 31;  // rounds the fold
  }
  __host__ __device__ __forceinline__ void mac(int32_t h, int32_t l, int2 c) {
    hh += (int64_t)h * c.x;
    m += (int64_t)h * c.y;
    m += (int64_t)l * c.x;
  }
  __host__ __device__ __forceinline__ void fold() {
    hh += m >> 32;
    m = (int64_t)1 << 31;
  }
};

// One line through an operator in even-odd form, integers in, raw sums out (units 2^(64 - t) of the input's).
// f: {t, SH}, then the even part A [OH][IH], the odd part B [OH][IH] and the middle column C [OH] as {high, low}
// halves of round(entry 2^t), t the largest scale with (row sum of a half) 2^t <= 2^61.  |sum and difference|
// of two inputs < 2^62, so the high products add up to less than 2^60; the cross products are folded into them
// after every two terms (2 (2^61 + 2^60) and the middle column's share stay below 2^63).
template <int DIN, int DOUT, int SYM>
__host__ __device__ __forceinline__ void fx_core(const int2* __restrict__ f, const int64_t (&F)[DIN], int64_t (&y)[DOUT]) {
  constexpr int IH = DIN / 2, OH = (DOUT + 1) / 2;
  int32_t eh[IH > 0 ? IH : 1], el[IH > 0 ? IH : 1], oh[IH > 0 ? IH : 1], ol[IH > 0 ? IH : 1], mh = 0, ml = 0;
#pragma unroll
  for (int i = 0; i < IH; ++i) {
    fx_split(F[i] + F[DIN - 1 - i], eh[i], el[i]);
    fx_split(F[i] - F[DIN - 1 - i], oh[i], ol[i]);
  }
  if (DIN & 1) fx_split(F[IH], mh, ml);
  const int2* __restrict__ A = f + 1;
  const int2* __restrict__ B = A + OH * IH;
  const int2* __restrict__ C = B + OH * IH;
#pragma unroll
  for (int q = 0; q < OH; ++q) {
    const bool centre = (DOUT & 1) && q == OH - 1;
    const bool need_e = !(centre && SYM < 0), need_o = !(centre && SYM > 0);
    FxAcc e, o;
    e.zero();
    o.zero();
    if ((DIN & 1) && need_e) e.mac(mh, ml, C[q]);
#pragma unroll
    for (int i = 0; i < IH; ++i) {
      if (need_e) e.mac(eh[i], el[i], A[q * IH + i]);
      if (need_o) o.mac(oh[i], ol[i], B[q * IH + i]);
      if ((i & 1) || i == IH - 1) {
        if (need_e) e.fold();
        if (need_o) o.fold();
      }
    }
    if (centre) {
      y[q] = SYM > 0 ? e.hh : o.hh;
    } else {
      y[q] = e.hh + o.hh;
      y[DOUT - 1 - q] = SYM > 0 ? e.hh - o.hh : o.hh - e.hh;
    }
  }
}

// The same from and to doubles, with the line's own exponent.
template <int NA, int DIN, int DOUT, int SYM>
__host__ __device__ __forceinline__ bool fx_line(const int2* __restrict__ f, const double (&x)[NA][DIN],
                                                 double (&y)[DOUT]) {
  int64_t F[DIN], Y[DOUT];
  int E;
  if (!fx_load<NA, DIN>(x, F, E)) return false;
  fx_core<DIN, DOUT, SYM>(f, F, Y);
  const int X = E + 75 - fx_shift<NA>() - f[0].x;
#pragma unroll
  for (int q = 0; q < DOUT; ++q) y[q] = fx_store(Y[q], X);
  return true;
}

// One value as an integer relative to a block's largest exponent E: x = F 2^(E - 1083), |F| < 2^61.
__device__ __forceinline__ int64_t fx_of(double x, int E) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  int s = E - (int)((h >> 20) & 0x7ffu);
  s = s < 63 ? s : 63;
  const uint64_t v = ((((uint64_t)((h & 0xfffffu) | 0x100000u) << 32) | l) << 8) >> s;
  return (int32_t)h < 0 ? -(int64_t)v : (int64_t)v;
}
// What a value adds to its block's maximum, and the exponent of a block from it (a block of zeros takes the lowest,
// so that a sum with another block keeps that block's).
__device__ __forceinline__ uint32_t fx_mag(double x) {
  return ((uint32_t)__double2hiint(x) & 0x7fffffffu) | (__double2loint(x) != 0 ? 1u : 0u);
}
__device__ __forceinline__ int fx_exp(uint32_t m) { return m ? (int)(m >> 20) : 300; }
__device__ __forceinline__ bool fx_exp_ok(uint32_t m) { return m == 0 || (m >> 20) - 300u <= 1400u; }

// ---------------------------------------------------------------------------
// float <-> double on the integer units, bit for bit the hardware conversions (which run on the FP64 pipe, two
// a cycle and SM).  For kernels that do little else: in the operator kernels, where the FP64 pipe has room, the
// extra instructions cost more than the conversions (the k = 3 cell kernel 2.14 -> 2.36 ms, measured).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double f64_of(double x) { return x; }
__device__ __forceinline__ double f64_of(float x) {
  const uint32_t b = __float_as_uint(x), a = b & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u)  // normal: rebias the exponent by 1023 - 127
    return __hiloint2double((int)((b & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(b << 29));
  if (a == 0) return __hiloint2double((int)b, 0);
  return (double)x;
}
template <typename T>
__device__ __forceinline__ T f32_of(double x);
template <>
__device__ __forceinline__ double f32_of<double>(double x) {
  return x;
}
template <>
__device__ __forceinline__ float f32_of<float>(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x), a = h & 0x7fffffffu;
  if (a - 0x38100000u < 0x0fd00000u) {  // the result is normal and cannot overflow
    // exponent and 23 mantissa bits, then round to nearest even on the 29 bits below
    const uint32_t t = ((a - 0x38000000u) << 3) | (l >> 29);
    const uint64_t r = (uint64_t)(l << 3) + 0x7fffffffu + (t & 1u);
    return __uint_as_float((h & 0x80000000u) | (t + (uint32_t)(r >> 32)));
  }
  if ((a | l) == 0) return __uint_as_float(h);
  return (float)x;
}

}  // namespace dgcns
