// fr_fixed.cuh -- block fixed point for the linear operators of the FP64 form.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM against 128 32-bit operations, so the FP64
// pipe bounds the element kernel while the integer pipes idle.  The linear parts of the method (the
// folded derivative, the correction terms, the traces) are contractions with a fixed small matrix;
// they are computed here on integers, exactly up to the operands, cut at 2^-59 of the element's
// largest value in the variable group, and one rounding of the sum at 2^-58 of the largest possible
// sum, against 2^-53 of its terms per operation of a chain of FP64 multiply-adds.  So terms k > 5 binary
// places below the group's largest value have fewer bits than in FP64: elements that span so much in density
// or energy are left to FP64 (fx_low).  A single small momentum is not: its residual holds the pressure, which
// rounds at the larger unit in FP64 as well (one momentum 2^-20 of the others, relative error of its residual
// at 3D p = 3: 6.9e-15 in FP64, 6.1e-15 so).
//
// A value x of an element is the 60-bit integer v = trunc(x 2^(1081 - E)), E the biased exponent of
// the largest magnitude of its group (density, momenta, energy) in the element, so |v| < 2^59.
// An operator entry c is the integer C = round(c 2^k), k the largest exponent at which the sum of
// |C| over the terms of one result stays below 2^61.  Both are held in two limbs,
//   v = vh 2^31 + vl, vh, vl of v's sign, |vl| < 2^31;   C = ch 2^31 + cl, |cl| <= 2^30,
// and a result is H = sum vh ch + (sum (vh cl + vl ch) + 2^30) >> 31: three 32x32+64 multiply-adds
// a term (the product vl cl lies below 2^-58 of the result's range).  Bounds: |sum vh ch| < 2^28 2^30
// and |sum (vh cl + vl ch)| < 2^28 2^30 n + 2^31 2^30 < 2^63 for the n <= 21 terms of any result here.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstring>

namespace frg {

constexpr int FX_GROUPS = 3;      // density, momenta, energy: one exponent each
constexpr int FX_E_MIN = 64;      // smallest group exponent: results never fall below the normal range
constexpr int FX_E_BAD = 2040;    // groups with infinities, NaN or values above 2^1017: results are NaN
constexpr int FX_SUM_BITS = 61;   // log2 of the bound on the sum of |C|
constexpr int FX_SPREAD = 5;      // exponents that a group may span with no fewer bits than FP64

struct FxAcc {
  long long h, m;
};
__host__ __device__ __forceinline__ void fx_mac(FxAcc& a, int2 v, int2 c) {
  a.h += (long long)v.x * c.x;
  a.m += (long long)v.x * c.y;
  a.m += (long long)v.y * c.x;
}
__host__ __device__ __forceinline__ long long fx_sum(const FxAcc& a) {
  return a.h + ((a.m + (1ll << 30)) >> 31);
}

__host__ __device__ __forceinline__ uint64_t fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return uint64_t(__double_as_longlong(x));
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double fx_from_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
// the high word of |x|: these order as the magnitudes, and >> 20 is the biased exponent
__host__ __device__ __forceinline__ uint32_t fx_mag(double x) { return uint32_t(fx_bits(x) >> 32) & 0x7FFFFFFFu; }

// limbs of trunc(x 2^(1081 - E)); |x| < 2^(E - 1022), E >= FX_E_MIN.  The significand with its
// leading one at bit 62 is shifted down by E - e + 4 (e: x's biased exponent); zeros and subnormals
// (e = 0) come out as 0.  (The hardware's conversion to 64-bit integers runs on the FP64 pipe.)
__host__ __device__ __forceinline__ int2 fx_limbs(double x, int E) {
  const uint64_t b = fx_bits(x);
  const int e = int(b >> 52) & 0x7FF;
  const uint64_t m = ((b << 10) & 0x3FFFFFFFFFFFFFFFull) | 0x4000000000000000ull;
  int s = E - e + 4;
  s = s < 63 ? s : 63;
  const uint64_t a = m >> s;
  const int sg = (int(uint32_t(b >> 32)) >> 31) | 1;
  return make_int2(int(a >> 31) * sg, int(uint32_t(a) & 0x7FFFFFFFu) * sg);
}

// v 2^(e - 1023), rounded to nearest (ties away from zero); e: biased exponent of one unit of v,
// at least 1 (and e + 62 below 2047); bad: NaN
__host__ __device__ __forceinline__ double fx_double(long long v, int e, bool bad) {
  const uint64_t s = uint64_t(v >> 63);
  uint64_t a = (uint64_t(v) ^ s) - s;  // below 2^62
#ifdef __CUDA_ARCH__
  const int z = __clzll((long long)a);
#else
  const int z = a ? __builtin_clzll(a) : 64;
#endif
  a <<= (z - 1) & 63;                              // the leading one at bit 62
  a = (a + 0x200) >> 10;                           // ... at bit 52 (a carry moves up)
  uint32_t hi = uint32_t(a >> 32) + (uint32_t(e + 62 - z) << 20);  // it counts one in the exponent field
  hi = v == 0 ? 0u : hi;
  hi |= (uint32_t(s) & 0x80000000u) | (bad ? 0x7FF80000u : 0u);
  return fx_from_bits((uint64_t(hi) << 32) | uint32_t(a));
}

// ---- sums of products of values (flux terms), each operand with its own exponent E ----
// x = v 2^(E - 1082) with 60-bit v (one bit more than the operands of the operator contractions, whose
// sums are longer), limbs v = vh 2^31 + vl with 0 <= vl < 2^31.  All partial products are kept: the sums
// below are in units of 2^(Ev + Ew - 2102 - pk), below 2^62 and wrong by less than 7 units (one for each
// operand cut at its last bit, and the rounding).
constexpr int FX_PK = 2, FX_PK3 = 1;  // pk of the sum of squares and of fx_dot3
constexpr int FX_P_MIN = 542;  // smallest exponent of an operand (2^-481): fx_half_sq's unit is normal
__host__ __device__ __forceinline__ long long fx_value(double x, int E) {
  const uint64_t b = fx_bits(x);
  const int e = int(b >> 52) & 0x7FF;
  const uint64_t m = ((b << 10) & 0x3FFFFFFFFFFFFFFFull) | 0x4000000000000000ull;
  int s = E - e + 3;
  s = s < 63 ? s : 63;
  const long long a = (long long)(m >> s), sg = (long long)b >> 63;
  return (a ^ sg) - sg;
}
__host__ __device__ __forceinline__ int2 fx_split(long long v) {
  return make_int2(int(v >> 31), int(uint32_t(v) & 0x7FFFFFFFu));
}
// a - b limb by limb: the low limbs' difference keeps its sign
__host__ __device__ __forceinline__ int2 fx_diff(int2 a, int2 b) { return make_int2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ int fx_pexp(uint32_t mag) {
  const int e = int(mag >> 20);
  return e < FX_P_MIN ? FX_P_MIN : e;
}
__host__ __device__ __forceinline__ int fx_punit(int Ev, int Ew, int pk) { return Ev + Ew - 1079 - pk; }
// no finite result for certain: an operand that is not finite, or a unit too large for the sum's range
__host__ __device__ __forceinline__ bool fx_pbad(int Ev, int Ew) {
  return Ev >= FX_E_BAD || Ew >= FX_E_BAD || fx_punit(Ev, Ew, FX_PK3) > 2046 - 62;
}
// a b + c d + e f, e a difference of two values (61 bits): |h| <= 2 2^58 + 2^59, |m| <= 4 2^60 + 2^61 +
// 2^60 + 3 2^31 < 2^63
__host__ __device__ __forceinline__ long long fx_dot3(int2 a, int2 b, int2 c, int2 d, int2 e, int2 f) {
  const long long h = (long long)a.x * b.x + (long long)c.x * d.x + (long long)e.x * f.x;
  long long m = (long long)a.x * b.y + (long long)a.y * b.x + (long long)c.x * d.y + (long long)c.y * d.x +
                (long long)e.x * f.y + (long long)e.y * f.x;
  m += (((long long)a.y * b.y) >> 31) + (((long long)c.y * d.y) >> 31) + (((long long)e.y * f.y) >> 31);
  return (h << FX_PK3) + ((m + (1ll << (30 - FX_PK3))) >> (31 - FX_PK3));
}
// sum of n <= 3 squares: h <= 3 2^58, |m| <= 3 2^60 (half of the cross products)
template <int n>
__host__ __device__ __forceinline__ long long fx_sum_sq(const int2* v) {
  long long h = 0, m = 0;
  unsigned long long l = 0;  // below 3 2^62
#pragma unroll
  for (int k = 0; k < n; ++k) {
    h += (long long)v[k].x * v[k].x;
    m += (long long)v[k].x * v[k].y;
    l += (unsigned long long)((long long)v[k].y * v[k].y);
  }
  m += (long long)(l >> 32);
  return (h << FX_PK) + ((m + (1ll << (29 - FX_PK))) >> (30 - FX_PK));
}
// half of it as a double, from limbs of exponent E: halved in its unit
template <int n>
__host__ __device__ __forceinline__ double fx_half_sq(const int2* v, int E) {
  return fx_double(fx_sum_sq<n>(v), fx_punit(E, E, FX_PK) - 1, fx_pbad(E, E));
}

// biased exponent of one unit of a result: values of group exponent E, entries scaled by 2^k
__host__ __device__ __forceinline__ int fx_unit(int E, int k) { return E + 4 - k; }

// one operator entry at scale 2^k
inline int2 fx_coef(double c, int k) {
  const long long C = llrint(ldexp(c, k));
  const long long h = (C + (1ll << 30)) >> 31;
  return make_int2(int(h), int(C - (h << 31)));
}
// ... and back, rounded to FP64 (k <= 67)
__device__ __forceinline__ double fx_coef_value(int2 c, int k) {
  return fma(double(c.x), 2147483648.0, double(c.y)) * __hiloint2double((1023 - k) << 20, 0);
}
// largest k with sum 2^k <= 2^FX_SUM_BITS; at most 67, so that the smallest group exponent leaves a
// unit (fx_unit) in the normal range
inline int fx_scale(double sum) {
  int e = 0;
  frexp(sum, &e);  // sum < 2^e
  const int k = FX_SUM_BITS - e;
  return k < 67 ? k : 67;
}

// Largest of each of K exponents over the N threads of one element, thread i of it, into s[K] of the
// element (zeroed before a barrier by the caller, read after one).  All threads of the block call it;
// those without a point bring zeros and act = false.  With N a power of two up to 16 an element lies in one
// warp and the values are stored, not accumulated.
template <int N, int K>
__device__ __forceinline__ void fx_group_max(const uint32_t (&w)[K], int i, bool act, uint32_t* s) {
  const int lane = threadIdx.x & 31;
  if constexpr (N % 32 == 0) {
    // whole warps belong to one element
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t m = __reduce_max_sync(~0u, w[k]);
      if (act && lane == 0) atomicMax(&s[k], m);
    }
  } else {
    constexpr int P = (K + 1) / 2;  // two to a register
    uint32_t p[P];
#pragma unroll
    for (int k = 0; k < P; ++k) p[k] = 2 * k + 1 < K ? w[2 * k] | (w[2 * k + 1] << 16) : w[2 * k];
    if constexpr (32 % N == 0) {
      // whole elements in a warp: one value per element, no atomics
#pragma unroll
      for (int o = 1; o < N; o <<= 1)
#pragma unroll
        for (int k = 0; k < P; ++k) p[k] = __vmaxu2(p[k], __shfl_xor_sync(~0u, p[k], o));
      if (act && i == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) s[k] = k & 1 ? p[k / 2] >> 16 : p[k / 2] & 0xFFFFu;
      }
    } else {
      // segments of N lanes that may cross warps: each segment's first lane in a warp collects it
#pragma unroll
      for (int o = 1; o < 32 && o < N; o <<= 1) {
        const bool in = i + o < N && lane + o < 32;
#pragma unroll
        for (int k = 0; k < P; ++k) {
          const uint32_t q = __shfl_down_sync(~0u, p[k], o);
          if (in) p[k] = __vmaxu2(p[k], q);
        }
      }
      if (act && (i == 0 || lane == 0)) {
#pragma unroll
        for (int k = 0; k < K; ++k) atomicMax(&s[k], k & 1 ? p[k / 2] >> 16 : p[k / 2] & 0xFFFFu);
      }
    }
  }
}
// the group of variable v of nv: 0 density, 1 momenta, 2 energy
__host__ __device__ constexpr int fx_group(int v, int nv) { return v == 0 ? 0 : (v == nv - 1 ? 2 : 1); }
// exponents of a point of state q: the largest of each group
template <int NV>
__device__ __forceinline__ void fx_state_exps(const double* q, uint32_t (&w)[FX_GROUPS]) {
  uint32_t m = fx_mag(q[1]);
#pragma unroll
  for (int v = 2; v < NV - 1; ++v) m = max(m, fx_mag(q[v]));
  w[0] = fx_mag(q[0]) >> 20;
  w[1] = m >> 20;
  w[2] = fx_mag(q[NV - 1]) >> 20;
}
// a point with exponent e too low for its element's largest, emax, to leave it FP64's bits
__device__ __forceinline__ bool fx_low(uint32_t e, uint32_t emax) { return e + FX_SPREAD < emax; }
// the same for a state with exponents w whose element has the largest ones s: by density and energy (a
// single small momentum, or the stagnation of all three, is no reason)
__device__ __forceinline__ bool fx_low_state(const uint32_t (&w)[FX_GROUPS], const uint32_t* s) {
  return fx_low(w[0], s[0]) || fx_low(w[2], s[2]);
}
__device__ __forceinline__ int fx_exp(uint32_t e) { return int(e) < FX_E_MIN ? FX_E_MIN : int(e); }

}  // namespace frg
