// 64-bit fixed point for the pair geometry of the FP64 form.
//
// GB300 issues two FP64 thread operations per SM and clock, one 64th of its
// integer and FP32 rate, so the FP64 form's loops over neighbours were bound
// by the FP64 pipe (85-89 % busy).  The geometry of a pair is bounded by the
// kernel support (r < 2h), so it needs no exponent: lengths are held in units
// of 2h as signed 64-bit integers with 62 fractional bits, nine more than the
// mantissa of a double between 1/2 and 1 has, and the distance, the kernel
// shapes and the sums are formed on the integer pipe.
//
//  - A coordinate x is x / (2h) 2^62 modulo 2^64.  Differences of
//    coordinates are exact modulo 2^64, which holds every difference below
//    2 (2h); so the range of the box costs no precision.
//  - r^2 is in units of 2^-60 (2h)^2, r in units of 2^-62 2h.
//  - The kernel shapes with t = 1 - r / 2h: F shape t^3, W shape t^4 (5 - 4t).
//    Near the cutoff they are far below one, where an absolute step is coarse:
//    the density and the filter, which the self term keeps away from zero, take
//    W at steps of 2^-61, the pair pass scales t up first (scaled_t).  What is
//    left there is the error of t itself, 2^-58.6 / t of its value (that of an
//    FP64 evaluation is about 2^-53 / t).
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace sphgb {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;

#ifdef __CUDACC__
#define SPH_FX __host__ __device__ __forceinline__
#else
#define SPH_FX inline
#endif

constexpr u64 kOne2 = 1ull << 60;    // (2h)^2 in units of r^2
constexpr u64 kNear2 = 1ull << 48;   // below (2h / 64)^2 a pair takes the FP64 route: there the
                                     // 2^-60 step of r^2 would show in r

SPH_FX u64 mulhi(u64 a, u64 b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (u64)(((unsigned __int128)a * b) >> 64);
#endif
}

SPH_FX u64 bits_of(double x) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(x);
#else
  u64 b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
SPH_FX double of_bits(u64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((i64)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}

// 1 / (2h) = (r1 2^64 + r0) 2^(-180 - eh), to 127 bits.
struct Unit {
  u64 r1, r0;
  int32_t eh;
};

inline Unit make_unit(double two_h) {
  Unit u;
  const u64 b = bits_of(two_h);
  const u64 m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);  // two_h is a normal number
  u.eh = (int32_t)((b >> 52) & 0x7FF) - 1075;
  unsigned __int128 rem = ((1ull << 52) - 1) % m;  // (2^180 - 1) / m by 64-bit digits
  unsigned __int128 a = (rem << 64) | ~0ull;
  u.r1 = (u64)(a / m);
  rem = a % m;
  a = (rem << 64) | ~0ull;
  u.r0 = (u64)(a / m);
  return u;
}

// x / (2h) 2^62 modulo 2^64, truncated towards zero (0 for a non-finite x and
// for one beyond 2^54 2h, where a double no longer resolves the support).
SPH_FX i64 to_fixed(double x, const Unit& U) {
  const u64 b = bits_of(x);
  const int ex = (int)((b >> 52) & 0x7FF);
  const u64 m = (b & 0xFFFFFFFFFFFFFull) | (ex ? (1ull << 52) : 0ull);
  const int s = 118 + U.eh - ((ex ? ex : 1) - 1075);  // m R >> s
  const u64 a = mulhi(m, U.r0), lo1 = m * U.r1;
  const u64 p0 = m * U.r0, p1 = lo1 + a;
  const u64 p2 = mulhi(m, U.r1) + (p1 < lo1 ? 1ull : 0ull);
  u64 q;
  if (s < 0 || s >= 192) q = 0;
  else {
    const u64 l = s < 64 ? p0 : (s < 128 ? p1 : p2), h = s < 64 ? p1 : (s < 128 ? p2 : 0ull);
    const int t = s & 63;
    q = t ? (l >> t) | (h << (64 - t)) : l;
  }
  if (ex == 0x7FF) q = 0;
  return (i64)((b >> 63) ? 0ull - q : q);
}

// v = h 2^32 + l with a signed low half.
struct Half {
  int h, l;
};
SPH_FX Half split(i64 v) {
  Half s;
  s.l = (int)(uint32_t)(u64)v;
  s.h = (int)(uint32_t)((u64)(v + 0x80000000ll) >> 32);
  return s;
}

// r^2 of a pair vector (|components| < 2^62.5): the products of the low
// halves, below one unit together, are left out.
SPH_FX u64 norm2(const Half& x, const Half& y, const Half& z) {
  const i64 hh = (i64)x.h * x.h + (i64)y.h * y.h + (i64)z.h * z.h;
  const i64 c = (i64)x.h * x.l + (i64)y.h * y.l + (i64)z.h * z.l + (1ll << 30);
  return (u64)(hh + (c >> 31));
}

SPH_FX float inv_sqrt(float x) {
#ifdef __CUDA_ARCH__
  float y;  // (x is a normal number: no scaling around the hardware estimate)
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / sqrtf(x);
#endif
}

// The integer nearest to a float below 2^22 in magnitude, on the FP32 and
// integer pipes.
SPH_FX int near_int(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_int(__fadd_rn(x, 12582912.0f)) - 0x4B400000;
#else
  return (int)lrintf(x);
#endif
}

// sqrt(r2) for kNear2 <= r2 < 2^60, in units of 2^-32: an integer estimate r0
// from the FP32 reciprocal square root y (30 bits, good to about 2^-21), and
// two corrections e y / 2 of the exact integer residual e = r2 - r^2, the
// first down to 2^-12, the second to 2^-32.
SPH_FX i64 root(u64 r2) {
#ifdef __CUDA_ARCH__
  const float f = __uint2float_rn((uint32_t)(r2 >> 28));
#else
  const float f = (float)(uint32_t)(r2 >> 28);
#endif
  const float y = inv_sqrt(f);
#ifdef __CUDA_ARCH__
  const uint32_t r0 = __float2uint_rn(f * y * 16384.0f);
#else
  const uint32_t r0 = (uint32_t)llrintf(f * y * 16384.0f);
#endif
  // 1 / (2 r0) = 2^-15 y
  const i64 e0 = (i64)(r2 - (u64)r0 * r0);
  const int d1 = near_int((float)(int)(e0 >> 9) * (y * 64.0f));  // 2^9 2^-15 2^12
  const i64 e1 = (e0 << 12) - (((i64)d1 * (int)r0) << 1) - (((i64)d1 * d1) >> 12);
  const int d2 = near_int((float)(int)(e1 >> 1) * (y * 64.0f));  // 2 2^-15 2^20
  return ((i64)r0 << 32) + ((i64)d1 << 20) + d2;
}

// t = 1 - r / 2h in units of 2^-64 (r2 as for root: 0 < t < 1).
SPH_FX u64 shape_t(u64 r2) { return (u64)((1ll << 62) - root(r2)) << 2; }
// The W shape over 8 from t and t^2, in units of 2^-64: t^4 (5 - 4t) / 8.
SPH_FX u64 shape_w8(u64 t, u64 t2) {
  return mulhi(mulhi(t2, t2), 0xA000000000000000ull - (t >> 1));
}

// Shapes scaled up by a power of two, which keep their precision where t is
// small: with T = t 2^lead, the F shape is mulhi(mulhi(T, T), T) 2^(-3 lead)
// and the W shape over 8 is shape_w8(t, mulhi(T, T)) 2^(-4 lead).
SPH_FX u64 scaled_t(u64 t, uint32_t lead) { return t << lead; }
// Leading zeros of a 64-bit value, 32 at most: of t, the lead that brings it
// into [1/2, 1), or up by 2^32.
SPH_FX uint32_t lead32(u64 v) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__clz((int)(uint32_t)(v >> 32));
#else
  return (v >> 32) ? (uint32_t)__builtin_clz((uint32_t)(v >> 32)) : 32u;
#endif
}

// Sum of W shapes (over 8, 2^-64) in 96 bits, and its value.
struct Sum96 {
  uint32_t w0 = 0, w1 = 0, w2 = 0;
  SPH_FX void add(u64 v) {
#ifdef __CUDA_ARCH__
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, 0;"
        : "+r"(w0), "+r"(w1), "+r"(w2)
        : "r"((uint32_t)v), "r"((uint32_t)(v >> 32)));
#else
    const u64 s = (((u64)w1 << 32) | w0) + v;
    if (s < v) ++w2;
    w0 = (uint32_t)s;
    w1 = (uint32_t)(s >> 32);
#endif
  }
  SPH_FX double shape_sum() const {  // (w2 2^64 + w1 2^32 + w0) 2^-61
    return (double)w2 * 8.0 + (double)(((u64)w1 << 32) | w0) * 4.336808689942017736e-19;
  }
};

// The high half of a 32 x 32-bit product plus c, and a full product plus a
// signed 32-bit addend: the instructions that the products below are made of
// (the compiler's 64-bit arithmetic takes about twice as many).
SPH_FX int mad_hi(int a, int b, int c) {
#ifdef __CUDA_ARCH__
  int r;
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
#else
  return (int)(((i64)a * b) >> 32) + c;
#endif
}
SPH_FX i64 mad_wide(int a, int b, i64 c) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (i64)a * b + c;
#endif
}
// a b / 2^64 within 1.3 units and without bias (|a|, |b| <= 2^62): the high
// parts of the two middle products, each truncated by half a unit on average,
// for which the constants stand; the product of the low halves, a quarter of
// a unit at most, is left out.
SPH_FX i64 mul(const Half& a, const Half& b) {
  return mad_wide(a.h, b.h, (i64)mad_hi(a.l, b.h, mad_hi(a.h, b.l, 1)));
}
// (a b - c d) / 2^64, likewise: one component of a cross product.
SPH_FX i64 mul_sub(const Half& a, const Half& b, const Half& c, const Half& d) {
  const int nc = -c.h, nd = -d.h;
  const int m = mad_hi(c.l, nd, mad_hi(nc, d.l, mad_hi(a.l, b.h, mad_hi(a.h, b.l, 2))));
  return mad_wide(a.h, b.h, mad_wide(nc, d.h, (i64)m));
}
SPH_FX i64 dot3(const Half* a, const Half* b) {
  int m = 3;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int k = 0; k < 3; ++k) m = mad_hi(a[k].l, b[k].h, mad_hi(a[k].h, b[k].l, m));
  return mad_wide(a[0].h, b[0].h, mad_wide(a[1].h, b[1].h, mad_wide(a[2].h, b[2].h, (i64)m)));
}

// 1 / rho in units of 2^-59 for rho (units of 2^-62) in [1/8, 1]: the FP32
// reciprocal z0 to 27 fractional bits, then z0 (1 + e + e^2), e = 1 - rho z0.
SPH_FX i64 recip(i64 rho) {
  const uint32_t rh = (uint32_t)((u64)rho >> 32), rl = (uint32_t)rho;
#ifdef __CUDA_ARCH__
  const uint32_t z0 = __float2uint_rn(__fdividef(1.4411518807585587e17f, __uint2float_rn(rh)));
#else
  const uint32_t z0 = (uint32_t)llrintf(1.4411518807585587e17f / (float)rh);  // 2^57 / (rho 2^30)
#endif
  const i64 e = (i64)((1ull << 62) - ((((u64)rh * z0) << 5) + (((u64)rl * z0) >> 27)));
  const int es = (int)(e >> 20);
  const i64 c = e + (((i64)es * es) >> 22);
  return (i64)((u64)z0 << 32) + (((i64)(int)(c >> 32) * (i64)z0) << 2) +
         (i64)(((u64)(uint32_t)c * z0) >> 30);
}

// The exponent of a double's magnitude: |x| < 2^(exponent_of(x)).
SPH_FX int exponent_of(double x) { return (int)((bits_of(x) >> 52) & 0x7FF) - 1022; }
// x 2^(61 - e), truncated, for |x| < 2^e (0 below the last place; a subnormal
// counts as 0).
SPH_FX i64 mantissa_at(double x, int e) {
  const u64 b = bits_of(x);
  const int ex = (int)((b >> 52) & 0x7FF);
  if (ex == 0) return 0;
  const u64 m = ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << 8;  // in [2^60, 2^61): x 2^(61 - ex + 1022)
  const int s = e - (ex - 1022);
  const u64 q = s < 63 ? m >> s : 0ull;
  return (i64)((b >> 63) ? 0ull - q : q);
}

// Signed sum in 96 bits.
struct Acc96 {
  uint32_t w0 = 0, w1 = 0, w2 = 0;
  SPH_FX void add3(uint32_t a, uint32_t b, uint32_t c) {
#ifdef __CUDA_ARCH__
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(w0), "+r"(w1), "+r"(w2)
        : "r"(a), "r"(b), "r"(c));
#else
    u64 s = (u64)w0 + a;
    w0 = (uint32_t)s;
    s = (s >> 32) + w1 + b;
    w1 = (uint32_t)s;
    w2 += c + (uint32_t)(s >> 32);
#endif
  }
  SPH_FX void add(i64 v) {
    const uint32_t h = (uint32_t)((u64)v >> 32);
    add3((uint32_t)v, h, (uint32_t)((int)h >> 31));
  }
  // v 2^s, 0 <= s < 32
  SPH_FX void add_shifted(i64 v, int s) {
    const uint32_t l = (uint32_t)v, h = (uint32_t)((u64)v >> 32), x = (uint32_t)((int)h >> 31);
#ifdef __CUDA_ARCH__
    add3(l << s, __funnelshift_l(l, h, s), __funnelshift_l(h, x, s));
#else
    add3(l << s, (uint32_t)((((u64)h << 32) | l) << s >> 32), (uint32_t)((((u64)x << 32) | h) << s >> 32));
#endif
  }
  // The sum times 2^e as a double, rounded to nearest (ties away from zero),
  // put together on the integer pipe; zero below and infinite above the
  // range of normal numbers.
  SPH_FX double value(int e) const {
    const bool neg = (int)w2 < 0;
    const uint32_t f = neg ? ~0u : 0u;
    Acc96 z;
    z.add3(w0 ^ f, w1 ^ f, w2 ^ f);
    z.add3(f & 1u, 0u, 0u);
    uint32_t a = z.w2, b = z.w1, c = z.w0;
    if (a == 0u) {
      a = b;
      b = c;
      c = 0u;
      e -= 32;
    }
    if (a == 0u) {
      a = b;
      b = c;
      c = 0u;
      e -= 32;
    }
    if (a == 0u) return 0.0;
#ifdef __CUDA_ARCH__
    const int lz = __clz((int)a);
    a = __funnelshift_l(b, a, lz);
    b = __funnelshift_l(c, b, lz);
#else
    const int lz = __builtin_clz(a);
    if (lz) {
      a = (a << lz) | (b >> (32 - lz));
      b = (b << lz) | (c >> (32 - lz));
    }
#endif
    // value = (a:b) 2^(e + 32 - lz), with the top bit of a set
    const u64 m = (((((u64)a << 32) | b) >> 10) + 1ull) >> 1;  // 53 bits (or 2^53)
    const int ex = e + 32 - lz + 63 + 1023;                    // biased exponent
    u64 r = m + ((u64)(uint32_t)(ex - 1) << 52);
    if (ex <= 0) r = 0;
    if (ex >= 2046) r = 0x7FF0000000000000ull;
    return of_bits(r | ((u64)neg << 63));
  }
};

}  // namespace fx
}  // namespace sphgb
