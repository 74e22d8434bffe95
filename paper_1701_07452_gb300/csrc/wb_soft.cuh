// FP64 arithmetic on the integer pipes (host and device: the same integer
// operations give the same bits on the CPU, where the tests check them).
#pragma once
#include <cuda_runtime.h>
#include <string.h>

#define WB_HD __host__ __device__ __forceinline__

WB_HD unsigned wb_hi32(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2hiint(x);
#else
  unsigned long long b;
  memcpy(&b, &x, 8);
  return (unsigned)(b >> 32);
#endif
}
WB_HD unsigned wb_lo32(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(x);
#else
  unsigned long long b;
  memcpy(&b, &x, 8);
  return (unsigned)b;
#endif
}
WB_HD double wb_make64(unsigned hi, unsigned lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const unsigned long long b = (unsigned long long)hi << 32 | lo;
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}

// FP32 approximations of 1/f (1 <= f < 2) and 1/sqrt(f) (1 <= f < 4), given
// the bits of f, in units of 2^-23: adding 1 leaves the value in the low bits
// of the sum (a sum of 2 included: the bit pattern goes on by one).
#ifndef WB_SEED_ULPS  // the CPU tests move the seeds by some units
#define WB_SEED_ULPS 0
#endif
WB_HD unsigned wb_seed_units(float y) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(__fadd_rn(y, 1.0f)) - 0x3f800000u;
#else
  const volatile float s = y + 1.0f;
  const float t = s;
  unsigned u;
  memcpy(&u, &t, 4);
  return u - 0x3f800000u + (y < 1.0f ? WB_SEED_ULPS : 0);
#endif
}
WB_HD unsigned wb_seed_rcp(unsigned fbits) {
  float y;
#ifdef __CUDA_ARCH__
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(fbits)));
#else
  float f;
  memcpy(&f, &fbits, 4);
  y = 1.0f / f;
#endif
  return wb_seed_units(y);
}
WB_HD unsigned wb_seed_rsqrt(unsigned fbits) {
  float y;
#ifdef __CUDA_ARCH__
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(fbits)));
#else
  float f;
  memcpy(&f, &fbits, 4);
  y = (float)(1.0 / __builtin_sqrt((double)f));
#endif
  return wb_seed_units(y);
}

// Reciprocal, reciprocal square root and square root of FP64 values on the
// integer pipes.  An SM of this GPU issues one FP64 warp instruction in about
// 19 cycles but two integer or FP32 ones every cycle beside it (measured: 32
// of them per DFMA cost no time), so a Newton step in FP64 (3 to 6 FP64
// instructions, 57 to 114 cycles) is replaced by one in 64-bit fixed point
// (30 to 50 integer instructions, 10 to 20 cycles).
//
// The significand M of x = M 2^(e-52) is taken as a 53- or 54-bit integer, the
// FP32 approximation of its reciprocal (square root) as an integer Y of 2^-23
// (|Y 2^-23 / y - 1| < 2^-21 with the truncation of M to FP32), the residual
//   E = 1 - M Y   or   E = 1 - M Y^2
// exactly modulo 2^64 (its leading 21 bits cancel, so nothing is lost), and
//   y = Y (1 + E + E^2)   or   y = Y (1 + (E + 3/4 E^2) / 2)
// with 60 bits, rounded once to 53: at most 0.52 ulp from the exact value (0.53
// for the square of 1/sqrt; checked on the CPU against exact integers with the
// seeds moved either way), where the FP64 forms these replace reached about
// 1.5 ulp.  The square root is M times the 63-bit y, again rounded once.
// With every reciprocal and root of the step done here the 256^3 step went from
// 69.6 to 58.6 ms and the 64^3 one from 1.62 to 1.39 ms.
// x not positive and normal gives NaN (rcp: x of either sign).

// The double whose significand is V shifted down by sh to 53 bits (leading one
// included), rounded to nearest; ex is the exponent field minus one, >= 0.
WB_HD double wb_round_pack(unsigned long long V, int sh, int ex, unsigned sign, bool ok) {
  const unsigned long long r = (V + (1ull << (sh - 1))) >> sh;
  const unsigned hi = ((unsigned)(r >> 32) + ((unsigned)ex << 20)) | sign;
  return wb_make64(ok ? hi : 0x7ff80000u, (unsigned)r);
}
// The same for a reciprocal, whose exponent field minus one may be negative: a
// subnormal, shifted further (one rounding all the same).
WB_HD double wb_round_pack_low(unsigned long long V, int sh, int ex, unsigned sign, bool ok) {
  const int low = ex < 0 ? -ex : 0;
  return wb_round_pack(V, sh + low, ex + low, sign, ok);
}

WB_HD double wb_rcp(double x) {
  const unsigned hi = wb_hi32(x), lo = wb_lo32(x);
  const unsigned ef = (hi >> 20) & 0x7ffu;
  const unsigned Mh = (hi & 0xfffffu) | 0x100000u;
  const unsigned Y = wb_seed_rcp(((hi << 3 | lo >> 29) & 0x7fffffu) | 0x3f800000u);  // 2^-23, in (2^22, 2^23]
  const unsigned long long acc = (unsigned long long)lo * Y + ((unsigned long long)(Mh * Y) << 32);
  const long long E = -(long long)acc;                                   // 2^-75, |E| < 2^54
  const int Eh = (int)(E >> 27);                                         // 2^-48
  const unsigned sq = (unsigned)(((long long)Eh * Eh) >> 32);            // 2^-64
  const long long C = (E >> 14) + (long long)(sq >> 3);                  // 2^-61
  const long long YC = (long long)((unsigned long long)Y * (unsigned)C +
                                   ((unsigned long long)(Y * (unsigned)(C >> 32)) << 32));  // 2^-84
  const unsigned long long R = ((unsigned long long)Y << 40) + (unsigned long long)(YC >> 21);  // 2^-63
  return wb_round_pack_low(R, 10, 2044 - (int)ef, hi & 0x80000000u, ef - 1u < 2046u);
}

// 1/sqrt(x), sqrt(x) and 1/x from one residual (a caller pays for the ones it uses)
struct WbRoots {
  double rsq, sq, rcp;
};

WB_HD WbRoots wb_roots(double x) {
  const unsigned hi = wb_hi32(x), lo = wb_lo32(x);
  // x = m 2^(2k), 1 <= m < 4, M = m 2^52
  const unsigned ef = hi >> 20, s = ~ef & 1u;
  const int k = ((int)ef - 1023) >> 1;
  const bool ok = hi - 0x100000u < 0x7fe00000u;
  const unsigned long long M = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << s;
  const unsigned Mh = (unsigned)(M >> 32), Ml = (unsigned)M;
  const unsigned Y = wb_seed_rsqrt((((hi << 3 | lo >> 29) & 0x7fffffu) | 0x3f800000u) + (s << 23));  // 2^-23, in (2^22, 2^23]
  const unsigned long long Z = (unsigned long long)Y * Y;
  const unsigned Zh = (unsigned)(Z >> 32), Zl = (unsigned)Z;
  unsigned long long acc = (unsigned long long)Mh * Zl + (((unsigned long long)Ml * Zl) >> 32);
  acc += (unsigned long long)Ml * Zh;
  acc += (unsigned long long)(Mh * Zh) << 32;
  const long long E = -(long long)acc;                                   // 2^-66, |E| < 2^46
  const int Eh = (int)(E >> 18);                                         // 2^-48
  const unsigned sq = (unsigned)(((long long)Eh * Eh) >> 32);            // 2^-64
  const long long C = (E >> 6) + (long long)((3u * sq) >> 6);            // 2^-60
  const long long YC = (long long)((unsigned long long)Y * (unsigned)C +
                                   ((unsigned long long)(Y * (unsigned)(C >> 32)) << 32));  // 2^-83
  const unsigned long long R = ((unsigned long long)Y << 40) + (unsigned long long)(YC >> 21);  // 2^-63
  const unsigned Rh = (unsigned)(R >> 32), Rl = (unsigned)R;
  WbRoots o;
  o.rsq = wb_round_pack(R, 10, 1021 - k, 0u, ok);
  const unsigned long long A = M << 10;                                  // 2^-62
  const unsigned Ah = (unsigned)(A >> 32), Al = (unsigned)A;
  o.sq = wb_round_pack((unsigned long long)Ah * Rh + (((unsigned long long)Ah * Rl) >> 32) +
                           (((unsigned long long)Al * Rh) >> 32), 9, 1022 + k, 0u, ok);  // 2^-61
  o.rcp = wb_round_pack_low((unsigned long long)Rh * Rh + (((unsigned long long)Rh * Rl) >> 31),  // 2^-62
                        9 - (int)s, 2044 - (int)ef, 0u, ok);
  return o;
}

WB_HD double wb_rsqrt(double x) { return wb_roots(x).rsq; }
WB_HD double wb_sqrt(double x) { return wb_roots(x).sq; }
