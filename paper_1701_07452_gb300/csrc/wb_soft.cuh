// FP64 arithmetic on the integer pipes.  Reciprocals and roots are the same integer
// operations on host and device (the FP32 seeds differ by an ulp or two, which the
// fixed-point step absorbs); the product's device form is PTX of its own (carry
// chains, funnel shifts).  The tests hold the host forms against exact integers
// and the device forms against the FP64 multiply and exact integers.
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

template <bool SURE>
WB_HD double wb_rcp_t(double x) {
  const unsigned hi = wb_hi32(x), lo = wb_lo32(x);
  const unsigned ef = (hi >> 20) & 0x7ffu;
  const unsigned Mh = (hi & 0xfffffu) | 0x100000u;
  const unsigned Y = wb_seed_rcp(((hi << 3 | lo >> 29) & 0x7fffffu) | 0x3f800000u);  // 2^-23, in (2^22, 2^23]
  const unsigned long long acc = (unsigned long long)lo * Y + ((unsigned long long)(Mh * Y) << 32);
  const long long D = (long long)acc;                                    // -E in 2^-75, |E| < 2^54
  const int Dh = (int)(D >> 27);                                         // 2^-48
  const unsigned sq = (unsigned)(((long long)Dh * Dh) >> 32);            // 2^-64
  const long long C = (D >> 14) - (long long)(sq >> 3);                  // -(E + E^2) in 2^-61
  const long long YC = (long long)((unsigned long long)Y * (unsigned)C +
                                   ((unsigned long long)(Y * (unsigned)(C >> 32)) << 32));  // 2^-84
  const unsigned long long R = ((unsigned long long)Y << 40) - (unsigned long long)(YC >> 21);  // 2^-63
  if (SURE) return wb_round_pack(R, 10, 2044 - (int)ef, hi & 0x80000000u, true);
  return wb_round_pack_low(R, 10, 2044 - (int)ef, hi & 0x80000000u, ef - 1u < 2046u);
}
WB_HD double wb_rcp(double x) { return wb_rcp_t<false>(x); }
// x known to be normal and below 2^1022 in magnitude
WB_HD double wb_rcp_sure(double x) { return wb_rcp_t<true>(x); }

// 1/sqrt(x), sqrt(x) and 1/x from one residual (a caller pays for the ones it uses)
struct WbRoots {
  double rsq, sq, rcp;
};

template <bool SURE>
WB_HD WbRoots wb_roots_t(double x) {
  const unsigned hi = wb_hi32(x), lo = wb_lo32(x);
  // x = m 2^(2k), 1 <= m < 4, M = m 2^52
  const unsigned ef = hi >> 20, s = ~ef & 1u;
  const int k = ((int)ef - 1023) >> 1;
  const bool ok = SURE || hi - 0x100000u < 0x7fe00000u;
  const unsigned long long M = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << s;
  const unsigned Mh = (unsigned)(M >> 32), Ml = (unsigned)M;
  const unsigned Y = wb_seed_rsqrt((((hi << 3 | lo >> 29) & 0x7fffffu) | 0x3f800000u) + (s << 23));  // 2^-23, in (2^22, 2^23]
  const unsigned long long Z = (unsigned long long)Y * Y;
  const unsigned Zh = (unsigned)(Z >> 32), Zl = (unsigned)Z;
  unsigned long long acc = (unsigned long long)Mh * Zl + (((unsigned long long)Ml * Zl) >> 32);
  acc += (unsigned long long)Ml * Zh;
  acc += (unsigned long long)(Mh * Zh) << 32;
  const long long D = (long long)acc;                                    // -E in 2^-66, |E| < 2^46
  const int Dh = (int)(D >> 18);                                         // 2^-48
  const unsigned sq = (unsigned)(((long long)Dh * Dh) >> 32);            // 2^-64
  const long long C = (D >> 6) - (long long)((3u * sq) >> 6);            // -(E + 3/4 E^2) in 2^-60
  const long long YC = (long long)((unsigned long long)Y * (unsigned)C +
                                   ((unsigned long long)(Y * (unsigned)(C >> 32)) << 32));  // 2^-83
  const unsigned long long R = ((unsigned long long)Y << 40) - (unsigned long long)(YC >> 21);  // 2^-63
  const unsigned Rh = (unsigned)(R >> 32), Rl = (unsigned)R;
  WbRoots o;
  o.rsq = wb_round_pack(R, 10, 1021 - k, 0u, ok);
  const unsigned long long A = M << 10;                                  // 2^-62
  const unsigned Ah = (unsigned)(A >> 32), Al = (unsigned)A;
  o.sq = wb_round_pack((unsigned long long)Ah * Rh + (((unsigned long long)Ah * Rl) >> 32) +
                           (((unsigned long long)Al * Rh) >> 32), 9, 1022 + k, 0u, ok);  // 2^-61
  const unsigned long long Q = (unsigned long long)Rh * Rh + (((unsigned long long)Rh * Rl) >> 31);  // 2^-62
  o.rcp = SURE ? wb_round_pack(Q << s, 9, 2044 - (int)ef, 0u, true)
               : wb_round_pack_low(Q, 9 - (int)s, 2044 - (int)ef, 0u, ok);
  return o;
}
WB_HD WbRoots wb_roots(double x) { return wb_roots_t<false>(x); }
// x known to be positive, normal and below 2^1022
WB_HD WbRoots wb_roots_sure(double x) { return wb_roots_t<true>(x); }

WB_HD double wb_rsqrt(double x) { return wb_roots(x).rsq; }
WB_HD double wb_sqrt(double x) { return wb_roots(x).sq; }

// x y rounded to nearest even on the integer pipes: the bits of the FP64
// multiply for factors that are normal or zero and products that are zero or of
// magnitude in [2^-1021, 2^1023).  Subnormal factors and products below the
// normal range count as zero; an infinity, a NaN or a product above it gives
// NaN (in the first and last normal binade either, by the factors' exponents).
// 40 integer instructions (four 32 x 32 bit multiplies among them), about 12
// cycles of an SM's other pipes against 19 of its FP64 pipe.  How many of the
// sweep's products run here was measured: of its 100, none 8.05 ms, half 6.95,
// three quarters 6.45 and all 6.38 ms per axis of a 256^3 box (the FP64 pipe 85,
// 84 and 77 % busy with none, three quarters and all).
template <bool FINITE, int KNOWN>
WB_HD double wb_smul_t(double x, double y) {
  const unsigned hx = wb_hi32(x), hy = wb_hi32(y), lx = wb_lo32(x), ly = wb_lo32(y);
  const unsigned ah = (hx & 0xfffffu) | 0x100000u;
  const unsigned bh = (hy << 11 | ly >> 21) | 0x80000000u, bl = ly << 11;
  unsigned t0, t1, t2, t3;  // limbs of the significands' product
#ifdef __CUDA_ARCH__
  asm("{\n\t.reg .u64 w0, w1, w2, w3;\n\t.reg .u32 a0, a1, b0, b1, c0, c1, d0;\n\t"
      "mul.wide.u32 w0, %5, %7;\n\tmul.wide.u32 w1, %4, %7;\n\t"
      "mul.wide.u32 w2, %5, %6;\n\tmul.wide.u32 w3, %4, %6;\n\t"
      "mov.b64 {%0, d0}, w0;\n\tmov.b64 {a0, a1}, w1;\n\tmov.b64 {b0, b1}, w2;\n\tmov.b64 {c0, c1}, w3;\n\t"
      "add.cc.u32 %1, d0, a0;\n\taddc.cc.u32 %2, c0, a1;\n\taddc.u32 %3, c1, 0;\n\t"
      "add.cc.u32 %1, %1, b0;\n\taddc.cc.u32 %2, %2, b1;\n\taddc.u32 %3, %3, 0;\n\t}"
      : "=r"(t0), "=&r"(t1), "=&r"(t2), "=&r"(t3)
      : "r"(ah), "r"(lx), "r"(bh), "r"(bl));
#else
  const unsigned long long w0 = (unsigned long long)lx * bl;
  const unsigned long long w1 = (unsigned long long)ah * bl + (w0 >> 32);
  const unsigned long long w2 = (unsigned long long)lx * bh + (unsigned)w1;
  const unsigned long long w3 = (unsigned long long)ah * bh + (w1 >> 32) + (w2 >> 32);
  t0 = (unsigned)w0; t1 = (unsigned)w2; t2 = (unsigned)w3; t3 = (unsigned)(w3 >> 32);
#endif
  // one bit up when the significands' product is below 2 (bit 20 of t3 clear)
  const unsigned n = (t3 >> 20) + 31u;
#ifdef __CUDA_ARCH__
  const unsigned r3 = __funnelshift_rc(t2, t3, n), r2 = __funnelshift_rc(t1, t2, n), g = __funnelshift_rc(t0, t1, n);
#else
  const unsigned s = 32u - n;
  const unsigned r3 = s ? t3 << 1 | t2 >> 31 : t3, r2 = s ? t2 << 1 | t1 >> 31 : t2, g = s ? t1 << 1 | t0 >> 31 : t1;
#endif
  const unsigned ea = hx & 0x7ff00000u, eb = hy & 0x7ff00000u, sign = (hx ^ hy) & 0x80000000u;
  const unsigned sum = ea + eb;
  const unsigned es = sum + (n << 20) - ((1024u + 31u) << 20) + sign;  // sign and exponent field minus one
  // g: guard bit and the bits below it; up when above half, or half and odd
  // (any bit of t0 counts as above)
  const unsigned c = (r2 & 1u) | (t0 < 1u ? t0 : 1u);
  unsigned lo, hi;
#ifdef __CUDA_ARCH__
  asm("{\n\t.reg .u32 y, z;\n\tadd.u32 y, %3, 0x7fffffff;\n\tadd.cc.u32 z, %2, y;\n\t"
      "addc.cc.u32 %0, %4, 0;\n\taddc.u32 %1, %5, %6;\n\t}"
      : "=&r"(lo), "=r"(hi)
      : "r"(g), "r"(c), "r"(r2), "r"(r3), "r"(es));
#else
  const unsigned long long r = ((unsigned long long)r3 << 32 | r2) + (((unsigned long long)g + c + 0x7fffffffu) >> 32);
  lo = (unsigned)r; hi = (unsigned)(r >> 32) + es;
#endif
  if (KNOWN != 7 && ((!(KNOWN & 1) && ea == 0u) || (!(KNOWN & 2) && eb == 0u) || sum < (1024u << 20))) {
    hi = sign;
    lo = 0u;
  }
  if (!FINITE && (ea == 0x7ff00000u || eb == 0x7ff00000u || sum > (3068u << 20))) hi = 0x7ff80000u;
  return wb_make64(hi, lo);
}
WB_HD double wb_smul(double x, double y) { return wb_smul_t<false, 0>(x, y); }
// The form the sweeps take: the same for finite factors whose product is known to stay below the top of
// the range (4 of the 40 instructions less, 6 % of a sweep).  KNOWN: 1, 2: x, y
// normal; 7: both, and the product above 2^-1021 (1 to 5 instructions less).
template <int KNOWN>
WB_HD double wb_smul_finite(double x, double y) { return wb_smul_t<true, KNOWN>(x, y); }
