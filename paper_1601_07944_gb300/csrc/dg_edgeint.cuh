/*
 * dg_edgeint.cuh -- the local Lax-Friedrichs edge flux with most of its arithmetic
 * in 64-bit integers.
 *
 * The flux of lax_friedrichs_edge takes 54 float64 operations a point, and this
 * GPU issues 2 float64 FMAs per clock and SM, but 128 integer instructions.  Here
 * the normal velocities, the pressures, the sound speeds and the dissipation are
 * formed in fixed point (60 to 62 bits relative to the largest value that the inputs'
 * exponents allow, so each step's error is below a float64 rounding of that), and only the ten multiply-adds of the four results stay in
 * float64.
 *
 * A fixed-point number is an int64 F and an exponent X that depends on the
 * exponents of the inputs alone: value = F 2^X.  Products keep the upper 62 bits,
 * mul(a, b) = a b / 2^62, from 31-bit halves.  Both sides share the exponent of
 * the momenta, of the energies and of w, so that sums need no alignment.
 *
 * Measured (256 x 256 mesh, one launch, float64 form -> here): k_face 47 -> 21 us
 * (p = 1), 66 -> 29 (p = 2), 87 -> 37 (p = 3), 105 -> 45 (p = 4), 124 -> 54 (p = 5);
 * k_face_mixed 88 -> 42 us (p = 3), 403 -> 173 us (512 x 512, p = 4).  Against 113-bit arithmetic the
 * error is 0.75-1.0 of the float64 form's (rms) over still, slow, supersonic and
 * discontinuous states.
 *
 * A point whose sides differ by more than 2^4 in density or energy, whose state is
 * not physical or not finite, whose exponents are far from one (beyond 2^300), or
 * whose (gamma - 1) P w may be below the normal range, is left to the float64 form:
 * edge_flux_fixed returns false and writes nothing.
 */
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define DG_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#define DG_HD inline
#endif

namespace dg {

// Fixed-point form of a face's geometry: the scaled normal s = h n (h = l / 2) and
// hk = h^2 gamma (gamma - 1), in the scales of fixed_of (s with the larger
// component's exponent es, hk normalised to [2^61, 2^62) with its own, ek).
struct alignas(16) FaceFix {
  long long sx, sy, hk;
  int es, ek;               // biased float64 exponents; es < 0: not usable
};

namespace fx {

DG_HD long long bits_of(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  long long v;
  std::memcpy(&v, &x, 8);
  return v;
#endif
}
DG_HD double of_bits(long long v) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(v);
#else
  double x;
  std::memcpy(&x, &v, 8);
  return x;
#endif
}
DG_HD int clz64(unsigned long long v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}
// approximate reciprocal and reciprocal square root of a float32 (about 2^-22)
DG_HD float rcp32(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}
DG_HD float rsqrt32(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / std::sqrt(x);
#endif
}
DG_HD float float_of_bits(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float f;
  std::memcpy(&f, &b, 4);
  return f;
#endif
}
DG_HD int to_int(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int)std::lrint(x);
#endif
}

struct Half2x31 { int h, l; };                              // h 2^31 + l, 0 <= l < 2^31
DG_HD Half2x31 cut(long long x) { return Half2x31{(int)(x >> 31), (int)((uint32_t)x & 0x7FFFFFFFu)}; }
// a b / 2^62 (to within 2 units, downwards), |a|, |b| < 2^62
DG_HD long long mul(Half2x31 a, Half2x31 b) {
  const long long c = (long long)a.h * b.l + (long long)a.l * b.h;
  return (long long)a.h * b.h + (c >> 31);
}
// the same for a b4 / 2^64 of unsigned numbers, the second taken times four: on the
// device four multiplies, where the halves above take eight instructions of the
// busier pipe
DG_HD unsigned long long umul(unsigned long long a, unsigned long long b4) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b4);
#else
  return (unsigned long long)(((unsigned __int128)a * b4) >> 64);
#endif
}
DG_HD long long shr(long long x, int d) { return x >> (d < 63 ? d : 63); }

// the same, rounded to nearest (a small negative x gives 0, not -1)
DG_HD long long shr_rn(long long x, int d) {
  d = d < 62 ? d : 62;
  return (x + ((1ll << d) >> 1)) >> d;
}

// x 2^(1083 - e), truncated toward zero, for a float64 x of biased exponent at most
// e (e >= 63, so that a zero comes out as 0): below 2^61.  F32: x is a float32 number
// (its low 29 bits are zero), here and below: the same results.
template <bool F32 = false>
DG_HD long long fixed_of(double x, int e, unsigned long long *magnitude = nullptr) {
  const long long b = bits_of(x);
  const int hi = (int)(b >> 32);
  const int own = (hi >> 20) & 0x7FF;
  const uint32_t mh = ((uint32_t)hi & 0xFFFFFu) | 0x100000u, l = (uint32_t)b;
  const unsigned long long m = ((unsigned long long)((mh << 8) | (l >> 24)) << 32) | (F32 ? 0u : l << 8);
  const int d = e - own;
  const long long v = (long long)(m >> (d < 63 ? d : 63));
  if (magnitude) *magnitude = (unsigned long long)v;
  const long long s = (long long)(hi >> 31);
  return (v ^ s) - s;
}

// F 2^X -> float64, rounded to nearest (0 for F = 0); the result's exponent is in
// the normal range
DG_HD double to_double(long long F, int X) {
  const long long s = F >> 63;
  const unsigned long long a = (unsigned long long)((F ^ s) - s);
  const int z = clz64(a);
  const unsigned long long n = a << (z & 63);
  unsigned long long r = (n >> 11) + ((n >> 10) & 1ull);
  r += (unsigned long long)(uint32_t)(X + 1085 - z) << 52;   // biased exponent X + 1086 - z, less the leading bit
  r = a == 0ull ? 0ull : r;
  return of_bits((long long)(r | ((unsigned long long)s & 0x8000000000000000ull)));
}

// 1/m for the mantissa m in [1, 2) of a float64, times 2^62: in [2^61, 2^62].
// A float32 estimate y0 (23 bits) and its residual d = 1 - m y0, exact in 84 bits,
// give y0 (1 + d + d^2); the next term is below 2^-64.
template <bool F32 = false>
DG_HD long long recip_mantissa(double x) {
  const long long b = bits_of(x);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  const uint32_t mh = (hi & 0xFFFFFu) | 0x100000u;
  const int ah = (int)((mh << 10) | (lo >> 22)), al = F32 ? 0 : (int)((lo << 9) & 0x7FFFFFFFu);   // m 2^61 = ah 2^31 + al
  const float f = float_of_bits(0x3F800000u | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
  const int y = to_int(rcp32(f) * 8388608.0f);                                          // [2^22, 2^23]
  // e = 2^84 - y m 2^61 = d 2^84
  const long long u = (1ll << 53) - (long long)ah * y;
  const long long e = (long long)((unsigned long long)u << 31) - (long long)al * y;
  const int eh = (int)(e >> 32);                                                        // d 2^52
  const uint32_t el = (uint32_t)e;
  const long long z = (long long)y * eh + (long long)(((unsigned long long)(uint32_t)y * el) >> 32);   // y0 d 2^75
  const long long z2 = z + (((long long)(int)(z >> 31) * eh) >> 21);
  return ((long long)y << 39) + (z2 >> 13);
}

// 1/x as a float64, rounded to nearest (to 2^-60 before that).  The sign is x's; a
// zero, denormal or non-finite x gives NaN, a result below the normal range zero.
DG_HD double recip_fixed(double x) {
  const long long b = bits_of(x);
  const int e = (int)(b >> 52) & 0x7FF;
  const long long y = recip_mantissa(x);                       // [2^61, 2^62]
  long long r = ((y + 256) >> 9) + ((long long)(2044 - e) << 52);
  r = e >= 2045 ? 0 : r;
  r |= b & (long long)0x8000000000000000ull;
  r = (unsigned)(e - 1) >= 2046u ? 0x7FF8000000000000ll : r;
  return of_bits(r);
}

// 1/sqrt(x) as a float64, rounded to nearest (to 2^-58 before that), for a positive
// normal x; NaN for any other.  x = v 4^k with v in [2^60, 2^62); a float32 estimate
// y (23 bits) of 2^53 / sqrt(v) and its residual e = 1 - v y^2 / 2^106, exact to
// 2^-61, give y (1 + e/2 + 3 e^2 / 8); the next term is below 2^-64.
DG_HD double rsqrt_fixed(double x) {
  const long long b = bits_of(x);
  const int be = (int)(b >> 52);                                // biased exponent (negative: x < 0)
  const int odd = ~be & 1;                                      // be - 1083 odd
  const long long v = ((b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll) << (8 + odd);
  const int k = (be - 1083 - odd) >> 1;
  const Half2x31 c = cut(v);
  const int y = to_int(rsqrt32((float)c.h) * 194368031998.42758f);              // 2^37.5
  const long long t = ((long long)c.h * y << 8) + (((long long)c.l * y) >> 23);   // v y / 2^23
  const Half2x31 tc = cut(t);
  const long long u = (1ll << 52) - (long long)tc.h * y;
  const long long e = (long long)((unsigned long long)u << 31) - (long long)tc.l * y;   // e 2^83
  const int eh = (int)(e >> 32);
  const long long z = (long long)y * eh + (long long)(((unsigned long long)(uint32_t)y * (uint32_t)e) >> 32);   // y e 2^51
  const long long q = ((long long)(int)(z >> 31) * eh * 3) >> 36;
  const long long r = ((long long)y << 38) + (z >> 14) + q;                     // 2^91 / sqrt(v)
  const long long out = ((r + 128) >> 8) + ((long long)(991 - k) << 52);
  return of_bits((unsigned)(be - 1) >= 2046u ? 0x7FF8000000000000ll : out);
}

// sqrt(v) 2^30 for v in [2^58, 2^62): in [2^59, 2^61), to 2^-55
DG_HD long long sqrt_fixed(long long v) {
  const float f = (float)(int)(v >> 31);                        // v 2^-31, 24 bits
  const float r = rsqrt32(f);                                   // 2^15.5 / sqrt(v)
  // b: sqrt(v) to within 2^10 (sqrt(v) = 2^15.5 f r), 2^31 at most
  const uint32_t b = (uint32_t)to_int(f * r * 181.01933598375618f) << 8;    // 2^15.5 / 2^8 = 2^7.5
  const long long e = v - (long long)((unsigned long long)b * b);           // |e| < 2^42
  // sqrt(v) = b + e / (2 b): the correction, 2^30 times, with a float32 quotient
  const float h = r * 2.1579186437577746e-05f * 0.5f;           // 1 / (2 sqrt(v)): 2^-15.5 / 2
  const int t = to_int((float)(int)(e >> 11) * (h * 2147483648.0f));        // e / (2 b) 2^20, below 2^31
  const long long c1 = (long long)((unsigned long long)b << 30) + (long long)t * 1024;
  // the rest, from c1^2 / 2^62 against v / 4
  const int e1 = (int)((v >> 2) - (long long)umul((unsigned long long)c1, (unsigned long long)c1 * 4));
  const int t1 = to_int((float)e1 * (h * 4294967296.0f));
  return c1 + t1;
}

}  // namespace fx

DG_HD int exponent_of(double x) { return (int)((fx::bits_of(x) >> 52) & 0x7FF); }
DG_HD FaceFix face_fix(double sx, double sy, double hk) {
  const int ex = exponent_of(sx), ey = exponent_of(sy), es = ex > ey ? ex : ey, ek = exponent_of(hk);
  const bool in = es > 723 && es < 1323 && ek > 723 && ek < 1323 && hk > 0.0;
  return FaceFix{fx::fixed_of(sx, es), fx::fixed_of(sy, es), fx::fixed_of(hk, ek) * 2, in ? es : -1, ek};
}

// l F_hat as lax_friedrichs_edge; g1 = gamma - 1 in fixed_of scale with its own
// biased exponent eg.  False: this point is not in the range above, nothing written.
template <bool F32 = false>
DG_HD bool edge_flux_fixed(const double ul[4], const double ur[4], const FaceFix &g, double sx, double sy, long long g1,
                           int eg, double out[4]) {
  using namespace fx;
  const int hiL0 = (int)(bits_of(ul[0]) >> 32), hiR0 = (int)(bits_of(ur[0]) >> 32);
  const int hiL3 = (int)(bits_of(ul[3]) >> 32), hiR3 = (int)(bits_of(ur[3]) >> 32);
  const int rL = hiL0 >> 20, rR = hiR0 >> 20;                   // (negative for a negative value)
  const int eL = hiL3 >> 20, eR = hiR3 >> 20;
  const uint32_t m1 = (uint32_t)(bits_of(ul[1]) >> 32) & 0x7FFFFFFFu, m2 = (uint32_t)(bits_of(ul[2]) >> 32) & 0x7FFFFFFFu;
  const uint32_t m3 = (uint32_t)(bits_of(ur[1]) >> 32) & 0x7FFFFFFFu, m4 = (uint32_t)(bits_of(ur[2]) >> 32) & 0x7FFFFFFFu;
  const uint32_t m12 = m1 > m2 ? m1 : m2, m34 = m3 > m4 ? m3 : m4;
  // (momenta below 2^-823, zero among them, count as zero: fixed_of gives 0 from 63
  // exponents down)
  const uint32_t mm = m12 > m34 ? m12 : m34;
  const int em = (int)((mm > (200u << 20) ? mm : (200u << 20)) >> 20);
  const int r0 = rL < rR ? rL : rR, r1 = rL < rR ? rR : rL;
  const int e0 = eL < eR ? eL : eR, eE = eL < eR ? eR : eL;
  // shift of the kinetic energy K to the scale of E, which is taken six bits down for
  // the subtraction: K of a physical state is below E, but that of another may be up
  // to 2^6 times as large
  const int dK = eE + 6 - 2 * em + r0 - 2;
  // the last: below it H's exponent, eE + (em - r0 + es - 1080) + eg - 957 less up to 63
  // leading zeros, could be negative (P w of the smallest normal numbers and less)
  bool ok = (r0 > 723) & (r1 < 1323) & (r1 - r0 <= 4) & (e0 > 723) & (eE < 1323) & (eE - e0 <= 4) & (em < 1323) &
            (dK >= 0) & (g.es > 0) & (eE + em - r0 + g.es + eg >= 2100);
  if (!ok) return false;
  const Half2x31 Sx = cut(g.sx), Sy = cut(g.sy);
  const Half2x31 G1 = cut(g1);
  long long w[2], Pf[2], yc[2], c[2];
  int xc[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const double *u = s ? ur : ul;
    const int re = s ? rR : rL;
    const long long y = recip_mantissa<F32>(u[0]);                   // 1/rho = y 2^(961 - re)
    yc[s] = y < (1ll << 62) ? y : (1ll << 62) - 1;
    const long long I = yc[s] >> (1 + re - r0);                 // 1/rho = I 2^(962 - r0)
    unsigned long long ax, ay;
    const Half2x31 Mx = cut(fixed_of<F32>(u[1], em, &ax)), My = cut(fixed_of<F32>(u[2], em, &ay));
    const long long mn = mul(Mx, Sx) + mul(My, Sy);
    const long long sn = mn >> 63;                              // X = em + es - r0 - 1080
    w[s] = ((long long)umul((unsigned long long)((mn ^ sn) - sn), (unsigned long long)I * 4) ^ sn) - sn;
    const unsigned long long q = umul(ax, ax * 4) + umul(ay, ay * 4);
    const long long K = (long long)umul(q, (unsigned long long)I * 4);   // |m|^2 / rho, X = 2 em - r0 - 1080
    // E - K lies in (-2^60, 2^55): its sign is taken before the scaling by 2^6, which
    // only a positive one leaves room for
    const long long d = fixed_of<F32>(u[3], eE + 6) - shr(K, dK);
    ok &= d > 0;
    Pf[s] = (long long)((unsigned long long)d << 6);            // p / (gamma - 1), X = eE - 1083
  }
  if (!ok) return false;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int z = clz64((unsigned long long)Pf[s]) - 2;         // Pf 2^z in [2^61, 2^62)
    const unsigned long long Pn = (unsigned long long)Pf[s] << z;
    // c^2 = hk P / rho, h^2 folded in: X = eE - 1083 - z - re + ek + 1
    long long c2 = (long long)umul(umul(Pn, (unsigned long long)yc[s] * 4), (unsigned long long)g.hk * 4);
    int x2 = eE - 1082 - z - (s ? rR : rL) + g.ek;
    c2 = (x2 & 1) ? c2 >> 1 : c2;
    x2 += x2 & 1;
    c[s] = sqrt_fixed(c2);
    xc[s] = x2 / 2 - 30;
  }
  const int xw = em + g.es - r0 - 1080;
  int xa = xw > xc[0] ? xw : xc[0];
  xa = (xa > xc[1] ? xa : xc[1]) + 1;
  const long long wl = shr_rn(w[0], xa - xw), wr = shr_rn(w[1], xa - xw);
  const long long al = (wl < 0 ? -wl : wl) + shr(c[0], xa - xc[0]), ar = (wr < 0 ? -wr : wr) + shr(c[1], xa - xc[1]);
  const long long la = al > ar ? al : ar;
  const double wa = to_double(wl + la, xa), wb = to_double(wr - la, xa);
  // (gamma - 1) (P_l + P_r) and (gamma - 1) (P_l w_l + P_r w_r)
  const double ps = to_double((long long)umul((unsigned long long)(Pf[0] + Pf[1]) >> 1, (unsigned long long)g1 * 4), eE - 1083 + 1 + 62 + eg - 1083);
  const long long pw = mul(cut(Pf[0]), cut(w[0])) + mul(cut(Pf[1]), cut(w[1]));
  const double H = to_double(mul(cut(pw), G1), eE - 1083 + 62 + xw + 62 + eg - 1083);
#ifdef __CUDA_ARCH__
  out[0] = fma(ul[0], wa, ur[0] * wb);
  out[1] = fma(ul[1], wa, fma(ur[1], wb, ps * sx));
  out[2] = fma(ul[2], wa, fma(ur[2], wb, ps * sy));
  out[3] = fma(ul[3], wa, fma(ur[3], wb, H));
#else
  out[0] = std::fma(ul[0], wa, ur[0] * wb);
  out[1] = std::fma(ul[1], wa, std::fma(ur[1], wb, ps * sx));
  out[2] = std::fma(ul[2], wa, std::fma(ur[2], wb, ps * sy));
  out[3] = std::fma(ul[3], wa, std::fma(ur[3], wb, H));
#endif
  return true;
}

}  // namespace dg
