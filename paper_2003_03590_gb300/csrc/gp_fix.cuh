// gp_fix.cuh -- 64-bit fixed-point arithmetic of the float64 transforms.
//
// GB300 executes 2 float64 operations per clock and SM but 128 integer ones: the float64 sweeps spent
// all their time in DADD / DFMA issue (one 256-point transform of a 256^3 field 0.73 ms, where its
// memory traffic takes 0.08 ms).  A transform is sums and rotations of numbers of one scale, which is
// what fixed point does: an addition is two integer instructions, a multiplication by a known
// |factor| <= 1 about a dozen, and both run on the wide integer pipes.
//
// Scale.  Every pencil has its own power of two: with S1 >= sum |z_i| over the pencil, values are kept
// as integers of unit S1 2^-62 (components below 2^62).  Every intermediate of the transform is a
// partial sum of rotated inputs, so its modulus is below S1 and nothing overflows, and the unit is at
// most L rms 2^-62: for the lengths here the inputs' rounding and the products' roundings (half a
// unit each, unbiased) stay below what a float64 transform of the pencil loses (relative to the
// pencil's norm, 256 points, random data: 0.65e-16 against 2.2e-16).  Values that are
// tiny beside the pencil's norm lose digits to the unit -- as they do, to the same rounding, in any
// float64 transform that mixes them with the pencil's large values.
//
// Products.  x * c for |c| <= 1 takes unsigned 64 x 64 products only: with x' = x + 2^63 (a flipped
// sign bit) and c64 = c 2^64, hi(x' c64) - c64 / 2 = x c for c in (0, 1); for a table factor of either
// sign u = (c + 1) / 2 is stored and x c = 2 x u - x.  The low x low partial product enters by its
// mean and half a unit is added before the cut, so the rounding is unbiased.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstring>

namespace gp {

struct cfix {
  long long x, y;
};
struct ufix2 {   // a table factor c + i s as ((c + 1) / 2, (s + 1) / 2) in units of 2^-64, even
  unsigned long long c, s;
};

// a component v of a table factor as ufix2 holds it.  The product of two rounded unit factors can lie an
// ulp outside [-1, 1]: it counts as 1 or -1 (unclamped, the sum below would wrap to the other sign).
inline unsigned long long fix_factor(double v) {
  if (!(v < 1.0)) return ~1ull;   // NaN too (see FixArgs::bad)
  if (v <= -1.0) return 0;
  return ((unsigned long long)(long long)std::nearbyint(std::ldexp(v, 62)) << 1) + (1ull << 63);   // (v + 1) 2^63
}

#define GP_HD __host__ __device__ __forceinline__

// (a b) / 2^64 rounded, the low x low partial product replaced by its mean
GP_HD unsigned long long umulhi_r(unsigned long long a, unsigned long long b) {
  const unsigned al = (unsigned)a, ah = (unsigned)(a >> 32), bl = (unsigned)b, bh = (unsigned)(b >> 32);
  const unsigned long long m = (unsigned long long)al * bh + 0xC0000000ull;   // 1/2 unit + mean of al bl 2^-32
  const unsigned long long n = (unsigned long long)ah * bl + (unsigned)m;
  return (unsigned long long)ah * bh + (m >> 32) + (n >> 32);
}
// x * c for a constant c in (0, 1), c64 = c 2^64 (even)
GP_HD long long fmulc(long long x, unsigned long long c64) {
  return (long long)(umulhi_r((unsigned long long)x ^ (1ull << 63), c64) - (c64 >> 1));
}
// z * (c + i s) for a table factor; |x|, |y| < 2^62
GP_HD cfix ftwmul(cfix z, ufix2 w) {
  const unsigned long long X = ((unsigned long long)z.x << 1) ^ (1ull << 63), Y = ((unsigned long long)z.y << 1) ^ (1ull << 63);
  const unsigned long long hc = w.c >> 1, hs = w.s >> 1;
  const long long xc = (long long)(umulhi_r(X, w.c) - hc) - z.x, ys = (long long)(umulhi_r(Y, w.s) - hs) - z.y;
  const long long xs = (long long)(umulhi_r(X, w.s) - hs) - z.x, yc = (long long)(umulhi_r(Y, w.c) - hc) - z.y;
  return cfix{xc - ys, xs + yc};
}

GP_HD cfix cadd(cfix a, cfix b) { return cfix{a.x + b.x, a.y + b.y}; }
GP_HD cfix csub(cfix a, cfix b) { return cfix{a.x - b.x, a.y - b.y}; }
template <bool INV> GP_HD cfix fmul_mi(cfix a) { return INV ? cfix{-a.y, a.x} : cfix{a.y, -a.x}; }

// cos(k pi / 16) 2^64, k = 1 .. 7, and sqrt(3)/2, 2/3 (even)
__host__ __device__ constexpr unsigned long long fix_cos(int k) {
  return k == 1 ? 0xfb14be7fbae58156ull
         : k == 2 ? 0xec835e79946a3146ull
         : k == 3 ? 0xd4db3148750d181aull
         : k == 4 ? 0xb504f333f9de6484ull
         : k == 5 ? 0x8e39d9cd73464364ull
         : k == 6 ? 0x61f78a9abaa58b46ull
         : 0x31f17078d34c156cull;
}
constexpr unsigned long long FIX_R2 = fix_cos(4), FIX_H3 = 0xddb3d742c265539eull, FIX_23 = 0xaaaaaaaaaaaaaaaaull;

// a * (c - i s) forward, a * (c + i s) inverse, c and s in (0, 1)
template <bool INV> GP_HD cfix frot(cfix a, unsigned long long c, unsigned long long s) {
  const long long xc = fmulc(a.x, c), ys = fmulc(a.y, s), yc = fmulc(a.y, c), xs = fmulc(a.x, s);
  return INV ? cfix{xc - ys, yc + xs} : cfix{xc + ys, yc - xs};
}
template <bool INV> GP_HD cfix frot45(cfix a) {   // * exp(-+ i pi/4)
  return INV ? cfix{fmulc(a.x - a.y, FIX_R2), fmulc(a.x + a.y, FIX_R2)}
             : cfix{fmulc(a.x + a.y, FIX_R2), fmulc(a.y - a.x, FIX_R2)};
}
// a * w32^EXP (forward, w32 = exp(-2 pi i / 32)) or its conjugate (inverse): a quarter turn at most
// by the signs, then a rotation by less than pi/2
template <bool INV, int EXP> GP_HD cfix frot32(cfix a) {
  constexpr int q = (EXP % 32) / 8, e = EXP % 8;
  if constexpr (q == 1) a = fmul_mi<INV>(a);
  if constexpr (q == 2) a = cfix{-a.x, -a.y};
  if constexpr (q == 3) a = fmul_mi<!INV>(a);
  if constexpr (e == 4) return frot45<INV>(a);
  else if constexpr (e != 0) {
    constexpr unsigned long long c = fix_cos(e), s = fix_cos(8 - e);
    return frot<INV>(a, c, s);
  }
  else return a;
}

template <bool INV> GP_HD void fdft4(cfix& a0, cfix& a1, cfix& a2, cfix& a3) {
  const cfix s0 = cadd(a0, a2), d0 = csub(a0, a2), s1 = cadd(a1, a3), d1 = csub(a1, a3);
  a0 = cadd(s0, s1);
  a2 = csub(s0, s1);
  const cfix m = fmul_mi<INV>(d1);
  a1 = cadd(d0, m);
  a3 = csub(d0, m);
}
template <bool INV> GP_HD void fdft8(cfix* v) {
  cfix e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  fdft4<INV>(e0, e1, e2, e3);
  fdft4<INV>(o0, o1, o2, o3);
  o1 = frot32<INV, 4>(o1);
  o2 = frot32<INV, 8>(o2);
  o3 = frot32<INV, 12>(o3);
  v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}
// R = 4 Q: Q-point transforms of the stride-4 subsequences, twiddles w_R^(n2 k1), 4-point ones over n2
template <bool INV, int Q, int K1 = 1> GP_HD void ftwid4(cfix* y) {
  if constexpr (K1 < Q) {
    y[4 * K1 + 1] = frot32<INV, (32 / (4 * Q)) * K1>(y[4 * K1 + 1]);
    y[4 * K1 + 2] = frot32<INV, 2 * (32 / (4 * Q)) * K1>(y[4 * K1 + 2]);
    y[4 * K1 + 3] = frot32<INV, 3 * (32 / (4 * Q)) * K1>(y[4 * K1 + 3]);
    ftwid4<INV, Q, K1 + 1>(y);
  }
}
template <bool INV, int Q> GP_HD void fdft4q(cfix* v) {
  cfix y[4 * Q];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
    cfix u[Q];
#pragma unroll
    for (int n1 = 0; n1 < Q; ++n1) u[n1] = v[4 * n1 + n2];
    if constexpr (Q == 8) fdft8<INV>(u);
    else fdft4<INV>(u[0], u[1], u[2], u[3]);
#pragma unroll
    for (int k1 = 0; k1 < Q; ++k1) y[4 * k1 + n2] = u[k1];
  }
  ftwid4<INV, Q>(y);
#pragma unroll
  for (int k1 = 0; k1 < Q; ++k1) {
    fdft4<INV>(y[4 * k1], y[4 * k1 + 1], y[4 * k1 + 2], y[4 * k1 + 3]);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[k1 + Q * k2] = y[4 * k1 + k2];
  }
}
template <bool INV> GP_HD void fdft3(cfix& a0, cfix& a1, cfix& a2) {
  const cfix t1 = cadd(a1, a2), d = csub(a1, a2);
  // a0 - t1 / 2, rounded up for one component and down for the other
  const cfix t2{a0.x - (t1.x >> 1), a0.y - ((t1.y + 1) >> 1)};
  const cfix t3 = fmul_mi<INV>(cfix{fmulc(d.x, FIX_H3), fmulc(d.y, FIX_H3)});   // -+ i (a1 - a2) sqrt(3)/2
  a0 = cadd(a0, t1);
  a1 = cadd(t2, t3);
  a2 = csub(t2, t3);
}
template <int R, bool INV> GP_HD void fdft(cfix* v) {
  if constexpr (R == 3) fdft3<INV>(v[0], v[1], v[2]);
  else if constexpr (R == 4) fdft4<INV>(v[0], v[1], v[2], v[3]);
  else if constexpr (R == 8) fdft8<INV>(v);
  else if constexpr (R == 16) fdft4q<INV, 4>(v);
  else fdft4q<INV, 8>(v);
}

// ---------------------------------------------------------------- float64 <-> fixed point
// an upper bound of the modulus of (a, b), a, b >= 0
GP_HD float mod_bound(float a, float b) { return a > b ? a + 0.41421360f * b : b + 0.41421360f * a; }

// v / 2^sh rounded to nearest, ties to even (a fixed direction would bias the norm: at 1024 points one
// value in two is a tie); 0 < sh < 64
GP_HD unsigned long long round_shift(unsigned long long v, int sh) {
  const unsigned long long q = v >> sh;
  return (v + ((1ull << (sh - 1)) - 1) + (q & 1)) >> sh;
}
// v 2^-r: rounded as round_shift for r > 0, exact for r <= 0
GP_HD long long rescale1(long long v, int r) {
  if (r <= 0) return v << (r > -64 ? -r : 63);
  if (r > 63) return 0;
  return (v + (long long)((1ull << (r - 1)) - 1) + ((v >> r) & 1)) >> r;
}
// d * 2^s rounded to an integer, d given by its bits; |d| 2^s < 2^62
GP_HD long long to_fix(unsigned long long bits, int s) {
  const int e = (int)((bits >> 52) & 0x7ff);
  unsigned long long m = bits & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  const int sh = (e ? e : 1) - 1075 + s;
  unsigned long long v;
  if (sh >= 0) v = m << sh;
  else if (sh > -55) v = round_shift(m, -sh);
  else v = 0;
  return (long long)bits < 0 ? -(long long)v : (long long)v;
}
// bits of v * 2^-s rounded to a double (|v| < 2^63)
GP_HD unsigned long long from_fix(long long v, int s) {
  const unsigned long long sign = (unsigned long long)v & (1ull << 63);
  unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = a ? __builtin_clzll(a) : 64;
#endif
  if (lz == 64) return sign;
  a <<= lz;                                            // bit 63 set
  // 53 bits kept; a carry out of the mantissa adds to the exponent
  const unsigned low = (unsigned)a & 0x7ffu;
  unsigned long long r = a >> 11;
  r += low > 0x400u || (low == 0x400u && (r & 1));
  const int e = 1085 - lz - s;
  if (e < 0 || e >= 2046) {                            // outside the normal range
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(scalbn((double)v, -s));
#else
    const double d = scalbn((double)v, -s);
    unsigned long long b;
    memcpy(&b, &d, 8);
    return b;
#endif
  }
  return sign | (((unsigned long long)e << 52) + r);
}

// ---------------------------------------------------------------- N(s) in fixed point
// psi <- exp(-i coef (|psi|^2 - shift)) psi.  The phase is kept as a fraction of a turn in units of
// 2^-64, which wraps by itself: turns = |psi|^2 kappa - shift kappa, kappa = coef / (2 pi) = m 2^-q.
// cos and sin of the phase: a table of 256 directions, and for the rest |theta| <= pi / 256 the
// Taylor series 1 - z/2 + z^2/24 - z^3/720 and theta (1 - z/6 + z^2/120 - z^3/5040), z = theta^2 (the
// first omitted terms are below 2^-66).
struct NlFix {
  unsigned long long m;   // 2^63 <= m < 2^64, or 0 for coef = 0
  unsigned long long tc;  // |shift kappa| modulo 1 in units of 2^-64
  int q;
  int neg;                // coef < 0
};
// from float64 coefficients, in integers (the same on every host)
inline NlFix nl_fix(double coef, double shift) {
  NlFix f{0, 0, 0, coef < 0.0 ? 1 : 0};
  int e = 0;
  const double mant = std::frexp(std::fabs(coef), &e);          // |coef| = mant 2^e
  if (mant == 0.0 || !std::isfinite(coef)) return f;            // (not finite: FixArgs::bad)
  const unsigned long long c = (unsigned long long)std::ldexp(mant, 53) << 11;   // mant 2^64
  // 1 / (2 pi) = 0x28BE60DB9391054A.7F09D5F47D4D3770 2^-64
  typedef unsigned __int128 u128;
  u128 p = (u128)c * 0x28BE60DB9391054Aull + (((u128)c * 0x7F09D5F47D4D3770ull) >> 64);   // mant / (2 pi) 2^128
  int lz = 0;
  while (!(p >> 127)) p <<= 1, ++lz;
  f.m = (unsigned long long)(p >> 64);                          // |kappa| = m 2^(e - 64 - lz)
  f.q = 64 + lz - e;
  if (shift != 0.0) f.tc = f.q >= 128 ? 0 : (f.q >= 64 ? f.m >> (f.q - 64) : (f.q > 0 ? f.m << (64 - f.q) : 0));
  return f;
}
GP_HD unsigned long long uhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
GP_HD long long smulhi(long long a, long long b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (long long)(((__int128)a * b) >> 64);
#endif
}
// (p 2^64 + l) >> sh, the low 64 bits
GP_HD unsigned long long shift128(unsigned long long p, unsigned long long l, int sh) {
  if (sh >= 128 || sh <= -64) return 0;
  if (sh >= 64) return p >> (sh - 64);
  if (sh > 0) return (l >> sh) | (p << (64 - sh));
  return l << -sh;
}
// v: fixed point with v 2^-s = psi, |components| < 2^62 (the larger, the more digits of |psi|^2);
// dir: the 256 directions exp(+2 pi i k / 256)
// (sh = 2 s + q - 126; not inlined: about 250 instructions, which unrolled over a thread's elements
// would not fit the instruction cache)
#ifdef __CUDACC__
__host__ __device__ __noinline__ static
#else
inline
#endif
cfix fnonlinear(cfix v, int sh, unsigned long long fm, unsigned long long tc, int neg, const ufix2* __restrict__ dir) {
  const unsigned long long ax = (unsigned long long)(v.x < 0 ? -v.x : v.x), ay = (unsigned long long)(v.y < 0 ? -v.y : v.y);
  const unsigned long long w = uhi(ax << 1, ax << 1) + uhi(ay << 1, ay << 1);   // |psi|^2 2^(2 s - 62)
  unsigned long long T = shift128(uhi(w, fm), w * fm, sh) - tc;
  if (!neg) T = 0ull - T;                                   // the phase of the factor
  const unsigned k = (unsigned)((T + (1ull << 55)) >> 56) & 255u;
  const long long r = (long long)(T - ((unsigned long long)k << 56));           // [-2^55, 2^55)
  const long long rho = fmulc(r * 256, 0xC90FDAA22168C234ull);   // theta 2^69 (constant: pi / 4)
  const unsigned long long ar = (unsigned long long)(rho < 0 ? -rho : rho);
  const unsigned long long z = uhi(ar, ar);                   // theta^2 2^74
  const unsigned long long z4 = uhi(z, z);                    // theta^4 2^84
  const unsigned u = (unsigned)(z4 >> 27);                    // theta^4 2^57
  const unsigned u6 = (unsigned)(((unsigned long long)u * (unsigned)(z >> 30)) >> 32);   // theta^6 2^69
  // 1 - cos and 1 - sin / theta in units of 2^-64
  const unsigned long long cm = (z >> 11) - (((unsigned long long)u * 2863311531u) >> 29) + (((unsigned long long)u6 * 186414u) >> 32);
  const unsigned long long sm = (uhi(z, 0x2AAAAAAAAAAAAAAAull) >> 10) - (((unsigned long long)u * 2290649225u) >> 31) +
                                (((unsigned long long)u6 * 26631u) >> 32);
  const long long sn = rho - fmulc(rho, sm & ~1ull);          // sin(theta) 2^69
#ifdef __CUDA_ARCH__
  const ulonglong2 d2 = __ldg(reinterpret_cast<const ulonglong2*>(dir + k));
  const cfix a = ftwmul(v, ufix2{d2.x, d2.y});
#else
  const cfix a = ftwmul(v, dir[k]);
#endif
  const unsigned long long c1 = cm & ~1ull;
  const long long ys = (smulhi(a.y, sn) + 16) >> 5, xs = (smulhi(a.x, sn) + 16) >> 5;
  return cfix{a.x - fmulc(a.x, c1) - ys, a.y - fmulc(a.y, c1) + xs};
}

}  // namespace gp
