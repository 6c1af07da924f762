// FP64 mat-vecs on the integer multiply-add units.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM, but 32 32 x 32 -> 64 bit
// integer multiply-adds (mad.wide.s32).  A real
// number of a mat-vec is therefore held as a 55-bit fixed-point value in two
// words,
//   v = (h 2^27 + l) 2^(E - 55),   |h| <= 2^28, |l| < 2^27,
// relative to an exponent E of its block (all links: one for the field;
// colour vectors: one per output site, raised while its 16 neighbours are
// read), and a product is three integer multiply-adds into two 64-bit sums,
//   hi += ah bh,   mid += ah bl + al bh,
// exact but for the term al bl (2^-57 of the blocks' scales at most), which is
// dropped.  The sums over the 96 real products of an output component neither
// round nor overflow:
//   |hi| <= 96 2^56 < 2^63,  |mid| <= 96 (2^28 2^27 + 2^26 2^28) < 2^63
// (the links' low words are balanced, |al| <= 2^26).  The result is rounded to
// FP64 once; a chain of FP64 FMAs rounds at each of its 96 steps.  Against a
// long-double Dslash of Gaussian vectors the 2-norm error is 1.5e-16, with
// FP64 FMAs 3.5e-16 (2.7e-16 against 3.5e-16 where neighbouring sites differ
// by factors up to e^8), the largest error of a component 5e-16 against 2e-15.
//
// The long links are 24 times smaller than the fat ones as a rule, and have 50 of
// the 55 bits; a neighbour much smaller than the site's largest has fewer too.
// That is enough beside the terms of the fat links and the larger neighbours, but
// not where the vector reaches a site by the long links only, or almost (point and
// wall sources, steep decays): such sites, told by the exponents of the vectors,
// are computed again with the two kinds apart, for which the long links' words
// hold FX_MORE more bits.  Rms over the sites of the error relative to the site, a
// point source's long-hop sites 2.0e-15 -> 8.8e-17; Gaussian vectors that decay in
// t as exp(-k |t|), 8^3 x 16, against a C Dslash in FP64:
//   k            0        0.5      0.7      1        1.5      2        3
//   before       1.9e-16  2.4e-16  3.2e-16  5.9e-16  1.5e-15  2.2e-15  2.3e-15
//   here         1.9e-16  2.3e-16  2.6e-16  2.5e-16  2.2e-16  2.3e-16  2.2e-16
//   FP64 FMAs    1.9e-16  1.9e-16  1.8e-16  1.7e-16  1.5e-16  1.3e-16  1.2e-16
// dirac_apply at 20^3 x 64: 221 us, with a point source 202, a wall 268, and 585
// where every site is computed again (k = 1; with FP64 FMAs 867 for any vector).
//
// What it bounds: the FP64 Dslash of one system at 20^3 x 64 went from
// 321.6 us (FP64 units 100 % busy) to 111 us, 0.82 of the HBM rate for its
// 2400 bytes per site; with 12 systems, where the links are read once, from
// 3550 to 1010 us (350 instructions per hop and system, 16 warps per SM: bound
// by their latency).
#pragma once

#include "sq_device.cuh"

namespace sq {

constexpr int FX_LOW = 27;                 // bits of a low word
constexpr int FX_BITS = 55;                // bits of a value
constexpr int FX_LOW_MASK = (1 << FX_LOW) - 1;
constexpr int FX_MORE = 5;                 // further bits of a long link
// A nonzero link's largest element is at least 2^-FX_FAT_LEAST (fat) or
// 2^-FX_LONG_LEAST (long) of the field's scale, and so held to 2^-51 of itself.
constexpr int FX_FAT_LEAST = 5, FX_LONG_LEAST = 9;
// How far the exponent of a site's largest fat-hop neighbour may be below that of
// all its neighbours: at most 8 times smaller, which costs 2.6e-16 (table above).
// In Gaussian vectors they are never further apart (all 48 components by fat hops
// 4 times smaller than one by long hops: some 10^-9 of the sites); with 1 here the
// sites of random fields that are cost 19 % of the time.
constexpr int FX_KINDS_APART = 2;
// Biased FP64 exponents the fixed-point path takes: below FX_MIN_E a vector
// counts as zero at every scale in use, from FX_MAX_E on (which includes
// infinities and NaN) the site is computed with FP64 FMAs.
constexpr int FX_MIN_E = 128, FX_MAX_E = 1900;

struct Fx { int h, l; };
struct FxVec { Fx re[3], im[3]; };

__device__ __forceinline__ int fx_hi_word(double v) { return __double2hiint(v); }

// Largest biased exponent of a colour vector's six components.
__device__ __forceinline__ int fx_max_exponent(const Vec3<double> &v) {
  int m = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    m = max(m, fx_hi_word(v.c[c].x) & 0x7fffffff);
    m = max(m, fx_hi_word(v.c[c].y) & 0x7fffffff);
  }
  return m >> 20;
}
__device__ __forceinline__ bool fx_any_nonzero(const Vec3<double> &v) {
  int m = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c)
    m |= (fx_hi_word(v.c[c].x) << 1) | __double2loint(v.c[c].x) | (fx_hi_word(v.c[c].y) << 1) |
         __double2loint(v.c[c].y);
  return m != 0;
}

// v (biased exponent <= E) as a fixed-point value relative to 2^(E - 1022),
// times sgn (+1 or -1): the 53-bit mantissa, shifted up by 2 and down by the
// distance of the exponents, the bits below the last one dropped.
__device__ __forceinline__ Fx fx_from_double(double v, int E, int sgn) {
  const unsigned H = (unsigned)__double2hiint(v), L = (unsigned)__double2loint(v);
  const int d = E - (int)((H >> 20) & 0x7ff);
  const unsigned mh = (H & 0xfffff) | 0x100000;
  const unsigned Mh = __funnelshift_l(L, mh, 2);
  unsigned Ml = __funnelshift_rc(L << 2, Mh, d);         // clamps at 32: then the high word
  Ml = __funnelshift_rc(Ml, 0, max(d - 32, 0));
  const unsigned Mr = __funnelshift_rc(Mh, 0, d);
  const int s = ((int)H >> 31) ^ (sgn >> 31);            // 0 or -1
  Fx o;
  o.h = ((int)__funnelshift_l(Ml, Mr, 32 - FX_LOW) ^ s) - s;
  o.l = ((int)(Ml & FX_LOW_MASK) ^ s) - s;
  return o;
}

// FP32 value as the FP64 value of the same number without the conversion
// unit; zero for zero and for FP32 denormals, infinities and NaN kept.
__device__ __forceinline__ double fx_widen(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned e = (b >> 23) & 0xff;
  unsigned E = e + 896;
  E = (e == 255) ? 2047 : E;
  const unsigned H = (b & 0x80000000u) | (E << 20) | ((b & 0x7fffff) >> 3);
  return e == 0 ? 0.0 : __hiloint2double((int)H, (int)(b << 29));
}

// In PTX: written as 64-bit C++ products the compiler turns some of them (words
// cut out of 64-bit values) into three instructions.
__device__ __forceinline__ void fx_mac1(long long &s, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s) : "r"(a), "r"(b));
}
__device__ __forceinline__ void fx_mac(long long &hi, long long &mid, const Fx a, const Fx b) {
  fx_mac1(hi, a.h, b.h);
  fx_mac1(mid, a.h, b.l);
  fx_mac1(mid, a.l, b.h);
}

struct FxAcc {
  long long hr[3], mr[3], hi[3], mi[3];  // real part: hr, mr; imaginary part: hi, mi
  int E;                                 // the vectors' exponent
};

__device__ __forceinline__ void fx_zero(FxAcc &a) {
#pragma unroll
  for (int c = 0; c < 3; ++c) a.hr[c] = a.mr[c] = a.hi[c] = a.mi[c] = 0;
  a.E = FX_MIN_E;
}

// Raise the exponent of the sums to E.
__device__ __forceinline__ void fx_raise(FxAcc &a, int E) {
  const int s = min(E - a.E, 63);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a.hr[c] >>= s; a.mr[c] >>= s;
    a.hi[c] >>= s; a.mi[c] >>= s;
  }
  a.E = E;
}

// acc += M v, M given as 9 (re, im) pairs of fixed-point values
__device__ __forceinline__ void fx_mat_vec(FxAcc &a, const int4 (&m)[9], const FxVec &v) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Fx nim = {-v.im[c].h, -v.im[c].l};
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int4 q = m[3 * r + c];
      const Fx mr = {q.y, q.x}, mi = {q.w, q.z};
      fx_mac(a.hr[r], a.mr[r], mr, v.re[c]);
      fx_mac(a.hi[r], a.mi[r], mr, v.im[c]);
      fx_mac(a.hr[r], a.mr[r], mi, nim);
      fx_mac(a.hi[r], a.mi[r], mi, v.re[c]);
    }
  }
}

// Colour c of the vector v (XS: v + d) relative to E, times sgn.
template <bool XS>
__device__ __forceinline__ void fx_colour(const Vec3<double> &v, const Vec3<double> &d, int E, int sgn,
                                          int c, Fx &re, Fx &im) {
  re = fx_from_double(v.c[c].x, E, sgn);
  im = fx_from_double(v.c[c].y, E, sgn);
  if (XS) {
    const Fx p = fx_from_double(d.c[c].x, E, sgn), q = fx_from_double(d.c[c].y, E, sgn);
    const int lr = re.l + p.l, li = im.l + q.l;
    re.h += p.h + (lr >> FX_LOW);
    re.l = lr & FX_LOW_MASK;
    im.h += q.h + (li >> FX_LOW);
    im.l = li & FX_LOW_MASK;
  }
}

// Products are in units of 2^(fixed_exp - FX_BITS) 2^(E - 1022 - FX_BITS), the
// sums' hi of 2^(2 FX_LOW) of these: that unit.
__device__ __forceinline__ double fx_unit(int fixed_exp, int E) {
  const int ex = fixed_exp + E - 1022 - 2 * FX_BITS + 2 * FX_LOW;
  return __hiloint2double((ex + 1023) << 20, 0);
}

// (hi 2^27 + mid) 2^27 in units of the operands' last bits, times `unit`
__device__ __forceinline__ double fx_to_double(long long hi, long long mid, double unit) {
  const double d = (double)(hi + (mid >> FX_LOW));
  const double r = (double)((int)mid & FX_LOW_MASK);
  return fma(r, 1.0 / (1 << FX_LOW), d) * unit;
}

// Stored form of a link element: (re.l, re.h, im.l, im.h), low words balanced.
__device__ __forceinline__ int2 fx_link_word(double v, double to_fixed) {
  const long long q = __double2ll_rn(v * to_fixed);
  const long long h = (q + (1ll << (FX_LOW - 1))) >> FX_LOW;
  return make_int2((int)(q - (h << FX_LOW)), (int)h);
}
// Of a long link: the low word 2^FX_MORE l + x, x = 0 .. 2^FX_MORE - 1 the further
// bits with half of their range added, so that a shift gives the rounded l.
__device__ __forceinline__ int2 fx_long_word(double v, double to_fixed) {
  constexpr int half = 1 << (FX_MORE - 1);
  const long long more = __double2ll_rn(v * (to_fixed * (1 << FX_MORE))) + half;
  const long long q = more >> FX_MORE, h = (q + (1ll << (FX_LOW - 1))) >> FX_LOW;
  return make_int2((int)(more - (h << (FX_LOW + FX_MORE))), (int)h);
}
__device__ __forceinline__ int4 fx_long_element(int4 q) {
  return make_int4(q.x >> FX_MORE, q.y, q.z >> FX_MORE, q.w);
}
__device__ __forceinline__ int fx_long_rest(int l) {
  return (l & ((1 << FX_MORE) - 1)) - (1 << (FX_MORE - 1));
}

}  // namespace sq
