// Fixed-point contraction of FP64 numbers with integer multiply-adds.
//
// The FP64 pipe does 1.8 multiply-adds per clock and SM, the integer pipe tens of
// 32 x 32 -> 64 bit ones, and a sum of products needs no exponents of its own once
// every number is taken relative to a power of two, as in a symmetric contraction
//   H_rc = 2^(a_r + a_c) h_rc,  x_c = 2^(Z - a_c) y_c,  |h|, |y| < 1,
//   sigma_r = 2^(a_r + Z) sum_c h_rc y_c,
// with one exponent a for the unknowns of F and one for the order parameters
// (per point, from the largest entries of the three parts of H) and one Z per
// point. h and y are 58-bit integers in two limbs of 29 bits with their sign, cut
// towards zero. Of the four limb products the leading one (below 2^58) goes to s1 and
// the two middle ones to s0; the last one, below 2^-58 of the product's scale, is left
// out. A sum takes FX_TERMS = 16 products at most: then s1 < 2^62, s0 < 2^63 - 2^35 and
// 2 s1 + s0 2^-28 < 2^63 - 2^7. Error of n products: two cut operands and the product
// left out, 2^-58 of 2^(a_r + Z) each, and 2^-59 for the final shift: at most
// (3 n + 1/2) 2^-58 of 2^(a_r + Z), whatever the size of the row's own terms.
// Used where the numbers of a sum share their scale: the rank-16 updates of the coarse
// inverse (one power of two per row and column of a tile) and the order-parameter
// columns of the Hessian. Not in the FP64 tangent application: its error is relative to
// 2^(a_r + Z), not to the row's own terms, and a penalty of 1e3 to 1e9 on one order
// parameter lifts that above the other rows' terms (in the root mean square of a row's
// error over sum |h x| 3.6e-15 in place of FP64's 7e-17 at 1e3, 1.5e-8 at 1e9). It took
// 426 us on 61x45x33 elements there against 581 us in FP64.
// Compiles for the host too (test of the arithmetic).
#pragma once

#include <cstdint>
#include <cstring>

namespace pfm {

#ifdef __CUDACC__
#define PFM_FX __host__ __device__ __forceinline__
#else
#define PFM_FX inline
#endif

PFM_FX uint64_t fx_bits(double v) {
#ifdef __CUDA_ARCH__
  return static_cast<uint64_t>(__double_as_longlong(v));
#else
  uint64_t u;
  std::memcpy(&u, &v, sizeof u);
  return u;
#endif
}
PFM_FX double fx_from_bits(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(static_cast<long long>(u));
#else
  double v;
  std::memcpy(&v, &u, sizeof v);
  return v;
#endif
}
PFM_FX int fx_clz(uint64_t a) {
#ifdef __CUDA_ARCH__
  return __clzll(static_cast<long long>(a));
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// high word of |v|: orders as |v| up to its low word; exponent e = top >> 20 with
// |v| < 2^(e - 1022) (e = 0: zero or below the normal numbers, read as zero)
PFM_FX unsigned fx_top(double v) { return unsigned(fx_bits(v) >> 32) & 0x7fffffffu; }

constexpr int FX_TERMS = 16;  // products per sum

// Scales of a point's Hessian, for a contraction that leaves the weak rows out of
// account (host test only, see above): a_F in the high and a_e in the low 16 bits, from
// the largest fx_top of its parts (F, F), (F, eta), (eta, eta); FX_NONE when an
// entry is not finite or a scale is outside +-FX_RANGE.
constexpr int FX_NONE = -2147483647 - 1;
constexpr int FX_RANGE = 400;
PFM_FX int fx_hess_scales(const unsigned top[3]) {
  const int e0 = int(top[0] >> 20), e1 = int(top[1] >> 20), e2 = int(top[2] >> 20);
  if (e0 == 0x7ff || e1 == 0x7ff || e2 == 0x7ff) return FX_NONE;
  if (e0 == 0 && e1 == 0 && e2 == 0) return 0;
  const int aF = e0 ? (e0 - 1021) >> 1 : -FX_RANGE;
  int ae = e2 ? (e2 - 1021) >> 1 : -FX_RANGE;
  if (e1 && e1 - 1022 - aF > ae) ae = e1 - 1022 - aF;
  if (aF < -FX_RANGE || aF > FX_RANGE || ae < -FX_RANGE || ae > FX_RANGE) return FX_NONE;
  return int((unsigned(aF) << 16) | (unsigned(ae) & 0xffffu));
}
PFM_FX int fx_scale_F(int hx) { return hx >> 16; }
PFM_FX int fx_scale_eta(int hx) { return int(int16_t(uint16_t(unsigned(hx) & 0xffffu))); }

// Z of its input from the largest fx_top of its two parts; false when the
// contraction does not take the point (then it goes through FP64).
PFM_FX bool fx_input_scale(int hx, unsigned topF, unsigned tope, int& Z) {
  const int eF = int(topF >> 20), ee = int(tope >> 20);
  const int zF = eF ? eF - 1022 + fx_scale_F(hx) : -3 * FX_RANGE;
  const int ze = ee ? ee - 1022 + fx_scale_eta(hx) : -3 * FX_RANGE;
  Z = eF == 0 && ee == 0 ? 0 : (zF > ze ? zF : ze);
  return hx != FX_NONE && eF != 0x7ff && ee != 0x7ff && Z >= -FX_RANGE && Z <= FX_RANGE;
}

// Limbs of v 2^-E as a 58-bit fraction, k = 1027 + E (truncated towards zero).
PFM_FX void fx_limbs(double v, int k, int& x1, int& x0) {
  const uint64_t u = fx_bits(v);
  const unsigned hi = unsigned(u >> 32), lo = unsigned(u);
  int r = k - int((hi >> 20) & 0x7ffu);  // >= 5: the mantissa's leading bit moves from bit 62 below bit 58
  r = r < 63 ? r : 63;
  const uint64_t w = ((uint64_t((hi & 0xfffffu) | 0x100000u) << 42) | (uint64_t(lo) << 10)) >> r;
  const int sg = (int(hi) >> 31) | 1;
  x1 = int(unsigned(w >> 29)) * sg;
  x0 = int(unsigned(w) & 0x1fffffffu) * sg;
}
// s1 + s0 2^-29 += h x, at most FX_TERMS times
PFM_FX void fx_mad(int64_t& s1, int64_t& s0, int h1, int h0, int x1, int x0) {
  s1 += int64_t(h1) * x1;
  s0 += int64_t(h1) * x0;
  s0 += int64_t(h0) * x1;
}
// (s1 + s0 2^-29) 2^-58 2^E rounded to nearest, k = 1027 + E
PFM_FX double fx_value(int64_t s1, int64_t s0, int k) {
  const int64_t t = 2 * s1 + (s0 >> 28);  // units of 2^-59
  const int64_t sg = t >> 63;
  const uint64_t a = uint64_t((t ^ sg) - sg);
  const int lz = fx_clz(a);
  const uint64_t q = (((a << (lz & 63)) >> 10) + 1) >> 1;  // 53 bits; the leading one counts in the exponent
  const uint64_t u = (uint64_t(unsigned(k - 1 - lz)) << 52) + q;
  return t == 0 ? 0.0 : fx_from_bits(u | (uint64_t(sg) << 63));
}

// Chains of such contractions: a block of numbers is kept as limbs x = h 2^29 + l
// with one power of two, x 2^(E - 58). After each contraction the sums are shifted
// to fill the 58 bits, so a stage loses about 2^-57 of its largest result.
struct Fx {
  int h, l;
};
// E with |v| < 2^E for the largest fx_top of a block (0: all zero); `ok` is cleared
// when a number is not finite or E is outside +-range
PFM_FX int fx_block_exponent(unsigned top, int range, bool& ok) {
  const int e = int(top >> 20);
  const int E = e ? e - 1022 : 0;
  ok = ok && e != 0x7ff && E >= -range && E <= range;
  return E;
}
PFM_FX Fx fx_of(double v, int E) {
  Fx x;
  fx_limbs(v, 1027 + E, x.h, x.l);
  return x;
}
PFM_FX void fx_mad(int64_t& s1, int64_t& s0, Fx a, Fx b) { fx_mad(s1, s0, a.h, a.l, b.h, b.l); }
PFM_FX int64_t fx_sum(int64_t s1, int64_t s0) { return 2 * s1 + (s0 >> 28); }  // units of 2^(E - 59)
// limbs of the block t (|t| < 2^62, units of 2^(E - 59)); returns the change of E
template <int N>
PFM_FX int fx_normalise(const int64_t (&t)[N], Fx (&x)[N]) {
  uint64_t m = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) m |= uint64_t(t[i] ^ (t[i] >> 63));
  const int lz = fx_clz(m);  // >= 2
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int64_t y = int64_t(uint64_t(t[i]) << ((lz - 2) & 63));  // below 2^62
    x[i].h = int(y >> 33);
    x[i].l = int(unsigned(y >> 4) & 0x1fffffffu);
  }
  return 5 - lz;
}

}  // namespace pfm
