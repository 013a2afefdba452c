// Block fixed-point arithmetic for the FP64 operators.
//
// GB300 issues two FP64 fused multiply-adds per clock and SM, and 61 integer multiply-adds of 32 x 32
// into 64 bits (both measured), so the products of the hopping term and the clover blocks are formed on
// integers.  A number is an integer v of at most 60 bits with a power-of-two unit shared by its group:
//   spinor site   12 reals of each chiral block, |x| < 2^e for all of them, x = v 2^(e-60); e is stored per
//                 (RHS, block, site): the site operators do not mix the blocks, and one may be much the smaller
//   link          near-unitary, entries of magnitude <= 1 + 1e-5, x = v 2^-58 (no exponent)
//   clover block  36 reals of one 6x6 block, |x| <= 2^e, x = v 2^(e-58); e per (block, site)
// For a product both factors are split as v = hi 2^31 + lo, and
//   a b = (ah bh) 2^62 + (ah bl + al bh) 2^31 + al bl:
// three multiply-adds into two 64-bit sums, the last term dropped.  The dropped terms are about 2^59 each
// whatever the factors, so both groups are brought to their full size before they meet; the products of
// a group's largest members (2^116 and more) are then right to 2^-56 or better, where FP64 rounds each of
// them to 2^-53 (qcd_selftest_fixed measures both against extended precision).  Products of smaller members have
// that same absolute error, where FP64's shrinks with them: a result is as good as FP64's by its group's size
// (norms over a chiral block, a matrix), not component by component.
//
// Bounds (the sums are exact integers, so only their final values have to fit):
//   half spinor h = s +- s', |h| < 2^61: hi < 2^30, 0 <= lo < 2^31
//   link: |hi| <= 2^27 + 1, |lo| <= 2^30; three complex products, six real ones:
//     |sum ah bh| < 2^59.7, |sum ah bl + al bh| <= 6 (2^58 + 2^60) < 2^62.9
//   w = (sum ah bh) + (sum ah bl + al bh >> 31), in units of 2^(e-56): |w| <= |row| |h| <= 2^2.3 2^56, so
//   eight hops stay below 2^61.4
//   clover: |hi| <= 2^27, |lo| <= 2^30 against |x| < 2^60 with hi <= 2^29, |lo| <= 2^30; eleven products:
//     |sum ah bl + al bh| <= 11 (2^57 + 2^59) < 2^62.8, and their value in units of 2^60 is below 2^61.5
//
// A block whose reals are not all finite carries the exponent FX_NAN: the largest exponent of its
// neighbours is what a result takes its unit from, so the mark spreads as a NaN does, and the
// conversion to double gives NaN.
#pragma once

#include "qcd_internal.cuh"

namespace qcd {

typedef long long i64;
typedef unsigned long long u64;

constexpr int FX_NAN = 1 << 24;      // exponent of a group with a non-finite member (and anything above FX_BIG)
constexpr int FX_BIG = 1 << 23;
constexpr int FX_ZERO = -(1 << 24);  // exponent of a group of zeros
constexpr int FX_SPINOR = 60, FX_LINK = 58, FX_CLOVER = 58, FX_SCALAR = 59;  // v = x 2^(this - e)

#define QCD_HD __host__ __device__ __forceinline__

// ------------------------------------------------------------------ limbs ----
struct FxLimb {
  int hi, lo;  // hi 2^31 + lo
};

// the limbs as 32-bit registers whose origin the compiler does not see: where it does, it takes their
// products as 64-bit ones of the masked sums, three multiply-adds each
QCD_HD FxLimb fx_limb(int hi, int lo) {
#ifdef __CUDA_ARCH__
  asm("" : "+r"(hi), "+r"(lo));
#endif
  return FxLimb{hi, lo};
}
// of a sum's value: 0 <= lo < 2^31
QCD_HD FxLimb fx_split(i64 v) { return fx_limb((int)(v >> 31), (int)v & 0x7fffffff); }
// -2^30 <= lo < 2^30, so that the dropped products of the low limbs have no bias: for the constant factor
// (link, clover entry, coefficient) and where the sums need the smaller range
QCD_HD FxLimb fx_split_balanced(i64 v) {
  const FxLimb a = fx_split(v + (1LL << 30));
  return fx_limb(a.hi, a.lo - (1 << 30));
}
QCD_HD FxLimb fx_neg(FxLimb a) { return FxLimb{-a.hi, -a.lo}; }
// -a where f = -1, a where f = 0
QCD_HD FxLimb fx_sign(FxLimb a, int f) { return FxLimb{(a.hi ^ f) - f, (a.lo ^ f) - f}; }
QCD_HD i64 fx_sign(i64 v, int f) { return (v ^ (i64)f) - (i64)f; }

// sum of products: h 2^62 + m 2^31
struct FxSum {
  i64 h, m;
};
// an empty sum whose fx_value<K> is rounded to nearest: cut off, values are low by half a unit in the mean
template <int K>
QCD_HD FxSum fx_sum() { return FxSum{0, 1LL << (30 - K)}; }
QCD_HD i64 fx_mad(int a, int b, i64 c) { return c + (i64)a * b; }
QCD_HD void fx_mac(FxSum& s, FxLimb a, FxLimb b) {
  s.h = fx_mad(a.hi, b.hi, s.h);
  s.m = fx_mad(a.hi, b.lo, s.m);
  s.m = fx_mad(a.lo, b.hi, s.m);
}
// the sum in units of 2^(62 - K), rounded if it began as fx_sum<K>
template <int K>
QCD_HD i64 fx_value(const FxSum& s) {
  return (i64)((u64)s.h << K) + (s.m >> (31 - K));
}

// v 2^-d rounded to nearest, d >= 0
QCD_HD i64 fx_down_rn(i64 v, int d) {
  if (d <= 0) return v;
  if (d > 62) return 0;
  return (v + (1LL << (d - 1))) >> d;
}

// ------------------------------------------------------- double <-> fixed ----
QCD_HD u64 fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(x);
#else
  u64 b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
QCD_HD double fx_from_bits(u64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((i64)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
QCD_HD int fx_clz(u64 m) {
#ifdef __CUDA_ARCH__
  return __clzll((i64)m);
#else
  return m ? __builtin_clzll(m) : 64;
#endif
}

// the exponent e of a group, |x| < 2^e for each member, from the largest bit pattern of their magnitudes
QCD_HD int fx_exponent(u64 max_bits) {
  const int E = (int)(max_bits >> 52);
  if (E == 0x7ff) return FX_NAN;
  if (max_bits == 0) return FX_ZERO;
  return (E > 1 ? E : 1) - 1022;
}

// x 2^(B - e) rounded to nearest, |x| < 2^e, B >= 53 (e from fx_exponent of the group)
template <int B>
QCD_HD i64 fx_of_double(double x, int e) {
  if (e <= FX_ZERO || e > FX_BIG) return 0;
  const u64 b = fx_bits(x);
  int E = (int)(b >> 52) & 0x7ff;
  i64 m = (i64)(b & ((1ULL << 52) - 1));
  if (E) m |= 1LL << 52;
  else E = 1;
  // x = m 2^(E - 1075), m < 2^53; at E - 1022 = e it becomes m 2^(B - 53)
  m = fx_down_rn(m << (B - 53), e + 1022 - E);
  return (b >> 63) ? -m : m;
}

// v 2^(e - B) as a double, rounded to nearest even
QCD_HD double fx_to_double(i64 v, int e, int B) {
  if (e > FX_BIG) return fx_from_bits(0x7ff8000000000000ULL);
  const u64 s = v < 0 ? 1ULL << 63 : 0ULL;
  u64 m = v < 0 ? 0ULL - (u64)v : (u64)v;
  if (m == 0) return 0.0;
  const int n = fx_clz(m);
  m <<= n;
  const int E = e - B + 63 - n + 1023;  // biased exponent of m's top bit
  if (E >= 1 && E < 2046) {
    u64 r = m >> 11;
    const u64 rest = m & 0x7ff;
    r += (rest > 0x400 || (rest == 0x400 && (r & 1))) ? 1 : 0;  // r <= 2^53: a carry raises the exponent
    return fx_from_bits(s | (((u64)(E - 1) << 52) + r));
  }
  // results at the ends of the double range: powers of two applied in two steps of at most 2^+-1000
  const int p = E - 1023 - 63;  // m 2^p
  const double x = (double)m;
  const int p1 = p < -1000 ? -1000 : (p > 900 ? 900 : p);
  int p2 = p - p1;
  p2 = p2 < -1000 ? -1000 : (p2 > 1000 ? 1000 : p2);
  const double y = x * fx_from_bits((u64)(p1 + 1023) << 52) * fx_from_bits((u64)(p2 + 1023) << 52);
  return s ? -y : y;
}

// a coefficient: v 2^(e - 59), limbs balanced
struct FxScalar {
  FxLimb v;
  int e;
};
inline FxScalar fx_scalar(double a) {
  u64 b = fx_bits(a) & ~(1ULL << 63);
  const int e = fx_exponent(b);
  return FxScalar{fx_split_balanced(fx_of_double<FX_SCALAR>(a, e)), e};
}

QCD_HD u64 fx_mag(double x) { return fx_bits(x) & ~(1ULL << 63); }

// ------------------------------------------------------------- field access ----
// Spinor sites in block fixed point ([rhs][12][Vh] pairs of 64-bit integers, exponents [rhs][2][Vh] in
// place of the FP16 norms), seen as doubles: for the kernels that convert fields or update vectors.
QCD_HD size_t eidx(int b, int Vh, int r, int h) { return ((size_t)2 * r + b) * Vh + h; }

template <>
struct SpinorIO<60> {
  static constexpr int NVEC = 12;
  template <int LD = LD_NC>
  __device__ static void load_block(const void* base, const float* ex, int Vh, int r, int h, int b,
                                    cx<double> s[6]) {
    if (!dbg_spinor(Vh, r, h)) {
      for (int c = 0; c < 6; c++) s[c] = {};
      return;
    }
    const longlong2* p = static_cast<const longlong2*>(base);
    const int e = ldv<LD>(reinterpret_cast<const int*>(ex) + eidx(b, Vh, r, h));
#pragma unroll
    for (int c = 0; c < 6; c++) {
      const longlong2 v = ldv<LD>(p + sidx<NVEC>(6 * b + c, Vh, r, h));
      s[c] = cmk(fx_to_double(v.x, e, FX_SPINOR), fx_to_double(v.y, e, FX_SPINOR));
    }
  }
};

// a link entry or a clover entry pair as stored: the limbs of two numbers
QCD_HD int4 fx_pack2(FxLimb a, FxLimb b) { return int4{a.hi, a.lo, b.hi, b.lo}; }

// one link (near-unitary) into [9][Vh] int4 at q
__device__ __forceinline__ void fx_store_link(int4* q, int Vh, const double2 u[9]) {
#pragma unroll
  for (int k = 0; k < 9; k++) {
    // |x| <= 1 + 1e-5 < 2: in units of 2^-58 (B = 59 for the bound 2^1)
    q[(size_t)k * Vh] = fx_pack2(fx_split_balanced(fx_of_double<FX_LINK + 1>(u[k].x, 1)),
                                 fx_split_balanced(fx_of_double<FX_LINK + 1>(u[k].y, 1)));
  }
}

// one chiral block (6 diagonal reals, 15 strictly-lower entries) into [18][Vh] int4 at q; its exponent
// is returned
__device__ __forceinline__ int fx_store_clover(int4* q, int Vh, const double d[6], const cx<double> L[15]) {
  u64 mx = 0;
#pragma unroll
  for (int k = 0; k < 6; k++) mx = fx_mag(d[k]) > mx ? fx_mag(d[k]) : mx;
#pragma unroll
  for (int k = 0; k < 15; k++) {
    mx = fx_mag(L[k].re) > mx ? fx_mag(L[k].re) : mx;
    mx = fx_mag(L[k].im) > mx ? fx_mag(L[k].im) : mx;
  }
  const int e = fx_exponent(mx);
  auto lim = [&](double x) { return fx_split_balanced(fx_of_double<FX_CLOVER>(x, e)); };
#pragma unroll
  for (int k = 0; k < 3; k++) q[(size_t)k * Vh] = fx_pack2(lim(d[2 * k]), lim(d[2 * k + 1]));
#pragma unroll
  for (int k = 0; k < 15; k++) q[(size_t)(3 + k) * Vh] = fx_pack2(lim(L[k].re), lim(L[k].im));
  return e;
}

}  // namespace qcd
