// Products of 3x3 complex matrices in block fixed point (qcd_fixed.cuh), a row at a time: a thread carries
// one row of a product of links from left to right, so that it holds three complex numbers and the
// matrices are read from memory where they are multiplied (three warps of a block take the three rows of
// the same sites).
//
// A matrix is in units of 2^-58 times its group's power of two, a row in the same or finer ones (up to 2^61 units
// for its largest entry), balanced limbs.  A product's sum of six real products of entries below 2^58 and 2^61
// stays exact: |sum ah bl + al bh| <= 6 (2^27 2^30 + 2^30 2^30) < 2^62.8.
//
// Field strength and gauge force depend on the links' differences from one alone.  FP64 products carry these
// to 2^-53 of themselves, products in fixed units to an absolute size; rows in units of 2^-61 make that 2^-59 a
// product.  Error of the gauge force on links exp(i eps H), relative to the force, at eps 0.2, 0.1, 0.05: 0.92, 0.95,
// 1.05e-16 (rows in units of 2^-58: 1.6, 2.5, 4.7e-16; FP64 kernel: 1.3e-16 at every eps).  Where all links of a
// result are within 2^-4 of one in each entry (below eps 0.05) the FP64 kernels form it.
#pragma once

#include "qcd_fixed.cuh"

namespace qcd {

struct FxRow {
  FxLimb re[3], im[3];
};

__device__ __forceinline__ FxRow fx_row(const cx<i64> v[3]) {
  FxRow r;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    r.re[k] = fx_split_balanced(v[k].re);
    r.im[k] = fx_split_balanced(v[k].im);
  }
  return r;
}

// row i of a stored link (DAG: of its adjoint) in units of 2^-61
template <bool DAG>
__device__ __forceinline__ FxRow fx_load_row_fine(const int4* __restrict__ q, size_t stride, int i) {
  // 8 (hi 2^31 + lo) with limbs of the same range
  auto times8 = [](int hi, int lo) {
    const int t = lo + (1 << 27);
    return fx_limb(8 * hi + (t >> 28), (int)((unsigned)t << 3 & 0x7fffffffu) - (1 << 30));
  };
  FxRow r;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int4 e = __ldg(q + (size_t)(DAG ? 3 * k + i : 3 * i + k) * stride);
    r.re[k] = times8(e.x, e.y);
    r.im[k] = DAG ? times8(-e.z, -e.w) : times8(e.z, e.w);
  }
  return r;
}

// row i of a stored matrix M (DAG: of M^dag, conj of column i); q: its first element, rows of stride
template <bool DAG>
__device__ __forceinline__ FxRow fx_load_row(const int4* __restrict__ q, size_t stride, int i) {
  FxRow r;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int4 e = __ldg(q + (size_t)(DAG ? 3 * k + i : 3 * i + k) * stride);
    r.re[k] = FxLimb{e.x, e.y};
    r.im[k] = DAG ? fx_neg(FxLimb{e.z, e.w}) : FxLimb{e.z, e.w};
  }
  return r;
}

// v M (DAG: v M^dag) in units of 2^(62 - K) of the products (K = 4: those of v), cut off, or ROUNDed
// where the results are added up with one sign
template <bool DAG, int K = 4, bool ROUND = false>
__device__ __forceinline__ void fx_row_mul(const FxRow& v, const int4* __restrict__ q, size_t stride, cx<i64> o[3]) {
  FxLimb n[3];  // -Im v for M, -Re v for M^dag
#pragma unroll
  for (int k = 0; k < 3; k++) n[k] = fx_neg(DAG ? v.re[k] : v.im[k]);
#pragma unroll
  for (int j = 0; j < 3; j++) {
    FxSum re = ROUND ? fx_sum<K>() : FxSum{}, im = ROUND ? fx_sum<K>() : FxSum{};
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const int4 e = __ldg(q + (size_t)(DAG ? 3 * j + k : 3 * k + j) * stride);
      const FxLimb a = {e.x, e.y}, b = {e.z, e.w};
      fx_mac(re, a, v.re[k]);
      fx_mac(re, b, DAG ? v.im[k] : n[k]);
      fx_mac(im, a, v.im[k]);
      fx_mac(im, b, DAG ? n[k] : v.re[k]);
    }
    o[j] = cmk(fx_value<K>(re), fx_value<K>(im));
  }
}
template <bool DAG>
__device__ __forceinline__ FxRow fx_row_times(const FxRow& v, const int4* __restrict__ q, size_t stride) {
  cx<i64> o[3];
  fx_row_mul<DAG>(v, q, stride, o);
  return fx_row(o);
}

// v 2^p as a double, rounded to nearest, for results well inside the double range (no subnormals, no
// overflow: -900 < p < 900)
__device__ __forceinline__ double fx_to_double_in_range(i64 v, int p) {
  const u64 m = (u64)(v < 0 ? -v : v);
  const int n = __clzll((i64)m);  // 64 for zero
  const u64 t = m << (n & 63);
  const u64 r = (t >> 11) + ((t >> 10) & 1);
  const u64 b = ((u64)(p + 63 - n + 1022) << 52) + r;
  return __longlong_as_double((i64)(m ? (b | ((u64)v & (1ULL << 63))) : 0));
}

// the stored link U_mu at displacement (s1 d1 + s2 d2) from the site of lexicographic coordinates c and
// parity p; d1 != d2, steps -1, 0, 1
struct FxSites {
  const int4* g;
  int Vh, X, Y, Z, T, c[4], p;
};
__device__ __forceinline__ int fx_half_at(const FxSites& f, int d1, int s1, int d2, int s2) {
  int q[4];
  const int L[4] = {f.X, f.Y, f.Z, f.T};
#pragma unroll
  for (int k = 0; k < 4; k++) {
    int v = f.c[k] + (k == d1 ? s1 : 0) + (k == d2 ? s2 : 0);
    q[k] = v < 0 ? v + L[k] : (v >= L[k] ? v - L[k] : v);
  }
  return (q[0] + f.X * (q[1] + f.Y * (q[2] + f.Z * q[3]))) >> 1;
}
__device__ __forceinline__ const int4* fx_link_at(const FxSites& f, int d1, int s1, int d2, int s2, int mu) {
  const int p = (f.p + s1 + s2) & 1;
  return f.g + (size_t)(p * 4 + mu) * 9 * f.Vh + fx_half_at(f, d1, s1, d2, s2);
}

}  // namespace qcd
