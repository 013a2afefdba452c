// Fermion force and Wilson gauge force from block fixed-point links and fields (qcd_fixed.cuh,
// qcd_fxmat.cuh): the sums of qcd_force.cu and qcd_md.cu for near-unitary links.
//
// Three warps of a block take the three rows of the result of 32 sites of one parity (or of their links in
// one direction, blockIdx.y); rows meet in shared memory where a dagger or a whole matrix is needed.  A
// stored matrix field is [field][9][V] int4 (limbs in units of 2^-58 of the matrix's power of two) with
// exponents [field][V], the site of parity p and half index h at p Vh + h.
//
// Against the FP64 kernels, which ran at 82 to 95% of the FP64 pipe (16^4, one pseudofermion): coefficients
// 172 -> 56 us, insertions 328 -> 119 us (with the coefficients' conversion), links 1526 -> 429 us, gauge force
// 741 -> 201 us, plaquette 206 -> 63 us.  Bound by instruction issue and the latency of the matrices' loads:
// the link kernel runs 4 blocks of 168 registers per SM (3 of 178 without the bound: 668 us; 5 of 128, which
// spill: 437 us here, but 2469 against 2449 us at 24^4 with two), the gauge force and insertions 7 of 96
// (6 of 108: 980 against 863 us and 628 against 575 us at 24^4).
#include <type_traits>

#include "qcd_dslash.cuh"
#include "qcd_force.h"
#include "qcd_fxmat.cuh"
#include "qcd_kernels.h"

namespace qcd {

QCD_DEBUG_TAKE(debug_take_force_fx)

namespace {

// common bound 2^bits of n numbers (0 for zeros)
template <int N>
__device__ __forceinline__ int fx_bits_n(const cx<i64> (&t)[N]) {
  u64 o = 0;
#pragma unroll
  for (int k = 0; k < N; k++) o |= (u64)(t[k].re ^ (t[k].re >> 63)) | (u64)(t[k].im ^ (t[k].im >> 63));
  return 64 - fx_clz(o);
}

// Before another term is added to a sum over right-hand sides: a sum that has grown to 2^most units is halved,
// and *down, the powers of two by which its unit is above the terms', goes up.  (The unit follows the sum's
// size: one chosen beforehand for n terms of the largest size costs log2(n) bits that sums of random signs do
// not use, 64 right-hand sides 1.6e-15 of the force against the FP64 kernels' 3.8e-16.)
template <int N>
__device__ __forceinline__ void fx_make_room(cx<i64> (&t)[N], int most, int* down) {
  if (fx_bits_n(t) <= most) return;
#pragma unroll
  for (int k = 0; k < N; k++) t[k] = cmk((t[k].re + 1) >> 1, (t[k].im + 1) >> 1);
  *down += 1;
}

// t 2^sh, rounded to nearest where sh < 0
__device__ __forceinline__ i64 fx_scaled(i64 t, int sh) {
  return sh >= 0 ? (i64)((u64)t << (sh < 63 ? sh : 63)) : fx_down_rn(t, -sh);
}

// exponent of a product of members of two groups (marked if either is, whatever the other)
__device__ __forceinline__ int fx_exp_sum(int a, int b) { return max(a, b) > FX_BIG ? FX_NAN : a + b; }

// t 2^-d, 0 <= d <= 62, rounded to nearest: many such terms are added, and cut off they would add up to a bias
__device__ __forceinline__ i64 fx_round_down(i64 t, int d) { return (t + ((1LL << d) >> 1)) >> d; }

// exponent of a matrix whose entries are below 2^bits units of 2^unit
__device__ __forceinline__ int fx_group_exp(int unit, int bits, bool bad) {
  return bad ? FX_NAN : (bits ? unit + bits : FX_ZERO);
}
__device__ __forceinline__ int fx_max3(const int (*e)[32], int lane) { return max(e[0][lane], max(e[1][lane], e[2][lane])); }

// the site of this thread: parity, half index, row
struct Where {
  int p, h, lane, row;
  bool valid;
};
__device__ __forceinline__ Where where(const Geom& g) {
  Where w;
  w.lane = threadIdx.x & 31;
  w.row = threadIdx.x >> 5;
  const int nb = (g.Vh + 31) / 32;
  w.p = (int)blockIdx.x / nb;
  w.h = ((int)blockIdx.x - w.p * nb) * 32 + w.lane;
  w.valid = w.h < g.Vh && dbg_link(g.Vh, w.p, 0, w.h);
  return w;
}

// colour a of the four spins of a spinor site, brought to 58 bits
__device__ __forceinline__ void load_colour(const longlong2* f, int Vh, int r, int h, int a, cx<i64> s[4]) {
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const longlong2 v = __ldg(f + sidx<12>(3 * k + a, Vh, r, h));
    s[k] = cmk((i64)v.x, (i64)v.y);
  }
}
__device__ __forceinline__ FxLimb limb58(i64 v, int down) { return fx_split_balanced((v + (1LL << (down - 1))) >> down); }

// ---- clover coefficients C_{mu nu}(x) = -i (kappa c_sw / 4) (S + S^dag), S the traceless part of
// sum_s [sigma_{mu nu} X]_s W_s^dag over the right-hand sides, W = Y (even sites), kappa^2 Y (odd).  sigma is
// block diagonal in chirality: with T_st = X_s W_t^dag inside block b (spins 0, 1 of it),
// D_b = T_00 - T_11, P_b = T_10 + T_01, Q_b = i (T_01 - T_10),
//   xy = D_0 + D_1, xz = Q_0 + Q_1, xt = P_1 - P_0, yz = P_0 + P_1, yt = Q_0 - Q_1, zt = D_1 - D_0,
// 18 complex products a row and right-hand side instead of 72.
struct FieldPair {  // a field on even and odd sites in block fixed point, exponents [rhs][2][Vh]
  const longlong2* v[2];
  const int* e[2];
};

__global__ void __launch_bounds__(96, 4) clover_coeff_fixed_kernel(Geom g, double f_even, double f_odd, int nrhs,
                                                                FieldPair X, FieldPair Y, double2* Cbuf) {
  __shared__ i64 sm[3][36][32];
  __shared__ int sd[3][32];
  const Where w = where(g);
  const int Vh = g.Vh;
  const size_t V = 2 * (size_t)Vh;
  cx<i64> S[18] = {};  // [plane][colour]
  int ex = FX_ZERO, down = 0;
  if (w.valid) {
    const int *eX = X.e[w.p] + w.h, *eY = Y.e[w.p] + w.h;
    for (int k = 0; k < 2 * nrhs; k++)  // (right-hand side, chiral block)
      ex = max(ex, fx_exp_sum(__ldg(eX + (size_t)k * Vh), __ldg(eY + (size_t)k * Vh)));
#pragma unroll 1
    for (int r = 0; r < nrhs; r++) {
      // units of 2^(eX + eY - 56) of a block, brought to the largest's and the sum's; a term is below 2^59 units of
      // the former, so the sum stays below 2^60
      if (r > 0) fx_make_room(S, 59, &down);
      int d[2];
#pragma unroll
      for (int b = 0; b < 2; b++) {
        const size_t o = eidx(b, Vh, r, 0);
        d[b] = min(ex - fx_exp_sum(__ldg(eX + o), __ldg(eY + o)) + down, 62);
      }
      cx<i64> xs[4];
      load_colour(X.v[w.p], Vh, r, w.h, w.row, xs);
      FxLimb xr[4], xi[4], nxr[4];
#pragma unroll
      for (int s = 0; s < 4; s++) {
        xr[s] = limb58(xs[s].re, 2);
        xi[s] = limb58(xs[s].im, 2);
        nxr[s] = fx_neg(xr[s]);
      }
#pragma unroll
      for (int c = 0; c < 3; c++) {
        cx<i64> ws[4];
        load_colour(Y.v[w.p], Vh, r, w.h, c, ws);
        FxLimb wr[4], wi[4];
#pragma unroll
        for (int s = 0; s < 4; s++) {
          wr[s] = limb58(ws[s].re, 2);
          wi[s] = limb58(ws[s].im, 2);
        }
        auto outer = [&](int s, int t) {  // X_s conj(W_t), s and t of one block
          FxSum re = fx_sum<2>(), im = fx_sum<2>();
          fx_mac(re, xr[s], wr[t]);
          fx_mac(re, xi[s], wi[t]);
          fx_mac(im, xi[s], wr[t]);
          fx_mac(im, nxr[s], wi[t]);
          return cmk(fx_round_down(fx_value<2>(re), d[s >> 1]), fx_round_down(fx_value<2>(im), d[s >> 1]));
        };
        cx<i64> D[2], P[2], Q[2];
#pragma unroll
        for (int b = 0; b < 2; b++) {
          const cx<i64> t01 = outer(2 * b, 2 * b + 1), t10 = outer(2 * b + 1, 2 * b);
          D[b] = outer(2 * b, 2 * b) - outer(2 * b + 1, 2 * b + 1);
          P[b] = t10 + t01;
          Q[b] = times_i(t01 - t10);
        }
        S[c] = S[c] + D[0] + D[1];
        S[3 + c] = S[3 + c] + Q[0] + Q[1];
        S[6 + c] = S[6 + c] + P[1] - P[0];
        S[9 + c] = S[9 + c] + P[0] + P[1];
        S[12 + c] = S[12 + c] + Q[0] - Q[1];
        S[15 + c] = S[15 + c] + D[1] - D[0];
      }
    }
  }
  sd[w.row][w.lane] = down;
  __syncthreads();
  const int most = max(sd[0][w.lane], max(sd[1][w.lane], sd[2][w.lane]));
#pragma unroll
  for (int k = 0; k < 18; k++) {
    S[k] = cmk(fx_round_down(S[k].re, min(most - down, 62)), fx_round_down(S[k].im, min(most - down, 62)));
    sm[w.row][2 * k][w.lane] = S[k].re;
    sm[w.row][2 * k + 1][w.lane] = S[k].im;
  }
  __syncthreads();
  if (!w.valid) return;
  const double f = w.p ? f_odd : f_even;
  // |X W| < 2^(eX + eY): a product in units of 2^(-58 - 58 + 60)
  const int e = ex > FX_BIG ? FX_NAN : ex + most - 56;
#pragma unroll
  for (int pl = 0; pl < 6; pl++) {
    const i64 tr = sm[0][6 * pl][w.lane] + sm[1][6 * pl + 2][w.lane] + sm[2][6 * pl + 4][w.lane];
    double2* q = Cbuf + ((size_t)pl * 9 + 3 * w.row) * V + (size_t)w.p * Vh + w.h;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      double2 o;
      if (c == w.row) {  // -i f (2 Re S_aa - 2/3 tr)
        o = make_double2(0.0, -f * (2.0 / 3.0) * fx_to_double(3 * S[3 * pl + c].re - tr, e, 0));
      } else {  // H = S_ac + conj(S_ca), -i f H
        const double hr = fx_to_double(S[3 * pl + c].re + sm[c][6 * pl + 2 * w.row][w.lane], e, 0);
        const double hi = fx_to_double(S[3 * pl + c].im - sm[c][6 * pl + 2 * w.row + 1][w.lane], e, 0);
        o = make_double2(f * hi, -f * hr);
      }
      q[(size_t)c * V] = o;
    }
  }
}

// ---- C from FP64 to block fixed point, one (site, plane) per thread
__global__ void __launch_bounds__(128) coeff_to_fixed_kernel(size_t V, const double2* Cbuf, int4* Cfx, int* eC) {
  const size_t j = (size_t)blockIdx.x * 128 + threadIdx.x;
  if (j >= 6 * V) return;
  const size_t pl = j / V, i = j - pl * V;
  const double2* q = Cbuf + pl * 9 * V + i;
  double2 v[9];
  u64 mx = 0;
#pragma unroll
  for (int k = 0; k < 9; k++) {
    v[k] = __ldg(q + (size_t)k * V);
    const u64 a = fx_mag(v[k].x), b = fx_mag(v[k].y);
    mx = max(mx, max(a, b));
  }
  const int e = fx_exponent(mx);
  int4* o = Cfx + pl * 9 * V + i;
#pragma unroll
  for (int k = 0; k < 9; k++)
    o[(size_t)k * V] = fx_pack2(fx_split_balanced(fx_of_double<58>(v[k].x, e)), fx_split_balanced(fx_of_double<58>(v[k].y, e)));
  eC[pl * V + i] = e;
}

__device__ __forceinline__ void plane_of(int pl, int& mu, int& nu) {
  mu = pl < 3 ? 0 : (pl < 5 ? 1 : 2);
  nu = pl < 3 ? pl + 1 : (pl < 5 ? pl - 1 : 3);
}

// ---- corner insertions E = C(x) U(x) + U(x) C(x + dir) of the two links of a plane at x: field
// blockIdx.y = 2 plane + (0: U_mu, 1: U_nu)
__global__ void __launch_bounds__(96, 7) edge_fixed_kernel(Geom g, const int4* __restrict__ gfx, const int4* __restrict__ Cfx,
                                                        const int* __restrict__ eC, int4* Efx, int* eE) {
  __shared__ int se[3][32];
  const Where w = where(g);
  const int Vh = g.Vh;
  const size_t V = 2 * (size_t)Vh;
  const int field = blockIdx.y, pl = field >> 1;
  int mu, nu;
  plane_of(pl, mu, nu);
  const int dir = field & 1 ? nu : mu;
  cx<i64> t[3] = {};
  int unit = 0, e = FX_ZERO;
  const size_t at = (size_t)w.p * Vh + w.h;
  if (w.valid) {
    const Site s = site_of(g, w.p, w.h);
    const size_t next = (size_t)(1 - w.p) * Vh + (neighbor_fwd(g, s, dir) >> 1);
    const int4* u = gfx + (size_t)(w.p * 4 + dir) * 9 * Vh + w.h;
    const int4* c = Cfx + (size_t)pl * 9 * V;
    const int e0 = __ldg(eC + pl * V + at), e1 = __ldg(eC + pl * V + next), em = max(e0, e1);
    cx<i64> o[3];
    fx_row_mul<false, 2, true>(fx_load_row<false>(c + at, V, w.row), u, Vh, t);
    fx_row_mul<false, 2, true>(fx_load_row<false>(u, Vh, w.row), c + next, V, o);
    const int d0 = min(em - e0, 62), d1 = min(em - e1, 62);
#pragma unroll
    for (int j = 0; j < 3; j++)
      t[j] = cmk(fx_round_down(t[j].re, d0) + fx_round_down(o[j].re, d1),
                 fx_round_down(t[j].im, d0) + fx_round_down(o[j].im, d1));
    unit = em - 56;
    e = fx_group_exp(unit, fx_bits_n(t), em > FX_BIG);
  }
  se[w.row][w.lane] = e;
  __syncthreads();
  if (!w.valid) return;
  e = fx_max3(se, w.lane);
  const int sh = e > FX_BIG ? -63 : unit - e + 58;
  int4* q = Efx + ((size_t)field * 9 + 3 * w.row) * V + at;
#pragma unroll
  for (int j = 0; j < 3; j++)
    q[(size_t)j * V] = fx_pack2(fx_split_balanced(fx_scaled(t[j].re, sh)), fx_split_balanced(fx_scaled(t[j].im, sh)));
  if (w.row == 0) eE[(size_t)field * V + at] = e;
}

// shared area of a block that needs its rows' matrices whole
struct RowsXch {
  int4 m[9][32];   // limbs of a matrix
  i64 v[3][6][32];  // rows of a result
  int e[3][32];
};

// v M (DAG: v M^dag) with M in shared memory, units of 2^(62 - K) of the products
template <bool DAG, int K>
__device__ __forceinline__ void row_mul_shared(const FxRow& v, const int4 (*m)[32], int lane, cx<i64> o[3]) {
#pragma unroll
  for (int j = 0; j < 3; j++) {
    FxSum re = fx_sum<K>(), im = fx_sum<K>();
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const int4 x = m[DAG ? 3 * j + k : 3 * k + j][lane];
      const FxLimb a = {x.x, x.y}, b = {x.z, x.w};
      fx_mac(re, a, v.re[k]);
      fx_mac(re, b, DAG ? v.im[k] : fx_neg(v.im[k]));
      fx_mac(im, a, v.im[k]);
      fx_mac(im, b, DAG ? fx_neg(v.re[k]) : v.re[k]);
    }
    o[j] = cmk(fx_value<K>(re), fx_value<K>(im));
  }
}

// out (canonical) = or += f P_TA(U M^dag) (DAG) or f P_TA(U M) for the matrix whose row w.row this thread
// holds as t in units of 2^unit; all threads of the block call it
template <bool DAG>
__device__ __forceinline__ void store_ta(const Geom& g, const Where& w, const int4* u, cx<i64> t[3], int unit, bool bad,
                                         double f, RowsXch& x, double2* q, bool accumulate) {
  int e = w.valid ? fx_group_exp(unit, fx_bits_n(*reinterpret_cast<cx<i64>(*)[3]>(t)), bad) : FX_ZERO;
  x.e[w.row][w.lane] = e;
  __syncthreads();
  e = fx_max3(x.e, w.lane);
  const int sh = e > FX_BIG || e <= FX_ZERO ? -63 : unit - e + 61;
#pragma unroll
  for (int j = 0; j < 3; j++)
    x.m[3 * w.row + j][w.lane] = fx_pack2(fx_split_balanced(fx_scaled(t[j].re, sh)), fx_split_balanced(fx_scaled(t[j].im, sh)));
  __syncthreads();
  cx<i64> M[3] = {};
  // units of 2^(e - 61 - 58 + 60), |M| < 2^60.4
  if (w.valid) row_mul_shared<DAG, 2>(fx_load_row<false>(u, g.Vh, w.row), x.m, w.lane, M);
#pragma unroll
  for (int j = 0; j < 3; j++) {
    x.v[w.row][2 * j][w.lane] = M[j].re;
    x.v[w.row][2 * j + 1][w.lane] = M[j].im;
  }
  __syncthreads();
  if (!w.valid) return;
  const int em = e > FX_BIG ? FX_NAN : (e <= FX_ZERO ? 0 : e - 59);
  const i64 tr = x.v[0][1][w.lane] + x.v[1][3][w.lane] + x.v[2][5][w.lane];
  // (M - M^dag) / 2 less its trace / 3
#pragma unroll
  for (int j = 0; j < 3; j++) {
    double2 o;
    if (j == w.row) {
      o = make_double2(0.0, f * (1.0 / 3.0) * fx_to_double(2 * M[j].im - (tr - M[j].im), em, 0));
    } else {
      o.x = 0.5 * f * fx_to_double(M[j].re - x.v[j][2 * w.row][w.lane], em, 0);
      o.y = 0.5 * f * fx_to_double(M[j].im + x.v[j][2 * w.row + 1][w.lane], em, 0);
    }
    if (accumulate) {
      const double2 was = q[j];
      o = make_double2(was.x + o.x, was.y + o.y);
    }
    q[j] = o;
  }
}

// ---- hopping part of a link's G, row `row`: the sum over the right-hand sides of A^dag + B with
//   A = (1 - g) X(y + l) Y(y)^dag,  B = (1 + g) X(y) Y(y + l)^dag.
// (1 -+ g) is twice a projector, so A = sum_k h_k hw_k^dag over its two rows k with h, hw the projected half
// spinors of X(y + l) and of Y(y), and likewise B: two outer products each instead of four.
template <int MU>
__device__ __forceinline__ void hop_force_fx(const Geom& g, const Where& w, int j, int nrhs, const FieldPair& X,
                                             const FieldPair& Y, cx<i64> t[3], int& unit, bool& bad) {
  const int Vh = g.Vh, p = w.p, n = 1 - w.p;
  // a site's exponent, the larger of its blocks' (the projections add one to the other)
  auto site_exp = [&](const int* e, int r, int h) { return max(__ldg(e + eidx(0, Vh, r, h)), __ldg(e + eidx(1, Vh, r, h))); };
  int em = FX_ZERO;
  for (int r = 0; r < nrhs; r++)
    em = max(em, max(fx_exp_sum(site_exp(X.e[n], r, j), site_exp(Y.e[p], r, w.h)),
                     fx_exp_sum(site_exp(X.e[p], r, w.h), site_exp(Y.e[n], r, j))));
#pragma unroll
  for (int b = 0; b < 3; b++) t[b] = {};
  int down = 0;
#pragma unroll 1
  for (int r = 0; r < nrhs; r++) {
    if (r > 0) fx_make_room(*reinterpret_cast<cx<i64>(*)[3]>(t), 60, &down);  // a right-hand side's A^dag + B: below 2^59
    const int dA = min(em - fx_exp_sum(site_exp(X.e[n], r, j), site_exp(Y.e[p], r, w.h)) + down, 62);
    const int dB = min(em - fx_exp_sum(site_exp(X.e[p], r, w.h), site_exp(Y.e[n], r, j)) + down, 62);
    // colour `row` of the projected Y(y) and X(y)
    cx<i64> s[12] = {}, hy[6], hx[6];
    auto colour = [&](const FieldPair& F, int par, int h, int a, cx<i64> q[12]) {  // in units of the site's exponent
      cx<i64> c4[4];
      load_colour(F.v[par], Vh, r, h, a, c4);
      const int e0 = __ldg(F.e[par] + eidx(0, Vh, r, h)), e1 = __ldg(F.e[par] + eidx(1, Vh, r, h));
      const int d0 = min(max(e1 - e0, 0), 63), d1 = min(max(e0 - e1, 0), 63);
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const int d = k < 2 ? d0 : d1;
        q[3 * k] = cmk(c4[k].re >> d, c4[k].im >> d);
      }
    };
    colour(Y, p, w.h, w.row, s);
    project<MU, -1>(s, hy);
    colour(X, p, w.h, w.row, s);
    project<MU, +1>(s, hx);
    FxLimb yr[2], yi[2], xr[2], xi[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
      yr[k] = limb58(hy[3 * k].re, 3);
      yi[k] = limb58(hy[3 * k].im, 3);
      xr[k] = limb58(hx[3 * k].re, 3);
      xi[k] = limb58(hx[3 * k].im, 3);
    }
#pragma unroll
    for (int b = 0; b < 3; b++) {
      cx<i64> h[6];
      colour(X, n, j, b, s);
      project<MU, -1>(s, h);
      FxSum re = fx_sum<2>(), im = fx_sum<2>();
#pragma unroll
      for (int k = 0; k < 2; k++) {  // (A^dag)_row,b: conj(h_k,b) hw_k,row
        const FxLimb a = limb58(h[3 * k].re, 3), c = limb58(h[3 * k].im, 3);
        fx_mac(re, a, yr[k]);
        fx_mac(re, c, yi[k]);
        fx_mac(im, a, yi[k]);
        fx_mac(im, fx_neg(c), yr[k]);
      }
      t[b].re += fx_round_down(fx_value<2>(re), dA);
      t[b].im += fx_round_down(fx_value<2>(im), dA);
      colour(Y, n, j, b, s);
      project<MU, +1>(s, h);
      re = im = fx_sum<2>();
#pragma unroll
      for (int k = 0; k < 2; k++) {  // B_row,b: h'_k,row conj(hw'_k,b)
        const FxLimb a = limb58(h[3 * k].re, 3), c = limb58(h[3 * k].im, 3);
        fx_mac(re, a, xr[k]);
        fx_mac(re, c, xi[k]);
        fx_mac(im, a, xi[k]);
        fx_mac(im, fx_neg(c), xr[k]);
      }
      t[b].re += fx_round_down(fx_value<2>(re), dB);
      t[b].im += fx_round_down(fx_value<2>(im), dB);
    }
  }
  // |h| < 2^61, brought to 2^58: products in units of 2^(2 (3 - 60) + 60)
  unit = em - 54 + down;
  bad = em > FX_BIG;
}

// ---- per link (y, lambda = blockIdx.y): the hopping term (scaled by hop) and, with E, the clover leaves
// through it.  For each other direction o, with sign + for lambda < o and - for lambda > o,
//   G += U_o(y) U_l(y+o) E_o(y+l)^dag - E_o(y) U_l(y+o) U_o(y+l)^dag
//      + U_o(y-o)^dag U_l(y-o) E_o(y-o+l) - E_o(y-o)^dag U_l(y-o) U_o(y-o+l),
// E_o the insertion into U_o in the plane of l and o.
__global__ void __launch_bounds__(96, 4) link_force_fixed_kernel(Geom g, FxScalar hop, FxScalar hop_bc, int nrhs,
                                                              const int4* __restrict__ gfx, FieldPair X, FieldPair Y,
                                                              const int4* __restrict__ Efx, const int* __restrict__ eE,
                                                              double2* out, int gradient) {
  __shared__ RowsXch xch;
  const Where w = where(g);
  const int Vh = g.Vh, lam = blockIdx.y;
  const size_t V = 2 * (size_t)Vh;
  cx<i64> G[3] = {};
  int unit = FX_ZERO, i = 0;
  bool bad = false;
  if (w.valid) {
    const Site s = site_of(g, w.p, w.h);
    i = s.i;
    const FxSites f = {gfx, Vh, g.X, g.Y, g.Z, g.T, {s.x, s.y, s.z, s.t}, w.p};
    // exponents of the insertions used: E_o at y, y + l, y - o, y - o + l
    int em = FX_ZERO;
#pragma unroll 1
    for (int k = 0; k < 3; k++) {
      const int o = k < lam ? k : k + 1, mu = min(lam, o), nu = max(lam, o);
      const int pl = mu == 0 ? nu - 1 : (mu == 1 ? nu + 1 : 5);
      const int* e = eE + (size_t)(2 * pl + (o == nu ? 1 : 0)) * V;
      const size_t same = (size_t)w.p * Vh, other = (size_t)(1 - w.p) * Vh;
      const int e0 = __ldg(e + same + w.h), e1 = __ldg(e + other + fx_half_at(f, lam, 1, o, 0));
      const int e2 = __ldg(e + other + fx_half_at(f, lam, 0, o, -1)), e3 = __ldg(e + same + fx_half_at(f, lam, 1, o, -1));
      em = max(em, max(max(e0, e1), max(e2, e3)));
    }
    bad = em > FX_BIG;
#pragma unroll 1
    for (int k = 0; k < 3; k++) {
      const int o = k < lam ? k : k + 1, mu = min(lam, o), nu = max(lam, o);
      const int pl = mu == 0 ? nu - 1 : (mu == 1 ? nu + 1 : 5);
      const int fld = 2 * pl + (o == nu ? 1 : 0);
      const int4* E = Efx + (size_t)fld * 9 * V;
      const int* e = eE + (size_t)fld * V;
      const size_t y = (size_t)w.p * Vh + w.h, yl = (size_t)(1 - w.p) * Vh + fx_half_at(f, lam, 1, o, 0);
      const size_t yo = (size_t)(1 - w.p) * Vh + fx_half_at(f, lam, 0, o, -1);
      const size_t yol = (size_t)w.p * Vh + fx_half_at(f, lam, 1, o, -1);
      const int neg = lam < o ? 0 : -1;
      auto add = [&](const cx<i64> t[3], int et, int m) {
        const int d = min(em - et, 63);
#pragma unroll
        for (int j = 0; j < 3; j++) {
          G[j].re += fx_sign(t[j].re >> d, m);
          G[j].im += fx_sign(t[j].im >> d, m);
        }
      };
      cx<i64> t[3];
      const int4* ul = fx_link_at(f, lam, 0, o, 1, lam);
      fx_row_mul<true, 2>(fx_row_times<false>(fx_load_row<false>(fx_link_at(f, lam, 0, o, 0, o), Vh, w.row), ul, Vh),
                          E + yl, V, t);
      add(t, __ldg(e + yl), neg);
      fx_row_mul<true, 2>(fx_row_times<false>(fx_load_row<false>(E + y, V, w.row), ul, Vh), fx_link_at(f, lam, 1, o, 0, o),
                          Vh, t);
      add(t, __ldg(e + y), ~neg);
      ul = fx_link_at(f, lam, 0, o, -1, lam);
      fx_row_mul<false, 2>(fx_row_times<false>(fx_load_row<true>(fx_link_at(f, lam, 0, o, -1, o), Vh, w.row), ul, Vh),
                           E + yol, V, t);
      add(t, __ldg(e + yol), neg);
      fx_row_mul<false, 2>(fx_row_times<false>(fx_load_row<true>(E + yo, V, w.row), ul, Vh),
                           fx_link_at(f, lam, 1, o, -1, o), Vh, t);
      add(t, __ldg(e + yo), ~neg);
    }
    unit = em - 56;
    if (nrhs > 0) {
      // the hopping part, at full size times its coefficient, onto the larger unit
      cx<i64> t[3];
      int uh = 0;
      bool badh = false;
      const int j = fx_half_at(f, lam, 1, (lam + 1) & 3, 0);
      switch (lam) {
        case 0: hop_force_fx<0>(g, w, j, nrhs, X, Y, t, uh, badh); break;
        case 1: hop_force_fx<1>(g, w, j, nrhs, X, Y, t, uh, badh); break;
        case 2: hop_force_fx<2>(g, w, j, nrhs, X, Y, t, uh, badh); break;
        default: hop_force_fx<3>(g, w, j, nrhs, X, Y, t, uh, badh); break;
      }
      const bool edge = lam == 3 && s.t == g.T - 1;
      const FxLimb sv = edge ? hop_bc.v : hop.v;
      const int se = edge ? hop_bc.e : hop.e;
      const int up = 59 - fx_bits_n(t);
      bad = bad || badh || se > FX_BIG;
      // products of the coefficient (units of 2^(se - 59)) and t 2^up, in units of 2^60
      uh = uh - up + se - 59 + 60;
      const int um = max(unit, uh), d0 = min(um - unit, 62), d1 = min(um - uh, 62);
#pragma unroll
      for (int b = 0; b < 3; b++) {
        FxSum re = fx_sum<2>(), im = fx_sum<2>();
        fx_mac(re, sv, fx_split_balanced(fx_scaled(t[b].re, up)));
        fx_mac(im, sv, fx_split_balanced(fx_scaled(t[b].im, up)));
        G[b].re = fx_round_down(G[b].re, d0) + fx_round_down(fx_value<2>(re), d1);
        G[b].im = fx_round_down(G[b].im, d0) + fx_round_down(fx_value<2>(im), d1);
      }
      unit = um;
    }
  }
  double2* q = out + ((size_t)i * 4 + lam) * 9 + 3 * w.row;
  if (gradient) {
    if (!w.valid) return;
    const int e = bad ? FX_NAN : unit;
#pragma unroll
    for (int j = 0; j < 3; j++) q[j] = make_double2(fx_to_double(G[j].re, e, 0), fx_to_double(G[j].im, e, 0));
    return;
  }
  // F = -1/2 P_TA(U G^dag)
  store_ta<true>(g, w, gfx + (size_t)(w.p * 4 + lam) * 9 * Vh + w.h, G, unit, bad, -0.5, xch, q, false);
}

// ---- Wilson gauge force (qcd_md.cu): the staple sum
//   A = sum_o U_o(y+l) U_l(y+o)^dag U_o(y)^dag + U_o(y+l-o)^dag U_l(y-o)^dag U_o(y-o),
// G = -(beta/3) A^dag, F = (beta/6) P_TA(U A)
__global__ void __launch_bounds__(96, 7) gauge_force_fixed_kernel(Geom g, double beta, const int4* __restrict__ gfx,
                                                               const unsigned char* __restrict__ weak, double2* out,
                                                               int gradient, int accumulate) {
  __shared__ RowsXch xch;
  Where w = where(g);
  const int Vh = g.Vh, lam = blockIdx.y;
  if (weak) {
    w.valid = w.valid && !(weak[(size_t)w.p * Vh + w.h] >> lam & 1);
    if (__syncthreads_or(w.valid) == 0) return;
  }
  cx<i64> A[3] = {};  // in units of 2^-60
  int i = 0;
  if (w.valid) {
    const Site s = site_of(g, w.p, w.h);
    i = s.i;
    const FxSites f = {gfx, Vh, g.X, g.Y, g.Z, g.T, {s.x, s.y, s.z, s.t}, w.p};
#pragma unroll 1
    for (int k = 0; k < 3; k++) {
      const int o = k < lam ? k : k + 1;
      cx<i64> t[3], u[3];
      fx_row_mul<true>(fx_row_times<true>(fx_load_row_fine<false>(fx_link_at(f, lam, 1, o, 0, o), Vh, w.row),
                                          fx_link_at(f, lam, 0, o, 1, lam), Vh),
                       fx_link_at(f, lam, 0, o, 0, o), Vh, t);
      fx_row_mul<false>(fx_row_times<true>(fx_load_row_fine<true>(fx_link_at(f, lam, 1, o, -1, o), Vh, w.row),
                                           fx_link_at(f, lam, 0, o, -1, lam), Vh),
                        fx_link_at(f, lam, 0, o, -1, o), Vh, u);
#pragma unroll
      for (int j = 0; j < 3; j++) {  // six terms of 2^60 at most
        A[j].re += (t[j].re + u[j].re) >> 1;
        A[j].im += (t[j].im + u[j].im) >> 1;
      }
    }
  }
  double2* q = out + ((size_t)i * 4 + lam) * 9;
  if (gradient) {
    if (!w.valid) return;
    const double f = -beta / 3.0;
#pragma unroll
    for (int j = 0; j < 3; j++) {  // G_j,row = f conj(A_row,j)
      double2 o = make_double2(f * fx_to_double_in_range(A[j].re, -60), -f * fx_to_double_in_range(A[j].im, -60));
      double2* qq = q + 3 * j + w.row;
      if (accumulate) {
        const double2 was = *qq;
        o = make_double2(was.x + o.x, was.y + o.y);
      }
      *qq = o;
    }
    return;
  }
  store_ta<false>(g, w, gfx + (size_t)(w.p * 4 + lam) * 9 * Vh + w.h, A, -60, false, beta / 6.0, xch, q + 3 * w.row,
                  accumulate != 0);
}

// ---- sum over sites and planes (blockIdx.y) of Re tr P_{mu nu}(x) / 3, a row of the two corner products each
__global__ void __launch_bounds__(96) plaquette_fixed_kernel(Geom g, const int4* __restrict__ gfx, ReduceArgs red) {
  const Where w = where(g);
  const int Vh = g.Vh;
  int mu, nu;
  plane_of(blockIdx.y, mu, nu);
  double v = 0.0;
  if (w.valid) {
    const Site s = site_of(g, w.p, w.h);
    const FxSites f = {gfx, Vh, g.X, g.Y, g.Z, g.T, {s.x, s.y, s.z, s.t}, w.p};
    // Re tr(U_mu(x) U_nu(x+mu) (U_nu(x) U_mu(x+nu))^dag)
    const FxRow a = fx_row_times<false>(fx_load_row<false>(fx_link_at(f, mu, 0, nu, 0, mu), Vh, w.row),
                                        fx_link_at(f, mu, 1, nu, 0, nu), Vh);
    const FxRow b = fx_row_times<false>(fx_load_row<false>(fx_link_at(f, mu, 0, nu, 0, nu), Vh, w.row),
                                        fx_link_at(f, mu, 0, nu, 1, mu), Vh);
    FxSum t = fx_sum<2>();
#pragma unroll
    for (int j = 0; j < 3; j++) {
      fx_mac(t, a.re[j], b.re[j]);
      fx_mac(t, a.im[j], b.im[j]);
    }
    v = fx_to_double_in_range(fx_value<2>(t), -56) / 3.0;
  }
  const int nblk = gridDim.x * gridDim.y;
  block_partial<96>(v, 0, blockIdx.x * gridDim.y + blockIdx.y, nblk, red);
  grid_finish<96>(1, nblk, nblk, red);
}

dim3 rows_grid(const Geom& g, int ny) { return dim3(2 * ((g.Vh + 31) / 32), ny); }

FieldPair pair_of(const void* even, const void* odd, const float* even_e, const float* odd_e) {
  return FieldPair{{static_cast<const longlong2*>(even), static_cast<const longlong2*>(odd)},
                   {reinterpret_cast<const int*>(even_e), reinterpret_cast<const int*>(odd_e)}};
}

}  // namespace

// bytes of a fixed matrix field set: n fields of V matrices, then their exponents
size_t fixed_matrix_bytes(const Geom& g, int n) { return (size_t)n * 2 * g.Vh * (9 * sizeof(int4) + sizeof(int)); }

void launch_force_coeff_fixed(const Geom& g, double kappa, double csw, int nrhs, const void* Xe, const void* Xo,
                              const void* Ye, const void* Yo, const float* xe, const float* xo, const float* ye,
                              const float* yo, double2* Cbuf, cudaStream_t st) {
  g_kernel_launches += 1;
  const double f = kappa * csw / 4.0;
  clover_coeff_fixed_kernel<<<rows_grid(g, 1), 96, 0, st>>>(g, f, f * kappa * kappa, nrhs,
                                                           pair_of(Xe, Xo, xe, xo), pair_of(Ye, Yo, ye, yo), Cbuf);
}

void launch_force_edges_fixed(const Geom& g, const void* gfx, const double2* Cbuf, void* Cfx, void* Efx, cudaStream_t st) {
  g_kernel_launches += 2;
  const size_t V = 2 * (size_t)g.Vh;
  int4 *c = static_cast<int4*>(Cfx), *e = static_cast<int4*>(Efx);
  int *ec = reinterpret_cast<int*>(c + 6 * 9 * V), *ee = reinterpret_cast<int*>(e + 12 * 9 * V);
  coeff_to_fixed_kernel<<<(unsigned)((6 * V + 127) / 128), 128, 0, st>>>(V, Cbuf, c, ec);
  edge_fixed_kernel<<<rows_grid(g, 12), 96, 0, st>>>(g, static_cast<const int4*>(gfx), c, ec, e, ee);
}

void launch_force_links_fixed(const Geom& g, double kappa, int nrhs, const void* gfx, const void* Xe, const void* Xo,
                              const void* Ye, const void* Yo, const float* xe, const float* xo, const float* ye,
                              const float* yo, const void* Efx, double2* out, bool gradient, cudaStream_t st) {
  g_kernel_launches += 1;
  const int4* e = static_cast<const int4*>(Efx);
  const double hop = 2.0 * kappa * kappa;
  link_force_fixed_kernel<<<rows_grid(g, 4), 96, 0, st>>>(
      g, fx_scalar(hop), fx_scalar(hop * g.t_bc), nrhs, static_cast<const int4*>(gfx),
      pair_of(Xe, Xo, xe, xo), pair_of(Ye, Yo, ye, yo), e, reinterpret_cast<const int*>(e + 12 * 9 * 2 * (size_t)g.Vh), out,
      gradient ? 1 : 0);
}

void launch_plaquette_fixed(const Geom& g, const void* gfx, const ReduceArgs& red, cudaStream_t st) {
  g_kernel_launches += 1;
  plaquette_fixed_kernel<<<rows_grid(g, 6), 96, 0, st>>>(g, static_cast<const int4*>(gfx), red);
}

void launch_gauge_force_fixed(const Geom& g, double beta, const void* gfx, const unsigned char* weak, double2* out,
                              bool gradient, bool accumulate, cudaStream_t st) {
  g_kernel_launches += 1;
  gauge_force_fixed_kernel<<<rows_grid(g, 4), 96, 0, st>>>(g, beta, static_cast<const int4*>(gfx), weak, out,
                                                           gradient ? 1 : 0, accumulate ? 1 : 0);
}

}  // namespace qcd
