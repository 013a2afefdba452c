// Hopping kernels of the FP64 operators on block fixed-point integers (qcd_fixed.cuh): the same operators
// and epilogues as the FP64 pair-unit kernel, for near-unitary links.
#include <math.h>

#include <type_traits>

#include "qcd_dslash.cuh"
#include "qcd_fixed.cuh"
#include "qcd_kernels.h"

namespace qcd {

QCD_DEBUG_TAKE(debug_take_dslash_fx)

namespace {

// Stages of the neighbour ring, and rows of 32 16-byte elements of one stage: the 9 of a link, which the
// RHS of a block share, and the 12 of each pair's neighbour spinor.
constexpr int FX_STAGES = 2;
__host__ __device__ constexpr int fx_stage_rows(int pairs) { return 9 + 12 * pairs; }

// exchange area of one pair of warps: the components a warp passes to its partner (rows 0-5 to warp 0, 6-17
// to warp 1); it takes the place of the pair's spinor rows of stage 0, which the last hop does not use
struct FxXch {
  i64 v[18][32];  // [component re, im][lane]
};
static_assert(sizeof(FxXch) <= 12 * 32 * sizeof(int4), "the exchange area fits a pair's spinor rows");

// One hop for row k of the projected half spinor.  (1 + sgn g_mu) psi has in row k (upper spin)
// h = psi_k + c psi_p, with p the lower spin that g_mu couples to k and c = sgn (g_mu)_kp, one of +-1 (IMAG
// false: mu = y, t) or +-i (IMAG: mu = x, z); w = U h is added to the sum of spin k (up), and conj(c) w to
// that of spin p (low).  BWD: the backward hop (sgn = +1), which takes U^dag.  sk, sp, u: the staged rows of
// the neighbour's spins k and p and of the link; neg = -1: (g_mu)_kp is -1 or -i (0: 1 or i); g5 = -1: gamma_5 psi in
// place of psi, which changes the sign of psi_p (0: psi itself); flip: -w in place of w; psi_k and psi_p are
// brought down by dk and dp powers of two, from their blocks' units to the sum's.
// What is cut off to the unit is low by half a unit in the mean (with all hops cut off alike, every component
// was by up to 2^-54 of its site's bound).  So the hops of y and t form -w and subtract it: in up their halves
// cancel those of x and z, in low the forward hop's cancel the backward one's.  Exact values stay exact.
template <bool IMAG, bool BWD>
__device__ __forceinline__ void hop_fx(const longlong2* sk, const longlong2* sp, const int4* u, int neg, int g5,
                                       bool flip, int dk, int dp, cx<i64> up[3], cx<i64> low[3]) {
  if (!BWD) neg = ~neg;  // c = -+1, -+i
  const int f = neg ^ g5;
  FxLimb re[3], im[3];
#pragma unroll
  for (int b = 0; b < 3; b++) {
    longlong2 x = sk[32 * b], y = sp[32 * b];
    x.x >>= dk;
    x.y >>= dk;
    y.x >>= dp;
    y.y >>= dp;
    const i64 hr = IMAG ? x.x + fx_sign(y.y, ~f) : fx_sign(y.x, ~f) - x.x;  // h, or -h of y and t
    const i64 hi = IMAG ? x.y + fx_sign(y.x, f) : fx_sign(y.y, ~f) - x.y;
    re[b] = fx_split(hr);
    im[b] = fx_split(hi);
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    FxSum wr = {}, wi = {};
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const int4 v = u[32 * (BWD ? 3 * b + a : 3 * a + b)];
      const FxLimb ur = {v.x, v.y}, ui = {v.z, v.w};
      fx_mac(wr, ur, re[b]);
      fx_mac(wi, ur, im[b]);
      // u h: (ur re - ui im, ur im + ui re); conj(u) h: (ur re + ui im, ur im - ui re)
      fx_mac(wr, ui, BWD ? im[b] : fx_neg(im[b]));
      fx_mac(wi, ui, BWD ? fx_neg(re[b]) : re[b]);
    }
    i64 x = fx_value<0>(wr), y = fx_value<0>(wi);
    if (!IMAG && flip) {
      x = -x;
      y = -y;
    }
    up[a].re += IMAG ? x : -x;
    up[a].im += IMAG ? y : -y;
    // conj(c) w: c = +-1: +-w; c = +-i: -+i w
    low[a].re += IMAG ? fx_sign(y, neg) : fx_sign(x, ~neg);
    low[a].im += IMAG ? fx_sign(x, ~neg) : fx_sign(y, ~neg);
  }
}

// y = C x for a 6x6 block stored as in fx_store_clover (|x| < 2^60): values in units of 2^60 of the products
__device__ __forceinline__ void clover_fx(const int4* __restrict__ q, int Vh, const cx<i64> x[6], cx<i64> y[6]) {
  FxLimb re[6], im[6];
  FxSum yr[6] = {}, yi[6] = {};
#pragma unroll
  for (int k = 0; k < 6; k++) {
    re[k] = fx_split_balanced(x[k].re);
    im[k] = fx_split_balanced(x[k].im);
  }
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int4 v = __ldg(q + (size_t)k * Vh);
    const FxLimb d0 = {v.x, v.y}, d1 = {v.z, v.w};
    fx_mac(yr[2 * k], d0, re[2 * k]);
    fx_mac(yi[2 * k], d0, im[2 * k]);
    fx_mac(yr[2 * k + 1], d1, re[2 * k + 1]);
    fx_mac(yi[2 * k + 1], d1, im[2 * k + 1]);
  }
  int k = 0;
#pragma unroll
  for (int i = 1; i < 6; i++) {
#pragma unroll
    for (int j = 0; j < i; j++) {
      const int4 v = __ldg(q + (size_t)(3 + k) * Vh);
      const FxLimb lr = {v.x, v.y}, li = {v.z, v.w}, nli = fx_neg(li);
      // y_i += L x_j, y_j += conj(L) x_i
      fx_mac(yr[i], lr, re[j]);
      fx_mac(yr[i], nli, im[j]);
      fx_mac(yi[i], lr, im[j]);
      fx_mac(yi[i], li, re[j]);
      fx_mac(yr[j], lr, re[i]);
      fx_mac(yr[j], li, im[i]);
      fx_mac(yi[j], lr, im[i]);
      fx_mac(yi[j], nli, re[i]);
      k++;
    }
  }
#pragma unroll
  for (int i = 0; i < 6; i++) y[i] = cmk(fx_value<2>(yr[i]), fx_value<2>(yi[i]));
}

// the magnitudes' common bound 2^bits of six complex numbers (0 for zeros)
__device__ __forceinline__ int fx_bits_of(const cx<i64> t[6]) {
  u64 o = 0;
#pragma unroll
  for (int k = 0; k < 6; k++) o |= (u64)(t[k].re ^ (t[k].re >> 63)) | (u64)(t[k].im ^ (t[k].im >> 63));
  return 64 - fx_clz(o);
}

// t -> t 2^sh: one shift up, or one down rounded to nearest
struct FxShift {
  int up, down;
  i64 half;
  __device__ __forceinline__ i64 operator()(i64 t) const { return ((i64)((u64)t << up) + half) >> down; }
};
__device__ __forceinline__ FxShift fx_shift(int sh) {
  FxShift f;
  f.up = min(max(sh, 0), 63);
  f.down = min(max(-sh, 0), 63);
  f.half = f.down > 0 && f.down < 63 ? 1LL << (f.down - 1) : 0;
  return f;
}
// from units of 2^unit to those of a stored site of exponent e (a marked group's values do not matter)
__device__ __forceinline__ FxShift fx_shift(int unit, int e) {
  return fx_shift(e > FX_BIG ? -63 : unit - e + FX_SPINOR);
}

// The epilogue of chiral block B of a site, RHS r, with the hopping sum v in units of 2^(eh - 56), and its
// stores.  Returns the thread's share of |out|^2 (do_norm) or of |r|^2 (EPI_XPAY_CG, EPI_RESID).
template <int EPI>
__device__ __forceinline__ double finish_fx(const DslashArgs& A, const FxScalar& sc, int hh, bool valid, int r, int B,
                                            cx<i64> v[6], int eh) {
  const int Vh = A.g.Vh;
  double nrm = 0.0;
  cx<i64> t[6];
  int unit = 0;
  bool bad = eh > FX_BIG;
  if (valid) {
    // v: the hopping sum of chiral block B in units of 2^(eh - 56)
    unit = eh - 56;
    if (EPI == EPI_NONE) {
#pragma unroll
      for (int k = 0; k < 6; k++) t[k] = v[k];
    } else {
      // v brought to full size, |v| < 2^60, in units of 2^unit
      const int bits = fx_bits_of(v);
      const FxShift full = fx_shift(60 - bits);
#pragma unroll
      for (int k = 0; k < 6; k++) v[k] = cmk(full(v[k].re), full(v[k].im));
      unit += bits - 60;
      const bool ok = dbg_clover(Vh, hh, B);
      const int4* cl = static_cast<const int4*>(A.clover) + (size_t)(18 * B) * Vh + (ok ? hh : 0);
      const int ec = __ldg(A.clover_e + (size_t)B * Vh + (ok ? hh : 0));
      bad = bad || ec > FX_BIG;
      if (EPI == EPI_CLOVER_INV) {
        clover_fx(cl, Vh, v, t);
        unit += ec + 2;
      } else {
        cx<i64> xs[6], cxs[6];
        const longlong2* px = static_cast<const longlong2*>(A.x);
        const int exx = __ldg(reinterpret_cast<const int*>(A.x_norm) + eidx(B, Vh, r, hh));
        bad = bad || exx > FX_BIG || sc.e > FX_BIG;
#pragma unroll
        for (int k = 0; k < 6; k++) {
          const longlong2 x = __ldg(px + sidx<12>(6 * B + k, Vh, r, hh));
          xs[k] = cmk((i64)x.x, (i64)x.y);
        }
        if (A.x_g5 && B == 1) {
#pragma unroll
          for (int k = 0; k < 6; k++) xs[k] = -xs[k];
        }
        clover_fx(cl, Vh, xs, cxs);
        // C x in units of 2^u1, a v in units of 2^u2 (each below 2^61.5)
        const int u1 = exx - FX_SPINOR + ec + 2, u2 = unit + sc.e - 1;
        unit = max(u1, u2);
        const int k1 = min(unit - u1, 63), k2 = min(unit - u2, 63);
#pragma unroll
        for (int k = 0; k < 6; k++) {
          FxSum pr = {}, pi = {};
          fx_mac(pr, sc.v, fx_split(v[k].re));
          fx_mac(pi, sc.v, fx_split(v[k].im));
          t[k].re = (cxs[k].re >> k1) + (fx_value<4>(pr) >> k2);
          t[k].im = (cxs[k].im >> k1) + (fx_value<4>(pi) >> k2);
        }
      }
    }
    if (A.out_g5 && B == 1) {
#pragma unroll
      for (int k = 0; k < 6; k++) t[k] = -t[k];
    }
  }
  if (EPI == EPI_XPAY_CG || EPI == EPI_RESID || A.out_f64) {
    if (valid) {
      cx<double> res[6];
      const int e = bad ? FX_NAN : unit;
#pragma unroll
      for (int k = 0; k < 6; k++) res[k] = cmk(fx_to_double(t[k].re, e, 0), fx_to_double(t[k].im, e, 0));
      if (EPI == EPI_XPAY_CG) {
        if (A.red.cg[r].active) {
          const double al = A.red.cg[r].alpha;
          cx<double> ps[6], xs[6], rs[6];
          SpinorIO<60>::load_block(A.cg_p, A.cg_p_norm, Vh, r, hh, B, ps);
          SpinorIO<64>::load_block(A.cg_x, nullptr, Vh, r, hh, B, xs);
          SpinorIO<64>::load_block(A.cg_r, nullptr, Vh, r, hh, B, rs);
#pragma unroll
          for (int k = 0; k < 6; k++) {
            xs[k].re = fma(al, ps[k].re, xs[k].re);
            xs[k].im = fma(al, ps[k].im, xs[k].im);
            rs[k].re = fma(-al, res[k].re, rs[k].re);
            rs[k].im = fma(-al, res[k].im, rs[k].im);
            nrm = fma(rs[k].re, rs[k].re, nrm);
            nrm = fma(rs[k].im, rs[k].im, nrm);
          }
          SpinorIO<64>::store_block(A.cg_x, nullptr, Vh, r, hh, B, xs);
          SpinorIO<64>::store_block(A.cg_r, nullptr, Vh, r, hh, B, rs);
        }
      } else if (EPI == EPI_RESID) {
        cx<double> bs[6];
        SpinorIO<64>::load_block(A.cg_p, nullptr, Vh, r, hh, B, bs);
#pragma unroll
        for (int k = 0; k < 6; k++) {
          res[k] = bs[k] - res[k];
          nrm = fma(res[k].re, res[k].re, nrm);
          nrm = fma(res[k].im, res[k].im, nrm);
        }
        if (A.r_f64) {
          SpinorIO<64>::store_block(A.cg_r, nullptr, Vh, r, hh, B, res);
        } else {
          cx<float> lo[6];
#pragma unroll
          for (int k = 0; k < 6; k++) lo[k] = cmk(narrow(res[k].re), narrow(res[k].im));
          SpinorIO<32>::store_block(A.cg_r, nullptr, Vh, r, hh, B, lo);
        }
      } else {
        SpinorIO<64>::store_block(A.out, nullptr, Vh, r, hh, B, res);
      }
    }
    return nrm;
  }
  if (valid && dbg_spinor(Vh, r, hh)) {
    const int bits = fx_bits_of(t);
    const int e = bad ? FX_NAN : (bits ? unit + bits : FX_ZERO);
    const FxShift f = fx_shift(unit, e);
    longlong2* po = static_cast<longlong2*>(A.out);
    FxSum n = {};
#pragma unroll
    for (int k = 0; k < 6; k++) {
      const i64 a = f(t[k].re), b = f(t[k].im);
      if (A.do_norm) {  // |v| < 2^60, summed as squares of v / 4
        const FxLimb x = fx_split(a >> 2), y = fx_split(b >> 2);
        n.h += (i64)x.hi * x.hi;
        n.h += (i64)y.hi * y.hi;
        n.m += (i64)x.hi * x.lo;
        n.m += (i64)y.hi * y.lo;
      }
      po[sidx<12>(6 * B + k, Vh, r, hh)] = make_longlong2(a, b);
    }
    reinterpret_cast<int*>(A.out_norm)[eidx(B, Vh, r, hh)] = e;
    if (A.do_norm) {
      const int u = e > FX_BIG ? FX_NAN : 2 * (e - FX_SPINOR + 2);
      nrm = fx_to_double(n.h, u + 62, 0) + fx_to_double(n.m, u + 32, 0);
    }
  }
  return nrm;
}

// Warp B of a pair: half-spinor row B of the eight hops of 32 output sites and RHS r, then chiral block B
// (warp 0 passes on its parts of spins 2 and 3, warp 1 spin 1).  With the rows, not the directions, shared
// out, a thread's sums are 9 complex numbers instead of 12.  The neighbours and links of the hops come
// through a ring of shared-memory stages filled by cp.async a hop ahead (loaded to registers where they are
// used, the loads' latency was half the time: 32^4, 340 us a pass).  The hops are a loop over one body (x
// and y, then z and t): written out, their 7000 instructions ran at the rate at which the instruction cache
// was refilled (16^4: 90 us a pass).  All threads of the block call it together.
// nbs: the block's neighbour half indices, [mu][bwd][lane].
// Returns the thread's share of |out|^2 (do_norm) or of |r|^2 (EPI_XPAY_CG).
template <int EPI, int PAIRS>
__device__ __forceinline__ double pair_fx(const DslashArgs& A, const FxScalar& sc, int hh, bool valid, int time, int r,
                                          int q, int B, const int (*nbs)[2][32], int4* ring) {
  constexpr int STAGE = fx_stage_rows(PAIRS) * 32;
  const int lane = threadIdx.x & 31;
  const int Vh = A.g.Vh;
  cx<i64> up[3] = {}, lxy[3] = {}, low[3] = {};
  // copies of hop j's spinor (its chiral block B) and, by pair 0, of its link (rows 0-4 by warp 0, 5-8 by warp 1)
  const int4* in = static_cast<const int4*>(A.in) + ((size_t)r * 12 + 6 * B) * Vh;
  const int4* gl = static_cast<const int4*>(A.gauge) + (size_t)(5 * B) * Vh;
  int4* const dst = ring + lane;
  auto fetch = [&](int mu, int bwd, int j) {
    if (hh < Vh) {
      const int nb = nbs[mu][bwd][lane], pl = bwd ? 1 - A.p : A.p, hl = bwd ? nb : hh;
      int4* buf = dst + (j % FX_STAGES) * STAGE;
      if (dbg_link(Vh, pl, mu, hl) && dbg_spinor(Vh, r, nb)) {
        if (q == 0) {
          const int4* u = gl + (size_t)((pl * 4 + mu) * 9) * Vh + hl;
#pragma unroll
          for (int k = 0; k < 5; k++) {
            if (k < 4 || B == 0) cp_async16(buf + 32 * (5 * B + k), u);
            u += Vh;
          }
        }
        if (valid) {
          const int4* p = in + nb;
#pragma unroll
          for (int k = 0; k < 6; k++) {
            cp_async16(buf + 32 * (9 + 12 * q + 6 * B + k), p);
            p += Vh;
          }
        }
      }
    }
    cp_async_commit();
  };
  using F = std::false_type;
  using T = std::true_type;
  static_assert(FX_STAGES == 2, "the loop below fetches one hop ahead");
  fetch(0, 0, 0);
  int eh = FX_ZERO;
  unsigned dwk[2] = {0, 0}, dwp[2] = {0, 0};
  if (valid) {
    const int* ex = reinterpret_cast<const int*>(A.in_norm) + eidx(0, Vh, r, 0);
    int ek[8], ep[8];  // of the neighbours' blocks 0 (spin k) and 1 (spin p)
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int nb = nbs[k >> 1][k & 1][lane];
      ek[k] = __ldg(ex + nb);
      ep[k] = __ldg(ex + Vh + nb);
    }
#pragma unroll
    for (int k = 0; k < 8; k++) eh = max(eh, max(ek[k], ep[k]));
    // the neighbours' shifts, eight bits each: byte 2 (mu >> 1) + bwd of word mu & 1
#pragma unroll
    for (int k = 0; k < 8; k++) {
      dwk[(k >> 1) & 1] |= (unsigned)min(eh - ek[k], 63) << (8 * (2 * (k >> 2) + (k & 1)));
      dwp[(k >> 1) & 1] |= (unsigned)min(eh - ep[k], 63) << (8 * (2 * (k >> 2) + (k & 1)));
    }
  }
  {
    const int g5 = A.in_g5 ? -1 : 0;
    const int tg = time + A.g.t0;
    const bool anti = A.g.t_bc < 0.0;
#pragma unroll 1
    for (int zt = 0; zt < 2; zt++) {
      // directions x, y (zt = 0), then z, t
      int z = zt;
      asm volatile("" : "+r"(z));  // one body for both: the loop is not to be split by zt
      const int p = z ? 2 + B : 3 - B;  // the lower spin
      if (z) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
          lxy[a] = low[a];
          low[a] = {};
        }
      }
      // hop j = 4 z + 2 ODD + BWD (the stage it takes is known: 4 z is even)
      auto hop = [&](auto odd_c, auto bwd_c) {
        constexpr bool ODD = decltype(odd_c)::value, BWD = decltype(bwd_c)::value;
        cp_async_wait_all();
        __syncthreads();
        if (!BWD) fetch(2 * z + (ODD ? 1 : 0), 1, 1);
        else if (!ODD) fetch(2 * z + 1, 0, 0);
        else if (!z) fetch(2, 0, 0);
        const int4* buf = dst + (BWD ? 1 : 0) * STAGE;
        const longlong2* sp = reinterpret_cast<const longlong2*>(buf) + 32 * (9 + 12 * q);
        // (g_mu)_Bp: x i, i; y -1, 1; z i, -i; t 1, 1 (B = 0, 1)
        const int neg = ODD ? (!z && B == 0 ? -1 : 0) : (z && B == 1 ? -1 : 0);
        const bool flip = ODD && z && anti && tg == (BWD ? 0 : A.g.Tg - 1);
        const int sh = 16 * z + (BWD ? 8 : 0);
        const int dk = (dwk[ODD ? 1 : 0] >> sh) & 63, dp = (dwp[ODD ? 1 : 0] >> sh) & 63;
        hop_fx<!ODD, BWD>(sp + 96 * B, sp + 96 * p, buf, neg, g5, flip, dk, dp, up, low);
      };
      hop(F(), F());
      hop(F(), T());
      hop(T(), F());
      hop(T(), T());
    }
  }
  FxXch* xch = reinterpret_cast<FxXch*>(ring + 32 * (9 + 12 * q));
  // warp 0 holds spin 0, and of spins 3, 2 the parts lxy, low; warp 1 spin 1, and of spins 2, 3 lxy, low
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const cx<i64> o = B == 0 ? low[a] : up[a];
    const int at = B == 0 ? 6 : 0;
    xch->v[at + 2 * a][lane] = o.re;
    xch->v[at + 2 * a + 1][lane] = o.im;
    if (B == 0) {
      xch->v[12 + 2 * a][lane] = lxy[a].re;
      xch->v[12 + 2 * a + 1][lane] = lxy[a].im;
    }
  }
  __syncthreads();
  // the hopping sum of chiral block B
  cx<i64> v[6] = {};
  if (valid) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const int at = B == 0 ? 0 : 6;
      const cx<i64> p0 = cmk(xch->v[at + 2 * a][lane], xch->v[at + 2 * a + 1][lane]);
      if (B == 0) {
        v[a] = up[a];
        v[3 + a] = p0;
      } else {
        v[a] = lxy[a] + p0;
        v[3 + a] = low[a] + cmk(xch->v[12 + 2 * a][lane], xch->v[12 + 2 * a + 1][lane]);
      }
    }
  }
  return finish_fx<EPI>(A, sc, hh, valid, r, B, v, eh);
}

// One pair of warps per (32 output sites, RHS); a block holds the pairs of PAIRS RHS of the same sites (nrhs is
// a multiple of PAIRS), which share the staged links.  Bound by instruction issue: 4290 instructions per warp, 1260 of them
// multiply-adds that take two issue slots, 45% of the slots issuing at 16 warps per SM (128 registers);
// 32^4, 1 RHS: 256 us a pass with the inverse clover block, 57% of DRAM throughput, bytes read once.
template <int EPI, int PAIRS>
__global__ void __launch_bounds__(64 * PAIRS, 8 / PAIRS) dslash_fixed_kernel(DslashArgs A,
                                                                                            FxScalar sc) {
  extern __shared__ __align__(16) int4 fx_ring[];
  __shared__ int nbs[4][2][32];
  if ((A.halt && *A.halt) || (A.gate && !*A.gate)) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, q = w >> 1;
  const int hh = blockIdx.x * 32 + lane;
  const bool site = hh < A.g.Vh;
  Site s{};
  if (site) {
    s = site_of(A.g, A.p, hh);
    if (q == 0) {  // warp 0: x, y; warp 1: z, t
#pragma unroll
      for (int m = 0; m < 2; m++) {
        nbs[2 * w + m][0][lane] = (w ? neighbor_fwd(A.g, s, 2 + m) : neighbor_fwd(A.g, s, m)) >> 1;
        nbs[2 * w + m][1][lane] = (w ? neighbor_bwd(A.g, s, 2 + m) : neighbor_bwd(A.g, s, m)) >> 1;
      }
    }
  }
  __syncthreads();
  const bool reduce = A.do_norm || EPI == EPI_XPAY_CG || EPI == EPI_RESID;
#pragma unroll 1
  for (int r0 = 0; r0 < A.nrhs; r0 += PAIRS) {
    const int r = r0 + q;
    if (r0 > 0) __syncthreads();  // the exchange area of the last RHS has been read
    double nrm = pair_fx<EPI, PAIRS>(A, sc, hh, site, s.t, r, q, w & 1, nbs, fx_ring);
    if (reduce) {
      for (int off = 16; off >= 1; off >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, off);
      if (lane == 0) {
        const long long slot = (long long)r * (2 * gridDim.x) + 2 * blockIdx.x + (w & 1);
        if (slot < A.red.capacity) A.red.partials[slot] = nrm;
        else A.red.ctl->overflow = 1;
      }
    }
  }
  if (reduce) grid_finish<0>(A.nrhs, gridDim.x, 2 * gridDim.x, A.red);
}

// The same for lattices whose pairs of warps would leave most of the GPU idle: four pairs per 32 output sites
// and RHS (blockIdx.y), one direction each, whose sums meet in shared memory; pair 0 finishes the sites.  A
// pass is then two hops and an epilogue long instead of eight hops and an epilogue, at the same work.
template <int EPI>
__global__ void __launch_bounds__(256, 2) dslash_fixed_split_kernel(DslashArgs A, FxScalar sc) {
  extern __shared__ __align__(16) int4 fx_ring[];
  if ((A.halt && *A.halt) || (A.gate && !*A.gate)) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, q = w >> 1, B = w & 1, r = blockIdx.y;
  const int hh = blockIdx.x * 32 + lane, Vh = A.g.Vh;
  const bool valid = hh < Vh && dbg_spinor(Vh, r, hh);
  constexpr int STAGE = fx_stage_rows(1) * 32;
  int4* mine = fx_ring + 2 * q * STAGE + lane;  // the forward hop's stage, then the backward one's
  Site s{};
  int eh = FX_ZERO, ef[2] = {0, 0}, eb[2] = {0, 0};  // [chiral block]
  if (valid) {
    s = site_of(A.g, A.p, hh);
    const int* ex = reinterpret_cast<const int*>(A.in_norm) + eidx(0, Vh, r, 0);
    const int nf = neighbor_fwd(A.g, s, q) >> 1, nb = neighbor_bwd(A.g, s, q) >> 1;
    const int4* in = static_cast<const int4*>(A.in) + ((size_t)r * 12 + 6 * B) * Vh;
    const int4* u = static_cast<const int4*>(A.gauge) + (size_t)(5 * B) * Vh;
    const int4* uf = u + (size_t)((A.p * 4 + q) * 9) * Vh + hh;
    const int4* ub = u + (size_t)(((1 - A.p) * 4 + q) * 9) * Vh + nb;
    const int4 *pf = in + nf, *pb = in + nb;
    if (dbg_link(Vh, 1 - A.p, q, nb) && dbg_spinor(Vh, r, nf)) {
#pragma unroll
      for (int k = 0; k < 6; k++) {
        cp_async16(mine + 32 * (9 + 6 * B + k), pf + (size_t)k * Vh);
        cp_async16(mine + STAGE + 32 * (9 + 6 * B + k), pb + (size_t)k * Vh);
      }
#pragma unroll
      for (int k = 0; k < 5; k++) {
        if (k < 4 || B == 0) {
          cp_async16(mine + 32 * (5 * B + k), uf + (size_t)k * Vh);
          cp_async16(mine + STAGE + 32 * (5 * B + k), ub + (size_t)k * Vh);
        }
      }
    }
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
      const int hf = neighbor_fwd(A.g, s, mu) >> 1, hb = neighbor_bwd(A.g, s, mu) >> 1;
#pragma unroll
      for (int k = 0; k < 2; k++) {
        const int a = __ldg(ex + (size_t)k * Vh + hf), b = __ldg(ex + (size_t)k * Vh + hb);
        eh = max(eh, max(a, b));
        ef[k] = mu == q ? a : ef[k];
        eb[k] = mu == q ? b : eb[k];
      }
    }
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  cx<i64> up[3] = {}, low[3] = {};
  {
    const int g5 = A.in_g5 ? -1 : 0, p = q < 2 ? 3 - B : 2 + B;
    const int fk = min(eh - ef[0], 63), fp = min(eh - ef[1], 63), bk = min(eh - eb[0], 63), bp = min(eh - eb[1], 63);
    const int tg = s.t + A.g.t0;
    const longlong2* sf = reinterpret_cast<const longlong2*>(mine) + 32 * 9;
    const longlong2* sb = sf + STAGE;
    if (q & 1) {  // (g_y)_Bp: -1, 1; (g_t)_Bp: 1, 1
      const int neg = q == 1 && B == 0 ? -1 : 0;
      const bool anti = q == 3 && A.g.t_bc < 0.0;
      hop_fx<false, false>(sf + 96 * B, sf + 96 * p, mine, neg, g5, anti && tg == A.g.Tg - 1, fk, fp, up, low);
      hop_fx<false, true>(sb + 96 * B, sb + 96 * p, mine + STAGE, neg, g5, anti && tg == 0, bk, bp, up, low);
    } else {  // (g_x)_Bp: i, i; (g_z)_Bp: i, -i
      const int neg = q == 2 && B == 1 ? -1 : 0;
      hop_fx<true, false>(sf + 96 * B, sf + 96 * p, mine, neg, g5, false, fk, fp, up, low);
      hop_fx<true, true>(sb + 96 * B, sb + 96 * p, mine + STAGE, neg, g5, false, bk, bp, up, low);
    }
  }
  __syncthreads();  // every pair has read its stages: the sums take their place
  i64 (*part)[12][32] = reinterpret_cast<i64 (*)[12][32]>(fx_ring);  // [warp][up, low: component re, im][lane]
#pragma unroll
  for (int a = 0; a < 3; a++) {
    part[w][2 * a][lane] = up[a].re;
    part[w][2 * a + 1][lane] = up[a].im;
    part[w][6 + 2 * a][lane] = low[a].re;
    part[w][6 + 2 * a + 1][lane] = low[a].im;
  }
  __syncthreads();
  cx<i64> v[6] = {};
  if (q == 0 && valid) {
#pragma unroll
    for (int d = 0; d < 4; d++)
#pragma unroll
      for (int a = 0; a < 3; a++) {
        // block 0: the upper spins 0, 1 of warps 0, 1; block 1: spin 2 from warp 1 (x, y) or 0 (z, t), spin 3
        // from the other
        const int w0 = 2 * d + (B == 0 ? 0 : (d < 2 ? 1 : 0)), w1 = 2 * d + (B == 0 ? 1 : (d < 2 ? 0 : 1));
        const int o = B == 0 ? 2 * a : 6 + 2 * a;
        v[a] = v[a] + cmk(part[w0][o][lane], part[w0][o + 1][lane]);
        v[3 + a] = v[3 + a] + cmk(part[w1][o][lane], part[w1][o + 1][lane]);
      }
  }
  double nrm = finish_fx<EPI>(A, sc, hh, valid && q == 0, r, B, v, eh);
  if (A.do_norm || EPI == EPI_XPAY_CG || EPI == EPI_RESID) {
    if (q == 0) {
      for (int off = 16; off >= 1; off >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, off);
      if (lane == 0) {
        const long long slot = (long long)r * (2 * gridDim.x) + 2 * blockIdx.x + B;
        if (slot < A.red.capacity) A.red.partials[slot] = nrm;
        else A.red.ctl->overflow = 1;
      }
    }
    grid_finish<256>(A.nrhs, (long long)gridDim.x * gridDim.y, 2 * gridDim.x, A.red);
  }
}

// out = C in on the sites of one parity, one thread per (site, RHS, chiral block)
__global__ void __launch_bounds__(128) clover_fixed_kernel(Geom g, const int4* clover, const int* clover_e,
                                                           const longlong2* in, const int* in_e, longlong2* out,
                                                           int* out_e, int nrhs) {
  const int Vh = g.Vh, n = Vh * nrhs, k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= 2 * n) return;
  const int b = k >= n, tid = k - b * n, r = tid / Vh, h = tid - r * Vh;
  if (!dbg_spinor(Vh, r, h) || !dbg_clover(Vh, h, b)) return;
  const int ex = in_e[eidx(b, Vh, r, h)], ec = clover_e[(size_t)b * Vh + h];
  cx<i64> x[6], t[6];
#pragma unroll
  for (int c = 0; c < 6; c++) {
    const longlong2 v = in[sidx<12>(6 * b + c, Vh, r, h)];
    x[c] = cmk((i64)v.x, (i64)v.y);
  }
  clover_fx(clover + (size_t)(18 * b) * Vh + h, Vh, x, t);
  const int unit = ex - FX_SPINOR + ec + 2, bits = fx_bits_of(t);
  const int e = ex > FX_BIG || ec > FX_BIG ? FX_NAN : (bits ? unit + bits : FX_ZERO);
  const FxShift f = fx_shift(unit, e);
#pragma unroll
  for (int c = 0; c < 6; c++) out[sidx<12>(6 * b + c, Vh, r, h)] = make_longlong2(f(t[c].re), f(t[c].im));
  out_e[eidx(b, Vh, r, h)] = e;
}

}  // namespace

void launch_clover_apply_fixed(const Geom& g, const void* clover, const int* clover_e, const void* in,
                               const float* in_e, void* out, float* out_e, int nrhs, cudaStream_t st) {
  g_kernel_launches += 1;
  const int B = 128;
  clover_fixed_kernel<<<(2 * g.Vh * nrhs + B - 1) / B, B, 0, st>>>(
      g, static_cast<const int4*>(clover), clover_e, static_cast<const longlong2*>(in),
      reinterpret_cast<const int*>(in_e), static_cast<longlong2*>(out), reinterpret_cast<int*>(out_e), nrhs);
}

namespace {

template <int EPI, int PAIRS>
void launch_fx_pairs(const DslashArgs& a, const FxScalar& sc, cudaStream_t st) {
  const size_t sh = sizeof(int4) * 32 * fx_stage_rows(PAIRS) * FX_STAGES;
  if (sh > 48 * 1024)
    cudaFuncSetAttribute(dslash_fixed_kernel<EPI, PAIRS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  dslash_fixed_kernel<EPI, PAIRS><<<(a.g.Vh + 31) / 32, 64 * PAIRS, sh, st>>>(a, sc);
}

// The split kernel where its blocks, one a unit of 32 sites and RHS, are no more than the SMs: a pass of one pair of
// warps a unit would leave the others idle (4^3 x 8, 8 units, split 10.4 us a pass, pairs 12.6; 8 x 8 x 16 x 16, 256
// units, 14.5 against 14.3; 12^3 x 20, 540 units, 23.0 against 18.2 us).
//
// Otherwise two RHS share a block's links from two RHS on, and four where all blocks of four are resident at once
// (two an SM), so that the wider block is there to fill the SMs.  Clover-inverse / xpay passes in us with 1, 2 or 4
// RHS a block, 4 RHS: 128 blocks of sites 38/41, 24/25, 19/20; 300: -, 30/33, 27/29; 473: -, 46/49, 48/54; 1024: 86/94,
// 75/82, 78/89; 24^3 x 32, 6912: 451/519, 431/476, 472/515.  8 RHS: 128: 71/78, 41/44, 31/33; 300: -, 54/58, 48/51;
// 6912: 905/1062, 859/946, 927/1002.
template <int EPI>
void launch_fx(const DslashArgs& a, const FxScalar& sc, cudaStream_t st) {
  const int nb = (a.g.Vh + 31) / 32;
  if ((long long)nb * a.nrhs <= a.sms) {
    constexpr size_t sh = sizeof(int4) * 32 * fx_stage_rows(1) * 8;
    cudaFuncSetAttribute(dslash_fixed_split_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    dslash_fixed_split_kernel<EPI><<<dim3(nb, a.nrhs), 256, sh, st>>>(a, sc);
    return;
  }
  if (a.nrhs >= 4 && nb <= 2 * a.sms) launch_fx_pairs<EPI, 4>(a, sc, st);
  else if (a.nrhs >= 2) launch_fx_pairs<EPI, 2>(a, sc, st);
  else launch_fx_pairs<EPI, 1>(a, sc, st);
}

}  // namespace

void launch_dslash_fixed(int epi, const DslashArgs& a, cudaStream_t st) {
  g_kernel_launches += 1;
  const FxScalar sc = fx_scalar(a.a);
  switch (epi) {
    case EPI_NONE: launch_fx<EPI_NONE>(a, sc, st); break;
    case EPI_CLOVER_INV: launch_fx<EPI_CLOVER_INV>(a, sc, st); break;
    case EPI_XPAY_CG: launch_fx<EPI_XPAY_CG>(a, sc, st); break;
    case EPI_RESID: launch_fx<EPI_RESID>(a, sc, st); break;
    default: launch_fx<EPI_XPAY>(a, sc, st); break;
  }
}

}  // namespace qcd

extern "C" long long qcd_selftest_fixed(void) {
  using namespace qcd;
  long long bad = 0;
  u64 state = 0x9E3779B97F4A7C15ULL;
  auto next = [&]() {
    state ^= state << 13;
    state ^= state >> 7;
    state ^= state << 17;
    return state;
  };
  // doubles there and back: exact for a group's largest member, whatever its exponent (subnormals included)
  for (int i = 0; i < 200000; i++) {
    const double x = fx_from_bits(next() & ~(i % 3 == 0 ? 0x7ff0000000000000ULL : 0x0010000000000000ULL));
    const int e = fx_exponent(fx_mag(x));
    if (e > FX_BIG) continue;
    if (fx_to_double(fx_of_double<FX_SPINOR>(x, e), e, FX_SPINOR) != x) bad++;
    // a member 2^30 below the group's largest keeps 2^-60 of that, rounded
    const double y = fx_to_double(fx_of_double<FX_SPINOR>(x, e + 30), e + 30, FX_SPINOR);
    const double step = e > -900 ? fx_from_bits((u64)(e + 30 - FX_SPINOR + 1022) << 52) : 0.0;
    if (e > -900 && e < 900 && !(fabs(y - x) <= step)) bad++;
  }
  if (fx_exponent(fx_mag(INFINITY)) != FX_NAN || fx_exponent(fx_mag(NAN)) != FX_NAN || fx_exponent(0) != FX_ZERO) bad++;
  if (fx_to_double(1, FX_NAN, FX_SPINOR) == fx_to_double(1, FX_NAN, FX_SPINOR)) bad++;  // NaN
  // limbs
  for (int i = 0; i < 100000; i++) {
    const i64 v = (i64)(next() >> 2) - (1LL << 61);
    const FxLimb a = fx_split(v), b = fx_split_balanced(v);
    if (((i64)a.hi * (1LL << 31)) + a.lo != v || a.lo < 0) bad++;
    if (((i64)b.hi * (1LL << 31)) + b.lo != v || b.lo < -(1 << 30) || b.lo >= (1 << 30)) bad++;
  }
  // sums of n products |a| <= 2^abits, |b| <= 2^bbits in units of 2^(62 - K): right to the n dropped terms
  auto sums = [&](int n, int abits, int bbits, bool balanced, int K) {
    for (int i = 0; i < 20000; i++) {
      FxSum s = {};
      __int128 exact = 0;
      for (int k = 0; k < n; k++) {
        i64 a = (i64)(next() >> (63 - abits)), b = (i64)(next() >> (63 - bbits));
        a -= 1LL << abits;
        b -= 1LL << bbits;
        if (i % 4 == 1) a = 1LL << abits, b = 1LL << bbits;                  // the largest sum
        if (i % 4 == 2) a = (1LL << abits) - (1LL << 30), b = (1LL << bbits) - 1;  // the largest low limbs
        if (i % 8 == 3) a = -a;
        // (a row's norm bounds the hops' sums: their largest factors do not all meet)
        if (n == 6) a >>= 1;
        exact += (__int128)a * b;
        fx_mac(s, fx_split_balanced(a), balanced ? fx_split_balanced(b) : fx_split(b));
      }
      const i64 got = K == 0 ? fx_value<0>(s) : (K == 2 ? fx_value<2>(s) : fx_value<4>(s));
      const __int128 diff = exact - (__int128)got * ((__int128)1 << (62 - K));
      const __int128 most = (__int128)n * ((__int128)1 << 61) + ((__int128)1 << (62 - K));
      if (diff > most || diff < -most) bad++;
    }
  };
  sums(6, FX_LINK, FX_SPINOR + 1, false, 0);   // a hop
  sums(11, FX_CLOVER, FX_SPINOR, true, 2);     // a row of a clover block
  sums(1, FX_SCALAR, FX_SPINOR, false, 4);     // a coefficient
  return bad;
}
