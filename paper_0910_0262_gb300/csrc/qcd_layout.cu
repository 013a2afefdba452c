// Layout kernels: canonical complex128 fields <-> checkerboarded structure-of-arrays.
//
// The paper pads MILC's site structs to 128-byte multiples and odd strides so
// that the Cell's DMA engine reaches full bank bandwidth (Sec. 3).  On a GPU
// the equivalent goal -- every byte fetched is a byte used -- is met by a
// component-major, site-minor layout per parity: consecutive threads (sites)
// read consecutive 8/16-byte words, so no padding is transferred at all.
#include "qcd_fxmat.cuh"
#include "qcd_kernels.h"

namespace qcd {

QCD_DEBUG_TAKE(debug_take_layout)

std::atomic<long long> g_kernel_launches{0};

namespace {

__device__ __forceinline__ void coords_of(const Geom& g, int i, int& x, int& y, int& z, int& t) {
  int c[4];
  lattice_coords(g, i, c);
  x = c[0];
  y = c[1];
  z = c[2];
  t = c[3];
}

// whether U U^dag = 1 to 1e-5 (rows 0, 1, 2 of v), in FP32
__device__ __forceinline__ bool near_unitary(const float2 v[9]) {
  float worst = 0.f;
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b <= a; b++) {
      float re = a == b ? -1.f : 0.f, im = 0.f;
#pragma unroll
      for (int k = 0; k < 3; k++) {
        const float2 x = v[3 * a + k], y = v[3 * b + k];
        re += x.x * y.x + x.y * y.y;
        im += x.y * y.x - x.x * y.y;
      }
      worst = fmaxf(worst, fmaxf(fabsf(re), fabsf(im)));
    }
  return worst < 1e-5f;
}

// whether an entry of U - 1 is 2^-4 or more (the bound of qcd_fxmat.cuh)
__device__ __forceinline__ bool far_from_one(const float2 v[9]) {
  float most = 0.f;
#pragma unroll
  for (int k = 0; k < 9; k++) most = fmaxf(most, fmaxf(fabsf(k % 4 == 0 ? v[k].x - 1.f : v[k].x), fabsf(v[k].y)));
  return most >= 0.0625f;
}

// canonical gauge U[i][mu][3][3] complex128 -> per-parity, per-direction SoA copies.  gfx: the block
// fixed-point copy, which serves near-unitary links only, with far; *not_unitary is set if one is not.
// *non_finite (may be null) is set if a link holds a non-finite value.
__global__ void pack_gauge_kernel(Geom g, const double2* __restrict__ U, double2* g64, void* g32, int recon32,
                                  void* g16, int recon16, int4* gfx, unsigned char* far, int* not_unitary,
                                  int* non_finite) {
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  const int V = 2 * g.Vh;
  if (tid >= V * 4) return;
  const int i = tid >> 2, mu = tid & 3;
  int x, y, z, t;
  coords_of(g, i, x, y, z, t);
  const int p = (x + y + z + t) & 1;
  const int h = i >> 1;
  const double2* src = U + (size_t)tid * 9;
  double2 u[9];
#pragma unroll
  for (int k = 0; k < 9; k++) u[k] = src[k];
  bool bad = false;
  float2 v[9];
#pragma unroll
  for (int k = 0; k < 9; k++) {
    bad |= !isfinite(u[k].x) || !isfinite(u[k].y);
    v[k] = make_float2(narrow_many(u[k].x), narrow_many(u[k].y));
  }
  if (bad && non_finite) *non_finite = 1;
  const size_t base = (size_t)(p * 4 + mu);
#pragma unroll
  for (int k = 0; k < 9; k++) g64[(base * 9 + k) * g.Vh + h] = u[k];
  if (gfx) {
    fx_store_link(gfx + base * 9 * g.Vh + h, g.Vh, u);
    // (a site's four links lie in neighbouring lanes; V is a multiple of 16, so warps are whole)
    const unsigned f = __ballot_sync(0xffffffffu, far_from_one(v));
    if (mu == 0) far[(size_t)p * g.Vh + h] = (unsigned char)(f >> (threadIdx.x & 28) & 15);
    if (!near_unitary(v)) *not_unitary = 1;
  }
  if (g32) {
    if (recon32 == 12) {
      float4* q = static_cast<float4*>(g32);
#pragma unroll
      for (int k = 0; k < 3; k++)
        q[(base * 3 + k) * g.Vh + h] = make_float4(v[2 * k].x, v[2 * k].y, v[2 * k + 1].x, v[2 * k + 1].y);
    } else {
      float2* q = static_cast<float2*>(g32);
#pragma unroll
      for (int k = 0; k < 9; k++) q[(base * 9 + k) * g.Vh + h] = v[k];
    }
  }
  if (g16) {
    if (recon16 == 12) {
      uint2* q = static_cast<uint2*>(g16);
#pragma unroll
      for (int k = 0; k < 3; k++) {
        q[(base * 3 + k) * g.Vh + h] =
            make_uint2(f2h(v[2 * k].x, v[2 * k].y), f2h(v[2 * k + 1].x, v[2 * k + 1].y));
      }
    } else {
      uint32_t* q = static_cast<uint32_t*>(g16);
#pragma unroll
      for (int k = 0; k < 9; k++) q[(base * 9 + k) * g.Vh + h] = f2h(v[k].x, v[k].y);
    }
  }
}

// Per site the planes and directions all of whose links are close to one (the twelve links of the four leaves of
// F_{mu nu}(x); the link U_l(x) and the 18 of its staples), for a whole block of 32 sites of a parity if for one of
// them: a block would take the time of both kernels to be shared out between them.
__global__ void __launch_bounds__(128) weak_sites_kernel(Geom g, const unsigned char* __restrict__ far,
                                                         unsigned char* weakF, unsigned char* weakG, int* any) {
  const int nb = (g.Vh + 31) / 32, blk = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (blk >= 2 * nb) return;
  const int p = blk >= nb, h = (blk - p * nb) * 32 + (threadIdx.x & 31);
  const bool valid = h < g.Vh;
  const Site s = site_of(g, p, valid ? h : 0);
  const FxSites f = {nullptr, g.Vh, g.X, g.Y, g.Z, g.T, {s.x, s.y, s.z, s.t}, p};
  // the far links of a site in its directions, a bit each
  auto at = [&](int d1, int s1, int d2, int s2) {
    return (int)__ldg(far + (size_t)((p + s1 + s2) & 1) * g.Vh + fx_half_at(f, d1, s1, d2, s2));
  };
  int fwd[4], bwd[4];
#pragma unroll
  for (int m = 0; m < 4; m++) {
    fwd[m] = at(m, 1, (m + 1) & 3, 0);
    bwd[m] = at(m, -1, (m + 1) & 3, 0);
  }
  const int here = at(0, 0, 1, 0);
  int wF = 0, force = 0;  // force: directions with a link in their staples that is far from one
  int pl = 0;
#pragma unroll
  for (int m = 0; m < 3; m++)
#pragma unroll
    for (int n = m + 1; n < 4; n++) {
      const int M = 1 << m, N = 1 << n, fb = at(m, 1, n, -1), bf = at(m, -1, n, 1), bb = at(m, -1, n, -1);
      // U_m and U_n here, U_n(x+m), U_m(x+n); with U_n(x+m-n), U_m(x-n), U_n(x-n) the staples of U_m, with
      // U_m(x-m+n), U_n(x-m), U_m(x-m) those of U_n
      const int both = (here & (M | N)) | (fwd[m] & N) | (fwd[n] & M);
      const int of_m = (fb & N) | (bwd[n] & (M | N)), of_n = (bf & M) | (bwd[m] & (M | N));
      if (!(both | of_m | of_n | (bb & (M | N)))) wF |= 1 << pl;
      if (both | of_m) force |= M;
      if (both | of_n) force |= N;
      pl++;
    }
  const int marks = __reduce_or_sync(0xffffffffu, valid ? wF | (~force & 15) << 6 : 0);
  if (!valid) return;
  weakF[(size_t)p * g.Vh + h] = (unsigned char)(marks & 63);
  weakG[(size_t)p * g.Vh + h] = (unsigned char)(marks >> 6);
  if (marks && (threadIdx.x & 31) == 0) atomicOr(any, (marks & 63 ? 1 : 0) | (marks >> 6 ? 2 : 0));
}

// Canonical sites are 12 consecutive complex128.  Reading them site by site is fine (a site's lines stay in
// L1 between its 12 loads), but a site's store instruction touches half of 32 sectors, so the way back moves a
// block's sites through shared memory and its lanes write consecutive 16-byte words: 32^3 x 64, 8 RHS, FP16
// to canonical 1037 -> 300 us, the time its bytes take (reads staged the same way: 328 -> 410 us).  Sites in
// shared memory are 13 words apart, so that eight lanes' 16-byte accesses hit distinct banks.  Three threads
// share a site, four components each (four threads, to block fixed point: two a chiral block): the conversions of
// block fixed point, some 25 instructions a number, are long chains on a small lattice (4^3 x 8, one thread per
// site: 10.7 us to canonical, 5.7 us from it; three: 5.9 and 4.8 us).
constexpr int LB = 128;         // sites of a block
constexpr int SITE_WORDS = 13;  // double2 words between sites in shared memory

template <int P>
__global__ void __launch_bounds__(3 * LB) spinor_to_native_kernel(Geom g, const double2* __restrict__ canon, void* nat,
                                                                  float* norm, int nrhs) {
  const int site = threadIdx.x % LB, part = threadIdx.x / LB;
  const int tid = blockIdx.x * LB + site;
  const bool valid = tid < g.Vh * nrhs;
  const int r = tid / g.Vh, h = tid - r * g.Vh;
  double2 v[4] = {};
  if (valid) {
    const double2* src = canon + (size_t)tid * 12 + 4 * part;
#pragma unroll
    for (int c = 0; c < 4; c++) v[c] = __ldg(src + c);
  }
  if constexpr (P == 64) {
    if (!valid || !dbg_spinor(g.Vh, r, h)) return;
#pragma unroll
    for (int c = 0; c < 4; c++) static_cast<double2*>(nat)[sidx<12>(4 * part + c, g.Vh, r, h)] = v[c];
  } else {
    // one branch for a thread's conversions: with one in each of them, loads wait behind the branches before them
    // (4^3 x 8, Mdag M in FP32, one thread per site and 24 branches: 26.8 us a pass; so 24.7)
    float2 f[4];
    bool common = true;
#pragma unroll
    for (int c = 0; c < 4; c++) common = common && narrow_common(v[c].x) && narrow_common(v[c].y);
    if (common) {
#pragma unroll
      for (int c = 0; c < 4; c++) f[c] = make_float2(narrow_of_common(v[c].x), narrow_of_common(v[c].y));
    } else {
#pragma unroll
      for (int c = 0; c < 4; c++) f[c] = make_float2(narrow_rare(v[c].x), narrow_rare(v[c].y));
    }
    if constexpr (P == 32) {
      if (!valid || !dbg_spinor(g.Vh, r, h)) return;
#pragma unroll
      for (int k = 0; k < 2; k++)
        static_cast<float4*>(nat)[sidx<6>(2 * part + k, g.Vh, r, h)] =
            make_float4(f[2 * k].x, f[2 * k].y, f[2 * k + 1].x, f[2 * k + 1].y);
    } else {
      __shared__ float sm[3][LB];
      float m = 0.f;
#pragma unroll
      for (int c = 0; c < 4; c++) m = fmaxf(m, fmaxf(fabsf(f[c].x), fabsf(f[c].y)));
      sm[part][site] = m;
      __syncthreads();
      if (!valid || !dbg_spinor(g.Vh, r, h)) return;
      m = fmaxf(sm[0][site], fmaxf(sm[1][site], sm[2][site]));
      const float inv = m > 0.f ? 1.0f / m : 0.f;
      static_cast<uint4*>(nat)[sidx<3>(part, g.Vh, r, h)] =
          make_uint4(f2h(f[0].x * inv, f[0].y * inv), f2h(f[1].x * inv, f[1].y * inv), f2h(f[2].x * inv, f[2].y * inv),
                     f2h(f[3].x * inv, f[3].y * inv));
      if (part == 0) norm[(size_t)r * g.Vh + h] = m;
    }
  }
}

// the same to block fixed point
__global__ void __launch_bounds__(4 * LB) spinor_to_fixed_kernel(Geom g, const double2* __restrict__ canon, longlong2* nat,
                                                                 int* ex, int nrhs) {
  __shared__ u64 sm[4][LB];
  const int site = threadIdx.x % LB, part = threadIdx.x / LB;
  const int tid = blockIdx.x * LB + site;  // (eight right-hand sides at most: below 2^31)
  const bool valid = tid < g.Vh * nrhs;
  const int r = tid / g.Vh, h = tid - r * g.Vh;
  double2 v[3];
  u64 mx = 0;
  if (valid) {
    const double2* src = canon + (size_t)tid * 12 + 3 * part;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      v[c] = src[c];
      mx = max(mx, max(fx_mag(v[c].x), fx_mag(v[c].y)));
    }
  }
  sm[part][site] = mx;
  __syncthreads();
  if (!valid || !dbg_spinor(g.Vh, r, h)) return;
  const int e = fx_exponent(max(mx, sm[part ^ 1][site]));
#pragma unroll
  for (int c = 0; c < 3; c++)
    nat[sidx<12>(3 * part + c, g.Vh, r, h)] =
        make_longlong2(fx_of_double<FX_SPINOR>(v[c].x, e), fx_of_double<FX_SPINOR>(v[c].y, e));
  if ((part & 1) == 0) ex[eidx(part >> 1, g.Vh, r, h)] = e;
}

// components 4 part .. 4 part + 3 of a site as doubles
template <int P>
__device__ __forceinline__ void load_part(const void* nat, const float* norm, int Vh, int r, int h, int part, double2 o[4]) {
  if (!dbg_spinor(Vh, r, h)) {
    for (int c = 0; c < 4; c++) o[c] = {};
    return;
  }
  if constexpr (P == 60) {
    const longlong2* p = static_cast<const longlong2*>(nat);
    // components 0-5 are those of block 0: part 1 holds two of each block
    const int* ex = reinterpret_cast<const int*>(norm);
    const int e0 = __ldg(ex + eidx(part == 2, Vh, r, h)), e1 = __ldg(ex + eidx(part > 0, Vh, r, h));
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const longlong2 v = __ldg(p + sidx<12>(4 * part + c, Vh, r, h));
      const int e = c < 2 ? e0 : e1;
      o[c] = make_double2(fx_to_double(v.x, e, FX_SPINOR), fx_to_double(v.y, e, FX_SPINOR));
    }
  } else if constexpr (P == 64) {
    const double2* p = static_cast<const double2*>(nat);
#pragma unroll
    for (int c = 0; c < 4; c++) o[c] = __ldg(p + sidx<12>(4 * part + c, Vh, r, h));
  } else if constexpr (P == 32) {
    const float4* p = static_cast<const float4*>(nat);
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const float4 v = __ldg(p + sidx<6>(2 * part + k, Vh, r, h));
      o[2 * k] = make_double2(widen(v.x), widen(v.y));
      o[2 * k + 1] = make_double2(widen(v.z), widen(v.w));
    }
  } else {
    const float n = __ldg(norm + (size_t)r * Vh + h);
    const uint4 v = __ldg(static_cast<const uint4*>(nat) + sidx<3>(part, Vh, r, h));
    const float2 a = h2f(v.x), b = h2f(v.y), c = h2f(v.z), d = h2f(v.w);
    o[0] = make_double2(widen(a.x * n), widen(a.y * n));
    o[1] = make_double2(widen(b.x * n), widen(b.y * n));
    o[2] = make_double2(widen(c.x * n), widen(c.y * n));
    o[3] = make_double2(widen(d.x * n), widen(d.y * n));
  }
}

template <int P>
__global__ void __launch_bounds__(3 * LB) spinor_to_canon_kernel(Geom g, const void* nat, const float* norm,
                                                                 double2* canon, int nrhs) {
  __shared__ double2 buf[LB * SITE_WORDS];
  const long long first = (long long)blockIdx.x * LB, n = (long long)g.Vh * nrhs;
  const int here = (int)min((long long)LB, n - first);
  const int mine = threadIdx.x % LB, part = threadIdx.x / LB;
  if (mine < here) {
    const int tid = (int)first + mine, r = tid / g.Vh, h = tid - r * g.Vh;
    double2 o[4];
    load_part<P>(nat, norm, g.Vh, r, h, part, o);
#pragma unroll
    for (int c = 0; c < 4; c++) buf[mine * SITE_WORDS + 4 * part + c] = o[c];
  }
  __syncthreads();
  double2* dst = canon + first * 12;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int j = k * 3 * LB + threadIdx.x, site = j / 12;
    if (site < here) dst[j] = buf[site * SITE_WORDS + (j - 12 * site)];
  }
}

__global__ void check_finite_kernel(const double* __restrict__ d, size_t n, int* flag) {
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  bool bad = false;
  for (; i < n; i += stride) bad |= !isfinite(d[i]);
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) *flag = 1;
}

inline int nblocks(long long n, int b) { return (int)((n + b - 1) / b); }

}  // namespace

void launch_pack_gauge(const Geom& g, const double2* canon, void* g64, void* g32, int recon32, void* g16,
                       int recon16, void* gfx, unsigned char* far, int* not_unitary, int* non_finite, cudaStream_t st) {
  g_kernel_launches += 1;
  const int B = 128;
  pack_gauge_kernel<<<nblocks(8LL * g.Vh, B), B, 0, st>>>(g, canon, static_cast<double2*>(g64), g32, recon32, g16,
                                                          recon16, static_cast<int4*>(gfx), far, not_unitary,
                                                          non_finite);
}

void launch_weak_sites(const Geom& g, const unsigned char* far, unsigned char* weakF, unsigned char* weakG, int* any,
                       cudaStream_t st) {
  g_kernel_launches += 1;
  weak_sites_kernel<<<nblocks(2 * ((g.Vh + 31) / 32), 4), 128, 0, st>>>(g, far, weakF, weakG, any);
}

void launch_spinor_to_native(int prec, const Geom& g, const double2* canon, void* nat, float* norm, int nrhs,
                             cudaStream_t st) {
  g_kernel_launches += 1;
  const int B = 3 * LB;
  const int nb = nblocks((long long)g.Vh * nrhs, LB);
  if (prec == 60)
    spinor_to_fixed_kernel<<<nb, 4 * LB, 0, st>>>(
        g, canon, static_cast<longlong2*>(nat), reinterpret_cast<int*>(norm), nrhs);
  else if (prec == 64) spinor_to_native_kernel<64><<<nb, B, 0, st>>>(g, canon, nat, norm, nrhs);
  else if (prec == 32) spinor_to_native_kernel<32><<<nb, B, 0, st>>>(g, canon, nat, norm, nrhs);
  else spinor_to_native_kernel<16><<<nb, B, 0, st>>>(g, canon, nat, norm, nrhs);
}

void launch_spinor_to_canon(int prec, const Geom& g, const void* nat, const float* norm, double2* canon, int nrhs,
                            cudaStream_t st) {
  g_kernel_launches += 1;
  const int B = 3 * LB;
  const int nb = nblocks((long long)g.Vh * nrhs, LB);
  if (prec == 60) spinor_to_canon_kernel<60><<<nb, B, 0, st>>>(g, nat, norm, canon, nrhs);
  else if (prec == 64) spinor_to_canon_kernel<64><<<nb, B, 0, st>>>(g, nat, norm, canon, nrhs);
  else if (prec == 32) spinor_to_canon_kernel<32><<<nb, B, 0, st>>>(g, nat, norm, canon, nrhs);
  else spinor_to_canon_kernel<16><<<nb, B, 0, st>>>(g, nat, norm, canon, nrhs);
}

void launch_check_finite(const double* data, size_t n, int* flag, cudaStream_t st) {
  if (n > 0) g_kernel_launches += 1;
  if (n == 0) return;
  const int B = 256;
  long long nb = (long long)((n + B - 1) / B);
  if (nb > 152 * 16) nb = 152 * 16;
  check_finite_kernel<<<(int)nb, B, 0, st>>>(data, n, flag);
}

void launch_zero(void* ptr, size_t bytes, cudaStream_t st) {
  if (bytes) cudaMemsetAsync(ptr, 0, bytes, st);
}

}  // namespace qcd
