// Device building blocks of the Wilson-Dirac stencil (the operator D of Eq. 1), shared by
// the single- and multi-right-hand-side kernels: site loads/stores of every storage type,
// link loads in both layouts, the spin projections (1 -/+ gamma_mu) of the chiral basis,
// colour transport by U or U^dag, reconstruction, and one hop in each direction.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "vec.cuh"

namespace wmg {
namespace stencil {

// 32-byte global accesses (sm_100 and later).  volatile: they stay behind the dependent-launch
// wait of dep_entry() in program order.
__device__ __forceinline__ void ld32(const void* p, float v[8]) {
  asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]),
                 "=f"(v[6]), "=f"(v[7])
               : "l"(p));
}
__device__ __forceinline__ void st32(void* p, const float v[8]) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]),
               "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void ld32(const void* p, double v[4]) {
  asm volatile("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
               : "l"(p));
}
__device__ __forceinline__ void st32(void* p, const double v[4]) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]),
               "d"(v[2]), "d"(v[3])
               : "memory");
}

// Loads/stores of one site's 12 complex numbers (complex float: 96 bytes, complex double: 192).
// Consecutive threads take consecutive sites, so a 16-byte load of a warp touches 32 half-used
// sectors in 24 lines, and the stencil is bound by the L1's passes over them (80 % busy, DRAM
// 41 %, ncu at 24^3x48).  32-byte accesses use every sector they touch: 201 -> 161 us per FP32
// stencil at 32^3x64 (two-row links), 256 -> 208 us with ABI links.  They need 32-byte aligned
// fields; StC64N / StC128N are the 16-byte forms for fields that are only 16-byte aligned.
template <typename S> struct SiteIO;

template <typename S> struct SiteIO32 {
  typedef typename S::real R;
  static constexpr int N = 32 / sizeof(R);        // reals per access
  static __device__ __forceinline__ void load(const typename S::elem* p, size_t site,
                                              cplx<R> v[12]) {
    const char* q = reinterpret_cast<const char*>(p + site * 12);
#pragma unroll
    for (int i = 0; i < 24 / N; ++i) {
      R t[N];
      ld32(q + 32 * i, t);
#pragma unroll
      for (int j = 0; j < N / 2; ++j) v[i * (N / 2) + j] = {t[2 * j], t[2 * j + 1]};
    }
  }
  static __device__ __forceinline__ void store(typename S::elem* p, size_t site,
                                               const cplx<R> v[12]) {
    char* q = reinterpret_cast<char*>(p + site * 12);
#pragma unroll
    for (int i = 0; i < 24 / N; ++i) {
      R t[N];
#pragma unroll
      for (int j = 0; j < N / 2; ++j) {
        t[2 * j] = v[i * (N / 2) + j].re;
        t[2 * j + 1] = v[i * (N / 2) + j].im;
      }
      st32(q + 32 * i, t);
    }
  }
};
template <> struct SiteIO<StC128> : SiteIO32<StC128> {};
template <> struct SiteIO<StC64> : SiteIO32<StC64> {};

// 16-byte forms
struct StC128N : StC128 {};
struct StC64N : StC64 {};
template <> struct SiteIO<StC128N> {
  static __device__ __forceinline__ void load(const double2* p, size_t site, zd v[12]) {
    const double2* q = p + site * 12;
#pragma unroll
    for (int i = 0; i < 12; ++i) { double2 t = __ldg(q + i); v[i] = {t.x, t.y}; }
  }
  static __device__ __forceinline__ void store(double2* p, size_t site, const zd v[12]) {
    double2* q = p + site * 12;
#pragma unroll
    for (int i = 0; i < 12; ++i) q[i] = make_double2(v[i].re, v[i].im);
  }
};
template <> struct SiteIO<StC64N> {
  static __device__ __forceinline__ void load(const float2* p, size_t site, zf v[12]) {
    const float4* q = reinterpret_cast<const float4*>(p + site * 12);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      float4 t = __ldg(q + i);
      v[2 * i] = {t.x, t.y};
      v[2 * i + 1] = {t.z, t.w};
    }
  }
  static __device__ __forceinline__ void store(float2* p, size_t site, const zf v[12]) {
    float4* q = reinterpret_cast<float4*>(p + site * 12);
#pragma unroll
    for (int i = 0; i < 6; ++i)
      q[i] = make_float4(v[2 * i].re, v[2 * i].im, v[2 * i + 1].re, v[2 * i + 1].im);
  }
};
template <typename H, typename S> struct SiteIOHalf {
  static __device__ __forceinline__ void load(const H* p, size_t site, zf v[12]) {
    const uint4* q = reinterpret_cast<const uint4*>(p + site * 12);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      uint4 t = __ldg(q + i);
      const H* h = reinterpret_cast<const H*>(&t);
#pragma unroll
      for (int j = 0; j < 4; ++j) v[4 * i + j] = S::ld(h, j);
    }
  }
  static __device__ __forceinline__ void store(H* p, size_t site, const zf v[12]) {
    uint4* q = reinterpret_cast<uint4*>(p + site * 12);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      uint4 t;
      H* h = reinterpret_cast<H*>(&t);
#pragma unroll
      for (int j = 0; j < 4; ++j) S::st(h, j, v[4 * i + j]);
      q[i] = t;
    }
  }
};
template <> struct SiteIO<StF16> : SiteIOHalf<__half2, StF16> {};
template <> struct SiteIO<StBF16> : SiteIOHalf<__nv_bfloat162, StBF16> {};

// Load the 3x3 link U_mu(site).  LL = 0: ABI layout [mu][site][3][3] (one link contiguous);
// LL = 1: lane-contiguous layout [mu][3x3 entry][site], so a warp reading one entry for 32
// consecutive sites touches one contiguous 32 x element_size span (the solver's copy);
// LL = 2: the same with the first two rows only, [mu][6 entry][site]: for U in SU(3) the rows
// are orthonormal and det U = 1, so the third row is the complex conjugate of the cross
// product of the first two (12 of the 18 reals cross HBM);
// LL = 3: ABI layout of 4- or 8-byte elements with a 16-byte aligned base: the aligned 16-byte
// pieces that cover the link (5 of a 72-byte link that starts at 0 or 8 mod 16, 3 of a 36-byte
// link that starts at 0, 4, 8 or 12 mod 16) instead of nine element loads, then a select by the
// offset (208 -> 205 us at 32^3x64 in FP32, 18.4 -> 16.5 us at 16^3x32).  The window never
// leaves the array: 4 V is a multiple of 4, so the first link starts and the last one ends on a
// 16-byte boundary.
template <typename S, int LL>
__device__ __forceinline__ void load_link(const typename S::elem* L, int V, int mu, int site,
                                          cplx<typename S::real> u[9]) {
  if constexpr (LL == 0) {
    size_t idx = ((size_t)mu * V + site) * 9;
#pragma unroll
    for (int i = 0; i < 9; ++i) u[i] = S::ld(L, idx + i);
  } else if constexpr (LL == 1) {
#pragma unroll
    for (int i = 0; i < 9; ++i) u[i] = S::ld(L, ((size_t)mu * 9 + i) * V + site);
  } else if constexpr (LL == 2) {
#pragma unroll
    for (int i = 0; i < 6; ++i) u[i] = S::ld(L, ((size_t)mu * 6 + i) * V + site);
    u[6] = conj(u[1] * u[5] - u[2] * u[4]);
    u[7] = conj(u[2] * u[3] - u[0] * u[5]);
    u[8] = conj(u[0] * u[4] - u[1] * u[3]);
  } else if constexpr (sizeof(typename S::elem) == 8) {
    const size_t e0 = ((size_t)mu * V + site) * 9;   // first element of the link
    const bool odd = (e0 & 1) != 0;
    const float4* q = reinterpret_cast<const float4*>(L) + (e0 >> 1);
    float w[20];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      float4 t = __ldg(q + i);
      w[4 * i] = t.x; w[4 * i + 1] = t.y; w[4 * i + 2] = t.z; w[4 * i + 3] = t.w;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i)
      u[i] = {odd ? w[2 * i + 2] : w[2 * i], odd ? w[2 * i + 3] : w[2 * i + 1]};
  } else {
    const size_t e0 = ((size_t)mu * V + site) * 9;
    const int off = (int)(e0 & 3);
    const uint4* q = reinterpret_cast<const uint4*>(L) + (e0 >> 2);
    unsigned w[12], x[11];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      uint4 t = __ldg(q + i);
      w[4 * i] = t.x; w[4 * i + 1] = t.y; w[4 * i + 2] = t.z; w[4 * i + 3] = t.w;
    }
    // shift by off = 2 b1 + b0 elements
#pragma unroll
    for (int i = 0; i < 11; ++i) x[i] = (off & 1) ? w[i + 1] : w[i];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      typename S::elem h;
      const unsigned v = (off & 2) ? x[i + 2] : x[i];
      memcpy(&h, &v, 4);
      u[i] = S::ld(&h, 0);
    }
  }
}

// Project psi with (1 + s gamma_mu) to the upper spin pair h (2 spins x 3 colours).
// mu = 0,1,2: h = psi_up - s i sigma_mu psi_dn; mu = 3: h = psi_up + s psi_dn.
template <int MU, int SGN, typename R>
__device__ __forceinline__ void project(const cplx<R> p[12], cplx<R> h[6]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    cplx<R> u0 = p[0 * 3 + c], u1 = p[1 * 3 + c], d0 = p[2 * 3 + c], d1 = p[3 * 3 + c];
    cplx<R> a, b;  // i sigma psi_dn, components 0 and 1
    if (MU == 0) { a = ti(d1); b = ti(d0); }
    else if (MU == 1) { a = d1; b = -d0; }
    else if (MU == 2) { a = ti(d0); b = tmi(d1); }
    else { a = d0; b = d1; }
    if (MU < 3) {
      if (SGN > 0) { h[c] = u0 - a; h[3 + c] = u1 - b; }
      else { h[c] = u0 + a; h[3 + c] = u1 + b; }
    } else {
      if (SGN > 0) { h[c] = u0 + a; h[3 + c] = u1 + b; }
      else { h[c] = u0 - a; h[3 + c] = u1 - b; }
    }
  }
}

// acc += c (1 + s gamma_mu) reconstructed from the transported half spinor g:
// upper = g; lower = s i sigma_mu g (mu < 3) or s g (mu = 3).  The hop's coefficient c (weight
// and boundary phase) rides on the multiply-adds: scaling the half spinor first would be 12
// multiplications more per hop (a tenth of the FP64 stencil's instructions).
template <int MU, int SGN, typename R>
__device__ __forceinline__ void accumulate(cplx<R> acc[12], const cplx<R> g[6], R c) {
  const R cs = SGN > 0 ? c : -c;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cplx<R> g0 = g[i], g1 = g[3 + i];
    cplx<R> a, b;  // i sigma g or g
    if (MU == 0) { a = ti(g1); b = ti(g0); }
    else if (MU == 1) { a = g1; b = -g0; }
    else if (MU == 2) { a = ti(g0); b = tmi(g1); }
    else { a = g0; b = g1; }
    acc[i].re = fma(c, g0.re, acc[i].re);
    acc[i].im = fma(c, g0.im, acc[i].im);
    acc[3 + i].re = fma(c, g1.re, acc[3 + i].re);
    acc[3 + i].im = fma(c, g1.im, acc[3 + i].im);
    acc[6 + i].re = fma(cs, a.re, acc[6 + i].re);
    acc[6 + i].im = fma(cs, a.im, acc[6 + i].im);
    acc[9 + i].re = fma(cs, b.re, acc[9 + i].re);
    acc[9 + i].im = fma(cs, b.im, acc[9 + i].im);
  }
}

template <typename R>
__device__ __forceinline__ void mul_link(const cplx<R> u[9], const cplx<R> h[6], cplx<R> g[6]) {
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      cplx<R> t = u[a * 3 + 0] * h[s * 3 + 0];
      cfma(t, u[a * 3 + 1], h[s * 3 + 1]);
      cfma(t, u[a * 3 + 2], h[s * 3 + 2]);
      g[s * 3 + a] = t;
    }
}
template <typename R>
__device__ __forceinline__ void mul_link_dag(const cplx<R> u[9], const cplx<R> h[6], cplx<R> g[6]) {
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      cplx<R> t = {0, 0};
      cfmac(t, u[0 * 3 + a], h[s * 3 + 0]);
      cfmac(t, u[1 * 3 + a], h[s * 3 + 1]);
      cfmac(t, u[2 * 3 + a], h[s * 3 + 2]);
      g[s * 3 + a] = t;
    }
}

// Sites of a CTA.  Off: consecutive sites.  On: a tile of t0 x t1 x t2 x t3 sites (t0 in half
// sites for a single-parity stencil), so that neighbours in y, z and t come from the CTA's own
// L1 lines more often: the L2 -> L1 traffic of a 128-site tile of a 16^3x32 lattice is 4 spinors
// per site instead of 5-6 (18.6 -> 18.0 us cold, 14.5 -> 12.5 us warm per FP32 stencil there,
// 164 -> 162 us at 32^3x64).  Chosen on the host by pick_tile.
struct TileMap {
  int on = 0;
  int sites = 0;          // t0 t1 t2 t3
  int t[4];               // tile extents
  int n[3];               // tiles along the first three axes
  unsigned tm[3], nm[3];  // reciprocals of t[0..2] (16 bit) and n[0..2] (32 bit, 0 for 1)
};

struct KGeom {
  int L[4];
  int stride[4];
  int V;
  float wf[4];
  double wd[4];
  int bc[4];
  double kappa;
  float kf;      // kappa in FP32: one FP64 conversion per thread would cost each warp 16 cycles
  bool unit;     // all four hop weights are 1
  // single-parity form only: when set, out_p = sub_p - (-kappa H_{p,1-p} in) (the even-odd
  // Schur complement and its source / reconstruction steps), sub with out's layout and stride
  const void* sub = nullptr;
  TileMap tile;
};

// res <- sub[rhs][i] - res for the single-parity form with a subtrahend field
template <typename S>
__device__ __forceinline__ void apply_sub(const KGeom& g, size_t rhs_off, int i,
                                          cplx<typename S::real> res[12]);

template <typename R> __device__ __forceinline__ R kap(const KGeom& g);
template <> __device__ __forceinline__ double kap<double>(const KGeom& g) { return g.kappa; }
template <> __device__ __forceinline__ float kap<float>(const KGeom& g) { return g.kf; }
template <typename R> __device__ __forceinline__ R wgt(const KGeom& g, int mu);
template <> __device__ __forceinline__ double wgt<double>(const KGeom& g, int mu) { return g.wd[mu]; }
template <> __device__ __forceinline__ float wgt<float>(const KGeom& g, int mu) { return g.wf[mu]; }

// forward hop of direction MU: (1 + SF gamma) U_mu(x) psi(x + mu)
template <int MU, int DAG, typename S, int LL>
__device__ __forceinline__ void hop_fwd(const KGeom& g, int site, const int c[4],
                                        const typename S::elem* in, size_t in_off,
                                        bool half_in, const typename S::elem* links,
                                        cplx<typename S::real> acc[12]) {
  typedef typename S::real R;
  constexpr int SF = DAG ? +1 : -1;  // forward projector sign
  R w = wgt<R>(g, MU);
  int nb = (c[MU] == g.L[MU] - 1) ? site - (g.L[MU] - 1) * g.stride[MU] : site + g.stride[MU];
  R cf = (c[MU] == g.L[MU] - 1 && g.bc[MU] < 0) ? -w : w;
  cplx<R> p[12], h[6], gg[6], u[9];
  SiteIO<S>::load(in + in_off, half_in ? (size_t)(nb >> 1) : (size_t)nb, p);
  project<MU, SF, R>(p, h);
  load_link<S, LL>(links, g.V, MU, site, u);
  mul_link<R>(u, h, gg);
  accumulate<MU, SF, R>(acc, gg, cf);
}

// backward hop of direction MU: (1 + SB gamma) U_mu(x - mu)^dag psi(x - mu)
template <int MU, int DAG, typename S, int LL>
__device__ __forceinline__ void hop_bwd(const KGeom& g, int site, const int c[4],
                                        const typename S::elem* in, size_t in_off,
                                        bool half_in, const typename S::elem* links,
                                        cplx<typename S::real> acc[12]) {
  typedef typename S::real R;
  constexpr int SB = DAG ? -1 : +1;  // backward projector sign
  R w = wgt<R>(g, MU);
  int nb = (c[MU] == 0) ? site + (g.L[MU] - 1) * g.stride[MU] : site - g.stride[MU];
  R cf = (c[MU] == 0 && g.bc[MU] < 0) ? -w : w;
  cplx<R> p[12], h[6], gg[6], u[9];
  SiteIO<S>::load(in + in_off, half_in ? (size_t)(nb >> 1) : (size_t)nb, p);
  project<MU, SB, R>(p, h);
  load_link<S, LL>(links, g.V, MU, nb, u);
  mul_link_dag<R>(u, h, gg);
  accumulate<MU, SB, R>(acc, gg, cf);
}

template <int MU, int DAG, typename S, int LL>
__device__ __forceinline__ void hop_pair(const KGeom& g, int site, const int c[4],
                                         const typename S::elem* in, size_t in_off,
                                         bool half_in, const typename S::elem* links,
                                         cplx<typename S::real> acc[12]) {
  hop_fwd<MU, DAG, S, LL>(g, site, c, in, in_off, half_in, links, acc);
  hop_bwd<MU, DAG, S, LL>(g, site, c, in, in_off, half_in, links, acc);
}

// ---- one thread per site and hop
// For lattices that leave the chip idle with a thread per site (4^4: two CTAs; 8^4: 32) the chain
// of eight dependent hops is the launch: FP64 on 4^4 17.8 us, of which the launch itself is a
// few (7.7 us in this form).  Here eight lanes share a site, lane `hop` takes direction hop / 2 (forward when even) with
// the spin projector's phases as operands, and the 12 sums are reduced and scattered over the
// lanes: every pair of lanes ends with the three colours of one spin.

// -x where `neg`, off the FP64 pipe
__device__ __forceinline__ float flip(float x, bool neg) {
  return __uint_as_float(__float_as_uint(x) ^ (neg ? 0x80000000u : 0u));
}
__device__ __forceinline__ double flip(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000u : 0), __double2loint(x));
}

// The two components of i sigma_mu d for mu < 3, d for mu = 3, are d[w], d[1 - w] (w = 1 for mu <
// 2) times one unit, i for even mu and 1 for odd, the second negated for mu = 1 and 2.  The unit is
// applied by exchanging real and imaginary parts and flipping signs, not by multiplying with it: an
// infinite component does not turn its neighbours into NaN, and FP64 multiply-adds, the bound of a
// filled chip, are left to the products and sums (8192 sites: 24.1 -> 18.6 us).
template <typename R>
struct HopPhase {
  bool swap, imag, neg1;        // neg1: the second component's sign
  // component c of the result, from d = its d[w] or d[1 - w], negated where `neg`
  __device__ __forceinline__ cplx<R> turn(cplx<R> d, int c, bool neg) const {
    const bool n = neg != (c && neg1);
    return {flip(imag ? d.im : d.re, n != imag), flip(imag ? d.re : d.im, n)};
  }
};
template <typename R>
__device__ __forceinline__ HopPhase<R> hop_phase(int mu) {
  return {mu < 2, (mu & 1) == 0, mu == 1 || mu == 2};
}

// The hop's term of H psi at `site`, reduced over the site's eight lanes: out = components 3 sp ..
// 3 sp + 2 of sum_mu w_mu [...], sp = hop >> 1.  All 32 lanes call it; inactive sites pass active =
// false and get zeros.
template <int DAG, typename S, int LL>
__device__ __forceinline__ void hop_lanes(const KGeom& g, bool active, int site, const int c[4],
                                          int hop, const typename S::elem* in, bool half_in,
                                          const typename S::elem* links,
                                          cplx<typename S::real> out[3]) {
  typedef typename S::real R;
  const int mu = hop >> 1;
  const bool fwd = (hop & 1) == 0;
  cplx<R> gg[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) gg[i] = {0, 0};
  const HopPhase<R> f = hop_phase<R>(mu);
  const bool neg = fwd != (DAG != 0);   // projector sign
  R w = 0;
  bool cneg = false;                    // coefficient: w, negated at an antiperiodic boundary
  if (active) {
    const int L = mu == 0 ? g.L[0] : mu == 1 ? g.L[1] : mu == 2 ? g.L[2] : g.L[3];
    const int st = mu == 0 ? g.stride[0] : mu == 1 ? g.stride[1] : mu == 2 ? g.stride[2] : g.stride[3];
    const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
    const int bc = mu == 0 ? g.bc[0] : mu == 1 ? g.bc[1] : mu == 2 ? g.bc[2] : g.bc[3];
    w = mu == 0 ? wgt<R>(g, 0) : mu == 1 ? wgt<R>(g, 1) : mu == 2 ? wgt<R>(g, 2) : wgt<R>(g, 3);
    const bool wrap = fwd ? cm == L - 1 : cm == 0;
    const int step = wrap ? -(L - 1) * st : st;
    const int nb = fwd ? site + step : site - step;
    cneg = wrap && bc < 0;
    cplx<R> p[12], u[9], h[6];
    SiteIO<S>::load(in, half_in ? (size_t)(nb >> 1) : (size_t)nb, p);
    load_link<S, LL>(links, g.V, mu, fwd ? site : nb, u);
    // h = psi_up - s i sigma psi_dn (mu < 3), psi_up + s psi_dn (mu = 3)
    const bool np = neg != (mu < 3);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const cplx<R> d0 = f.swap ? p[9 + k] : p[6 + k], d1 = f.swap ? p[6 + k] : p[9 + k];
      h[k] = p[k] + f.turn(d0, 0, np);
      h[3 + k] = p[3 + k] + f.turn(d1, 1, np);
    }
    // U h or U^dag h
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      cplx<R> t0 = {0, 0}, t1 = {0, 0};
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const cplx<R> q = fwd ? u[a * 3 + b] : u[b * 3 + a];
        const cplx<R> m = {q.re, flip(q.im, !fwd)};
        cfma(t0, m, h[b]);
        cfma(t1, m, h[3 + b]);
      }
      gg[a] = t0;
      gg[3 + a] = t1;
    }
  }
  // unit weights (uniform over the launch) need no multiplications
  if (!g.unit) {
#pragma unroll
    for (int k = 0; k < 6; ++k) gg[k] = w * gg[k];
  }
  // upper pair g, lower pair s i sigma g (s g): lanes 0-3 keep the upper, 4-7 the lower
  const bool low = (hop & 4) != 0;
  cplx<R> keep[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const cplx<R> g0 = f.swap ? gg[3 + k] : gg[k], g1 = f.swap ? gg[k] : gg[3 + k];
    const cplx<R> up0 = {flip(gg[k].re, cneg), flip(gg[k].im, cneg)};
    const cplx<R> up1 = {flip(gg[3 + k].re, cneg), flip(gg[3 + k].im, cneg)};
    const cplx<R> lo0 = f.turn(g0, 0, cneg != neg), lo1 = f.turn(g1, 1, cneg != neg);
    const cplx<R> s0 = low ? up0 : lo0, s1 = low ? up1 : lo1;
    keep[k] = low ? lo0 : up0;
    keep[3 + k] = low ? lo1 : up1;
    keep[k].re += __shfl_xor_sync(0xffffffffu, s0.re, 4);
    keep[k].im += __shfl_xor_sync(0xffffffffu, s0.im, 4);
    keep[3 + k].re += __shfl_xor_sync(0xffffffffu, s1.re, 4);
    keep[3 + k].im += __shfl_xor_sync(0xffffffffu, s1.im, 4);
  }
  const bool odd = (hop & 2) != 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const cplx<R> send = odd ? keep[k] : keep[3 + k];
    cplx<R> t = odd ? keep[3 + k] : keep[k];
    t.re += __shfl_xor_sync(0xffffffffu, send.re, 2);
    t.im += __shfl_xor_sync(0xffffffffu, send.im, 2);
    t.re += __shfl_xor_sync(0xffffffffu, t.re, 1);
    t.im += __shfl_xor_sync(0xffffffffu, t.im, 1);
    out[k] = t;
  }
}

// Site index of thread i (parity < 0: lexicographic; else the i-th site of that parity)
// and its coordinates.
__device__ __forceinline__ int stencil_site(const KGeom& g, int parity, int i, int c[4]) {
  int site;
  if (parity < 0) {
    site = i;
  } else {
    int s0 = 2 * i;
    int x0 = s0 % g.L[0];
    int rest = s0 / g.L[0];
    int y = rest % g.L[1];
    int z = (rest / g.L[1]) % g.L[2];
    int t = rest / (g.L[1] * g.L[2]);
    site = s0 + (((x0 + y + z + t) & 1) != parity ? 1 : 0);
  }
  c[0] = site % g.L[0];
  int rest = site / g.L[0];
  c[1] = rest % g.L[1];
  rest /= g.L[1];
  c[2] = rest % g.L[2];
  c[3] = rest / g.L[2];
  return site;
}

// Work item of thread `u` (of `per` sites per CTA) in CTA blockIdx.x: output index i (the site,
// or the checkerboard index of a single-parity stencil), lattice site and coordinates; false when
// there is none.
__device__ __forceinline__ bool stencil_work(const KGeom& g, int parity, int nsites, int u, int per,
                                             int& i, int& site, int c[4]) {
  const TileMap& m = g.tile;
  if (!m.on) {
    i = blockIdx.x * per + u;
    if (i >= nsites) return false;
    site = stencil_site(g, parity, i, c);
    return true;
  }
  if (u >= m.sites) return false;
  unsigned r = (unsigned)u, b = blockIdx.x;
  int x[4];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const unsigned q = (r * m.tm[a]) >> 16;
    const unsigned bq = m.nm[a] ? __umulhi(b, m.nm[a]) : b;
    x[a] = (int)(b - bq * m.n[a]) * m.t[a] + (int)(r - q * m.t[a]);
    r = q;
    b = bq;
  }
  x[3] = (int)b * m.t[3] + (int)r;
  const int row = x[1] + g.L[1] * (x[2] + g.L[2] * x[3]);
  c[0] = parity < 0 ? x[0] : 2 * x[0] + ((x[1] + x[2] + x[3] + parity) & 1);
  c[1] = x[1];
  c[2] = x[2];
  c[3] = x[3];
  site = c[0] + g.L[0] * row;
  i = parity < 0 ? site : site >> 1;
  return true;
}

template <typename S>
__device__ __forceinline__ void apply_sub(const KGeom& g, size_t rhs_off, int i,
                                          cplx<typename S::real> res[12]) {
  if (!g.sub) return;
  cplx<typename S::real> b[12];
  SiteIO<S>::load(static_cast<const typename S::elem*>(g.sub) + rhs_off, (size_t)i, b);
#pragma unroll
  for (int k = 0; k < 12; ++k) res[k] = b[k] - res[k];
}

inline KGeom to_kgeom(const Geom& g) {
  KGeom k;
  k.unit = true;
  for (int m = 0; m < 4; ++m) {
    k.unit = k.unit && g.w[m] == 1.0;
    k.L[m] = g.L[m];
    k.wf[m] = (float)g.w[m];
    k.wd[m] = g.w[m];
    k.bc[m] = g.bc[m];
  }
  k.stride[0] = 1;
  k.stride[1] = g.L[0];
  k.stride[2] = g.L[0] * g.L[1];
  k.stride[3] = g.L[0] * g.L[1] * g.L[2];
  k.V = g.V;
  k.kappa = g.kappa;
  k.kf = (float)g.kappa;
  return k;
}

// Tile of at most `most` sites for the stencil of the given parity (< 0: full lattice); off when
// no tile beats consecutive sites (csrc/dslash.cu).
TileMap pick_tile(const int L[4], int parity, int most);
// CTAs of a launch over nsites sites with `per` site slots per CTA
inline int stencil_ctas(const TileMap& m, int nsites, int per) {
  return m.on ? nsites / m.sites : (nsites + per - 1) / per;
}

// Whether storage S is compiled for links of form LL (load_link).  The windowed form is for fields
// with S's widest accesses; element-wise ABI links are for what is less aligned, and a choice for
// half storage.
template <typename S>
constexpr bool link_form(int ll) {
  if (std::is_same<typename S::real, double>::value) return ll < 2;
  if (std::is_same<S, StC64>::value) return ll > 0;
  if (std::is_same<S, StC64N>::value) return ll < 3;
  return true;
}

// The stencil in launch shape v with links of form ll (dslash_forms.cuh, one instantiation per
// storage type in dslash_<storage>.cu).
template <typename S>
void launch_stencil(int v, int dagger, int ll, void* out, const void* in, const void* links,
                    const KGeom& k, int parity, int nsites, int nrhs, cudaStream_t st,
                    size_t in_stride, size_t out_stride);

}  // namespace stencil
}  // namespace wmg
