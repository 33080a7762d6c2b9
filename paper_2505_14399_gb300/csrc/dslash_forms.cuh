// Kernels of the Wilson-Dirac stencil (the operator D of Eq. 1) and the launch shapes that the
// autotuner chooses from, for one storage type; csrc/dslash_<storage>.cu instantiate them, one
// translation unit each, so that they compile side by side.
//
// One thread per output site and right-hand side: each of the 8 hops loads the neighbour spinor,
// projects it to a 2-spin half spinor with (1 -/+ gamma_mu) in the chiral basis, multiplies by
// U_mu(x) or U_mu(x-mu)^dag, and reconstructs the lower spin pair from the upper one.  Spinor loads
// are 32-byte vector loads of the [site][spin][colour] layout (16-byte where the fields are only so
// aligned); links are read through the read-only path.  Further shapes take one thread per site and
// hop, or 2 and 4 right-hand sides per thread: there each link is loaded once
// and applied to NR spinors (the test-vector streams of the setup smoothing, Eq. 2, and batched
// solves), and every thread keeps NR independent neighbour loads in flight per hop.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "stencil.cuh"
#include "vec.cuh"

namespace wmg {
namespace {

using namespace stencil;

// parity < 0: out = in - kappa H in (full lattice).  parity p >= 0: out_p = -kappa H in_{1-p}
// on half-lattice (checkerboard-indexed) fields.
template <typename S, int DAG, int TPB, int MINB, int LL>
__global__ void __launch_bounds__(TPB, MINB)
dslash_kernel(typename S::elem* __restrict__ out, const typename S::elem* __restrict__ in,
              const typename S::elem* __restrict__ links, KGeom g, int parity, int nsites,
              size_t in_stride, size_t out_stride) {
  dep_entry();
  typedef typename S::real R;
  const size_t rhs = blockIdx.y;
  int i, site, c[4];
  if (!stencil_work(g, parity, nsites, threadIdx.x, TPB, i, site, c)) return;
  cplx<R> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {0, 0};
  bool half_in = parity >= 0;
  size_t in_off = rhs * in_stride;
  hop_pair<0, DAG, S, LL>(g, site, c, in, in_off, half_in, links, acc);
  hop_pair<1, DAG, S, LL>(g, site, c, in, in_off, half_in, links, acc);
  hop_pair<2, DAG, S, LL>(g, site, c, in, in_off, half_in, links, acc);
  hop_pair<3, DAG, S, LL>(g, site, c, in, in_off, half_in, links, acc);
  R mk = -kap<R>(g);
  cplx<R> res[12];
  if (parity < 0) {
    cplx<R> p[12];
    SiteIO<S>::load(in + in_off, (size_t)site, p);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      res[k].re = fma(mk, acc[k].re, p[k].re);
      res[k].im = fma(mk, acc[k].im, p[k].im);
    }
    SiteIO<S>::store(out + rhs * out_stride, (size_t)site, res);
  } else {
#pragma unroll
    for (int k = 0; k < 12; ++k) res[k] = mk * acc[k];
    apply_sub<S>(g, rhs * out_stride, i, res);
    SiteIO<S>::store(out + rhs * out_stride, (size_t)i, res);
  }
}

// One thread per site and hop (hop_lanes), consecutive sites; lane pairs write one spin each.
template <typename S, int DAG, int LL>
__global__ void __launch_bounds__(128)
dslash_hop_kernel(typename S::elem* __restrict__ out, const typename S::elem* __restrict__ in,
                  const typename S::elem* __restrict__ links, KGeom g, int parity, int nsites,
                  size_t in_stride, size_t out_stride) {
  dep_entry();
  typedef typename S::real R;
  const int i = blockIdx.x * (blockDim.x >> 3) + (threadIdx.x >> 3), hop = threadIdx.x & 7;
  const bool active = i < nsites;
  int c[4] = {0, 0, 0, 0}, site = 0;
  if (active) site = stencil_site(g, parity, i, c);
  const size_t rhs = blockIdx.y;
  const typename S::elem* inr = in + rhs * in_stride;
  cplx<R> acc[3];
  hop_lanes<DAG, S, LL>(g, active, site, c, hop, inr, parity >= 0, links, acc);
  if (!active || (hop & 1)) return;
  const R mk = -kap<R>(g);
  const size_t e0 = (size_t)i * 12 + 3 * (hop >> 1);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cplx<R> r = mk * acc[k];
    if (parity < 0) {
      const cplx<R> x = S::ld(inr, e0 + k);
      r = {fma(mk, acc[k].re, x.re), fma(mk, acc[k].im, x.im)};
    } else if (g.sub) {
      r = S::ld(static_cast<const typename S::elem*>(g.sub) + rhs * out_stride, e0 + k) - r;
    }
    S::st(out + rhs * out_stride, e0 + k, r);
  }
}

template <int MU, int DAG, typename S, int LL, int NR>
__device__ __forceinline__ void hop_fwd_m(const KGeom& g, int site, const int c[4],
                                          const typename S::elem* in, size_t in_stride, int nr,
                                          bool half_in, const typename S::elem* links,
                                          cplx<typename S::real> acc[NR][12]) {
  typedef typename S::real R;
  constexpr int SF = DAG ? +1 : -1;
  R w = wgt<R>(g, MU);
  int nb = (c[MU] == g.L[MU] - 1) ? site - (g.L[MU] - 1) * g.stride[MU] : site + g.stride[MU];
  R cf = (c[MU] == g.L[MU] - 1 && g.bc[MU] < 0) ? -w : w;
  size_t idx = half_in ? (size_t)(nb >> 1) : (size_t)nb;
  cplx<R> u[9];
  load_link<S, LL>(links, g.V, MU, site, u);
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    // a ragged last group re-reads its last right-hand side (discarded at the store), so the
    // loads carry no branch and all NR can be in flight at once
    {
      cplx<R> p[12], h[6], gg[6];
      SiteIO<S>::load(in + (r < nr ? r : nr - 1) * in_stride, idx, p);
      project<MU, SF, R>(p, h);
      mul_link<R>(u, h, gg);
      accumulate<MU, SF, R>(acc[r], gg, cf);
    }
  }
}

template <int MU, int DAG, typename S, int LL, int NR>
__device__ __forceinline__ void hop_bwd_m(const KGeom& g, int site, const int c[4],
                                          const typename S::elem* in, size_t in_stride, int nr,
                                          bool half_in, const typename S::elem* links,
                                          cplx<typename S::real> acc[NR][12]) {
  typedef typename S::real R;
  constexpr int SB = DAG ? -1 : +1;
  R w = wgt<R>(g, MU);
  int nb = (c[MU] == 0) ? site + (g.L[MU] - 1) * g.stride[MU] : site - g.stride[MU];
  R cf = (c[MU] == 0 && g.bc[MU] < 0) ? -w : w;
  size_t idx = half_in ? (size_t)(nb >> 1) : (size_t)nb;
  cplx<R> u[9];
  load_link<S, LL>(links, g.V, MU, nb, u);
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    // a ragged last group re-reads its last right-hand side (discarded at the store), so the
    // loads carry no branch and all NR can be in flight at once
    {
      cplx<R> p[12], h[6], gg[6];
      SiteIO<S>::load(in + (r < nr ? r : nr - 1) * in_stride, idx, p);
      project<MU, SB, R>(p, h);
      mul_link_dag<R>(u, h, gg);
      accumulate<MU, SB, R>(acc[r], gg, cf);
    }
  }
}

// One thread per site and group of NR right-hand sides (grid.y = groups); the last group
// may hold fewer than NR.
template <typename S, int DAG, int NR, int LL, int MINB>
__global__ void __launch_bounds__(128, MINB)
dslash_mrhs_kernel(typename S::elem* __restrict__ out, const typename S::elem* __restrict__ in,
                   const typename S::elem* __restrict__ links, KGeom g, int parity, int nsites,
                   int nrhs, size_t in_stride, size_t out_stride) {
  dep_entry();
  typedef typename S::real R;
  int i, site, c[4];
  if (!stencil_work(g, parity, nsites, threadIdx.x, 128, i, site, c)) return;
  const int r0 = blockIdx.y * NR;
  const int nr = min(NR, nrhs - r0);
  const bool half_in = parity >= 0;
  const typename S::elem* inr = in + (size_t)r0 * in_stride;
  cplx<R> acc[NR][12];
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[r][k] = {0, 0};
  hop_fwd_m<0, DAG, S, LL, NR>(g, site, c, inr, in_stride, nr, half_in, links, acc);
  hop_bwd_m<0, DAG, S, LL, NR>(g, site, c, inr, in_stride, nr, half_in, links, acc);
  hop_fwd_m<1, DAG, S, LL, NR>(g, site, c, inr, in_stride, nr, half_in, links, acc);
  hop_bwd_m<1, DAG, S, LL, NR>(g, site, c, inr, in_stride, nr, half_in, links, acc);
  hop_fwd_m<2, DAG, S, LL, NR>(g, site, c, inr, in_stride, nr, half_in, links, acc);
  hop_bwd_m<2, DAG, S, LL, NR>(g, site, c, inr, in_stride, nr, half_in, links, acc);
  hop_fwd_m<3, DAG, S, LL, NR>(g, site, c, inr, in_stride, nr, half_in, links, acc);
  hop_bwd_m<3, DAG, S, LL, NR>(g, site, c, inr, in_stride, nr, half_in, links, acc);
  const R mk = -kap<R>(g);
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    if (r < nr) {
      cplx<R> res[12];
      typename S::elem* o = out + (size_t)(r0 + r) * out_stride;
      if (parity < 0) {
        cplx<R> p[12];
        SiteIO<S>::load(inr + r * in_stride, (size_t)site, p);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
          res[k].re = fma(mk, acc[r][k].re, p[k].re);
          res[k].im = fma(mk, acc[r][k].im, p[k].im);
        }
        SiteIO<S>::store(o, (size_t)site, res);
      } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) res[k] = mk * acc[r][k];
        apply_sub<S>(g, (size_t)(r0 + r) * out_stride, i, res);
        SiteIO<S>::store(o, (size_t)i, res);
      }
    }
  }
}

template <typename S, int DAG, int LL, int MINB>
void launch_site(void* out, const void* in, const void* links, const KGeom& k, int parity,
                 int nsites, int nrhs, cudaStream_t st, size_t is, size_t os) {
  typedef typename S::elem E;
  dim3 grid(stencil_ctas(k.tile, nsites, 128), nrhs);
  launch_dep(dslash_kernel<S, DAG, 128, MINB, LL>, grid, 128, 0, st, (E*)out, (const E*)in,
             (const E*)links, k, parity, nsites, is, os);
}

// register caps measured best on GB300: 2 right-hand sides per thread at <= 128 registers, 4
// uncapped (a 168-register cap spills)
template <typename S, int DAG, int LL, int NR>
void launch_mrhs(void* out, const void* in, const void* links, const KGeom& k, int parity,
                 int nsites, int nrhs, cudaStream_t st, size_t is, size_t os) {
  typedef typename S::elem E;
  dim3 grid(stencil_ctas(k.tile, nsites, 128), (nrhs + NR - 1) / NR);
  launch_dep(dslash_mrhs_kernel<S, DAG, NR, LL, NR == 2 ? 4 : 1>, grid, 128, 0, st, (E*)out,
             (const E*)in, (const E*)links, k, parity, nsites, nrhs, is, os);
}

template <typename S, int DAG, int LL>
void launch_form(int v, void* out, const void* in, const void* links, const KGeom& k, int parity,
                 int nsites, int nrhs, cudaStream_t st, size_t is, size_t os) {
  typedef typename S::elem E;
  constexpr bool f64 = std::is_same<typename S::real, double>::value;
  if (v == 2) {
    // one warp per CTA until every SM has a few of them
    const int t = (long long)nsites * nrhs < 4LL * 16 * num_sms() ? 32 : 128;
    dim3 grid((nsites + t / 8 - 1) / (t / 8), nrhs);
    launch_dep(dslash_hop_kernel<S, DAG, LL>, grid, t, 0, st, (E*)out, (const E*)in,
               (const E*)links, k, parity, nsites, is, os);
    return;
  }
  if constexpr (f64) {
    if (v == 3) {
      KGeom kc = k;
      kc.tile.on = 0;
      return launch_site<S, DAG, LL, 1>(out, in, links, kc, parity, nsites, nrhs, st, is, os);
    }
  } else {
    if (v == 3) return launch_site<S, DAG, LL, 6>(out, in, links, k, parity, nsites, nrhs, st, is, os);
    if (v == 4) return launch_mrhs<S, DAG, LL, 2>(out, in, links, k, parity, nsites, nrhs, st, is, os);
    if (v == 5) return launch_mrhs<S, DAG, LL, 4>(out, in, links, k, parity, nsites, nrhs, st, is, os);
  }
  if (v == 1) return launch_site<S, DAG, LL, 4>(out, in, links, k, parity, nsites, nrhs, st, is, os);
  launch_site<S, DAG, LL, 1>(out, in, links, k, parity, nsites, nrhs, st, is, os);
}

}  // namespace

namespace stencil {

template <typename S>
void launch_stencil(int v, int dagger, int ll, void* out, const void* in, const void* links,
                    const KGeom& k, int parity, int nsites, int nrhs, cudaStream_t st, size_t is,
                    size_t os) {
  auto go = [&](auto l) {
    constexpr int LL = decltype(l)::value;
    if constexpr (link_form<S>(LL)) {
      if (dagger) launch_form<S, 1, LL>(v, out, in, links, k, parity, nsites, nrhs, st, is, os);
      else launch_form<S, 0, LL>(v, out, in, links, k, parity, nsites, nrhs, st, is, os);
    }
  };
  if (ll == 0) go(std::integral_constant<int, 0>{});
  else if (ll == 1) go(std::integral_constant<int, 1>{});
  else if (ll == 2) go(std::integral_constant<int, 2>{});
  else go(std::integral_constant<int, 3>{});
}

}  // namespace stencil

#define WMG_STENCIL(S)                                                                        \
  template void stencil::launch_stencil<S>(int, int, int, void*, const void*, const void*,    \
                                           const stencil::KGeom&, int, int, int, cudaStream_t, \
                                           size_t, size_t);

}  // namespace wmg
