// Wilson-Dirac stencil (the operator D of Eq. 1), full and single-parity, any storage.
//
// The kernels are in dslash_forms.cuh; here are the choice of launch shape, link layouts and tiles.
#include <cstring>
#include <type_traits>

#include "bits.cuh"
#include "common.cuh"
#include "internal.h"
#include "stencil.cuh"
#include "vec.cuh"

namespace wmg {
namespace {

using namespace stencil;

// Launch shapes (dslash_forms.cuh), searched by the autotuner per (dtype, link form, alignment,
// parity, dagger, volume, nrhs): 0 and 1 one site per thread, 128 threads, registers uncapped and
// capped at 128; 2 one thread per site and hop.  FP32 arithmetic: 3 one site per thread at 80
// registers, 4 and 5 take 2 and 4 right-hand sides per thread, candidates when nrhs > 1; 6, 7 and 8
// (4-byte types) are 3, 4 and 5 on consecutive sites, ABI links read element by element: with the
// links shared by several right-hand sides, the windows' selects and the tiles can cost more than
// they save (bf16, 12 right-hand sides at 16^3x32: 103 -> 98 us).  FP64: 3 as 0 with consecutive
// sites (12x10x14x18: 62 us instead of 77, the tile's part-filled warps cost FP64 issue); 2 and 4
// right-hand sides per thread spill kilobytes (78 and 139 us against 19 at 8^4, 2 right-hand sides).
// Two threads per site in FP64 (20 us there, alone) are slower in a chain of dependent launches: their
// 128 CTAs are placed while the SMs still drain, several to one SM (a solve at 8^3x16: 11.2 ms
// against 8.8 with one thread per site and hop).
constexpr int kNumForms = 6, kNumSingle = 4, kNumF64 = 4, kNumHalf = 9;

// S: the storage type; SN: its form for fields that are only 16-byte aligned.  Fields or ABI links
// less aligned than S's accesses and the windowed links want run the same shapes on 16-byte accesses
// and element loads, under tuning keys of their own; in FP32 arithmetic on consecutive sites, which
// mostly suit those accesses better than tiles (complex float at 16^3x32, 1 / 4 / 12 right-hand
// sides: 20.4 / 63 / 165 us, with tiles 21.6 / 71 / 186), with the uncapped single-site shape and
// the several-right-hand-side ones on tiles as kTiled more candidates (8^4, 12 right-hand sides: 9
// us, consecutive sites 12-14).
constexpr int kTiled = 3, kTiledSingle = 1;

template <typename S, typename SN>
int launch_typed(void* out, const void* in, const void* links, const Geom& g, int parity,
                 int dagger, int nrhs, cudaStream_t st, size_t in_stride, size_t out_stride,
                 int dtype, int layout, const void* subf) {
  constexpr bool f64 = std::is_same<S, StC128>::value;
  constexpr bool site32 = !std::is_same<S, SN>::value;   // 32-byte site accesses
  if (layout == 2 && f64)
    return fail(MG_EINVAL, "dslash: two-row links are not used with complex double fields");
  KGeom k = to_kgeom(g);
  k.sub = parity >= 0 ? subf : nullptr;
  k.tile = pick_tile(g.L, parity, 128);
  int nsites = parity < 0 ? g.V : g.V / 2;
  const size_t es = sizeof(typename S::elem);
  uintptr_t al = (uintptr_t)out | (uintptr_t)in | (uintptr_t)k.sub;
  if (nrhs > 1) al |= (in_stride * es) | (out_stride * es);
  if (al & 15) return fail(MG_EINVAL, "dslash: spinor fields must be 16-byte aligned");
  if ((uintptr_t)links & (es - 1)) return fail(MG_EINVAL, "dslash: links misaligned for their dtype");
  bool wide = !site32 || (al & 31) == 0;
  // the windowed link loads (load_link, LL = 3) start at a 16-byte boundary
  if (layout == 0 && !f64) wide = wide && ((uintptr_t)links & 15) == 0;
  const int forms = f64 ? kNumF64 : nrhs == 1 ? kNumSingle : kNumForms;
  auto run = [&](int v) {
    if (!wide) {
      KGeom kn = k;
      if (!f64) kn.tile.on = k.tile.on && v >= forms;
      if (v >= forms) v = v == forms ? 0 : v - forms + 3;   // 0, 4, 5 on tiles
      launch_stencil<SN>(v, dagger, layout, out, in, links, kn, parity, nsites, nrhs, st, in_stride, out_stride);
      return;
    }
    if (v >= kNumForms) {   // half storage only
      KGeom kc = k;
      kc.tile.on = 0;
      launch_stencil<S>(v - 3, dagger, layout, out, in, links, kc, parity, nsites, nrhs, st, in_stride, out_stride);
      return;
    }
    launch_stencil<S>(v, dagger, layout == 0 && !f64 ? 3 : layout, out, in, links, k, parity, nsites,
                      nrhs, st, in_stride, out_stride);
  };
  const int more = f64 ? 0 : !wide ? (nrhs == 1 ? kTiledSingle : kTiled)
                   : nrhs > 1 && es == 4 ? kNumHalf - kNumForms : 0;
  int v = tuned_variant(dtype + 16 * layout + (wide ? 0 : 64), parity, dagger, g.V, nrhs, st, forms + more, run);
  if (v < 0) return fail(MG_ECUDA, "dslash autotune failed");
  // algorithmic bytes: in + out spinors per rhs and each link once (parity: all 4V links),
  // 18 reals per link whatever the stored form
  double real_bytes = (double)sizeof(typename S::real) * (sizeof(typename S::elem) == 4 ? 0.5 : 1.0);
  double per_site = parity < 0 ? 48.0 * nrhs + 72.0 : 48.0 * nrhs + 144.0;
  const char* name = dtype == MG_C128 ? "dslash_c128" : dtype == MG_C64 ? "dslash_c64"
                     : dtype == MG_F16 ? "dslash_f16" : "dslash_bf16";
  ProfScope ps(name, per_site * real_bytes * nsites, 1320.0 * nsites * nrhs, st);
  run(v);
  WMG_LAUNCHED();
  return MG_OK;
}

template <typename E>
__global__ void link_to_lanes_kernel(E* dst, const zd* __restrict__ src, int V, int ne) {
  typedef typename VecT<E>::R R;
  size_t total = (size_t)4 * V * ne;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    // e enumerates the destination [mu][entry][site], entries 0 .. ne - 1 (row-major)
    size_t site = e % V, rest = e / V;
    int entry = (int)(rest % ne), mu = (int)(rest / ne);
    zd v = src[((size_t)mu * V + site) * 9 + entry];
    VecT<E>::st(dst, e, cplx<R>{(R)v.re, (R)v.im});
  }
}

}  // namespace

template <typename E>
int link_to_lanes_v(E* dst, const zd* src, int V, cudaStream_t st, int rows) {
  size_t total = (size_t)4 * V * 3 * rows;
  size_t g = (total + 255) / 256, cap = (size_t)num_sms() * 16;
  link_to_lanes_kernel<E><<<(unsigned)(g < cap ? g : cap), 256, 0, st>>>(dst, src, V, 3 * rows);
  WMG_LAUNCHED();
  return MG_OK;
}
template int link_to_lanes_v<zd>(zd*, const zd*, int, cudaStream_t, int);
template int link_to_lanes_v<zf>(zf*, const zd*, int, cudaStream_t, int);
template int link_to_lanes_v<zh>(zh*, const zd*, int, cudaStream_t, int);
template int link_to_lanes_v<zbf>(zbf*, const zd*, int, cudaStream_t, int);

namespace {

// |U U^dag - 1| and |det U - 1| of one link, largest entry, in double-float arithmetic on the
// FP32 units (error-free products and sums, ~2^-48 relative: deviations are resolved far below
// 1e-9).  Entries that are not finite, or whose products leave the FP32 range, give a huge value: a
// deviation that is not a number (inf - inf in the error-free sums) is one.
__device__ float su3_deviation(const zdf u[9]) {
  float worst = 0.f;
  auto take = [&](float d) { worst = d <= 3e38f ? fmaxf(worst, d) : 3e38f; };
  // U U^dag - 1: the six entries a <= b of the Hermitian matrix
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = a; b < 3; ++b) {
      zdfacc s{};
#pragma unroll
      for (int c = 0; c < 3; ++c) zdf_fmac(s, u[b * 3 + c], u[a * 3 + c]);   // u_ac conj(u_bc)
      zdf v = zdf_norm(s);
      if (a == b) v.re = df_add(v.re, {-1.0f, 0.0f});
      take(fabsf(v.re.hi));
      take(fabsf(v.im.hi));
    }
  // det U - 1 by cofactors of the first row
  zdfacc t{};
  zdf_fma(t, u[4], u[8]);
  zdf_fma(t, zdf_neg(u[5]), u[7]);
  const zdf c0 = zdf_norm(t);
  t = zdfacc{};
  zdf_fma(t, u[3], u[8]);
  zdf_fma(t, zdf_neg(u[5]), u[6]);
  const zdf c1 = zdf_norm(t);
  t = zdfacc{};
  zdf_fma(t, u[3], u[7]);
  zdf_fma(t, zdf_neg(u[4]), u[6]);
  const zdf c2 = zdf_norm(t);
  t = zdfacc{};
  zdf_fma(t, u[0], c0);
  zdf_fma(t, zdf_neg(u[1]), c1);
  zdf_fma(t, u[2], c2);
  zdf det = zdf_norm(t);
  det.re = df_add(det.re, {-1.0f, 0.0f});
  take(sqrtf(det.re.hi * det.re.hi + det.im.hi * det.im.hi));
  return worst;
}

// Everything a handle keeps of its links, in one pass over them: the ABI copy, its double-float
// form, the lane-contiguous FP64 and FP32 stencil copies (the latter with `rows` rows) and the
// largest deviation from SU(3) (bits of a non-negative float, ordered like the values).  Null
// outputs are skipped.  A CTA's links go through shared memory, so loads and stores are coalesced
// in both layouts; the conversions stay off the FP64 pipe (bits.cuh).  The separate passes (copy,
// two layouts, conversion, check) took 225 us at 16^3x32, this one 97 us (85 us without the check).
constexpr int LPT = 128;
__global__ void __launch_bounds__(LPT)
links_prepare_kernel(zd* copy, zdf* df_, zd* lanes64, zf* lanes32, int rows, unsigned* dev,
                     const zd* __restrict__ src, int V) {
  __shared__ zd su[LPT * 9];
  const size_t n = (size_t)4 * V, l0 = (size_t)blockIdx.x * LPT;
  const int nl = (int)min((size_t)LPT, n - l0);
  for (int e = threadIdx.x; e < nl * 9; e += LPT) {
    const zd v = src[l0 * 9 + e];
    su[e] = v;
    if (copy) copy[l0 * 9 + e] = v;
    if (df_) {
      const zdf q = zdf_from_bits(v);
      reinterpret_cast<float4*>(df_)[l0 * 9 + e] = make_float4(q.re.hi, q.re.lo, q.im.hi, q.im.lo);
    }
  }
  __syncthreads();
  float worst = 0.f;
  if ((int)threadIdx.x < nl) {
    const size_t l = l0 + threadIdx.x, mu = l / V, site = l - mu * V;
    const zd* u = su + threadIdx.x * 9;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const zd v = u[i];
      if (lanes64) lanes64[(mu * 9 + i) * V + site] = v;
      if (lanes32 && i < 3 * rows)
        lanes32[(mu * 3 * rows + i) * V + site] = {f32_from_bits(v.re), f32_from_bits(v.im)};
    }
    if (dev) {
      zdf q[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) q[i] = zdf_from_bits(u[i]);
      worst = su3_deviation(q);
    }
  }
  if (!dev) return;
  // warp, then CTA maximum: one atomic per CTA
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, o));
  __shared__ float wmax[LPT / 32];
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = worst;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = wmax[0];
    for (int w = 1; w < LPT / 32; ++w) m = fmaxf(m, wmax[w]);
    atomicMax(dev, __float_as_uint(m));
  }
}

}  // namespace

int links_prepare(zd* copy, zdf* df_, zd* lanes64, zf* lanes32, int rows, double* deviation,
                  const zd* src, int V, cudaStream_t st) {
  unsigned* d = nullptr;
  if (deviation) {
    WMG_CUDA(scratch_alloc(&d, sizeof(*d), st));
    WMG_CUDA(cudaMemsetAsync(d, 0, sizeof(*d), st));
  }
  links_prepare_kernel<<<(unsigned)(((size_t)4 * V + LPT - 1) / LPT), LPT, 0, st>>>(
      copy, df_, lanes64, lanes32, rows, d, src, V);
  WMG_LAUNCHED();
  if (deviation) {
    unsigned bits = 0;
    WMG_CUDA(cudaMemcpyAsync(&bits, d, sizeof(bits), cudaMemcpyDeviceToHost, st));
    WMG_CUDA(cudaStreamSynchronize(st));
    scratch_free(d, st);
    float f;
    std::memcpy(&f, &bits, sizeof(f));
    *deviation = f;
  }
  return MG_OK;
}

namespace stencil {

// The tile of at most `most` sites with the least L2 -> L1 traffic per site: its own spinors, the
// 2 / t_mu neighbours outside it in every direction it does not span, and the links' part-used
// 32-byte sectors, times the idle lanes of its last warp.  Consecutive sites are the tile's rival:
// `most` of them span x, and y as far as they reach.
TileMap pick_tile(const int L[4], int parity, int most) {
  struct Key {
    int L[4], half, most;
  };
  struct Entry {
    Key k;
    TileMap m;
  };
  // the last few answers of this thread (a solver asks for the same two lattices again and again)
  static thread_local Entry cache[4];
  static thread_local int used = 0, next = 0;
  const Key key = {{L[0], L[1], L[2], L[3]}, parity >= 0 ? 1 : 0, most};
  for (int i = 0; i < used; ++i)
    if (std::memcmp(&cache[i].k, &key, sizeof(Key)) == 0) return cache[i].m;
  const int E[4] = {key.half ? L[0] / 2 : L[0], L[1], L[2], L[3]};
  auto halo = [](int t, int e) { return t == e ? 0.0 : 2.0 / t; };
  TileMap m;
  // consecutive sites: rows of x, then of y, inside one CTA
  const int lx = E[0] < most ? E[0] : most;
  const int ly = E[0] < most ? (most / E[0] < E[1] ? most / E[0] : E[1]) : 1;
  double best = 96.0 * (1.0 + halo(lx, E[0]) + halo(ly, E[1]) + halo(1, E[2]) + halo(1, E[3])) +
                384.0 + 192.0 / lx;
  const int xmin = E[0] < 8 ? E[0] : 8;
  for (int a = xmin; a <= E[0] && a <= most; ++a) {
    if (E[0] % a) continue;
    for (int b = 1; b <= E[1] && a * b <= most; ++b) {
      if (E[1] % b) continue;
      for (int c = 1; c <= E[2] && a * b * c <= most; ++c) {
        if (E[2] % c) continue;
        for (int d = 1; d <= E[3] && a * b * c * d <= most; ++d) {
          if (E[3] % d) continue;
          const int n = a * b * c * d;
          const double links = (a % 4 ? (8.0 * a + 24.0) / (8.0 * a) : 1.0) + 0.5 / a;
          const double cost = (96.0 * (1.0 + halo(a, E[0]) + halo(b, E[1]) + halo(c, E[2]) +
                                       halo(d, E[3])) + 384.0 * links) *
                              ((n + 31) / 32 * 32) / n;
          if (cost < best - 1e-9) {
            best = cost;
            m.on = 1;
            m.t[0] = a; m.t[1] = b; m.t[2] = c; m.t[3] = d;
          }
        }
      }
    }
  }
  if (m.on) {
    m.sites = m.t[0] * m.t[1] * m.t[2] * m.t[3];
    const long long tiles = (long long)E[0] * E[1] * E[2] * E[3] / m.sites;
    for (int a = 0; a < 3; ++a) {
      m.n[a] = E[a] / m.t[a];
      // u / t = (u tm) >> 16 for u t < 2^16 (u, t <= 128); b / n = high word of b nm for
      // b n < 2^32
      m.tm[a] = (65536u + m.t[a] - 1) / m.t[a];
      m.nm[a] = m.n[a] == 1 ? 0u : 0xffffffffu / (unsigned)m.n[a] + 1u;
      if (tiles * m.n[a] >= (1LL << 32)) m.on = 0;
    }
  }
  cache[next] = {key, m};
  next = (next + 1) % 4;
  if (used < 4) ++used;
  return m;
}

}  // namespace stencil

int dslash_launch(int dtype, void* out, const void* in, const void* links, const Geom& g,
                  int parity, int dagger, int nrhs, cudaStream_t st, size_t in_stride,
                  size_t out_stride, int link_layout, const void* sub) {
  size_t half = (size_t)12 * (parity < 0 ? g.V : g.V / 2);
  if (in_stride == 0) in_stride = half;
  if (out_stride == 0) out_stride = half;
  switch (dtype) {
    case MG_C128:
      return launch_typed<StC128, StC128N>(out, in, links, g, parity, dagger, nrhs, st, in_stride, out_stride, dtype,
                                  link_layout, sub);
    case MG_C64:
      return launch_typed<StC64, StC64N>(out, in, links, g, parity, dagger, nrhs, st, in_stride, out_stride, dtype,
                                  link_layout, sub);
    case MG_F16:
      return launch_typed<StF16, StF16>(out, in, links, g, parity, dagger, nrhs, st, in_stride, out_stride, dtype,
                                  link_layout, sub);
    case MG_BF16:
      return launch_typed<StBF16, StBF16>(out, in, links, g, parity, dagger, nrhs, st, in_stride, out_stride, dtype,
                                  link_layout, sub);
  }
  return fail(MG_EINVAL, "dslash: unknown dtype");
}

}  // namespace wmg

extern "C" int wilson_dslash(void* out, const void* in, const void* links, const int dims[4],
                             double kappa, const double hop_weight[4], const int bc_phase[4],
                             int parity, int dagger, int dtype, int nrhs, void* stream) {
  using namespace wmg;
  if (!out || !in || !links || !dims) return fail(MG_EINVAL, "wilson_dslash: NULL pointer");
  if (nrhs < 1) return fail(MG_EINVAL, "wilson_dslash: nrhs < 1");
  if (parity < -1 || parity > 1) return fail(MG_EINVAL, "wilson_dslash: parity must be -1, 0 or 1");
  if (dtype < MG_C128 || dtype > MG_BF16) return fail(MG_EINVAL, "wilson_dslash: bad dtype");
  double w1[4] = {1, 1, 1, 1};
  int bc1[4] = {1, 1, 1, 1};
  Geom g;
  WMG_TRY(make_geom(g, dims, kappa, hop_weight ? hop_weight : w1, bc_phase ? bc_phase : bc1,
                    parity >= 0));
  if (out == in) return fail(MG_EINVAL, "wilson_dslash: out must not alias in");
  cudaStream_t st = (cudaStream_t)stream;
  size_t eb = dtype_bytes(dtype);
  size_t fsites = parity < 0 ? (size_t)g.V : (size_t)g.V / 2;
  size_t fbytes = fsites * 12 * eb * nrhs;
  size_t lbytes = (size_t)4 * g.V * 9 * eb;
  Staged sin, sl, sout;
  WMG_TRY(stage_in(sin, in, fbytes, st));
  WMG_TRY(stage_in(sl, links, lbytes, st));
  WMG_TRY(stage_out_alloc(sout, out, fbytes, st));
  WMG_TRY(dslash_launch(dtype, sout.dev, sin.dev, sl.dev, g, parity, dagger, nrhs, st, 0, 0));
  WMG_TRY(stage_out_finish(sout, out, fbytes, st));
  return MG_OK;
}
