// Batched streaming chiral SVD (Algorithm 3, Eqs. 7-8) over all aggregates and both
// chiralities at once.
//
// Every (aggregate j, chirality alpha) owns a tile A = [Phi_{s-1} | Psi_s] of M = 6 n_d
// rows (Eq. 3 split) stored column-major in FP64, or in double-float (zdf, the same 16 bytes)
// when the sums run in double-float: those tiles then stay double-float from the gather to
// the final prolongator, so no kernel converts them on the FP64 units.  One stream is:
//   gather   : chiral split of the r new smoothed vectors into columns kk.. of all tiles
//   gram     : G = A^dag A (c x c Hermitian, c = kk + r), one CTA per tile
//   eig      : parallel cyclic Jacobi (Brent-Luk ordering) on G in shared memory,
//              eigenvalues sorted descending (ties by index) -> Sigma^2 and V
//   update   : Phi_s = A V_k (= U_k Sigma_k, Eq. 7), or U_k = A V_k Sigma_k^{-1} at the end
// An optional second pass (G of A V over all c columns, eig, rotate) restores the
// accuracy lost by forming A^dag A (its rotations are relative to sigma_i sigma_j).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "bits.cuh"
#include "df64.cuh"
#include "internal.h"

namespace wmg {

namespace {

// One thread per component pair of a site, for every vector in turn: coalesced loads, stores of
// 32 contiguous bytes in runs of 96, and the aggregate's index arithmetic once for all vectors
// (8 vectors at 16^3x32: 120 -> 55 us).
template <typename R, typename TO>
__global__ void __launch_bounds__(256)
gather_kernel(TO* tiles, int cmax, int col0, const cplx<R>* __restrict__ f, int nvec, Blocking B) {
  const unsigned e = blockIdx.x * 256u + threadIdx.x;
  const unsigned n = 6u * B.nd * B.d;
  if (e >= n) return;
  const int s = (int)(e / 6), p = (int)(e - 6 * (unsigned)s), alpha = p / 3;
  int j, l;
  B.block_of(s, &j, &l);
  TO* dst = tiles + ((size_t)(2 * j + alpha) * cmax + col0) * B.M + 6 * l + 2 * (p - 3 * alpha);
  for (int v = 0; v < nvec; ++v, dst += B.M) {
    const cplx<R>* src = f + 2 * ((size_t)v * n + e);
    const cplx<R> x = src[0], y = src[1];
    if constexpr (std::is_same<TO, zdf>::value) {
      const zdf a = zdf_from(x), b = zdf_from(y);
      float4* d4 = reinterpret_cast<float4*>(dst);
      d4[0] = make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo);
      d4[1] = make_float4(b.re.hi, b.re.lo, b.im.hi, b.im.lo);
    } else {
      dst[0] = {(double)x.re, (double)x.im};
      dst[1] = {(double)y.re, (double)y.im};
    }
  }
}

constexpr int GT = 256;   // threads per tile CTA
// threads per Jacobi CTA: a round's work is about (c/2)(c/2 + 1)/2 A blocks and c^2/2 V
// entries, a few per thread at 128, and 128-thread CTAs keep every tile of a launch resident
// at once (8 per SM)
constexpr int JT = 128;
constexpr int GR = 32;    // rows staged per chunk
constexpr int MAXC = 64;  // max columns per tile

// G = A^dag A in FP64, upper triangle computed, mirrored.  MAXP: column pairs per thread
// (>= pairs / blockDim), which sets the accumulator registers.
// The first kd columns may be known to be orthogonal with squared norms lamp[t][0..kd-1]
// (the previous stream's Phi = A V_k, whose Gram matrix is V_k^dag G V_k = Lambda_k): their
// block is then written as that diagonal and only the pairs (i, j), i <= j, j >= kd are summed.
template <int MAXP>
__global__ void __launch_bounds__(GT) gram_kernel(zd* G, const zd* __restrict__ tiles, int cmax,
                                                  int c, int M, int kd, const double* lamp,
                                                  int cprev) {
  extern __shared__ zd sA[];  // [GR][c]
  int t = blockIdx.x;
  const zd* A = tiles + (size_t)t * cmax * M;
  const int nth = blockDim.x;
  const int npairs = c * (c + 1) / 2 - kd * (kd + 1) / 2;
  zd acc[MAXP];
  int pi[MAXP], pj[MAXP];
#pragma unroll
  for (int q = 0; q < MAXP; ++q) {
    acc[q] = zd{};
    int p = threadIdx.x + q * nth;
    // p -> (i, j) with i <= j and j >= kd, column by column (column j holds j + 1 pairs)
    int j = kd, rem = p;
    while (j < c && rem >= j + 1) { rem -= j + 1; ++j; }
    pi[q] = rem;
    pj[q] = j;
  }
  zd* Gt = G + (size_t)t * c * c;
  for (int e = threadIdx.x; e < kd * kd; e += nth) {
    const int i = e / kd, j = e % kd;
    Gt[i * c + j] = i == j ? zd{lamp[(size_t)t * cprev + i], 0.0} : zd{0.0, 0.0};
  }
  for (int r0 = 0; r0 < M; r0 += GR) {
    int nr = min(GR, M - r0);
    __syncthreads();
    for (int e = threadIdx.x; e < nr * c; e += nth) {
      int col = e / nr, rr = e % nr;
      sA[rr * c + col] = A[(size_t)col * M + r0 + rr];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < MAXP; ++q) {
      int p = threadIdx.x + q * nth;
      if (p < npairs) {
        zd a = acc[q];
        for (int rr = 0; rr < nr; ++rr) cfmac(a, sA[rr * c + pi[q]], sA[rr * c + pj[q]]);
        acc[q] = a;
      }
    }
  }
#pragma unroll
  for (int q = 0; q < MAXP; ++q) {
    int p = threadIdx.x + q * nth;
    if (p < npairs) {
      zd v = acc[q];
      Gt[pi[q] * c + pj[q]] = v;
      if (pi[q] != pj[q]) Gt[pj[q] * c + pi[q]] = conj(v);
    }
  }
}

// G = A^dag A on double-float tiles, on the FP32 units, with biased accumulators (df64.cuh).
// A thread sums a 2 x 2 block of column pairs over every eighth row, the block's two right
// columns in the two halves of packed instructions: its four operands come from shared memory
// once per four products (24 packed instructions per two products), the eight row groups of a
// block are neighbouring lanes, so a quarter warp reads eight rows at an odd stride (no bank
// conflicts) and the groups meet in shuffles.  Rows arrive in chunks of GR through registers
// (loads of the next chunk in flight during this one's products) and two shared buffers, one
// barrier per chunk.  A group's sums over a chunk (four rows) start at a bias from the norms n of
// the columns over those rows (Cauchy and Schwarz: every partial sum is within n_i n_j) and then
// join a (hi, lo) total.  Against one long double-float sum (df_fma, 12 instructions per product)
// it is half the instructions and more exact: P^dag P of orthonormal 1536-row tiles (the Galerkin
// diagonal) is off by 1.4e-14 instead of 5.6e-13, of 192-row tiles by 2.4e-14 instead of 7.4e-14.
// 16^3x32, four streams (c = 8, 16, 20, 20): 1.88 -> 1.11 ms; 16 384 tiles of 192 x 24: 1.44 ms.
// kd, lamp: as for gram_kernel.  cn[t][i] (leading dimension cld, may be null): the columns'
// squared norms.  nt: 2 x 2 blocks in all, ntc of them per CTA (blockIdx.y picks the slice).
constexpr int GDF_G = 8;        // row groups
constexpr int GDF_T = 40;       // blocks per CTA at most (320 threads)
// PRE: staged column pairs of a row per thread and chunk at most (2, or 4 above 40 columns)
template <int PRE>
__global__ void __launch_bounds__(GDF_T * GDF_G, 2)
gram_df_kernel(zd* G, float* cn, int cld, const zdf* __restrict__ tiles, int cmax, int c, int M,
               int kd, const double* lamp, int cprev, int nt, int ntc) {
  extern __shared__ __align__(16) unsigned char smraw_gd[];
  const int np = (c + 1) / 2, ld = np | 1;      // column pairs, odd row stride
  // [2][re, im][GR][ld]: (hi, hi, lo, lo) of a column pair
  float4* sA = reinterpret_cast<float4*>(smraw_gd);
  float2* snrm = reinterpret_cast<float2*>(sA + 4 * GR * ld);   // [2][GDF_G][np]
  const int t = blockIdx.x, nth = blockDim.x;
  const zdf* A = tiles + (size_t)t * cmax * M;
  const int g = threadIdx.x & (GDF_G - 1);
  int blk = blockIdx.y * ntc + (threadIdx.x / GDF_G);
  const bool work = (int)(threadIdx.x / GDF_G) < ntc && blk < nt;
  if (!work) blk = nt - 1;
  // block index -> (I, J), I <= J, J >= kd / 2, column pair by column pair
  int J = kd / 2, I = blk;
  while (I >= J + 1) { I -= J + 1; ++J; }
  const zdf zero = {{0.f, 0.f}, {0.f, 0.f}};
  zdf pre[PRE][2];
  const int npre = GR * np;
  auto load = [&](int r0) {
#pragma unroll
    for (int u = 0; u < PRE; ++u) {
      const int e = threadIdx.x + u * nth;   // whole warps: 32 rows of one column pair
      const int col = 2 * (e / GR), r = r0 + (e & (GR - 1));
      pre[u][0] = pre[u][1] = zero;
      if (e < npre && r < M) {
        pre[u][0] = zdf_ld(A + (size_t)col * M + r);
        if (col + 1 < c) pre[u][1] = zdf_ld(A + (size_t)(col + 1) * M + r);
      }
    }
  };
  f32x2 th[2][2] = {}, tl[2][2] = {};
  load(0);
  int buf = 0;
  for (int r0 = 0; r0 < M; r0 += GR, buf ^= 1) {
    float4* sre = sA + buf * 2 * GR * ld;
    float4* sim = sre + GR * ld;
    float2* sn = snrm + buf * GDF_G * np;
#pragma unroll
    for (int u = 0; u < PRE; ++u) {
      const int e = threadIdx.x + u * nth;
      if (e < npre) {
        const int at = (e & (GR - 1)) * ld + e / GR;
        const zdf &v = pre[u][0], &w = pre[u][1];
        sre[at] = make_float4(v.re.hi, w.re.hi, v.re.lo, w.re.lo);
        sim[at] = make_float4(v.im.hi, w.im.hi, v.im.lo, w.im.lo);
        // squared norms over the rows of each group: lanes g, g + 8, g + 16, g + 24
        float n0 = fmaf(v.re.hi, v.re.hi, v.im.hi * v.im.hi);
        float n1 = fmaf(w.re.hi, w.re.hi, w.im.hi * w.im.hi);
#pragma unroll
        for (int o = GDF_G; o < 32; o <<= 1) {
          n0 += __shfl_xor_sync(0xffffffffu, n0, o);
          n1 += __shfl_xor_sync(0xffffffffu, n1, o);
        }
        if ((threadIdx.x & 31) < GDF_G)
          sn[(threadIdx.x & 31) * np + e / GR] = make_float2(sqrtf(n0), sqrtf(n1));
      }
    }
    __syncthreads();
    if (r0 + GR < M) load(r0 + GR);
    const float2 ni = sn[g * np + I], nj = sn[g * np + J];
    zbacc2 acc[2];
    f32x2 C[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      acc[q] = zbacc2{};
      const float n = 1.001f * (q ? ni.y : ni.x);
      C[q] = f2_pack(bacc_bias(n * nj.x), bacc_bias(n * nj.y));
      acc[q].re.s = acc[q].im.s = C[q];
    }
#pragma unroll
    for (int u = 0; u < GR / GDF_G; ++u) {
      const int row = (g + u * GDF_G) * ld;
      const float4 ar = sre[row + I], ai = sim[row + I];
      const zdf2 b = {df2_ld(sre + row + J), df2_ld(sim + row + J)};
      zbacc2_fmac(acc[0], zdf_dup({{ar.x, ar.z}, {ai.x, ai.z}}), b);
      zbacc2_fmac(acc[1], zdf_dup({{ar.y, ar.w}, {ai.y, ai.w}}), b);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        const bacc2& a = z ? acc[q].im : acc[q].re;
        const df2 v = df2_two_sum(th[q][z], f2_sub(a.s, C[q]));
        th[q][z] = v.hi;
        tl[q][z] = f2_add(tl[q][z], f2_add(v.lo, f2_add(a.e, a.x)));
      }
  }
  zd* Gt = G + (size_t)t * c * c;
  if (blockIdx.y == 0)
    for (int e = threadIdx.x; e < kd * kd; e += nth) {
      const int i = e / kd, j = e % kd;
      const double l = lamp[(size_t)t * cprev + i];
      Gt[i * c + j] = i == j ? zd{l, 0.0} : zd{0.0, 0.0};
      if (i == j && cn) cn[(size_t)t * cld + i] = fmaxf((float)l, 0.0f);   // noise: either sign
    }
  // sums over the eight lanes of a block, scattered: lane g ends with value g (entry g >> 1, real
  // part or, g odd, imaginary part) after 4 + 2 + 1 additions
  df x[8];
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    const f32x2 h = th[v >> 2][v & 1], l = tl[v >> 2][v & 1];
    x[v] = (v & 2) ? df_two_sum(f2_hi(h), f2_hi(l)) : df_two_sum(f2_lo(h), f2_lo(l));
  }
#pragma unroll
  for (int o = GDF_G / 2; o > 0; o >>= 1) {
    const bool up = (g & o) != 0;
#pragma unroll
    for (int v = 0; v < o; ++v) {
      const df send = up ? x[v] : x[v + o], keep = up ? x[v + o] : x[v];
      const df y = {__shfl_xor_sync(0xffffffffu, send.hi, o), __shfl_xor_sync(0xffffffffu, send.lo, o)};
      x[v] = df_add(keep, y);
    }
  }
  const int i = 2 * I + (g >> 2), j = 2 * J + ((g >> 1) & 1), im = g & 1;
  if (work && i <= j && j < c && j >= kd) {
    const double w = im && i == j ? 0.0 : df_val_bits(x[0]);
    reinterpret_cast<double*>(Gt + i * c + j)[im] = w;
    if (i != j) reinterpret_cast<double*>(Gt + j * c + i)[im] = im ? -w : w;
    else if (cn && !im) cn[(size_t)t * cld + i] = df_to_float(x[0]);
  }
}

// Parallel cyclic Jacobi on a Hermitian c x c matrix per CTA (Brent-Luk round robin).
// Rotation angles are computed in FP64 from the current entries; DF applies the rotations
// to the matrix and the eigenvector basis in double-float arithmetic on the FP32 units
// (this GPU's FP64 rate is ~1/64 of its FP32 rate), otherwise in FP64.
template <typename T> struct JacOps;
template <> struct JacOps<zd> {
  static __device__ __forceinline__ zd from(zd v) { return v; }
  static __device__ __forceinline__ zd val(zd v) { return v; }
  static __device__ __forceinline__ zd zero() { return {0, 0}; }
  static __device__ __forceinline__ zd one() { return {1, 0}; }
  static __device__ __forceinline__ zd cj(zd v) { return {v.re, -v.im}; }
};
template <> struct JacOps<zdf> {
  static __device__ __forceinline__ zdf from(zd v) { return zdf_from(v); }
  static __device__ __forceinline__ zd val(zdf v) { return {df_val(v.re), df_val(v.im)}; }
  static __device__ __forceinline__ zdf zero() { return {{0.f, 0.f}, {0.f, 0.f}}; }
  static __device__ __forceinline__ zdf one() { return {{1.f, 0.f}, {0.f, 0.f}}; }
  static __device__ __forceinline__ zdf cj(zdf v) { return {v.re, df_neg(v.im)}; }
};

// (xa, xb) <- (c xa - s ph xb, s xa + c ph xb), c and s real, ph a unit phase
__device__ __forceinline__ void rot_pair(zd& xa, zd& xb, double c, double s, zd ph) {
  zd e = ph * xb;
  zd na = c * xa - s * e;
  xb = s * xa + c * e;
  xa = na;
}
__device__ __forceinline__ void rot_pair(zdf& xa, zdf& xb, df c, df s, zdf ph) {
  zdf e = {df_dot2(ph.re, xb.re, df_neg(ph.im), xb.im), df_dot2(ph.re, xb.im, ph.im, xb.re)};
  df ms = df_neg(s);
  zdf na = {df_dot2(c, xa.re, ms, e.re), df_dot2(c, xa.im, ms, e.im)};
  xb = {df_dot2(s, xa.re, c, e.re), df_dot2(s, xa.im, c, e.im)};
  xa = na;
}

template <bool DF>
__global__ void __launch_bounds__(JT) jacobi_kernel(double* lam, zd* Vec, const zd* G, int c,
                                                    double rtol) {
  typedef typename std::conditional<DF, zdf, zd>::type T;
  typedef typename std::conditional<DF, df, double>::type TR;
  typedef JacOps<T> J;
  extern __shared__ zd sm[];
  int ce = c + (c & 1);              // padded to even
  int np = ce / 2;
  T* A = reinterpret_cast<T*>(sm);    // ce x ce
  T* Vv = A + ce * ce;                // ce x ce
  T* rph = Vv + ce * ce;              // [np] e^{-i phi}
  TR* rcT = reinterpret_cast<TR*>(rph + np);   // [np] cos
  TR* rsT = rcT + np;                          // [np] sin
  int* pa = reinterpret_cast<int*>(rsT + np);    // [ce - 1][np] pair (a < b) of each round
  int* pb = pa + (ce - 1) * np;
  int* rflag = pb + (ce - 1) * np;               // [np] pair rotated in this round
  __shared__ double dg[MAXC];
  int t = blockIdx.x;
  const zd* Gt = G + (size_t)t * c * c;
  const float rtol2 = (float)(rtol * rtol);
  // double-float: scaled by a power of two (exact) to a largest diagonal entry in [1/2, 1), since
  // the angles square FP32 copies of the entries
  __shared__ double gscale[2];   // 2^-e, 2^e
  if constexpr (DF) {
    if (threadIdx.x < 32) {
      double m = 0;
      for (int i = threadIdx.x; i < c; i += 32) m = fmax(m, fabs(Gt[i * c + i].re));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (threadIdx.x == 0) {
        int e = 0;
        if (m > 0 && isfinite(m)) frexp(m, &e);
        gscale[0] = ldexp(1.0, -e);
        gscale[1] = ldexp(1.0, e);
      }
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < ce * ce; e += blockDim.x) {
    int i = e / ce, j = e % ce;
    zd v = (i < c && j < c) ? Gt[i * c + j] : zd{0, 0};
    if constexpr (DF) v = gscale[0] * v;
    A[e] = J::from(v);
    Vv[e] = (i == j) ? J::one() : J::zero();
  }
  // the round-robin schedule of all ce - 1 rounds of a sweep, once: pairs (top[p], bot[p])
  // start as (2p, 2p + 1); after each round top[0] stays, the others move one place
  if (threadIdx.x == 0) {
    int top[MAXC / 2], bot[MAXC / 2];
    for (int p = 0; p < np; ++p) { top[p] = 2 * p; bot[p] = 2 * p + 1; }
    for (int round = 0; round < ce - 1; ++round) {
      for (int p = 0; p < np; ++p) {
        pa[round * np + p] = min(top[p], bot[p]);
        pb[round * np + p] = max(top[p], bot[p]);
      }
      if (np > 1) {
        int tlast = top[np - 1];
        int b0 = bot[0];
        for (int p = np - 1; p > 1; --p) top[p] = top[p - 1];
        top[1] = b0;
        for (int p = 0; p < np - 1; ++p) bot[p] = bot[p + 1];
        bot[np - 1] = tlast;
      }
    }
  }
  __syncthreads();
  for (int sweep = 0; sweep < 30; ++sweep) {
    int rotated = 0;   // this thread computed a rotation in this sweep
    for (int round = 0; round < ce - 1; ++round) {
      // rotation parameters
      for (int p = threadIdx.x; p < np; p += blockDim.x) {
        const int a = pa[round * np + p], b = pb[round * np + p];
        int f = 0;
        if constexpr (DF) {
          // The angle comes from FP32 copies (the diagonal difference formed in df64 first,
          // so close eigenvalues keep their separation); cos, sin and the phase are then
          // made an exact rotation in df64 (c = (1 + t^2)^-1/2, s = t c, |phase| = 1) by
          // Newton reciprocal square roots on the FP32 units.  An angle good to FP32 leaves
          // ~1e-7 of the pair's coupling, removed when the pair comes round again; the
          // rotation applied is unitary to df64 accuracy either way.
          df cT = {1.f, 0.f}, sT = {0.f, 0.f};
          zdf phT = {{1.f, 0.f}, {0.f, 0.f}};
          if (b < c) {
            zdf g = A[a * ce + b];
            df da = A[a * ce + a].re, db = A[b * ce + b].re;
            float gr = df_to_float(g.re), gi = df_to_float(g.im);
            float ag2 = fmaf(gr, gr, gi * gi);
            if (ag2 > rtol2 * fabsf(da.hi * db.hi) && ag2 > 0.f) {
              float ia = rsqrtf(ag2);            // 1 / |g|
              float zeta = 0.5f * df_to_float(df_add(db, df_neg(da))) * ia;
              float tt = fabsf(zeta) > 1e18f
                             ? 0.5f / zeta
                             : copysignf(1.f, zeta) / (fabsf(zeta) + sqrtf(fmaf(zeta, zeta, 1.f)));
              cT = df_rsqrt(df_add({1.f, 0.f}, df_two_prod(tt, tt)));
              sT = df_mul_f(cT, tt);
              float pr = gr * ia, pi = -gi * ia;   // e^{-i phi} to FP32, then normalised
              df q = df_rsqrt(df_add(df_two_prod(pr, pr), df_two_prod(pi, pi)));
              phT = {df_mul_f(q, pr), df_mul_f(q, pi)};
              f = 1;
            }
          }
          rcT[p] = cT;
          rsT[p] = sT;
          rph[p] = phT;
        } else {
          double c0 = 1.0, s = 0.0;
          zd ph = {1, 0};
          if (b < c) {
            zd g = J::val(A[a * ce + b]);
            double ag = sqrt(norm2(g));
            double da = J::val(A[a * ce + a]).re, db = J::val(A[b * ce + b]).re;
            if (ag > rtol * sqrt(fabs(da * db)) && ag > 1e-300) {
              double zeta = (db - da) / (2.0 * ag);
              double tt = (zeta >= 0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
              c0 = 1.0 / sqrt(1.0 + tt * tt);
              s = tt * c0;
              ph = {g.re / ag, -g.im / ag};  // e^{-i phi}
              f = 1;
            }
          }
          rcT[p] = c0;
          rsT[p] = s;
          rph[p] = J::from(ph);
        }
        rflag[p] = f;
        rotated |= f;
      }
      __syncthreads();
      // A <- J^dag A J and V <- V J in one pass.  The pairs of a round are disjoint, so the
      // 2 x 2 block of A on the rows of pair p and the columns of pair p' is closed under both
      // rotations: its rows turn with pair p (new_a = c A_a - s e^{i phi} A_b, new_b = s A_a +
      // c e^{i phi} A_b), then its columns with pair p' (phase e^{-i phi}).  A stays Hermitian,
      // so only blocks p <= p' are computed and each p < p' block is mirrored (conjugate
      // transpose) into (p', p); V's columns turn like A's.
      {
        const int nblk = np * (np + 1) / 2;
        for (int e = threadIdx.x; e < nblk + np * ce; e += blockDim.x) {
          if (e < nblk) {
            // block (p, p2), p <= p2, from the packed upper-triangle index
            int p = 0, rem = e;
            while (rem >= np - p) { rem -= np - p; ++p; }
            const int p2 = p + rem;
            const bool fr = rflag[p] != 0, fc = rflag[p2] != 0;
            if (!fr && !fc) continue;
            const int a = pa[round * np + p], b = pb[round * np + p];
            const int a2 = pa[round * np + p2], b2 = pb[round * np + p2];
            T x00 = A[a * ce + a2], x01 = A[a * ce + b2];
            T x10 = A[b * ce + a2], x11 = A[b * ce + b2];
            if (fr) {
              T eph = rph[p];
              if constexpr (DF) eph.im = df_neg(eph.im);
              else eph.im = -eph.im;
              rot_pair(x00, x10, rcT[p], rsT[p], eph);
              rot_pair(x01, x11, rcT[p], rsT[p], eph);
            }
            if (fc) {
              const T mph = rph[p2];
              rot_pair(x00, x01, rcT[p2], rsT[p2], mph);
              rot_pair(x10, x11, rcT[p2], rsT[p2], mph);
            }
            if (p == p2) {
              if constexpr (!DF) {
                // with the exact FP64 angle the rotated pair's coupling is zero
                if (fr) x01 = x10 = J::zero();
              }
            } else {
              A[a2 * ce + a] = J::cj(x00);
              A[b2 * ce + a] = J::cj(x01);
              A[a2 * ce + b] = J::cj(x10);
              A[b2 * ce + b] = J::cj(x11);
            }
            A[a * ce + a2] = x00;
            A[a * ce + b2] = x01;
            A[b * ce + a2] = x10;
            A[b * ce + b2] = x11;
          } else {
            const int ev = e - nblk;
            const int p = ev / ce, k = ev % ce;
            if (!rflag[p]) continue;
            const int a = pa[round * np + p], b = pb[round * np + p];
            T va = Vv[k * ce + a], vb = Vv[k * ce + b];
            rot_pair(va, vb, rcT[p], rsT[p], rph[p]);
            Vv[k * ce + a] = va;
            Vv[k * ce + b] = vb;
          }
        }
      }
      __syncthreads();
    }
    // a barrier that also ORs the flags: every thread takes the same exit decision
    if (!__syncthreads_or(rotated)) break;
  }
  for (int i = threadIdx.x; i < c; i += blockDim.x) dg[i] = J::val(A[i * ce + i]).re;
  __syncthreads();
  // sort eigenvalues descending (stable by index), thread 0; the df64 path compares the
  // normalised (hi, lo) pairs on the FP32 units
  __shared__ int order[MAXC];
  if (threadIdx.x == 0) {
    // stable insertion sort by value descending (ties keep index order)
    for (int i = 0; i < c; ++i) order[i] = i;
    for (int i = 1; i < c; ++i) {
      int key = order[i];
      int j = i - 1;
      if constexpr (DF) {
        df kv = A[key * ce + key].re;
        while (j >= 0 && df_less(A[order[j] * ce + order[j]].re, kv)) {
          order[j + 1] = order[j];
          --j;
        }
      } else {
        double kv = dg[key];
        while (j >= 0 && dg[order[j]] < kv) {
          order[j + 1] = order[j];
          --j;
        }
      }
      order[j + 1] = key;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < c; i += blockDim.x) lam[(size_t)t * c + i] = DF ? gscale[1] * dg[order[i]] : dg[order[i]];
  zd* Vt = Vec + (size_t)t * c * c;
  for (int e = threadIdx.x; e < c * c; e += blockDim.x) {
    int row = e / c, i = e % c;
    Vt[row * c + i] = J::val(Vv[row * ce + order[i]]);
  }
}

constexpr int UK = 64;  // max output columns per update

// out = A V (FP64), optionally with columns scaled by 1 / sqrt(lam)
__global__ void __launch_bounds__(GT) update_kernel(zd* out, int cmax_out,
                                                    const zd* __restrict__ tiles, int cmax, int c,
                                                    const zd* __restrict__ Vec, const double* lam,
                                                    int kout, int scale_inv, int M) {
  extern __shared__ zd sV[];  // [c][kout]
  int t = blockIdx.x;
  const zd* Vt = Vec + (size_t)t * c * c;
  for (int e = threadIdx.x; e < c * kout; e += blockDim.x) {
    int row = e / kout, i = e % kout;
    zd v = Vt[row * c + i];
    if (scale_inv) {
      double l = lam[(size_t)t * c + i];
      double f = l > 0 ? 1.0 / sqrt(l) : 0.0;
      v = f * v;
    }
    sV[e] = v;
  }
  __syncthreads();
  const zd* A = tiles + (size_t)t * cmax * M;
  zd* O = out + (size_t)t * cmax_out * M;
  for (int r = threadIdx.x; r < M; r += blockDim.x) {
    for (int i0 = 0; i0 < kout; i0 += 16) {
      zd acc[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) acc[q] = zd{};
      for (int col = 0; col < c; ++col) {
        zd a0 = A[(size_t)col * M + r];
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (i0 + q < kout) cfma(acc[q], a0, sV[col * kout + i0 + q]);
      }
#pragma unroll
      for (int q = 0; q < 16; ++q)
        if (i0 + q < kout) O[(size_t)(i0 + q) * M + r] = acc[q];
    }
  }
}

// The same on double-float tiles, on the FP32 units with biased accumulators (df64.cuh): a thread
// takes one row and OB output columns at a time, two outputs per packed instruction, and adds the
// columns of A in groups of UDG.  A group's bias comes from Cauchy and Schwarz with the columns
// scaled by their norms n_c (cn, squared, from the Gram kernel): every partial sum of the group's
// A_rc V_ci lies within R F_i, R^2 = sum_c |A_rc|^2 / n_c^2 and F_i^2 = sum_c n_c^2 |V_ci|^2,
// which follows small singular values; the group then joins a (hi, lo) total.  Groups of four
// lose less than one sum over all columns by the square of their number (its bias is larger, and
// it collects more roundings): relative error of a column 4.8e-13 -> 6e-14 at c = 20 (float32
// emulation); the streaming SVD's P is then as exact as with the 12-instruction df_fma or more.
// 16^3x32, four streams (c x kout = 8 x 8, 16 x 12, 20 x 12 twice): 2.52 -> 1.22 ms.
// Each CTA takes `rows` rows of a tile (blockIdx.y picks them).  kp: kout padded to a multiple of
// OB (even).
constexpr int UDT = 128, UDG = 4;
template <int OB>
__global__ void __launch_bounds__(UDT, 4)
update_df_kernel(zdf* out, int cmax_out, const zdf* __restrict__ tiles, int cmax, int c,
                 const zd* __restrict__ Vec, const double* lam, const float* __restrict__ cn,
                 int cld, int kout, int kp, int scale_inv, int M, int rows) {
  extern __shared__ __align__(16) unsigned char smraw_ud[];
  const int ng = (c + UDG - 1) / UDG, cpad = ng * UDG;
  // [cpad][kp / 2][re, im]: (hi, hi, lo, lo) of an output pair
  float4* sV = reinterpret_cast<float4*>(smraw_ud);
  float* sF = reinterpret_cast<float*>(sV + (size_t)cpad * kp);  // [ng][kp] F_i of a group
  float* sI = sF + ng * kp;                                      // [cpad] 1 / n_c
  float* sN = sI + cpad;                                         // [cpad] n_c / max
  __shared__ float nmax;
  const int t = blockIdx.x;
  const zd* Vt = Vec + (size_t)t * c * c;
  if (threadIdx.x < 32) {
    float m = 0.f;
    for (int q = threadIdx.x; q < c; q += 32) m = fmaxf(m, sqrtf(cn[(size_t)t * cld + q]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    // Any positive weights n_c bound the sums, but one far below its column's true norm makes R, and
    // with it the bias of its whole group, too large.  A kept null direction's norm is eigenvalue
    // noise, down to zero (the column itself stays below 1e-7 of the largest), so no weight is below
    // 2^-24 of the largest; columns of that size are below what the Gram matrix resolves.
    for (int q = threadIdx.x; q < cpad; q += 32) {
      const float n = q < c ? fmaxf(sqrtf(cn[(size_t)t * cld + q]), 0x1p-24f * m) : 0.f;
      sI[q] = n > 1e-20f ? 1.0f / n : 0.0f;   // below: n^2 has lost its digits
      sN[q] = m > 0.f ? n / m : 0.f;
    }
    if (threadIdx.x == 0) nmax = m;
  }
  for (int e = threadIdx.x; e < cpad * kp; e += UDT) {
    const int row = e / kp, i = e % kp;
    zdf w = {{0.f, 0.f}, {0.f, 0.f}};
    if (i < kout && row < c) {
      zd v = Vt[row * c + i];
      if (scale_inv) {
        double l = lam[(size_t)t * c + i];
        double f = l > 0 ? 1.0 / sqrt(l) : 0.0;
        v = f * v;
      }
      w = zdf_from(v);
    }
    float* q = reinterpret_cast<float*>(sV + (size_t)row * kp + (i & ~1)) + (i & 1);
    q[0] = w.re.hi; q[2] = w.re.lo; q[4] = w.im.hi; q[6] = w.im.lo;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < ng * kp; e += UDT) {
    const int g = e / kp, i = e % kp;
    float f = 0.f;
    for (int q = g * UDG; q < (g + 1) * UDG; ++q) {
      const float* v = reinterpret_cast<const float*>(sV + (size_t)q * kp + (i & ~1)) + (i & 1);
      const float x = sN[q] * v[0], y = sN[q] * v[4];
      f = fmaf(x, x, fmaf(y, y, f));
    }
    sF[e] = 1.001f * nmax * sqrtf(f);
  }
  __syncthreads();
  const zdf* A = tiles + (size_t)t * cmax * M;
  zdf* O = out + (size_t)t * cmax_out * M;
  const int r1 = min(M, ((int)blockIdx.y + 1) * rows);
  const zdf zero = {{0.f, 0.f}, {0.f, 0.f}};
  for (int r = blockIdx.y * rows + threadIdx.x; r < r1; r += UDT) {
    for (int i0 = 0; i0 < kout; i0 += OB) {
      f32x2 th[OB / 2][2], tl[OB / 2][2];
#pragma unroll
      for (int q = 0; q < OB / 2; ++q) th[q][0] = th[q][1] = tl[q][0] = tl[q][1] = 0;
      zdf a[UDG];
#pragma unroll
      for (int u = 0; u < UDG; ++u) a[u] = u < c ? zdf_ld(A + (size_t)u * M + r) : zero;
      for (int g = 0; g < ng; ++g) {
        float R = 0.f;
        zdfdup ad[UDG];
#pragma unroll
        for (int u = 0; u < UDG; ++u) {
          const float x = sI[g * UDG + u] * a[u].re.hi, y = sI[g * UDG + u] * a[u].im.hi;
          R = fmaf(x, x, fmaf(y, y, R));
          ad[u] = zdf_dup(a[u]);
          const int col = (g + 1) * UDG + u;   // the next group's loads, under this one's products
          a[u] = col < c ? zdf_ld(A + (size_t)col * M + r) : zero;
        }
        R = sqrtf(R);
        const float4* v = sV + (size_t)g * UDG * kp + i0;
#pragma unroll
        for (int q = 0; q < OB / 2; ++q) {
          const float2 F = *reinterpret_cast<const float2*>(sF + g * kp + i0 + 2 * q);
          const f32x2 C = f2_pack(bacc_bias(R * F.x), bacc_bias(R * F.y));
          zbacc2 acc = {};
          acc.re.s = acc.im.s = C;
#pragma unroll
          for (int u = 0; u < UDG; ++u)
            zbacc2_fma(acc, ad[u], {df2_ld(v + u * kp + 2 * q), df2_ld(v + u * kp + 2 * q + 1)});
#pragma unroll
          for (int z = 0; z < 2; ++z) {
            const bacc2& b = z ? acc.im : acc.re;
            const df2 w = df2_two_sum(th[q][z], f2_sub(b.s, C));
            th[q][z] = w.hi;
            tl[q][z] = f2_add(tl[q][z], f2_add(w.lo, f2_add(b.e, b.x)));
          }
        }
      }
#pragma unroll
      for (int q = 0; q < OB; ++q) {
        if (i0 + q < kout) {
          df x[2];
#pragma unroll
          for (int z = 0; z < 2; ++z) {
            const f32x2 h = th[q >> 1][z], l = tl[q >> 1][z];
            x[z] = (q & 1) ? df_two_sum(f2_hi(h), f2_hi(l)) : df_two_sum(f2_lo(h), f2_lo(l));
          }
          reinterpret_cast<float4*>(O)[(size_t)(i0 + q) * M + r] =
              make_float4(x[0].hi, x[0].lo, x[1].hi, x[1].lo);
        }
      }
    }
  }
}

__global__ void __launch_bounds__(GT) phase_kernel(zd* tiles, int cmax, int k, int M) {
  __shared__ double sh[64];
  __shared__ zd q;
  int t = blockIdx.x;
  zd* A = tiles + (size_t)t * cmax * M;
  for (int i = 0; i < k; ++i) {
    zd* col = A + (size_t)i * M;
    double a = 0, b = 0;
    for (int r = threadIdx.x; r < M; r += blockDim.x) {
      a += col[r].re;
      b += col[r].im;
    }
    // block sum
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
    }
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { sh[2 * wid] = a; sh[2 * wid + 1] = b; }
    __syncthreads();
    if (threadIdx.x == 0) {
      double sa = 0, sb = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { sa += sh[2 * w]; sb += sh[2 * w + 1]; }
      double m = sqrt(sa * sa + sb * sb);
      q = m > 0 ? zd{sa / m, -sb / m} : zd{1, 0};
    }
    __syncthreads();
    zd f = q;
    for (int r = threadIdx.x; r < M; r += blockDim.x) col[r] = col[r] * f;
    __syncthreads();
  }
}

// The same canonical phase on double-float tiles, in double-float arithmetic: the column sum
// accumulated error-free on the FP32 units, q = conj(s) / |s| normalised by a Newton
// reciprocal square root, each entry multiplied by q.
// OUT: instead of writing the phased columns back, write them as the outputs P [tile][k][M]
// in complex double, complex float (rounded) and, if Pdf is not null, double-float.
template <bool OUT>
__global__ void __launch_bounds__(GT) phase_df_kernel(zdf* tiles, int cmax, int k, int M, zd* P,
                                                      zf* P32, zdf* Pdf) {
  __shared__ df sh[2][GT / 32];
  __shared__ zdf q;
  int t = blockIdx.x;
  zdf* A = tiles + (size_t)t * cmax * M;
  const df one = {1.0f, 0.0f};
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i = 0; i < k; ++i) {
    zdf* col = A + (size_t)i * M;
    dfacc a{0.f, 0.f}, b{0.f, 0.f};
    for (int r = threadIdx.x; r < M; r += blockDim.x) {
      zdf v = col[r];
      df_fma(a, v.re, one);
      df_fma(b, v.im, one);
    }
    df ar = df_norm(a), br = df_norm(b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      df x = {__shfl_down_sync(0xffffffffu, ar.hi, o), __shfl_down_sync(0xffffffffu, ar.lo, o)};
      df y = {__shfl_down_sync(0xffffffffu, br.hi, o), __shfl_down_sync(0xffffffffu, br.lo, o)};
      ar = df_add(ar, x);
      br = df_add(br, y);
    }
    if (lane == 0) { sh[0][wid] = ar; sh[1][wid] = br; }
    __syncthreads();
    if (threadIdx.x == 0) {
      df sa = {0.f, 0.f}, sb = {0.f, 0.f};
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        sa = df_add(sa, sh[0][w]);
        sb = df_add(sb, sh[1][w]);
      }
      df n2 = df_add(df_mul(sa, sa), df_mul(sb, sb));
      if (n2.hi > 0.f) {
        df inv = df_rsqrt(n2);
        q = {df_mul(sa, inv), df_neg(df_mul(sb, inv))};
      } else {
        q = {one, {0.f, 0.f}};
      }
    }
    __syncthreads();
    zdf f = q;
    const size_t o = ((size_t)t * k + i) * M;
    for (int r = threadIdx.x; r < M; r += blockDim.x) {
      zdf v = col[r];
      zdf w = {df_dot2(v.re, f.re, df_neg(v.im), f.im), df_dot2(v.re, f.im, v.im, f.re)};
      if (OUT) {
        P[o + r] = {df_val_bits(w.re), df_val_bits(w.im)};
        P32[o + r] = {df_to_float(w.re), df_to_float(w.im)};
        if (Pdf) Pdf[o + r] = w;
      } else {
        col[r] = w;
      }
    }
    __syncthreads();
  }
}

// Least-squares interpolation weights (Eq. 9): with the tile A = U Sigma V^dag (V and
// Sigma^2 from the Gram eigen-decomposition), V_c = Sigma_k V_k^dag and Omega = diag(omega),
//   P = A Omega V_c^dag (V_c Omega V_c^dag)^{-1} = A W,  W = Omega V_k B^{-1} Sigma_k^{-1},
//   B = V_k^dag Omega V_k (k x k, Hermitian positive definite for omega > 0).
// One CTA per tile: B in shared memory, inverted by Gauss-Jordan elimination with partial
// pivoting in FP64; W[t][row][i] (leading dimension c, columns i < k) for tile_update.
__global__ void __launch_bounds__(GT) ls_weights_kernel(zd* W, const zd* __restrict__ Vec,
                                                        const double* __restrict__ lam,
                                                        const double* __restrict__ omega, int c,
                                                        int k) {
  extern __shared__ zd lsm[];
  zd* Bm = lsm;                  // [k][2k]: B | I, reduced to I | B^-1
  zd* fc = Bm + (size_t)k * 2 * k;   // [k] the pivot column's factors of one elimination step
  __shared__ int piv;
  const int t = blockIdx.x, w2 = 2 * k;
  const zd* V = Vec + (size_t)t * c * c;   // V[row * c + i]
  for (int e = threadIdx.x; e < k * w2; e += blockDim.x) {
    int a = e / w2, b = e % w2;
    zd s = {0, 0};
    if (b < k) {
      for (int r = 0; r < c; ++r) cfmac(s, V[r * c + a], omega[r] * V[r * c + b]);
    } else {
      s = {(b - k) == a ? 1.0 : 0.0, 0.0};
    }
    Bm[e] = s;
  }
  __syncthreads();
  for (int col = 0; col < k; ++col) {
    if (threadIdx.x == 0) {
      int p = col;
      double m = -1;
      for (int r = col; r < k; ++r) {
        double v = norm2(Bm[r * w2 + col]);
        if (v > m) { m = v; p = r; }
      }
      piv = p;
    }
    __syncthreads();
    if (piv != col)
      for (int b = threadIdx.x; b < w2; b += blockDim.x) {
        zd x = Bm[col * w2 + b];
        Bm[col * w2 + b] = Bm[piv * w2 + b];
        Bm[piv * w2 + b] = x;
      }
    __syncthreads();
    zd pv = Bm[col * w2 + col];
    double d = norm2(pv);
    zd inv = d > 0 ? zd{pv.re / d, -pv.im / d} : zd{0, 0};
    __syncthreads();
    for (int b = threadIdx.x; b < w2; b += blockDim.x) Bm[col * w2 + b] = Bm[col * w2 + b] * inv;
    for (int r = threadIdx.x; r < k; r += blockDim.x) fc[r] = Bm[r * w2 + col];
    __syncthreads();
    for (int e = threadIdx.x; e < k * w2; e += blockDim.x) {
      int r = e / w2, b = e % w2;
      if (r == col) continue;
      Bm[e] = Bm[e] - fc[r] * Bm[col * w2 + b];
    }
    __syncthreads();
  }
  zd* Wt = W + (size_t)t * c * c;
  for (int e = threadIdx.x; e < c * k; e += blockDim.x) {
    int r = e / k, i = e % k;
    zd s = {0, 0};
    for (int a = 0; a < k; ++a) cfma(s, V[r * c + a], Bm[a * w2 + k + i]);
    double l = lam[(size_t)t * c + i];
    double f = l > 0 ? omega[r] / sqrt(l) : 0.0;
    Wt[r * c + i] = f * s;
  }
}

__global__ void sigma_kernel(double* sig, int ldsig, const double* lam, int c, int kk, int ntiles) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ntiles * kk) return;
  int t = e / kk, i = e % kk;
  double l = lam[(size_t)t * c + i];
  sig[(size_t)t * ldsig + i] = l > 0 ? sqrt(l) : 0.0;
}

}  // namespace

int make_blocking(Blocking& B, const int dims[4], const int block[4]) {
  B.nd = 1;
  B.d = 1;
  for (int m = 0; m < 4; ++m) {
    if (block[m] < 1 || dims[m] % block[m] != 0)
      return fail(MG_EINVAL, "aggregate extents must divide the lattice extents");
    B.L[m] = dims[m];
    B.b[m] = block[m];
    B.C[m] = dims[m] / block[m];
    B.nd *= block[m];
    B.d *= B.C[m];
  }
  B.M = 6 * B.nd;
  return MG_OK;
}

template <typename R>
int chiral_gather(void* tiles, int cmax, int col0, const cplx<R>* fields, int nvec,
                  const Blocking& B, cudaStream_t st, bool df64) {
  const unsigned grid = (6u * B.nd * B.d + 255) / 256;
  if (df64) gather_kernel<R, zdf><<<grid, 256, 0, st>>>((zdf*)tiles, cmax, col0, fields, nvec, B);
  else gather_kernel<R, zd><<<grid, 256, 0, st>>>((zd*)tiles, cmax, col0, fields, nvec, B);
  WMG_LAUNCHED();
  return MG_OK;
}
template int chiral_gather<float>(void*, int, int, const zf*, int, const Blocking&, cudaStream_t, bool);
template int chiral_gather<double>(void*, int, int, const zd*, int, const Blocking&, cudaStream_t, bool);

int tile_gram(zd* G, const void* tiles, int cmax, int c, const Blocking& B, cudaStream_t st,
              bool df64, int kd, const double* lam_prev, int c_prev, float* cn, int cld) {
  if (c > MAXC) return fail(MG_EINVAL, "tile_gram: more than 64 columns");
  if (kd < 0 || kd > c || (kd > 0 && (!lam_prev || c_prev < kd)))
    return fail(MG_EINVAL, "tile_gram: bad known-diagonal block");
  const int npairs = c * (c + 1) / 2 - kd * (kd + 1) / 2;
  ProfScope ps(df64 ? "svd_gram_df64" : "svd_gram_fp64", 16.0 * B.M * c * B.d * 2,
               8.0 * B.M * npairs * B.d * 2, st);
  if (df64) {
    // 2 x 2 blocks of column pairs, in equal slices of at most GDF_T per CTA; enough threads that
    // a chunk's column pairs are at most PRE per thread
    const int cp = (c + 1) / 2, J0 = kd / 2;
    const int nt = cp * (cp + 1) / 2 - J0 * (J0 + 1) / 2;
    const int ny = nt < 1 ? 1 : (nt + GDF_T - 1) / GDF_T;
    const int ntc = nt < 1 ? 1 : (nt + ny - 1) / ny;
    const int pre = cp <= 2 * GDF_T * GDF_G / GR ? 2 : 4;
    const int need = std::max(ntc * GDF_G, (GR * cp + pre - 1) / pre);
    const int nth = (need + 31) / 32 * 32;
    const size_t sh = sizeof(float4) * 4 * GR * (cp | 1) + sizeof(float2) * 2 * GDF_G * cp;
    auto kernel = pre == 2 ? gram_df_kernel<2> : gram_df_kernel<4>;
    WMG_TRY(smem_attr(kernel, sh));
    kernel<<<dim3(B.d * 2, ny), nth, sh, st>>>(G, cn, cld, (const zdf*)tiles, cmax, c, B.M, kd,
                                               lam_prev, c_prev, std::max(nt, 1), ntc);
    WMG_LAUNCHED();
    return MG_OK;
  }
  size_t sh = sizeof(zd) * GR * c;
  // one thread per summed pair where they fit one CTA (whole warps, at least two)
  const int nth = npairs >= GT ? GT : std::max(64, (npairs + 31) / 32 * 32);
  int np = (npairs + nth - 1) / nth;
  auto go = [&](auto mp) {
    gram_kernel<decltype(mp)::value><<<B.d * 2, nth, sh, st>>>(G, (const zd*)tiles, cmax, c, B.M,
                                                               kd, lam_prev, c_prev);
  };
  if (np <= 1) go(std::integral_constant<int, 1>{});
  else if (np <= 2) go(std::integral_constant<int, 2>{});
  else if (np <= 4) go(std::integral_constant<int, 4>{});
  else go(std::integral_constant<int, 9>{});
  WMG_LAUNCHED();
  return MG_OK;
}

int tile_eig(double* lam, zd* Vec, zd* G, int c, int ntiles, cudaStream_t st, double rtol,
             bool df64) {
  if (c > MAXC) return fail(MG_EINVAL, "tile_eig: more than 64 columns");
  int ce = c + (c & 1), np = ce / 2;
  // A, V, phases (16-byte complex in both arithmetics), cos, sin (8 bytes), the round-robin
  // schedule and the rotation flags
  size_t sh = sizeof(zd) * (2 * ce * ce + np) + sizeof(double) * 2 * np +
              sizeof(int) * (2 * (ce - 1) * np + np) + 64;
  WMG_TRY(smem_attr(df64 ? jacobi_kernel<true> : jacobi_kernel<false>, sh));
  ProfScope ps(df64 ? "svd_jacobi_df64" : "svd_jacobi_fp64", 32.0 * c * c * ntiles, 0.0, st);
  if (df64) jacobi_kernel<true><<<ntiles, JT, sh, st>>>(lam, Vec, G, c, rtol);
  else jacobi_kernel<false><<<ntiles, JT, sh, st>>>(lam, Vec, G, c, rtol);
  WMG_LAUNCHED();
  return MG_OK;
}

int tile_update(void* out, int cmax_out, const void* tiles, int cmax, int c, const zd* Vec,
                const double* lam, int kout, int scale_inv, const Blocking& B, cudaStream_t st,
                bool df64, const float* cn, int cld) {
  if (kout > UK || c > MAXC) return fail(MG_EINVAL, "tile_update: too many columns");
  ProfScope ps(df64 ? "svd_update_df64" : "svd_update_fp64", 16.0 * B.M * (c + kout) * B.d * 2,
               8.0 * B.M * c * kout * B.d * 2, st);
  if (df64) {
    if (!cn) return fail(MG_EINVAL, "tile_update: no column norms");
    // output columns in equal groups of at most 12 (four floats of totals each stay in registers);
    // 256 rows per CTA: ten waves of CTAs on 1024 tiles of 1536 rows instead of five and a bit
    const int ng = (kout + 11) / 12, per = (kout + ng - 1) / ng;
    const int ob = per <= 4 ? 4 : per <= 6 ? 6 : per <= 8 ? 8 : per <= 10 ? 10 : 12;
    const int kp = (kout + ob - 1) / ob * ob, cg = (c + UDG - 1) / UDG;
    const int rows = 2 * UDT;
    const dim3 grid(B.d * 2, (B.M + rows - 1) / rows);
    const size_t sh = sizeof(zdf) * (size_t)cg * UDG * kp + sizeof(float) * (cg * kp + 2 * cg * UDG);
    auto go = [&](auto kernel) -> int {
      WMG_TRY(smem_attr(kernel, sh));
      kernel<<<grid, UDT, sh, st>>>((zdf*)out, cmax_out, (const zdf*)tiles, cmax, c, Vec, lam, cn,
                                    cld, kout, kp, scale_inv, B.M, rows);
      return MG_OK;
    };
    if (ob == 4) WMG_TRY(go(update_df_kernel<4>));
    else if (ob == 6) WMG_TRY(go(update_df_kernel<6>));
    else if (ob == 8) WMG_TRY(go(update_df_kernel<8>));
    else if (ob == 10) WMG_TRY(go(update_df_kernel<10>));
    else WMG_TRY(go(update_df_kernel<12>));
    WMG_LAUNCHED();
    return MG_OK;
  }
  size_t sh = sizeof(zd) * c * kout;
  WMG_TRY(smem_attr(update_kernel, sh));
  update_kernel<<<B.d * 2, GT, sh, st>>>((zd*)out, cmax_out, (const zd*)tiles, cmax, c, Vec, lam,
                                         kout, scale_inv, B.M);
  WMG_LAUNCHED();
  return MG_OK;
}

int tile_canonical_phase(void* tiles, int cmax, int k, const Blocking& B, cudaStream_t st,
                         bool df64) {
  if (df64) phase_df_kernel<false><<<B.d * 2, GT, 0, st>>>((zdf*)tiles, cmax, k, B.M, nullptr, nullptr, nullptr);
  else phase_kernel<<<B.d * 2, GT, 0, st>>>((zd*)tiles, cmax, k, B.M);
  WMG_LAUNCHED();
  return MG_OK;
}

int tile_phase_outputs(zd* P, zf* P32, zdf* Pdf, void* tiles, int cmax, int k,
                       const Blocking& B, cudaStream_t st) {
  phase_df_kernel<true><<<B.d * 2, GT, 0, st>>>((zdf*)tiles, cmax, k, B.M, P, P32, Pdf);
  WMG_LAUNCHED();
  return MG_OK;
}

int tile_ls_weights(zd* W, const zd* Vec, const double* lam, const double* omega, int c, int k,
                    int ntiles, cudaStream_t st) {
  if (k > c || c > MAXC) return fail(MG_EINVAL, "tile_ls_weights: bad sizes");
  size_t sh = sizeof(zd) * ((size_t)k * 2 * k + k);
  WMG_TRY(smem_attr(ls_weights_kernel, sh));
  ls_weights_kernel<<<ntiles, GT, sh, st>>>(W, Vec, lam, omega, c, k);
  WMG_LAUNCHED();
  return MG_OK;
}

int tile_sigma(double* sig, int ldsig, const double* lam, int c, int kk, int ntiles,
               cudaStream_t st) {
  int tot = ntiles * kk;
  sigma_kernel<<<(tot + 255) / 256, 256, 0, st>>>(sig, ldsig, lam, c, kk, ntiles);
  WMG_LAUNCHED();
  return MG_OK;
}

}  // namespace wmg
