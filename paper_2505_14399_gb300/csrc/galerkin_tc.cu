// Forward-hop blocks of the Galerkin coarse operator (Eq. 5) on the tcgen05 tensor cores, at
// double-float accuracy.
//
// CTA (j, mu) accumulates, over the fine sites x of aggregate j, C[a][b] =
// sum_{x,r} conj(Pt[x][r][a]) Ch[x][r][b] (the staged reconstruction-folded P(x) and the
// spin-projected, colour-transported P(x + mu), as in the FP32-unit kernel of coarse.cu).
// Every staged double-float entry v satisfies |v| < 2 (|P| <= 1 entrywise for orthonormal
// columns; |U h| <= sqrt(3) for unitary U and |h| <= 1), so it is written exactly enough as
// fixed-point digits in base 256,
//     v = sum_{i < NS} s_i 2^{-6-8i},  s_i integers, |s_i| <= 128,  NS = 7
// (error at most 2^-55),
// each digit exact in fp16 (kept as s_i 2^-8).  A product of digit planes is an integer matrix
// product: fp16 x fp16 tensor-core MMAs with FP32 accumulation are exact while the partial sums stay
// below 2^24, which holds for three staging batches (7 digit pairs x 3 x 48 stacked rows x
// 128^2 = 0.984 2^24).  Digit pairs i + j = d of the same weight 2^{-12-8d} share FP32
// accumulator columns; pairs with i + j >= NS (weight below 2^-68) are dropped.  After every
// third batch the exact FP32 sums are scaled by their weights (exact) and added to double-float
// accumulators with error-free two-sums, so the result carries double-float accuracy (~2^-48
// relative), not fp16's.
//
// A batch is NB = 4 sites: 24 staged rows, three groups of eight.  One tcgen05.mma covers one
// group (K = 16: eight rows against the real parts of Pt, the same eight against the imaginary
// parts) and one digit i of Ch:
//   A, M rows = columns b of (Re C | Im C): the planes (Ch_re, Ch_im, -Ch_re) of a digit lie one
//      after the other, so K half 0 reads (Ch_re | Ch_im) and K half 1, one plane further,
//      (Ch_im | -Ch_re): three stored planes serve as a 2 x 2 block;
//   B, N columns = the digits j = 0 .. 6 - i of Pt side by side, so that the pair (i, j) lands in
//      accumulator columns (i + j) 8 T4 .. without an instruction per pair.
// Operands are MN-major without swizzle: a core matrix is eight rows of eight columns (128
// contiguous bytes), written by one warp store (8 rows x 4 column pairs of packed fp16) without
// bank conflicts, at addresses that are constants of the thread.  Rows and columns of padding
// hold garbage; it stays in accumulator rows and columns that nothing reads.
//
// The planes are double-buffered: a warp of its own issues a batch's products and the others go
// on to stage the next batch, so that only staging (double-float colour transport and digit
// split, on two columns at once in packed FP32 instructions) and every third batch's fold are on
// the critical path.  With warp-level mma.sync (bf16 digits) the products, their ldmatrix reads
// and the accumulators lived in the staging warps, which met at two barriers per batch: 2.57 ms
// at 16^3x32, k = 12 (blocks of 4^4) and 18.6 ms at 16^3x64, k = 24 (2x2x2x4); here 1.42 and
// 9.25 ms.  (These and the times below hold the finish pass and the range flag's round trip, 0.05
// and 1.5 ms; the contraction alone takes 1.37 and 7.74 ms.)  Bound now by the staging warps' FP32 and issue slots (k = 12: about 4700 cycles a
// batch, two CTAs per SM), for small blocks also by a CTA's start, four folds and two outputs (k =
// 24, 32 sites: together a third of its 78 000 cycles).  P(x) is loaded between the transport and
// the digits: before the transport its eight registers made the loop spill (1.54 against 1.48 ms,
// 9.5 against 9.3 ms with the rest as it is).  Tried and slower: Ch and Pt staged by different
// warps (2.27 ms, k = 12), a persistent grid whose feeder warp copies and issues everything (2.5
// ms: the feeder is a serial chain; 3.4 ms with 96-byte bulk copies).

#include "bits.cuh"
#include "common.cuh"
#include "df64.cuh"
#include "galerkin.cuh"
#include "internal.h"
#include "tcdigits.cuh"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace wmg {

namespace {

constexpr int TC_MAXT4 = 6;            // 2k <= 48

constexpr int NB = 4;                  // fine sites staged per batch
constexpr int NG = NB * 6 / 8;         // groups of eight staged rows per batch
constexpr int FOLD = 3;                // batches between folds
constexpr int TC_WAIT = 1 << 18;       // polls of a completion barrier before giving up
static_assert(NB * 6 == 8 * NG, "whole groups of rows");
static_assert((long)TC_NS * FOLD * NB * 6 * 2 * 128 * 128 < (1l << 24), "exact FP32 sums");

// Per column-tile count T4 (columns of a plane: 8 T4 >= 2k).
template <int T4>
struct TcCfg {
  static constexpr int NR = 8 * T4;
  static constexpr int ITEMS = NG * T4;                     // staging warps
  // and one that issues the products (T4 = 2: a staging warp does, three CTAs of seven warps
  // would not keep their registers)
  static constexpr int WARPS = T4 == 2 ? ITEMS : ITEMS + 1;
  static constexpr int M = 2 * NR <= 64 ? 64 : 128;         // MMA rows (2 NR used)
  static constexpr int NPAD = M == 128 ? 16 : 8;            // granule of N
  // column groups of the fold: four warps (a quarter of the accumulator lanes each) per group
  static constexpr int FG = T4 == 6 ? 4 : T4 >= 3 ? 2 : 1;
  static constexpr int CPG = NR / FG;
  static constexpr int DCOLS = (TC_NS * NR + NPAD - 1) / NPAD * NPAD;
  static constexpr int TCOLS = DCOLS <= 64 ? 64 : DCOLS <= 128 ? 128 : DCOLS <= 256 ? 256 : 512;
  // resident CTAs per SM asked of the register allocator; MINB TCOLS <= 512
  static constexpr int MINB = T4 == 1 ? 4 : T4 == 2 ? 3 : T4 == 3 ? 2 : 1;
  static constexpr int PLANE = T4 * 128;                    // bytes of one plane of 8 rows
  static constexpr int A_BYTES = TC_NS * NG * 3 * PLANE;
  static constexpr int B_BYTES = NG * 2 * TC_NS * PLANE;
  static constexpr int BUF = A_BYTES + B_BYTES;
  static constexpr int NRP = NR + 4;   // raw row stride: 3 NRP = 4 mod 8 sixteen-byte units
  static constexpr int RAW = NB * 6 * NRP + NB * 9;         // double-float complex values
  static_assert(WARPS >= 4 * FG && CPG % 4 == 0 && MINB * TCOLS <= 512, "fold groups");
};

// dynamic shared memory: two digit buffers (A then B planes; the padding rows' reads past A's
// end stay inside B, those past B's end inside what follows), two raw buffers (P(x + mu)
// components, U), the per-site tables
template <int T4>
constexpr size_t tc_fixed_bytes() {
  return 2 * (size_t)TcCfg<T4>::BUF + 2 * sizeof(zdf) * (size_t)TcCfg<T4>::RAW;
}
inline size_t tc_cta_bytes(int t4, int nd) {
  const size_t tab = sizeof(int) * 3 * (size_t)nd;
  switch (t4) {
    case 1: return tc_fixed_bytes<1>() + tab;
    case 2: return tc_fixed_bytes<2>() + tab;
    case 3: return tc_fixed_bytes<3>() + tab;
    case 4: return tc_fixed_bytes<4>() + tab;
    case 5: return tc_fixed_bytes<5>() + tab;
    default: return tc_fixed_bytes<6>() + tab;
  }
}

__device__ __forceinline__ zdf2 zdf2_pair(const zdf& a, const zdf& b) {
  return {{f2_pack(a.re.hi, b.re.hi), f2_pack(a.re.lo, b.re.lo)},
          {f2_pack(a.im.hi, b.im.hi), f2_pack(a.im.lo, b.im.lo)}};
}
// a / b for 0 <= a < 2^20, b > 0: the quotient of the floats is within 2^-22 a / b of
// (a + 1/2) / b, which is at least 1 / (2 b) away from an integer
__device__ __forceinline__ int small_div(int a, int b) {
  return (int)__fdividef((float)a + 0.5f, (float)b);
}
__device__ __forceinline__ df2 df2_xor(df2 a, f32x2 m) { return {a.hi ^ m, a.lo ^ m}; }
__device__ __forceinline__ f32x2 sign_mask(bool neg) { return neg ? 0x8000000080000000ull : 0ull; }

template <int T4>
__global__ void __launch_bounds__(32 * TcCfg<T4>::WARPS, TcCfg<T4>::MINB)
galerkin_tc_kernel(zd* Op, zd* Xpart, const zdf* __restrict__ Pdf, int k,
                   const zdf* __restrict__ Ldf, HopGeom g, Blocking B, int* range_flag) {
  using C = TcCfg<T4>;
  constexpr int NR = C::NR, PLANE = C::PLANE, NRP = C::NRP;
  constexpr int NT = 32 * C::WARPS;
  extern __shared__ __align__(128) unsigned char tc_raw[];
  zdf* raw = reinterpret_cast<zdf*>(tc_raw + 2 * (size_t)C::BUF);   // [2][RAW]
  const int nd = B.nd;
  int* ty = reinterpret_cast<int*>(raw + 2 * (size_t)C::RAW);   // P offset of y = x + mu, column 0
  int* tx = ty + nd;                                            // P offset of x
  int* tu = tx + nd;                                            // 2 (link offset of x) + sign
  __shared__ uint64_t mbar[2];
  __shared__ uint32_t s_tmem;
  const int n2k = 2 * k, KP = (k + 1) & ~1;
  const int j = blockIdx.x, mu = blockIdx.y, dir = 2 * mu;
  const double coef = -g.kappa * g.w[mu];
  const int ne = n2k * n2k;
  const int M = B.M;
  const size_t V = (size_t)B.nd * B.d;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  bool bad = false, dead = false;

  // ---- per-site tables, hops inside the aggregate first (pass 0), then the crossing ones: a
  // hop crosses when its local coordinate mu is the last one
  const int b0 = B.b[0], b1 = B.b[1], b2 = B.b[2];
  const int lstride = mu == 0 ? 1 : mu == 1 ? b0 : mu == 2 ? b0 * b1 : b0 * b1 * b2;
  const int bm = mu == 0 ? b0 : mu == 1 ? b1 : mu == 2 ? b2 : B.b[3];
  const int n1 = small_div(nd, bm), n0 = nd - n1;
  int jc[4];
  jc[0] = j % B.C[0];
  int jr = j / B.C[0];
  jc[1] = jr % B.C[1]; jr /= B.C[1];
  jc[2] = jr % B.C[2]; jc[3] = jr / B.C[2];
  const int bstride = mu == 0 ? 1 : mu == 1 ? B.C[0] : mu == 2 ? B.C[0] * B.C[1]
                                                             : B.C[0] * B.C[1] * B.C[2];
  const int Cm = mu == 0 ? B.C[0] : mu == 1 ? B.C[1] : mu == 2 ? B.C[2] : B.C[3];
  const int jm = mu == 0 ? jc[0] : mu == 1 ? jc[1] : mu == 2 ? jc[2] : jc[3];
  const int bcm = mu == 0 ? g.bc[0] : mu == 1 ? g.bc[1] : mu == 2 ? g.bc[2] : g.bc[3];
  const bool last = jm == Cm - 1;   // crossing hops leave the lattice
  const int jn = last ? j - (Cm - 1) * bstride : j + bstride;
  const int tj = 2 * j * k * M, tn = 2 * jn * k * M;
  const int x0 = jc[0] * b0 +
                 B.L[0] * (jc[1] * b1 + B.L[1] * (jc[2] * b2 + B.L[2] * jc[3] * B.b[3]));
  for (int l = tid; l < nd; l += NT) {
    const int r1 = small_div(l, b0), r2 = small_div(r1, b1), r3 = small_div(r2, b2);
    const int c0 = l - r1 * b0, c1 = r1 - r2 * b1, c2 = r2 - r3 * b2;
    const int cm = mu == 0 ? c0 : mu == 1 ? c1 : mu == 2 ? c2 : r3;
    // hi: the coordinates above mu, lo: below (as a local index)
    const int hi = mu == 0 ? r1 : mu == 1 ? r2 : mu == 2 ? r3 : 0;
    const int lo = l - lstride * (cm + bm * hi);
    const bool cross = cm == bm - 1;
    const int e = cross ? n0 + lo + lstride * hi : lo + lstride * (cm + (bm - 1) * hi);
    const int x = x0 + c0 + B.L[0] * (c1 + B.L[1] * (c2 + B.L[2] * r3));
    tx[e] = tj + l * 6;
    ty[e] = cross ? tn + (l - (bm - 1) * lstride) * 6 : tj + (l + lstride) * 6;
    tu[e] = 2 * (x * 9) + ((cross && last && bcm < 0) ? 1 : 0);
  }
  if (wid == C::WARPS - 1) tc5_alloc(&s_tmem, C::TCOLS);
  if (tid == 0) {
    mbar_init(&mbar[0], 1);
    mbar_init(&mbar[1], 1);
    mbar_init_fence();
  }
  tc5_fence_before();
  __syncthreads();
  tc5_fence_after();
  const uint32_t tmem = s_tmem;

  // ---- constants of this thread
  // copies: pieces (16 bytes) of P(x + mu), two per thread: site of the batch, source and
  // destination offset (h < 0: none); then the links, one piece for the first 9 NB threads
  int cph[2], cps[2], cpd[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int p = tid + u * NT;
    const int h = small_div(p, 6 * n2k), rem = p - h * 6 * n2k;
    const int col = rem / 6, part = rem - 6 * col;
    const int chi = col >= k, i = col - (chi ? k : 0);
    // pair q = chi KP / 2 + i / 2 keeps its columns in slots q and KP + q: the staging threads,
    // which take consecutive pairs, read consecutive 16-byte slots
    const int q = chi * (KP / 2) + (i >> 1);
    cph[u] = h < NB ? h : -1;
    cps[u] = col * M + part;
    cpd[u] = (h * 6 + part) * NRP + q + ((i & 1) ? KP : 0);
  }
  // staging: a column pair sq (one chirality: padded to an even count) of one batch row
  // Warp w runs on scheduler w % 4, so both CTAs of an SM would give their ninth item to the same
  // one (T4 = 3): the accumulator allocation tells them apart (1.48 -> 1.42 ms at k = 12).
  const int cta = (int)((tmem & 0xffffu) / C::TCOLS);
  const int item = T4 == 3 && wid >= 8 ? 8 + (((wid - 8) ^ cta) & 1) : wid;
  const int sg = item / T4, pg = item % T4, lrow = lane >> 2, sq = 4 * pg + (lane & 3);
  const bool dn = sq >= KP / 2;
  const int si = 2 * (sq - (dn ? KP / 2 : 0)), scol = (dn ? k : 0) + si;
  const int scol1 = si + 1 < k ? M : 0;   // an odd k's last pair repeats its column
  const int slot1 = si + 1 < k ? KP : 0;
  // Row of a batch: site, component row of the half spinor read and the power i^rot.  Columns of
  // chirality 1 take i sigma_mu psi_dn (mu < 3) or -psi_dn (mu = 3): one component of the pair
  // times a power of i, which commutes with the colour transport.
  struct Row {
    int h, spin, cc;
    bool odd;          // odd powers swap (re, im)
    f32x2 sgx, sgy;    // signs of the two results
  };
  auto row_of = [&](int row) {
    Row w;
    w.h = row / 6;
    const int r = row - 6 * w.h, ss = r / 3;
    w.cc = r - 3 * ss;
    w.spin = 3 * ((!dn || mu >= 2) ? ss : 1 - ss);
    const int rot = !dn ? 0 : mu == 0 ? 1 : mu == 1 ? 2 * ss : mu == 2 ? 1 + 2 * ss : 2;
    w.odd = rot & 1;
    w.sgx = sign_mask(rot == 1 || rot == 2);
    w.sgy = sign_mask(rot & 2);
    return w;
  };
  unsigned char* const sA = tc_raw + 3 * PLANE * sg + 128 * pg + 4 * lane;
  unsigned char* const sB = tc_raw + C::A_BYTES + 2 * TC_NS * PLANE * sg + 128 * pg + 4 * lane;
  const bool stager = item < C::ITEMS && sq < KP;
  const Row w = row_of(8 * sg + lrow);
  // fold: quarter of the lanes, column group
  const int fq = wid & 3, fg = wid >> 2;
  const int frow = C::M == 128 ? 32 * fq + lane : lane < 16 ? 16 * fq + lane : 2 * NR;
  const bool folder = fg < C::FG && (C::M == 128 ? 32 : 16) * fq < 2 * NR;
  const uint32_t ftm = tmem + ((uint32_t)(32 * fq) << 16) + (uint32_t)(fg * C::CPG);

  const int nb0 = (n0 + NB - 1) / NB, nbt = nb0 + (n1 + NB - 1) / NB;
  auto batch = [&](int t, int& e0, int& nb) {
    e0 = t < nb0 ? t * NB : n0 + (t - nb0) * NB;
    nb = min(NB, (t < nb0 ? n0 : nd) - e0);
  };
  // issue the raw inputs of batch t (cp.async, one group)
  auto prefetch = [&](int t) {
    if (t < nbt) {
      int e0, nb;
      batch(t, e0, nb);
      zdf* dst = raw + (size_t)(t & 1) * C::RAW;
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (cph[u] >= 0 && cph[u] < nb) cp_async16(dst + cpd[u], Pdf + ty[e0 + cph[u]] + cps[u]);
      if (tid < 9 * nb) {
        const int h = tid / 9;
        cp_async16(dst + NB * 6 * NRP + tid,
                   Ldf + (size_t)mu * V * 9 + (tu[e0 + h] >> 1) + (tid - 9 * h));
      }
    }
    cp_async_commit();
  };

  prefetch(0);
  prefetch(1);
  cp_async_wait<1>();
  __syncthreads();

  dfacc2 dacc[C::CPG / 2];
#pragma unroll
  for (int c = 0; c < C::CPG / 2; ++c) dacc[c] = {0, 0};
  // wait until the products of batch t are done (bounded: a timeout raises the range flag)
  auto wait_mma = [&](int t) {
    if (!dead && !mbar_wait(&mbar[t & 1], (t >> 1) & 1, TC_WAIT)) dead = true;
  };
  // add the exact sums, scaled by 2^{-12-8d}, to the double-float accumulators
  auto fold = [&]() {
    tc5_fence_after();
    if (folder) {
#pragma unroll
      for (int c4 = 0; c4 < C::CPG / 4; ++c4) {
        float v[TC_NS][4];
#pragma unroll
        for (int d = 0; d < TC_NS; ++d) tc5_ld4(v[d], ftm + d * NR + 4 * c4);
        tc5_wait_ld();
        float wgt = 16.0f;   // 2^{-12-8d} 2^16
#pragma unroll
        for (int d = 0; d < TC_NS; ++d) {
          const f32x2 w2 = f2_dup(wgt);
#pragma unroll
          for (int e = 0; e < 2; ++e)
            acc_fma(dacc[2 * c4 + e], f2_pack(v[d][2 * e], v[d][2 * e + 1]), w2);
          wgt *= 1.0f / 256.0f;
        }
      }
    }
    tc5_fence_before();
  };
  // a pass's blocks: accumulators -> shared memory (a digit buffer that is not in use) -> Op /
  // Xpart
  auto output = [&](int pass, int buf) {
    df* sOut = reinterpret_cast<df*>(tc_raw + (size_t)buf * C::BUF);   // [2 NR][NR + 1]
    constexpr int LO = NR + 1;
    static_assert(sizeof(df) * 2 * NR * LO <= (size_t)C::BUF, "blocks fit a digit buffer");
    if (folder && frow < 2 * NR) {
      df* o = sOut + (size_t)frow * LO + fg * C::CPG;
#pragma unroll
      for (int c = 0; c < C::CPG / 2; ++c) {
        const df2 v = df2_norm(dacc[c]);
        o[2 * c] = {f2_lo(v.hi), f2_lo(v.lo)};
        o[2 * c + 1] = {f2_hi(v.hi), f2_hi(v.lo)};
        dacc[c] = {0, 0};
      }
    }
    __syncthreads();
    zd* out = pass == 1 ? Op + ((size_t)j * 9 + 1 + dir) * ne
                        : Xpart + ((size_t)mu * B.d + j) * ne;
    const int db = small_div(NT, n2k), da = NT - db * n2k;
    int b = small_div(tid, n2k), a = tid - b * n2k;
    for (int e = tid; e < ne; e += NT) {
      const int sb = b < k ? b : KP + b - k, sa = a < k ? a : KP + a - k;
      const df re = sOut[(size_t)sb * LO + sa], im = sOut[(size_t)(NR + sb) * LO + sa];
      out[e] = {coef * df_val_bits(re), coef * df_val_bits(im)};   // column-major
      b += db;
      a += da;
      if (a >= n2k) { a -= n2k; ++b; }
    }
  };
  int nacc = 0;   // batches in the accumulators
  for (int t = 0; t < nbt; ++t) {
    const int buf = t & 1;
    int e0, nb;
    batch(t, e0, nb);
    unsigned char* const A = sA + (size_t)buf * C::BUF;
    unsigned char* const Bp = sB + (size_t)buf * C::BUF;
    const bool act = stager && w.h < nb;
    if (t >= 2) wait_mma(t - 2);   // its products have read this digit buffer
    // Ch (spin-projected, transported P(x + mu)) and Pt (reconstruction-folded P(x)) in
    // double-float, written as digit planes: every digit of the two columns of a pair goes
    // out as one 32-bit store
    if (act) {
      const zdf* rw = raw + (size_t)buf * C::RAW;
      const zdf* U = rw + NB * 6 * NRP + w.h * 9 + w.cc * 3;
      const zdf* Py = rw + (size_t)(w.h * 6 + w.spin) * NRP + sq;
      const f32x2 neg = sign_mask(tu[e0 + w.h] & 1);
      dfacc2 tre, tim;
#pragma unroll
      for (int c2 = 0; c2 < 3; ++c2) {
        const zdf u = U[c2];
        const zdf2 v = zdf2_pair(Py[c2 * NRP], Py[c2 * NRP + slot1]);
        const df2 ur = df2_dup(u.re), ui = df2_dup(u.im), mi = df2_dup(df_neg(u.im));
        const f32x2 mr = f2_dup(-u.re.hi);
        dfacc2_fma(tre, ur, mr, v.re, c2 == 0);
        dfacc2_fma(tre, mi, ui.hi, v.im, false);
        dfacc2_fma(tim, ur, mr, v.im, c2 == 0);
        dfacc2_fma(tim, ui, mi.hi, v.re, false);
      }
      // P(x), used last: straight from global memory, swapped for odd powers of i
      const float2* px = reinterpret_cast<const float2*>(Pdf + (size_t)tx[e0 + w.h] +
                                                         (size_t)scol * M + w.spin + w.cc);
      const float2 pxv[4] = {__ldg(px + w.odd), __ldg(px + !w.odd), __ldg(px + 2 * scol1 + w.odd),
                             __ldg(px + 2 * scol1 + !w.odd)};
      const df2 nre = df2_norm(tre), nim = df2_norm(tim);
      bad |= !(tc_in_range(nre) && tc_in_range(nim));
      unsigned dr[TC_NS], di[TC_NS];
      tc_digits2(df2_xor(w.odd ? nim : nre, w.sgx ^ neg), dr);
      tc_digits2(df2_xor(w.odd ? nre : nim, w.sgy ^ neg), di);
#pragma unroll
      for (int i = 0; i < TC_NS; ++i) {
        unsigned char* a = A + i * NG * 3 * PLANE;
        *reinterpret_cast<unsigned*>(a) = dr[i];
        *reinterpret_cast<unsigned*>(a + PLANE) = di[i];
        *reinterpret_cast<unsigned*>(a + 2 * PLANE) = dr[i] ^ 0x80008000u;   // -Ch_re
      }
      const df2 ptr = df2_xor({f2_pack(pxv[0].x, pxv[2].x), f2_pack(pxv[0].y, pxv[2].y)}, w.sgx);
      const df2 pti = df2_xor({f2_pack(pxv[1].x, pxv[3].x), f2_pack(pxv[1].y, pxv[3].y)}, w.sgy);
      bad |= !(tc_in_range(ptr) && tc_in_range(pti));
      tc_digits2(ptr, dr);
      tc_digits2(pti, di);
#pragma unroll
      for (int i = 0; i < TC_NS; ++i) {
        *reinterpret_cast<unsigned*>(Bp + i * PLANE) = dr[i];
        *reinterpret_cast<unsigned*>(Bp + (TC_NS + i) * PLANE) = di[i];
      }
    } else if (stager) {   // a short batch: its unused rows are zero in every plane
#pragma unroll
      for (int i = 0; i < TC_NS; ++i) {
#pragma unroll
        for (int p = 0; p < 3; ++p)
          *reinterpret_cast<unsigned*>(A + (i * NG * 3 + p) * PLANE) = 0u;
        *reinterpret_cast<unsigned*>(Bp + i * PLANE) = 0u;
        *reinterpret_cast<unsigned*>(Bp + (TC_NS + i) * PLANE) = 0u;
      }
    }
    cp_async_wait<0>();     // batch t + 1's inputs
    fence_proxy_async();    // the digit planes, to the tensor core's reads
    __syncthreads();
    prefetch(t + 2);        // its buffer was read by this batch's staging
    if (nacc == FOLD || t == nb0) {
      if (nacc > 0) {
        wait_mma(t - 1);
        fold();
      }
      if (t == nb0) output(0, buf ^ 1);
      nacc = 0;
      __syncthreads();           // the accumulators (and the output's buffer) have been read
    }
    if (item == C::WARPS - 1 && lane == 0) {
      tc5_fence_after();
      constexpr uint32_t idesc = tc5_idesc_f16_mn(C::M, 0);
      const uint32_t a0 = smem_addr(tc_raw + (size_t)buf * C::BUF), b0 = a0 + C::A_BYTES;
      // MN-major, no swizzle: 128 bytes between column octets, one plane (A) or the real and
      // imaginary planes of all digits (B) between the two halves of K
      const uint64_t ad = tc5_desc(a0, PLANE, 128), bd = tc5_desc(b0, TC_NS * PLANE, 128);
#pragma unroll 1
      for (int gq = 0; gq < NG; ++gq) {
#pragma unroll
        for (int i = 0; i < TC_NS; ++i) {
          const uint64_t da = ad + (uint64_t)((i * NG + gq) * 3 * (PLANE >> 4));
          const uint64_t db = bd + (uint64_t)(gq * 2 * TC_NS * (PLANE >> 4));
          const int n = ((TC_NS - i) * NR + C::NPAD - 1) / C::NPAD * C::NPAD;
          const uint32_t acc = (nacc > 0 || gq > 0 || i > 0) ? 1u : 0u;
          const int n1st = n > 256 ? 256 : n;
          tc5_mma(tmem + i * NR, da, db, idesc | tc5_idesc_n(n1st), acc);
          if (n > 256)
            tc5_mma(tmem + i * NR + 256, da, db + (uint64_t)(256 / 8 * (128 >> 4)),
                    idesc | tc5_idesc_n(n - 256), acc);
        }
      }
      tc5_commit(&mbar[buf]);
    }
    ++nacc;
  }
  wait_mma(nbt - 1);
  fold();
  output(1, nbt & 1);
  __syncthreads();
  if (wid == C::WARPS - 1) tc5_dealloc(tmem, C::TCOLS);
  if (bad || dead) atomicExch(range_flag, 1);
}

template <int T4>
int launch_tc(zd* Op, zd* Xpart, const zdf* Pdf, int k, const zdf* Ldf, const HopGeom& g,
              const Blocking& B, int* range_flag, cudaStream_t st) {
  size_t sh = tc_cta_bytes(T4, B.nd);
  WMG_TRY(smem_attr(galerkin_tc_kernel<T4>, sh));
  if (TcCfg<T4>::MINB > 1)   // room for several CTAs: the largest shared-memory carveout
    WMG_CUDA(cudaFuncSetAttribute(galerkin_tc_kernel<T4>,
                                  cudaFuncAttributePreferredSharedMemoryCarveout,
                                  (int)cudaSharedmemCarveoutMaxShared));
  galerkin_tc_kernel<T4><<<dim3(B.d, 4), 32 * TcCfg<T4>::WARPS, sh, st>>>(Op, Xpart, Pdf, k, Ldf, g,
                                                                          B, range_flag);
  WMG_LAUNCHED();
  return MG_OK;
}

constexpr size_t kTcSmemMax = (size_t)227 * 1024 - 1024;

}  // namespace

bool galerkin_tc_supported(int k, const Blocking& B) {
  if (k < 1 || (k + 3) / 4 > TC_MAXT4) return false;
  // shared memory of one CTA, and tile and link offsets that fit an int
  const int t4 = (k + 3) / 4;
  return tc_cta_bytes(t4, B.nd) <= kTcSmemMax &&
         (size_t)B.d * 2 * k * B.M < ((size_t)1 << 31) &&
         (size_t)B.d * B.nd * 18 < ((size_t)1 << 31);
}

double galerkin_tc_issued_flops(int k, const Blocking& B) {
  // digit-plane products issued: 28 digit pairs of an M x (8 T4) x (12 NB) real product per
  // batch and hop direction, about n_d / NB + 1 batches per CTA
  const int t4 = (k + 3) / 4;
  const double m = t4 <= 4 ? 64.0 : 128.0;
  return 2.0 * m * (8.0 * t4) * (12.0 * NB) * 28.0 * 4.0 * B.d * ((double)B.nd / NB + 1.0);
}

int galerkin_hops_tc(zd* Op, zd* Xpart, const zdf* Pdf, int k, const zdf* Ldf, const HopGeom& g,
                     const Blocking& B, int* range_flag, cudaStream_t st) {
  switch ((k + 3) / 4) {
    case 1: return launch_tc<1>(Op, Xpart, Pdf, k, Ldf, g, B, range_flag, st);
    case 2: return launch_tc<2>(Op, Xpart, Pdf, k, Ldf, g, B, range_flag, st);
    case 3: return launch_tc<3>(Op, Xpart, Pdf, k, Ldf, g, B, range_flag, st);
    case 4: return launch_tc<4>(Op, Xpart, Pdf, k, Ldf, g, B, range_flag, st);
    case 5: return launch_tc<5>(Op, Xpart, Pdf, k, Ldf, g, B, range_flag, st);
    case 6: return launch_tc<6>(Op, Xpart, Pdf, k, Ldf, g, B, range_flag, st);
    default: return fail(MG_EINVAL, "galerkin (tensor pipe): 2k > 48");
  }
}

}  // namespace wmg
