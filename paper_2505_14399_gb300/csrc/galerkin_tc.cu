// Forward-hop blocks of the Galerkin coarse operator (Eq. 5) on the tensor pipe, at
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
// each digit exact in bfloat16.  A product of digit planes is an integer matrix product:
// bf16 x bf16 tensor-core MMAs with FP32 accumulation are exact while the partial sums stay
// below 2^24, which holds for three staging batches (7 digit pairs x 3 x 48 stacked rows x
// 128^2 = 0.984 2^24).  Digit pairs i + j = d of the same weight 2^{-12-8d} share an FP32
// accumulator; pairs with i + j >= NS (weight below 2^-68) are dropped.  After every third batch
// (every one where a warp's tiles leave no registers for that) the exact FP32 sums are
// scaled by their weights (exact) and added to double-float accumulators with error-free
// two-sums, so the result carries double-float accuracy (~2^-48 relative), not bf16's.
//
// The complex product is one real GEMM per digit pair: with K = 6 NB rows (NB sites x 6 half-
// spinor rows) per batch, stacked as k' = [re rows | im rows] (12 NB),
//     A'[b'][k'] : rows b < 2k = (Ch_re | Ch_im), rows 2k + b = (Ch_im | -Ch_re),
//     B'[a][k']  : (Pt_re | Pt_im),
// C'[b'][a] = sum_k' A'[b'][k'] B'[a][k'] gives Re C[a][b] (b' = b) and Im C[a][b] (b' = 2k+b).
// mma.sync m16n8k16 (row.col) tiles: 16 rows b' x 8 columns a, one warp per tile.  The digit
// planes are stored k'-major (SA[k'][b'], SB[k'][a]) so that staging threads with consecutive
// columns write consecutive addresses, and read with ldmatrix .trans; every row stride is an
// odd number of 16-byte units, so the eight rows of an ldmatrix phase hit distinct banks.
// A batch is NB = 4 sites: three k' steps of 16 stacked rows.  For 2k <= 24 two CTAs (three and
// four for 2k <= 16 and 8) share an SM, so one CTA's staging overlaps the other's products.
//
// Staging (double-float colour transport, digit split) runs on two adjacent columns at once in
// packed FP32 instructions.  It was the bound, with the per-batch fold: 3.11 ms at 16^3x32, k =
// 12, tensor pipe a fifth busy; 2.57 ms now (21.7 -> 19.8 ms at 16^3x64, k = 24), where the FP32
// pipe is busy 61 % of the time, the tensor pipe 27 %, and the warps wait for the barriers
// between staging and products.
#include <cuda_bf16.h>

#include "common.cuh"
#include "df64.cuh"
#include "galerkin.cuh"
#include "internal.h"
#include "tcdigits.cuh"
#include "tma.cuh"

namespace wmg {

namespace {

constexpr int TC_MAXT4 = 6;            // 2k <= 48

constexpr int NB = 4;                  // fine sites staged per batch
constexpr int KB = NB * 6;             // staged rows per batch
constexpr int TCK = 2 * KB;            // stacked real rows per batch

// Per column-tile count T4 (2k <= 8 T4): tiles, warps.
template <int T4>
struct TcCfg {
  static constexpr int NTILES = T4 * T4;
  static constexpr int MAXW = T4 == 6 ? 18 : 16;           // warps that take tiles, at most
  static constexpr int TPW = (NTILES + MAXW - 1) / MAXW;   // tiles per warp
  static constexpr int NW = (NTILES + TPW - 1) / TPW;
  // warps of the CTA: one staging item (row, column pair) per thread
  static constexpr int WARPS = NW > 3 * T4 ? NW : 3 * T4;
  // resident CTAs per SM asked of the register allocator
  static constexpr int MINB = T4 == 1 ? 4 : T4 == 2 ? 3 : T4 == 3 ? 2 : 1;
  // batches between folds
  static constexpr int FOLD = TPW == 1 ? 3 : 1;
};

// Row strides (bf16) of the k'-major digit planes: odd multiples of 8 (16 bytes).
__host__ __device__ constexpr int tc_lda(int t4) { return 16 * t4 + 8; }
__host__ __device__ constexpr int tc_ldb(int t4) { return 8 * t4 + ((t4 & 1) ? 0 : 8); }
__host__ __device__ constexpr size_t tc_smem(int t4) {
  return sizeof(__nv_bfloat16) * (size_t)TC_NS * TCK * (tc_lda(t4) + tc_ldb(t4));
}

// Shared memory of one CTA beyond the digit planes: two raw input buffers (P(x + mu) and P(x)
// column segments of 6 double-float values, U_mu(x)) and the per-site tables.
// Raw P segments are stored [site][6 components][column slot], rows padded to 8 T4 + 1 slots
// so that the copies (consecutive components of one column) spread over the banks; column b
// sits in slot (b odd ? k : 0) + b / 2, so that the staging threads, which take the column
// pairs (2q, 2q + 1) for consecutive q, read consecutive 16-byte slots.
__host__ __device__ constexpr int tc_nrp(int t4) { return 8 * t4 + 1; }
__host__ __device__ constexpr size_t tc_raw_bytes(int t4) {
  return sizeof(zdf) * 2 * ((size_t)2 * NB * 6 * tc_nrp(t4) + NB * 9);
}
__host__ __device__ inline size_t tc_table_bytes(int nd) { return sizeof(int) * 8 * (size_t)nd + 16; }
__host__ __device__ inline size_t tc_cta_bytes(int t4, int nd) {
  return tc_smem(t4) + tc_raw_bytes(t4) + tc_table_bytes(nd);
}

// i^rot x for the two halves of x, rot 0 .. 3 per half (sign changes and swaps: exact)
__device__ __forceinline__ zdf2 rot_i(zdf2 x, int rot0, int rot1) {
  auto one = [](float re, float im, int rot, float& ore, float& oim) {
    const float a = (rot & 1) ? im : re, b = (rot & 1) ? re : im;
    // rot 1: (-im, re), 2: (-re, -im), 3: (im, -re)
    const unsigned sa = (rot == 1 || rot == 2) ? 0x80000000u : 0u;
    const unsigned sb = (rot & 2) ? 0x80000000u : 0u;
    ore = __uint_as_float(__float_as_uint(a) ^ sa);
    oim = __uint_as_float(__float_as_uint(b) ^ sb);
  };
  float h[4], l[4];
  one(f2_lo(x.re.hi), f2_lo(x.im.hi), rot0, h[0], h[1]);
  one(f2_hi(x.re.hi), f2_hi(x.im.hi), rot1, h[2], h[3]);
  one(f2_lo(x.re.lo), f2_lo(x.im.lo), rot0, l[0], l[1]);
  one(f2_hi(x.re.lo), f2_hi(x.im.lo), rot1, l[2], l[3]);
  return {{f2_pack(h[0], h[2]), f2_pack(l[0], l[2])}, {f2_pack(h[1], h[3]), f2_pack(l[1], l[3])}};
}
__device__ __forceinline__ zdf2 zdf2_pair(const zdf& a, const zdf& b) {
  return {{f2_pack(a.re.hi, b.re.hi), f2_pack(a.re.lo, b.re.lo)},
          {f2_pack(a.im.hi, b.im.hi), f2_pack(a.im.lo, b.im.lo)}};
}

template <int T4>
__global__ void __launch_bounds__(32 * TcCfg<T4>::WARPS, TcCfg<T4>::MINB)
galerkin_tc_kernel(zd* Op, zd* Xpart, const zdf* __restrict__ Pdf, int k,
                   const zdf* __restrict__ Ldf, HopGeom g, Blocking B, int* range_flag) {
  using C = TcCfg<T4>;
  constexpr int NR = 8 * T4;                  // columns a (>= 2k)
  constexpr int NTILES = C::NTILES;
  constexpr int NW = C::NW;
  constexpr int TPW = C::TPW;                 // tiles per warp
  constexpr int K = TCK;
  constexpr int ND = TC_NS;                   // digit-pair weights d = i + j < NS
  constexpr int LDA = tc_lda(T4), LDB = tc_ldb(T4);
  extern __shared__ __align__(16) unsigned char tc_raw[];
  __nv_bfloat16* SA = reinterpret_cast<__nv_bfloat16*>(tc_raw);   // [NS][K][LDA]
  __nv_bfloat16* SB = SA + (size_t)TC_NS * K * LDA;                // [NS][K][LDB]
  constexpr int NRP = tc_nrp(T4);
  zdf* sPy = reinterpret_cast<zdf*>(tc_raw + tc_smem(T4));     // [2][NB][6][NRP]
  zdf* sPx = sPy + (size_t)2 * NB * 6 * NRP;                       // [2][NB][6][NRP]
  zdf* sU = sPx + (size_t)2 * NB * 6 * NRP;                        // [2][NB][9]
  const int nd = B.nd;
  int* tx = reinterpret_cast<int*>(tc_raw + tc_smem(T4) + tc_raw_bytes(T4));   // site x
  int* toy = tx + nd;      // P offset of (2 j(y)) k M, y = x + mu
  int* tox = toy + nd;     // P offset of (2 j(x)) k M
  int* tly = tox + nd;     // local site of y, x
  int* tlx = tly + nd;
  int* tng = tlx + nd;     // antiperiodic sign of the hop
  int* sel = tng + nd;     // [2][nd]: local sites of pass 0, then of pass 1
  __shared__ int nsel[2];
  const int n2k = 2 * k;
  const int j = blockIdx.x, mu = blockIdx.y, dir = 2 * mu;
  const double coef = -g.kappa * g.w[mu];
  const int ne = n2k * n2k;
  const int M = B.M;
  const size_t V = (size_t)B.nd * B.d;
  const int lane = threadIdx.x & 31;
  const int wid = threadIdx.x >> 5;   // tile slot; warps beyond NW only stage
  const size_t plane16 = tc_smem(T4) / 16;   // 16-byte chunks of SA + SB
  bool bad = false;

  // ---- per-site tables of this aggregate, and the two passes' site lists
  for (int l = threadIdx.x; l < nd; l += blockDim.x) {
    int x = B.site(j, l);
    int c[4];
    c[0] = x % g.L[0];
    int r = x / g.L[0];
    c[1] = r % g.L[1]; r /= g.L[1];
    c[2] = r % g.L[2]; c[3] = r / g.L[2];
    bool wrap = c[mu] == g.L[mu] - 1;
    int y = wrap ? x - (g.L[mu] - 1) * g.stride[mu] : x + g.stride[mu];
    int jy, ly, jx, lx;
    B.block_of(y, &jy, &ly);
    B.block_of(x, &jx, &lx);
    tx[l] = x;
    toy[l] = 2 * jy * k * M;
    tox[l] = 2 * jx * k * M;
    tly[l] = ly;
    tlx[l] = lx;
    tng[l] = (wrap && g.bc[mu] < 0) ? 1 : 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // a hop crosses the aggregate when the local coordinate mu is the last one
    int n0 = 0, n1 = 0;
    const int bm = B.b[mu];
    int stride = 1;
    for (int m = 0; m < mu; ++m) stride *= B.b[m];
    for (int l = 0; l < nd; ++l) {
      bool cross = (l / stride) % bm == bm - 1;
      if (cross) sel[nd + n1++] = l;
      else sel[n0++] = l;
    }
    nsel[0] = n0;
    nsel[1] = n1;
  }
  __syncthreads();

  const int pps = 2 * n2k * 6 + 9;   // 16-byte pieces per site (one double-float complex each)
  // q / pps as a multiply-high: with m = ceil(2^32 / pps), floor(q m / 2^32) = floor(q / pps)
  // whenever q pps < 2^32 (here q < NB pps and pps <= 585)
  const unsigned pps_m = 0xffffffffu / (unsigned)pps + 1u;
  // staging assignment: thread -> column pair sq of staged rows srow0, srow0 + srows, ...
  // (threads beyond srows * k stage nothing)
  const int srows = blockDim.x / k;
  const int sq = threadIdx.x % k;
  const int srow0 = threadIdx.x < srows * k ? threadIdx.x / k : 6 * NB;
  // issue the raw inputs of batch b of pass p into buffer buf (cp.async, one group)
  auto prefetch = [&](int p, int b, int buf) {
    const int* ls = sel + p * nd;
    const int h0 = b * NB;
    const int nb = min(NB, nsel[p] - h0);
    for (int q = threadIdx.x; q < nb * pps; q += blockDim.x) {
      int h = (int)__umulhi((unsigned)q, pps_m), rem = q - h * pps;
      int l = ls[h0 + h];
      const zdf* src;
      zdf* dst;
      if (rem < n2k * 6) {
        int bcol = rem / 6, part = rem - bcol * 6;
        src = Pdf + (size_t)toy[l] + (size_t)bcol * M + tly[l] * 6 + part;
        dst = sPy + (((size_t)buf * NB + h) * 6 + part) * NRP + ((bcol & 1) ? k : 0) + (bcol >> 1);
      } else if (rem < 2 * n2k * 6) {
        rem -= n2k * 6;
        int bcol = rem / 6, part = rem - bcol * 6;
        src = Pdf + (size_t)tox[l] + (size_t)bcol * M + tlx[l] * 6 + part;
        dst = sPx + (((size_t)buf * NB + h) * 6 + part) * NRP + ((bcol & 1) ? k : 0) + (bcol >> 1);
      } else {
        int part = rem - 2 * n2k * 6;
        src = Ldf + ((size_t)mu * V + tx[l]) * 9 + part;
        dst = sU + ((size_t)buf * NB + h) * 9 + part;
      }
      cp_async16(dst, src);
    }
    cp_async_commit();
  };

  for (int pass = 0; pass < 2; ++pass) {  // 0: hops inside the aggregate, 1: crossing hops
    // zero both digit planes: padding rows and columns stay zero for the whole pass
    for (size_t e = threadIdx.x; e < plane16; e += blockDim.x)
      reinterpret_cast<uint4*>(tc_raw)[e] = make_uint4(0u, 0u, 0u, 0u);
    dfacc2 dacc[TPW][2];
    float acc[TPW][ND][4];
#pragma unroll
    for (int t = 0; t < TPW; ++t) dacc[t][0] = dacc[t][1] = {0, 0};
    const int nbat = (nsel[pass] + NB - 1) / NB;
    if (nbat > 0) prefetch(pass, 0, 0);
    for (int b = 0; b < nbat; ++b) {
      const int buf = b & 1;
      if (b + 1 < nbat) {
        prefetch(pass, b + 1, buf ^ 1);   // its buffer was last read by batch b - 1's staging
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();   // batch b's inputs are in; every warp finished batch b - 1's products
      const int nb = min(NB, nsel[pass] - b * NB);
      const int* ls = sel + pass * nd + b * NB;
      if (nb < NB) {
        // a short batch: its unused stacked rows k' are zero in every digit plane
        const int k0 = nb * 6, kn = KB - k0;
        for (int e = threadIdx.x; e < TC_NS * 2 * kn * (LDA + LDB); e += blockDim.x) {
          int col = e % (LDA + LDB), rr = e / (LDA + LDB);
          int i = rr / (2 * kn), q = rr % (2 * kn);
          int kk = (q < kn) ? k0 + q : KB + k0 + (q - kn);
          if (col < LDA) SA[((size_t)i * K + kk) * LDA + col] = __float2bfloat16_rn(0.0f);
          else SB[((size_t)i * K + kk) * LDB + (col - LDA)] = __float2bfloat16_rn(0.0f);
        }
      }
      // stage from shared memory: Ch (spin-projected, transported P(x + mu)) and Pt
      // (reconstruction-folded P(x)) in double-float, written as digit planes; a thread takes
      // the adjacent columns 2q and 2q + 1 of one row, so every digit goes out as a packed
      // bf16 pair (one 32-bit store)
      const zdf* py = sPy + (size_t)buf * NB * 6 * NRP;
      const zdf* px = sPx + (size_t)buf * NB * 6 * NRP;
      const zdf* pu = sU + (size_t)buf * NB * 9;
      for (int rr = srow0; rr < nb * 6; rr += srows) {
        const int h = rr / 6, r = rr - 6 * (rr / 6);
        const int q = sq;
        const int s = r / 3, cc = r - 3 * s;
        const zdf* U = pu + h * 9 + cc * 3;
        const bool neg = tng[ls[h]] != 0;
        // columns of chirality 1 take i sigma_mu psi_dn (mu < 3) or -psi_dn (mu = 3): one
        // component of the pair times a power of i, which commutes with the colour transport
        const zdf* Py = py + (size_t)h * 6 * NRP + q;
        const zdf* Px = px + (size_t)h * 6 * NRP + q;
        int pi[2], rot[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const bool up = 2 * q + u < k;
          pi[u] = u * k + NRP * 3 * ((up || mu >= 2) ? s : 1 - s);   // column slot, spin row
          rot[u] = up ? 0 : mu == 0 ? 1 : mu == 1 ? 2 * s : mu == 2 ? 1 + 2 * s : 2;
        }
        dfacc2 tre, tim;
#pragma unroll
        for (int c2 = 0; c2 < 3; ++c2) {
          const zdf u = U[c2];
          const zdf2 v = zdf2_pair(Py[pi[0] + c2 * NRP], Py[pi[1] + c2 * NRP]);
          const df2 ur = df2_dup(u.re), ui = df2_dup(u.im), mi = df2_dup(df_neg(u.im));
          const f32x2 mr = f2_dup(-u.re.hi);
          dfacc2_fma(tre, ur, mr, v.re, c2 == 0);
          dfacc2_fma(tre, mi, ui.hi, v.im, false);
          dfacc2_fma(tim, ur, mr, v.im, c2 == 0);
          dfacc2_fma(tim, ui, mi.hi, v.re, false);
        }
        const int kk = h * 6 + r;
        f32x2 dr[TC_NS], di[TC_NS];
        {
          const int n2 = neg ? 2 : 0;
          const zdf2 ch = rot_i({df2_norm(tre), df2_norm(tim)}, (rot[0] + n2) & 3, (rot[1] + n2) & 3);
          bad |= !(tc_in_range(ch.re) && tc_in_range(ch.im));
          tc_digits2(ch.re, dr);
          tc_digits2(ch.im, di);
#pragma unroll
          for (int i = 0; i < TC_NS; ++i) {
            __nv_bfloat16* a0 = SA + ((size_t)i * K + kk) * LDA;          // re rows k
            __nv_bfloat16* a1 = SA + ((size_t)i * K + KB + kk) * LDA;     // im rows k
            const unsigned pr = tc_pack(dr[i]), pim = tc_pack(di[i]);
            *reinterpret_cast<unsigned*>(a0 + 2 * q) = pr;
            *reinterpret_cast<unsigned*>(a1 + 2 * q) = pim;
            *reinterpret_cast<unsigned*>(a0 + n2k + 2 * q) = pim;
            *reinterpret_cast<unsigned*>(a1 + n2k + 2 * q) = pr ^ 0x80008000u;   // -Ch_re
          }
        }
        {
          const zdf2 pt = rot_i(zdf2_pair(Px[pi[0] + cc * NRP], Px[pi[1] + cc * NRP]), rot[0], rot[1]);
          bad |= !(tc_in_range(pt.re) && tc_in_range(pt.im));
          tc_digits2(pt.re, dr);
          tc_digits2(pt.im, di);
#pragma unroll
          for (int i = 0; i < TC_NS; ++i) {
            *reinterpret_cast<unsigned*>(SB + ((size_t)i * K + kk) * LDB + 2 * q) = tc_pack(dr[i]);
            *reinterpret_cast<unsigned*>(SB + ((size_t)i * K + KB + kk) * LDB + 2 * q) =
                tc_pack(di[i]);
          }
        }
      }
      __syncthreads();
      // exact digit-plane products of this warp's output tiles, folded into double-float
      const bool start = b % C::FOLD == 0, fold = b % C::FOLD == C::FOLD - 1 || b == nbat - 1;
#pragma unroll
      for (int tt = 0; tt < TPW; ++tt) {
        const int tile = wid + tt * NW;
        if (wid < NW && tile < NTILES) {
          const int mt = tile / T4, nt = tile % T4;
          if (start) {
#pragma unroll
            for (int d = 0; d < ND; ++d)
#pragma unroll
              for (int e = 0; e < 4; ++e) acc[tt][d][e] = 0.0f;
          }
          // ldmatrix .trans row addresses: A matrices (b' 0-7 | 8-15) x (k 0-7 | 8-15) in the
          // order of the A fragment, B matrices k 0-7 | 8-15 for columns a of this tile
          const int mq = lane >> 3, rr = lane & 7;
          const __nv_bfloat16* arow = SA + (size_t)(8 * (mq >> 1) + rr) * LDA + 16 * mt + 8 * (mq & 1);
          const __nv_bfloat16* brow = SB + (size_t)(8 * (mq & 1) + rr) * LDB + 8 * nt;
#pragma unroll 1
          for (int ks = 0; ks < K / 16; ++ks) {
            unsigned bfr[TC_NS][2];
#pragma unroll
            for (int i = 0; i < TC_NS; ++i)
              ldm_x2t(bfr[i], brow + ((size_t)i * K + 16 * ks) * LDB);
#pragma unroll
            for (int i = 0; i < TC_NS; ++i) {
              unsigned af[4];
              ldm_x4t(af, arow + ((size_t)i * K + 16 * ks) * LDA);
#pragma unroll
              for (int jd = 0; jd < TC_NS; ++jd)
                if (i + jd < ND) mma_bf16(acc[tt][i + jd], af, bfr[jd]);
            }
          }
          if (fold) {
            // weights 2^{-12-8d}: exact FP32 constants
            float wgt = 1.0f / 4096.0f;
#pragma unroll
            for (int d = 0; d < ND; ++d) {
              const f32x2 w2 = f2_dup(wgt);
#pragma unroll
              for (int e = 0; e < 2; ++e)
                acc_add(dacc[tt][e], f2_mul(f2_pack(acc[tt][d][2 * e], acc[tt][d][2 * e + 1]), w2));
              wgt *= 1.0f / 256.0f;
            }
          }
        }
      }
    }
    // this pass's blocks: tiles -> shared memory (over the digit planes) -> Op / Xpart
    __syncthreads();
    df* sOut = reinterpret_cast<df*>(tc_raw);   // [16 T4][NR]
#pragma unroll
    for (int tt = 0; tt < TPW; ++tt) {
      const int tile = wid + tt * NW;
      if (wid < NW && tile < NTILES) {
        const int mt = tile / T4, nt = tile % T4;
        const int row = 16 * mt + (lane >> 2), col = 8 * nt + 2 * (lane & 3);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const df2 v = df2_norm(dacc[tt][e]);
          df* o = sOut + (size_t)(row + 8 * e) * NR + col;
          o[0] = {f2_lo(v.hi), f2_lo(v.lo)};
          o[1] = {f2_hi(v.hi), f2_hi(v.lo)};
        }
      }
    }
    __syncthreads();
    zd* out = pass == 1 ? Op + ((size_t)j * 9 + 1 + dir) * ne
                        : Xpart + ((size_t)mu * B.d + j) * ne;
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
      int b = e / n2k, a = e % n2k;
      df re = sOut[(size_t)b * NR + a], im = sOut[(size_t)(n2k + b) * NR + a];
      out[(size_t)b * n2k + a] = {coef * df_val(re), coef * df_val(im)};   // column-major
    }
    __syncthreads();
  }
  if (bad) atomicExch(range_flag, 1);
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
  // shared memory of one CTA, and tile offsets that fit an int
  const int t4 = (k + 3) / 4;
  return tc_cta_bytes(t4, B.nd) <= kTcSmemMax &&
         (size_t)B.d * 2 * k * B.M < ((size_t)1 << 31);
}

double galerkin_tc_issued_flops(int k, const Blocking& B) {
  // bf16 digit-plane products issued: 28 digit pairs of a (16 T4) x (8 T4) x (12 NB) real
  // product per batch and hop direction, about n_d / NB + 1 batches per CTA
  const int t4 = (k + 3) / 4;
  return 2.0 * (16.0 * t4) * (8.0 * t4) * (12.0 * NB) * 28.0 * 4.0 * B.d *
         ((double)B.nd / NB + 1.0);
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
