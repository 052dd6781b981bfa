// dm_split.cu -- the Legendre stages (spin-weighted synthesis and analysis of
// the dual messenger step, Algorithm 1) in FP64-class or FP32-class arithmetic
// as exact integer products on the tensor cores.
//
// Method: the error-free splitting of a matrix product (Ozaki, Ogita, Oishi &
// Rump 2012).  Each operand is written, relative to a power-of-two scale, as a
// fixed-point number of S digits in base 512, every digit an integer in
// [-256, 256] and so exact in BF16.  A product of two digits is at most 2^16,
// and the FP32 accumulators of tcgen05.mma (kind::f16) add integers exactly up
// to 2^24.  Digit products of equal weight (i + j = k) share one accumulator;
// after every 128 terms the accumulators are added to 64-bit integers, so no
// rounding happens between the splitting of the inputs (2^-54 of the scale for
// S = 6, 2^-27 for S = 3) and the final conversion, but for the dropped
// products i + j > S (i + j >= S for S = 3).
//
// Is 128 terms short enough?  Weights 0 and 1 hold 1 and 2 products a term:
// 2^24 at most.  From weight 4 on a unit is 2^-52 of the largest term, so a sum
// beyond 2^24 would cost no more than FP64 does.  Weights 2 and 3 (3 and 4
// products) could pass 2^24 only where three digits of both operands keep their
// signs over a chunk; a digit that varies adds up as noise, near 2^20.  Harmonic
// functions of few values on a ring (orders n / 4, n / 8, ... against a map of
// that period) reach 0.82 of 2^24 over all amplitudes.  lambda_00 is the same
// on every ring: against a constant map it reaches 1.17 (0.6 % of amplitudes pass
// 1).  Its tile of the analysis therefore drains every 64 terms, where weights 2
// and 3 cannot pass; every other function changes over 128 rings by far more
// than a unit of its third digit (relative 2^-26).
// S = 6 serves DM_FP64, DM_FLOAT_FLOAT, the anchors and the diagnostics; S = 3
// (27 bits against the 24 of FP32) the mixed mode's batches outside the BF16
// kernels.
//
// Why: this GPU's FP64 pipe runs 2 FMA a clock and SM (1.26 TFLOP/s measured).
// The recurrence kernels spend 23 FP64 instructions per (l, m, ring pair) and
// right-hand side; here the Legendre values are kept as digits (36 bytes per
// triple for the three functions) and the contraction costs 12 x 26 BF16
// multiply-adds on a pipe a thousand times wider.
//
// The functions and columns.  With P+- = Q +- iU and a+- = -(aE +- i aB):
//   P+_N = sum_l a+ p,          P-_S = sum_l sg a- p,
//   P+_S = sum_l a+ q,          P-_N = sum_l sg a- q,
// p = 2lambda, q = sg -2lambda, sg = (-1)^{l+m} (the mirror ring's parity), and
//   T_N = sum_l aT lambda,      T_S = sum_l sg aT lambda.
// So every function meets four real columns per right-hand side, X = (a+ re,
// im, sg a- re, im) for p and q alike.  The analysis is the transpose:
//   g+ = sum_r p P+_N + q P+_S,   sg g- = sum_r p P-_S + q P-_N,
//   aE = -(g+ + g-) / 2,  aB = -(g+ - g-) / 2i,  aT = sum_r lambda (T_N + sg T_S).
//
// Table: digit planes of 8 x 8 core matrices (8 multipoles x 8 ring pairs, the
// pairs contiguous, 128 bytes).  The synthesis reads them as an MN-major
// operand (rows = ring pairs, K = multipoles), the analysis as a K-major one
// (rows = multipoles, K = ring pairs), both by one 4-D TMA box per K step, so
// one table serves both directions.  Row scale: one exponent per (m, ring
// pair) for lambda and one for p, q, that of the largest value over l, so that
// rows far below the others (high orders near the poles) keep their relative
// precision down to the 2^-600 where the recurrence begins to count; the K
// range of a tile starts at the first multipole or ring pair whose digits are
// not all zero (18 % of the K steps are left out at nside 512 / lmax 1024).
//
// Kernel: one persistent CTA per SM.  Warp 8 streams the operands (TMA), warp
// 9 issues the MMAs, warps 0-7 drain the accumulators.  The B operand holds
// the digits of the columns one below the other, so that digit i of A meets
// digits 0 .. G-1-i of B in one MMA whose result lands on the accumulators
// i .. G-1 (G = 7 weights for S = 6).  Two accumulator sets alternate every 128
// terms, so draining overlaps the next MMAs.
#include <algorithm>
#include <cmath>
#include <vector>

#include "dm_internal.h"
#include "dm_rec.cuh"
#include "dm_split.cuh"
#include "dm_tc.cuh"

namespace dmwf {

using namespace tc;

constexpr int SPLIT_ROWS = 128;        // rows of a tile (ring pairs or multipoles)
constexpr int SPLIT_CHUNK = 8;         // K steps of 16 per drain (half of it in the analysis tile of l = 0)
constexpr int SPLIT_MIN_EXP = -600;    // smallest row scale
// Drain warps: 16 where the columns divide (the drain is latency bound).  Both
// stages and the rings' products alike, a solve at nside 128 with 8 right-hand
// sides 24.6 -> 23.2 ms, alm2map at nside 256 with 64 8.73 -> 7.98 ms.
__host__ __device__ constexpr int split_drain_warps(int nq) { return nq % 2 == 0 ? 16 : 8; }
__host__ __device__ constexpr int split_threads(int nq) { return 32 * (split_drain_warps(nq) + 2); }
constexpr int SPLIT_MAX_STAGES = 12;

// One tile of work: 128 rows of one order and part, K steps [k0, k0 + nk) of each function.
struct SplitTile {
  int m, row;      // order; row tile
  int part;        // 0: temperature, 1: polarisation
  int k0, nk;      // first K step and number of K steps
  int trow;        // table row (octet of multipoles) of the tile's first row octet (analysis) or K step 0 (synthesis)
  int xstep;       // K step 0 of the tile in the column scratch, in steps (of one column tile)
  int xlen;        // K steps of the whole order (scratch stride between column tiles)
  int chunk;       // K steps per drain
};

// Launches of both directions for one kind of batch: device tile lists, and
// per launch (m0, m1, first tile, tiles).
struct SplitLaunches {
  int nct = 0, n0 = 0, S = 0;
  SplitTile *tiles[2] = {nullptr, nullptr};
  std::vector<int> launch[2];
};

// Digit tables of a plan, shared by the views that serving makes of it.
struct SplitTables {
  int16_t *esc = nullptr;          // [2][mmax + 1][npairs] row exponents (lambda; p, q)
  unsigned char *dig = nullptr;    // [6][3 rows_cap][npoct][128 bytes]
  int64_t rows_cap = 0;            // table rows (octets of multipoles) per function of the largest slab
  std::vector<int> slab;           // slab boundaries in m
  bool full = false;               // one slab that stays valid
  int npoct = 0;
  const int *roff_dev = nullptr;   // first table row of each order, behind esc
  CUtensorMap map_syn[2], map_ana[2];  // [0]: all six digits, [1]: the first three
  std::vector<int> roff;           // [mmax + 2] first table row of each order
  std::vector<int> ks_syn, ks_ana; // first K step per (part, m, row tile), from lfirst
  unsigned char *x = nullptr;      // column digits of one launch: six digits of every right-hand side, whatever runs
  int *xexp = nullptr;             // [mmax + 1][batch][2] column exponents, behind x
  int batch = 0;                   // the plan's right-hand sides (its views have one)
  std::vector<SplitLaunches> cuts; // launches per kind of batch (a plan's own and its one-RHS views') and S: four at most
  int64_t bytes = 0;               // device memory held
  bool disabled = false;           // the plan's owner chose the direct kernels
  Shortage shortage;               // the tables did not fit: the direct kernels run
};

namespace {

__device__ __forceinline__ int64_t sp_alm_base(int lmax, int m) { return (int64_t)m * (2 * lmax + 1 - m) / 2; }

// ------------------------------------------------------------------ tables

// Row exponents and the first multipole with a non-zero digit (l - m): one
// thread per ring pair and order.  The running maximum of a row grows through
// buckets of 16 exponents; the multipole at which it entered each is kept, so
// that one pass of the recurrence finds the first value within 2^-55 of the
// final maximum and above 2^floor_exp (to a bucket, never late).
constexpr int SC_BUCKETS = 40;  // exponents -600 .. 39
__global__ void __launch_bounds__(64) k_split_scale(const PairDev *__restrict__ pairs,
                                                    const RecCoef *__restrict__ rec,
                                                    const double *__restrict__ seed,
                                                    const int *__restrict__ seed_exp, int16_t *__restrict__ esc,
                                                    uint16_t *__restrict__ lfirst, int lmax, int mmax, int npairs,
                                                    int floor_exp) {
  __shared__ uint16_t enter[2][SC_BUCKETS][64];
  __shared__ RecCoef sc[64];
  const int m = blockIdx.y, t = threadIdx.x, p = min((int)blockIdx.x * 64 + t, npairs - 1);
  const double x = pairs[p].x;
  Rec s;
  rec_init(s, seed, seed_exp, m, p, npairs);
  const int64_t base = sp_alm_base(lmax, m);
  int e[2] = {SPLIT_MIN_EXP - 1, SPLIT_MIN_EXP - 1}, top[2] = {-1, -1};
  for (int lc = m; lc <= lmax; lc += 64) {
    __syncthreads();
    if (lc + t <= lmax) sc[t] = rec[base + lc + t + 1];
    __syncthreads();
    for (int j = 0; j < min(64, lmax + 1 - lc); ++j) {
      const int l = lc + j;
      if (s.S == 0) {
        const int v[2] = {exp_of(s.l0), max(exp_of(s.p0), exp_of(s.q0))};
#pragma unroll
        for (int f = 0; f < 2; ++f)
          if (v[f] > e[f]) {
            e[f] = v[f];
            const int bk = min(SC_BUCKETS - 1, (v[f] - SPLIT_MIN_EXP) >> 4);
            while (top[f] < bk) enter[f][++top[f]][t] = (uint16_t)(l - m);
          }
      }
      if (l < lmax) rec_advance(s, sc[j], x, m, l, seed, p, npairs);
    }
  }
  if ((int)blockIdx.x * 64 + t >= npairs) return;
  for (int f = 0; f < 2; ++f) {
    const int64_t o = ((int64_t)f * (mmax + 1) + m) * npairs + p;
    esc[o] = (int16_t)max(e[f], SPLIT_MIN_EXP);
    const int thr = max(e[f] - 55, floor_exp), bk = max(0, (thr - SPLIT_MIN_EXP) >> 4);
    lfirst[o] = (uint16_t)(top[f] < 0 || e[f] < thr ? lmax - m + 1 : enter[f][min(bk, top[f])][t]);
  }
}

// First K step of every row tile, in units of 16: grid (orders, 2), ks[part][m][0 .. npt) for the
// synthesis (multipoles of the tile's first visible row), then [npt, npt + nlt) for the analysis
// (first ring pair visible at the tile's last multipole).
__global__ void k_split_ks(const uint16_t *__restrict__ lfirst, int *__restrict__ ks, int mmax, int npairs, int npt,
                           int nlt) {
  const int m = blockIdx.x, part = blockIdx.y;
  const uint16_t *f = lfirst + ((int64_t)part * (mmax + 1) + m) * npairs;
  int *o = ks + ((int64_t)part * (mmax + 1) + m) * (npt + nlt);
  for (int t = threadIdx.x; t < npt + nlt; t += blockDim.x) {
    if (t < npt) {
      int lo = 65535;
      for (int q = 128 * t; q < min(npairs, 128 * t + 128); ++q) lo = min(lo, (int)f[q]);
      o[t] = lo / 16;
    } else {
      const int l = 128 * (t - npt) + 127;
      int q = 0;
      while (q < npairs && f[q] > l) ++q;
      o[t] = q / 16;
    }
  }
}

constexpr int GEN_PST = 144;                      // staged bytes per (digit, pair octet): 128 + padding
constexpr int GEN_STAGE = 3 * SPLIT_S * 16 * GEN_PST;

// Digits of the orders [m0, m0 + gridDim.y): one thread per ring pair runs the
// FP64 recurrence; eight multipoles of 128 pairs are staged in shared memory
// and written as whole core matrices.
__global__ void __launch_bounds__(128) k_split_gen(const PairDev *__restrict__ pairs,
                                                   const RecCoef *__restrict__ rec,
                                                   const double *__restrict__ seed,
                                                   const int *__restrict__ seed_exp,
                                                   const int16_t *__restrict__ esc, unsigned char *__restrict__ dig,
                                                   int lmax, int mmax, int npairs, int npoct, int m0, int row0,
                                                   const int *__restrict__ roff, int64_t rows_cap,
                                                   const SolveState *__restrict__ state, int batch) {
  extern __shared__ __align__(16) unsigned char stage[];
  __shared__ RecCoef sc[64];
  if (state != nullptr) {  // a slab for right-hand sides of which none goes on
    int live = 0;
    for (int b = threadIdx.x; b < batch; b += 128) live |= !state[b].done;
    if (!__syncthreads_or(live)) return;
  }
  const int m = m0 + blockIdx.y, t = threadIdx.x, p = blockIdx.x * 128 + t;
  const bool act = p < npairs;
  const int pp = act ? p : npairs - 1;
  const double x = pairs[pp].x;
  Rec s;
  rec_init(s, seed, seed_exp, m, pp, npairs);
  const int64_t base = sp_alm_base(lmax, m), eo = (int64_t)m * npairs + pp;
  const int e0 = esc[eo], e2 = esc[(int64_t)(mmax + 1) * npairs + eo];
  const int noct = 2 * ((lmax - m + 16) / 16);
  const int nco = min(16, npoct - (int)blockIdx.x * 16);  // pair octets of this block in the table
  const int64_t trow = roff[m] - row0;
  unsigned char *mine = stage + (t >> 3) * GEN_PST + (t & 7) * 2;
  for (int oc = 0; oc < noct; ++oc) {
    if ((oc & 7) == 0) {
      if (t < 64 && m + 8 * oc + t <= lmax) sc[t] = rec[base + m + 8 * oc + t + 1];
      __syncthreads();
    }
    for (int r = 0; r < 8; ++r) {
      const int l = m + 8 * oc + r;
      long long v[3] = {0, 0, 0};
      if (l <= lmax && act && s.S == 0) {
        v[0] = fixed53(s.l0, e0);
        v[1] = fixed53(s.p0, e2);
        v[2] = fixed53(s.q0, e2);
        if ((l + m) & 1) v[2] = -v[2];
      }
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        int d[SPLIT_S];
        Fixed<SPLIT_S>::digits(v[f], d);
#pragma unroll
        for (int k = 0; k < SPLIT_S; ++k)
          *reinterpret_cast<uint16_t *>(mine + (f * SPLIT_S + k) * 16 * GEN_PST + r * 16) = bf16_one(d[k]);
      }
      if (l < lmax) rec_advance(s, sc[(8 * oc + r) & 63], x, m, l, seed, pp, npairs);
    }
    __syncthreads();
    if (t < 8 * nco) {
#pragma unroll
      for (int fd = 0; fd < 3 * SPLIT_S; ++fd) {
        const int f = fd / SPLIT_S, d = fd % SPLIT_S;
        const int64_t row = (int64_t)f * rows_cap + trow + oc;
        const uint4 w = *reinterpret_cast<const uint4 *>(stage + (fd * 16 + (t >> 3)) * GEN_PST + (t & 7) * 16);
        *reinterpret_cast<uint4 *>(dig + ((((int64_t)d * 3 * rows_cap + row) * npoct + blockIdx.x * 16) * 128) +
                                   t * 16) = w;
      }
    }
    __syncthreads();
  }
}

// ----------------------------------------------------------------- columns
// Digits of the columns.  One K step of one column tile is S x N0 rows of 16
// values in the K-major core-matrix order (row j N0 + 4 r + c: digit j of
// column c of the tile's right-hand side r).

// Synthesis columns of order m0 + blockIdx.x and right-hand side blockIdx.y;
// blockIdx.z = part.  xoff: K steps of the orders before m0 + blockIdx.x in
// this launch; the polarisation region follows the temperature one (xpart bytes).
template <int S, typename C>
__global__ void __launch_bounds__(128) k_split_xsyn(const C *__restrict__ alm, unsigned char *__restrict__ x,
                                                    int *__restrict__ xexp, const int *__restrict__ roff, int m0,
                                                    int lmax, int64_t nalm, int batch, int nb, int nct, int n0,
                                                    int64_t xpart, const SolveState *__restrict__ state) {
  __shared__ int red[4];
  const int m = m0 + blockIdx.x, b = blockIdx.y, part = blockIdx.z;
  if (state != nullptr && state[b].done) return;
  const int64_t base = sp_alm_base(lmax, m);
  const C *a0 = alm + (int64_t)b * 3 * nalm + base + m;
  const int n = lmax - m + 1, nk = (n + 15) / 16;
  using R = decltype(C::x);
  auto comp = [&](int c, int i) -> R {  // column c of multipole m + i (sg not applied)
    if (i >= n) return R(0);
    if (part == 0) {
      const C t = a0[i];
      return (c & 1) ? t.y : t.x;
    }
    const C e = a0[i + nalm], bb = a0[i + 2 * nalm];
    // a+ = -(E + iB), a- = -(E - iB)
    switch (c) {
      case 0: return bb.y - e.x;
      case 1: return -(e.y + bb.x);
      case 2: return -(e.x + bb.y);
      default: return bb.x - e.y;
    }
  };
  int ex = -100000;
  for (int i = threadIdx.x; i < n; i += 128)
    for (int c = 0; c < (part == 0 ? 2 : 4); ++c) ex = max(ex, exp_of(comp(c, i)));
  ex = max(-1000, block_max(ex, red));
  if (ex >= SPLIT_NAN) ex = SPLIT_NAN;
  if (threadIdx.x == 0) xexp[((int64_t)m * batch + b) * 2 + part] = ex;
  const int ct = b / nb, r = b - ct * nb;
  const int64_t blk = (int64_t)S * n0 * 32;
  const int64_t k0 = (int64_t)(roff[m] - roff[m0]) / 2 * nct + (int64_t)ct * nk;
  unsigned char *xo = x + part * xpart + k0 * blk;
  const int nconv = part == 0 ? 2 : 4;
  const int lc = part == 0 ? 1 : 2;  // neighbouring items write neighbouring 16-byte rows
  for (int it = threadIdx.x; it < 4 * nk * nconv; it += 128) {
    const int hf = it & 1, c = (it >> 1) & (nconv - 1), oc = it >> (1 + lc);
    typename Fixed<S>::type v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = ex >= SPLIT_NAN ? 0 : Fixed<S>::of(comp(c, 8 * oc + 4 * hf + i), ex);
    if (part == 1 && c >= 2) {  // sg a-
      v[1] = -v[1];
      v[3] = -v[3];
    }
    put_digits<S, 4>(xo + (int64_t)(oc >> 1) * blk, n0, 4 * r + c, oc & 1, hf, v, part == 0, 4 * r + c + 2);
  }
}

// Analysis columns of order m0 + blockIdx.x: T (re, im of N, of S), then for
// the polarisation (P+_N, P-_S) of p and (P+_S, P-_N) of q, scaled by the
// row exponents.  The three regions lie xpart bytes apart.  The columns are
// formed once, into shared memory (slot(p): one of padding every 8, so that
// threads on neighbouring octets read different banks).
template <int S, typename C>
__global__ void __launch_bounds__(256) k_split_xana(const C *__restrict__ rc, unsigned char *__restrict__ x,
                                                    int *__restrict__ xexp, const int16_t *__restrict__ esc, int m0,
                                                    int mmax, int npairs, int batch, int nb, int nct, int n0,
                                                    int64_t xpart, const SolveState *__restrict__ state, int pchunk) {
  using R = decltype(C::x);
  extern __shared__ __align__(16) unsigned char xs_raw[];
  R *col = reinterpret_cast<R *>(xs_raw);  // [columns][slots of a chunk of ring pairs]
  __shared__ int red[8];
  const int m = m0 + blockIdx.x, b = blockIdx.y, part = blockIdx.z;
  if (state != nullptr && state[b].done) return;
  const int64_t fs = (int64_t)(mmax + 1) * npairs * 2;  // field stride
  const C *g0 = rc + ((int64_t)b * 3 * (mmax + 1) + m) * npairs * 2;
  const int16_t *es = esc + ((int64_t)part * (mmax + 1) + m) * npairs;
  const int nk = (npairs + 15) / 16, ld = pchunk + pchunk / 8, nconv = part == 0 ? 4 : 8;
  const bool whole = pchunk >= npairs;
  auto slot = [](int p) { return p + (p >> 3); };
  // the columns of pair p (0, 1: N of T or P+_N; 2, 3: S or P-_S; 4, 5: P+_S; 6, 7: P-_N)
  auto form = [&](int p, R v[8]) {
    const bool eq = p == npairs - 1;  // the equator has no mirror ring
    C z;
    z.x = z.y = 0;
    if (part == 0) {
      const C n = g0[2 * p], s = eq ? z : g0[2 * p + 1];
      v[0] = n.x;
      v[1] = n.y;
      v[2] = s.x;
      v[3] = s.y;
      return;
    }
    const C qn = g0[fs + 2 * p], un = g0[2 * fs + 2 * p];
    const C qs = eq ? z : g0[fs + 2 * p + 1], us = eq ? z : g0[2 * fs + 2 * p + 1];
    v[0] = qn.x - un.y;
    v[1] = qn.y + un.x;
    v[2] = qs.x + us.y;
    v[3] = qs.y - us.x;
    v[4] = qs.x - us.y;
    v[5] = qs.y + us.x;
    v[6] = qn.x + un.y;
    v[7] = qn.y - un.x;
  };
  int ex = -100000;
  for (int p = threadIdx.x; p < npairs; p += 256) {
    R v[8];
    form(p, v);
    const int e0 = es[p];
    for (int c = 0; c < nconv; ++c) {
      const int e = exp_of(v[c]);
      ex = max(ex, e >= SPLIT_NAN || e < -10000 ? e : e + e0);
      if (whole) col[c * ld + slot(p)] = v[c];
    }
  }
  ex = max(-1000, block_max(ex, red));
  if (ex >= SPLIT_NAN - 1024) ex = SPLIT_NAN;
  if (threadIdx.x == 0) xexp[((int64_t)m * batch + b) * 2 + part] = ex;
  const int ct = b / nb, r = b - ct * nb;
  const int64_t blk = (int64_t)S * n0 * 32;
  const int64_t k0 = ((int64_t)(m - m0) * nct + ct) * nk;
  for (int p0 = 0; p0 < 16 * nk; p0 += pchunk) {
    if (!whole) {
      __syncthreads();
      for (int p = p0 + threadIdx.x; p < min(npairs, p0 + pchunk); p += 256) {
        R v[8];
        form(p, v);
        for (int c = 0; c < nconv; ++c) col[c * ld + slot(p - p0)] = v[c];
      }
      __syncthreads();
    }
    const int nh = min(pchunk, 16 * nk - p0) / 4;  // groups of four pairs
    for (int it = threadIdx.x; it < nh * nconv; it += 256) {
      // neighbouring items write neighbouring 16-byte rows
      const int r8 = it >> 3, no = nh / 2, reg = r8 / no, ol = r8 - reg * no;
      const int c = 4 * reg + ((it >> 1) & 3), pl = 8 * ol + 4 * (it & 1), p = p0 + pl, oc = p >> 3;
      typename Fixed<S>::type v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        v[i] = (ex >= SPLIT_NAN || p + i >= npairs) ? 0 : Fixed<S>::of(col[c * ld + slot(pl + i)], ex - es[p + i]);
      unsigned char *xo = x + (int64_t)(part == 0 ? 0 : 1 + (c >> 2)) * xpart + k0 * blk;
      put_digits<S, 4>(xo + (int64_t)(oc >> 1) * blk, n0, 4 * r + (c & 3), oc & 1, it & 1, v, false, 0);
    }
  }
}

// ------------------------------------------------------------- the products

// K steps per stage: the copies of three digits are half as large, and the
// waits and issues of a stage then cost more than its bytes (a stage of one
// step ran at 4.4 TB/s).
__host__ __device__ constexpr int stage_steps(int S) { return S == 3 ? 2 : 1; }

struct SplitArgs {
  const SplitTile *tiles;
  int ntiles, nct, nb, batch;
  const unsigned char *x;
  int64_t xpart;
  const int *xexp;
  const int16_t *esc;
  int rows_cap;
  int lmax, mmax, npairs;
  int64_t nalm;
  void *out;               // rc (synthesis) or analysis sums
  int64_t out_bstride;     // analysis: values between right-hand sides
  const SolveState *state;
  int nstages;
  int *err;
};

// SYN: rows are ring pairs, K the multipoles; else rows are multipoles, K the
// ring pairs.  N0 = 8 NQ columns, four per right-hand side.
template <bool SYN, int S, int NQ>
__global__ void __launch_bounds__(split_threads(NQ), 1) k_split(const __grid_constant__ CUtensorMap map,
                                                            const SplitArgs A) {
  constexpr int N0 = 8 * NQ, DRAIN = split_drain_warps(NQ), THREADS = split_threads(NQ);
  constexpr int QW = 8 * NQ / DRAIN;  // right-hand sides per drain warp
  constexpr int G = Weights<S>::G;
  constexpr int SET = (G * N0 + ((N0 & 15) ? 8 : 0) + 15) / 16 * 16;  // accumulator columns of one set
  constexpr int COLS = 2 * SET <= 64 ? 64 : (2 * SET <= 128 ? 128 : (2 * SET <= 256 ? 256 : 512));
  constexpr int KS = stage_steps(S);  // K steps of 16 per stage
  constexpr int ABYTES = S * 4096 * KS, BBYTES = S * N0 * 32;  // (B: of one K step)
  // zero rows behind the last digit's: the first MMA of a chunk clears every
  // accumulator, G of them from S digits, and an N is rounded up to 16
  constexpr int ZBYTES = (N0 + 8) * 32, STAGE = ABYTES + KS * BBYTES + ZBYTES;
  using cplx = typename OutT<S>::cplx;
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t bars[2 * SPLIT_MAX_STAGES + 5];
  __shared__ uint32_t tslot;
  __shared__ int cta_bad;
  __shared__ uint32_t live_mask[16];  // column tiles with an unfinished right-hand side (nct <= 512)
  uint64_t *full = bars, *empty = bars + SPLIT_MAX_STAGES, *tfull = bars + 2 * SPLIT_MAX_STAGES, *tempty = tfull + 2,
           *fin = tempty + 2;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NS = A.nstages;
  if (tid == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], DRAIN);
    }
    mbar_init(fin, 1);
    cta_bad = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 16) live_mask[tid] = 0;
  for (int i = tid; i < NS * (ZBYTES / 16); i += THREADS)
    *reinterpret_cast<uint4 *>(sm + (size_t)(i / (ZBYTES / 16)) * STAGE + ABYTES + KS * BBYTES +
                              (i % (ZBYTES / 16)) * 16) =
        make_uint4(0, 0, 0, 0);
  fence_proxy_async();
  if (warp == 0) tmem_alloc(&tslot, COLS);
  __syncthreads();
  for (int b = tid; b < A.batch; b += THREADS)
    if (A.state == nullptr || !A.state[b].done) atomicOr(&live_mask[(b / A.nb) >> 5], 1u << ((b / A.nb) & 31));
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tbase = tslot;
  const int total = A.ntiles * A.nct;
  int issued = 0;  // stages filled (producer)
  const uint32_t sm_a = smem_u32(sm), full_a = smem_u32(full), empty_a = smem_u32(empty);

  if (warp == DRAIN) {
    if (lane == 0) {
      bool ok = true;
      StageAt at;
      for (int t = blockIdx.x; ok && t < total; t += gridDim.x) {
        const int ct = t % A.nct;
        if (!((live_mask[ct >> 5] >> (ct & 31)) & 1u)) continue;
        const SplitTile T = A.tiles[t / A.nct];
        const int nfun = T.part == 0 ? 1 : 2;
        const int zrow = T.part * A.rows_cap + T.trow;
        const unsigned char *x0 = A.x + (int64_t)T.part * A.xpart +
                                  (T.xstep * (int64_t)A.nct + (int64_t)ct * T.xlen + T.k0) * BBYTES;
        // chunks alternate p and q over the same K steps
        for (int k0 = 0; ok && k0 < T.nk; k0 += T.chunk)
          for (int fun = 0; ok && fun < nfun; ++fun)
            for (int k = k0; k < min(k0 + T.chunk, T.nk); k += KS) {
              if (issued >= NS && !mbar_wait_at(empty_a + 8 * at.s, at.phase ^ 1, A.err)) {
                ok = false;
                break;
              }
              const uint32_t dst = sm_a + at.s * STAGE, bar = full_a + 8 * at.s;
              const uint32_t xb = KS > 1 ? min(KS, T.nk - k) * BBYTES : BBYTES;  // no column digits beyond the tile's
              mbar_expect_tx_at(bar, ABYTES + xb);
              const int z = zrow + fun * A.rows_cap;
              if (SYN)
                tma_box_at(dst, &map, 16 * T.row, z + 2 * (T.k0 + k), bar);
              else
                tma_box_at(dst, &map, 2 * (T.k0 + k), z, bar);
              bulk_g2s_at(dst + ABYTES, x0 + (SYN ? 0 : fun * A.xpart) + (int64_t)k * BBYTES, xb, bar);
              ++issued;
              at.next(NS);
            }
      }
      if (!ok) cta_bad = 1;
    }
  } else if (warp == DRAIN + 1) {
    if (lane == 0) {
      bool ok = true;
      int cc = 0;
      StageAt at;
      // K-major rows (multipoles): K neighbours 128 bytes apart, row octets 256; MN-major rows (ring
      // pairs): K neighbours 2048 bytes apart, row octets 128
      const uint64_t ad0 = SYN ? split_desc(sm_a, 2048, 128) : split_desc(sm_a, 128, 256 * KS);
      const uint64_t bd0 = split_desc(sm_a + ABYTES, 128, 256);
      for (int t = blockIdx.x; ok && t < total; t += gridDim.x) {
        const int ct = t % A.nct;
        if (!((live_mask[ct >> 5] >> (ct & 31)) & 1u)) continue;
        const SplitTile *T = A.tiles + t / A.nct;
        const int nk = T->nk, nfun = T->part == 0 ? 1 : 2, chunk = T->chunk;
        const int nch = nfun * ((nk + chunk - 1) / chunk);
        for (int c = 0; ok && c < nch; ++c, ++cc) {
          const int set = cc & 1;
          if (cc >= 2 && !mbar_wait(&tempty[set], ((cc >> 1) - 1) & 1, A.err)) {
            ok = false;
            break;
          }
          fence_after_sync();
          const int nstep = min(chunk, nk - (nfun == 2 ? c >> 1 : c) * chunk);
          const uint32_t d = tbase + set * SET;
          for (int k = 0; k < nstep; k += KS) {
            if (!mbar_wait_at(full_a + 8 * at.s, at.phase, A.err)) {
              ok = false;
              break;
            }
            fence_after_sync();
            const uint64_t off = (uint64_t)(at.s * (STAGE >> 4));
            if (k == 0)
              split_step<S, N0, 4096 * KS, SYN, true>(d, ad0 + off, bd0 + off);
            else
              split_step<S, N0, 4096 * KS, SYN, false>(d, ad0 + off, bd0 + off);
#pragma unroll
            for (int h = 1; h < KS; ++h)
              if (k + h < nstep)
                split_step<S, N0, 4096 * KS, SYN, false>(d, ad0 + off + h * ((SYN ? 4096 : 256) >> 4),
                                                         bd0 + off + h * (BBYTES >> 4));
            commit_at(empty_a + 8 * at.s);
            at.next(NS);
          }
          if (ok) commit(&tfull[set]);
        }
      }
      if (!ok) cta_bad = 1;
      commit(fin);
      mbar_wait(fin, 0, A.err);  // every MMA has finished before the tensor memory goes
    }
  } else {
    const int part = warp >> 2, wq = warp & 3;
    bool ok = true;
    int cc = 0;
    for (int t = blockIdx.x; ok && t < total; t += gridDim.x) {
      const int ct = t % A.nct;
      if (!((live_mask[ct >> 5] >> (ct & 31)) & 1u)) continue;
      const SplitTile T = A.tiles[t / A.nct];
      const int nfun = T.part == 0 ? 1 : 2;
      const int nch = nfun * ((T.nk + T.chunk - 1) / T.chunk);
      const int nrhs = min(QW, min(A.nb, A.batch - ct * A.nb) - part * QW);  // of this warp group (may be <= 0)
      constexpr int NF = SYN ? 2 : 1;
      Acc<S> acc[NF][QW][4];
      for (int c = 0; c < nch; ++c, ++cc) {
        const int set = cc & 1;
        if (!mbar_wait(&tfull[set], (cc >> 1) & 1, A.err)) {
          ok = false;
          break;
        }
        __syncwarp();
        fence_after_sync();
        const uint32_t tcol = tbase + ((uint32_t)(wq * 32) << 16) + set * SET + part * QW * 4;
        const int fa = SYN && nfun == 2 ? (c & 1) : 0;
#pragma unroll
        for (int q = 0; q < QW; ++q) {
          if (q >= nrhs) break;
          uint32_t g[G][4];
#pragma unroll
          for (int k = 0; k < G; ++k) tmem_ld4(tcol + k * N0 + q * 4, g[k]);
          tmem_wait_ld();
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            int w[G];
#pragma unroll
            for (int k = 0; k < G; ++k) w[k] = __float2int_rn(__uint_as_float(g[k][v]));
            if (NF == 2 && fa)
              acc[NF - 1][q][v].add(w);
            else
              acc[0][q][v].add(w);
          }
        }
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[set]);
      }
      if (!ok) break;
      // results of this tile
      const int row = T.row * SPLIT_ROWS + wq * 32 + lane;
      if (SYN) {
        if (row < A.npairs) {
          const int er = A.esc[((int64_t)T.part * (A.mmax + 1) + T.m) * A.npairs + row];
          cplx *rc = reinterpret_cast<cplx *>(A.out);
          const bool equator = row == A.npairs - 1;
#pragma unroll
          for (int q = 0; q < QW; ++q) {
            if (q >= nrhs) break;
            const int b = ct * A.nb + part * QW + q;
            if (A.state != nullptr && A.state[b].done) continue;
            const int ex = A.xexp[((int64_t)T.m * A.batch + b) * 2 + T.part];
            const int e = ex + er;
            const bool bad = ex >= SPLIT_NAN;
            const typename OutT<S>::real nan = (typename OutT<S>::real)NAN;
            const int64_t fstr = (int64_t)(A.mmax + 1) * A.npairs * 2;
            cplx *o = rc + ((int64_t)b * 3 * (A.mmax + 1) + T.m) * A.npairs * 2 + 2 * (int64_t)row;
            if (T.part == 0) {
              const Acc<S> *v = acc[0][q];
              o[0] = bad ? mk<S>(nan, nan) : mk<S>(value_of(v[0], e), value_of(v[1], e));
              if (!equator) o[1] = bad ? mk<S>(nan, nan) : mk<S>(value_of(v[2], e), value_of(v[3], e));
            } else {
              // p: (P+_N, P-_S), q: (P+_S, P-_N); Q = (P+ + P-) / 2, U = (P+ - P-) / 2i
              const Acc<S> *vp = acc[0][q], *vq = acc[NF - 1][q];
              o += fstr;
              o[0] = bad ? mk<S>(nan, nan) : mk<S>(value_of(vp[0], vq[2], 1, e - 1), value_of(vp[1], vq[3], 1, e - 1));
              o[fstr] = bad ? mk<S>(nan, nan)
                            : mk<S>(value_of(vp[1], vq[3], -1, e - 1), value_of(vq[2], vp[0], -1, e - 1));
              if (!equator) {
                o[1] = bad ? mk<S>(nan, nan)
                           : mk<S>(value_of(vq[0], vp[2], 1, e - 1), value_of(vq[1], vp[3], 1, e - 1));
                o[fstr + 1] = bad ? mk<S>(nan, nan)
                                  : mk<S>(value_of(vq[1], vp[3], -1, e - 1), value_of(vp[2], vq[0], -1, e - 1));
              }
            }
          }
        }
      } else {
        const int l = T.m + row;
        if (l <= A.lmax) {
          cplx *out = reinterpret_cast<cplx *>(A.out);
          const int64_t i = sp_alm_base(A.lmax, T.m) + l;
          const int sg = ((l + T.m) & 1) ? -1 : 1;
#pragma unroll
          for (int q = 0; q < QW; ++q) {
            if (q >= nrhs) break;
            const int b = ct * A.nb + part * QW + q;
            if (A.state != nullptr && A.state[b].done) continue;
            const int e = A.xexp[((int64_t)T.m * A.batch + b) * 2 + T.part];
            const bool bad = e >= SPLIT_NAN;
            const typename OutT<S>::real nan = (typename OutT<S>::real)NAN;
            const Acc<S> *v = acc[0][q];
            cplx *o = out + (int64_t)b * A.out_bstride + i;
            if (T.part == 0) {
              o[0] = bad ? mk<S>(nan, nan) : mk<S>(value_of(v[0], v[2], sg, e), value_of(v[1], v[3], sg, e));
            } else {
              // aE = -(g+ + g-) / 2, aB = i (g+ - g-) / 2 with g- = sg v[2, 3]
              o[A.nalm] = bad ? mk<S>(nan, nan)
                              : mk<S>(-value_of(v[0], v[2], sg, e - 1), -value_of(v[1], v[3], sg, e - 1));
              o[2 * A.nalm] = bad ? mk<S>(nan, nan)
                                  : mk<S>(-value_of(v[1], v[3], -sg, e - 1), value_of(v[0], v[2], -sg, e - 1));
            }
          }
        }
      }
    }
    if (!ok && lane == 0) cta_bad = 1;
  }
  __syncthreads();
  // after a wait that gave up, the copies still in flight (at most the last
  // phase of each stage) land before the shared memory goes away
  if (cta_bad && warp == DRAIN && lane == 0)
    for (int c = max(0, issued - NS); c < issued; ++c) mbar_wait(&full[c % NS], (c / NS) & 1, A.err);
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tbase, COLS);
}

// ---------------------------------------------------------------- host side

// columns of one tile: right-hand sides per tile and N0 / 8 for a batch
void split_cols(int batch, int *nct, int *nb, int *nq) {
  *nct = (batch + 7) / 8;
  *nb = (batch + *nct - 1) / *nct;
  *nq = (*nb + 1) / 2;
}

}  // namespace

static int table_rows(int lmax, int m) { return 2 * ((lmax - m + 16) / 16); }

size_t split_table_bytes(int lmax, int mmax, int npairs) {
  double rows = 0;
  for (int m = 0; m <= mmax; ++m) rows += table_rows(lmax, m);
  return (size_t)(rows * 3 * SPLIT_S * 128.0 * ((npairs + 7) / 8));
}

bool split_whole(const dm_plan *p) {
  const SplitTables *T = p->split;
  if (!T || T->disabled) return false;
  if (T->dig) return T->full;
  const int64_t bytes = (int64_t)split_table_bytes(p->lmax, p->mmax, p->npairs);
  return bytes <= p->ffs_cap || (!p->ffs_cap_set && bytes <= p->split_cap);  // (one slab may hold all of it)
}

size_t split_order_bytes(int lmax, int npairs) {
  return (size_t)table_rows(lmax, 0) * 3 * SPLIT_S * 128 * ((npairs + 7) / 8);
}

static void drop_cuts(SplitTables *T) {
  for (SplitLaunches &c : T->cuts)
    for (SplitTile *t : c.tiles)
      if (t) cudaFree(t);
  T->cuts.clear();
}

int64_t split_bytes(const dm_plan *p) { return p->split ? p->split->bytes : 0; }

// All that the device holds of the tables goes.
static void drop_tables(SplitTables *T) {
  drop_cuts(T);
  for (void *q : {(void *)T->esc, (void *)T->dig, (void *)T->x})
    if (q) cudaFree(q);
  T->esc = nullptr;
  T->dig = T->x = nullptr;
  T->xexp = nullptr;
  T->full = false;
  T->slab.clear();
  T->bytes = 0;
}

void split_release(dm_plan *p) {
  if (!p->split) return;
  drop_tables(p->split);
  delete p->split;
  p->split = nullptr;
}

void split_new(dm_plan *p) {
  p->split = new SplitTables();
  p->split->batch = p->batch;
}

void split_disable(dm_plan *p) { p->split->disabled = true; }

// Column digits of one launch: those of every order, at most cap bytes unless
// one order alone takes more.
size_t split_scratch_bytes(int lmax, int npairs, int batch, int64_t cap) {
  int nct, nb, nq;
  split_cols(batch, &nct, &nb, &nq);
  const double blk = (double)SPLIT_S * 8 * nq * 32 * nct, nkp = (npairs + 15) / 16;
  const double one = blk * std::max(3.0 * nkp, (double)table_rows(lmax, 0)), all = one * (lmax + 1);
  return (size_t)std::max(one, std::min(all, (double)cap));
}

// Forget the digit slabs (a new slab size); the row exponents stay.
void split_forget(dm_plan *p) {
  SplitTables *T = p->split;
  if (!T) return;
  if (T->dig) {
    T->bytes -= (int64_t)SPLIT_S * 3 * T->rows_cap * T->npoct * 128;
    cudaFree(T->dig);
  }
  T->dig = nullptr;
  T->full = false;
  T->slab.clear();
  drop_cuts(T);
}

cudaError_t first_steps(const uint16_t *lfirst, int *ks, int mmax, int npairs, int npt, int nlt) {
  k_split_ks<<<dim3(mmax + 1, 2), 32>>>(lfirst, ks, mmax, npairs, npt, nlt);
  return cudaGetLastError();
}

// First K steps (units of 16 multipoles or ring pairs) of every tile of 128
// ring pairs and of 128 multipoles whose values reach 2^floor_exp, as k_split_ks
// lays them out, in a new device array.
cudaError_t visible_steps(dm_plan *p, int floor_exp, int **out) {
  const int nm = p->mmax + 1, npt = (p->npairs + 127) / 128, nlt = (p->lmax + 128) / 128;
  const size_t n = 2 * (size_t)nm * p->npairs;
  int16_t *esc = nullptr;
  int *ks = nullptr;
  cudaError_t e = cudaMalloc(&esc, sizeof(int16_t) * 2 * n);
  if (!e) e = cudaMalloc(&ks, sizeof(int) * 2 * nm * (size_t)(npt + nlt));
  if (!e) {
    uint16_t *lf = reinterpret_cast<uint16_t *>(esc + n);
    k_split_scale<<<dim3((p->npairs + 63) / 64, nm), 64>>>(p->pairs, p->rec, p->seed, p->seed_exp, esc, lf, p->lmax,
                                                           p->mmax, p->npairs, floor_exp);
    k_split_ks<<<dim3(nm, 2), 32>>>(lf, ks, p->mmax, p->npairs, npt, nlt);
    e = cudaGetLastError();
  }
  if (!e) e = cudaDeviceSynchronize();
  cudaFree(esc);
  if (e) {
    cudaFree(ks);
    return e;
  }
  *out = ks;
  return cudaSuccess;
}

// Row exponents, first visible multipoles, column scratch, slabs and tensor
// maps: once per plan, and kept until it goes, because a captured graph may
// name them (the slabs until dm_set_ff_slab_bytes).  The whole table is kept
// when it takes at most p->split_cap bytes, else slabs of p->ffs_cap bytes are
// generated before their products.
static cudaError_t split_setup(dm_plan *p, cudaStream_t st) {
  SplitTables *T = p->split;
  const int nm = p->mmax + 1, lmax = p->lmax, npairs = p->npairs;
  cudaError_t e = cudaSuccess;
  if (!encode_fn()) return cudaErrorNotSupported;
  if (!T->esc) {
    const size_t n = 2 * (size_t)nm * npairs;
    T->npoct = (npairs + 7) / 8;
    T->roff.assign(nm + 1, 0);
    for (int m = 0; m < nm; ++m) T->roff[m + 1] = T->roff[m] + table_rows(lmax, m);
    // the exponents and, behind them, the first table row of each order
    const size_t eb = (sizeof(int16_t) * n + 15) / 16 * 16;
    const int npt = (npairs + 127) / 128, nlt = (lmax + 128) / 128;
    const size_t nks = 2 * (size_t)nm * (npt + nlt);
    unsigned char *esc = nullptr, *tmp = nullptr;  // tmp: first multipoles, then K steps
    if ((e = table_alloc(p, (void **)&esc, eb + sizeof(int) * (nm + 1)))) return e;
    if ((e = table_alloc(p, (void **)&tmp, (sizeof(uint16_t) * n + 15) / 16 * 16 + sizeof(int) * nks))) {
      cudaFree(esc);
      return e;
    }
    uint16_t *lf = reinterpret_cast<uint16_t *>(tmp);
    int *ks = reinterpret_cast<int *>(tmp + (sizeof(uint16_t) * n + 15) / 16 * 16);
    std::vector<int> h(nks);
    e = cudaMemcpyAsync(esc + eb, T->roff.data(), sizeof(int) * (nm + 1), cudaMemcpyHostToDevice, st);
    if (!e) {
      k_split_scale<<<dim3((npairs + 63) / 64, nm), 64, 0, st>>>(p->pairs, p->rec, p->seed, p->seed_exp,
                                                                 reinterpret_cast<int16_t *>(esc), lf, lmax, p->mmax,
                                                                 npairs, -100000);
      k_split_ks<<<dim3(nm, 2), 32, 0, st>>>(lf, ks, p->mmax, npairs, npt, nlt);
      e = cudaGetLastError();
    }
    if (!e) e = cudaMemcpyAsync(h.data(), ks, sizeof(int) * nks, cudaMemcpyDeviceToHost, st);
    if (!e) e = cudaStreamSynchronize(st);
    cudaFree(tmp);
    if (e) {
      cudaFree(esc);
      return e;
    }
    T->esc = reinterpret_cast<int16_t *>(esc);
    T->roff_dev = reinterpret_cast<const int *>(esc + eb);
    T->bytes += (int64_t)(eb + sizeof(int) * (nm + 1));
    T->ks_syn.resize(2 * (size_t)nm * npt);
    T->ks_ana.resize(2 * (size_t)nm * nlt);
    for (int r = 0; r < 2 * nm; ++r) {
      std::copy_n(&h[(size_t)r * (npt + nlt)], npt, &T->ks_syn[(size_t)r * npt]);
      std::copy_n(&h[(size_t)r * (npt + nlt) + npt], nlt, &T->ks_ana[(size_t)r * nlt]);
    }
  }
  if (!T->x) {
    const size_t xb = (split_scratch_bytes(lmax, npairs, T->batch, p->scratch_cap) + 127) / 128 * 128;
    const size_t all = xb + sizeof(int) * 2 * (size_t)nm * T->batch;
    if ((e = table_alloc(p, (void **)&T->x, all))) return e;
    T->xexp = reinterpret_cast<int *>(T->x + xb);
    T->bytes += (int64_t)all;
  }
  if (!T->dig) {
    const size_t row_bytes = (size_t)3 * SPLIT_S * 128 * T->npoct;
    const size_t whole = row_bytes * (size_t)T->roff[nm];
    const bool keep = !p->ffs_cap_set && whole <= (size_t)p->split_cap;
    for (int attempt = keep ? 0 : 1; attempt < 2; ++attempt) {
      const size_t cap = attempt == 0 ? whole : (size_t)p->ffs_cap;
      T->slab.assign(1, 0);
      int most = 0;
      for (int m = 0, first = 0; m < nm; ++m) {
        if (m > first && row_bytes * (size_t)(T->roff[m + 1] - T->roff[first]) > cap) {
          T->slab.push_back(m);
          first = m;
        }
        most = std::max(most, T->roff[m + 1] - T->roff[first]);
      }
      T->slab.push_back(nm);
      T->rows_cap = most;
      e = table_alloc(p, (void **)&T->dig, row_bytes * (size_t)most);
      if (e != cudaErrorMemoryAllocation) break;
    }
    if (e) return e;
    T->bytes += (int64_t)(row_bytes * (size_t)T->rows_cap);
    for (int k = 0; k < 2; ++k)
      for (int dir = 0; dir < 2; ++dir) {
        const cuuint64_t dims[4] = {64, (cuuint64_t)T->npoct, (cuuint64_t)(3 * T->rows_cap), SPLIT_S};
        const cuuint64_t strides[3] = {128, (cuuint64_t)T->npoct * 128, (cuuint64_t)(3 * T->rows_cap) * T->npoct * 128};
        const unsigned S = k == 0 ? 6 : 3, ks = stage_steps(S);
        const cuuint32_t box[4] = {64, dir == 0 ? 16u : 2 * ks, dir == 0 ? 2 * ks : 16u, S};
        const cuuint32_t one[4] = {1, 1, 1, 1};
        CUtensorMap *map = dir == 0 ? &T->map_syn[k] : &T->map_ana[k];
        if (encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, T->dig, dims, strides, box, one,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
          return cudaErrorInvalidValue;
      }
    if (T->slab.size() == 2) {  // the whole table: generated once
      if ((e = dyn_smem_allow(k_split_gen, GEN_STAGE))) return e;
      k_split_gen<<<dim3((npairs + 127) / 128, nm), 128, GEN_STAGE, st>>>(
          p->pairs, p->rec, p->seed, p->seed_exp, T->esc, T->dig, lmax, p->mmax, npairs, T->npoct, 0, 0,
          T->roff_dev, T->rows_cap, nullptr, 0);
      if ((e = cudaGetLastError())) return e;
      T->full = true;
    }
  }
  return cudaSuccess;
}

// Launches and tile lists for a batch: each launch takes orders of one slab
// whose column digits fit the scratch; tiles in order of falling K length.
static cudaError_t split_cut(dm_plan *p, int S, cudaStream_t st) {
  SplitTables *T = p->split;
  const int nm = p->mmax + 1, lmax = p->lmax, npairs = p->npairs;
  SplitLaunches C;
  int nb, nq;
  split_cols(p->batch, &C.nct, &nb, &nq);
  C.n0 = 8 * nq;
  C.S = S;
  cudaError_t e = cudaSuccess;
  const size_t blk = (size_t)S * C.n0 * 32, cap = (size_t)p->scratch_cap;
  const int npt = (npairs + 127) / 128, nlt = (lmax + 128) / 128, nkp = (npairs + 15) / 16;
  for (int dir = 0; dir < 2 && !e; ++dir) {
    std::vector<SplitTile> tiles;
    for (size_t k = 0; k + 1 < T->slab.size(); ++k) {
      int m0 = T->slab[k];
      while (m0 < T->slab[k + 1]) {
        int m1 = m0;
        size_t bytes = 0;
        for (; m1 < T->slab[k + 1]; ++m1) {
          const size_t add = blk * C.nct * (dir == 0 ? (size_t)(T->roff[m1 + 1] - T->roff[m1]) : 3 * (size_t)nkp);
          if (m1 > m0 && bytes + add > cap) break;
          bytes += add;
        }
        const size_t first = tiles.size();
        for (int m = m0; m < m1; ++m)
          for (int part = 0; part < 2; ++part)
            for (int r = 0; r < (dir == 0 ? npt : (lmax - m + 128) / 128); ++r) {
              SplitTile t;
              t.m = m;
              t.row = r;
              t.part = part;
              t.xlen = dir == 0 ? (T->roff[m + 1] - T->roff[m]) / 2 : nkp;
              t.k0 = std::min(t.xlen, dir == 0 ? T->ks_syn[((size_t)part * nm + m) * npt + r]
                                               : T->ks_ana[((size_t)part * nm + m) * nlt + r]);
              t.nk = t.xlen - t.k0;
              t.chunk = dir == 1 && m == 0 && part == 0 && r == 0 ? SPLIT_CHUNK / 2 : SPLIT_CHUNK;
              t.trow = T->roff[m] - T->roff[T->slab[k]] + (dir == 0 ? 0 : 16 * r);
              t.xstep = dir == 0 ? (T->roff[m] - T->roff[m0]) / 2 : (m - m0) * nkp;
              tiles.push_back(t);
            }
        std::stable_sort(tiles.begin() + first, tiles.end(), [](const SplitTile &a, const SplitTile &b) {
          return a.nk * (1 + a.part) > b.nk * (1 + b.part);
        });
        C.launch[dir].insert(C.launch[dir].end(), {m0, m1, (int)first, (int)(tiles.size() - first)});
        m0 = m1;
      }
    }
    e = cudaMalloc(&C.tiles[dir], sizeof(SplitTile) * tiles.size());
    if (!e)
      e = cudaMemcpyAsync(C.tiles[dir], tiles.data(), sizeof(SplitTile) * tiles.size(), cudaMemcpyHostToDevice, st);
    if (!e) e = cudaStreamSynchronize(st);
  }
  if (e) {
    for (SplitTile *t : C.tiles)
      if (t) cudaFree(t);
    return e;
  }
  T->cuts.push_back(C);
  return cudaSuccess;
}

static const SplitLaunches *split_find(const dm_plan *p, int S) {
  const SplitTables *T = p->split;
  int nct, nb, nq;
  split_cols(p->batch, &nct, &nb, &nq);
  if (!T->dig) return nullptr;
  for (const SplitLaunches &c : T->cuts)
    if (c.nct == nct && c.n0 == 8 * nq && c.S == S) return &c;
  return nullptr;
}

// The launches of the plan's batch when the split products can run: the
// tables exist or can be made now; else null (tables that do not fit, a
// stream under capture, where nothing can be allocated).
static cudaError_t split_ready(dm_plan *p, int S, cudaStream_t st, const SplitLaunches **out) {
  SplitTables *T = p->split;
  *out = nullptr;
  if (!T || T->disabled) return cudaSuccess;
  if ((*out = split_find(p, S))) return cudaSuccess;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return cudaSuccess;
  }
  if (T->shortage.lasts(p)) return cudaSuccess;
  const bool fresh = T->cuts.empty();
  cudaError_t e = split_setup(p, st);
  if (!e) e = split_cut(p, S, st);
  if (e) {
    if (fresh) drop_tables(T);  // no launch has named them yet
    cudaGetLastError();
    if (e == cudaErrorNotSupported) T->disabled = true;
    if (e == cudaErrorMemoryAllocation) T->shortage.note(p);
    return e == cudaErrorMemoryAllocation || e == cudaErrorNotSupported ? cudaSuccess : e;
  }
  T->shortage = Shortage();
  *out = split_find(p, S);
  return cudaSuccess;
}

template <bool SYN, int S, typename C2>
static cudaError_t split_run(dm_plan *p, const SplitLaunches &C, const C2 *in, void *out, int64_t out_bstride,
                             cudaStream_t st) {
  SplitTables *T = p->split;
  int nct, nb, nq;
  split_cols(p->batch, &nct, &nb, &nq);
  const int n0 = 8 * nq;
  const SolveState *state = p->state_active ? p->state : nullptr;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if (cudaError_t r = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) return r;
  const std::vector<int> &L = C.launch[SYN ? 0 : 1];
  cudaError_t e;
  int slab_made = -1;
  for (size_t k = 0; k < L.size(); k += 4) {
    const int m0 = L[k], m1 = L[k + 1], nt = L[k + 3];
    if (!T->full) {
      const int s = (int)(std::upper_bound(T->slab.begin(), T->slab.end(), m0) - T->slab.begin()) - 1;
      if (s != slab_made) {
        if ((e = dyn_smem_allow(k_split_gen, GEN_STAGE))) return e;
        k_split_gen<<<dim3((p->npairs + 127) / 128, T->slab[s + 1] - T->slab[s]), 128, GEN_STAGE, st>>>(
            p->pairs, p->rec, p->seed, p->seed_exp, T->esc, T->dig, p->lmax, p->mmax, p->npairs, T->npoct, T->slab[s],
            T->roff[T->slab[s]], T->roff_dev, T->rows_cap, state, p->batch);
        slab_made = s;
      }
    }
    const int64_t blk = (int64_t)S * n0 * 32;
    int64_t xpart;
    if (SYN) {
      xpart = blk * nct * ((T->roff[m1] - T->roff[m0]) / 2);
      k_split_xsyn<S, C2><<<dim3(m1 - m0, p->batch, 2), 128, 0, st>>>(
          in, T->x, T->xexp, T->roff_dev, m0, p->lmax, p->nalm, p->batch, nb, nct, n0, xpart, state);
    } else {
      xpart = blk * nct * ((int64_t)(m1 - m0) * ((p->npairs + 15) / 16));
      // columns of up to 1024 ring pairs in shared memory at a time
      const int pchunk = std::min(1024, (p->npairs + 15) / 16 * 16);
      const size_t xsm = sizeof(C2) / 2 * 8 * (size_t)(pchunk + pchunk / 8);
      if ((e = dyn_smem_allow(k_split_xana<S, C2>, xsm))) return e;
      k_split_xana<S, C2><<<dim3(m1 - m0, p->batch, 2), 256, xsm, st>>>(in, T->x, T->xexp, T->esc, m0, p->mmax,
                                                                       p->npairs, p->batch, nb, nct, n0, xpart, state,
                                                                       pchunk);
    }
    SplitArgs A;
    A.tiles = C.tiles[SYN ? 0 : 1] + L[k + 2];
    A.ntiles = nt;
    A.nct = nct;
    A.nb = nb;
    A.batch = p->batch;
    A.x = T->x;
    A.xpart = xpart;
    A.xexp = T->xexp;
    A.esc = T->esc;
    A.rows_cap = (int)T->rows_cap;
    A.lmax = p->lmax;
    A.mmax = p->mmax;
    A.npairs = p->npairs;
    A.nalm = p->nalm;
    A.out = out;
    A.out_bstride = out_bstride;
    A.state = state;
    A.err = p->tc_err;
    const int stage = stage_steps(S) * (S * 4096 + S * n0 * 32) + (n0 + 8) * 32;
    A.nstages = std::min(SPLIT_MAX_STAGES, (int)((224u << 10) / stage));
    const size_t smem = (size_t)A.nstages * stage;
    const CUtensorMap &map = SYN ? T->map_syn[S == 3] : T->map_ana[S == 3];
    const int grid = std::min(sms, nt * nct);
    auto go = [&](auto kern) {
      cudaError_t r = dyn_smem_allow(kern, smem);
      if (r) return r;
      kern<<<grid, split_threads(nq), smem, st>>>(map, A);
      return cudaGetLastError();
    };
    switch (nq) {
      case 1: e = go(k_split<SYN, S, 1>); break;
      case 2: e = go(k_split<SYN, S, 2>); break;
      case 3: e = go(k_split<SYN, S, 3>); break;
      default: e = go(k_split<SYN, S, 4>); break;
    }
    if (e) return e;
  }
  return cudaSuccess;
}

// The digits of a slab are made in each stage call, for any number of
// right-hand sides; the direct kernels run their recurrence once for each.  One
// iteration, slabs and direct kernels: nside 512 / lmax 1535, one right-hand
// side 109 and 100 ms, two 110 and 200; nside 1024 / lmax 2048, one 460 and 351.
// Digits are fixed-point: a value far below the largest of its row or column
// keeps few bits or none.  No pixel and no sum notices, but the coefficients of
// a red spectrum near the poles (lambda of low multipoles beside that of the
// highest) are such values: the calls that return them take the direct kernels.
static bool direct64(const dm_plan *p) { return p->each_value || (p->batch == 1 && !split_whole(p)); }

// FP64-class synthesis of alm into p->rc; *ran = false when the direct
// kernels have to do it.
cudaError_t split_synthesis64(dm_plan *p, const double2 *alm, cudaStream_t st, bool *ran) {
  const SplitLaunches *c = nullptr;
  const cudaError_t e = direct64(p) ? cudaSuccess : split_ready(p, 6, st, &c);
  *ran = c != nullptr;
  if (e) return e;
  return c ? split_run<true, 6>(p, *c, alm, p->rc, 0, st) : cudaSuccess;
}
// FP64-class analysis of p->rc into slot 0 of p->apart
cudaError_t split_analysis64(dm_plan *p, cudaStream_t st, bool *ran) {
  const SplitLaunches *c = nullptr;
  const cudaError_t e = direct64(p) ? cudaSuccess : split_ready(p, 6, st, &c);
  *ran = c != nullptr;
  if (e) return e;
  return c ? split_run<false, 6>(p, *c, p->rc, p->apart, (int64_t)p->nslot * 3 * p->nalm, st) : cudaSuccess;
}

// The mixed mode's stages for batches outside the BF16 kernels: of the FP32
// state e32 (or of alm) into p->rc32, and of p->rc32 into p->apart32.
cudaError_t split_synthesis32(dm_plan *p, const double2 *alm, const float2 *e32, cudaStream_t st) {
  const SplitLaunches *c = nullptr;
  if (const cudaError_t e = split_ready(p, 3, st, &c)) return e;
  if (!c) return cudaErrorMemoryAllocation;
  return e32 ? split_run<true, 3>(p, *c, e32, p->rc32, 0, st) : split_run<true, 3>(p, *c, alm, p->rc32, 0, st);
}
cudaError_t split_analysis32(dm_plan *p, cudaStream_t st) {
  const SplitLaunches *c = nullptr;
  if (const cudaError_t e = split_ready(p, 3, st, &c)) return e;
  if (!c) return cudaErrorMemoryAllocation;
  return split_run<false, 3>(p, *c, p->rc32, p->apart32, 3 * p->nalm, st);
}

}  // namespace dmwf
