// dm_dft.cu -- the FP64-class ring transforms (inverse and forward ring DFTs of
// the dual messenger step, Algorithm 1, with the update of Eq. 9 between them)
// as exact integer products on the tensor cores (split products, dm_split.cu).
//
// Why: an FFT in FP64 is bound by the FP64 pipe (2 FMA a clock and SM), and the
// polar rings of 4i pixels need Bluestein's convolution, four transforms of
// twice the size.  A ring's DFT is a product with a matrix that every
// right-hand side, field and ring of the same length shares, and the tensor
// cores do 26 digit products faster than the FP64 pipe does the FFT.
//
// Folding.  The pixels of a ring sit at phi_j = 2 pi (j + s) / n, s = 1/2 or 0,
// and n is a multiple of 4, so the ring maps onto itself under phi -> -phi and
// phi -> pi - phi.  With cos m(pi - phi) = (-1)^m cos m phi and
// sin m(pi - phi) = -(-1)^m sin m phi, the four pixels of an orbit combine to
// one value for each of four matrices: cosines and sines of even and of odd m
// (CE, CO, SE, SO), each of about n/4 x n/4: a quarter of the plain product
// each way.  Orders beyond n/2 alias: F_{kn+q} = (-1)^{2sk} F_q and
// F_{kn-q} = (-1)^{2sk} conj F_q, so only q <= n/2 meet the matrix.
//
// Passes of an iteration: k_dft_xinv (alias fold of F_m, digits), k_dft<false>
// (orbit sums, FP64), k_dft_pix (unfold, s, Cauchy partials, t - s = w (d - s),
// fold, digits), k_dft<true> (F_q, q <= n/2), k_dft_alias (the orders beyond).
// One matrix set per ring length and shift (each polar radius; two for the
// belt), kept as digit planes of 8 x 8 core matrices (4 matrices x n^2/16 x 12
// bytes: 268 MB in all at nside 256, 2.1 GB at nside 512) that serve both
// directions, K-major forward and MN-major inverse.
#include <algorithm>
#include <vector>

#include "dm_fft.cuh"
#include "dm_internal.h"
#include "dm_split.cuh"

namespace dmwf {

constexpr int DFT_CHUNK = 8;       // K steps of 16 per drain
// Warps that drain the accumulators (FP32 to integer, 64-bit sums: latency
// bound; with 8 the tensor pipe was 48 % busy): 16 where the column quads
// divide.  Forward products of 32 columns, 8 and 16 warps: flat N = 1024, 16
// right-hand sides 987 and 905 us; nside 100, 5 right-hand sides 49 and 42.
// The inverse ones, half the sums, stay as they were (855 and 866).
__host__ __device__ constexpr int dft_drain_warps(int nq) { return nq % 2 == 0 ? 16 : 8; }
__host__ __device__ constexpr int dft_threads(int nq) { return 32 * (dft_drain_warps(nq) + 2); }
constexpr int DFT_MAX_STAGES = 8;
constexpr size_t DFT_SMEM = 224u << 10;  // dynamic shared memory that a block may have here
// Below this many pixels of a plan (all right-hand sides) the FFT kernels are
// faster: a stage here is five dependent launches of few tiles, there one to
// three.  64 iterations of a solve, products against FFTs: nside 16, B 1 22.1
// and 11.5 ms; nside 64, B 1 23.8 and 19.7; nside 64, B 2 (the line) 26.7 and
// 30.0; nside 32, B 8 (the line) 28.9 and 29.8; nside 128, B 2 58 and 101.
constexpr int64_t DFT_MIN_PIXELS = 12 * 64 * 64 * 2;
// The rows and columns of a flat patch have no Bluestein rings, and on a small
// grid nothing makes up for the passes around the products: from 2^18 pixels
// on, of grids below 256 from 2^18 (256 / N)^2, below 128 never.  20 iterations
// of a solve, products against FFTs: N = 64, B 24 5.5 and 3.7 ms, B 400 54 and
// 48; N = 128, B 24 8.4 and 8.1, B 100 28.6 and 30.5 (the line: 64); N = 256, B 2
// 3.5 and 3.2, B 4 (the line) 4.9 and 5.0, B 8 7.4 and 8.4; N = 512, B 1 4.6 and
// 5.0; N = 1024, B 1 12.7 and 18.2.
static bool flat_products(int N, int batch) {
  const int64_t px = (int64_t)N * N * batch, line = (int64_t)1 << 18;
  return N >= 256 ? px >= line : N >= 128 && px * N * N >= line * 256 * 256;
}
constexpr size_t DFT_SCRATCH = (size_t)1 << 30;  // column digits of one direction and group of right-hand sides

// A matrix set: the rings of one length and shift.
struct DftSet {
  int n, nj;            // pixels; orbits (n/4, or n/4 + 1 without the half-pixel shift)
  int shift;            // 1: s = 1/2
  int mx;               // largest order kept (min(mmax, n/2))
  int rq;               // row octets of each matrix (even)
  int nyo;              // column octets (orbits)
  int pair0, npr;       // pairs of this length in the pair list
};
// The same in a cut of nl lanes (right-hand sides x fields of a group).
struct DftCol {
  int nct, w, n0;       // column tiles, columns per tile, padded columns
  int ksi, ksf;         // K steps of the inverse and forward products
  int col0;             // first column of the set
  int64_t xi, xf;       // bytes into the inverse and forward column digits
  int64_t v;            // values into the orbit sums
  int njp;              // padded orbits
};
struct DftTile {
  int set, fun;         // matrix: CE 0, CO 1, SE 2, SO 3 (forward: the parity; cosine and sine in one tile)
  int row, ct, ks;
  int z, zfun;          // table row octet of the tile; distance to the sine matrix
  int n0;
  int64_t x, xfun;      // column digits of K step 0; distance to the sine columns
  int b0, b1;           // first and last right-hand side (of the group) with a column here
};
struct DftCut {
  int nl = 0;
  DftCol *cols = nullptr;              // device
  DftTile *tiles[2][5] = {};           // device, by direction and NQ
  int ntiles[2][5] = {};
};
struct DftTables {
  int batch = 0;                       // the plan's right-hand sides (its views have one)
  std::vector<DftSet> sets;
  std::vector<int64_t> off;            // digit table offset of each set
  unsigned char *dig = nullptr;
  DftSet *sets_dev = nullptr;
  CUtensorMap *maps = nullptr;         // device: [set][inverse, forward]
  int *pair_of = nullptr, *set_of = nullptr;  // pair list and its sets
  int nlist = 0;
  std::vector<DftCut> cuts;            // by lanes: the groups of the plan and of its one-RHS views, three at most
  unsigned char *x = nullptr;          // column digits of the largest group
  double *v = nullptr;                 // orbit sums
  int *xexp = nullptr;                 // [2][xexp_n] column exponents
  int xexp_n = 0;
  int64_t bytes = 0;
  bool disabled = false;               // the plan's owner chose the FFT kernels, or the matrices pass dft_cap
  Shortage shortage;                   // they did not fit
};

namespace {

// cos(pi t / n), n a multiple of 4: the argument is brought into [0, pi/4] in
// integers, so that the rounding of t / n costs less than the result's own
__device__ double cos_frac(long long t, long long n) {
  t %= 2 * n;
  if (t < 0) t += 2 * n;
  if (t > n) t = 2 * n - t;
  double sgn = 1.0;
  if (2 * t > n) {
    t = n - t;
    sgn = -1.0;
  }
  if (4 * t > n) return sgn * sinpi((double)(n / 2 - t) / (double)n);
  return sgn * cospi((double)t / (double)n);
}

// Digits of one set: one thread per (matrix, row, octet of orbits).
__global__ void k_dft_gen(const DftSet s, unsigned char *__restrict__ dig) {
  const int64_t total = (int64_t)4 * s.rq * 8 * s.nyo;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int jo = (int)(i % s.nyo), rr = (int)(i / s.nyo), fun = rr / (8 * s.rq), r = rr % (8 * s.rq);
    const int q = 2 * r + (fun & 1);
    long long v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int j = 8 * jo + k;
      v[k] = 0;
      if (q <= s.mx && j < s.nj) {
        const long long t = (long long)q * (2 * j + s.shift);  // q phi_j = pi t / n
        const double c = cos_frac(fun < 2 ? t : t - s.n / 2, s.n);
        v[k] = c == 1.0 ? 1ll << 53 : (c == -1.0 ? -(1ll << 53) : fixed53(c, 0));
      }
    }
    int d[8][SPLIT_S];
#pragma unroll
    for (int k = 0; k < 8; ++k) Fixed<SPLIT_S>::digits(v[k], d[k]);
#pragma unroll
    for (int j = 0; j < SPLIT_S; ++j) {
      uint4 w;
      w.x = bf16_pair(d[0][j], d[1][j]);
      w.y = bf16_pair(d[2][j], d[3][j]);
      w.z = bf16_pair(d[4][j], d[5][j]);
      w.w = bf16_pair(d[6][j], d[7][j]);
      *reinterpret_cast<uint4 *>(
          dig + ((((int64_t)j * 4 * s.rq + fun * s.rq + (r >> 3)) * s.nyo + jo) * 128 + (r & 7) * 16)) = w;
    }
  }
}

// Columns of a set run over the pairs' two sides, then over the lanes, so that a
// tile holds as few right-hand sides as it can: it is left out once they are
// finished.
__device__ __forceinline__ int col_of(const DftSet &s, int pair, int lane) { return (lane * s.npr + pair) * 2; }
// a column's tile and place there
__device__ __forceinline__ void col_place(const DftCol &c, int col, int &ct, int &cit) {
  ct = col / c.w;
  cit = col - ct * c.w;
}

// Slot of the i-th value of a row of staged values: one slot of padding every
// 4, so that threads on neighbouring groups of 4 read different banks.
__device__ __forceinline__ int slot4(int i) { return i + (i >> 2); }
__host__ __device__ constexpr int slots4(int n) { return n + n / 4 + 1; }

// Digits of four staged values per item, the items ordered so that the 16-byte
// rows of the two sides (neighbouring columns) leave as one 32-byte sector.
// row(side, fun) -> staged values; col/place of side 0 in ct, cit.
template <typename Row>
__device__ __forceinline__ void digit_items(unsigned char *x, const DftCol &C, int ks, int ct, int cit, int count,
                                            const int e[2], int nsides, Row row) {
  const int64_t blk = (int64_t)SPLIT_S * C.n0 * 32;
  for (int it = threadIdx.x; it < 4 * 4 * ks * 2; it += blockDim.x) {
    const int hf = it & 1, side = (it >> 1) & 1, r = it >> 2, fun = r / (2 * ks), o = r - fun * 2 * ks;
    if (side >= nsides) continue;
    const double *v = row(side, fun);
    long long d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = 8 * o + 4 * hf + i;
      d[i] = (e[side] >= SPLIT_NAN || j >= count) ? 0 : fixed53(v[slot4(j)], e[side]);
    }
    put_digits<6, 4>(x + (((int64_t)fun * C.nct + ct) * ks + (o >> 1)) * blk, C.n0, cit + side, o & 1, hf, d, false,
                     0);
  }
}

// Inverse columns of one pair and lane (both sides): C_q = sum of the orders
// that alias to q, times 2 beyond m = 0; cosines meet Re C, sines Im C.
__global__ void __launch_bounds__(128) k_dft_xinv(const double2 *__restrict__ rc, unsigned char *__restrict__ x,
                                                  int *__restrict__ xexp, const DftSet *__restrict__ sets,
                                                  const DftCol *__restrict__ cols, const int *__restrict__ pair_of,
                                                  const int *__restrict__ set_of, int lane0, int mmax,
                                                  int npairs, int eq, const SolveState *__restrict__ state) {
  extern __shared__ __align__(16) double vals[];  // [side][CE, CO, SE, SO][slots of an order's half]
  __shared__ double2 part[256];                   // partial alias sums of the short rings
  __shared__ int red[4];
  const int g = blockIdx.x, lane = blockIdx.y, pair = pair_of[g];
  if (state != nullptr && state[(lane0 + lane) / 3].done) return;
  const DftSet S = sets[set_of[g]];
  const DftCol C = cols[set_of[g]];
  const int n = S.n, h = n / 2, nq = S.mx + 1, ld = slots4(S.mx / 2 + 1);
  const bool equator = pair == eq;
  const double2 *src = rc + ((int64_t)(lane0 + lane) * (mmax + 1) * npairs + pair) * 2;
  const int64_t ms = (int64_t)npairs * 2;
  int ex[2] = {-100000, -100000};
  auto keep = [&](int q, int side, double2 v) {
    double *o = vals + (side * 4 + (q & 1)) * ld + slot4(q >> 1);
    o[0] = v.x;
    o[2 * ld] = v.y;
    ex[side] = max(ex[side], max(exp_of(v.x), exp_of(v.y)));
  };
  // short rings: groups of threads share the aliases of an order
  const int ng = nq < 128 ? 128 / nq : 1, grp = ng > 1 ? threadIdx.x / nq : 0;
  for (int q = ng > 1 ? threadIdx.x % nq : threadIdx.x; q < nq && grp < ng; q += 128) {
    double2 a = make_double2(0, 0), b = make_double2(0, 0);
    auto add = [&](int m, double re, double im) {  // re, im: signs of the real and imaginary parts
      const double2 u = src[m * ms], w = equator ? make_double2(0, 0) : src[m * ms + 1];
      a.x = fma(re, u.x, a.x);
      a.y = fma(im, u.y, a.y);
      b.x = fma(re, w.x, b.x);
      b.y = fma(im, w.y, b.y);
    };
    if (grp == 0) add(q, q ? 2.0 : 1.0, q ? 2.0 : 1.0);
    for (int k = 1 + grp; k * n - q <= mmax; k += ng) {
      const double sg = (S.shift & k & 1) ? -2.0 : 2.0;
      if (q > 0 && q < h) add(k * n - q, sg, -sg);
      if (k * n + q <= mmax) add(k * n + q, sg, sg);
    }
    if (ng > 1) {
      part[(2 * grp) * nq + q] = a;
      part[(2 * grp + 1) * nq + q] = b;
      break;
    }
    keep(q, 0, a);
    keep(q, 1, b);
  }
  __syncthreads();
  if (ng > 1) {  // the groups' sums, in order
    const int q = threadIdx.x;
    if (q < nq)
      for (int side = 0; side < 2; ++side) {
        double2 a = part[side * nq + q];
        for (int g2 = 1; g2 < ng; ++g2) {
          const double2 u = part[(2 * g2 + side) * nq + q];
          a.x += u.x;
          a.y += u.y;
        }
        keep(q, side, a);
      }
  }
  int e[2];
  const int col = col_of(S, g - S.pair0, lane), nsides = equator ? 1 : 2;
  for (int side = 0; side < 2; ++side) {
    e[side] = max(-1000, block_max(ex[side], red));  // (its barriers cover the staged values too)
    if (e[side] >= SPLIT_NAN) e[side] = SPLIT_NAN;
    if (threadIdx.x == 0 && side < nsides) xexp[C.col0 + col + side] = e[side];
  }
  int ct, cit;
  col_place(C, col, ct, cit);
  // rows of the odd matrices end half an order earlier when mx is even
  const int ne = S.mx / 2 + 1, no = (S.mx + 1) / 2;
  if (no < ne && threadIdx.x < 4) vals[(2 * threadIdx.x + 1) * ld + slot4(no)] = 0.0;
  __syncthreads();
  digit_items(x + C.xi, C, C.ksi, ct, cit, ne, e, nsides,
              [&](int side, int fun) { return vals + (side * 4 + fun) * ld; });
}

// One pair of rings and lane (threads 0-127 the northern ring, 128-255 the
// southern): pixels from the orbit sums (inverse), their update or output, and
// the orbit combinations of the forward product as digits.  The loads of an
// orbit's four pixels go out together: the pass is bound by their latency and
// the FP64 pipe, not by its bytes.
template <int MODE>
__global__ void __launch_bounds__(256) k_dft_pix(const RingDev *__restrict__ rings, const double *__restrict__ v,
                                                 unsigned char *__restrict__ x, const int *__restrict__ xexp_in,
                                                 int *__restrict__ xexp_out, const DftSet *__restrict__ sets,
                                                 const DftCol *__restrict__ cols, const int *__restrict__ pair_of,
                                                 const int *__restrict__ set_of, int lane0, int eq,
                                                 int nrings, int64_t npix, const double *__restrict__ in_map,
                                                 double *__restrict__ out_map, const double *__restrict__ w,
                                                 const double *__restrict__ wd, double *__restrict__ norms,
                                                 const SolveState *__restrict__ state) {
  extern __shared__ __align__(16) double so[];  // [side][CE, CO, SE, SO][slots of nj]
  __shared__ int red[8];
  __shared__ double rsum[8][2];
  const int g = blockIdx.x, lane = blockIdx.y, pair = pair_of[g], side = threadIdx.x >> 7, tx = threadIdx.x & 127;
  const int al = lane0 + lane;
  if ((MODE == RING_ITER || MODE == RING_INIT) && state != nullptr && state[al / 3].done) return;
  const DftSet S = sets[set_of[g]];
  const DftCol C = cols[set_of[g]];
  const int nsides = pair == eq ? 1 : 2;
  const bool on = side < nsides;
  const int ring = side ? nrings - 1 - pair : pair;
  const int col = col_of(S, g - S.pair0, lane);
  const int n = S.n, nj = S.nj, ld = slots4(nj);
  double dd = 0.0, ss = 0.0;
  int ex = -100000;
  if (on) {
    const int64_t mo = (int64_t)al * npix + rings[ring].start;
    const double *vc = v + C.v + (int64_t)(col + side) * 4 * C.njp;
    double *sv = so + side * 4 * ld;
    bool bad = false;
    if (MODE == RING_ITER || MODE == RING_INV_MAP) bad = xexp_in[C.col0 + col + side] >= SPLIT_NAN;
    // orbit j: its mirrors under phi -> pi - phi, -phi and pi + phi; without
    // the shift orbit 0 stands for the two half orbits phi = 0, pi and
    // phi = pi/2, 3 pi/2
    for (int j = tx; j < n / 4; j += 128) {
      const bool two = !S.shift && j == 0;
      int at[4] = {j, (S.shift ? n / 2 - 1 : n / 2) - j, (S.shift ? n - 1 : n) - j, n / 2 + j};
      if (two) {
        at[1] = n / 2;
        at[2] = n / 4;
        at[3] = 3 * (n / 4);
      }
      double p[4], pw[4], pd[4], o[4], r[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (MODE == RING_ITER) {
          p[k] = out_map[mo + at[k]];
          pw[k] = w[mo + at[k]];
          pd[k] = wd[mo + at[k]];
        } else if (MODE == RING_INIT) {
          pw[k] = w[mo + at[k]];
          p[k] = in_map[mo + at[k]];
        } else if (MODE == RING_FWD_MAP) {
          p[k] = in_map[mo + at[k]];
        }
      }
      if (MODE == RING_ITER || MODE == RING_INV_MAP) {
        const double ce = vc[j], co = vc[C.njp + j], se = vc[2 * C.njp + j], sn = vc[3 * C.njp + j];
        const double a1 = ce + co, a2 = ce - co, b1 = sn + se, b2 = sn - se;
        o[0] = a1 - b1;
        o[1] = a2 - b2;
        o[2] = a1 + b1;
        o[3] = a2 + b2;
        if (two) {
          const double c4 = vc[n / 4] + vc[C.njp + n / 4], s4 = vc[2 * C.njp + n / 4] + vc[3 * C.njp + n / 4];
          o[0] = a1;
          o[1] = a2;
          o[2] = c4 - s4;
          o[3] = c4 + s4;
        }
        if (bad) o[0] = o[1] = o[2] = o[3] = NAN;
#pragma unroll
        for (int k = 0; k < 4; ++k) out_map[mo + at[k]] = o[k];
      }
      if (MODE == RING_INV_MAP) continue;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (MODE == RING_ITER) {
          const double d = o[k] - p[k];
          dd = fma(d, d, dd);
          ss = fma(o[k], o[k], ss);
          r[k] = fma(-pw[k], o[k], pd[k]);
        } else if (MODE == RING_INIT) {
          r[k] = pw[k] > 0.0 ? p[k] : 0.0;
        } else {
          r[k] = p[k];
        }
      }
      auto keep = [&](int i, double ce, double co, double se, double sn) {
        sv[slot4(i)] = ce;
        sv[ld + slot4(i)] = co;
        sv[2 * ld + slot4(i)] = se;
        sv[3 * ld + slot4(i)] = sn;
        ex = max(max(ex, max(exp_of(ce), exp_of(co))), max(exp_of(se), exp_of(sn)));
      };
      if (two) {
        keep(0, r[0] + r[1], r[0] - r[1], 0.0, 0.0);
        keep(n / 4, r[2] + r[3], 0.0, 0.0, r[2] - r[3]);
      } else {
        const double c0 = r[0] + r[2], c1 = r[1] + r[3], d0 = r[0] - r[2], d1 = r[1] - r[3];
        keep(j, c0 + c1, c0 - c1, d0 - d1, d0 + d1);
      }
    }
  }
  if (MODE == RING_INV_MAP) return;
  if (MODE == RING_ITER) {
    for (int o = 16; o > 0; o >>= 1) {
      dd += __shfl_down_sync(0xffffffffu, dd, o);
      ss += __shfl_down_sync(0xffffffffu, ss, o);
    }
    if ((threadIdx.x & 31) == 0) {
      rsum[threadIdx.x >> 5][0] = dd;
      rsum[threadIdx.x >> 5][1] = ss;
    }
  }
  for (int o = 16; o > 0; o >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ex;
  __syncthreads();
  int e[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    e[k] = max(-1000, max(max(red[4 * k], red[4 * k + 1]), max(red[4 * k + 2], red[4 * k + 3])));
    if (e[k] >= SPLIT_NAN) e[k] = SPLIT_NAN;
  }
  if (tx == 0 && on) {
    xexp_out[C.col0 + col + side] = e[side];
    if (MODE == RING_ITER) {
      const int64_t no = ((int64_t)al * nrings + ring) * 2;
      const int q = 4 * side;
      norms[no] = (rsum[q][0] + rsum[q + 1][0]) + (rsum[q + 2][0] + rsum[q + 3][0]);
      norms[no + 1] = (rsum[q][1] + rsum[q + 1][1]) + (rsum[q + 2][1] + rsum[q + 3][1]);
    }
  }
  int ct, cit;
  col_place(C, col, ct, cit);
  digit_items(x + C.xf, C, C.ksf, ct, cit, nj, e, nsides,
              [&](int sd, int fun) { return so + (sd * 4 + fun) * ld; });
}

// Orders beyond n/2 from the ones they alias with: thread = pair, so that the
// stores of one order run along the pairs; blockIdx.y the order, blockIdx.z
// the lane.  (In the products' epilogue one thread wrote all aliases of its
// order: the shortest rings then took longest.)
__global__ void __launch_bounds__(128) k_dft_alias(double2 *__restrict__ rc, int lane0, int mmax, int npairs,
                                                   int nside, int nrun, const SolveState *__restrict__ state) {
  const int m = blockIdx.y + 3, p = blockIdx.x * 128 + threadIdx.x, al = lane0 + blockIdx.z;
  const int n = 4 * min(p + 1, nside);  // the orders up to n / 2 are the products' own
  if (p >= nrun || 2 * m <= n) return;
  if (state != nullptr && state[al / 3].done) return;
  const bool shift = p < nside || !((p - nside + 1) & 1);
  const int k0 = m / n, r = m - k0 * n;
  const bool fold = 2 * r > n;
  const int q = fold ? n - r : r, k = fold ? k0 + 1 : k0;
  const double re = (shift && (k & 1)) ? -1.0 : 1.0, im = fold ? -re : re;
  double2 *o = rc + ((int64_t)al * (mmax + 1) * npairs + p) * 2;
  const double2 a = o[(int64_t)q * npairs * 2];
  o[(int64_t)m * npairs * 2] = make_double2(re * a.x, im * a.y);
  if (p == npairs - 1) return;  // the equator has no mirror ring
  const double2 b = o[(int64_t)q * npairs * 2 + 1];
  o[(int64_t)m * npairs * 2 + 1] = make_double2(re * b.x, im * b.y);
}

// ---- the columns of a flat patch: complex transforms of the same length over
// the N rows.  Column kx takes the place of a row pair, its real and imaginary
// parts those of the two rows, so tables, cuts and products are the rows' own.
// At N = 1024 with 16 right-hand sides, against one FP64 FFT kernel each:
// synthesis 2.53 -> 1.66 ms (digits 0.53, products 0.86, unfolding 0.27),
// analysis 2.79 -> 1.64 (digits 0.32, products 0.91, epilogue 0.41).
constexpr int FLAT_NB = 8;  // right-hand sides per block (the E/B rotation of a column is formed once)

// Column digits of field f: C_q = h_q + h_-q to the cosines, i (h_q - h_-q) to
// the sines, h the rotated modes.  grid (columns, 3 x groups of FLAT_NB).
__global__ void __launch_bounds__(256) k_flat_xsyn(const double2 *__restrict__ alm, unsigned char *__restrict__ x,
                                                   int *__restrict__ xexp, const DftSet *__restrict__ sets,
                                                   const DftCol *__restrict__ cols, int nl, int b0, double inv_area,
                                                   int64_t nmodes, const SolveState *__restrict__ state) {
  extern __shared__ __align__(16) double vals[];  // [re, im][CE, CO, SE, SO][slots], then cos, sin 2 phi
  __shared__ int red[8];
  const DftSet S = sets[0];
  const DftCol C = cols[0];
  const int N = S.n, ne = N / 4, ld = slots4(ne), kx = blockIdx.x, f = blockIdx.y % 3;
  double *rot = vals + 8 * ld;
  if (f > 0)
    for (int q = threadIdx.x; q < N / 2; q += 256) {
      double c, s;
      rot2(kx, q, c, s);
      rot[2 * q] = inv_area * c;
      rot[2 * q + 1] = inv_area * s;
    }
  for (int b = (blockIdx.y / 3) * FLAT_NB; b < min(nl / 3, (int)(blockIdx.y / 3 + 1) * FLAT_NB); ++b) {
    if (state != nullptr && state[b0 + b].done) continue;
    __syncthreads();
    const double2 *a = alm + (int64_t)(b0 + b) * 3 * nmodes + (int64_t)kx * N;
    int ex[2] = {-100000, -100000};
    for (int q = threadIdx.x; q < N / 2; q += 256) {
      auto mode = [&](int ky, double sgn) {
        if (f == 0) return make_double2(inv_area * a[ky].x, inv_area * a[ky].y);
        const double2 e = a[nmodes + ky], bb = a[2 * nmodes + ky];
        const double c = rot[2 * q], s = sgn * rot[2 * q + 1];
        return f == 1 ? make_double2(e.x * c - bb.x * s, e.y * c - bb.y * s)
                      : make_double2(e.x * s + bb.x * c, e.y * s + bb.y * c);
      };
      const double2 hp = mode(q, 1.0);
      double2 cs = hp, sn = make_double2(0, 0);
      if (q > 0) {
        const double2 hm = mode(N - q, -1.0);
        cs = make_double2(hp.x + hm.x, hp.y + hm.y);
        sn = make_double2(hp.x - hm.x, hp.y - hm.y);
      }
      auto keep = [&](int ri, double c, double t) {
        double *o = vals + (ri * 4 + (q & 1)) * ld + slot4(q >> 1);
        o[0] = c;
        o[2 * ld] = t;
        ex[ri] = max(ex[ri], max(exp_of(c), exp_of(t)));
      };
      keep(0, cs.x, sn.y);
      keep(1, cs.y, -sn.x);
    }
    int e[2];
    const int col = col_of(S, kx, 3 * b + f);
    for (int ri = 0; ri < 2; ++ri) {
      e[ri] = max(-1000, block_max(ex[ri], red));  // (its barriers cover the staged values too)
      if (e[ri] >= SPLIT_NAN) e[ri] = SPLIT_NAN;
      if (threadIdx.x == 0) xexp[C.col0 + col + ri] = e[ri];
    }
    int ct, cit;
    col_place(C, col, ct, cit);
    digit_items(x + C.xi, C, C.ksi, ct, cit, ne, e, 2, [&](int ri, int fun) { return vals + (ri * 4 + fun) * ld; });
  }
}

// Place of row y in a column of the ring coefficients (pairs (y, N - 1 - y)).
__device__ __forceinline__ int flat_place(int y, int N) { return y < N / 2 ? 2 * y : 2 * (N - 1 - y) + 1; }

// The rows of orbit j under y -> N - y and N/2 - y; orbit 0 stands for the half
// orbits y = 0, N/2 and y = N/4, 3N/4.
__device__ __forceinline__ void flat_orbit(int j, int N, int at[4]) {
  at[0] = j;
  at[1] = N / 2 - j;
  at[2] = j ? N - j : N / 4;
  at[3] = j ? N / 2 + j : 3 * (N / 4);
}

// Orbit sums of a column into its rows.  grid (columns, lanes)
__global__ void __launch_bounds__(256) k_flat_unfold(const double *__restrict__ v, const int *__restrict__ xexp,
                                                     double2 *__restrict__ rc, const DftSet *__restrict__ sets,
                                                     const DftCol *__restrict__ cols, int lane0, int mmax,
                                                     const SolveState *__restrict__ state) {
  const int kx = blockIdx.x, lane = blockIdx.y, al = lane0 + lane;
  if (state != nullptr && state[al / 3].done) return;
  const DftCol C = cols[0];
  const int N = sets[0].n, col = col_of(sets[0], kx, lane);
  const double *vc = v + C.v + (int64_t)col * 4 * C.njp;
  double2 *o = rc + ((int64_t)al * (mmax + 1) + kx) * N;
  for (int j = threadIdx.x; j < N / 4; j += 256) {
    double s[2][4];
#pragma unroll
    for (int ri = 0; ri < 2; ++ri) {
      const double *u = vc + ri * 4 * C.njp;
      const double ce = u[j], co = u[C.njp + j], se = u[2 * C.njp + j], so = u[3 * C.njp + j];
      const double a1 = ce + co, a2 = ce - co, b1 = so + se, b2 = so - se;
      s[ri][0] = a1 - b1;
      s[ri][1] = a2 - b2;
      s[ri][2] = a1 + b1;
      s[ri][3] = a2 + b2;
      if (j == 0) {
        const int h = N / 4;
        const double c4 = u[h] + u[C.njp + h], s4 = u[2 * C.njp + h] + u[3 * C.njp + h];
        s[ri][0] = a1;
        s[ri][1] = a2;
        s[ri][2] = c4 - s4;
        s[ri][3] = c4 + s4;
      }
      if (xexp[C.col0 + col + ri] >= SPLIT_NAN) s[ri][0] = s[ri][1] = s[ri][2] = s[ri][3] = NAN;
    }
    int at[4];
    flat_orbit(j, N, at);
#pragma unroll
    for (int k = 0; k < 4; ++k) o[flat_place(at[k], N)] = make_double2(s[0][k], s[1][k]);
  }
}

// The rows of a column folded over their orbits, as digits.  grid (columns, lanes)
__global__ void __launch_bounds__(256) k_flat_xana(const double2 *__restrict__ rc, unsigned char *__restrict__ x,
                                                   int *__restrict__ xexp, const DftSet *__restrict__ sets,
                                                   const DftCol *__restrict__ cols, int lane0, int mmax,
                                                   const SolveState *__restrict__ state) {
  extern __shared__ __align__(16) double vals[];  // [re, im][CE, CO, SE, SO][slots of nj]
  __shared__ int red[8];
  const int kx = blockIdx.x, lane = blockIdx.y, al = lane0 + lane;
  if (state != nullptr && state[al / 3].done) return;
  const DftSet S = sets[0];
  const DftCol C = cols[0];
  const int N = S.n, ld = slots4(S.nj), col = col_of(S, kx, lane);
  const double2 *src = rc + ((int64_t)al * (mmax + 1) + kx) * N;
  int ex[2] = {-100000, -100000};
  for (int j = threadIdx.x; j < N / 4; j += 256) {
    int at[4];
    flat_orbit(j, N, at);
    double2 r[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) r[k] = src[flat_place(at[k], N)];
#pragma unroll
    for (int ri = 0; ri < 2; ++ri) {
      double y[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) y[k] = ri ? r[k].y : r[k].x;
      auto keep = [&](int i, double ce, double co, double se, double so) {
        double *o = vals + ri * 4 * ld + slot4(i);
        o[0] = ce;
        o[ld] = co;
        o[2 * ld] = se;
        o[3 * ld] = so;
        ex[ri] = max(max(ex[ri], max(exp_of(ce), exp_of(co))), max(exp_of(se), exp_of(so)));
      };
      if (j == 0) {
        keep(0, y[0] + y[1], y[0] - y[1], 0.0, 0.0);
        keep(N / 4, y[2] + y[3], 0.0, 0.0, y[2] - y[3]);
      } else {
        const double c0 = y[0] + y[2], c1 = y[1] + y[3], d0 = y[0] - y[2], d1 = y[1] - y[3];
        keep(j, c0 + c1, c0 - c1, d0 - d1, d0 + d1);
      }
    }
  }
  int e[2];
  for (int ri = 0; ri < 2; ++ri) {
    e[ri] = max(-1000, block_max(ex[ri], red));
    if (e[ri] >= SPLIT_NAN) e[ri] = SPLIT_NAN;
    if (threadIdx.x == 0) xexp[C.col0 + col + ri] = e[ri];
  }
  int ct, cit;
  col_place(C, col, ct, cit);
  digit_items(x + C.xf, C, C.ksf, ct, cit, S.nj, e, 2, [&](int ri, int fun) { return vals + (ri * 4 + fun) * ld; });
}

struct DftArgs {
  const DftTile *tiles;
  int ntiles;
  const CUtensorMap *maps;
  const DftSet *sets;
  const DftCol *cols;
  const int *pair_of;
  const unsigned char *x;
  const int *xexp;
  int nl, lane0, mmax, npairs;
  int eq;               // the pair without a mirror ring (-1: none)
  bool columns;         // forward: columns of a flat patch, modes +-q of complex sums
  double *v;            // inverse: orbit sums
  double2 *rc;          // forward: ring coefficients
  const SolveState *state;
  int nstages;
  int *err;
};

__device__ __forceinline__ void map_acquire(const CUtensorMap *map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(map) : "memory");
}

// FWD: rows are orders of one parity (cosine and sine sums in one tile), K the
// orbits; else rows are orbits of one matrix, K the orders.  The structure of
// the Legendre products (k_split): the first warps drain, then one streams
// and one issues.
template <bool FWD, int NQ>
__global__ void __launch_bounds__(dft_threads(NQ), 1) k_dft(const DftArgs A) {
  constexpr int DRAIN = dft_drain_warps(NQ), THREADS = dft_threads(NQ), QW = 8 * NQ / DRAIN;  // QW: column quads per warp
  constexpr int S = SPLIT_S, G = Weights<S>::G, N0 = 8 * NQ;
  constexpr int SET = (G * N0 + ((N0 & 15) ? 8 : 0) + 15) / 16 * 16;
  constexpr int COLS = 2 * SET <= 128 ? 128 : (2 * SET <= 256 ? 256 : 512);
  constexpr int ABYTES = S * 4096, BBYTES = S * N0 * 32, ZBYTES = (N0 + 8) * 32, STAGE = ABYTES + BBYTES + ZBYTES;
  constexpr int NF = FWD ? 2 : 1;
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t bars[2 * DFT_MAX_STAGES + 5];
  __shared__ uint32_t tslot;
  __shared__ int cta_bad;
  __shared__ uint32_t live[128];  // unfinished right-hand sides of the group (4096 at most)
  uint64_t *full = bars, *empty = bars + DFT_MAX_STAGES, *tfull = bars + 2 * DFT_MAX_STAGES, *tempty = tfull + 2,
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
  for (int i = tid; i < NS * (ZBYTES / 16); i += THREADS)
    *reinterpret_cast<uint4 *>(sm + (size_t)(i / (ZBYTES / 16)) * STAGE + ABYTES + BBYTES + (i % (ZBYTES / 16)) * 16) =
        make_uint4(0, 0, 0, 0);
  fence_proxy_async();
  if (warp == 0) tmem_alloc(&tslot, COLS);
  if (A.state != nullptr)
    for (int b = tid; (b & ~31) < A.nl / 3; b += THREADS) {
      const uint32_t word = __ballot_sync(0xffffffffu, b < A.nl / 3 && !A.state[A.lane0 / 3 + b].done);
      if (lane == 0) live[b >> 5] = word;
    }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  auto finished = [&](const DftTile &T) {  // the same for every role: the states do not change under the kernel
    if (A.state == nullptr) return false;
    for (int b = T.b0; b <= T.b1; ++b)
      if ((live[b >> 5] >> (b & 31)) & 1u) return false;
    return true;
  };
  const uint32_t tbase = tslot;
  int issued = 0;
  const uint32_t sm_a = smem_u32(sm), full_a = smem_u32(full), empty_a = smem_u32(empty);

  if (warp == DRAIN) {
    if (lane == 0) {
      bool ok = true;
      StageAt at;
      for (int t = blockIdx.x; ok && t < A.ntiles; t += gridDim.x) {
        const DftTile T = A.tiles[t];
        if (finished(T)) continue;
        const CUtensorMap *map = A.maps + 2 * T.set + (FWD ? 1 : 0);
        map_acquire(map);
        for (int k0 = 0; ok && k0 < T.ks; k0 += DFT_CHUNK)
          for (int f = 0; ok && f < NF; ++f)
            for (int k = k0; k < min(k0 + DFT_CHUNK, T.ks); ++k) {
              if (issued >= NS && !mbar_wait_at(empty_a + 8 * at.s, at.phase ^ 1, A.err)) {
                ok = false;
                break;
              }
              const uint32_t dst = sm_a + at.s * STAGE, bar = full_a + 8 * at.s;
              mbar_expect_tx_at(bar, ABYTES + BBYTES);
              const int z = T.z + f * T.zfun;
              if (FWD)
                tma_box_at(dst, map, 2 * k, z, bar);
              else
                tma_box_at(dst, map, 16 * T.row, z + 2 * k, bar);
              bulk_g2s_at(dst + ABYTES, A.x + T.x + f * T.xfun + (int64_t)k * BBYTES, BBYTES, bar);
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
      const uint64_t ad0 = FWD ? split_desc(sm_a, 128, 256) : split_desc(sm_a, 2048, 128);
      const uint64_t bd0 = split_desc(sm_a + ABYTES, 128, 256);
      for (int t = blockIdx.x; ok && t < A.ntiles; t += gridDim.x) {
        if (finished(A.tiles[t])) continue;
        const int ks = A.tiles[t].ks, nch = NF * ((ks + DFT_CHUNK - 1) / DFT_CHUNK);
        for (int c = 0; ok && c < nch; ++c, ++cc) {
          const int set = cc & 1;
          if (cc >= 2 && !mbar_wait(&tempty[set], ((cc >> 1) - 1) & 1, A.err)) {
            ok = false;
            break;
          }
          fence_after_sync();
          const int nstep = min(DFT_CHUNK, ks - (c / NF) * DFT_CHUNK);
          const uint32_t d = tbase + set * SET;
          for (int k = 0; k < nstep; ++k) {
            if (!mbar_wait_at(full_a + 8 * at.s, at.phase, A.err)) {
              ok = false;
              break;
            }
            fence_after_sync();
            const uint64_t off = (uint64_t)(at.s * (STAGE >> 4));
            if (k == 0)
              split_step<S, N0, 4096, !FWD, true>(d, ad0 + off, bd0 + off);
            else
              split_step<S, N0, 4096, !FWD, false>(d, ad0 + off, bd0 + off);
            commit_at(empty_a + 8 * at.s);
            at.next(NS);
          }
          if (ok) commit(&tfull[set]);
        }
      }
      if (!ok) cta_bad = 1;
      commit(fin);
      mbar_wait(fin, 0, A.err);
    }
  } else {
    const int part = warp >> 2, wq = warp & 3;
    bool ok = true;
    int cc = 0;
    for (int t = blockIdx.x; ok && t < A.ntiles; t += gridDim.x) {
      const DftTile T = A.tiles[t];
      if (finished(T)) continue;
      const DftSet D = A.sets[T.set];
      const DftCol C = A.cols[T.set];
      const int ncol = D.npr * A.nl * 2, c0 = T.ct * C.w + part * QW * 4;
      const int cend = min(ncol, (T.ct + 1) * C.w);  // columns of the tile end here
      const int nch = NF * ((T.ks + DFT_CHUNK - 1) / DFT_CHUNK);
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
#pragma unroll
        for (int q = 0; q < QW; ++q) {
          if (c0 + 4 * q >= cend) break;
          uint32_t g[G][4];
#pragma unroll
          for (int k = 0; k < G; ++k) tmem_ld4(tcol + k * N0 + q * 4, g[k]);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            int w[G];
#pragma unroll
            for (int k = 0; k < G; ++k) w[k] = __float2int_rn(__uint_as_float(g[k][e]));
            if (NF == 2 && (c & 1))
              acc[NF - 1][q][e].add(w);
            else
              acc[0][q][e].add(w);
          }
        }
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[set]);
      }
      if (!ok) break;
      const int row = T.row * 128 + wq * 32 + lane;
      if (!FWD) {
        if (row < D.nj) {
#pragma unroll
          for (int q = 0; q < QW; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int col = c0 + 4 * q + e;
              if (col >= cend) break;
              A.v[C.v + ((int64_t)col * 4 + T.fun) * C.njp + row] = value_of(acc[0][q][e], A.xexp[C.col0 + col]);
            }
        }
      } else {
        const int qo = 2 * row + T.fun;  // the order
        if (qo <= D.mx) {
#pragma unroll
          for (int q = 0; q < QW; ++q)
#pragma unroll
            for (int e = 0; e < 4; e += 2) {  // the two sides of one pair and lane
              const int col = c0 + 4 * q + e;
              if (col >= cend) break;
              const int pc = col >> 1, ln = pc / D.npr, pl = pc - ln * D.npr, al = A.lane0 + ln;
              if (A.state != nullptr && A.state[al / 3].done) continue;
              const int pair = A.pair_of[D.pair0 + pl];
              const bool equator = pair == A.eq;
              const int en = A.xexp[C.col0 + col], es = equator ? 0 : A.xexp[C.col0 + col + 1];
              double2 f = make_double2(value_of(acc[0][q][e], en), -value_of(acc[NF - 1][q][e], en));
              double2 s = make_double2(value_of(acc[0][q][e + 1], es), -value_of(acc[NF - 1][q][e + 1], es));
              if (en >= SPLIT_NAN) f.x = f.y = NAN;
              if (es >= SPLIT_NAN) s.x = s.y = NAN;
              if (A.columns) {  // f, s: the sums of the real and imaginary parts
                double2 *o = A.rc + ((int64_t)al * (A.mmax + 1) + pair) * D.n;
                o[qo] = make_double2(f.x - s.y, f.y + s.x);
                if (qo > 0) o[D.n - qo] = make_double2(f.x + s.y, s.x - f.y);
                continue;
              }
              double2 *o = A.rc + (((int64_t)al * (A.mmax + 1) + qo) * A.npairs + pair) * 2;
              o[0] = f;
              if (!equator) o[1] = s;
            }
        }
      }
    }
    if (!ok && lane == 0) cta_bad = 1;
  }
  __syncthreads();
  if (cta_bad && warp == DRAIN && lane == 0)
    for (int c = max(0, issued - NS); c < issued; ++c) mbar_wait(&full[c % NS], (c / NS) & 1, A.err);
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tbase, COLS);
}

void drop_cut(DftCut &c) {
  if (c.cols) cudaFree(c.cols);
  for (auto &d : c.tiles)
    for (DftTile *t : d)
      if (t) cudaFree(t);
}

}  // namespace

// Matrix sets of a plan: polar radii, then the belt with and without the shift; a flat patch has one.
static std::vector<DftSet> dft_sets(const dm_plan *p, std::vector<int> *pairs, std::vector<int> *set_of) {
  std::vector<DftSet> sets;
  auto make = [&](int n, int shift) {
    DftSet s{};
    s.n = n;
    s.shift = shift;
    s.nj = n / 4 + (shift ? 0 : 1);
    s.mx = std::min(p->mmax, n / 2);
    s.rq = 2 * ((s.mx / 2 + 16) / 16);
    s.nyo = (s.nj + 7) / 8;
    s.pair0 = (int)pairs->size();
    return s;
  };
  if (p->flat) {  // every row of the grid
    DftSet s = make(p->flatN, 0);
    for (int q = 0; q < p->npairs; ++q) pairs->push_back(q);
    s.npr = p->npairs;
    sets.push_back(s);
    set_of->assign(p->npairs, 0);
    return sets;
  }
  for (int i = 1; i < p->nside; ++i) {
    DftSet s = make(4 * i, 1);
    s.npr = 1;
    pairs->push_back(i - 1);
    sets.push_back(s);
  }
  for (int shift = 1; shift >= 0; --shift) {
    DftSet s = make(4 * p->nside, shift);
    for (int q = p->nside - 1; q < p->npairs; ++q)
      if (p->rings_h[q].shift == shift) pairs->push_back(q);
    s.npr = (int)pairs->size() - s.pair0;
    if (s.npr > 0) sets.push_back(s);
  }
  for (size_t k = 0; k < sets.size(); ++k)
    for (int q = 0; q < sets[k].npr; ++q) set_of->push_back((int)k);
  return sets;
}

static size_t set_bytes(const DftSet &s) { return (size_t)SPLIT_S * 4 * s.rq * s.nyo * 128; }

// Bytes of the matrix sets of a sphere plan.
size_t dft_table_bytes(int nside, int mmax) {
  double b = 0;
  for (int i = 1; i <= nside; ++i)
    b += (double)SPLIT_S * 4 * 2 * ((std::min(mmax, 2 * i) / 2 + 16) / 16) * ((i + 8) / 8) * 128 * (i == nside ? 2 : 1);
  return (size_t)b;
}

// All that the device holds of the tables goes.
static void drop_tables(DftTables *T) {
  for (DftCut &c : T->cuts) drop_cut(c);
  T->cuts.clear();
  for (void *q : {(void *)T->dig, (void *)T->sets_dev, (void *)T->maps, (void *)T->pair_of, (void *)T->set_of,
                  (void *)T->x, (void *)T->v, (void *)T->xexp})
    if (q) cudaFree(q);
  T->dig = T->x = nullptr;
  T->sets_dev = nullptr;
  T->maps = nullptr;
  T->pair_of = T->set_of = T->xexp = nullptr;
  T->v = nullptr;
  T->xexp_n = 0;
  T->bytes = 0;
}

void dft_release(dm_plan *p) {
  if (!p->dft) return;
  drop_tables(p->dft);
  delete p->dft;
  p->dft = nullptr;
}
void dft_new(dm_plan *p) {
  p->dft = new DftTables();
  p->dft->batch = p->batch;
}
void dft_disable(dm_plan *p) { p->dft->disabled = true; }
int64_t dft_bytes(const dm_plan *p) { return p->dft ? p->dft->bytes : 0; }

// Column digits of nl lanes: bytes of the larger direction.
static size_t cut_layout(const DftTables *T, int nl, std::vector<DftCol> *cols, int *ncol, size_t *vcount) {
  size_t xi = 0, xf = 0, v = 0;
  int c0 = 0;
  cols->clear();
  for (const DftSet &s : T->sets) {
    DftCol c{};
    const int n = s.npr * nl * 2;
    c.nct = (n + 31) / 32;
    c.w = ((n + c.nct - 1) / c.nct + 3) / 4 * 4;
    c.nct = (n + c.w - 1) / c.w;
    c.n0 = (c.w + 7) / 8 * 8;
    c.ksi = s.rq / 2;
    c.ksf = (s.nj + 15) / 16;
    c.col0 = c0;
    c.njp = (s.nj + 3) / 4 * 4;
    c.xi = (int64_t)xi;
    c.xf = (int64_t)xf;
    c.v = (int64_t)v;
    const size_t blk = (size_t)SPLIT_S * c.n0 * 32;
    xi += 4 * (size_t)c.nct * c.ksi * blk;
    xf += 4 * (size_t)c.nct * c.ksf * blk;
    v += (size_t)n * 4 * c.njp;
    c0 += n;
    cols->push_back(c);
  }
  *ncol = c0;
  *vcount = v;
  return std::max(xi, xf);
}

// Right-hand sides per group: as many as the column digits of DFT_SCRATCH bytes hold.
static int dft_group(const DftTables *T, int batch) {
  std::vector<DftCol> cols;
  int nc;
  size_t v;
  int g = batch;
  while (g > 1 && cut_layout(T, 3 * g, &cols, &nc, &v) > DFT_SCRATCH) g = (g + 1) / 2;
  return g;
}

// Matrix sets, tensor maps and the scratch of the largest group: once per plan,
// and kept until it goes, because a captured graph may name them.
static cudaError_t dft_setup(dm_plan *p, cudaStream_t st) {
  DftTables *T = p->dft;
  if (T->dig) return cudaSuccess;
  if (!encode_fn()) return cudaErrorNotSupported;
  std::vector<int> pairs, set_of;
  T->sets = dft_sets(p, &pairs, &set_of);
  T->nlist = (int)pairs.size();
  const int ns = (int)T->sets.size();
  int64_t total = 0;
  T->off.clear();
  for (const DftSet &s : T->sets) {
    T->off.push_back(total);
    total += (int64_t)set_bytes(s);
  }
  cudaError_t e;
  unsigned char *dig = nullptr;
  auto up = [&](auto **dst, const auto *src, size_t count) {
    if (*dst == nullptr)
      if (cudaError_t r = cudaMalloc((void **)dst, sizeof(*src) * count)) return r;
    return cudaMemcpyAsync((void *)*dst, src, sizeof(*src) * count, cudaMemcpyHostToDevice, st);
  };
  // the scratch of one right-hand side, of a whole group and of the last one
  size_t xb = 0, vc = 0;
  int nc = 0;
  const int g = dft_group(T, T->batch);
  for (int n : {1, g, T->batch % g}) {
    if (n == 0) continue;
    std::vector<DftCol> cols;
    int c;
    size_t v;
    xb = std::max(xb, cut_layout(T, 3 * n, &cols, &c, &v));
    vc = std::max(vc, v);
    nc = std::max(nc, c);
  }
  if (!T->x) {
    if ((e = table_alloc(p, (void **)&T->x, xb))) return e;
    T->bytes += (int64_t)xb;
  }
  if (!T->v) {
    if ((e = table_alloc(p, (void **)&T->v, sizeof(double) * vc))) return e;
    T->bytes += (int64_t)(sizeof(double) * vc);
  }
  if (!T->xexp) {
    if ((e = table_alloc(p, (void **)&T->xexp, sizeof(int) * 2 * nc))) return e;
    T->xexp_n = nc;
    T->bytes += (int64_t)(sizeof(int) * 2 * nc);
  }
  if ((e = table_alloc(p, (void **)&dig, (size_t)total))) return e;
  std::vector<CUtensorMap> maps(2 * ns);
  for (int k = 0; k < ns && !e; ++k) {
    const DftSet &s = T->sets[k];
    for (int dir = 0; dir < 2; ++dir) {
      const cuuint64_t dims[4] = {64, (cuuint64_t)s.nyo, (cuuint64_t)(4 * s.rq), SPLIT_S};
      const cuuint64_t strides[3] = {128, (cuuint64_t)s.nyo * 128, (cuuint64_t)(4 * s.rq) * s.nyo * 128};
      const cuuint32_t box[4] = {64, dir == 0 ? 16u : 2u, dir == 0 ? 2u : 16u, SPLIT_S};
      const cuuint32_t one[4] = {1, 1, 1, 1};
      if (encode_fn()(&maps[2 * k + dir], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, dig + T->off[k], dims, strides, box,
                      one, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        e = cudaErrorInvalidValue;
    }
    const int64_t items = (int64_t)4 * s.rq * 8 * s.nyo;
    k_dft_gen<<<(unsigned)std::min<int64_t>((items + 127) / 128, 4096), 128, 0, st>>>(s, dig + T->off[k]);
  }
  if (!e) e = cudaGetLastError();
  if (!e) e = up(&T->maps, maps.data(), maps.size());
  if (!e) e = up(&T->sets_dev, T->sets.data(), T->sets.size());
  if (!e) e = up(&T->pair_of, pairs.data(), pairs.size());
  if (!e) e = up(&T->set_of, set_of.data(), set_of.size());
  if (!e) e = cudaStreamSynchronize(st);
  if (e) {
    cudaFree(dig);
    return e;
  }
  T->dig = dig;
  T->bytes += total + (int64_t)(sizeof(CUtensorMap) * maps.size() + sizeof(DftSet) * ns + 2 * sizeof(int) * pairs.size());
  return cudaSuccess;
}

static cudaError_t dft_cut(dm_plan *p, int nl, cudaStream_t st) {
  DftTables *T = p->dft;
  DftCut K;
  K.nl = nl;
  std::vector<DftCol> cols;
  int ncol;
  size_t vcount;
  cut_layout(T, nl, &cols, &ncol, &vcount);
  cudaError_t e = cudaMalloc(&K.cols, sizeof(DftCol) * cols.size());
  if (!e) e = cudaMemcpyAsync(K.cols, cols.data(), sizeof(DftCol) * cols.size(), cudaMemcpyHostToDevice, st);
  for (int dir = 0; dir < 2 && !e; ++dir) {
    std::vector<DftTile> tiles[5];
    for (int k = 0; k < (int)T->sets.size(); ++k) {
      const DftSet &s = T->sets[k];
      const DftCol &c = cols[k];
      const int64_t blk = (int64_t)SPLIT_S * c.n0 * 32;
      const int ks = dir == 0 ? c.ksi : c.ksf;
      for (int fun = 0; fun < (dir == 0 ? 4 : 2); ++fun) {
        const int rows = dir == 0 ? s.nj : (s.mx - fun) / 2 + (s.mx >= fun ? 1 : 0);
        for (int r = 0; r < (rows + 127) / 128; ++r)
          for (int ct = 0; ct < c.nct; ++ct) {
            DftTile t{};
            t.set = k;
            t.fun = fun;
            t.row = r;
            t.ct = ct;
            t.ks = ks;
            t.z = fun * s.rq + (dir == 0 ? 0 : 16 * r);
            t.zfun = 2 * s.rq;
            t.n0 = c.n0;
            t.b0 = ct * c.w / (6 * s.npr);
            t.b1 = (std::min(2 * s.npr * nl, (ct + 1) * c.w) - 1) / (6 * s.npr);
            t.x = (dir == 0 ? c.xi : c.xf) + ((int64_t)fun * c.nct + ct) * ks * blk;
            t.xfun = (int64_t)2 * c.nct * ks * blk;
            tiles[c.n0 / 8].push_back(t);
          }
      }
    }
    for (int q = 1; q < 5 && !e; ++q) {
      if (tiles[q].empty()) continue;
      std::stable_sort(tiles[q].begin(), tiles[q].end(), [](const DftTile &a, const DftTile &b) { return a.ks > b.ks; });
      e = cudaMalloc(&K.tiles[dir][q], sizeof(DftTile) * tiles[q].size());
      if (!e)
        e = cudaMemcpyAsync(K.tiles[dir][q], tiles[q].data(), sizeof(DftTile) * tiles[q].size(),
                            cudaMemcpyHostToDevice, st);
      if (!e) e = cudaStreamSynchronize(st);
      K.ntiles[dir][q] = (int)tiles[q].size();
    }
  }
  if (!e) e = cudaStreamSynchronize(st);
  if (e) {
    drop_cut(K);
    return e;
  }
  T->cuts.push_back(K);
  return cudaSuccess;
}

size_t dft_scratch_bytes(int nside, int batch) {  // bound of the column digits and orbit sums
  const double px = 12.0 * nside * nside * 3 * batch;
  return (size_t)(std::min(1.5 * px * 12.0, 2.0 * (double)DFT_SCRATCH) + std::min(1.3 * px * 8.0, 1.5 * (double)DFT_SCRATCH)) +
         ((size_t)32 << 20);
}

static const DftCut *dft_find(const DftTables *T, int nl) {
  for (const DftCut &c : T->cuts)
    if (c.nl == nl) return &c;
  return nullptr;
}

template <bool FWD>
static cudaError_t dft_products(dm_plan *p, const DftCut &K, int lane0, const SolveState *state, cudaStream_t st,
                                bool columns = false) {
  DftTables *T = p->dft;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if (cudaError_t r = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) return r;
  for (int q = 4; q >= 1; --q) {
    const int nt = K.ntiles[FWD][q];
    if (nt == 0) continue;
    DftArgs A;
    A.tiles = K.tiles[FWD][q];
    A.ntiles = nt;
    A.maps = T->maps;
    A.sets = T->sets_dev;
    A.cols = K.cols;
    A.pair_of = T->pair_of;
    A.x = T->x;
    A.xexp = T->xexp + (FWD ? T->xexp_n : 0);
    A.nl = K.nl;
    A.lane0 = lane0;
    A.mmax = p->mmax;
    A.npairs = p->npairs;
    A.eq = p->flat ? -1 : p->npairs - 1;
    A.columns = columns;
    A.v = T->v;
    A.rc = p->rc;
    A.state = state;
    A.err = p->tc_err;
    const int n0 = 8 * q, stage = SPLIT_S * 4096 + SPLIT_S * n0 * 32 + (n0 + 8) * 32;
    A.nstages = std::min(DFT_MAX_STAGES, (int)((224u << 10) / stage));
    const size_t smem = (size_t)A.nstages * stage;
    auto go = [&](auto kern) {
      if (cudaError_t r = dyn_smem_allow(kern, smem)) return r;
      kern<<<std::min(sms, nt), dft_threads(q), smem, st>>>(A);
      return cudaGetLastError();
    };
    cudaError_t e;
    switch (q) {
      case 1: e = go(k_dft<FWD, 1>); break;
      case 2: e = go(k_dft<FWD, 2>); break;
      case 3: e = go(k_dft<FWD, 3>); break;
      default: e = go(k_dft<FWD, 4>); break;
    }
    if (e) return e;
  }
  return cudaSuccess;
}

static size_t xinv_smem(const dm_plan *p) { return sizeof(double) * 8 * slots4(p->mmax / 2 + 1); }
static size_t pix_smem(const dm_plan *p) { return sizeof(double) * 8 * slots4((p->flat ? p->flatN / 4 : p->nside) + 1); }

// Whether the products run; then their tables and the cuts of all groups exist.
cudaError_t dft_use(dm_plan *p, cudaStream_t st, bool *use) {
  DftTables *T = p->dft;
  *use = false;
  if (!T || T->disabled || p->ring_fft || p->tune_only_class >= 0) return cudaSuccess;
  if (p->flat ? !flat_products(p->flatN, p->batch) : p->npix * p->batch < DFT_MIN_PIXELS) return cudaSuccess;
  if (std::max(xinv_smem(p), pix_smem(p)) > DFT_SMEM) return cudaSuccess;
  const int B = p->batch;
  auto found = [&](int gb) {
    for (int b0 = 0; b0 < B; b0 += gb)
      if (!dft_find(T, 3 * std::min(gb, B - b0))) return false;
    return true;
  };
  if (T->dig && found(dft_group(T, B))) {
    *use = true;
    return cudaSuccess;
  }
  if (!T->dig && !p->flat && (int64_t)dft_table_bytes(p->nside, p->mmax) > p->dft_cap) {
    T->disabled = true;
    return cudaSuccess;
  }
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return cudaSuccess;
  }
  if (T->shortage.lasts(p)) return cudaSuccess;
  const bool fresh = T->cuts.empty();
  cudaError_t e = dft_setup(p, st);
  const int gb = e ? B : dft_group(T, B);
  for (int b0 = 0; !e && b0 < B; b0 += gb)
    if (!dft_find(T, 3 * std::min(gb, B - b0))) e = dft_cut(p, 3 * std::min(gb, B - b0), st);
  if (e) {
    if (fresh) drop_tables(T);  // no launch has named them yet
    cudaGetLastError();
    if (e == cudaErrorNotSupported) T->disabled = true;
    if (e == cudaErrorMemoryAllocation) T->shortage.note(p);
    return e == cudaErrorMemoryAllocation || e == cudaErrorNotSupported ? cudaSuccess : e;
  }
  T->shortage = Shortage();
  *use = true;
  return cudaSuccess;
}

// The FP64 ring stage (modes of ring_stage) as split products; *ran = false
// when the FFT kernels have to do it.
cudaError_t dft_ring_stage(dm_plan *p, int mode, const double *in_map, double *out_map, cudaStream_t st, bool *ran) {
  const cudaError_t eu = dft_use(p, st, ran);
  if (eu || !*ran) return eu;
  const int gb = dft_group(p->dft, p->batch);
  DftTables *T = p->dft;
  const int eq = p->flat ? -1 : p->npairs - 1;
  const SolveState *state = (mode == RING_ITER || mode == RING_INIT) ? p->state : nullptr;
  for (int b0 = 0; b0 < p->batch; b0 += gb) {
    const int nl = 3 * std::min(gb, p->batch - b0), lane0 = 3 * b0;
    const DftCut *K = dft_find(T, nl);
    cudaError_t e;
    int *ei = T->xexp, *ef = T->xexp + T->xexp_n;
    if (mode == RING_ITER || mode == RING_INV_MAP) {
      const size_t sm = xinv_smem(p);
      if ((e = dyn_smem_allow(k_dft_xinv, sm))) return e;
      k_dft_xinv<<<dim3(T->nlist, nl), 128, sm, st>>>(p->rc, T->x, ei, T->sets_dev, K->cols, T->pair_of, T->set_of,
                                                      lane0, p->mmax, p->npairs, eq, state);
      if ((e = dft_products<false>(p, *K, lane0, state, st))) return e;
    }
    const size_t sp = pix_smem(p);
    auto pix = [&](auto kern) {
      if (cudaError_t r = dyn_smem_allow(kern, sp)) return r;
      kern<<<dim3(T->nlist, nl), 256, sp, st>>>(p->rings, T->v, T->x, ei, ef, T->sets_dev, K->cols, T->pair_of,
                                                T->set_of, lane0, eq, p->nrings, p->npix, in_map, out_map, p->w,
                                                p->wd, p->norms, state);
      return cudaGetLastError();
    };
    switch (mode) {
      case RING_ITER: e = pix(k_dft_pix<RING_ITER>); break;
      case RING_INV_MAP: e = pix(k_dft_pix<RING_INV_MAP>); break;
      case RING_INIT: e = pix(k_dft_pix<RING_INIT>); break;
      default: e = pix(k_dft_pix<RING_FWD_MAP>); break;
    }
    if (e) return e;
    if (mode == RING_INV_MAP) continue;
    if ((e = dft_products<true>(p, *K, lane0, state, st))) return e;
    // pairs with orders beyond n / 2: the shorter polar rings, and the belt where mmax exceeds 2 nside
    const int nrun = p->flat ? 0 : p->mmax > 2 * p->nside ? p->npairs : std::min(p->nside - 1, (p->mmax + 1) / 2);
    if (nrun > 0 && p->mmax >= 3) {
      k_dft_alias<<<dim3((nrun + 127) / 128, p->mmax - 2, nl), 128, 0, st>>>(p->rc, lane0, p->mmax, p->npairs,
                                                                             p->nside, nrun, state);
      if ((e = cudaGetLastError())) return e;
    }
  }
  return cudaSuccess;
}

// Column transforms of a flat patch as the same products; *ran = false when
// the FFT kernels have to do them.  Synthesis: modes to the ring coefficients;
// analysis: in place, to F[lane][kx][ky] (without the Nyquist modes).
cudaError_t dft_flat_columns(dm_plan *p, const double2 *alm, const SolveState *state, cudaStream_t st, bool *ran) {
  const cudaError_t eu = dft_use(p, st, ran);
  if (eu || !*ran) return eu;
  DftTables *T = p->dft;
  const int N = p->flatN, gb = dft_group(p->dft, p->batch);
  const size_t sx = sizeof(double) * (8 * slots4(N / 4) + N), sf = sizeof(double) * 8 * slots4(N / 4 + 1);
  for (int b0 = 0; b0 < p->batch; b0 += gb) {
    const int nb = std::min(gb, p->batch - b0), nl = 3 * nb, lane0 = 3 * b0;
    const DftCut *K = dft_find(T, nl);
    cudaError_t e;
    int *ei = T->xexp, *ef = T->xexp + T->xexp_n;
    if (alm) {
      if ((e = dyn_smem_allow(k_flat_xsyn, sx))) return e;
      k_flat_xsyn<<<dim3(N / 2, 3 * ((nb + FLAT_NB - 1) / FLAT_NB)), 256, sx, st>>>(
          alm, T->x, ei, T->sets_dev, K->cols, nl, b0, 1.0 / (p->flatL * p->flatL), p->nmodes, state);
      if ((e = dft_products<false>(p, *K, lane0, state, st))) return e;
      k_flat_unfold<<<dim3(N / 2, nl), 256, 0, st>>>(T->v, ei, p->rc, T->sets_dev, K->cols, lane0, p->mmax,
                                                     state);
      if ((e = cudaGetLastError())) return e;
    } else {
      if ((e = dyn_smem_allow(k_flat_xana, sf))) return e;
      k_flat_xana<<<dim3(N / 2, nl), 256, sf, st>>>(p->rc, T->x, ef, T->sets_dev, K->cols, lane0, p->mmax,
                                                    state);
      if ((e = dft_products<true>(p, *K, lane0, state, st, true))) return e;
    }
  }
  return cudaSuccess;
}

}  // namespace dmwf
