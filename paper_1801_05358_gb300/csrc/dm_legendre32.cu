// dm_legendre32.cu -- the mixed mode's Legendre stages on the FP32 pipe, from
// FP32 tables (12 bytes per multipole, order and ring pair for lambda, lam+
// and lam-): the synthesis of small plans, the analysis of small plans and of
// one or two right-hand sides, and both wherever no digit table is kept whole.
//
// With few columns the tables are the work, read once.  The split products
// (dm_split.cu) read 18 bytes per triple for any number of columns up to 32,
// in tiles of 128 ring pairs and behind a pass that makes the columns' digits:
// they take over where a plan fills them.
#include "dm_internal.h"
#include "dm_tc_tiles.cuh"

namespace dmwf {

namespace {

// The synthesis runs here below this many table rows and columns of an order
// (npairs x multipoles).  alm2map, k_syn32 and split products: nside 32, B 9
// 39.5 and 47.5 us; nside 64, B 3 49.8 and 53.3, B 17 110 and 130; nside 100
// (below the line), B 3 92 and 102, B 9 199 and 186; nside 128 (above), B 1 124
// and 91, B 9 271 and 235.
constexpr int64_t SYN32_MAX = 48 * 1024;
// The analysis of more than two right-hand sides runs here below this many.
// map2alm, k_ana32 and split products: nside 64 / lmax 128, B 12 79.9 and 89.1 us,
// B 25 149 and 167, B 50 291 and 304; nside 64 / lmax 190 (the line), B 12 102 and
// 115, B 17 152 and 155, B 50 402 and 393.
constexpr int64_t ANA32_MAX = 24 * 1024;

constexpr int SYN_THREADS = 128;
constexpr int SYN_CH = 64;
constexpr int SYN_UNROLL = 8;  // multipoles whose 24 table loads are in flight together

// Synthesis: thread = ring pair, NB right-hand sides, the sum over l in
// registers; the coefficients of 64 multipoles staged at a time.
// grid (batch / NB, pair blocks, orders).
template <int NB, typename T2>
__global__ void __launch_bounds__(SYN_THREADS) k_syn32(const float *__restrict__ tab, int ld,
                                                       const T2 *__restrict__ alm, float2 *__restrict__ rc, int lmax,
                                                       int mmax, int npairs, int64_t nalm,
                                                       const SolveState *__restrict__ state) {
  __shared__ float2 sT[NB][SYN_CH], sE[NB][SYN_CH], sB[NB][SYN_CH];
  const int b0 = blockIdx.x * NB, m = blockIdx.z;
  bool any = state == nullptr;
  for (int k = 0; k < NB && !any; ++k) any = !state[b0 + k].done;
  if (!any) return;
  const int p = blockIdx.y * SYN_THREADS + threadIdx.x, pp = min(p, npairs - 1);
  float2 v[NB][3][2];  // field, parity of l - m
#pragma unroll
  for (int k = 0; k < NB; ++k)
#pragma unroll
    for (int f = 0; f < 3; ++f) v[k][f][0] = v[k][f][1] = make_float2(0.f, 0.f);
  const int64_t base = abase(lmax, m), plane = nalm * (int64_t)ld;
  const float *tp = tab + base * ld + pp;
  for (int lc = m; lc <= lmax; lc += SYN_CH) {
    const int cnt = min(SYN_CH, lmax + 1 - lc);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt * NB; i += SYN_THREADS) {
      const int k = i / cnt, j = i - k * cnt;
      const T2 *a = alm + (int64_t)(b0 + k) * 3 * nalm + base + lc + j;
      sT[k][j] = make_float2((float)a[0].x, (float)a[0].y);
      sE[k][j] = make_float2((float)-a[nalm].x, (float)-a[nalm].y);
      sB[k][j] = make_float2((float)-a[2 * nalm].x, (float)-a[2 * nalm].y);
    }
    __syncthreads();
    const float *tc = tp + (int64_t)lc * ld;
    auto term = [&](int j, int e, float lam, float lp, float lq) {  // e: parity of l - m
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        const float2 t = sT[k][j], ne = sE[k][j], nb = sB[k][j];
        float2 &T = v[k][0][e], &Q = v[k][1][e], &U = v[k][2][e], &Qo = v[k][1][1 - e], &Uo = v[k][2][1 - e];
        T.x = fmaf(t.x, lam, T.x);
        T.y = fmaf(t.y, lam, T.y);
        Q.x = fmaf(ne.x, lp, Q.x);
        Q.y = fmaf(ne.y, lp, Q.y);
        U.x = fmaf(nb.x, lp, U.x);
        U.y = fmaf(nb.y, lp, U.y);
        Qo.x = fmaf(-nb.y, lq, Qo.x);
        Qo.y = fmaf(nb.x, lq, Qo.y);
        Uo.x = fmaf(ne.y, lq, Uo.x);
        Uo.y = fmaf(-ne.x, lq, Uo.y);
      }
    };
    for (int j = 0; j < cnt; j += SYN_UNROLL) {  // lc - m is a multiple of 64
      float t[SYN_UNROLL][3];
#pragma unroll
      for (int i = 0; i < SYN_UNROLL; ++i) {
        const int64_t o = (int64_t)min(j + i, cnt - 1) * ld;
        t[i][0] = tc[o];
        t[i][1] = tc[plane + o];
        t[i][2] = tc[2 * plane + o];
      }
#pragma unroll
      for (int i = 0; i < SYN_UNROLL; ++i)
        if (j + i < cnt) term(j + i, i & 1, t[i][0], t[i][1], t[i][2]);
    }
  }
  if (p >= npairs) return;
#pragma unroll
  for (int k = 0; k < NB; ++k) {
    const int b = b0 + k;
    if (state != nullptr && state[b].done) continue;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      float2 *o = rc + (((int64_t)(b * 3 + f) * (mmax + 1) + m) * npairs + p) * 2;
      const float2 x = v[k][f][0], y = v[k][f][1];
      o[0] = make_float2(x.x + y.x, x.y + y.y);
      if (p != npairs - 1) o[1] = make_float2(x.x - y.x, x.y - y.y);
    }
  }
}

constexpr int A32_WARPS = 8;
// multipoles per warp and pass: with four right-hand sides two, so that two blocks share an SM
__host__ __device__ constexpr int a32_rows(int nb) { return nb == 4 ? 2 : 4; }
constexpr int A32_LB = 128;    // multipoles per block

// The sums over a warp of N values a lane, each left in the lanes that the
// folding assigns it to: every step halves the values that a lane still holds
// (N = 48: 48 shuffles instead of 240 for a tree each, more than the products
// of 64 ring pairs); what is added to what is as in the trees.
template <int N, int O>
__device__ __forceinline__ void fold_sums(float *a, int lane, int &first) {
  if constexpr (O > 0) {
    if constexpr (N % 2 == 0) {
      const bool up = lane & O;
#pragma unroll
      for (int i = 0; i < N / 2; ++i) {
        const float keep = up ? a[N / 2 + i] : a[i], give = up ? a[i] : a[N / 2 + i];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, give, O);
      }
      if (up) first += N / 2;
      fold_sums<N / 2, O / 2>(a, lane, first);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) a[i] += __shfl_xor_sync(0xffffffffu, a[i], O);
      fold_sums<N, O / 2>(a, lane, first);
    }
  }
}
// values that a lane is left with, and the lane bits of those that share them
__host__ __device__ constexpr int folded(int n, int o) { return o == 0 ? n : folded(n % 2 ? n : n / 2, o / 2); }
__host__ __device__ constexpr int sharers(int n, int o) {
  return o == 0 ? 0 : (n % 2 ? o : 0) | sharers(n % 2 ? n : n / 2, o / 2);
}

// Analysis: each warp takes a32_rows multipoles and all ring pairs, 16 bytes per
// lane, function and multipole (12 loads in flight); values below
// 2^TC_FLOOR_EXP (the evanescent region) are not read.  At nside 256, one
// right-hand side: 105 us, split products 203.  grid (batch / NB, blocks of
// A32_LB multipoles, orders): blocks that read the same values run together and
// find them in L2; dynamic shared memory [NB][12][ldp]:
// (T, Q, U) x (even re, im, odd re, im) of every ring pair.
template <int NB>
__global__ void __launch_bounds__(32 * A32_WARPS, NB == 4 ? 2 : 0) k_ana32(const float *__restrict__ tab, int ldt,
                                                          const int *__restrict__ ks,
                                                          int npt, int nlt, const float2 *__restrict__ rc,
                                                          float2 *__restrict__ out, int lmax, int mmax, int npairs,
                                                          int64_t nalm, int ldp, int batch,
                                                          const SolveState *__restrict__ state) {
  constexpr int A32_ROWS = a32_rows(NB);
  extern __shared__ __align__(16) float G[];
  const int m = blockIdx.z, lb = blockIdx.y * A32_LB;  // l - m of the block's first multipole
  if (lb > lmax - m) return;
  const int b0 = blockIdx.x * NB, nb = NB == 4 ? min(NB, batch - b0) : NB;  // (of four the last block may hold fewer)
  rc += (int64_t)b0 * 3 * (mmax + 1) * npairs * 2;
  out += (int64_t)b0 * 3 * nalm;
  if (state != nullptr) state += b0;
  bool any = state == nullptr;
  for (int k = 0; k < nb && !any; ++k) any = !state[k].done;
  if (!any) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // first ring pair visible at the block's last multipole, down to a multiple of 128
  const int64_t kr = (int64_t)m * (npt + nlt) + npt + min(nlt - 1, lb / 128), ks2 = (int64_t)(mmax + 1) * (npt + nlt);
  const int p0 = min(16 * min(ks[kr], ks[kr + ks2]), npairs - 1) & ~127;
  for (int i = tid; i < (ldp - p0) * 3 * NB; i += 32 * A32_WARPS) {
    const int p = p0 + i % (ldp - p0), kf = i / (ldp - p0);
    float2 n = make_float2(0.f, 0.f), s = n;
    if (p < npairs && kf < 3 * nb) {
      const float2 *g = rc + ((int64_t)kf * (mmax + 1) + m) * npairs * 2 + 2 * p;
      n = g[0];
      if (p != npairs - 1) s = g[1];
    }
    float *o = G + (int64_t)kf * 4 * ldp + p;
    o[0] = n.x + s.x;
    o[ldp] = n.y + s.y;
    o[2 * ldp] = n.x - s.x;
    o[3 * ldp] = n.y - s.y;
  }
  __syncthreads();
  const int64_t base = abase(lmax, m), plane = nalm * (int64_t)ldt;
  for (int r0 = lb + warp * A32_ROWS; r0 < min(lb + A32_LB, lmax - m + 1); r0 += A32_WARPS * A32_ROWS) {
    float acc[A32_ROWS][NB][6];
#pragma unroll
    for (int r = 0; r < A32_ROWS; ++r)
#pragma unroll
      for (int k = 0; k < NB; ++k)
#pragma unroll
        for (int c = 0; c < 6; ++c) acc[r][k][c] = 0.f;
    for (int p = p0 + 4 * lane; p < npairs; p += 128) {
      float4 t[A32_ROWS][3];
#pragma unroll
      for (int r = 0; r < A32_ROWS; ++r) {
        const int l = min(m + r0 + r, lmax);
#pragma unroll
        for (int f = 0; f < 3; ++f)
          t[r][f] = __ldg(reinterpret_cast<const float4 *>(tab + f * plane + (base + l) * ldt + p));
      }
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        float4 g[12];
#pragma unroll
        for (int c = 0; c < 12; ++c)
          g[c] = *reinterpret_cast<const float4 *>(G + ((int64_t)k * 12 + c) * ldp + p);
        const float *gf = reinterpret_cast<const float *>(g);
#pragma unroll
        for (int r = 0; r < A32_ROWS; ++r) {
          const int q = (r & 1) * 2, o = 2 - q;  // this parity (of l - m; r0 is a multiple of 4) and the other
          const float *lam = reinterpret_cast<const float *>(&t[r][0]);
          const float *lp = reinterpret_cast<const float *>(&t[r][1]), *lq = reinterpret_cast<const float *>(&t[r][2]);
          float *a = acc[r][k];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            a[0] = fmaf(lam[e], gf[4 * (0 + q) + e], a[0]);
            a[1] = fmaf(lam[e], gf[4 * (1 + q) + e], a[1]);
            // aE = -(lam+ Q + i lam- U'), aB = -(lam+ U - i lam- Q') (' : the other parity)
            a[2] = fmaf(-lp[e], gf[4 * (4 + q) + e], fmaf(lq[e], gf[4 * (9 + o) + e], a[2]));
            a[3] = fmaf(-lp[e], gf[4 * (5 + q) + e], fmaf(-lq[e], gf[4 * (8 + o) + e], a[3]));
            a[4] = fmaf(-lp[e], gf[4 * (8 + q) + e], fmaf(-lq[e], gf[4 * (5 + o) + e], a[4]));
            a[5] = fmaf(-lp[e], gf[4 * (9 + q) + e], fmaf(lq[e], gf[4 * (4 + o) + e], a[5]));
          }
        }
      }
    }
    if constexpr (NB > 1) {
      constexpr int V = A32_ROWS * NB * 6;
      float *v = &acc[0][0][0];
      int first = 0;
      fold_sums<V, 16>(v, lane, first);
      if ((lane & sharers(V, 16)) == 0)
#pragma unroll
        for (int i = 0; i < folded(V, 16); ++i) {
          const int r = (first + i) / (6 * NB), k = (first + i) / 6 % NB, c = (first + i) % 6;
          if (r0 + r <= lmax - m && k < nb && (state == nullptr || !state[k].done))
            reinterpret_cast<float *>(out)[2 * ((int64_t)(3 * k + c / 2) * nalm + base + m + r0 + r) + c % 2] = v[i];
        }
    } else {
#pragma unroll
      for (int r = 0; r < A32_ROWS; ++r)
#pragma unroll
        for (int k = 0; k < NB; ++k) {
#pragma unroll
          for (int c = 0; c < 6; ++c)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc[r][k][c] += __shfl_xor_sync(0xffffffffu, acc[r][k][c], o);
          if (lane == 0 && r0 + r <= lmax - m && (state == nullptr || !state[k].done)) {
            float2 *o = out + (int64_t)k * 3 * nalm + base + m + r0 + r;
            o[0] = make_float2(acc[r][k][0], acc[r][k][1]);
            o[nalm] = make_float2(acc[r][k][2], acc[r][k][3]);
            o[2 * nalm] = make_float2(acc[r][k][4], acc[r][k][5]);
          }
        }
    }
  }
}

int table_ld(const dm_plan *p) { return (p->npairs + 3) & ~3; }  // 16-byte rows
int64_t order_entries(const dm_plan *p) { return (int64_t)p->npairs * (p->lmax + 1); }

// The FP32 kernels take every size and batch where the split products would
// have to make their digits again in each stage call (no whole table), when the
// tensor cores are turned off and where every value's precision counts.  An iteration at nside 1024 / lmax 2048, one
// and three right-hand sides: 14.5 and 28.5 ms here, 425 and 426 with slabs of
// digits; at nside 512 / lmax 1535 with seven, slabs 103, whole digits 8.6.
bool instead(const dm_plan *p) { return !p->use_tc || p->each_value || !split_whole(p); }

// The FP32 tables, made on first use: not while the stream is captured, on a
// plan that shares another's tables, or where they leave no room for the
// anchors' digits (a slab at least).
bool tables(dm_plan *p, cudaStream_t st) {
  if (p->tab32) return true;
  const double bytes = 12.0 * (double)p->nalm * table_ld(p);
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (p->is_view || cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return false;
  }
  if (p->tab32_short.lasts(p)) return false;
  const double digits =
      split_bytes(p) > 0 ? 0.0  // made already
                         : std::min((double)p->ffs_cap, (double)split_table_bytes(p->lmax, p->mmax, p->npairs)) +
                               (double)split_scratch_bytes(p->lmax, p->npairs, p->batch, p->scratch_cap);
  if (bytes + digits > (double)table_room(p)) {
    p->tab32_short.note(p);
    return false;
  }
  float *t = nullptr;
  int *ks = nullptr;
  cudaError_t e = table_alloc(p, (void **)&t, (size_t)bytes);
  if (!e && table_ld(p) != p->npairs) e = cudaMemsetAsync(t, 0, (size_t)bytes, st);
  if (!e) e = gen_tables32(p, t, table_ld(p), st);
  if (!e && !p->tc_ks) e = visible_steps(p, TC_FLOOR_EXP, &ks);
  if (e) {
    cudaGetLastError();
    cudaFree(t);
    p->tab32_short.note(p);
    return false;
  }
  p->tab32 = t;
  if (ks) p->tc_ks = ks;
  p->bytes += (int64_t)bytes;
  return true;
}

constexpr size_t ANA32_SMEM = 220u << 10;
size_t ana32_smem(const dm_plan *p, int nb) {
  return sizeof(float) * 12 * (size_t)((p->npairs + 127) / 128 * 128) * nb;
}

}  // namespace

bool syn32_ready(dm_plan *p, cudaStream_t st) {
  return (order_entries(p) < SYN32_MAX || instead(p)) && tables(p, st);
}

bool ana32_ready(dm_plan *p, cudaStream_t st) {
  if (p->batch > 2 && order_entries(p) >= ANA32_MAX && !instead(p)) return false;
  return ana32_smem(p, 1) <= ANA32_SMEM && tables(p, st);
}

cudaError_t syn32(dm_plan *p, const double2 *alm, const float2 *e32, cudaStream_t st) {
  const SolveState *state = p->state_active ? p->state : nullptr;
  const int nb = p->batch % 4 == 0 ? 4 : 1;
  const dim3 g(p->batch / nb, (p->npairs + SYN_THREADS - 1) / SYN_THREADS, p->mmax + 1);
  auto go = [&](auto kern, const auto *a) {
    kern<<<g, SYN_THREADS, 0, st>>>(p->tab32, table_ld(p), a, p->rc32, p->lmax, p->mmax, p->npairs, p->nalm, state);
    return cudaGetLastError();
  };
  if (e32) return nb == 4 ? go(k_syn32<4, float2>, e32) : go(k_syn32<1, float2>, e32);
  return nb == 4 ? go(k_syn32<4, double2>, alm) : go(k_syn32<1, double2>, alm);
}

cudaError_t ana32(dm_plan *p, cudaStream_t st) {
  const SolveState *state = p->state_active ? p->state : nullptr;
  const int npt = (p->npairs + 127) / 128, nlt = (p->lmax + 128) / 128;
  // four where that still makes 200 blocks for the 152 SMs (map2alm, four a block and one or two: nside 32, B 9, 195
  // blocks, 34.9 and 31.3 us; nside 21, B 25, 301, 45.1 and 48.4; nside 8, B 50, 221, 30.7 and 34.8)
  const int64_t blocks4 = (int64_t)((p->batch + 3) / 4) * (p->mmax + 1) * ((p->lmax + A32_LB) / A32_LB);
  int nb = p->batch >= 8 && blocks4 >= 200 ? 4 : p->batch % 2 == 0 ? 2 : 1;
  while (ana32_smem(p, nb) > ANA32_SMEM) nb /= 2;
  auto go = [&](auto kern) {
    const size_t sm = ana32_smem(p, nb);
    if (cudaError_t e = dyn_smem_allow(kern, sm)) return e;
    kern<<<dim3((p->batch + nb - 1) / nb, (p->lmax + A32_LB) / A32_LB, p->mmax + 1), 32 * A32_WARPS, sm, st>>>(
        p->tab32, table_ld(p), p->tc_ks, npt, nlt, p->rc32, p->apart32, p->lmax, p->mmax, p->npairs, p->nalm,
        npt * 128, p->batch, state);
    return cudaGetLastError();
  };
  return nb == 1 ? go(k_ana32<1>) : nb == 2 ? go(k_ana32<2>) : go(k_ana32<4>);
}

}  // namespace dmwf
