// dm_split.cuh -- digits, exact sums and operand access of the split products
// (dm_split.cu: the Legendre stages; dm_dft.cu: the ring transforms).  A value
// is a fixed-point number of S digits in base 512 relative to a power-of-two
// scale; the method is described in dm_split.cu.
#pragma once

#include <cuda.h>

#include "dm_internal.h"
#include "dm_tc.cuh"

namespace dmwf {

using namespace tc;

constexpr int SPLIT_S = 6;             // digits of the table
constexpr int SPLIT_NAN = 1 << 20;     // column exponent of a column with a non-finite value

namespace {

// floor(log2 |x|) + 1 of a finite non-zero double from its bits; very small for 0 and denormals
__device__ __forceinline__ int exp_of(double x) {
  const int f = (__double2hiint(x) >> 20) & 0x7ff;
  return f == 0 ? -100000 : (f == 0x7ff ? SPLIT_NAN : f - 1022);
}

// x 2^(53 - e) rounded to the nearest integer, |x| <= 2^e: integer operations only
__device__ __forceinline__ long long fixed53(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int f = (int)((b >> 52) & 0x7ff);
  if (f == 0) return 0;
  const int sh = e - (f - 1022);  // >= 0
  long long v = (b & 0xfffffffffffffll) | 0x10000000000000ll;
  if (sh > 54) return 0;
  if (sh > 0) v = (v + (1ll << (sh - 1))) >> sh;
  return b < 0 ? -v : v;
}

// the FP32 forms: exponent, and x 2^(26 - e) rounded (27 bits: three digits)
__device__ __forceinline__ int exp_of(float x) {
  const int f = (__float_as_int(x) >> 23) & 0xff;
  return f == 0 ? -100000 : (f == 0xff ? SPLIT_NAN : f - 126);
}
__device__ __forceinline__ int fixed26(float x, int e) {
  const int b = __float_as_int(x), f = (b >> 23) & 0xff;
  if (f == 0) return 0;
  const int sh = e - (f - 126);  // >= 0
  int v = ((b & 0x7fffff) | 0x800000) << 2;
  if (sh > 27) return 0;
  if (sh > 0) v = (v + (1 << (sh - 1))) >> sh;
  return b < 0 ? -v : v;
}
__device__ __forceinline__ int fixed26(double x, int e) {
  const long long v = fixed53(x, e);
  return (int)((v + (1ll << 26)) >> 27);
}

// digit of the lowest weight, [-256, 255], taken off v
__device__ __forceinline__ int take_digit(int &v) {
  const int d = (int)(((unsigned)v + 256u) & 511u) - 256;
  v = (v - d) >> 9;
  return d;
}

// Fixed-point numbers of S digits and their digits (index 0: the highest weight)
template <int S>
struct Fixed;
template <>
struct Fixed<6> {
  using type = long long;
  static __device__ __forceinline__ type of(double x, int e) { return fixed53(x, e); }
  // two halves of three digits in 32 bits each
  static __device__ __forceinline__ void digits(type v, int d[6]) {
    int lo = (int)(((unsigned)(int)v + (1u << 26)) & ((1u << 27) - 1)) - (1 << 26);
    int hi = (int)((v - lo) >> 27);
    d[5] = take_digit(lo);
    d[4] = take_digit(lo);
    d[3] = lo;
    d[2] = take_digit(hi);
    d[1] = take_digit(hi);
    d[0] = hi;
  }
};
template <>
struct Fixed<3> {
  using type = int;
  template <typename R>
  static __device__ __forceinline__ type of(R x, int e) {
    return fixed26(x, e);
  }
  static __device__ __forceinline__ void digits(type v, int d[3]) {
    d[2] = take_digit(v);
    d[1] = take_digit(v);
    d[0] = v;
  }
};

// two small integers as a BF16 pair (exact for |d| <= 256)
__device__ __forceinline__ uint32_t bf16_pair(int d0, int d1) {
  const float f0 = __uint_as_float(0x4B400000u + (unsigned)d0) - 12582912.0f;
  const float f1 = __uint_as_float(0x4B400000u + (unsigned)d1) - 12582912.0f;
  return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
}
__device__ __forceinline__ uint16_t bf16_one(int d) {
  const float f = __uint_as_float(0x4B400000u + (unsigned)d) - 12582912.0f;
  return (uint16_t)(__float_as_uint(f) >> 16);
}

// NV (4 or 8) consecutive K values of one column, the first at K index part
// NV of the octet ko of the step, as digit rows: row j n0 + row holds digit j.
// alt: the same with the odd K values negated goes to row_alt.
template <int S, int NV>
__device__ __forceinline__ void put_digits(unsigned char *step, int n0, int row, int ko, int part,
                                           const typename Fixed<S>::type v[NV], bool alt, int row_alt) {
  int d[NV][S];
#pragma unroll
  for (int i = 0; i < NV; ++i) Fixed<S>::digits(v[i], d[i]);
#pragma unroll
  for (int j = 0; j < S; ++j) {
    uint32_t w[NV / 2];
#pragma unroll
    for (int i = 0; i < NV / 2; ++i) w[i] = bf16_pair(d[2 * i][j], d[2 * i + 1][j]);
    const int n = j * n0 + row;
    unsigned char *o = step + (n >> 3) * 256 + ko * 128 + (n & 7) * 16 + part * (2 * NV);
    if (NV == 8)
      *reinterpret_cast<uint4 *>(o) = make_uint4(w[0], w[1], w[NV / 2 - 2], w[NV / 2 - 1]);
    else
      *reinterpret_cast<uint2 *>(o) = make_uint2(w[0], w[1]);
    if (alt) {
      const int n2 = j * n0 + row_alt;
      unsigned char *o2 = step + (n2 >> 3) * 256 + ko * 128 + (n2 & 7) * 16 + part * (2 * NV);
#pragma unroll
      for (int i = 0; i < NV / 2; ++i) w[i] ^= 0x80000000u;
      if (NV == 8)
        *reinterpret_cast<uint4 *>(o2) = make_uint4(w[0], w[1], w[NV / 2 - 2], w[NV / 2 - 1]);
      else
        *reinterpret_cast<uint2 *>(o2) = make_uint2(w[0], w[1]);
    }
  }
}

__device__ __forceinline__ int block_max(int v, int *red) {
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  int r = red[0];
  for (int i = 1; i < (int)(blockDim.x >> 5); ++i) r = max(r, red[i]);
  __syncthreads();
  return r;
}

// (hi 2^36 + lo) 2^(e - 70) rounded to FP64, integer operations only; the sum of two such numbers
// divides by two through e.  Results below the normal range are zero.
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, int e) {
  __int128 t = ((__int128)hi << 36) + lo;
  const bool neg = t < 0;
  const unsigned __int128 u = neg ? (unsigned __int128)(-t) : (unsigned __int128)t;
  const unsigned long long uh = (unsigned long long)(u >> 64), ul = (unsigned long long)u;
  if ((uh | ul) == 0) return 0.0;
  const int n = uh ? 127 - __clzll((long long)uh) : 63 - __clzll((long long)ul);  // top bit
  unsigned long long mant;  // 53 bits, possibly 2^53 after rounding
  if (n > 52) {
    const unsigned long long q = (unsigned long long)(u >> (n - 53));
    mant = (q + 1) >> 1;
  } else {
    mant = ul << (52 - n);
  }
  const int ex = n + e - 70 + 1023;
  if (ex <= 0) return 0.0;
  if (ex >= 0x7ff) return __longlong_as_double((neg ? 0xfff0000000000000ull : 0x7ff0000000000000ull));
  unsigned long long bits = ((unsigned long long)ex << 52) + (mant - (1ull << 52));
  if (neg) bits |= 1ull << 63;
  return __longlong_as_double((long long)bits);
}

// digit weights kept: those of i + j < G
template <int S>
struct Weights {
  static constexpr int G = S == 6 ? 7 : S;
};

// sums of one output in units of the digit weights: hi for weights 0 .. 2, lo for 3 .. 6
template <int S>
struct Acc;
template <>
struct Acc<6> {
  long long hi = 0, lo = 0;
  __device__ __forceinline__ void add(const int *g) {
    hi += (long long)g[0] * (1 << 18) + (long long)g[1] * (1 << 9) + g[2];
    lo += (long long)g[3] * (1 << 27) + (long long)g[4] * (1 << 18) + (long long)g[5] * (1 << 9) + g[6];
  }
};
template <>
struct Acc<3> {
  long long hi = 0;
  __device__ __forceinline__ void add(const int *g) {
    hi += (long long)g[0] * (1 << 18) + (long long)g[1] * (1 << 9) + g[2];
  }
};

// a + s b (s = +-1), scaled by 2^e relative to the digit weights
__device__ __forceinline__ double value_of(const Acc<6> &a, const Acc<6> &b, int s, int e) {
  return fixed_to_double(s > 0 ? a.hi + b.hi : a.hi - b.hi, s > 0 ? a.lo + b.lo : a.lo - b.lo, e);
}
__device__ __forceinline__ double value_of(const Acc<6> &a, int e) { return fixed_to_double(a.hi, a.lo, e); }
__device__ __forceinline__ float scale_float(long long v, int e) {  // v 2^(e - 34)
  e -= 34;
  const int e1 = max(-126, min(127, e / 2)), e2 = max(-126, min(127, e - e1));
  return (float)v * __uint_as_float((unsigned)(e1 + 127) << 23) * __uint_as_float((unsigned)(e2 + 127) << 23);
}
__device__ __forceinline__ float value_of(const Acc<3> &a, const Acc<3> &b, int s, int e) {
  return scale_float(s > 0 ? a.hi + b.hi : a.hi - b.hi, e);
}
__device__ __forceinline__ float value_of(const Acc<3> &a, int e) { return scale_float(a.hi, e); }

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t r[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tma_box_at(uint32_t dst, const CUtensorMap *map, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(dst),
      "l"(map), "r"(0), "r"(y), "r"(z), "r"(0), "r"(bar)
      : "memory");
}

// matrix descriptor, no swizzle: byte offsets between core matrices (lead, stride)
__device__ __forceinline__ uint64_t split_desc(uint32_t saddr, uint32_t lead, uint32_t stride) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | (uint64_t)((lead >> 4) & 0x3FFF) << 16 |
         (uint64_t)((stride >> 4) & 0x3FFF) << 32 | (uint64_t)1 << 46;
}

// The MMAs of one K step: digit i of A (AD bytes apart from ad on) with the
// digits of B (rows from bd on) that it meets, added to the accumulators
// d + i N0; FIRST: the first step of a chunk, whose first MMA clears all G
// weights (its extra rows are zero).  N is rounded up to 16: the extra rows are
// another digit's or zero, the extra columns unused.  One thread issues all of
// a CTA's MMAs, so that everything here is known when compiled but the
// addresses: descriptors rebuilt and divisions by the stage count made it the
// bound of the kernel (870 cycles a K step of three MMAs).
template <int S, int N0, int AD, bool A_MN, bool FIRST, int I = 0>
__device__ __forceinline__ void split_step(uint32_t d, uint64_t ad, uint64_t bd) {
  if constexpr (I < S) {
    constexpr int G = Weights<S>::G, nd = (FIRST && I == 0) ? G : (S < G - I ? S : G - I);
    constexpr int N = (nd * N0 + 15) / 16 * 16;
    constexpr uint32_t idesc = idesc_bf16(128, N) | (A_MN ? 1u << 15 : 0u);  // bit 15: A is MN-major
    mma_bf16_c<!(FIRST && I == 0)>(d + I * N0, ad + I * (AD >> 4), bd, idesc);
    split_step<S, N0, AD, A_MN, FIRST, I + 1>(d, ad, bd);
  }
}

// Position in the ring of stages
struct StageAt {
  int s = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void next(int ns) {
    if (++s == ns) {
      s = 0;
      phase ^= 1;
    }
  }
};

template <int S>
struct OutT {
  using real = double;
  using cplx = double2;
};
template <>
struct OutT<3> {
  using real = float;
  using cplx = float2;
};

template <int S>
__device__ __forceinline__ typename OutT<S>::cplx mk(typename OutT<S>::real x, typename OutT<S>::real y) {
  typename OutT<S>::cplx c;
  c.x = x;
  c.y = y;
  return c;
}

// ---------------------------------------------------------------- host side

using EncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                              const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeFn encode_fn() {
  static EncodeFn fn = [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return (EncodeFn)f;
  }();
  return fn;
}

}  // namespace

}  // namespace dmwf
