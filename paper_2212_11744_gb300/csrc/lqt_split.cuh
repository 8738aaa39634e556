// FP64 matrix products on the FP16 tensor core: every operand is written as a
// sum of small integers (digits), so that all products and sums inside the
// tensor core are exact, and the digits' partial sums are put together as a
// 64-bit integer.  The scheme is Ozaki, Ogita, Oishi and Rump's error-free
// splitting (Numerical Algorithms 59, 2012) with the splitting done on the
// integer pipe.
//
// Why: an FP64 warp instruction occupies a sub-partition of this GPU for 64
// cycles (1.25 TFLOP/s in all), mma.sync m16n8k16 with FP16 inputs for 2 and
// an integer instruction for 1, so a product of FP64 accuracy made of 21 to 28
// FP16 products and some 35 integer instructions per operand entry leaves the
// FP64 pipe free and takes a fraction of its time.
//
// A vector (a row of the left operand, a column of the right one) with largest
// biased exponent E is held as v = x 2^(kBias - E), an integer of S ND - 2
// bits and a sign (rounded half up), cut into ND digits of S bits, balanced
// (-2^(S-1) .. 2^(S-1) - 1; an FP16 number holds them exactly).  Digit i = 0
// is the most significant.  Products of digits i and j with i + j < ND are
// kept: sum w = i + j has weight 2^(S (2 (ND - 1) - w)).  A sum of K products
// stays below 2^24 in the FP32 accumulator, and so exact, for K 2^(2S - 2)
// (w + 1) <= 2^24: with S = 10, K = 16 up to w = 3; with S = 9, K = 64 up to
// w = 3; beyond that a sum can only reach 2^24 when the result itself is of
// full size, and its rounding lies below 2^-58 of it.  What is dropped (i + j
// >= ND) and the rounding of v are below 2^-57 of the row's largest entry
// times the column's: an FP64 product's own rounding is 2^-53 of each term.
#pragma once

#include <cstdint>

#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace lqt {
namespace split {

template <int S_, int ND_, int UNIT_>
struct Cfg {
  static constexpr int S = S_, ND = ND_;
  static constexpr int SH = S * ND - 54;     // left shift of the 53-bit significand
  static constexpr int kBias = 1074 + SH;    // x = v 2^(E - kBias)
  static constexpr int UNIT = UNIT_;         // log2 of the unit of the 64-bit result
};
using C16 = Cfg<10, 6, 60>;  // inner dimension up to 16
using C64 = Cfg<9, 7, 66>;   // inner dimension up to 64

__device__ __forceinline__ int biased_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// v's digits, biased to be non-negative, in bits 1 .. S ND of the result (bit
// 0 is the rounding bit).
template <class C>
__device__ __forceinline__ unsigned long long digits(double x, int E) {
  constexpr unsigned long long kOffset = [] {
    unsigned long long b = 1;
    for (int i = 0; i < C::ND; ++i) b += 1ull << (C::S * i + C::S);  // 2 * 2^(S-1) 2^(S i)
    return b;
  }();
  const unsigned xh = (unsigned)__double2hiint(x), xl = (unsigned)__double2loint(x);
  const int ex = (int)((xh >> 20) & 0x7ff);
  const unsigned mh = ex ? ((xh & 0xfffffu) | 0x100000u) : 0u;  // subnormals count as zero
  const unsigned ml = ex ? xl : 0u;
  int d = E - ex;
  d = d > 63 ? 63 : d;
  const unsigned long long w = ((((unsigned long long)mh << 32) | ml) << C::SH) >> d;
  const unsigned long long s = (unsigned long long)((long long)(int)xh >> 63);
  return (w ^ s) - s + kOffset;
}

// Digit i of two neighbouring entries as a pair of FP16 numbers.
template <class C>
__device__ __forceinline__ unsigned digit_pair(unsigned long long a, unsigned long long b, int i) {
  constexpr unsigned m = (1u << C::S) - 1u;
  const int p = 1 + C::S * (C::ND - 1 - i);
  const unsigned ua = (unsigned)(a >> p) & m, ub = (unsigned)(b >> p) & m;
  // 1024 + u is the FP16 number 0x6400 | u for u < 1024
  const unsigned h = ua | (ub << 16) | 0x64006400u;
  const __half2 off = __float2half2_rn((float)(1024 + (1 << (C::S - 1))));
  const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&h), off);
  return *reinterpret_cast<const unsigned*>(&r);
}

__device__ __forceinline__ void mma16816(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The digit sums of one output as an integer: the output is that integer times
// 2^(UNIT + Ea - kBias + Eb - kBias).
template <class C>
__device__ __forceinline__ long long to_int(const float (&acc)[C::ND][4], int q) {
  // sums whose weight lies below the unit are added in FP32 to the first one
  // there (rounded at the unit), the others are integers
  long long r = 0;
  float low = 0.0f;
#pragma unroll
  for (int w = C::ND - 1; w >= 0; --w) {
    const int a = C::S * (2 * (C::ND - 1) - w) - C::UNIT;
    if (a <= 0) {
      low = fmaf(acc[w][q], exp2f((float)a), low);
      if (a == 0 || C::S * (2 * (C::ND - 1) - (w - 1)) - C::UNIT > 0) r = (long long)__float2int_rn(low);
    } else {
      r += (long long)__float2int_rn(acc[w][q]) * (1ll << a);
    }
  }
  return r;
}

// r 2^e as a double (round to nearest, ties away; overflow to infinity,
// underflow to zero).
__device__ __forceinline__ double to_double(long long r, int e) {
  const long long s = r >> 63;
  unsigned long long a = (unsigned long long)((r ^ s) - s);
  const int lz = __clzll((long long)a);
  a <<= (lz & 63);
  const int be = 1023 + 63 - lz + e;  // biased exponent of the leading bit
  unsigned long long v = ((unsigned long long)(unsigned)(be - 1) << 52) + (a >> 11) + ((a >> 10) & 1ull);
  if (be < 1 || r == 0) v = 0;
  if (be > 2046) v = 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(v | ((unsigned long long)s & 0x8000000000000000ull)));
}

// r 2^(UNIT + ea + eb - 2 kBias) + diag as a double, diag = 0, 1 or -1 added
// before the one rounding; where 1.0 is too large for the 64-bit integer the
// product is below 2^-1 of its last bits and an FP64 addition does.
template <class C>
__device__ __forceinline__ double finish(long long r, int ea, int eb, int diag) {
  const int p = 2 * C::kBias - C::UNIT - ea - eb;  // 1.0 = 2^p units
  if (diag != 0 && p < 62) r += p >= 0 ? (long long)diag * (1ll << p) : 0ll;
  double v = to_double(r, -p);
  if (diag != 0 && p >= 62) v += (double)diag;
  if (ea == 0x7ff || eb == 0x7ff) v = __longlong_as_double(0x7ff8000000000000ll);
  return v;
}

// ---------------------------------------------------------------------------
// 16 x 16 x 16, one warp or a CTA of two, operands in shared memory
// ---------------------------------------------------------------------------

// A 16 x 16 operand: entry k of vector v (a row of the left operand, a column
// of the right one) at p[v sv + k sk], p an offset (doubles) from the CTA's
// dynamic shared memory.
struct Mat16 {
  int p, sv, sk;
};
enum Store16 { kSet = 0, kSubtract = 1 };

template <int NW>
__device__ __forceinline__ void sync16() {
  if constexpr (NW == 1)
    __syncwarp();
  else
    __syncthreads();
}

// Entries k = c, c + 1, c + 8, c + 9 of vector v of m and the vector's largest
// exponent (c = 2 (lane % 4); the four lanes of a vector are neighbours).
__device__ __forceinline__ int load_vector(int lane, const double* sm, Mat16 m, int v, double (&x)[4]) {
  const double* s = sm + m.p + v * m.sv + 2 * (lane & 3) * m.sk;
  x[0] = s[0];
  x[1] = s[m.sk];
  x[2] = s[8 * m.sk];
  x[3] = s[9 * m.sk];
  int e = max(max(biased_exp(x[0]), biased_exp(x[1])), max(biased_exp(x[2]), biased_exp(x[3])));
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
  return max(e, __shfl_xor_sync(0xffffffffu, e, 2));
}

// out(i, j) = sum_k a(i, k) b(k, j) + diag (i == j) (kSet), or out -= the
// product (kSubtract); out at p + i sv + j sk.  out may be one of the operands
// (they are in registers before it is written).  A row or column with an
// infinity or NaN gives NaN.  Two warps (NW = 2, the whole CTA) take eight
// columns each.  Returns the largest biased exponent of the entries this warp
// set (a bound on them).  Not inlined: some 1000 instructions, of which a
// combination runs fourteen copies' worth; inlined, its code no longer fits
// the instruction caches and a warp waits on fetches.
template <int NW>
static __device__ __noinline__ int product16(Mat16 ma, Mat16 mb, Mat16 mo, int diag, int store) {
  extern __shared__ __align__(16) double split_smem[];
  constexpr int kTiles = 2 / NW;  // 8-column tiles of this warp
  const int lane = threadIdx.x & 31;
  const int g = lane >> 2, c = 2 * (lane & 3);
  const int t0 = NW == 1 ? 0 : (int)(threadIdx.x >> 5);
  unsigned a[C16::ND][4], b[kTiles][C16::ND][2];
  int ea[2], eb[kTiles];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    double x[4];
    ea[r] = load_vector(lane, split_smem, ma, g + 8 * r, x);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned long long u = digits<C16>(x[2 * h], ea[r]), v = digits<C16>(x[2 * h + 1], ea[r]);
#pragma unroll
      for (int i = 0; i < C16::ND; ++i) a[i][r + 2 * h] = digit_pair<C16>(u, v, i);
    }
  }
#pragma unroll
  for (int t = 0; t < kTiles; ++t) {
    double x[4];
    eb[t] = load_vector(lane, split_smem, mb, g + 8 * (t0 + t), x);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned long long u = digits<C16>(x[2 * h], eb[t]), v = digits<C16>(x[2 * h + 1], eb[t]);
#pragma unroll
      for (int i = 0; i < C16::ND; ++i) b[t][i][h] = digit_pair<C16>(u, v, i);
    }
  }
  sync16<NW>();
  int top = 0;
#pragma unroll
  for (int t = 0; t < kTiles; ++t) {
    float acc[C16::ND][4];
#pragma unroll
    for (int w = 0; w < C16::ND; ++w)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[w][q] = 0.0f;
    // one digit of the rows at a time, so that neighbouring instructions add
    // to different sums
#pragma unroll
    for (int i = 0; i < C16::ND; ++i)
#pragma unroll
      for (int j = 0; j < C16::ND - i; ++j) mma16816(acc[i + j], a[i], b[t][j][0], b[t][j][1]);
    // exponents of columns c and c + 1 of the tile: lanes 4 c .. and 4 (c + 1) ..
    const int e0 = __shfl_sync(0xffffffffu, eb[t], 4 * c), e1 = __shfl_sync(0xffffffffu, eb[t], 4 * c + 4);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = g + 8 * (q >> 1), j = 8 * (t0 + t) + c + (q & 1);
      const double v = finish<C16>(to_int<C16>(acc, q), ea[q >> 1], (q & 1) ? e1 : e0, i == j ? diag : 0);
      top = max(top, biased_exp(v));
      double* o = split_smem + mo.p + i * mo.sv + j * mo.sk;
      *o = store == kSubtract ? *o - v : v;
    }
  }
  sync16<NW>();
  return __reduce_max_sync(0xffffffffu, top);
}

}  // namespace split
}  // namespace lqt
