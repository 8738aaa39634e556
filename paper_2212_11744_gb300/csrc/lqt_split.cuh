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
// times the column's.
//
// That bound is for the row and the column, where an FP64 product rounds every
// term to 2^-53 of itself.  In states of mixed units, x = D x' with D diagonal,
// rows and columns are graded oppositely and the bound is max D / min D larger
// than an FP64 product's.  So every product is measured (grade()): row i's and
// column i's largest magnitudes against the largest term of diagonal entry i,
//     grade = max_i (Ea_i + Eb_i - max_k (e(a_ik) + e(b_ki))).
// With d_i = sqrt(row maximum i / column maximum i) the error of entry (i, j) is
// below 2^(grade - 57) d_i / d_j times the square root of the diagonal entries'
// terms: a relative error of that size in the units d.  Dense elements of one
// scale have grades up to 5, mixed units of ratio R about log2 R.  Above
// kGradeLimit a product is formed in FP64; a combination whose C J is above
// kFoldLimit, where the error of its later products starts to pass an FP64
// elimination's (S of 64 elements folded at n = 16, split products over FP64:
// 0.97 at ratio 2^3, 1.6 at 2^5, 75 at 2^20), forms all of them in FP64.  In the
// units x' S is then as exact at ratio 2^34 as at 1 (3e-15; an elimination, whose
// pivots feel D, leaves 8e-13).
// Measuring costs some 5% (n = 16, T = 8192: 1.93 -> 2.05 ms; n = 64, T = 4096: 16.5
// -> 17.1; 256 problems: 37.4 -> 39.7).  The FP64 products of a graded problem:
// n = 16, T = 8192 at ratio 2^34 3.90 ms, n = 64, T = 512 23.9 ms (7.3 at ratio 1).
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

constexpr int kGradeLimit = 5;   // a product of a larger grade is formed in FP64
constexpr int kFoldLimit = 3;    // C J of a larger grade: all products of the combination in FP64
constexpr int kAllFp64 = -1;     // below every grade
constexpr int kNoLimit = 1 << 12;  // above every grade of normal operands
constexpr int kGradeOdd = 1 << 13; // operands that have no digits: see odd_vector()

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

// Whether a vector with largest biased exponent E has no digits: an infinity or
// NaN, or nonzero (bits: its entries' bits but the signs, or'ed) and so small
// that its entries or the products' last digits are subnormal.  Such a product
// is formed in FP64.
__device__ __forceinline__ bool odd_vector(int E, unsigned bits) { return E == 0x7ff || (E < 64 && bits != 0u); }
__device__ __forceinline__ unsigned magnitude_bits(double x) {
  return ((unsigned)__double2hiint(x) << 1) | (unsigned)__double2loint(x);
}

// Grade of diagonal entry i: the largest biased exponents of row i and column i
// and the largest sum of the exponents of a term (see the head of this file).
__device__ __forceinline__ int grade(int Ea, int Eb, int term) {
  if (Ea == 0 || Eb == 0) return 0;  // a zero vector
  return Ea + Eb < 1023 + 64 ? kGradeOdd : Ea + Eb - term;
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
// kTry: as kSet, but above the limit nothing is written and kGraded returned.
enum Store { kSet = 0, kSubtract = 1, kTry = 2 };
constexpr int kGraded = -1;

template <int NW>
__device__ __forceinline__ void sync16() {
  if constexpr (NW == 1)
    __syncwarp();
  else
    __syncthreads();
}

// Whether x holds in any thread of the warp or CTA; orders their earlier
// accesses to shared memory before the later ones.
template <int NW>
__device__ __forceinline__ bool any16(bool x) {
  if constexpr (NW == 1) {
    __syncwarp();
    return __any_sync(0xffffffffu, x);
  } else {
    return __syncthreads_or(x) != 0;
  }
}

// Entries k = c, c + 1, c + 8, c + 9 of vector v of m and the vector's largest
// exponent (c = 2 (lane % 4); the four lanes of a vector are neighbours).
__device__ __forceinline__ int load_vector(int lane, const double* sm, Mat16 m, int v, double (&x)[4],
                                           unsigned (&h)[4], bool& odd) {
  const double* s = sm + m.p + v * m.sv + 2 * (lane & 3) * m.sk;
  x[0] = s[0];
  x[1] = s[m.sk];
  x[2] = s[8 * m.sk];
  x[3] = s[9 * m.sk];
#pragma unroll
  for (int q = 0; q < 4; ++q) h[q] = (unsigned)__double2hiint(x[q]) & 0x7ff00000u;  // the exponent in place
  unsigned t = max(max(h[0], h[1]), max(h[2], h[3]));
  t = max(t, __shfl_xor_sync(0xffffffffu, t, 1));
  t = max(t, __shfl_xor_sync(0xffffffffu, t, 2));
  const int e = (int)(t >> 20);
  if (e < 64 || e == 0x7ff)
    odd = odd || odd_vector(e, magnitude_bits(x[0]) | magnitude_bits(x[1]) | magnitude_bits(x[2]) | magnitude_bits(x[3]));
  return e;
}

// out(i, j) = sum_k a(i, k) b(k, j) + diag (i == j) (kSet), or out -= the
// product (kSubtract); out at p + i sv + j sk.  out may be one of the operands
// (all reads of them come before the writes).  Above the limit the product is
// formed in FP64, its terms in ascending k.  Two warps (NW = 2, the whole CTA)
// take eight columns each.  Returns the largest biased exponent of the entries
// this warp set (a bound on them).  Not inlined: some 1000 instructions, of
// which a combination runs fourteen copies' worth; inlined, its code no longer
// fits the instruction caches and a warp waits on fetches.
template <int NW>
static __device__ __noinline__ int product16(Mat16 ma, Mat16 mb, Mat16 mo, int diag, int store,
                                             int limit = kGradeLimit) {
  extern __shared__ __align__(16) double split_smem[];
  constexpr int kTiles = 2 / NW;  // 8-column tiles of this warp
  const int lane = threadIdx.x & 31;
  const int g = lane >> 2, c = 2 * (lane & 3);
  const int t0 = NW == 1 ? 0 : (int)(threadIdx.x >> 5);
  unsigned a[C16::ND][4], b[kTiles][C16::ND][2];
  int ea[2], eb[kTiles];
  unsigned ha[2][4];
  int top = 0;
  bool graded = limit < 0;
  if (!graded) {
    bool odd = false;
    int worst = 0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      double x[4];
      ea[r] = load_vector(lane, split_smem, ma, g + 8 * r, x, ha[r], odd);
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
      unsigned hb[4];
      eb[t] = load_vector(lane, split_smem, mb, g + 8 * (t0 + t), x, hb, odd);
      // diagonal entry i = g + 8 (t0 + t): this lane holds the same k of both
      const int r = t0 + t;
      unsigned term = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) term = max(term, (r ? ha[1][q] : ha[0][q]) + hb[q]);
      term = max(term, __shfl_xor_sync(0xffffffffu, term, 1));
      term = max(term, __shfl_xor_sync(0xffffffffu, term, 2));
      worst = max(worst, grade(r ? ea[1] : ea[0], eb[t], (int)(term >> 20)));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const unsigned long long u = digits<C16>(x[2 * h], eb[t]), v = digits<C16>(x[2 * h + 1], eb[t]);
#pragma unroll
        for (int i = 0; i < C16::ND; ++i) b[t][i][h] = digit_pair<C16>(u, v, i);
      }
    }
    graded = any16<NW>(odd || worst > limit);  // a barrier, too
  }
  if (graded) {
    if (store == kTry) return kGraded;
    double s[kTiles][4];
#pragma unroll
    for (int t = 0; t < kTiles; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) s[t][q] = 0.0;
#pragma unroll 1
    for (int k = 0; k < 16; ++k)
#pragma unroll
      for (int t = 0; t < kTiles; ++t)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = g + 8 * (q >> 1), j = 8 * (t0 + t) + c + (q & 1);
          s[t][q] = fma(split_smem[ma.p + i * ma.sv + k * ma.sk], split_smem[mb.p + j * mb.sv + k * mb.sk], s[t][q]);
        }
    sync16<NW>();
#pragma unroll
    for (int t = 0; t < kTiles; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = g + 8 * (q >> 1), j = 8 * (t0 + t) + c + (q & 1);
        const double v = s[t][q] + (i == j ? (double)diag : 0.0);
        top = max(top, biased_exp(v));
        double* o = split_smem + mo.p + i * mo.sv + j * mo.sk;
        *o = store == kSubtract ? *o - v : v;
      }
    sync16<NW>();
    return __reduce_max_sync(0xffffffffu, top);
  }
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
