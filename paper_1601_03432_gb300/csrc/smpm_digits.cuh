// Exact fixed-point products on the tensor cores ("digits"): y = A x for small
// dense A, accurate relative to A's rows and the whole vector x, where the FP64 pipe of this part (2 FMA
// per clock and SM) or the FP32 pipe's shared-memory loads are the bound.
//
// A number is held as a signed integer X = v 2^(B-e) (|X| <= 2^B; B = 62 for
// FP64, 30 for FP32, 94 for single products, see tile8_wide) relative to an exponent e shared by a row of A or a
// column of x, and cut into base-256 digits in [-128, 127] (ND = 8, 4 or 12): with
// the bias 0x80..80 added, the digits are the bytes of X, less 128.  Digits
// are exact in fp16, their products are integers of at most 2^14, and up to
// 8 x 128 of them add exactly in the FP32 accumulators of mma.sync (at most
// 2^24; tests/test_gpu_accumulators.py).  Products of digits i and j weigh 256^(i+j);
// those of one weight share an accumulator, and the weights below 256^GMIN
// are left out.  The sums are put together in integers and rounded once.
//
// Error, for K columns, as a share of row maximum times column maximum (each at
// least half of its power of two): the operands lose up to K 2^-60 (K 2^-28 in FP32),
// the left-out weights up to 7 K 2^14 256^6 2^-122 = K 2^-57 (2 K 2^14 256 2^-58 = K 2^-35) if
// all their digits are extreme and of one sign, about 2^-8 of that for digits of
// mixed signs.  This is a bound relative to the largest entries, as a GMRES solve with
// its normwise tolerance needs it; a chain of K FP64 FMAs loses up to K 2^-53 of the
// sum of magnitudes of the entry itself, which is less where that sum is below
// 2^-4 of the two maxima (solves on local and widely ranging right-hand sides end
// with the same errors either way).  The products that are results by themselves,
// y = S v, take operands of 94 bits (tile8_wide).
//
// mma.sync m16n8k16 rather than tcgen05 in the solves: the operands are one
// element's 4n x 4n matrix and eight columns (or the eight digits of one
// column), far below a tcgen05 tile, and each warp works on its own element.
// The class apply of y = S v on a large grid is a contraction that would fill
// tcgen05 tiles; that form has not been built.
//
// Fragments of A (host: pack_digits): tile (mt, kt) of 16 x 16 entries, lane
// (g = lane / 4, q = lane % 4) holds rows g, g + 8 and columns 2q, 2q+1, 2q+8,
// 2q+9; 8 bytes per digit (the biased digits in the order of the mma
// registers), two digits per 16-byte word: [mt][kt][digit / 2][lane].
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

namespace {

template <typename S>
struct Digits;
template <>
struct Digits<double> {
  static constexpr int ND = 8, GMIN = 7, NG = 8, B = 62;
};
template <>
struct Digits<float> {
  static constexpr int ND = 4, GMIN = 2, NG = 5, B = 30;
};

struct Wide {};  // FP64 operands of 94 bits: the class apply (tile8_wide)
template <>
struct Digits<Wide> {
  static constexpr int ND = 12, GMIN = 11, NG = 12, B = 94;
};

constexpr short kBadRow = 32767;  // row exponent of a matrix row with an Inf or NaN

__host__ __device__ constexpr int digit_tiles(int m) { return (m + 15) / 16; }
// uint4 words of one packed rows x cols matrix
template <typename S>
__host__ __device__ constexpr size_t digit_words(int rows, int cols) {
  return (size_t)digit_tiles(rows) * digit_tiles(cols) * (Digits<S>::ND / 2) * 32;
}
// uint4 words of the packed eight columns of a vector of `len` entries
template <typename S>
__host__ __device__ constexpr int digit_bwords(int len) {
  return digit_tiles(len) * (Digits<S>::ND / 2) * 32;
}

__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// two biased digits (bytes in halves 0x64dd: the fp16 number 1024 + byte) less 1152
__device__ __forceinline__ uint32_t digit_half2(uint32_t w) {
  const uint32_t bias = 0x64806480u;
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), *reinterpret_cast<const __half2*>(&bias));
  return *reinterpret_cast<const uint32_t*>(&h);
}
// A registers of one digit from its 8 bytes
__device__ __forceinline__ void digit_a(uint32_t w0, uint32_t w1, uint32_t (&a)[4]) {
  a[0] = digit_half2(__byte_perm(w0, 0x64646464u, 0x4140));
  a[1] = digit_half2(__byte_perm(w0, 0x64646464u, 0x4342));
  a[2] = digit_half2(__byte_perm(w1, 0x64646464u, 0x4140));
  a[3] = digit_half2(__byte_perm(w1, 0x64646464u, 0x4342));
}

// biased exponent field of v (0 for zero and subnormals, the largest value for Inf and NaN)
__device__ __forceinline__ int exp_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ int exp_field(float v) { return (__float_as_int(v) >> 23) & 0xff; }

// biased fixed-point digits of v relative to a column whose largest exponent field is E (>= 1)
__device__ __forceinline__ uint64_t to_digits(double v, int E) {
  const long long bits = __double_as_longlong(v);
  const int ev = (int)((bits >> 52) & 0x7ff);
  long long m = bits & 0xfffffffffffffLL;
  if (ev) m |= 1LL << 52;
  const int sh = 9 - (E - (ev ? ev : 1));  // m < 2^53 -> below 2^62
  long long x;
  if (sh >= 0) x = m << sh;
  else x = -sh < 60 ? (m + (1LL << (-sh - 1))) >> -sh : 0;
  x = bits < 0 ? -x : x;
  return (uint64_t)x + 0x8080808080808080ull;
}
__device__ __forceinline__ uint32_t to_digits(float v, int E) {
  const int bits = __float_as_int(v);
  const int ev = (bits >> 23) & 0xff;
  int m = bits & 0x7fffff;
  if (ev) m |= 1 << 23;
  const int sh = 6 - (E - (ev ? ev : 1));  // m < 2^24 -> below 2^30
  int x;
  if (sh >= 0) x = m << sh;
  else x = -sh < 28 ? (m + (1 << (-sh - 1))) >> -sh : 0;
  x = bits < 0 ? -x : x;
  return (uint32_t)x + 0x80808080u;
}

// the same to 94 bits, as three words
struct Bits96 {
  uint32_t w[3];
};
__device__ __forceinline__ Bits96 to_digits96(double v, int E) {
  const long long bits = __double_as_longlong(v);
  const int ev = (int)((bits >> 52) & 0x7ff);
  unsigned long long m = bits & 0xfffffffffffffLL;
  if (ev) m |= 1ULL << 52;
  const int sh = 41 - (E - (ev ? ev : 1));  // m < 2^53 -> below 2^94
  unsigned long long lo;
  uint32_t hi = 0;
  if (sh >= 0) {
    lo = m << sh;
    if (sh > 0) hi = (uint32_t)(m >> (64 - sh));
  } else {
    lo = -sh < 60 ? (m + (1ULL << (-sh - 1))) >> -sh : 0;
  }
  if (bits < 0) {
    lo = 0 - lo;
    hi = ~hi + (lo == 0);
  }
  const unsigned long long b = lo + 0x8080808080808080ull;
  hi += 0x80808080u + (b < lo);
  return {{(uint32_t)b, (uint32_t)(b >> 32), hi}};
}

// byte j of a and b as the two low halves' digits
template <typename U>
__device__ __forceinline__ uint32_t digit_pair(U a, U b, int j) {
  uint32_t wa, wb;
  if constexpr (sizeof(U) == 8) {
    wa = j < 4 ? (uint32_t)a : (uint32_t)(a >> 32);
    wb = j < 4 ? (uint32_t)b : (uint32_t)(b >> 32);
  } else {
    wa = a;
    wb = b;
  }
  const uint32_t p = __byte_perm(wa, wb, (uint32_t)((j & 3) | ((4 + (j & 3)) << 8)));  // bytes 0 and 2
  return digit_half2((p & 0x00ff00ffu) | 0x64006400u);
}

// value 2^s of the integer hi 2^32 + lo (|hi| < 2^62, |lo| < 2^62), rounded to
// nearest; s such that the result is a normal number unless it is zero
__device__ __forceinline__ double digits_value(long long hi, long long lo, int s) {
  hi += lo >> 32;
  uint32_t l = (uint32_t)lo;  // value = hi 2^32 + l
  const bool neg = hi < 0;
  if (neg) {
    hi = ~hi;
    l = ~l;  // magnitude - 1; the missing unit is far below the rounding unless hi is 0
    if (++l == 0) ++hi;
  }
  unsigned long long h = (unsigned long long)hi;
  int e = 32;
  if (h == 0) {
    if (l == 0) return 0.0;
    h = (unsigned long long)l << 32;
    l = 0;
    e = -32;
  }
  const int z = __clzll((long long)h);
  if (z) h = (h << z) | (z < 32 ? (unsigned long long)(l >> (32 - z)) : ((unsigned long long)l << (z - 32)));
  e -= z;
  unsigned long long m = (h >> 11) + ((h >> 10) & 1);  // 53 bits, nearest
  // value = m 2^(e + 11): the exponent field of m (implicit bit included) is added below
  const long long bits = (long long)m + ((long long)(e + 11 + s + 1023 + 52 - 1) << 52);
  return __longlong_as_double(neg ? (bits | (1LL << 63)) : bits);
}

// v 2^s for any s (two exact factors where the scale itself is out of range)
__device__ __forceinline__ double scale2(double v, int s) {
  if (s < -1000 || s > 1000) {
    const int h = s / 2;
    return v * __longlong_as_double((long long)(1023 + max(-1022, min(1023, h))) << 52) *
           __longlong_as_double((long long)(1023 + max(-1022, min(1023, s - h))) << 52);
  }
  return v * __longlong_as_double((long long)(1023 + s) << 52);
}

// Result from the summed weights hi 2^32 + lo (units of 256^GMIN); er: exponent
// of A's row, E: the column's largest exponent field.  Inf or NaN in the column
// gives NaN, as does a row marked kBadRow.
__device__ __noinline__ double digits_far(long long hi, long long lo, int er, int E) {  // exponents out of the usual range
  if (E == 0x7ff || er == kBadRow) return __longlong_as_double(0x7ff8000000000000LL);
  return scale2(digits_value(hi, lo, 0), er + E - 1022 + 56 - 124);
}
__device__ __forceinline__ double digits_result(long long hi, long long lo, int er, int E, double) {
  if (E >= 600 && E <= 1400 && er != kBadRow)
    return digits_value(hi, lo, er + E - 1022 + 56 - 124);  // 256^7 2^(er - 62) 2^(E - 1022 - 62)
  return digits_far(hi, lo, er, E);
}
__device__ __noinline__ float digits_far32(long long hi, long long lo, int er, int E) {
  return (float)digits_value(hi, lo, er + E - 126 + 16 - 60);
}
__device__ __forceinline__ float digits_result(long long hi, long long lo, int er, int E, float) {
  if (E == 0xff || er == kBadRow) return __int_as_float(0x7fc00000);
  return (float)digits_value(hi, lo, er + E - 126 + 16 - 60);  // 256^2 2^(er - 30) 2^(E - 126 - 30), FP64 exponents
}

// The same in a few FP64 operations (the halves are below 2^53: one rounding),
// for the one-column products, where few instructions count more than FP64
// throughput.
__device__ __forceinline__ double pow2(int s) { return __longlong_as_double((long long)(1023 + s) << 52); }
__device__ __forceinline__ double digits_short(long long hi, long long lo, int er, int E, double) {
  const int s = er + E - 1022 + 56 - 124;
  if (E >= 600 && E <= 1400 && er != kBadRow) return fma((double)hi, pow2(s + 32), (double)lo * pow2(s));
  return digits_far(hi, lo, er, E);
}
__device__ __forceinline__ float digits_short(long long hi, long long lo, int er, int E, float) {
  // hi 2^32 + lo < 2^57: rounded once from the integer, then scaled exactly
  if (E == 0xff || er == kBadRow) return __int_as_float(0x7fc00000);
  const int s = er + E - 126 + 16 - 60;
  const float t = __ll2float_rn((hi << 32) + lo);
  return s > -120 && s < 60 ? t * __int_as_float((127 + s) << 23) : digits_far32(hi, lo, er, E);
}

// ---- eight columns -----------------------------------------------------------
// k tile kt of eight packed columns: the lane's entries of column lane / 4
template <typename S>
__device__ __forceinline__ void pack_tile(uint4* Bf, int kt, int lane, const S (&v)[4], int E) {
  constexpr int ND = Digits<S>::ND;
  decltype(to_digits(S(0), 1)) Y[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) Y[u] = to_digits(v[u], E);
#pragma unroll
  for (int j = 0; j < ND; j += 2)
    Bf[(kt * (ND / 2) + j / 2) * 32 + lane] = make_uint4(digit_pair(Y[0], Y[1], j), digit_pair(Y[2], Y[3], j),
                                                         digit_pair(Y[0], Y[1], j + 1), digit_pair(Y[2], Y[3], j + 1));
}

// The routines below are calls, one copy each: the solve kernels run them from
// a dozen places, each once per phase and a few warps at a time, and inlined
// there the instruction fetches took longer than the products (a 64 x 64
// block solve 25 k cycles instead of 12 k).
//
// Packs eight columns, entry (k, c) at x[k ldk + c ldc] (shared memory, or
// global memory that no other CTA writes; columns >= nc are zero), k < len,
// into Bf (digit_bwords words) and returns the largest exponent field (>= 1) of
// column g = lane / 4.  One warp (it packs the k tiles part, part + parts, ...:
// several warps share the work, each finding the exponents itself).
template <typename S>
__device__ __noinline__ int pack_cols(uint4* Bf, const S* x, int ldk, int ldc, int len, int nc, int lane, int part,
                                      int parts) {
  const int g = lane >> 2, q = lane & 3, kt_n = digit_tiles(len);
  const S* xc = x + (size_t)min(g, nc - 1) * ldc;
  const int klen = g < nc ? len : 0;
  int E = 1;
  for (int kt = 0; kt < kt_n; ++kt)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = kt * 16 + 2 * q + (u & 1) + 8 * (u >> 1);
      if (k < klen) E = max(E, exp_field(xc[k * ldk]));
    }
  E = max(E, __shfl_xor_sync(0xffffffffu, E, 1));
  E = max(E, __shfl_xor_sync(0xffffffffu, E, 2));
  for (int kt = part; kt < kt_n; kt += parts) {
    S v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = kt * 16 + 2 * q + (u & 1) + 8 * (u >> 1);
      v[u] = k < klen ? xc[k * ldk] : S(0);
    }
    pack_tile<S>(Bf, kt, lane, v, E);
  }
  __syncwarp();
  return E;
}

// A's fragments of k tile kt of a row tile, ND / 2 words per lane (shared or
// global memory)
template <typename S>
__device__ __forceinline__ void ld_frag(uint4 (&f)[Digits<S>::ND / 2], const uint4* __restrict__ A, int kt) {
#pragma unroll
  for (int p = 0; p < Digits<S>::ND / 2; ++p) f[p] = A[(kt * (Digits<S>::ND / 2) + p) * 32];
}

// The values a lane (g, q) holds of a row tile times eight columns: z[v] is row
// 16 mt + g + 8 (v >> 1), column 2q + (v & 1).
template <typename S>
struct Tile8 {
  S z[4];
};

// Row tile mt of A times the packed columns (row indices beyond rows give
// arbitrary values).  Af: A's fragments (two k tiles ahead), er: its row
// exponents, E: the exponent field of column lane / 4 (from pack_cols).
template <typename S>
__device__ __forceinline__ Tile8<S> tile8_products(const uint4* Af, const short* __restrict__ er,
                                                   const uint4* Bf, int rows, int kt_n, int mt, int lane, int E) {
  constexpr int ND = Digits<S>::ND, GMIN = Digits<S>::GMIN, NG = Digits<S>::NG;
  const int g = lane >> 2, q = lane & 3, row0 = mt * 16 + g;
  const uint4* A = Af + (size_t)mt * kt_n * (ND / 2) * 32 + lane;
  uint4 a0[ND / 2], a1[ND / 2];
  ld_frag<S>(a0, A, 0);
  if (kt_n > 1) ld_frag<S>(a1, A, 1);
  const int er0 = row0 < rows ? __ldg(er + row0) : 0, er1 = row0 + 8 < rows ? __ldg(er + row0 + 8) : 0;
  float acc[NG][4];
#pragma unroll
  for (int c = 0; c < NG; ++c)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[c][v] = 0.f;
  for (int kt = 0; kt < kt_n; ++kt) {
    uint4 av[ND / 2], bv[ND / 2];
#pragma unroll
    for (int p = 0; p < ND / 2; ++p) {
      av[p] = a0[p];
      a0[p] = a1[p];
      bv[p] = Bf[(kt * (ND / 2) + p) * 32 + lane];
    }
    if (kt + 2 < kt_n) ld_frag<S>(a1, A, kt + 2);
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      uint32_t a[4];
      const uint4 w = av[i / 2];
      digit_a((i & 1) ? w.z : w.x, (i & 1) ? w.w : w.y, a);
#pragma unroll
      for (int j = 0; j < ND; ++j) {
        if (i + j < GMIN) continue;
        const uint4 b = bv[j / 2];
        mma_16816(acc[i + j - GMIN], a, (j & 1) ? b.z : b.x, (j & 1) ? b.w : b.y);
      }
    }
  }
  Tile8<S> o;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const int Ec = __shfl_sync(0xffffffffu, E, 4 * (2 * q + (v & 1)));  // column 2q + (v & 1): lanes 8q, 8q + 4
    long long lo = 0, hi = 0;
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const long long t = (long long)__float2int_rn(acc[k][v]) << (8 * (k & 3));
      if (k < 4) lo += t;
      else hi += t;
    }
    o.z[v] = digits_result(hi, lo, v < 2 ? er0 : er1, Ec, S(0));
  }
  return o;
}
template <typename S>
__device__ __noinline__ Tile8<S> digits_tile8(const uint4* Af, const short* __restrict__ er,
                                              const uint4* Bf, int rows, int kt_n, int mt, int lane, int E) {
  return tile8_products<S>(Af, er, Bf, rows, kt_n, mt, lane, E);
}

// ---- eight columns, 94-bit operands ---------------------------------------------
// For the single products y = S v, whose every entry is a result of its own: T_e's
// rows span up to 2^30 and more (slots of the far face against the near ones), so
// an entry can be that much smaller than row maximum times column maximum, and
// 62 bits relative to those left it 25 bits or fewer.  With rows that span at most
// 2^R the error of an entry is below that of a chain of K FMAs, K 2^-53 of its sum of
// magnitudes, as far as R <= 35: that sum is at least 2^-R of row maximum times
// column maximum, of which the operands lose K 2^-92 and the left-out weights, at
// most (11 K 2^14 256^10) 2^-188, four times K 2^-90.5.
//
// A weight takes up to 12 products per column: K <= 80 columns add exactly in an
// accumulator (12 * 80 * 2^14 < 2^24), so the sums of more than five k tiles are
// taken out halfway.

// value of hi 2^64 + mid 2^32 + lo (each below 2^52), times 2^s
__device__ __forceinline__ double wide_value(long long hi, long long mid, long long lo, int s) {
  mid += lo >> 32;
  hi += mid >> 32;
  unsigned long long t = ((unsigned long long)(uint32_t)mid << 32) | (uint32_t)lo;
  const bool neg = hi < 0;
  if (neg) {
    t = 0 - t;
    hi = ~hi + (t == 0);
  }
  double v = fma((double)hi, 0x1p64, (double)t);
  v = neg ? -v : v;
  return s > -1000 && s < 850 ? v * __longlong_as_double((long long)(1023 + s) << 52) : scale2(v, s);
}

__device__ __forceinline__ void pack_tile_wide(uint4* Bf, int lane, const double (&v)[4], int E) {
  Bits96 Y[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) Y[u] = to_digits96(v[u], E);
#pragma unroll
  for (int j = 0; j < 12; j += 2)
    Bf[j / 2 * 32 + lane] = make_uint4(digit_pair(Y[0].w[j / 4], Y[1].w[j / 4], j & 3), digit_pair(Y[2].w[j / 4], Y[3].w[j / 4], j & 3),
                                       digit_pair(Y[0].w[j / 4], Y[1].w[j / 4], (j & 3) + 1),
                                       digit_pair(Y[2].w[j / 4], Y[3].w[j / 4], (j & 3) + 1));
}

// Row tile mt of A times the packed columns, as tile8_products.
__device__ __forceinline__ Tile8<double> tile8_wide(const uint4* Af, const short* __restrict__ er, const uint4* Bf, int rows,
                                                    int kt_n, int mt, int lane, int E) {
  constexpr int ND = Digits<Wide>::ND, GMIN = Digits<Wide>::GMIN, NG = Digits<Wide>::NG, H = ND / 2;
  const int g = lane >> 2, q = lane & 3, row0 = mt * 16 + g;
  const uint4* A = Af + (size_t)mt * kt_n * H * 32 + lane;
  uint4 nx[H];
  ld_frag<Wide>(nx, A, 0);
  const int er0 = row0 < rows ? __ldg(er + row0) : 0, er1 = row0 + 8 < rows ? __ldg(er + row0 + 8) : 0;
  long long sum[4][3] = {};  // per value: weights 0-3, 4-7, 8-11 (units of 256^GMIN, 256^4, 256^8 of it)
  const int half = kt_n > 5 ? (kt_n + 1) / 2 : kt_n;
#pragma unroll 1
  for (int k0 = 0; k0 < kt_n; k0 += half) {
    float acc[NG][4];
#pragma unroll
    for (int c = 0; c < NG; ++c)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[c][v] = 0.f;
#pragma unroll 1
    for (int kt = k0; kt < min(k0 + half, kt_n); ++kt) {
      uint4 av[H], bv[H];
#pragma unroll
      for (int p = 0; p < H; ++p) {
        av[p] = nx[p];
        bv[p] = Bf[(kt * H + p) * 32 + lane];
      }
      if (kt + 1 < kt_n) ld_frag<Wide>(nx, A, kt + 1);
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        uint32_t a[4];
        const uint4 w = av[i / 2];
        digit_a((i & 1) ? w.z : w.x, (i & 1) ? w.w : w.y, a);
#pragma unroll
        for (int j = 0; j < ND; ++j) {
          if (i + j < GMIN) continue;
          const uint4 b = bv[j / 2];
          mma_16816(acc[i + j - GMIN], a, (j & 1) ? b.z : b.x, (j & 1) ? b.w : b.y);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
      for (int c = 0; c < NG; ++c) sum[v][c / 4] += (long long)__float2int_rn(acc[c][v]) << (8 * (c & 3));
  }
  Tile8<double> o;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const int Ec = __shfl_sync(0xffffffffu, E, 4 * (2 * q + (v & 1)));
    // 256^11 2^(er - 94) 2^(E - 1022 - 94)
    o.z[v] = wide_value(sum[v][2], sum[v][1], sum[v][0], (v < 2 ? er0 : er1) + Ec - 1022 + 88 - 188);
  }
  return o;
}

// ---- one column --------------------------------------------------------------
// The eight mma columns are the weights: digit i of A meets digit n + GMIN - i
// of x in column n, so the digits of A share one accumulator tile (two, by
// parity, for shorter chains).  Bf: one fragment per digit i of A
// (digit_bwords words).  x: len entries (as for pack_cols); returns the largest
// exponent field (>= 1).  One warp packs the k tiles part, part + parts, ...
template <typename S>
__device__ __noinline__ int pack_one(uint4* Bf, const S* x, int len, int lane, int part, int parts) {
  constexpr int ND = Digits<S>::ND, GMIN = Digits<S>::GMIN, NG = Digits<S>::NG, OFF = ND - 1 - GMIN;
  const int g = lane >> 2, q = lane & 3, kt_n = digit_tiles(len);
  int E = 1;
#pragma unroll 1
  for (int k = lane; k < len; k += 32) E = max(E, exp_field(x[k]));
  E = __reduce_max_sync(0xffffffffu, E);
  constexpr unsigned long long kFill = 0x8080808080808080ull;
#pragma unroll 1
  for (int kt = part; kt < kt_n; kt += parts) {
    unsigned long long Y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = kt * 16 + 2 * q + (u & 1) + 8 * (u >> 1);
      unsigned long long y = to_digits(k < len ? x[k] : S(0), E);
      if (sizeof(S) == 4) y = ((y | (kFill << 32)) << (8 * OFF)) | (kFill >> (64 - 8 * (OFF > 0 ? OFF : 1)));
      // digits moved down by g places, zeros moved in at the top
      if (g > 0) y = (y >> (8 * g)) | (kFill << (64 - 8 * g));
      Y[u] = y;
    }
    uint32_t r[ND][2];
#pragma unroll
    for (int i = 0; i < ND; ++i) {  // digit g + GMIN - i of x is now at place GMIN - i + OFF = ND - 1 - i
      r[i][0] = g < NG ? digit_pair(Y[0], Y[1], ND - 1 - i) : 0u;
      r[i][1] = g < NG ? digit_pair(Y[2], Y[3], ND - 1 - i) : 0u;
    }
#pragma unroll
    for (int i = 0; i < ND; i += 2)
      Bf[(kt * (ND / 2) + i / 2) * 32 + lane] = make_uint4(r[i][0], r[i][1], r[i + 1][0], r[i + 1][1]);
  }
  __syncwarp();
  return E;
}

// row of a row tile whose value digits_tile1 leaves in this lane, -1: none
__device__ __forceinline__ int tile1_row(int mt, int lane, int rows) {
  const int q = lane & 3, row = mt * 16 + (lane >> 2) + (q < 2 ? 0 : 8);
  return !(q & 1) && row < rows ? row : -1;
}

// Row tile mt of A times the packed column: the value of row tile1_row.
template <typename S>
__device__ __noinline__ S digits_tile1(const uint4* Af, const short* __restrict__ er, const uint4* Bf,
                                       int rows, int kt_n, int mt, int lane, int E) {
  constexpr int ND = Digits<S>::ND;
  const int q = lane & 3, row = tile1_row(mt, lane, rows);
  const uint4* A = Af + (size_t)mt * kt_n * (ND / 2) * 32 + lane;
  uint4 a0[ND / 2], a1[ND / 2];
  ld_frag<S>(a0, A, 0);
  if (kt_n > 1) ld_frag<S>(a1, A, 1);
  const int err = row >= 0 ? __ldg(er + row) : 0;
  float acc[2][4];
#pragma unroll
  for (int v = 0; v < 8; ++v) acc[v >> 2][v & 3] = 0.f;
  auto step = [&](uint4 (&f)[ND / 2], int kt) {  // k tile kt, whose fragments f then become those of kt + 2
    uint4 b[ND / 2];
#pragma unroll
    for (int p = 0; p < ND / 2; ++p) b[p] = Bf[(kt * (ND / 2) + p) * 32 + lane];
    uint32_t a[ND][4];
#pragma unroll
    for (int p = 0; p < ND / 2; ++p) {
      digit_a(f[p].x, f[p].y, a[2 * p]);
      digit_a(f[p].z, f[p].w, a[2 * p + 1]);
    }
    if (kt + 2 < kt_n) ld_frag<S>(f, A, kt + 2);
#pragma unroll
    for (int p = 0; p < ND / 2; ++p) {
      mma_16816(acc[0], a[2 * p], b[p].x, b[p].y);
      mma_16816(acc[1], a[2 * p + 1], b[p].z, b[p].w);
    }
  };
#pragma unroll 1
  for (int kt = 0; kt < kt_n; kt += 2) {
    step(a0, kt);
    if (kt + 1 < kt_n) step(a1, kt + 1);
  }
  // lane holds weights 2q, 2q + 1 of rows g and g + 8 (each accumulator stays
  // within 2^24, exact, for up to 256 columns); the quad adds them up: row g ends in lane
  // q = 0, row g + 8 in lane q = 2
  const int m0 = (q & 1) ? 1 << 16 : 1;
  long long w[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int s0 = __float2int_rn(acc[0][2 * h]) + __float2int_rn(acc[1][2 * h]);
    const int s1 = __float2int_rn(acc[0][2 * h + 1]) + __float2int_rn(acc[1][2 * h + 1]);
    w[h] = (long long)s0 * m0 + (long long)s1 * (m0 << 8);
    w[h] += __shfl_xor_sync(0xffffffffu, w[h], 1);
  }
  const long long got = __shfl_xor_sync(0xffffffffu, q < 2 ? w[1] : w[0], 2);
  return digits_short(q < 2 ? got : w[1], q < 2 ? w[0] : got, err, E, S(0));
}

// v 2^sh rounded to an integer (below 2^62, or 2^94 in 128 bits)
template <typename U>
inline U to_fixed(double v, int sh) {
  if constexpr (sizeof(U) == 8) {
    return (U)std::llrint(std::ldexp(v, sh));
  } else {
    int e = 0;
    const double m = std::frexp(v, &e);  // |v| 2^sh = |m| 2^(e + sh)
    const int up = e + sh - 53;          // places that 53 bits of m move up
    if (up <= 0) return (U)(__int128)std::llrint(std::ldexp(m, e + sh));
    return (U)((__int128)std::llrint(std::ldexp(m, 53)) << up);
  }
}

// Packs count row-major rows x cols matrices: fragments (digit_words each) and
// row exponents (rows each, within +-400: the results' exponents are formed
// without checks).  A row with an Inf or NaN, or above 2^400, is marked.
template <typename S>
void pack_digits(const double* A, int rows, int cols, size_t count, std::vector<uint4>* frag, std::vector<short>* er) {
  constexpr int ND = Digits<S>::ND, B = Digits<S>::B;
  const int mt_n = digit_tiles(rows), kt_n = digit_tiles(cols);
  frag->assign(count * digit_words<S>(rows, cols), make_uint4(0, 0, 0, 0));
  er->assign(count * rows, 0);
  using U = typename std::conditional<(ND > 8), unsigned __int128, uint64_t>::type;
  U kBias = 0;
  for (int i = 0; i < ND; ++i) kBias |= (U)0x80 << (8 * i);
#pragma omp parallel for schedule(static) if (count > 16)
  for (long long c = 0; c < (long long)count; ++c) {
    const double* a = A + c * rows * cols;
    std::vector<U> Y((size_t)mt_n * 16 * kt_n * 16, kBias);
    for (int r = 0; r < rows; ++r) {
      double mx = 0;
      bool ok = true;
      for (int k = 0; k < cols; ++k) {
        const double v = std::fabs(a[(size_t)r * cols + k]);
        ok = ok && v < 0x1p400;
        if (v > mx) mx = v;
      }
      int e = 0;
      if (ok && mx > 0) std::frexp(mx, &e);
      e = std::max(e, -400);
      (*er)[c * rows + r] = ok ? (short)e : kBadRow;
      if (!ok) continue;
      for (int k = 0; k < cols; ++k)
        Y[(size_t)r * kt_n * 16 + k] = kBias + to_fixed<U>(a[(size_t)r * cols + k], B - e);
    }
    uint4* f = frag->data() + c * digit_words<S>(rows, cols);
    for (int mt = 0; mt < mt_n; ++mt)
      for (int kt = 0; kt < kt_n; ++kt)
        for (int p = 0; p < ND / 2; ++p)
          for (int lane = 0; lane < 32; ++lane) {
            const int g = lane / 4, q = lane % 4;
            uint32_t w[4];
            for (int h = 0; h < 4; ++h) {  // h: digit 2p + (h / 2), columns 2q + 8 (h % 2) of rows g, g + 8
              w[h] = 0;
              for (int b = 0; b < 4; ++b) {
                const int row = mt * 16 + g + 8 * (b / 2), col = kt * 16 + 2 * q + (b % 2) + 8 * (h % 2);
                const U y = Y[(size_t)row * kt_n * 16 + col];
                w[h] |= (uint32_t)((y >> (8 * (2 * p + h / 2))) & 0xff) << (8 * b);
              }
            }
            f[((size_t)(mt * kt_n + kt) * (ND / 2) + p) * 32 + lane] = make_uint4(w[0], w[1], w[2], w[3]);
          }
  }
}

}  // namespace
