// pcz_device.cuh -- device-side building blocks of the PCZ block coder used as
// the compressor C / decompressor D of the multi-component framework
// (Algorithm 1 and 2 of Magri & Lindstrom, Sec. 4).  GPU path only.
//
// The coder is zfp-style (Sec. 4.4, Sec. 6.1): one exponent per 4^d brick and
// component, an exactly invertible integer lifting transform, negabinary
// coefficients and group-tested bit planes (Sec. 2).  The paper does not fix
// the coder's internals; the project rules R4..R15 do, and each is restated
// where it is implemented.  All floating-point work here is IEEE
// round-to-nearest with no contraction by the compiler, and the only arithmetic
// on T values that rounds is one add or one subtract (explicit _rn intrinsics) and
// the conversion of an integer coefficient.  What else runs in floating point is
// exact: products by powers of two that stay normal, their fused adds (which round
// once, as the add does), and the lifting, in float, of values that need at most
// 24 bits.  Scales outside those ranges work on the bit patterns with integer
// operations.
#pragma once

#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "pcz_kernels.h"

namespace pcz {
constexpr int kModeZero = 0, kModeCoded = 1, kModeRaw = 2;

// ---------------------------------------------------------------------------
// Field types.  P = integer width = bits of T.
// ---------------------------------------------------------------------------
template <typename T>
struct Fmt;

template <>
struct Fmt<float> {
  using U = uint32_t;
  using S = int32_t;
  static constexpr int P = 32;
  static constexpr int MANT = 24;    // significand bits, hidden bit included
  static constexpr int EMIN = -125;  // frexp exponent of the smallest normal
  static constexpr int EBITS = 8;    // stored block exponent width
  static constexpr int EBIAS = 126;  // stored = emax + EBIAS
  static constexpr int BIAS = 127;   // IEEE exponent bias
  static constexpr int EXPW = 8;     // IEEE exponent field width
  static constexpr U SIGN = 0x80000000u, ABS = 0x7FFFFFFFu, INF = 0x7F800000u;
  static constexpr U NBM = 0xAAAAAAAAu;
  __device__ static U bits(float v) { return __float_as_uint(v); }
  __device__ static float val(U b) { return __uint_as_float(b); }
  __device__ static float add(float a, float b) { return __fadd_rn(a, b); }
  __device__ static float sub(float a, float b) { return __fsub_rn(a, b); }
  __device__ static int clz(U a) { return __clz(a); }
};

template <>
struct Fmt<double> {
  using U = uint64_t;
  using S = int64_t;
  static constexpr int P = 64;
  static constexpr int MANT = 53;
  static constexpr int EMIN = -1021;
  static constexpr int EBITS = 11;
  static constexpr int EBIAS = 1022;
  static constexpr int BIAS = 1023;
  static constexpr int EXPW = 11;
  static constexpr U SIGN = 0x8000000000000000ull, ABS = 0x7FFFFFFFFFFFFFFFull, INF = 0x7FF0000000000000ull;
  static constexpr U NBM = 0xAAAAAAAAAAAAAAAAull;
  __device__ static U bits(double v) { return (U)__double_as_longlong(v); }
  __device__ static double val(U b) { return __longlong_as_double((long long)b); }
  __device__ static double add(double a, double b) { return __dadd_rn(a, b); }
  __device__ static double sub(double a, double b) { return __dsub_rn(a, b); }
  __device__ static int clz(U a) { return __clzll((long long)a); }
};

// Brick geometry for dimensionality D: N = 4^D coefficients, G = 2D headroom
// bits for the forward transform's growth (R6), C guard planes (R10): the
// smallest c with 2^c above (2/3) * 2.75^D, the inverse transform's worst-case
// error per unit of truncated coefficient.
template <int D>
struct Geo {
  static constexpr int N = D == 1 ? 4 : D == 2 ? 16 : 64;
  static constexpr int G = 2 * D;
  static constexpr int C = D == 1 ? 1 : D == 2 ? 3 : 4;
};

// ---------------------------------------------------------------------------
// Wrapping P-bit integer arithmetic (two's complement, modulo 2^P).
// ---------------------------------------------------------------------------
template <typename S>
__device__ __forceinline__ S wadd(S a, S b) {
  using U = typename std::make_unsigned<S>::type;
  return (S)((U)a + (U)b);
}
template <typename S>
__device__ __forceinline__ S wsub(S a, S b) {
  using U = typename std::make_unsigned<S>::type;
  return (S)((U)a - (U)b);
}

// R7: forward lifting of one 4-vector: integer Haar on the pairs, Haar on the
// pair means, then the second difference and the fine slope minus half the
// coarse slope.  a,b,c,d -> (mean, coarse slope, e1, e2).
template <typename S>
__device__ __forceinline__ void lift_fwd(S& a, S& b, S& c, S& d) {
  S d1 = wsub(b, a);
  S s1 = wadd(a, d1 >> 1);
  S d2 = wsub(d, c);
  S s2 = wadd(c, d2 >> 1);
  S d0 = wsub(s2, s1);
  S s0 = wadd(s1, d0 >> 1);
  S e2 = wsub(d2, d1);
  S e1 = wsub(d1, d0 >> 1);
  a = s0;
  b = d0;
  c = e1;
  d = e2;
}

// R7 inverse: the forward steps replayed backwards with opposite signs.
template <typename S>
__device__ __forceinline__ void lift_inv(S& a, S& b, S& c, S& d) {
  S s0 = a, d0 = b, e1 = c, e2 = d;
  S d1 = wadd(e1, d0 >> 1);
  S d2 = wadd(e2, d1);
  S s1 = wsub(s0, d0 >> 1);
  S s2 = wadd(s1, d0);
  a = wsub(s1, d1 >> 1);
  b = wadd(a, d1);
  c = wsub(s2, d2 >> 1);
  d = wadd(c, d2);
}

// lift_inv in float, the same values wherever every shift of lift_inv divides an
// even number and no value needs more than 24 bits: 8 operations instead of 11,
// on the pipe that integer work leaves idle.
__device__ __forceinline__ void lift_inv(float& a, float& b, float& c, float& d) {
  const float s0 = a, d0 = b, e1 = c, e2 = d;
  const float d1 = __fmaf_rn(0.5f, d0, e1);
  const float d2 = __fadd_rn(e2, d1);
  const float s1 = __fmaf_rn(-0.5f, d0, s0);
  const float s2 = __fadd_rn(s1, d0);
  a = __fmaf_rn(-0.5f, d1, s1);
  b = __fadd_rn(a, d1);
  c = __fmaf_rn(-0.5f, d2, s2);
  d = __fadd_rn(c, d2);
}

// R9: negabinary map and its inverse, modulo 2^P.
template <typename T>
__device__ __forceinline__ typename Fmt<T>::U nb_fwd(typename Fmt<T>::S q) {
  using F = Fmt<T>;
  return (typename F::U)(((typename F::U)q + F::NBM) ^ F::NBM);
}
template <typename T>
__device__ __forceinline__ typename Fmt<T>::S nb_inv(typename Fmt<T>::U u) {
  using F = Fmt<T>;
  return (typename F::S)((u ^ F::NBM) - F::NBM);
}

// IEEE biased exponent field of a bit pattern.
template <typename T>
__device__ __forceinline__ int biased_exp(typename Fmt<T>::U b) {
  using F = Fmt<T>;
  return (int)((b >> (F::MANT - 1)) & ((1u << F::EXPW) - 1));
}

// R6: block exponent from the largest biased exponent over the brick: emax is
// the frexp exponent of the largest magnitude, floored at the smallest normal's
// (subnormals and zeros carry biased exponent 0).
template <typename T>
__device__ __forceinline__ int block_emax_from_be(int be_max) {
  using F = Fmt<T>;
  return (be_max > 1 ? be_max : 1) - (F::BIAS - 1);
}

// R6: q = sign(e) * floor(|e| * 2^s), computed exactly on the bit pattern:
// |e| = m * 2^ex with m the integer significand.
template <typename T>
__device__ __forceinline__ typename Fmt<T>::S quantize(typename Fmt<T>::U b, int s) {
  using F = Fmt<T>;
  using U = typename F::U;
  using S = typename F::S;
  int be = biased_exp<T>(b);
  U m = b & ((U(1) << (F::MANT - 1)) - 1);
  if (be) m |= U(1) << (F::MANT - 1);
  int ex = (be ? be : 1) - F::BIAS - (F::MANT - 1);
  int sh = ex + s;
  U a;
  if (sh >= 0)
    a = sh >= F::P ? U(0) : (m << sh);
  else
    a = -sh >= F::P ? U(0) : (m >> (-sh));
  S q = (S)a;
  return (b & F::SIGN) ? (S)(0 - (U)q) : q;
}

// R13: the T value nearest to q * 2^-s (ties to even, one rounding, IEEE signed
// zero, +-inf beyond the largest finite value), as a bit pattern.
template <typename T>
__device__ __forceinline__ typename Fmt<T>::U dequantize_bits(typename Fmt<T>::S q, int s) {
  using F = Fmt<T>;
  using U = typename F::U;
  if (q == 0) return U(0);
  U a = q < 0 ? (U)(U(0) - (U)q) : (U)q;
  int nb = F::P - F::clz(a);            // bit length of |q|
  int E = nb - s;                       // frexp exponent of the exact value
  int qe = (E > F::EMIN ? E : F::EMIN) - F::MANT;  // exponent of the last place
  int sh = qe + s;                      // low bits of |q| below that place
  U r;
  if (sh <= 0) {
    r = a << (-sh);
  } else if (sh > F::P) {
    r = 0;
  } else if (sh == F::P) {
    r = a > (U(1) << (F::P - 1)) ? U(1) : U(0);
  } else {
    r = a >> sh;
    U rem = a & ((U(1) << sh) - 1);
    U half = U(1) << (sh - 1);
    if (rem > half || (rem == half && (r & 1))) r += 1;
  }
  int ef = qe - (F::EMIN - F::MANT);    // biased exponent - 1 for a normal result
  U out;
  if (ef >= (1 << F::EXPW) - 2) {
    out = F::INF;
  } else {
    out = ((U)ef << (F::MANT - 1)) + r;  // a carry out of r bumps the exponent
    if (out > F::INF) out = F::INF;
  }
  return q < 0 ? (out | F::SIGN) : out;
}

// R13 for float64 when the result is known to be normal and finite (s in
// [-960, 1022], see dequantize_line): the 53 leading bits of |q| rounded to
// nearest, ties to even, by adding half an ulp less one plus the kept lsb
// before the shift.  A carry out of the 53 bits moves into the exponent field.
__device__ __forceinline__ uint64_t dequantize_f64_normal(int64_t q, int s) {
  if (q == 0) return 0ull;
  const uint64_t a = q < 0 ? 0ull - (uint64_t)q : (uint64_t)q;
  const int nb = 64 - __clzll((long long)a);  // |q| < 2^nb, so a + half stays below 2^64
  const int sh = nb - 53;
  uint64_t r;
  if (sh > 0)
    r = (a + ((1ull << (sh - 1)) - 1ull) + ((a >> sh) & 1ull)) >> sh;
  else
    r = a << (-sh);
  const uint64_t bits = ((uint64_t)(nb - s + 1021) << 52) + r;  // r's bit 52 completes the exponent
  return q < 0 ? (bits | Fmt<double>::SIGN) : bits;
}

// R13 for the 4 values of a line that share the block's scale s.
//  float: when 2^-s is a normal float, int -> float rounding followed by the
//    exact multiplication by 2^-s is the single correct rounding for every q
//    (|q| >= 1 keeps the result normal; overflow gives +-inf as IEEE does;
//    q = 0 gives +0), so the test is made once per line.
//  double with EXP: int64 -> double rounding (one rounding), then 2^-s applied
//    by subtracting s from the exponent field.  For |q| in [1, 2^63] the
//    rounded value's biased exponent lies in [1023, 1086], so for s in
//    [-960, 1022] the scaled one lies in [1, 2046]: normal and finite, the
//    scaling exact, the field never borrows from or carries into the sign.
//    This spends one conversion instead of some 25 integer instructions, for
//    kernels whose integer pipe is the busier one.
//  Other cases take the integer path (dequantize_bits).
template <typename T, bool EXP>
__device__ __forceinline__ void dequantize_line(const typename Fmt<T>::S* q, int s, T* v) {
  if constexpr (sizeof(T) == 4) {
    if (s >= -127 && s <= 126) {
      const float sc = __uint_as_float((uint32_t)(127 - s) << 23);
#pragma unroll
      for (int m = 0; m < 4; ++m) v[m] = __fmul_rn(__int2float_rn(q[m]), sc);
      return;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = __uint_as_float(dequantize_bits<float>(q[m], s));
  } else {
    if (EXP && s >= -960 && s <= 1022) {
      const uint32_t adj = (uint32_t)s << 20;  // s in the exponent field of the high word
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const double d = __ll2double_rn(q[m]);
        const uint32_t hi = (uint32_t)__double2hiint(d);
        v[m] = __hiloint2double((int)(hi ? hi - adj : 0u), __double2loint(d));  // q = 0 stays +0
      }
      return;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = Fmt<double>::val(dequantize_bits<double>(q[m], s));
  }
}

// R13 for a float64 coefficient decoded in 32-bit integers in units of 2^e:
// the coefficient is q = r * 2^e exactly, |r| < 2^31, and 1 <= |q| < 2^63 when
// r != 0.  For s in [-960, 1022] the result q * 2^-s is then normal and finite
// (the bound of dequantize_line), so no rounding is needed: with |r|'s leading
// one moved to bit 31, the 31 bits below it are the top of the 52-bit
// fraction, and the biased exponent is 1023 + (31 - clz|r|) + e - s.  Pass
// eb = (1053 + e - s) << 20 (that exponent minus 1, plus clz|r|, in the high
// word's exponent field; the leading one, added at bit 20, completes it).
// r = 0 gives +0.  Integer instructions only: no int -> double conversion,
// whose FP64 pipe the partial-sum adds keep busy.
__device__ __forceinline__ double scaled_i32_to_f64(int32_t r, uint32_t eb) {
  const uint32_t a = (uint32_t)abs(r);
  const uint32_t z = (uint32_t)__clz(a);
  const uint32_t n = __funnelshift_l(0u, a, z);  // |r| << clz; 0 for r = 0
  const uint32_t hw = ((n >> 11) + eb - (z << 20)) | ((uint32_t)r & 0x80000000u);
  return __hiloint2double(a ? (int)hw : 0, (int)(n << 21));
}

// r * 2^e for a float r, exactly, where the result is a normal double (or r is
// 0): adj = (896 + e) << 20, the change of exponent bias in the high word.
__device__ __forceinline__ double scaled_f32_to_f64(float r, uint32_t adj) {
  const int b = __float_as_int(r);
  const uint32_t hi = ((uint32_t)(b >> 3) & 0x8FFFFFFFu) + adj;
  return __hiloint2double(r == 0.0f ? 0 : (int)hi, b << 29);
}

// ---------------------------------------------------------------------------
// R8: sequency order of the coefficients, ties by brick position.  make_perm(n).pos[r]
// = brick position of the r-th coded coefficient of n; make_rank below is the
// inverse for 4^3 (kRank3 in the 3D kernels).  Built at compile time by ranking
// every position.
// ---------------------------------------------------------------------------
struct PermTable {
  int8_t pos[64];
};

__host__ __device__ constexpr int seq_key(int p) { return (p & 3) + ((p >> 2) & 3) + (p >> 4); }

__host__ __device__ constexpr PermTable make_perm(int n) {
  PermTable t{};
  for (int p = 0; p < n; ++p) {
    int rank = 0;
    for (int q = 0; q < n; ++q)
      if (seq_key(q) < seq_key(p) || (seq_key(q) == seq_key(p) && q < p)) ++rank;
    t.pos[rank] = (int8_t)p;
  }
  return t;
}

// ---------------------------------------------------------------------------
// Debug builds (-DPCZ_DEBUG) check buffer accesses: a failed check sets bit
// `site` of this translation unit's check word and skips the access (no trap,
// so a bad index cannot fault the GPU), and pc_debug_status reports the word.
// Release builds compile the checks out.  Sites: 0 the 3D chunk bit buffer,
// 1 the 3D plane tables, 2 the 1D/2D chunk bit buffer, 3 the retrieval plane
// slots and spill.
// ---------------------------------------------------------------------------
#ifdef PCZ_DEBUG
static __device__ unsigned int g_pcz_check;
#define PCZ_CHECK(cond, site) ((cond) ? true : (atomicOr(&g_pcz_check, 1u << (site)), false))
#else
#define PCZ_CHECK(cond, site) true
#endif

// This translation unit's check word (0 in release builds); reset clears it.
static inline uint32_t read_check_word(int reset) {
#ifdef PCZ_DEBUG
  unsigned int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_pcz_check, sizeof(v)) != cudaSuccess) v = ~0u;
  if (reset) {
    const unsigned int z = 0;
    cudaMemcpyToSymbol(g_pcz_check, &z, sizeof(z));
  }
  return v;
#else
  (void)reset;
  return 0;
#endif
}

// ---------------------------------------------------------------------------
// Bit writes into a shared-memory bit buffer (bit b = bit b%32 of word b/32):
// OR v into bits [off, off + 64).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void or_bits(uint32_t* buf, uint32_t off, uint64_t v) {
  if (!v) return;
  uint32_t w = off >> 5, sh = off & 31;
  uint64_t lo = v << sh;
  uint32_t hi = sh ? (uint32_t)(v >> (64 - sh)) : 0u;
  if ((uint32_t)lo) atomicOr(buf + w, (uint32_t)lo);
  if ((uint32_t)(lo >> 32)) atomicOr(buf + w + 1, (uint32_t)(lo >> 32));
  if (hi) atomicOr(buf + w + 2, hi);
}

// or_bits into a buffer of cap_bits bits, checked in debug builds.
__device__ __forceinline__ void or_bits_in(uint32_t* buf, uint32_t off, uint64_t v, uint32_t cap_bits, int site) {
#ifdef PCZ_DEBUG
  if (v && !PCZ_CHECK(off + (uint32_t)(64 - __clzll((long long)v)) <= cap_bits, site)) return;
#endif
  or_bits(buf, off, v);
}

// 64 bits of a word stream starting at bit pos (bit b = bit b%64 of word
// b/64); words at or beyond nwords read as zero.
__device__ __forceinline__ uint64_t peek64(const uint64_t* __restrict__ w, uint64_t nwords, uint64_t pos) {
  uint64_t i = pos >> 6;
  uint32_t sh = (uint32_t)(pos & 63);
  uint64_t a = i < nwords ? __ldg(w + i) : 0ull;
  if (!sh) return a;
  uint64_t b = i + 1 < nwords ? __ldg(w + i + 1) : 0ull;
  return (a >> sh) | (b << (64 - sh));
}

// The largest 64-bit value over the lanes of `mask` (every lane of it calls):
// the largest high word, then the largest low word among the lanes that hold
// it -- two warp reductions (redux) instead of a shuffle ladder.
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned mask, unsigned long long v) {
  const unsigned hi = __reduce_max_sync(mask, (unsigned)(v >> 32));
  const unsigned lo = __reduce_max_sync(mask, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
  return ((unsigned long long)hi << 32) | lo;
}

// One x-line of a brick (4 consecutive values) between registers and memory:
// a single 16-byte access per 16 bytes when the line is whole and aligned
// (fewer transactions, which matters most when the memory is on the host side
// of the C2C link), element by element otherwise.
template <typename T>
__device__ __forceinline__ void store_line(T* dst, const T* v, const bool* ok) {
  if (ok[0] && ok[1] && ok[2] && ok[3] && ((uintptr_t)dst & 15) == 0) {
    if constexpr (sizeof(T) == 4) {
      *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
      reinterpret_cast<double2*>(dst)[0] = make_double2(v[0], v[1]);
      reinterpret_cast<double2*>(dst)[1] = make_double2(v[2], v[3]);
    }
    return;
  }
#pragma unroll
  for (int m = 0; m < 4; ++m)
    if (ok[m]) dst[m] = v[m];
}

// Loads the line's first nv (1..4) values; lanes past them repeat the last
// (R4 edge replication along x).
template <typename T>
__device__ __forceinline__ void load_line(const T* src, int nv, T* v) {
  if (nv == 4 && ((uintptr_t)src & 15) == 0) {
    if constexpr (sizeof(T) == 4) {
      const float4 a = *reinterpret_cast<const float4*>(src);
      v[0] = a.x;
      v[1] = a.y;
      v[2] = a.z;
      v[3] = a.w;
    } else {
      const double2 a = reinterpret_cast<const double2*>(src)[0];
      const double2 b = reinterpret_cast<const double2*>(src)[1];
      v[0] = a.x;
      v[1] = a.y;
      v[2] = b.x;
      v[3] = b.y;
    }
    return;
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = src[min(m, nv - 1)];
}

// Bit transposes within a lane.  transpose8: word i holds 8 bits (planes) each
// of the coefficients i, i + 8, i + 4 and i + 12 (from its low byte up);
// afterwards word j holds planes j and j + 4 of the 16 coefficients.  transpose16: word i holds 16 bits (planes) of
// coefficient i in its low half and of coefficient i + 8 in its high half;
// afterwards word j holds plane j of the 16 coefficients in its low half and
// plane j + 8 in its high half.  transpose32: word i holds 32 bits of
// coefficient i; afterwards word j holds planes j and j + 16.  Stages of 4, 2
// and 1 exchange bit groups between two words with a shift and a logic op per
// result; the stage of 8 is one byte permute per result.
template <int N, int K>
__device__ __forceinline__ void exchange_stage(uint32_t (&a)[N], uint32_t m) {
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (!(i & K)) {
      const uint32_t x = a[i], y = a[i + K];
      a[i] = (x & m) | ((y << K) & ~m);
      a[i + K] = ((x >> K) & m) | (y & ~m);
    }
}
__device__ __forceinline__ void transpose8(uint32_t (&a)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t t = (a[i] ^ (a[i] >> 12)) & 0x0000F0F0u;
    a[i] ^= t ^ (t << 12);
  }
  exchange_stage<4, 2>(a, 0x33333333u);
  exchange_stage<4, 1>(a, 0x55555555u);
}
// transpose8 backwards: word j holds planes j and j + 4; afterwards word i holds
// the bytes of coefficients i, i + 8, i + 4 and i + 12.
__device__ __forceinline__ void untranspose8(uint32_t (&a)[4]) {
  exchange_stage<4, 1>(a, 0x55555555u);
  exchange_stage<4, 2>(a, 0x33333333u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t t = (a[i] ^ (a[i] >> 12)) & 0x0000F0F0u;
    a[i] ^= t ^ (t << 12);
  }
}
__device__ __forceinline__ void untranspose16(uint32_t (&a)[8]) {  // transpose16 backwards
  exchange_stage<8, 1>(a, 0x55555555u);
  exchange_stage<8, 2>(a, 0x33333333u);
  exchange_stage<8, 4>(a, 0x0F0F0F0Fu);
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = __byte_perm(a[i], 0u, 0x3120);
}
__device__ __forceinline__ void transpose16(uint32_t (&a)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = __byte_perm(a[i], 0u, 0x3120);
  exchange_stage<8, 4>(a, 0x0F0F0F0Fu);
  exchange_stage<8, 2>(a, 0x33333333u);
  exchange_stage<8, 1>(a, 0x55555555u);
}
__device__ __forceinline__ void transpose32_lane(uint32_t (&a)[16]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t x = a[i], y = a[i + 8];
    a[i] = __byte_perm(x, y, 0x6240);
    a[i + 8] = __byte_perm(x, y, 0x7351);
  }
  exchange_stage<16, 4>(a, 0x0F0F0F0Fu);
  exchange_stage<16, 2>(a, 0x33333333u);
  exchange_stage<16, 1>(a, 0x55555555u);
}

// |v| as an integer that orders like it (NaN above +inf above every finite
// value): the bit pattern without its sign.  float64 masks the high word only:
// masking the whole pattern is recognised as fabs and emitted as an add on the
// FP64 pipe, which costs as much as a real one.
__device__ __forceinline__ uint32_t magnitude(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }
__device__ __forceinline__ uint64_t magnitude(double v) {
  return ((uint64_t)((uint32_t)__double2hiint(v) & 0x7FFFFFFFu) << 32) | (uint32_t)__double2loint(v);
}

// The largest magnitude of a lane's N values.  float32 takes the maximum of |v|
// with NaN propagated, one instruction per value; a NaN's own bits, which that
// maximum does not keep, are looked up.
__device__ __forceinline__ float max_abs_nan(float a, float b) {
  float r;
  asm("{\n .reg .f32 t;\n abs.f32 t, %2;\n max.NaN.f32 %0, %1, t;\n}\n" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
template <typename T, int N>
__device__ __forceinline__ typename Fmt<T>::U lane_max(const T* e) {
  using U = typename Fmt<T>::U;
  U m;
  if constexpr (sizeof(T) == 4) {
    float f = 0.0f;
#pragma unroll
    for (int v = 0; v < N; ++v) f = max_abs_nan(f, e[v]);
    m = __float_as_uint(f);
    if (m > Fmt<T>::INF) {
      m = 0;
#pragma unroll
      for (int v = 0; v < N; ++v) m = max(m, magnitude(e[v]));
    }
  } else {
    m = magnitude(e[0]);
#pragma unroll
    for (int v = 1; v < N; ++v) {
      const U a = magnitude(e[v]);
      m = a > m ? a : m;
    }
  }
  return m;
}

// R6 and R13 for blocks whose scale is outside the common range, out of line.
template <typename T>
__device__ __noinline__ typename Fmt<T>::S quantize_any(typename Fmt<T>::U b, int s) {
  return quantize<T>(b, s);
}
template <typename T>
__device__ __noinline__ typename Fmt<T>::U dequantize_any(typename Fmt<T>::S q, int s) {
  return dequantize_bits<T>(q, s);
}

// R6 for float64 in a block whose scale s lies in [-960, 1000], with Q = 53 + G
// quantisation bits (c = 1075 + G - s): q = sign(e) * ((the 53-bit significand
// << G) >> r) with r = c - biased exponent, which is at least 0 because
// |q| < 2^Q.  A subnormal e, taken with a hidden bit it does not have, is
// shifted out entirely (r >= 75 + G).  c = 4096 gives 0 for every e.
template <int G>
__device__ __forceinline__ int64_t quantize_f64_normal(double e, int c) {
  const uint32_t hi = (uint32_t)__double2hiint(e), lo = (uint32_t)__double2loint(e);
  const uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
  const int r = min(c - (int)((hi >> 20) & 0x7FFu), 63);
  const int64_t a = (int64_t)((m << G) >> r);
  const int64_t sg = (int64_t)((int32_t)hi >> 31);
  return (a ^ sg) - sg;
}

// Group-test code of 8 coefficient bits (R11): each bit in turn, and after
// each 1 the 1 of the next token's test bit.  Its length is 8 + popc(bits).
struct alignas(4) SpreadTable {
  uint16_t code[256];
};
constexpr SpreadTable make_spread() {
  SpreadTable t{};
  for (int v = 0; v < 256; ++v) {
    unsigned code = 0, len = 0;
    for (int j = 0; j < 8; ++j)
      if ((v >> j) & 1) {
        code |= 3u << len;
        len += 2;
      } else {
        ++len;
      }
    t.code[v] = (uint16_t)code;
  }
  return t;
}
static __device__ const SpreadTable kSpread = make_spread();
constexpr int kSpreadBytes = (int)sizeof(SpreadTable);

// Sequential reader of one block's bits with 32-bit positions relative to
// the start of the word that holds the block's first bit: the two current
// words in 32-bit halves, one load per 64 bits consumed, and a 64-bit window
// at any position made of two funnel shifts.  Words at or beyond the
// payload's end read as zero.  Positions must not decrease.
struct BlockBits {
  const uint64_t* __restrict__ w;  // the payload from the block's first word
  uint32_t nw;                     // words readable from w
  uint32_t wi;                     // index of the word in a0:a1
  uint32_t a0, a1, b0, b1;         // words wi and wi + 1
  __device__ __forceinline__ uint64_t ld(uint32_t i) const { return i < nw ? __ldg(w + i) : 0ull; }
  __device__ __forceinline__ void set(uint64_t lo, uint64_t hi) {
    a0 = (uint32_t)lo;
    a1 = (uint32_t)(lo >> 32);
    b0 = (uint32_t)hi;
    b1 = (uint32_t)(hi >> 32);
  }
  // bit position of the block's first bit within the reader's frame: off & 63
  __device__ __forceinline__ void init(const uint64_t* words, uint64_t nwords, uint64_t off) {
    const uint64_t w0 = off >> 6;
    w = words + w0;
    nw = w0 < nwords ? (uint32_t)min(nwords - w0, (uint64_t)0xffffffffu) : 0u;
    wi = 0;
    set(ld(0), ld(1));
  }
  __device__ __forceinline__ void advance() {  // by one word
    a0 = b0;
    a1 = b1;
    const uint64_t nb = ld(++wi + 1);
    b0 = (uint32_t)nb;
    b1 = (uint32_t)(nb >> 32);
  }
  __device__ __forceinline__ uint64_t peek(uint32_t pos) {
    const uint32_t i = pos >> 6;
    if (i != wi) {
      if (i == wi + 1) {
        advance();
      } else {
        set(ld(i), ld(i + 1));
        wi = i;
      }
    }
    return window(pos);
  }
  // 64 bits from pos, which lies in word wi
  __device__ __forceinline__ uint64_t window(uint32_t pos) const {
    const bool up = pos & 32u;  // window starts in the word's upper half
    const uint32_t x0 = up ? a1 : a0, x1 = up ? b0 : a1, x2 = up ? b1 : b0;
    return ((uint64_t)__funnelshift_r(x1, x2, pos) << 32) | __funnelshift_r(x0, x1, pos);
  }
};

// Byte table of the group-test part as a two-state machine: in state "test"
// a 0 ends the part and a 1 starts a run; in state "run" every bit is the
// next coefficient's bit and a 1 ends the run.  Entry 256 * state + byte: byte 0
// the byte's coefficient bits, byte 1 the state after it, byte 2 how many
// coefficients, byte 3 128 when the part ends in the byte, plus the bits used up
// to and including the closing test bit, minus 1.
constexpr int kTokLut = 512;  // entries (2 states x 256 bytes)

struct alignas(16) TokenTable {
  uint32_t entry[kTokLut];
};
constexpr TokenTable make_tokens() {
  TokenTable t{};
  for (int idx = 0; idx < kTokLut; ++idx) {
    unsigned st = (unsigned)idx >> 8, out = 0, cnt = 0, end = 0;
    for (int j = 0; j < 8 && !end; ++j) {
      const unsigned bit = ((unsigned)idx >> j) & 1u;
      if (st == 0) {
        if (bit)
          st = 1;
        else
          end = 128u + (unsigned)j;
      } else {
        out |= bit << cnt;
        ++cnt;
        if (bit) st = 0;
      }
    }
    t.entry[idx] = out | (st << 8) | (cnt << 16) | (end << 24);
  }
  return t;
}
static __device__ const TokenTable kTokens = make_tokens();

// A CTA's copy of the table in shared memory; read after the next barrier.
template <int THREADS>
__device__ __forceinline__ void load_tokens(uint32_t* at) {
  for (int i = threadIdx.x; i < kTokLut; i += THREADS) at[i] = kTokens.entry[i];
}

// The entry for byte `j` (0..3) of g after entry e (0 at the start of a part):
// one byte permute forms the index from e's state byte, whose clear sign bit
// fills the upper bytes.
__device__ __forceinline__ uint32_t token_index(uint32_t e, uint32_t g, int j) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(e), "r"(g), "r"(0x9914 + j));
  return r;
}
__device__ __forceinline__ int token_count(uint32_t e) { return (int)__byte_perm(e, 0u, 0x4442); }

// Rank of each brick position in coded order (R8).
constexpr PermTable make_rank() {
  const PermTable perm = make_perm(64);
  PermTable t{};
  for (int r = 0; r < 64; ++r) t.pos[perm.pos[r]] = (int8_t)r;
  return t;
}
// Places of a lane's coefficients x + 4 z (x = 0..3, y = q) in coded order, a
// byte each: rank r at 16 (r / 16) + 4 (r & 3) + 2 ((r >> 2) & 1) + ((r >> 3) & 1),
// the order in which the bit transposes take 16 coefficients.
__device__ __forceinline__ uint32_t coded_places(const int8_t* rank, int q, int z) {
  uint32_t v = 0;
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const int r = rank[x + 4 * q + 16 * z];
    v |= (uint32_t)((r & 48) + 4 * (r & 3) + 2 * ((r >> 2) & 1) + ((r >> 3) & 1)) << (8 * x);
  }
  return v;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Exchange between the z-planes and the y-planes of a warp's 8 bricks in shared
// memory: 16-byte vectors of 4 values along x (64-bit values: two sets of 2
// each), vector (y, z) of brick b at `at`.  Both directions are free of bank
// conflicts.
struct LineSet {
  static constexpr int kVectors = 38 * 4;
  static __device__ __forceinline__ int at(int b, int y, int z) { return (b >> 1) * 38 + (b & 1) + 10 * z + 2 * y; }
};

// 4 values along x to and from the work area, in 16-byte vectors (`set`
// vectors between a 64-bit line's two halves).
__device__ __forceinline__ void put_line(uint4* a, int, const int32_t* v) {
  *a = make_uint4((uint32_t)v[0], (uint32_t)v[1], (uint32_t)v[2], (uint32_t)v[3]);
}
__device__ __forceinline__ void get_line(const uint4* a, int, int32_t* v) {
  const uint4 r = *a;
  v[0] = (int32_t)r.x;
  v[1] = (int32_t)r.y;
  v[2] = (int32_t)r.z;
  v[3] = (int32_t)r.w;
}
__device__ __forceinline__ void put_line(uint4* a, int, const float* v) {
  *reinterpret_cast<float4*>(a) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void get_line(const uint4* a, int, float* v) {
  const float4 r = *reinterpret_cast<const float4*>(a);
  v[0] = r.x;
  v[1] = r.y;
  v[2] = r.z;
  v[3] = r.w;
}
__device__ __forceinline__ void put_line(uint4* a, int set, const int64_t* v) {
  longlong2* d = reinterpret_cast<longlong2*>(a);
  d[0] = make_longlong2(v[0], v[1]);
  d[set] = make_longlong2(v[2], v[3]);
}
__device__ __forceinline__ void get_line(const uint4* a, int set, int64_t* v) {
  const longlong2* d = reinterpret_cast<const longlong2*>(a);
  const longlong2 p = d[0], r = d[set];
  v[0] = p.x;
  v[1] = p.y;
  v[2] = r.x;
  v[3] = r.y;
}

// R7 on a warp's 8 bricks.  v: the lane's z-plane q (value x + 4 y) on entry;
// on return its y-plane q of coefficients (coefficient x + 4 z).  One exchange
// through the work area: a lane lifts along x and y in registers, then along z.
template <typename S>
__device__ __forceinline__ void lift_fwd_bricks(S* v, uint4* zw, uint4* yw, int set) {
#pragma unroll
  for (int y = 0; y < 4; ++y) lift_fwd(v[4 * y], v[4 * y + 1], v[4 * y + 2], v[4 * y + 3]);
#pragma unroll
  for (int x = 0; x < 4; ++x) lift_fwd(v[x], v[x + 4], v[x + 8], v[x + 12]);
#pragma unroll
  for (int y = 0; y < 4; ++y) put_line(zw + 2 * y, set, v + 4 * y);
  __syncwarp();
#pragma unroll
  for (int z = 0; z < 4; ++z) get_line(yw + 10 * z, set, v + 4 * z);
  __syncwarp();
#pragma unroll
  for (int x = 0; x < 4; ++x) lift_fwd(v[x], v[x + 4], v[x + 8], v[x + 12]);
}

// The inverse: coefficients of the lane's y-plane in, values of its z-plane out.
template <typename S>
__device__ __forceinline__ void lift_inv_bricks(S* v, uint4* zw, uint4* yw, int set) {
#pragma unroll
  for (int x = 0; x < 4; ++x) lift_inv(v[x], v[x + 4], v[x + 8], v[x + 12]);
#pragma unroll
  for (int z = 0; z < 4; ++z) put_line(yw + 10 * z, set, v + 4 * z);
  __syncwarp();
#pragma unroll
  for (int y = 0; y < 4; ++y) get_line(zw + 2 * y, set, v + 4 * y);
  __syncwarp();
#pragma unroll
  for (int x = 0; x < 4; ++x) lift_inv(v[x], v[x + 4], v[x + 8], v[x + 12]);
#pragma unroll
  for (int y = 0; y < 4; ++y) lift_inv(v[4 * y], v[4 * y + 1], v[4 * y + 2], v[4 * y + 3]);
}

// n / d for an invariant d, by one high multiply (DivMagic).
__device__ __forceinline__ uint32_t div_by(uint32_t n, const DivMagic& D) {
  const uint32_t t = __umulhi(D.m, n);
  return (t + ((n - t) >> D.s1)) >> D.s2;
}

// Brick g of the job's box (x fastest): its coordinates.
__device__ __forceinline__ void brick_of(const BoxJob& J, int64_t g, int64_t* bx, int64_t* by, int64_t* bz) {
  if (J.nbox < (1ll << 32)) {  // 32-bit division by the box's invariant extents
    const uint32_t g32 = (uint32_t)g;
    const uint32_t r = div_by(g32, J.dv_bn0);
    const uint32_t z = div_by(r, J.dv_bn1);
    *bx = J.bl[0] + (int64_t)(g32 - r * (uint32_t)J.bn[0]);
    *by = J.bl[1] + (int64_t)(r - z * (uint32_t)J.bn[1]);
    *bz = J.bl[2] + (int64_t)z;
  } else {
    *bx = J.bl[0] + g % J.bn[0];
    const int64_t r = g / J.bn[0];
    *by = J.bl[1] + r % J.bn[1];
    *bz = J.bl[2] + r / J.bn[1];
  }
}

}  // namespace pcz
