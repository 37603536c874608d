// Block fixed-point arithmetic on the integer pipe, for the double-precision
// element kernels.
//
// Why: GB300 issues 2 FP64 operations per SM and clock, one warp instruction
// per 64 clocks of an SM sub-partition, while the same sub-partition issues a
// 32 x 32 + 64 bit multiply-add (IMAD.WIDE) every 2 clocks and 32-bit integer
// operations every 1 to 2 clocks (measured: 1.9 DFMA, 58 IMAD.WIDE, 110 IADD
// lane operations per SM and clock; the pipes run side by side). A
// double-precision product sum written as integer multiply-adds of 61-bit
// numbers therefore costs a tenth of its FP64 form and carries more bits.
//
// A quantity is a small group of numbers that share one exponent: a component
// of the nodal velocities, an axis of the cofactor vectors, a row of the
// gradient. Its members are 64-bit integers X with |X| < 2^61, real value
// X 2^(e - 61). Products use two 32-bit limbs, X = h 2^32 + l with l signed
// (one instruction to make: h takes the carry of l's sign bit):
//   X Y / 2^64 = h h' + (h l' + l h') / 2^32 + l l' / 2^64,
// three multiply-adds per product, the last term (a quarter unit, zero mean)
// dropped; sums of products accumulate in the two 64-bit accumulators and are
// combined once, by a fourth multiply-add. An absolute error of about one
// unit, 2^-58 of the operands' bound, takes the place of the 2^-53 relative
// error of each rounded double operation. Groups that may be much smaller
// than their bound are normalised: shifted left until the largest member is in
// [2^60, 2^61). Terms of different exponents are shifted right to the largest
// one before they are added.
#pragma once

#include <cstdint>
#include <cstring>

#include "fastmath.cuh"

namespace nsrhs {
namespace fixed {

// ---- bits of doubles, and the integer instructions used ----

// What the arithmetic relies on: shift counts that are not negative, no bits lost
// at the top. A host build that defines it (tests/fixedpoint) counts violations.
#if !defined(NSRHS_FIXED_EXPECT)
#define NSRHS_FIXED_EXPECT(ok)
#endif

#if defined(__CUDA_ARCH__)
__device__ __forceinline__ int32_t hi_word(double x) { return __double2hiint(x); }
__device__ __forceinline__ uint32_t lo_word(double x) { return (uint32_t)__double2loint(x); }
__device__ __forceinline__ double make_double(uint64_t b) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ int clz32(uint32_t x) { return __clz((int)x); }
__device__ __forceinline__ int imax(int a, int b) { return max(a, b); }
__device__ __forceinline__ uint32_t umin(uint32_t a, uint32_t b) { return min(a, b); }
// Whether x holds in any thread of the warp that is here: a branch that the warp takes together.
__device__ __forceinline__ bool any_lane(bool x) { return __any_sync(__activemask(), x) != 0; }
// a b + c, one instruction.
__device__ __forceinline__ int64_t mad_wide(int32_t a, int32_t b, int64_t c) {
  int64_t d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
// x 2^-k (floor), x 2^k mod 2^64, for any k >= 0: the instructions clamp.
__device__ __forceinline__ int64_t shr(int64_t x, int k) {
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(k));
  return r;
}
__device__ __forceinline__ uint64_t shru(uint64_t x, int k) {
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(k));
  return r;
}
__device__ __forceinline__ int64_t shl(int64_t x, int k) {
  int64_t r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(k));
  return r;
}
#else
inline uint64_t bits_of(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
inline int32_t hi_word(double x) { return (int32_t)(bits_of(x) >> 32); }
inline uint32_t lo_word(double x) { return (uint32_t)bits_of(x); }
inline double make_double(uint64_t b) { double x; std::memcpy(&x, &b, 8); return x; }
inline int clz32(uint32_t x) { return x ? __builtin_clz(x) : 32; }
inline int imax(int a, int b) { return a > b ? a : b; }
inline uint32_t umin(uint32_t a, uint32_t b) { return a < b ? a : b; }
inline bool any_lane(bool x) { return x; }
inline int64_t mad_wide(int32_t a, int32_t b, int64_t c) {
  int64_t d;
  const bool over = __builtin_add_overflow((int64_t)a * b, c, &d);
  NSRHS_FIXED_EXPECT(!over);
  (void)over;
  return d;
}
// A negative count is a large one, as for the instructions.
inline int64_t shr(int64_t x, int k) {
  NSRHS_FIXED_EXPECT(k >= 0);
  return x >> ((uint32_t)k < 63u ? k : 63);
}
inline uint64_t shru(uint64_t x, int k) {
  NSRHS_FIXED_EXPECT(k >= 0);
  return (uint32_t)k > 63u ? 0 : x >> k;
}
inline int64_t shl(int64_t x, int k) {
  const int64_t r = (uint32_t)k > 63u ? 0 : (int64_t)((uint64_t)x << k);
  NSRHS_FIXED_EXPECT(k >= 0 && shr(r, k) == x);
  return r;
}
#endif
__device__ __forceinline__ int32_t hi32(int64_t x) { return (int32_t)(x >> 32); }

// x 2^-k rounded (ties up), k >= 0, |x| < 2^62.
__device__ __forceinline__ int64_t shr_round(int64_t x, int k) { return (shr(x * 2, k) + 1) >> 1; }

// ---- conversions ----

// Exponents of groups that hold only zeros: far below every other one, so
// that such a group never decides an alignment.
constexpr int kZeroExp = -4000;

// Exponent (E - 1022 of group_exp) of a group of zeros.
constexpr int kRestExp = 128 - 1022;

__device__ __forceinline__ int32_t hi_abs(double x) { return hi_word(x) & 0x7fffffff; }

// Biased exponent of a group from the largest |high word| of its members.
// Members too far below the largest become 0; a group of zeros gets an
// exponent so small that every member shifts to 0.
__device__ __forceinline__ int group_exp(int32_t mh) { return imax(mh >> 20, 128); }

// Whether a group's largest member is 0 or within 2^-100 .. 2^100; infinities
// and NaN are not.
__device__ __forceinline__ bool in_range(int32_t mh) {
  return mh == 0 || (uint32_t)((mh >> 20) - 923) <= 200u;
}

// x as a fixed-point member of the group with biased exponent E:
// |result| < 2^B, real value = result 2^(E - 1022 - B). 53 <= B <= 63.
template <int B>
__device__ __forceinline__ int64_t to_fixed(double x, int E) {
  const int32_t hi = hi_word(x);
  const uint64_t m =
      ((uint64_t)(uint32_t)((hi & 0xfffff) | 0x100000) << 32 | lo_word(x)) << (B - 53);
  const int64_t a = (int64_t)shru(m, E - ((hi & 0x7fffffff) >> 20));
  return hi < 0 ? -a : a;
}

// Exponent of a positive normal double, and its mantissa in [2^59, 2^60):
// x = result 2^(e - 60).
__device__ __forceinline__ int scalar_exp(double x) { return ((hi_word(x) >> 20) & 0x7ff) - 1022; }
__device__ __forceinline__ int64_t scalar_fixed(double x, int& e) {
  const int32_t hi = hi_word(x);
  e = ((hi >> 20) & 0x7ff) - 1022;
  return (int64_t)(((uint64_t)(uint32_t)((hi & 0xfffff) | 0x100000) << 32 | lo_word(x)) << 7);
}

// X 2^(e - 60) as a double, rounded to nearest (ties up), |X| < 2^63.
__device__ __forceinline__ double to_double(int64_t x, int e) {
  const uint64_t a = (uint64_t)(x < 0 ? -x : x);
  uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a;
  int k = e + 1025;
  if (ah == 0u) {  // up by 31: the leading bit stays below 2^63
    ah = al >> 1;
    al <<= 31;
    k -= 31;
  }
  const int n = clz32(ah);  // n >= 1 (32 for x = 1, where v is still right)
  NSRHS_FIXED_EXPECT(x == 0 || (k - n >= 0 && k - n < 2046));
  // leading bit to 2^62, then the 53 leading bits rounded
  const uint64_t v = ((uint64_t)shl((int64_t)((uint64_t)ah << 32 | al), n - 1) + 512u) >> 10;
  const uint32_t hi = (uint32_t)(v >> 32) + ((uint32_t)(k - n) << 20);
  const uint32_t h = x == 0 ? 0u : hi | ((uint32_t)(x >> 32) & 0x80000000u);
  return make_double((uint64_t)h << 32 | (uint32_t)v);
}

// ---- products ----

struct Limb {
  int32_t h, l;
};
__device__ __forceinline__ constexpr Limb limb(int64_t x) {
  return {(int32_t)((uint32_t)(x >> 32) + ((uint32_t)x >> 31)), (int32_t)(uint32_t)x};
}
__device__ __forceinline__ int64_t top(const Limb& a) { return a.h < 0 ? -(int64_t)a.h : a.h; }
__device__ __forceinline__ int64_t whole(const Limb& a) {
  return (int64_t)((uint64_t)(uint32_t)(a.h - (int32_t)((uint32_t)a.l >> 31)) << 32 | (uint32_t)a.l);
}

// Sum of products of limbs, at most 3 of |X|, |Y| < 2^61; fin() = (sum) / 2^64.
struct Acc {
  int64_t H, M;
};
__device__ __forceinline__ Acc acc_start(int64_t h = 0) { return {h, 1ll << 31}; }
__device__ __forceinline__ void mac(Acc& s, const Limb& a, const Limb& b) {
  s.H = mad_wide(a.h, b.h, s.H);
  s.M = mad_wide(a.h, b.l, s.M);
  s.M = mad_wide(a.l, b.h, s.M);
}
__device__ __forceinline__ int64_t fin(const Acc& s) { return s.H + hi32(s.M); }
__device__ __forceinline__ int64_t mul(const Limb& a, const Limb& b) {
  Acc s = acc_start();
  mac(s, a, b);
  return fin(s);
}
// 8 a b / 2^64, |a| <= 2^60, |b| <= 2^61: keeps the scale of b. The factor
// is split over both high limbs: a.h may be 2^28 and b.h 2^29 (a mantissa of
// ones rounds up to the next power of two).
__device__ __forceinline__ int64_t mul8(const Limb& a, const Limb& b) {
  NSRHS_FIXED_EXPECT(top(a) <= 1 << 28 && top(b) <= 1 << 29);
  int64_t M = mad_wide(a.h, b.l, 1ll << 31);
  M = mad_wide(a.l, b.h, M);
  return mad_wide(hi32(M), 8, mad_wide(a.h * 4, b.h * 2, 0));
}
// a0 b0 + a1 b1 + a2 b2
__device__ __forceinline__ int64_t dot3(const Limb& a0, const Limb& b0, const Limb& a1,
                                        const Limb& b1, const Limb& a2, const Limb& b2,
                                        int64_t h = 0) {
  Acc s = acc_start(h);
  mac(s, a0, b0);
  mac(s, a1, b1);
  mac(s, a2, b2);
  return fin(s);
}
// The same times 2^S and to the unit (S more bits): |a| <= 2^61 for S = 1,
// 2^60 for S = 2, 3; |b| <= 2^61.
template <int S>
__device__ __forceinline__ Acc accx_start(int64_t h = 0) { return {h, 1ll << (31 - S)}; }
template <int S>
__device__ __forceinline__ void macx(Acc& s, const Limb& a, const Limb& b) {
  NSRHS_FIXED_EXPECT(top(a) < 1 << (S == 1 ? 30 : 29) && top(b) < 1ll << (S == 3 ? 30 : 31));
  s.H = mad_wide(a.h * (S == 1 ? 2 : 4), b.h * (S == 3 ? 2 : 1), s.H);
  s.M = mad_wide(a.h, b.l, s.M);
  s.M = mad_wide(a.l, b.h, s.M);
}
template <int S>
__device__ __forceinline__ int64_t finx(const Acc& s) { return s.H + (s.M >> (32 - S)); }
template <int S>
__device__ __forceinline__ int64_t mulx(const Limb& a, const Limb& b) {
  Acc s = accx_start<S>();
  macx<S>(s, a, b);
  return finx<S>(s);
}
template <int S>
__device__ __forceinline__ int64_t dot3x(const Limb& a0, const Limb& b0, const Limb& a1,
                                         const Limb& b1, const Limb& a2, const Limb& b2) {
  Acc s = accx_start<S>();
  macx<S>(s, a0, b0);
  macx<S>(s, a1, b1);
  macx<S>(s, a2, b2);
  return finx<S>(s);
}
// x x summed over three members
__device__ __forceinline__ int64_t square3(const Limb& a, const Limb& b, const Limb& c) {
  int64_t H = mad_wide(a.h, a.h, 0), M = 1ll << 30;
  H = mad_wide(b.h, b.h, H);
  H = mad_wide(c.h, c.h, H);
  M = mad_wide(a.h, a.l, M);
  M = mad_wide(b.h, b.l, M);
  M = mad_wide(c.h, c.l, M);
  return mad_wide(hi32(M), 2, H);
}

// ---- normalisation ----

__device__ __forceinline__ uint32_t mag(int64_t x) {
  const int32_t h = hi32(x);
  return (uint32_t)(h ^ (h >> 31));
}
// Left shift (>= 0 if all members are below 2^61) that brings the largest
// member, by the OR of the members' mag(), to [2^60, 2^61); at most 29:
// members below 2^32 keep their absolute precision of one unit.
__device__ __forceinline__ int norm_shift(uint32_t m) { return clz32(m) - 3; }

// To [2^59, 2^60), over all 64 bits, for differences of doubles, which are
// exact however small they are; -1 if all members are 0.
__device__ __forceinline__ int norm_shift64(int64_t a, int64_t b, int64_t c) {
  const uint64_t o = (uint64_t)((a ^ (a >> 63)) | (b ^ (b >> 63)) | (c ^ (c >> 63)));
  const uint32_t oh = (uint32_t)(o >> 32), ol = (uint32_t)o;
  const int n = oh ? clz32(oh) : 32 + clz32(ol);
  return (a | b | c) == 0 ? -1 : n - 4;
}

}  // namespace fixed
}  // namespace nsrhs
