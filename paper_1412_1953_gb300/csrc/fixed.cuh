// Sums of FP64 products on the integer pipes.
//
// This part issues a warp's FP64 instruction over 64 cycles of its quarter of an SM, a 32 x 32 ->
// 64-bit integer multiply-add over 4 and other integer operations over 2 (measured: 1.7, 32.6 and
// 66 lane operations per clock and SM).  A complex FP64 multiply-add is 4 FP64 instructions, 256
// cycles; below it is 12 integer multiply-adds and, for an operand not converted before, about 32
// integer operations, 48 and 64 cycles that overlap.
//
// A double x = +-m 2^(e - 1075) (m the 53-bit significand, e the biased exponent) becomes, for a
// common exponent E >= e, the integer nearest to +-16 m 2^(e - E) of at most 57 bits, that is x to
// within 2^(E - 1080): four bits more than a double of the largest magnitude keeps, so an operand
// that shares E with one up to 16 times as large is still exact to its last bit.  It is held as two
// limbs h 2^29 + l (|h| <= 2^28, |l| <= 2^28).  In a product (h h' 2^58 + (h l' + l h')
// 2^29 + l l') the last term, below 2^-56 of the largest product, is dropped; the sums of the others
// are exact in 64 bits for FX_TERMS complex terms, and are then rounded to a double once.  (Gram-Schmidt
// sums take 59 bits and FX_TERMS_59 terms: a quarter of the error at the same cost.)  What is
// dropped must have no mean, or a long sum that cancels keeps it, so low limbs lie about zero and
// conversions round without a preference.  (With low limbs of the operands' signs and cut conversions, a dot product of
// 1023^2 skewed, nearly cancelling terms was 1e-17 to 1e-16 |v| |w| off its 64-bit value, and 2e-19
// with FP64 multiply-adds.)
//
// An operand far below the one whose exponent it shares has fewer bits than its double, so a sum on a
// common exponent is good to the largest operands' scale, not to its own terms', where these are
// small.  Each kernel therefore looks for a term near the largest, and takes FP64 instructions for the chunk,
// tile or entry that has none: within 2^-FX_NEAR with 57 bits, 2^-6 with 59 (U_NEAR, C_NEAR), so that the
// roundings of FP64 multiply-adds of the same terms are no smaller.  That costs a few instructions a
// product; the stencils, with few products a value, lost to it what the integers gave and are FP64.
//
// Largest exponents outside FX_MIN..FX_MAX (nothing but zeros and subnormals, huge, infinite or
// NaN operands) take the FP64 instructions; fx_ok tells.
#pragma once
#include "common.cuh"

constexpr int FX_MIN = 600, FX_MAX = 1446;       // biased exponents; a product's scale stays normal
constexpr int FX_TERMS = 8;                      // complex terms between two roundings
constexpr int FX_TERMS_59 = 6;                   // the same for limbs of 59 bits

// How many powers of two below the largest operands' product a sum's own largest term may lie.
constexpr int FX_NEAR = 4;

__device__ __forceinline__ int fx_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ bool fx_ok(int E) { return (unsigned)(E - FX_MIN) <= (unsigned)(FX_MAX - FX_MIN); }

struct FxLimbs {
  int h, l;
};
// x, of exponent e, for the common exponent E >= e: the significand left-justified in 64 bits, its 57 bits
// from position 7 + E - e on rounded, split at 2^29 with l in [-2^28, 2^28), and the sign multiplied in (on
// the other integer pipe).  Ties, one in 2^d of the values that lose d bits, go away from zero, or
// towards it with down = 1: long sums alternate it by lane, so that ties leave no mean either.
// X = 2: 59 bits, split at 2^30.
template <int X = 0>
__device__ __forceinline__ FxLimbs fx_limbs(double x, int e, int E, int down = 0) {
  static_assert(X == 0 || X == 2, "57 or 59 bits");
  constexpr int S = 29 + X / 2;
  const int hi = __double2hiint(x), s = (hi >> 31) | 1;
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned a1 = __funnelshift_l(lo, ((unsigned)hi & 0xfffffu) | 0x100000u, 11), a0 = lo << 11;
  unsigned long long r;                                  // with a bit more, for rounding; 0 for E - e > 57
  asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(((unsigned long long)a1 << 32 | a0) - down), "r"(E + 6 - X - e));
  r += (1u << S) + 1;
  const int h = (int)(r >> (S + 1)), l = (int)(((unsigned)r & ((2u << S) - 1)) >> 1) - (1 << (S - 1));
  return FxLimbs{h * s, l * s};
}
__device__ __forceinline__ FxLimbs fx_neg(FxLimbs a) { return FxLimbs{-a.h, -a.l}; }

// The two exact partial sums of sum a b.
struct FxSum {
  long long hh, mid;
};
__device__ __forceinline__ void fx_mac(FxSum& s, FxLimbs a, FxLimbs b) {
  s.hh += (long long)a.h * b.h;
  s.mid += (long long)a.h * b.l;
  s.mid += (long long)a.l * b.h;
}
// Carry the middle sum into the upper one, so that FX_TERMS more terms fit (the upper sum itself
// holds 4 FX_TERMS terms, of 59 bits 2 FX_TERMS_59).
template <int X = 0>
__device__ __forceinline__ void fx_carry(FxSum& s) {
  constexpr int S = 29 + X / 2;
  s.hh += (s.mid + (1LL << (S - 1))) >> S;
  s.mid = 0;
}
// (re, im) += a b for complex a = (ax, ay), b = (bx, by).
__device__ __forceinline__ void fx_cmac(FxSum& re, FxSum& im, int4 a, int4 b) {
  const FxLimbs ax{a.x, a.y}, ay{a.z, a.w}, bx{b.x, b.y}, by{b.z, b.w};
  fx_mac(re, ax, bx);
  fx_mac(re, fx_neg(ay), by);
  fx_mac(im, ax, by);
  fx_mac(im, ay, bx);
}
__device__ __forceinline__ int fx_exp(cplx z) { return max(fx_exp(z.x), fx_exp(z.y)); }
template <int X = 0>
__device__ __forceinline__ int4 fx_limbs(cplx z, int E, int down = 0) {
  const FxLimbs x = fx_limbs<X>(z.x, fx_exp(z.x), E, down), y = fx_limbs<X>(z.y, fx_exp(z.y), E, down);
  return make_int4(x.h, x.l, y.h, y.l);
}
// acc + the sum of products with exponents that add up to E2, rounded; the sum is cleared.
template <int X = 0>
__device__ __forceinline__ double fx_flush(FxSum& s, int E2, double acc) {
  constexpr int S = 29 + X / 2;
  const long long t = s.hh + ((s.mid + (1LL << (S - 1))) >> S);
  s.hh = s.mid = 0;
  return fma((double)t, __hiloint2double((E2 - 2100 - X + 1023) << 20, 0), acc);
}
