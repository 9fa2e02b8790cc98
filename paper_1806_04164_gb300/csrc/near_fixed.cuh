// Near part of PIE_FP64 problems in fixed point on the integer pipe.
//
// GB300 does two FP64 fused multiply-adds per clock and SM, and the near part
// takes 48 per triangle pair: 24 clocks a pair on the pipe that also bounds the
// far part, against 5.8 clocks of memory traffic (128 B a pair).  The integer
// pipe multiplies 32 x 32 -> 64 bits and accumulates at 54 a clock and SM
// (measured).  With integers of two limbs, h 2^28 + l, a product takes three such
// multiply-adds in two sums, h h' and h l' + l h' (l l' is below 2^-60 of the
// largest product and left out), so a pair takes 2.7 clocks of it and leaves the
// FP64 pipe to the far part.
//
// A pair's moments are stored as integers of up to 58 bits times a power of two
// that the test row shares (set-up), the sources' coefficients become 56-bit
// integers times powers of two shared by a leaf box's sources when they are
// staged.  Real and imaginary parts have powers of their own, in moments and
// coefficients alike: at low frequency the imaginary (radiated) part of a moment
// is k h / 4 of the real one and less, and where the coefficients are real it
// alone makes the imaginary part of the product.  So every sum takes products of one
// part with one part: four where a complex product has two.
//
// Error: the sums are exact but for l l' and the last bit of x, so what remains is the
// rounding of the factors, to 2^-59 of the row's largest moment and 2^-57 of the
// stage's largest coefficient of their part (FP64 rounds every product and partial
// sum, to 2^-53 of itself).  In the norm of either part that is no more than
// FP64's; an entry far below its neighbours in the row or stage
// keeps as many digits fewer, as it adds as much less to their sum.
#pragma once
#include <cstdint>

#include "device.cuh"

namespace pie {

// Limbs: -2^27 <= l < 2^27, |h| <= 2^30 (moments) or 2^28 (coefficients).  A lane sums
// at most kFixedStage / 32 = 12 entries, 4 real products each, before the sums
// are taken out.  The row's exponents keep the sum of the moments' integers over
// those below 2^61 (2^33 in h), so |sum h h'| < 2^61 and |sum h l' + l h'| <
// 2^28 48 2^27 + 2^27 2^33 < 2^62.
constexpr int kLimb = 28;
constexpr int kFixedStage = 384;
constexpr int kMomentBits = 58, kCoefBits = 56, kLaneBits = 61;

// Exponents of one test row, [0] of the real and [1] of the imaginary parts: a
// moment is its integer times 2^e, with e = m0 for m0, m0 + delta for ms, mt for mt
// and mt + delta for mts, delta the leaf box's (about log2 of its edges,
// FixedNear::delta).  One delta for both pairs of groups lets the products a mts and
// beta mt, a ms and beta m0 share a sum (a takes the exponent of beta less delta).
struct alignas(16) FixedRow {
  int32_t m0[2], mt[2];
};
constexpr int32_t kFixedNan = 1 << 20;  // exponent of a row with a moment that is not finite

// Moments: planes of int4, [part][4][nnz]: plane g holds moments 2 g and 2 g + 1 of
// m0, mt(3), ms(3), mts as (h, l, h, l).
constexpr int kFixedPlanes = 4;

struct FixedNear {
  const int4* mom;       // [2][kFixedPlanes][nnz]
  const FixedRow* row;   // [T]
  const int32_t* delta;  // [nleaf]
};

__device__ __forceinline__ int exponent_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// v as an integer times 2^(f - 1075), rounded to nearest; f at least v's exponent field less 10.
__device__ __forceinline__ int2 fixed_encode(double v, int f) {
  const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
  const uint64_t m = (uint64_t(uint32_t(hi & 0xfffff) | (e ? 0x100000u : 0u)) << 32) | uint32_t(__double2loint(v));
  const int s = f - max(e, 1);
  const uint64_t r = s <= 0 ? m << -s : s > 54 ? 0 : (m + (uint64_t(1) << (s - 1))) >> s;
  const int64_t x = hi < 0 ? -int64_t(r) : int64_t(r);
  const int l = int(uint32_t(x) << (32 - kLimb)) >> (32 - kLimb);
  return make_int2(int((x - l) >> kLimb), l);
}

__device__ __forceinline__ double fixed_value(int h, int l) { return fma(double(h), double(1 << kLimb), double(l)); }

// (hi 2^32 + lo) 2^e to about an ulp: hi is rounded where it has more than 53 bits,
// then the sum (the conversions are four operations on the FP64 pipe, which the
// far part needs; scalbn only where the result leaves the normal range).
__device__ __forceinline__ double fixed_scale(int64_t hi, uint32_t lo, int e) {
  const double v = fma(double(hi), 4294967296.0, double(lo));
  const int f = exponent_field(v);
  if (f == 0 || f + e <= 0 || f + e >= 0x7ff) return scalbn(v, e);
  return __hiloint2double(__double2hiint(v) + e * (1 << 20), __double2loint(v));
}

// Moment q of entry e in row t of leaf box b, as a double.
__device__ __forceinline__ cd fixed_moment(const FixedNear& f, int64_t nnz, int q, int64_t e, int64_t t, int b) {
  const FixedRow r = f.row[t];
  if (r.m0[0] == kFixedNan) return mk<double>(nan(""), nan(""));
  const bool test = (q >= 1 && q <= 3) || q == 7, source = q >= 4;
  double v[2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const int4 m = f.mom[(p * kFixedPlanes + q / 2) * nnz + e];
    v[p] = scalbn(q % 2 ? fixed_value(m.z, m.w) : fixed_value(m.x, m.y),
                  (test ? r.mt[p] : r.m0[p]) + (source ? f.delta[b] : 0));
  }
  return mk<double>(v[0], v[1]);
}

}  // namespace pie
