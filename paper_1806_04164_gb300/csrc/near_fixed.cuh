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
// staged.  Sums are exact: the error is that of the two roundings, 2^-59 and
// 2^-57 of the largest factors, where FP64 rounds every product and partial sum
// (24,576 triangles, against 64-bit sums: 1.4e-15 of the product, 1.6e-15 with
// FP64 multiply-adds).
#pragma once
#include <cstdint>

#include "device.cuh"

namespace pie {

// Limbs: -2^27 <= l < 2^27, |h| <= 2^30 (moments) or 2^28 (coefficients).  A lane sums
// at most kFixedStage / 32 = 12 entries, 8 real products each, before the sums
// are taken out.  The row's exponents keep the sum of the moments' integers over
// those below 2^61 (2^33 in h), so |sum h h'| < 2^61 and |sum h l' + l h'| <
// 2^28 96 2^27 + 2^27 2^33 < 2^62.
constexpr int kLimb = 28;
constexpr int kFixedStage = 384;
constexpr int kMomentBits = 58, kCoefBits = 56, kLaneBits = 61;

// Exponents of one test row: a moment is its integer times 2^e, with e = m0 for
// m0, m0 + delta for ms, mt for mt and mt + delta for mts, delta the leaf box's
// (about log2 of its edges, FixedNear::delta).  One delta for both pairs of groups lets
// the products a mts and beta mt, a ms and beta m0 share a sum (a takes the
// exponent of beta less delta).
struct FixedRow {
  int32_t m0, mt;
};
constexpr int32_t kFixedNan = 1 << 20;  // exponent of a row with a moment that is not finite

struct FixedNear {
  const int4* mom;       // [8][nnz] (re h, re l, im h, im l)
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

// (hi 2^32 + lo) 2^e, rounded once (the conversions are four operations on the FP64
// pipe, which the far part needs; scalbn only where the result leaves the
// normal range).
__device__ __forceinline__ double fixed_scale(int64_t hi, uint32_t lo, int e) {
  const double v = fma(double(hi), 4294967296.0, double(lo));
  const int f = exponent_field(v);
  if (f == 0 || f + e <= 0 || f + e >= 0x7ff) return scalbn(v, e);
  return __hiloint2double(__double2hiint(v) + e * (1 << 20), __double2loint(v));
}

// Moment q of entry e in row t of leaf box b, as a double.
__device__ __forceinline__ cd fixed_moment(const FixedNear& f, int64_t nnz, int q, int64_t e, int64_t t, int b) {
  const int4 m = f.mom[q * nnz + e];
  const FixedRow r = f.row[t];
  const bool test = (q >= 1 && q <= 3) || q == 7, source = q >= 4;
  const int x = (test ? r.mt : r.m0) + (source ? f.delta[b] : 0);
  if (r.m0 == kFixedNan) return mk<double>(nan(""), nan(""));
  return mk<double>(scalbn(fixed_value(m.x, m.y), x), scalbn(fixed_value(m.z, m.w), x));
}

}  // namespace pie
