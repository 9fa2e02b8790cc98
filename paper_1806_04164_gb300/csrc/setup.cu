// Operator set-up on the device, all in FP64 (Sections 2-3):
//  - near pair moments of g over triangle pairs in neighbouring leaf boxes,
//    with closed-form static inner integrals for near-singular pairs (rule
//    averaged over both orders of the pair);
//  - leaf radiation tables (Pi, M) at the leaf wavenumber kappa_L;
//  - translation operators of Eq. (5) per level and offset;
//  - interpolation filter (degree rescale) and phases.
#include <cstring>
#include <cmath>
#include <type_traits>

#include "near_fixed.cuh"

namespace pie {

constexpr double kFourPi = 4.0 * kPi;
constexpr int kMaxTau = 30;

// ------------------------------------------------------------ pair moments
//
// Both kernels below bind on the FP64 pipe (two fused multiply-adds per clock
// and SM), so they are written for few double operations per point pair.  The
// 7-point rule on a triangle is its centroid c and two orbits c + s_o v_k
// (v_k = vertex k - c, s_o = 1 - 3 a_o, weights w_o), so sums over its points
// need sum_o w_o g and sum_o w_o s_o g per corner only.  The stored centroid's
// rounding e = sum_k v_k / 3 is added to the first moments at the end.
// e^{ikR}/R needs no sincos: cos(kR) and sin(kR)/R are power series in (kR)^2,
// NT terms of each.

struct Rule7 {
  double w0, w[2], s[2], ws[2];  // ws = w s
};

__device__ __forceinline__ Rule7 load_rule7(const double* __restrict__ r) {
  const double s0 = 1.0 - 3.0 * r[5], s1 = 1.0 - 3.0 * r[17];
  return Rule7{r[3], {r[7], r[19]}, {s0, s1}, {r[7] * s0, r[19] * s1}};
}

// Coefficients in R^2 of cos(kR), sin(kR)/(kR) and 2 (1 - cos kR)/(kR)^2.
constexpr int kNearTerms = 11;
struct NearSeries {
  double c[kNearTerms], s[kNearTerms], r[kNearTerms];
};

static NearSeries near_series(double k) {
  NearSeries t;
  double* v[3] = {t.c, t.s, t.r};
  for (int N = 0; N < 3; ++N) {
    double a = 1.0;
    for (int n = 0; n < kNearTerms; ++n) {
      if (n > 0) a *= -k * k / double((2 * n + N) * (2 * n + N - 1));
      v[N][n] = a;
    }
  }
  return t;
}

// The first NT terms by Horner.
template <int NT>
__device__ __forceinline__ double even_series(const double* c, double z) {
  double v = c[NT - 1];
#pragma unroll
  for (int n = NT - 2; n >= 0; --n) v = fma(v, z, c[n]);
  return v;
}

// ln(a/b), a, b > 0 (normal): a is scaled by the power of two that brings a/b
// into [2/3, 3/2], then ln = 2 atanh(t), t = (a - b)/(a + b), |t| <= 0.2, by its
// Taylor series (11 terms: t^24/23 < 1e-17): one division for the ratio and the
// logarithm together (25 double operations; log(a / b) took 41).
__device__ __forceinline__ double log_ratio(double a, double b) {
  const int ha = __double2hiint(a);
  const int q = (ha - __double2hiint(b) + (1 << 19)) >> 20;
  const double as = __hiloint2double(ha - (q << 20), __double2loint(a));
  const double t = (as - b) / (as + b), z = t * t;
  double p = 1.0 / 23;
#pragma unroll
  for (int n = 10; n >= 1; --n) p = fma(p, z, 1.0 / (2 * n + 1));
  const double t2 = t + t, qd = double(q);
  // ln 2 to 1e-33 as a sum of two doubles
  return fma(qd, 0.69314718055994530942, fma(qd, 2.3190468138462996e-17, fma(t2 * z, p, t2)));
}

struct Moments {
  double m0r, m0i, mtr[3], mti[3], msr[3], msi[3], mtsr, mtsi;
};

// One outer point's share at weight w and weighted test offset wu = w (r - c_t):
// K = sum_j w_j g, K1 = sum_j w_j u_j g.
__device__ __forceinline__ void add_point(Moments& o, double w, const double (&wu)[3], double Kr, double Ki,
                                          const double (&K1r)[3], const double (&K1i)[3]) {
  o.m0r = fma(w, Kr, o.m0r);
  o.m0i = fma(w, Ki, o.m0i);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    o.mtr[d] = fma(wu[d], Kr, o.mtr[d]);
    o.mti[d] = fma(wu[d], Ki, o.mti[d]);
    o.msr[d] = fma(w, K1r[d], o.msr[d]);
    o.msi[d] = fma(w, K1i[d], o.msi[d]);
    o.mtsr = fma(wu[d], K1r[d], o.mtsr);
    o.mtsi = fma(wu[d], K1i[d], o.mtsi);
  }
}

// The centroid rounding e of the source triangle in the first moments.
__device__ __forceinline__ void add_centroid(Moments& o, const double (&e)[3]) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    o.msr[d] = fma(e[d], o.m0r, o.msr[d]);
    o.msi[d] = fma(e[d], o.m0i, o.msi[d]);
    o.mtsr = fma(e[d], o.mtr[d], o.mtsr);
    o.mtsi = fma(e[d], o.mti[d], o.mtsi);
  }
}

// The row's test points for the regular pairs: r, w, w (r - c_t) of the 7-point rule.
struct TestPoint {
  double r[3], w, wu[3];
};

// Regular pair by the 7 x 7 rule.  NT = 0: sincos (boxes large in wavelengths).
// The imaginary parts are summed without their factor k.
template <int NT>
__device__ __forceinline__ void moments_regular(const TestPoint* __restrict__ tp, const double* __restrict__ vs,
                                                const double* __restrict__ cs, double As, double k,
                                                const NearSeries& G, const Rule7& R, Moments& o) {
  double v[3][3], e[3];
  const double c[3] = {cs[0], cs[1], cs[2]};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q][d] = vs[3 * q + d] - c[d];
    e[d] = (v[0][d] + v[1][d] + v[2][d]) / 3.0;
  }
  o = Moments{};
  // e^{ikR}/R = cos(kR)/R + i k sin(kR)/(kR)
  auto green = [&](double q2, double& gr, double& gi) {
    const double ri = rsqrt(q2);
    if constexpr (NT == 0) {
      double sn, cn;
      sincos(k * (q2 * ri), &sn, &cn);
      gr = ri * cn;
      gi = ri * sn;
    } else {
      gr = ri * even_series<NT>(G.c, q2);
      gi = even_series<NT>(G.s, q2);
    }
  };
#pragma unroll 1
  for (int i = 0; i < 7; ++i) {
    const double x[3] = {tp[i].r[0] - c[0], tp[i].r[1] - c[1], tp[i].r[2] - c[2]};
    double Kr, Ki, K1r[3] = {0, 0, 0}, K1i[3] = {0, 0, 0};
    green(x[0] * x[0] + x[1] * x[1] + x[2] * x[2], Kr, Ki);
    Kr *= R.w0;
    Ki *= R.w0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      double hr = 0, hi = 0;
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const double dx = fma(-R.s[p], v[q][0], x[0]), dy = fma(-R.s[p], v[q][1], x[1]),
                     dz = fma(-R.s[p], v[q][2], x[2]);
        double gr, gi;
        green(dx * dx + dy * dy + dz * dz, gr, gi);
        Kr = fma(R.w[p], gr, Kr);
        Ki = fma(R.w[p], gi, Ki);
        hr = fma(R.ws[p], gr, hr);
        hi = fma(R.ws[p], gi, hi);
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        K1r[d] = fma(v[q][d], hr, K1r[d]);
        K1i[d] = fma(v[q][d], hi, K1i[d]);
      }
    }
    const double wu[3] = {tp[i].wu[0], tp[i].wu[1], tp[i].wu[2]};
    add_point(o, tp[i].w, wu, Kr, Ki, K1r, K1i);
  }
  add_centroid(o, e);
  const double fr = As * (1.0 / kFourPi), fi = NT == 0 ? fr : fr * k;
  o.m0r *= fr;
  o.m0i *= fi;
  o.mtsr *= fr;
  o.mtsi *= fi;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    o.mtr[d] *= fr;
    o.mti[d] *= fi;
    o.msr[d] *= fr;
    o.msi[d] *= fi;
  }
}

// Near-singular pair, test triangle t, source s: outer 8 x 8 collapsed Gauss
// rule (points lane, lane + NL, ...: NL lanes share the pair), the static
// inner integrals int 1/R and int (r'-r)/R over the flat source triangle in
// closed form (Wilton et al. 1984; Graglia 1993), the rest
// (e^{ikR} - 1)/R by the 7-point rule.  With unit normal n, height
// d = n.(r - v0), per edge a->b: tangent s, outward normal m = s x n,
// l+ = (b-r).s, l- = (a-r).s, P0 = (a-r).m, R0^2 = P0^2 + d^2,
// f = ln((R+ + l+)/(R- + l-)):
//   I1 = sum P0 f - |d| W,  Ir = 1/2 sum m [R0^2 f + l+R+ - l-R-] - d n I1,
// W the solid angle of the triangle, one arctangent by van Oosterom and
// Strackee (1983) instead of two per edge.  Adds to o.
template <int NT, int NL>
__device__ __forceinline__ void moments_singular(const double* __restrict__ vt, const double* __restrict__ ct,
                                                 double At, const double* __restrict__ vs,
                                                 const double* __restrict__ cs, double As, double k,
                                                 const NearSeries& G, const Rule7& R7,
                                                 const double* __restrict__ rule64, int lane, Moments& o) {
  double v[3][3], s[3][3], m[3][3], n[3], el[3], e[3];
  const double c[3] = {cs[0], cs[1], cs[2]};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q][d] = vs[3 * q + d] - c[d];
    e[d] = (v[0][d] + v[1][d] + v[2][d]) / 3.0;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
#pragma unroll
    for (int d = 0; d < 3; ++d) s[q][d] = vs[3 * ((q + 1) % 3) + d] - vs[3 * q + d];
    el[q] = sqrt(s[q][0] * s[q][0] + s[q][1] * s[q][1] + s[q][2] * s[q][2]);
  }
  // the normal from s_0 x s_1 = e1 x (e2 - e1) = e1 x e2
  n[0] = s[0][1] * s[1][2] - s[0][2] * s[1][1];
  n[1] = s[0][2] * s[1][0] - s[0][0] * s[1][2];
  n[2] = s[0][0] * s[1][1] - s[0][1] * s[1][0];
  const double nn = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
#pragma unroll
  for (int d = 0; d < 3; ++d) n[d] /= nn;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
#pragma unroll
    for (int d = 0; d < 3; ++d) s[q][d] /= el[q];
    m[q][0] = s[q][1] * n[2] - s[q][2] * n[1];
    m[q][1] = s[q][2] * n[0] - s[q][0] * n[2];
    m[q][2] = s[q][0] * n[1] - s[q][1] * n[0];
  }
  const double fr = -0.5 * k * k * As, fi = k * As;
  Moments a{};
#pragma unroll 1
  for (int i = lane; i < 64; i += NL) {
    double wu[3], x[3];
    const double wi = rule64[4 * i + 3] * (At * (1.0 / kFourPi));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double r = rule64[4 * i] * vt[d] + rule64[4 * i + 1] * vt[3 + d] + rule64[4 * i + 2] * vt[6 + d];
      wu[d] = wi * (r - ct[d]);
      x[d] = r - c[d];
    }
    // static part
    double p[3][3], Rv[3];  // r - vertex, its length
#pragma unroll
    for (int q = 0; q < 3; ++q) {
#pragma unroll
      for (int d = 0; d < 3; ++d) p[q][d] = x[d] - v[q][d];
      Rv[q] = sqrt(p[q][0] * p[q][0] + p[q][1] * p[q][1] + p[q][2] * p[q][2]);
    }
    const double h = n[0] * p[0][0] + n[1] * p[0][1] + n[2] * p[0][2], ah = fabs(h);
    double I1 = 0, Ip[3] = {0, 0, 0}, den = Rv[0] * Rv[1] * Rv[2];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int q1 = (q + 1) % 3;
      const double Rm = Rv[q], Rp = Rv[q1];
      const double lm = -(p[q][0] * s[q][0] + p[q][1] * s[q][1] + p[q][2] * s[q][2]), lp = lm + el[q];
      const double P0 = -(p[q][0] * m[q][0] + p[q][1] * m[q][1] + p[q][2] * m[q][2]);
      const double R02 = P0 * P0 + h * h;
      const bool right = lm >= 0, left = lp <= 0;
      const double up = left ? Rm - lm : right ? Rp + lp : (Rp + lp) * (Rm - lm);
      const double dn = left ? Rp - lp : right ? Rm + lm : R02;
      const double f = R02 > 1e-24 * el[q] * el[q] ? log_ratio(up, dn) : 0.0;
      I1 = fma(P0, f, I1);
      const double w = 0.5 * (R02 * f + lp * Rp - lm * Rm);
#pragma unroll
      for (int d = 0; d < 3; ++d) Ip[d] = fma(w, m[q][d], Ip[d]);
      den = fma(p[q][0] * p[q1][0] + p[q][1] * p[q1][1] + p[q][2] * p[q1][2], Rv[(q + 2) % 3], den);
    }
    I1 -= 2.0 * ah * atan2(ah * nn, den);
    // the rest, (e^{ikR} - 1)/R = -k^2/2 R [2 (1 - cos kR)/(kR)^2] + i k sin(kR)/(kR)
    double gr, gi, Kr, Ki, K1r[3] = {0, 0, 0}, K1i[3] = {0, 0, 0};
    auto rem = [&](double q2) {
      gr = q2 * rsqrt(q2 + 1e-300) * even_series<NT>(G.r, q2);  // R = 0 at a shared point
      gi = even_series<NT>(G.s, q2);
    };
    rem(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
    Kr = R7.w0 * gr;
    Ki = R7.w0 * gi;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      double hr = 0, hi = 0;
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const double dx = fma(-R7.s[b], v[q][0], x[0]), dy = fma(-R7.s[b], v[q][1], x[1]),
                     dz = fma(-R7.s[b], v[q][2], x[2]);
        rem(dx * dx + dy * dy + dz * dz);
        Kr = fma(R7.w[b], gr, Kr);
        Ki = fma(R7.w[b], gi, Ki);
        hr = fma(R7.ws[b], gr, hr);
        hi = fma(R7.ws[b], gi, hi);
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        K1r[d] = fma(v[q][d], hr, K1r[d]);
        K1i[d] = fma(v[q][d], hi, K1i[d]);
      }
    }
    Kr = fma(fr, Kr, I1);
    Ki *= fi;
    // (only the rule's imaginary part takes the centroid's rounding: the
    // static part is exact about c and dwarfs the real remainder)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      K1r[d] = fma(fr, K1r[d], fma(fma(-h, n[d], x[d]), I1, Ip[d]));
      K1i[d] = fma(e[d], Ki, fi * K1i[d]);
    }
    add_point(a, wi, wu, Kr, Ki, K1r, K1i);
  }
  o.m0r += a.m0r;
  o.m0i += a.m0i;
  o.mtsr += a.mtsr;
  o.mtsi += a.mtsi;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    o.mtr[d] += a.mtr[d];
    o.mti[d] += a.mti[d];
    o.msr[d] += a.msr[d];
    o.msi[d] += a.msi[d];
  }
}

// Near-singular test: ((dx*dx + dy*dy) + dz*dz) < 2.25 max(h_t^2, h_s^2), in
// round-to-nearest double with no contraction.
__device__ __forceinline__ bool near_singular(const double* ct, const double* cs, double h2t, double h2s) {
  double dx = __dsub_rn(ct[0], cs[0]), dy = __dsub_rn(ct[1], cs[1]), dz = __dsub_rn(ct[2], cs[2]);
  double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  return d2 < __dmul_rn(2.25, fmax(h2t, h2s));
}

// Near-part set-up in three passes, so that the few expensive near-singular
// pairs do not stall the warps computing the regular ones:
//  1. k_count_singular: count the near-singular pairs with t < s;
//  2. k_near_regular: regular pairs by the 7 x 7 rule; near-singular pairs
//     are appended to a list;
//  3. k_near_singular: kSingLanes lanes per listed pair compute the rule in
//     both orders and average; then the pairs (t, t).
// Every unordered pair is computed once and written as (t,s) and (s,t) (mt and
// ms swapped), which keeps Z^T = Z: a row lists its sources in ascending order,
// so the pairs t < s of a row are its tail past t's own position, and lanes
// walk that tail flat, as the product kernel does.
struct NearGeom {
  const int32_t* leaf_of;
  const int32_t* leaf_start;
  const int32_t* near_ptr;
  const int32_t* near_idx;
  const int32_t* near_off;
  const int64_t* row_ptr;
  const double* vert;
  const double* cent;
  const double* area;
  const double* h2;
};

// Position of source s within the row of a triangle of box b (-1: not near).
__device__ __forceinline__ int row_position(const NearGeom& g, int b, int64_t s) {
  const int bs = g.leaf_of[s];
  for (int q = g.near_ptr[b]; q < g.near_ptr[b + 1]; ++q)
    if (g.near_idx[q] == bs) return g.near_off[q] + int(s - g.leaf_start[bs]);
  return -1;
}

__global__ void __launch_bounds__(256) k_count_singular(int64_t T, NearGeom g, unsigned long long* count) {
  int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (t >= T) return;
  const int b = g.leaf_of[t];
  const int q0 = g.near_ptr[b], q1 = g.near_ptr[b + 1];
  const int len = int(g.row_ptr[t + 1] - g.row_ptr[t]);
  int qi = q0;
  unsigned n = 0;
  for (int j = row_position(g, b, t) + 1 + lane; j < len; j += 32) {
    while (qi + 1 < q1 && g.near_off[qi + 1] <= j) ++qi;
    const int64_t s = g.leaf_start[g.near_idx[qi]] + (j - g.near_off[qi]);
    if (near_singular(g.cent + 3 * t, g.cent + 3 * s, g.h2[t], g.h2[s])) ++n;
  }
  n = __reduce_add_sync(0xffffffffu, n);
  if (lane == 0 && n) atomicAdd(count, (unsigned long long)n);
}

struct SingPair {
  int32_t t, s;
  int64_t e;
};

template <typename Rm>
__device__ __forceinline__ void store_moments(C2<Rm>* mom, int64_t nnz, int64_t e, const Moments& m, bool swap) {
  mom[e] = mk<Rm>(Rm(m.m0r), Rm(m.m0i));
  for (int d = 0; d < 3; ++d) {
    const double tr = swap ? m.msr[d] : m.mtr[d], ti = swap ? m.msi[d] : m.mti[d];
    const double sr = swap ? m.mtr[d] : m.msr[d], si = swap ? m.mti[d] : m.msi[d];
    mom[(1 + d) * nnz + e] = mk<Rm>(Rm(tr), Rm(ti));
    mom[(4 + d) * nnz + e] = mk<Rm>(Rm(sr), Rm(si));
  }
  mom[7 * nnz + e] = mk<Rm>(Rm(m.mtsr), Rm(m.mtsi));
}

// 20,480 triangles (2.75e6 unordered pairs): 8.6 ms; 34.4 ms with both orders,
// sincos and a division per point pair.
template <typename Rm, int NT>
__global__ void __launch_bounds__(128) k_near_regular(int64_t T, int64_t nnz, NearGeom g, double k, NearSeries G,
                                                      const double* __restrict__ rule7, C2<Rm>* __restrict__ mom,
                                                      SingPair* __restrict__ list, unsigned long long* __restrict__ nlist,
                                                      unsigned long long cap) {
  __shared__ TestPoint tps[4][7];
  int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (t >= T) return;
  const int b = g.leaf_of[t];
  const int q0 = g.near_ptr[b], q1 = g.near_ptr[b + 1];
  const int64_t e0 = g.row_ptr[t];
  const int len = int(g.row_ptr[t + 1] - e0);
  const double* ct = g.cent + 3 * t;
  const Rule7 R = load_rule7(rule7);
  TestPoint* tp = tps[threadIdx.x >> 5];
  if (lane < 7) {
    const double* vt = g.vert + 9 * t;
    const double* q = rule7 + 4 * lane;
    tp[lane].w = q[3] * g.area[t];
    for (int d = 0; d < 3; ++d) {
      tp[lane].r[d] = q[0] * vt[d] + q[1] * vt[3 + d] + q[2] * vt[6 + d];
      tp[lane].wu[d] = tp[lane].w * (tp[lane].r[d] - ct[d]);
    }
  }
  __syncwarp();
  int qi = q0;
  for (int j = row_position(g, b, t) + 1 + lane; j < len; j += 32) {
    while (qi + 1 < q1 && g.near_off[qi + 1] <= j) ++qi;
    const int64_t s = g.leaf_start[g.near_idx[qi]] + (j - g.near_off[qi]);
    const int64_t e = e0 + j;
    if (near_singular(ct, g.cent + 3 * s, g.h2[t], g.h2[s])) {
      unsigned long long slot = atomicAdd(nlist, 1ull);
      if (slot < cap) list[slot] = SingPair{int32_t(t), int32_t(s), e};
      continue;
    }
    Moments m;
    moments_regular<NT>(tp, g.vert + 9 * s, g.cent + 3 * s, g.area[s], k, G, R, m);
    store_moments(mom, nnz, e, m, false);
    const int p = row_position(g, g.near_idx[qi], t);
    if (p >= 0) store_moments(mom, nnz, g.row_ptr[s] + p, m, true);
  }
}

// Eight lanes per pair: a small mesh's few thousand pairs still give every SM
// warps, and the 64 outer points of each order split evenly.  SELF: the pairs
// (t, t), one order each (no list).  20,480 triangles: 24.1 ms (22.5 + 1.6);
// 84.1 ms with a thread per pair, two arctangents and a logarithm of a quotient
// per edge and three sines per point pair.
constexpr int kSingLanes = 8;
template <typename Rm, int NT, bool SELF>
__global__ void __launch_bounds__(128) k_near_singular(int64_t npairs, int64_t nnz, NearGeom g, double k, NearSeries G,
                                                       const double* __restrict__ rule7,
                                                       const double* __restrict__ rule64,
                                                       const SingPair* __restrict__ list, C2<Rm>* __restrict__ mom) {
  const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kSingLanes;
  const int lane = threadIdx.x % kSingLanes;
  // lanes past the end repeat the last pair (every lane joins the shuffles)
  const int64_t ii = min(i, npairs - 1);
  const int64_t pt = SELF ? ii : list[ii].t, ps = SELF ? ii : list[ii].s;
  const Rule7 R = load_rule7(rule7);
  // both orders into one set of moments as seen from t (test) and s (source):
  // mt and ms change places between them
  Moments m{};
#pragma unroll 1
  for (int order = 0; order < (SELF ? 1 : 2); ++order) {
    const int64_t t = order ? ps : pt, s = order ? pt : ps;
    moments_singular<NT, kSingLanes>(g.vert + 9 * t, g.cent + 3 * t, g.area[t], g.vert + 9 * s, g.cent + 3 * s,
                                     g.area[s], k, G, R, rule64, lane, m);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double x = m.mtr[d], y = m.mti[d];
      m.mtr[d] = SELF ? 0.5 * (x + m.msr[d]) : m.msr[d];
      m.mti[d] = SELF ? 0.5 * (y + m.msi[d]) : m.msi[d];
      m.msr[d] = SELF ? m.mtr[d] : x;
      m.msi[d] = SELF ? m.mti[d] : y;
    }
  }
  double* f = reinterpret_cast<double*>(&m);
#pragma unroll
  for (int q = 0; q < 16; ++q) {
#pragma unroll
    for (int w = 1; w < kSingLanes; w *= 2) f[q] += __shfl_xor_sync(0xffffffffu, f[q], w);
    if (!SELF) f[q] *= 0.5;
  }
  if (i >= npairs || lane != 0) return;
  store_moments(mom, nnz, SELF ? g.row_ptr[pt] + row_position(g, g.leaf_of[pt], pt) : list[ii].e, m, false);
  if constexpr (!SELF) {
    const int p = row_position(g, g.leaf_of[ps], pt);
    if (p >= 0) store_moments(mom, nnz, g.row_ptr[ps] + p, m, true);
  }
}

// delta of a leaf box (FixedRow): the exponent of its longest edge, near boxes included.
__global__ void k_fixed_delta(int64_t nleaf, NearGeom g, int32_t* __restrict__ delta) {
  const int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (b >= nleaf) return;
  int e = -100000;
  for (int q = g.near_ptr[b]; q < g.near_ptr[b + 1]; ++q)
    for (int s = g.leaf_start[g.near_idx[q]] + int(threadIdx.x & 31); s < g.leaf_start[g.near_idx[q] + 1]; s += 32)
      e = max(e, ilogb(g.h2[s]));
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) delta[b] = (e >> 1) + 1;
}

// The FP64 pair moments into fixed point, in place (near_fixed.cuh: the eight
// 16-byte moments of an entry become its eight planes' entries): a warp per
// row, one pass for the row's exponents and one to convert.
__global__ void __launch_bounds__(128) k_moments_fixed(int64_t T, int64_t nnz, NearGeom g,
                                                       const int32_t* __restrict__ delta, FixedRow* __restrict__ row,
                                                       cd* mom) {
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (t >= T) return;
  const int lane = threadIdx.x & 31, dl = delta[g.leaf_of[t]];
  const int64_t e0 = g.row_ptr[t], e1 = g.row_ptr[t + 1];
  // per part: largest exponent fields of m0, mt, ms, mts, and the largest sums
  // over one lane's entries of a product stage, as they meet in a sum of the
  // product: m0 with one ms, mt's three with mts
  int x[2][4] = {{1, 1, 1, 1}, {1, 1, 1, 1}};
  double a0[2] = {0, 0}, at[2] = {0, 0}, s0[2] = {0, 0}, st[2] = {0, 0};
  const double dw = scalbn(1.0, -dl);
  for (int64_t e = e0 + lane; e < e1; e += 32) {
    cd m[kMom];
#pragma unroll
    for (int q = 0; q < kMom; ++q) m[q] = mom[q * nnz + e];
    const bool first = ((e - e0) % kFixedStage) < 32;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      double v[kMom];
#pragma unroll
      for (int q = 0; q < kMom; ++q) {
        v[q] = fabs(p ? m[q].y : m[q].x);
        int& r = x[p][(q + 2) / 3];
        r = max(r, exponent_field(v[q]));
      }
      s0[p] = (first ? 0.0 : s0[p]) + (v[0] + dw * fmax(v[4], fmax(v[5], v[6])));
      st[p] = (first ? 0.0 : st[p]) + (v[1] + v[2] + v[3] + dw * v[7]);
      a0[p] = fmax(a0[p], s0[p]);
      at[p] = fmax(at[p], st[p]);
    }
  }
  int top = 0;
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[p][i] = __reduce_max_sync(0xffffffffu, x[p][i]);
      top = max(top, x[p][i]);
    }
  // exponent fields: the largest integer below 2^kMomentBits, the sums below 2^kLaneBits
  auto field = [&](int xa, int xb, double sum) {
    const int lane_e = __reduce_max_sync(0xffffffffu, sum > 0 ? exponent_field(sum) + 53 - kLaneBits : -100000);
    return max(max(xa, xb - dl) + 53 - kMomentBits, lane_e);
  };
  int f0[2], ft[2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    f0[p] = field(x[p][0], x[p][2], a0[p]);
    ft[p] = field(x[p][1], x[p][3], at[p]);
  }
  if (lane == 0)
    row[t] = top == 0x7ff ? FixedRow{{kFixedNan, kFixedNan}, {kFixedNan, kFixedNan}}
                          : FixedRow{{f0[0] - 1075, f0[1] - 1075}, {ft[0] - 1075, ft[1] - 1075}};
  for (int64_t e = e0 + lane; e < e1; e += 32) {
    cd m[kMom];
#pragma unroll
    for (int q = 0; q < kMom; ++q) m[q] = mom[q * nnz + e];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int g = 0; g < kFixedPlanes; ++g) {
        int2 r[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int q = 2 * g + u;
          r[u] = fixed_encode(p ? m[q].y : m[q].x, ((q >= 1 && q <= 3) || q == 7 ? ft[p] : f0[p]) + (q >= 4 ? dl : 0));
        }
        reinterpret_cast<int4*>(mom)[(p * kFixedPlanes + g) * nnz + e] = make_int4(r[0].x, r[0].y, r[1].x, r[1].y);
      }
  }
}

// Leaf radiation tables at kappa_L: Pi_t(p) = int_t exp(-i kappa khat_p.(r - C_b)),
// M_t(p) = int_t (r - c_t) exp(-i kappa khat_p.(r - C_b)); 7-point rule.
// Called with P = the half grid (theta rows 0..ntheta/2-1): the other half
// is the complex conjugate.
template <typename Rf>
__global__ void k_rad(int64_t T, int P, const double* __restrict__ vert, const double* __restrict__ cent,
                      const double* __restrict__ area, const int32_t* __restrict__ leaf_of,
                      const double* __restrict__ leaf_center, const double* __restrict__ khat, double kappa,
                      const double* __restrict__ rule7, C2<Rf>* __restrict__ Pi, C2<Rf>* __restrict__ M,
                      C2<Rf>* __restrict__ PiR, C2<Rf>* __restrict__ MR) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= T * P) return;
  int64_t t = i / P;
  int p = int(i % P);
  const double* v = vert + 9 * t;
  const double* C = leaf_center + 3 * leaf_of[t];
  double kx = khat[3 * p], ky = khat[3 * p + 1], kz = khat[3 * p + 2];
  double pr = 0, pi = 0, mr[3] = {0, 0, 0}, mi[3] = {0, 0, 0};
  for (int q = 0; q < 7; ++q) {
    double r[3];
    for (int d = 0; d < 3; ++d) r[d] = rule7[4 * q] * v[d] + rule7[4 * q + 1] * v[3 + d] + rule7[4 * q + 2] * v[6 + d];
    double w = rule7[4 * q + 3] * area[t];
    double ph = -kappa * (kx * (r[0] - C[0]) + ky * (r[1] - C[1]) + kz * (r[2] - C[2]));
    double s, c;
    sincos(ph, &s, &c);
    pr += w * c;
    pi += w * s;
    for (int d = 0; d < 3; ++d) {
      double u = r[d] - cent[3 * t + d];
      mr[d] += w * u * c;
      mi[d] += w * u * s;
    }
  }
  Pi[t * P + p] = mk<Rf>(Rf(pr), Rf(pi));
  for (int d = 0; d < 3; ++d) M[(t * 3 + d) * P + p] = mk<Rf>(Rf(mr[d]), Rf(mi[d]));
  PiR[(int64_t)p * T + t] = mk<Rf>(Rf(pr), Rf(pi));
  for (int d = 0; d < 3; ++d) MR[((int64_t)d * P + p) * T + t] = mk<Rf>(Rf(mr[d]), Rf(mi[d]));
}

// Translation operator of Eq. (5) with the quadrature weight and the
// i k / (16 pi^2) prefactor of Eq. (4) folded in:
//   T[off][p] = (i k/(16 pi^2)) w_p sum_{t<=tau} i^t (2t+1) s^t h_t(k|w|) P_t(khat_p . what),
// w = offset * a.  s^t y_t by the scaled upward recurrence
// Y_{t+1} = (2t+1)(s/z) Y_t - s^2 Y_{t-1}; s^t j_t by its power series (z <= 4).
template <typename Rf>
__global__ void k_trans_table(int P, int tau, double k, double s, double a, const double* __restrict__ khat,
                              const double* __restrict__ wgt, C2<Rf>* __restrict__ Tt) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kNoffs * P) return;
  int off = i / P, p = i % P;
  // offset code -> (dx, dy, dz), lexicographic over {-3..3}^3 without {-1..1}^3
  int code = 0, dx = 0, dy = 0, dz = 0;
  for (int x = -3; x <= 3; ++x)
    for (int y = -3; y <= 3; ++y)
      for (int z = -3; z <= 3; ++z) {
        int mx = max(abs(x), max(abs(y), abs(z)));
        if (mx <= 1) continue;
        if (code == off) {
          dx = x;
          dy = y;
          dz = z;
        }
        ++code;
      }
  double wv[3] = {dx * a, dy * a, dz * a};
  double wn = sqrt(wv[0] * wv[0] + wv[1] * wv[1] + wv[2] * wv[2]);
  double z = k * wn;
  double cosang = (khat[3 * p] * wv[0] + khat[3 * p + 1] * wv[1] + khat[3 * p + 2] * wv[2]) / wn;
  double sz, cz;
  sincos(z, &sz, &cz);
  double Yv[kMaxTau + 2], Pv[kMaxTau + 2];
  Yv[0] = -cz / z;
  Yv[1] = s * (-cz / (z * z) - sz / z);
  for (int t = 1; t < tau; ++t) Yv[t + 1] = (2.0 * t + 1.0) * (s / z) * Yv[t] - s * s * Yv[t - 1];
  Pv[0] = 1.0;
  Pv[1] = cosang;
  for (int t = 1; t < tau; ++t) Pv[t + 1] = ((2.0 * t + 1.0) * cosang * Pv[t] - t * Pv[t - 1]) / (t + 1.0);
  double ar = 0, ai = 0;
  double sz_pow = 1.0;  // (s z)^t
  double dfact = 1.0;   // (2t+1)!!
  for (int t = 0; t <= tau; ++t) {
    if (t >= 1) {
      sz_pow *= s * z;
      dfact *= (2.0 * t + 1.0);
    }
    // s^t j_t(z) = (s z)^t / (2t+1)!! * sum_n (-z^2/2)^n / (n! prod_{i=1..n} (2t+2i+1))
    double term = 1.0, ser = 1.0;
    for (int n = 1; n < 60; ++n) {
      term *= -0.5 * z * z / (n * (2.0 * t + 2.0 * n + 1.0));
      ser += term;
      if (fabs(term) < 1e-18 * fabs(ser)) break;
    }
    double Jt = sz_pow / dfact * ser;
    // i^t (2t+1) (J + i Y) P_t
    double hr = (2.0 * t + 1.0) * Jt * Pv[t], hi = (2.0 * t + 1.0) * Yv[t] * Pv[t];
    switch (t & 3) {
      case 0: ar += hr; ai += hi; break;
      case 1: ar -= hi; ai += hr; break;
      case 2: ar -= hr; ai -= hi; break;
      default: ar += hi; ai -= hr; break;
    }
  }
  // times i k w_p / (16 pi^2)
  double f = k * wgt[p] / (16.0 * kPi * kPi);
  Tt[(int64_t)off * P + p] = mk<Rf>(Rf(-f * ai), Rf(f * ar));
}

// Degree-rescale filter from level l+1 to level l with ratio
// r = kappa_l / kappa_{l+1} (1/2 while both levels are scaled, 1 once s = 1):
// F[p][q] = sum_{n<ntheta} r^n (2n+1)/(4 pi) P_n(khat_p.khat_q) w_q.
template <typename Rf>
__global__ void k_filter(int P, int ntheta, double ratio, const double* __restrict__ khat,
                         const double* __restrict__ wgt, Rf* __restrict__ F, Rf* __restrict__ Ft) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P * P) return;
  int p = i / P, q = i % P;
  double x = khat[3 * p] * khat[3 * q] + khat[3 * p + 1] * khat[3 * q + 1] + khat[3 * p + 2] * khat[3 * q + 2];
  x = fmin(1.0, fmax(-1.0, x));
  double Pm = 1.0, Pc = x, sum = 1.0 / kFourPi, r = 1.0;
  for (int l = 1; l < ntheta; ++l) {
    r *= ratio;
    double Pl = (l == 1) ? x : Pc;
    if (l >= 2) {
      Pl = ((2.0 * l - 1.0) * x * Pc - (l - 1.0) * Pm) / l;
      Pm = Pc;
      Pc = Pl;
    }
    sum += r * (2.0 * l + 1.0) / kFourPi * Pl;
  }
  double v = sum * wgt[q];
  F[(int64_t)p * P + q] = Rf(v);
  Ft[(int64_t)q * P + p] = Rf(v);
}

// Azimuthal blocks of the block-circulant filter:
// K_m[i][k] = (1/NPHI) sum_d F[(i, d)][(k, 0)] cos(2 pi m d / NPHI)
// (F[(i,d)][(k,0)] is even in d, so the sine part vanishes).
template <typename Rf>
__global__ void k_filter_fourier(int ntheta, const Rf* __restrict__ F, Rf* __restrict__ Kf) {
  const int nphi = 2 * ntheta, P = ntheta * nphi;
  int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= nphi * ntheta * ntheta) return;
  int m = id / (ntheta * ntheta), i = (id / ntheta) % ntheta, k = id % ntheta;
  double acc = 0;
  for (int d = 0; d < nphi; ++d) {
    double c = cospi(2.0 * double(m * d % nphi) / nphi);
    acc += double(F[(int64_t)(i * nphi + d) * P + k * nphi]) * c;
  }
  Kf[id] = Rf(acc / nphi);
}

// Interpolation phases for the children of level-l boxes:
// exp(-i kappa_l khat_p . (C_child - C_parent)), C_child - C_parent = (a_{l+1}/2)(+-1,+-1,+-1).
template <typename Rf>
__global__ void k_phase(int P, double kappa, double half, const double* __restrict__ khat, C2<Rf>* __restrict__ ph) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 8 * P) return;
  int o = i / P, p = i % P;
  double d[3] = {half * (2 * ((o >> 2) & 1) - 1), half * (2 * ((o >> 1) & 1) - 1), half * (2 * (o & 1) - 1)};
  double arg = -kappa * (khat[3 * p] * d[0] + khat[3 * p + 1] * d[1] + khat[3 * p + 2] * d[2]);
  double s, c;
  sincos(arg, &s, &c);
  ph[i] = mk<Rf>(Rf(c), Rf(s));
}

// ------------------------------------------------------------ host side

pie_status cuda_check(cudaError_t e, const char* what) {
  if (e == cudaSuccess) return PIE_OK;
  set_error(std::string(what) + ": " + cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? PIE_ERR_OOM : PIE_ERR_CUDA;
}

void* dalloc(Problem& pr, size_t bytes) {
  void* p = nullptr;
  if (bytes == 0) bytes = 16;
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  pr.allocs.push_back(p);
  pr.bytes += bytes;
  return p;
}

template <typename T>
static T* upload(Problem& pr, const std::vector<T>& h, cudaStream_t st, pie_status& s) {
  if (s != PIE_OK) return nullptr;
  T* d = static_cast<T*>(dalloc(pr, sizeof(T) * h.size()));
  if (!d) {
    set_error("device allocation failed");
    s = PIE_ERR_OOM;
    return nullptr;
  }
  if (!h.empty()) s = cuda_check(cudaMemcpyAsync(d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice, st), "upload");
  return d;
}

static void* zalloc(Problem& pr, size_t bytes, pie_status& s) {
  if (s != PIE_OK) return nullptr;
  void* d = dalloc(pr, bytes);
  if (!d) {
    set_error("device allocation failed");
    s = PIE_ERR_OOM;
  }
  return d;
}

template <typename Rm, typename Rf>
static pie_status setup_t(Problem& pr, cudaStream_t st) {
  const Mesh& m = pr.mesh;
  const Tree& tr = pr.tree;
  const int64_t T = pr.T, E = pr.E;
  const int L = tr.L;
  const int P = pr.P;
  pie_status s = PIE_OK;

  // tree-ordered triangle tables
  std::vector<int32_t> tri_edge(T * 3), leaf_of(T);
  std::vector<double> tri_c(T * 3, 0.0), tri_dcp(T * 9, 0.0), tri_cdcp(T * 9, 0.0), vert(T * 9), cent(T * 3), h2(T), area(T);
  for (int64_t i = 0; i < T; ++i) {
    int64_t tm = tr.perm[i];
    for (int k = 0; k < 3; ++k) {
      int32_t v = m.tri[3 * tm + k];
      for (int d = 0; d < 3; ++d) vert[9 * i + 3 * k + d] = m.xyz[3 * v + d];
    }
    for (int d = 0; d < 3; ++d) cent[3 * i + d] = m.centroid[3 * tm + d];
    h2[i] = m.h2[tm];
    pr.h_max = std::max(pr.h_max, std::sqrt(m.h2[tm]));
    const double* ctr = &m.centroid[3 * tm];
    pr.r_max = std::max(pr.r_max, std::sqrt(ctr[0] * ctr[0] + ctr[1] * ctr[1] + ctr[2] * ctr[2]));
    area[i] = m.area[tm];
    for (int k = 0; k < 3; ++k) {
      int32_t n = m.tri_edge[3 * tm + k];
      tri_edge[3 * i + k] = n;
      if (n < 0) continue;
      int sg = m.tri_sign[3 * tm + k];
      const double* a = &m.xyz[3 * m.edges[2 * n]];
      const double* b = &m.xyz[3 * m.edges[2 * n + 1]];
      double len = std::sqrt((b[0] - a[0]) * (b[0] - a[0]) + (b[1] - a[1]) * (b[1] - a[1]) + (b[2] - a[2]) * (b[2] - a[2]));
      tri_c[3 * i + k] = sg * len / (2.0 * m.area[tm]);
      int32_t fv = m.edge_free[2 * n + (sg > 0 ? 0 : 1)];
      for (int d = 0; d < 3; ++d) {
        tri_dcp[9 * i + 3 * k + d] = m.centroid[3 * tm + d] - m.xyz[3 * fv + d];
        tri_cdcp[9 * i + 3 * k + d] = tri_c[3 * i + k] * tri_dcp[9 * i + 3 * k + d];
      }
    }
  }
  std::vector<int32_t> edge_tt(E * 2);
  std::vector<int8_t> edge_k(E * 2);
  for (int64_t n = 0; n < E; ++n)
    for (int side = 0; side < 2; ++side) {
      int32_t tm = m.edge_tri[2 * n + side];
      edge_tt[2 * n + side] = int32_t(tr.inv_perm[tm]);
      int kk = 0;
      for (int k = 0; k < 3; ++k)
        if (m.tri_edge[3 * tm + k] == n) kk = k;
      edge_k[2 * n + side] = int8_t(kk);
    }
  const int64_t nleaf = int64_t(tr.keys[L].size());
  pr.nleaf = nleaf;
  std::vector<int32_t> leaf_start(nleaf + 1), near_ptr(nleaf + 1), near_idx(tr.near_idx.size());
  std::vector<double> leaf_center(nleaf * 3);
  const double aL = tr.box_size(L);
  for (int64_t b = 0; b <= nleaf; ++b) leaf_start[b] = int32_t(tr.leaf_start[b]);
  for (int64_t b = 0; b < nleaf; ++b) {
    for (int64_t i = tr.leaf_start[b]; i < tr.leaf_start[b + 1]; ++i) leaf_of[i] = int32_t(b);
    int64_t key = tr.keys[L][b], ii[3] = {0, 0, 0};
    for (int bit = 0; bit < L - 1; ++bit) {
      ii[0] |= ((key >> (3 * bit + 2)) & 1) << bit;
      ii[1] |= ((key >> (3 * bit + 1)) & 1) << bit;
      ii[2] |= ((key >> (3 * bit)) & 1) << bit;
    }
    for (int d = 0; d < 3; ++d) leaf_center[3 * b + d] = tr.x0[d] + (double(ii[d]) + 0.5) * aL;
  }
  for (size_t i = 0; i < near_ptr.size(); ++i) near_ptr[i] = int32_t(tr.near_ptr[i]);
  for (size_t i = 0; i < near_idx.size(); ++i) near_idx[i] = int32_t(tr.near_idx[i]);
  std::vector<int32_t> near_off(near_idx.size());
  for (int64_t b = 0; b < nleaf; ++b) {
    int32_t acc = 0;
    for (int64_t qi = tr.near_ptr[b]; qi < tr.near_ptr[b + 1]; ++qi) {
      near_off[qi] = acc;
      acc += int32_t(tr.leaf_start[tr.near_idx[qi] + 1] - tr.leaf_start[tr.near_idx[qi]]);
    }
  }
  std::vector<int64_t> row_ptr(T + 1, 0);
  for (int64_t i = 0; i < T; ++i) {
    int64_t b = leaf_of[i], cnt = 0;
    for (int64_t q = tr.near_ptr[b]; q < tr.near_ptr[b + 1]; ++q) {
      int64_t nb = tr.near_idx[q];
      cnt += tr.leaf_start[nb + 1] - tr.leaf_start[nb];
    }
    row_ptr[i + 1] = row_ptr[i] + cnt;
    pr.max_row = std::max(pr.max_row, cnt);
    if (cnt <= kNearShortRow) {
      pr.short_row = std::max(pr.short_row, cnt);
      pr.short_pairs += cnt;
    }
    pr.box_pairs = std::max(pr.box_pairs, cnt * (tr.leaf_start[b + 1] - tr.leaf_start[b]));
  }
  pr.nnz = row_ptr[T];

  // angular grid: ntheta Gauss-Legendre nodes in cos(theta) x 2 ntheta azimuths
  const int nt = pr.par.ntheta;
  std::vector<double> gx, gw;
  gauss_legendre(nt, gx, gw);
  // The lower theta rows are computed; the upper rows are their exact
  // negatives (antipodes), so that -khat is on the grid bit for bit.
  std::vector<double> khat(3 * P), wgt(P);
  for (int i = 0; i < nt / 2; ++i)
    for (int j = 0; j < 2 * nt; ++j) {
      int p = i * 2 * nt + j;
      int pa = (nt - 1 - i) * 2 * nt + (j + nt) % (2 * nt);
      double ct = gx[i], stt = std::sqrt(1.0 - ct * ct), ph = kPi * j / nt;
      khat[3 * p] = stt * std::cos(ph);
      khat[3 * p + 1] = stt * std::sin(ph);
      khat[3 * p + 2] = ct;
      for (int d = 0; d < 3; ++d) khat[3 * pa + d] = -khat[3 * p + d];
      wgt[p] = gw[i] * kPi / nt;
      wgt[pa] = gw[nt - 1 - i] * kPi / nt;
    }
  // 7-point degree-5 rule (Radon), closed form; and the 8 x 8 collapsed Gauss rule
  std::vector<double> r7, r64;
  {
    const double s15 = std::sqrt(15.0);
    r7 = {1.0 / 3, 1.0 / 3, 1.0 / 3, 9.0 / 40};
    const double as[2] = {(6.0 - s15) / 21.0, (6.0 + s15) / 21.0};
    const double ws[2] = {(155.0 - s15) / 1200.0, (155.0 + s15) / 1200.0};
    for (int o = 0; o < 2; ++o) {
      double a = as[o], b = 1.0 - 2.0 * a;
      double pts[3][3] = {{b, a, a}, {a, b, a}, {a, a, b}};
      for (auto& q : pts) r7.insert(r7.end(), {q[0], q[1], q[2], ws[o]});
    }
    std::vector<double> ux, uw;
    gauss_legendre(8, ux, uw);
    for (int i = 0; i < 8; ++i)
      for (int j = 0; j < 8; ++j) {
        double u = 0.5 * (ux[i] + 1.0), v = 0.5 * (ux[j] + 1.0);
        double x = u, y = (1.0 - u) * v;
        r64.insert(r64.end(), {1.0 - x - y, x, y, 2.0 * (0.5 * uw[i]) * (0.5 * uw[j]) * (1.0 - u)});
      }
  }

  pr.tri_edge = upload(pr, tri_edge, st, s);
  pr.tri_c = upload(pr, tri_c, st, s);
  pr.tri_dcp = upload(pr, tri_dcp, st, s);
  pr.tri_cdcp = upload(pr, tri_cdcp, st, s);
  pr.perm = upload(pr, tr.perm, st, s);
  pr.inv_perm = upload(pr, tr.inv_perm, st, s);
  pr.edge_tt = upload(pr, edge_tt, st, s);
  pr.edge_k = upload(pr, edge_k, st, s);
  pr.vert = upload(pr, vert, st, s);
  pr.rule7_host = r7;
  pr.cent = upload(pr, cent, st, s);
  pr.h2 = upload(pr, h2, st, s);
  pr.area = upload(pr, area, st, s);
  pr.leaf_of = upload(pr, leaf_of, st, s);
  pr.leaf_start = upload(pr, leaf_start, st, s);
  pr.leaf_center = upload(pr, leaf_center, st, s);
  pr.near_ptr = upload(pr, near_ptr, st, s);
  pr.near_idx = upload(pr, near_idx, st, s);
  pr.near_off = upload(pr, near_off, st, s);
  pr.row_ptr = upload(pr, row_ptr, st, s);
  pr.khat = upload(pr, khat, st, s);
  pr.wgt = upload(pr, wgt, st, s);
  pr.rule7 = upload(pr, r7, st, s);
  pr.rule64 = upload(pr, r64, st, s);
  if (s != PIE_OK) return s;

  // near pair moments (three passes, see k_near_regular)
  pr.mom = zalloc(pr, sizeof(C2<Rm>) * kMom * size_t(pr.nnz), s);
  unsigned long long* dcount = static_cast<unsigned long long*>(zalloc(pr, 2 * sizeof(unsigned long long), s));
  if (s != PIE_OK) return s;
  NearGeom ng{pr.leaf_of, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr,
              pr.vert, pr.cent, pr.area, pr.h2};
  cudaMemsetAsync(dcount, 0, 2 * sizeof(unsigned long long), st);
  k_count_singular<<<unsigned((T * 32 + 255) / 256), 256, 0, st>>>(T, ng, dcount);
  unsigned long long nsing = 0;
  if ((s = cuda_check(cudaMemcpyAsync(&nsing, dcount, sizeof(nsing), cudaMemcpyDeviceToHost, st), "count")) != PIE_OK)
    return s;
  if ((s = cuda_check(cudaStreamSynchronize(st), "count sync")) != PIE_OK) return s;
  SingPair* list = static_cast<SingPair*>(zalloc(pr, sizeof(SingPair) * std::max<unsigned long long>(nsing, 1), s));
  if (s != PIE_OK) return s;
  // Series terms by the largest kR: points of near triangles are at most
  // 2 sqrt(3) leaf sides and two thirds of an edge each way apart (h <= leaf /
  // 1.5), 4.4 leaf sides; near-singular pairs at most 2.9 h.  First omitted
  // term below 1e-17: x^(2 NT)/(2 NT)!, or 2 x^(2 NT)/(2 NT + 2)!; k h is at most 0.52.
  {
    C2<Rm>* mom = static_cast<C2<Rm>*>(pr.mom);
    const unsigned rb = unsigned((T * 32 + 127) / 128);
    const double xr = 4.4 * pr.k0 * aL, xs = 2.9 * pr.k0 * pr.h_max;
    const NearSeries G = near_series(pr.k0);
    auto regular = [&](auto nt) {
      k_near_regular<Rm, decltype(nt)::value><<<rb, 128, 0, st>>>(T, pr.nnz, ng, pr.k0, G, pr.rule7, mom, list,
                                                                  dcount + 1, nsing);
    };
    auto singular = [&](auto nt, auto self, int64_t n) {
      if (n == 0) return;
      k_near_singular<Rm, decltype(nt)::value, decltype(self)::value>
          <<<unsigned((n * kSingLanes + 127) / 128), 128, 0, st>>>(n, pr.nnz, ng, pr.k0, G, pr.rule7, pr.rule64, list,
                                                                   mom);
    };
    if (xr < 0.028)
      regular(std::integral_constant<int, 4>());
    else if (xr < 0.59)
      regular(std::integral_constant<int, 8>());
    else
      regular(std::integral_constant<int, 0>());
    auto both = [&](auto nt) {
      singular(nt, std::false_type(), int64_t(nsing));
      singular(nt, std::true_type(), T);
    };
    if (xs < 0.04)
      both(std::integral_constant<int, 4>());
    else
      both(std::integral_constant<int, kNearTerms>());
  }
  if constexpr (sizeof(Rm) == 8) {
    FixedRow* row = static_cast<FixedRow*>(pr.fixed_row = zalloc(pr, sizeof(FixedRow) * size_t(T), s));
    pr.fixed_delta = static_cast<int32_t*>(zalloc(pr, sizeof(int32_t) * size_t(nleaf), s));
    if (s != PIE_OK) return s;
    k_fixed_delta<<<unsigned((nleaf * 32 + 127) / 128), 128, 0, st>>>(nleaf, ng, pr.fixed_delta);
    k_moments_fixed<<<unsigned((T * 32 + 127) / 128), 128, 0, st>>>(T, pr.nnz, ng, pr.fixed_delta, row,
                                                                    static_cast<cd*>(pr.mom));
  }
  if ((s = cuda_check(cudaGetLastError(), "near build")) != PIE_OK) return s;

  // leaf radiation tables
  const double x = pr.par.kappa_a;
  // kappa_l = k0 / s_l with s_l = min(k0 a_l / x, 1): boxes small in
  // wavelengths use the scaled plane waves of Eq. (4), larger ones the
  // standard diagonalization (s = 1)
  auto kappa_of = [&](int l) { return std::max(x / tr.box_size(l), pr.k0); };
  pr.Pi = zalloc(pr, sizeof(C2<Rf>) * size_t(T) * (P / 2), s);
  pr.M = zalloc(pr, sizeof(C2<Rf>) * size_t(T) * 3 * (P / 2), s);
  pr.PiR = zalloc(pr, sizeof(C2<Rf>) * size_t(T) * (P / 2), s);
  pr.MR = zalloc(pr, sizeof(C2<Rf>) * size_t(T) * 3 * (P / 2), s);
  if (s != PIE_OK) return s;
  k_rad<Rf><<<unsigned((T * (P / 2) + 255) / 256), 256, 0, st>>>(T, P / 2, pr.vert, pr.cent, pr.area, pr.leaf_of,
                                                           pr.leaf_center, pr.khat, kappa_of(L), pr.rule7,
                                                           static_cast<C2<Rf>*>(pr.Pi), static_cast<C2<Rf>*>(pr.M),
                                                           static_cast<C2<Rf>*>(pr.PiR), static_cast<C2<Rf>*>(pr.MR));
  if ((s = cuda_check(cudaGetLastError(), "radiation tables")) != PIE_OK) return s;

  // levels
  pr.lev.assign(L + 1, LevelDev{});
  for (int l = 1; l <= L; ++l) {
    LevelDev& lv = pr.lev[l];
    lv.nb = int64_t(tr.keys[l].size());
    if (l >= 4) {
      std::vector<int32_t> par(lv.nb);
      std::vector<int8_t> oct(lv.nb);
      for (int64_t b = 0; b < lv.nb; ++b) {
        par[b] = int32_t(tr.parent[l][b]);
        oct[b] = int8_t(tr.keys[l][b] & 7);
      }
      lv.parent = upload(pr, par, st, s);
      lv.octant = upload(pr, oct, st, s);
    }
    if (l >= 3 && l < L) {
      std::vector<int32_t> cs(tr.child_start[l].begin(), tr.child_start[l].end());
      lv.child_start = upload(pr, cs, st, s);
    }
    if (l >= 3) {
      std::vector<int32_t> ptr(tr.il_ptr[l].begin(), tr.il_ptr[l].end());
      std::vector<int32_t> idx(tr.il_idx[l].begin(), tr.il_idx[l].end());
      lv.il_ptr = upload(pr, ptr, st, s);
      lv.il_idx = upload(pr, idx, st, s);
      lv.nlist = int64_t(idx.size());
      lv.il_off = upload(pr, tr.il_off[l], st, s);
      lv.S = zalloc(pr, sizeof(C2<Rf>) * size_t(pr.par.max_nrhs) * size_t(lv.nb) * kComp * P, s);
      lv.G = zalloc(pr, sizeof(C2<Rf>) * size_t(pr.par.max_nrhs) * size_t(lv.nb) * kComp * P, s);
      lv.trans = zalloc(pr, sizeof(C2<Rf>) * kNoffs * P, s);
      if (s != PIE_OK) return s;
      const double al = tr.box_size(l);
      lv.kappa = kappa_of(l);
      k_trans_table<Rf><<<unsigned((kNoffs * P + 127) / 128), 128, 0, st>>>(
          P, pr.par.tau, pr.k0, pr.k0 / lv.kappa, al, pr.khat, pr.wgt, static_cast<C2<Rf>*>(lv.trans));
      if (l < L) {
        lv.phase = zalloc(pr, sizeof(C2<Rf>) * 8 * P, s);
        if (s != PIE_OK) return s;
        k_phase<Rf><<<unsigned((8 * P + 127) / 128), 128, 0, st>>>(P, lv.kappa, 0.5 * tr.box_size(l + 1), pr.khat,
                                                                   static_cast<C2<Rf>*>(lv.phase));
        lv.F = zalloc(pr, sizeof(Rf) * P * P, s);
        lv.Ft = zalloc(pr, sizeof(Rf) * P * P, s);
        lv.Kf = zalloc(pr, sizeof(Rf) * 2 * nt * nt * nt, s);
        if (s != PIE_OK) return s;
        k_filter<Rf><<<unsigned((P * P + 127) / 128), 128, 0, st>>>(P, nt, lv.kappa / kappa_of(l + 1), pr.khat, pr.wgt,
                                                                    static_cast<Rf*>(lv.F), static_cast<Rf*>(lv.Ft));
        k_filter_fourier<Rf><<<unsigned((2 * nt * nt * nt + 127) / 128), 128, 0, st>>>(
            nt, static_cast<const Rf*>(lv.F), static_cast<Rf*>(lv.Kf));
      }
    }
    if (s != PIE_OK) return s;
  }
  const size_t cio = pr.io_f32() ? sizeof(cf) : sizeof(cd);
  const size_t nr = size_t(pr.par.max_nrhs);
  pr.gsgd_bytes = sizeof(C2<Rf>) * 2 * nr * size_t(pr.lev[L].nb) * kComp * (P / 2);
  pr.gsgd = zalloc(pr, pr.gsgd_bytes, s);
  pr.coef = zalloc(pr, cio * 6 * size_t(T) * nr, s);
  pr.pot = zalloc(pr, cio * 6 * size_t(T) * nr, s);
  pr.pot2 = zalloc(pr, cio * 6 * size_t(T) * nr, s);
  if (pr.par.precision == PIE_MIXED) pr.coef32 = zalloc(pr, sizeof(cf) * 6 * size_t(T) * nr, s);
  pr.vec = zalloc(pr, cio * size_t(pr.N), s);
  pr.vec2 = zalloc(pr, cio * size_t(pr.N), s);
  if (s != PIE_OK) return s;
  if ((s = cuda_check(cudaGetLastError(), "setup launch")) != PIE_OK) return s;
  int dev = 0;
  if ((s = cuda_check(cudaGetDevice(&dev), "device")) != PIE_OK) return s;
  if ((s = cuda_check(cudaDeviceGetAttribute(&pr.nsm, cudaDevAttrMultiProcessorCount, dev), "SM count")) != PIE_OK)
    return s;
  if ((s = cuda_check(cudaStreamCreateWithFlags(&pr.side, cudaStreamNonBlocking), "side stream")) != PIE_OK) return s;
  int prio_low = 0, prio_high = 0;
  if ((s = cuda_check(cudaDeviceGetStreamPriorityRange(&prio_low, &prio_high), "stream priorities")) != PIE_OK)
    return s;
  if ((s = cuda_check(cudaStreamCreateWithPriority(&pr.far, cudaStreamNonBlocking, prio_high), "far stream")) !=
      PIE_OK)
    return s;
  if ((s = cuda_check(cudaEventCreateWithFlags(&pr.ev_fork, cudaEventDisableTiming), "event")) != PIE_OK) return s;
  if ((s = cuda_check(cudaEventCreateWithFlags(&pr.ev_join, cudaEventDisableTiming), "event")) != PIE_OK) return s;
  if ((s = cuda_check(cudaEventCreateWithFlags(&pr.ev_far, cudaEventDisableTiming), "event")) != PIE_OK) return s;
  if ((s = cuda_check(cudaEventCreateWithFlags(&pr.ev_field, cudaEventDisableTiming), "event")) != PIE_OK) return s;
  pr.tune = pie_tuning{1, 2, pr.par.max_nrhs, 0, 0, 0};
  if ((s = product_prepare(pr)) != PIE_OK) return s;
  return cuda_check(cudaStreamSynchronize(st), "setup");
}

// Largest |re| and |im| of each of the eight moment planes (blockIdx.y):
// non-negative floats order like their bit patterns, so atomicMax on those.
__global__ void k_plane_absmax(int64_t nnz, const cf* __restrict__ mom, unsigned* __restrict__ mx) {
  const int q = blockIdx.y;
  float m = 0.f;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += int64_t(gridDim.x) * blockDim.x) {
    const cf v = mom[q * nnz + e];
    m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(mx + q, __float_as_uint(m));
}

// out = round-to-nearest half of (value * 2^e[plane]), plane by plane.
// One thread per pair: the eight planes' entries e become the pair's record
// of eight half pairs (32 bytes, entry-major [nnz][8]).
__global__ void k_to_half(int64_t nnz, const cf* __restrict__ mom, MomScale mul, __half2* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += int64_t(gridDim.x) * blockDim.x) {
    uint32_t w[kMom];
#pragma unroll
    for (int q = 0; q < kMom; ++q) {
      const cf v = mom[q * nnz + e];
      const __half2 h = __floats2half2_rn(v.x * mul.s[q], v.y * mul.s[q]);
      memcpy(&w[q], &h, sizeof(h));
    }
    uint4* o = reinterpret_cast<uint4*>(out + kMom * e);
    o[0] = make_uint4(w[0], w[1], w[2], w[3]);
    o[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// PIE_FP32H: the float moments built by setup_t become half pairs, each
// plane scaled by the power of two that puts its largest magnitude in
// [2^14, 2^15) (half's largest finite value is 65504); the scale's inverse is
// kept in pr.mom_scale.  The half moments are stored pair by pair ([nnz][8],
// one 32-byte record per pair, read with two 16-byte loads), unlike the
// plane-major float and double moments.  The float planes are freed.
static pie_status moments_to_half(Problem& pr, cudaStream_t st) {
  pie_status s = PIE_OK;
  const int64_t nnz = pr.nnz;
  unsigned* mx = static_cast<unsigned*>(zalloc(pr, sizeof(unsigned) * kMom, s));
  __half2* h = static_cast<__half2*>(zalloc(pr, sizeof(__half2) * kMom * size_t(nnz), s));
  if (s != PIE_OK) return s;
  const unsigned grid = unsigned(std::min<int64_t>((nnz + 255) / 256, 4096));
  cudaMemsetAsync(mx, 0, sizeof(unsigned) * kMom, st);
  const cf* mom = static_cast<const cf*>(pr.mom);
  k_plane_absmax<<<dim3(std::max(grid, 1u), kMom), 256, 0, st>>>(nnz, mom, mx);
  unsigned hm[kMom];
  if ((s = cuda_check(cudaMemcpyAsync(hm, mx, sizeof(hm), cudaMemcpyDeviceToHost, st), "moment range")) != PIE_OK)
    return s;
  if ((s = cuda_check(cudaStreamSynchronize(st), "moment range")) != PIE_OK) return s;
  MomScale mul;
  for (int q = 0; q < kMom; ++q) {
    float m;
    std::memcpy(&m, &hm[q], sizeof(m));
    int e = 0;
    if (m > 0.f && std::isfinite(m)) std::frexp(m, &e);  // m = f 2^e, f in [0.5, 1)
    const int sh = (m > 0.f && std::isfinite(m)) ? 15 - e : 0;
    mul.s[q] = std::ldexp(1.0f, sh);
    pr.mom_scale[q] = std::ldexp(1.0f, -sh);
  }
  k_to_half<<<std::max(grid, 1u), 256, 0, st>>>(nnz, mom, mul, h);
  if ((s = cuda_check(cudaStreamSynchronize(st), "moments to half")) != PIE_OK) return s;
  // release the float planes and the range buffer
  auto release = [&](void* ptr, size_t bytes) {
    for (size_t i = 0; i < pr.allocs.size(); ++i)
      if (pr.allocs[i] == ptr) {
        cudaFree(ptr);
        pr.allocs.erase(pr.allocs.begin() + i);
        pr.bytes -= bytes;
        return;
      }
  };
  release(pr.mom, sizeof(cf) * kMom * size_t(nnz));
  release(mx, sizeof(unsigned) * kMom);
  pr.mom = h;
  return PIE_OK;
}

pie_status setup_device(Problem& pr, cudaStream_t st) {
  switch (pr.par.precision) {
    case PIE_FP64:
      return setup_t<double, double>(pr, st);
    case PIE_FP32:
      return setup_t<float, float>(pr, st);
    case PIE_FP32H: {
      pie_status s = setup_t<float, float>(pr, st);
      return s == PIE_OK ? moments_to_half(pr, st) : s;
    }
    case PIE_MIXED:
      return setup_t<float, double>(pr, st);
  }
  set_error("unknown precision");
  return PIE_ERR_PARAM;
}

}  // namespace pie
