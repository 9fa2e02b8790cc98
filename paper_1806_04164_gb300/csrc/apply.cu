// One MLFMA matrix-vector product y = Z x for the PIEs (Section 3):
// local coefficients, near pair products, leaf aggregation, interpolation,
// translation (Eq. (5) operators), anterpolation, leaf disaggregation and
// Galerkin assembly (Section 2).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <type_traits>

#include "near_fixed.cuh"

namespace pie {

// a0: affine restriction of J to every triangle (tree order),
// J|_t = a (r - c_t) + beta, and the pulse densities sigma, d = 2a + w^2 eps0 sigma.
// tri_cdcp: tri_c times tri_dcp, multiplied once at set-up (the FP64 pipe bounds
// the kernel).
template <typename Rio>
__global__ void k_coef(int64_t T, int64_t E, const C2<Rio>* __restrict__ x, const int64_t* __restrict__ perm,
                       const int32_t* __restrict__ tri_edge, const double* __restrict__ tri_c,
                       const double* __restrict__ tri_cdcp, double w2e, C2<Rio>* __restrict__ coef,
                       cf* __restrict__ coef32, int64_t sx = 0, int64_t sc = 0,
                       const double* __restrict__ scale = nullptr) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= T) return;
  // right-hand side blockIdx.y (strides sx, sc between right-hand sides)
  x += blockIdx.y * sx;
  if (coef) coef += blockIdx.y * sc;
  if (coef32) coef32 += blockIdx.y * sc;
  // scale (may be null): the input is scale x, rounded to the io precision
  auto entry = [&](int64_t n) {
    const C2<Rio> v = x[n];
    return scale ? mk<Rio>(Rio(scale[n] * double(v.x)), Rio(scale[n] * double(v.y))) : v;
  };
  double ar = 0, ai = 0, br[3] = {0, 0, 0}, bi[3] = {0, 0, 0};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    int32_t n = tri_edge[3 * t + k];
    if (n < 0) continue;
    double c = tri_c[3 * t + k];
    const C2<Rio> v = entry(n);
    double xr = double(v.x), xi = double(v.y);
    ar += c * xr;
    ai += c * xi;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double cd_ = tri_cdcp[9 * t + 3 * k + d];
      br[d] += cd_ * xr;
      bi[d] += cd_ * xi;
    }
  }
  C2<Rio> s = entry(E + perm[t]);
  double sr = double(s.x), si = double(s.y);
  double v[12] = {ar, ai, br[0], bi[0], br[1], bi[1], br[2], bi[2], sr, si, 2.0 * ar + w2e * sr, 2.0 * ai + w2e * si};
  if (coef) {
    C2<Rio>* o = coef + 6 * t;
    for (int q = 0; q < 6; ++q) o[q] = mk<Rio>(Rio(v[2 * q]), Rio(v[2 * q + 1]));
  }
  if (coef32) {  // float copy for a float near part: converted once per triangle
    cf* o = coef32 + 6 * t;
    for (int q = 0; q < 6; ++q) o[q] = mk<float>(float(v[2 * q]), float(v[2 * q + 1]));
  }
}

// PIE_FP32H pair record: eight half pairs (m0, mt_xyz, ms_xyz, mts) at
// momh[8 e .. 8 e + 7], 32 bytes, read as two streaming 16-byte loads.
__device__ __forceinline__ void load_half_record(const __half2* __restrict__ momh, int64_t e, uint4& lo, uint4& hi) {
  const uint4* p = reinterpret_cast<const uint4*>(momh) + 2 * e;
  lo = __ldcs(p);
  hi = __ldcs(p + 1);
}

// The record's moments in float: each half pair times its plane's scale.
template <typename Rm>
__device__ __forceinline__ void unpack_half(const uint4& lo, const uint4& hi, const MomScale& msc, C2<Rm>* m) {
  const uint32_t w[kMom] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
  for (int q = 0; q < kMom; ++q) {
    __half2 h;
    memcpy(&h, &w[q], sizeof(h));
    const float2 v = __half22float2(h);
    m[q] = mk<Rm>(Rm(v.x * msc.s[q]), Rm(v.y * msc.s[q]));
  }
}

template <typename Rm>
__device__ __forceinline__ void unpack_half_record(const __half2* __restrict__ momh, int64_t e, const MomScale& msc,
                                                   C2<Rm>* m) {
  uint4 lo, hi;
  load_half_record(momh, e, lo, hi);
  unpack_half<Rm>(lo, hi, msc, m);
}

// a1: near part.  One warp per test triangle t; lanes run over the source
// triangles of the neighbouring leaf boxes (contiguous in tree order), whose
// eight pair moments are stored plane by plane ([8][nnz]), so a warp reads
// 32 consecutive entries of each plane (measured faster than per-pair
// records with vector loads).  Writes pot[t] (initialises it).  H16: the
// moments come from momh (PIE_FP32H: one record of eight half pairs per
// pair, 32 bytes, two 16-byte loads) times their plane's scale.
template <typename Rm, typename Rio, int RB = 1, bool H16 = false>
__global__ void __launch_bounds__(256) k_near(int64_t T, int64_t nnz, const int32_t* __restrict__ leaf_of,
                                              const int32_t* __restrict__ leaf_start,
                                              const int32_t* __restrict__ near_ptr,
                                              const int32_t* __restrict__ near_idx,
                                              const int32_t* __restrict__ near_off,
                                              const int64_t* __restrict__ row_ptr, const C2<Rm>* __restrict__ mom,
                                              const __half2* __restrict__ momh, MomScale msc,
                                              const C2<Rm>* __restrict__ coef, Rm mu0, C2<Rio>* __restrict__ pot,
                                              int nrhs = 1, int64_t sc = 0, int64_t sp = 0) {
  const int lane = threadIdx.x & 31;
  // right-hand sides r0 .. r0 + RB - 1 share every moment load
  const int r0 = blockIdx.y * RB;
  // one warp per test triangle, with a grid stride when the grid is smaller
  // than T warps (a bounded share of the SMs beside the far part)
  const int64_t wstride = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; t < T; t += wstride) {
    const int b = leaf_of[t];
    const int q0 = near_ptr[b], q1 = near_ptr[b + 1];
    const int64_t e0 = row_ptr[t];
    const int len = int(row_ptr[t + 1] - e0);
    C2<Rm> acc[RB][6];
#pragma unroll
    for (int r = 0; r < RB; ++r)
#pragma unroll
      for (int i = 0; i < 6; ++i) acc[r][i] = mk<Rm>(0, 0);
    // the row is the concatenation of the near boxes' source ranges; lanes walk
    // it flat (32 consecutive entries per step), each lane keeping a cursor on
    // the near box that holds its position
    int qi = q0;
    for (int j = lane; j < len; j += 32) {
      while (qi + 1 < q1 && near_off[qi + 1] <= j) ++qi;
      const int64_t s = leaf_start[near_idx[qi]] + (j - near_off[qi]);
      const int64_t ee = e0 + j;
      C2<Rm> m0, mt0, mt1, mt2, ms0, ms1, ms2, mts;
      if constexpr (H16) {
        C2<Rm> m[kMom];
        unpack_half_record(momh, ee, msc, m);
        m0 = m[0], mt0 = m[1], mt1 = m[2], mt2 = m[3], ms0 = m[4], ms1 = m[5], ms2 = m[6], mts = m[7];
      } else {
        m0 = mom[ee];
        mt0 = mom[nnz + ee], mt1 = mom[2 * nnz + ee], mt2 = mom[3 * nnz + ee];
        ms0 = mom[4 * nnz + ee], ms1 = mom[5 * nnz + ee], ms2 = mom[6 * nnz + ee];
        mts = mom[7 * nnz + ee];
      }
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        if (r0 + r >= nrhs) break;
        const C2<Rm>* c = coef + (r0 + r) * sc + 6 * s;
        C2<Rm> a = c[0], b0 = c[1], b1 = c[2], b2 = c[3], sg = c[4], dd = c[5];
        cfma(acc[r][0], a, mts);
        cfma(acc[r][0], b0, mt0);
        cfma(acc[r][0], b1, mt1);
        cfma(acc[r][0], b2, mt2);
        cfma(acc[r][1], a, ms0);
        cfma(acc[r][1], b0, m0);
        cfma(acc[r][2], a, ms1);
        cfma(acc[r][2], b1, m0);
        cfma(acc[r][3], a, ms2);
        cfma(acc[r][3], b2, m0);
        cfma(acc[r][4], sg, m0);
        cfma(acc[r][5], dd, m0);
      }
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      if (r0 + r >= nrhs) break;
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        acc[r][i].x = warp_sum(acc[r][i].x);
        acc[r][i].y = warp_sum(acc[r][i].y);
      }
      if (lane == 0) {
        C2<Rio>* o = pot + (r0 + r) * sp + 6 * t;
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = mk<Rio>(Rio(mu0 * acc[r][i].x), Rio(mu0 * acc[r][i].y));
        o[4] = cvt<Rio>(acc[r][4]);
        o[5] = cvt<Rio>(acc[r][5]);
      }
    }
  }
}

// The twelve components of six complex sums over a warp: each step of the
// butterfly sum keeps half of the values on either side, so the adds of one
// value are those of warp_sum (same bits) and a row takes 13 shuffles instead of
// 60.  Component i ends on lane 16 (i / 6) + 8 (i % 6 / 3) + 4 (i % 3 / 2) + 2 (i % 3 % 2).
__device__ __forceinline__ float warp_sum12(const cf* a, int lane, int* component) {
  float v[12];
#pragma unroll
  for (int i = 0; i < 6; ++i) v[2 * i] = a[i].x, v[2 * i + 1] = a[i].y;
  const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4, h1 = lane & 2;
  auto step = [](bool up, float lo, float hi, int o) {
    const float keep = up ? hi : lo, send = up ? lo : hi;
    return keep + __shfl_xor_sync(0xffffffffu, send, o);
  };
  float w[6], x[3], y[2];
#pragma unroll
  for (int i = 0; i < 6; ++i) w[i] = step(h4, v[i], v[6 + i], 16);
#pragma unroll
  for (int i = 0; i < 3; ++i) x[i] = step(h3, w[i], w[3 + i], 8);
  y[0] = step(h2, x[0], x[2], 4);
  y[1] = step(h2, x[1], 0.f, 4);
  const float z = step(h1, y[0], y[1], 2);
  // lanes 4 + 2 of each eight (and every odd lane) hold nothing of their own
  *component = (lane & 1) || (h2 && h1) ? -1 : (h4 ? 6 : 0) + (h3 ? 3 : 0) + (h2 ? 2 : 0) + (h1 ? 1 : 0);
  return z + __shfl_xor_sync(0xffffffffu, z, 1);
}

// The twelve products of one pair into a right-hand side's sums; m: m0, mt(3),
// ms(3), mts; c: a, beta(3), sigma, d.
__device__ __forceinline__ void near_accumulate(cf* a, const cf* m, const cf* c) {
  cfma(a[0], c[0], m[7]);
  cfma(a[0], c[1], m[1]);
  cfma(a[0], c[2], m[2]);
  cfma(a[0], c[3], m[3]);
  cfma(a[1], c[0], m[4]);
  cfma(a[1], c[1], m[0]);
  cfma(a[2], c[0], m[5]);
  cfma(a[2], c[2], m[0]);
  cfma(a[3], c[0], m[6]);
  cfma(a[3], c[3], m[0]);
  cfma(a[4], c[4], m[0]);
  cfma(a[5], c[5], m[0]);
}

// A source's six staged coefficients, source by source in shared memory: three
// 16-byte loads, and eight lanes at 48 bytes apart meet every bank once.
__device__ __forceinline__ void load_coefs(const cf* src, cf* c) {
  const float4* p = reinterpret_cast<const float4*>(src);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float4 v = p[k];
    c[2 * k] = mk<float>(v.x, v.y);
    c[2 * k + 1] = mk<float>(v.z, v.w);
  }
}

// a1, float near part, one right-hand side: one block per leaf box (grid
// stride over boxes).  Every test triangle of a box runs over the same source
// list (the concatenated source ranges of its near boxes), so the block stages
// those sources' coefficients in shared memory ([stage][6], dynamic shared
// memory), and its warps take
// the box's test triangles in turn, lanes over the row as in k_near (lane j,
// j + 32, ...): the same operations in the same order as in k_near, so the same
// result to the last bit.  nsplit shares a box's test triangles among several
// blocks when the leaf boxes alone do not fill the SMs.  Rows longer than stage read
// the coefficients from global memory instead (near_box_stage).
// Half-precision records reach shared memory by cp.async kNearAhead steps of 32
// entries ahead, across rows: 327,680 triangles 607 -> 540 us (loads of four
// records at a time left the memory idle at every row's end; float moments read
// 94 % of the copy rate as they are).
constexpr int kNearAhead = 3;
constexpr int kNearBoxThreads = 128;  // 256 measured 8 % slower (FP32H)
constexpr size_t kNearSmemMax = 232448;  // what a block may have: 227 KB
template <bool H16>
constexpr size_t near_box_smem(int stage) {
  return size_t(6) * stage * sizeof(cf) + (H16 ? size_t(4) * (kNearAhead + 1) * 64 * sizeof(uint4) : 0);
}
// Sources staged, one size for all boxes: the longest row while that pays, for long
// rows take blocks off every SM, short ones' too, and room from the far part.  Float
// moments: up to 1344 sources, three blocks an SM and 60 KB of first-level cache
// (81,920 triangles, rows of 838 to 1311: 1.28 ms, 1.33 from global memory; up to
// 1541: 2.17, 1.71; 2947: 4.90, 2.74); up to 2400, two blocks, where one box is the
// critical path (cylinder of 40,960 triangles, rows to 2030 and one box with 2.7
// times an SM's share of the pairs: 1.48, 1.88).  Half records, whose loads hide less: as
// many as fit (up to 1541: 1.03, 1.64; 2947: 2.48, 2.50, the product 2.72, 4.30).
// Beyond, the short rows only, at six blocks an SM, where they hold half of the
// pairs (327,680 triangles of rows near 270 and 5120 of rows to 2377: the product
// 11.4 ms with the longest row staged, 10.0 with short rows, 10.1 with none), else
// none: the first-level cache then has the memory (rows of 3244 to 5170: near part
// 12.5 ms with those staged that fit, 5.0 with room for 512 sources, 4.6 with none).
constexpr int kNearFloatRow = 1344, kNearPathRow = 2400;
template <bool H16>
static int near_box_stage(const Problem& pr) {
  const int fit = int((kNearSmemMax - near_box_smem<H16>(0)) / (6 * sizeof(cf))) / 32 * 32;
  const bool path = 2 * pr.box_pairs * pr.nsm > 3 * pr.nnz;  // 1.5 times an SM's share
  const int64_t most = H16 ? fit : path ? kNearPathRow : kNearFloatRow;
  const int64_t row = pr.max_row <= most ? pr.max_row : 2 * pr.short_pairs >= pr.nnz ? pr.short_row : 0;
  return int((row + 31) / 32 * 32);
}

template <typename Rio, bool H16>
__global__ void __launch_bounds__(kNearBoxThreads, 6)
    k_near_box(int64_t nleaf, int nsplit, int stage, int64_t nnz, const int32_t* __restrict__ leaf_start,
               const int32_t* __restrict__ near_ptr, const int32_t* __restrict__ near_idx,
               const int32_t* __restrict__ near_off, const int64_t* __restrict__ row_ptr,
               const cf* __restrict__ mom, const __half2* __restrict__ momh, MomScale msc,
               const cf* __restrict__ coef, float mu0, C2<Rio>* __restrict__ pot, int64_t sc = 0, int64_t sp = 0) {
  extern __shared__ __align__(16) unsigned char near_smem[];
  constexpr int NS = kNearAhead + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  uint4* ring = reinterpret_cast<uint4*>(near_smem) + warp * NS * 64;  // [NS][64 half records]
  cf* cs = reinterpret_cast<cf*>(near_smem + (H16 ? size_t(4) * NS * 64 * sizeof(uint4) : 0));  // [stage][6]
  coef += blockIdx.y * sc;
  pot += blockIdx.y * sp;
  for (int64_t bi = blockIdx.x; bi < nleaf * nsplit; bi += gridDim.x) {
    const int64_t b = bi / nsplit;
    const int q0 = near_ptr[b], q1 = near_ptr[b + 1];
    const int t0 = leaf_start[b], t1 = leaf_start[b + 1];
    const int64_t base = row_ptr[t0];
    const int len = int(row_ptr[t0 + 1] - base);
    const bool staged = len <= stage;
    __syncthreads();  // the previous box's readers are done with cs
    if (staged) {
      int qi = q0;  // j grows: the cursor only moves forward
      for (int i = threadIdx.x; i < 3 * len; i += blockDim.x) {  // thirds of a source's 48 bytes
        const int j = i / 3;
        while (qi + 1 < q1 && near_off[qi + 1] <= j) ++qi;
        const cf* src = coef + 6 * (int64_t(leaf_start[near_idx[qi]]) + (j - near_off[qi])) + 2 * (i % 3);
        cp_async(reinterpret_cast<float4*>(cs) + i, reinterpret_cast<const float4*>(src));
      }
    }
    cp_async_wait_all();
    __syncthreads();
    const int tfirst = t0 + int(bi % nsplit) * nwarp + warp, tstep = nwarp * nsplit;
    // the (row, 32 entries) step after the last one sent on its way, and its slot
    int ft = tfirst, fi = 0, fslot = 0;
    const int per_row = (len + 31) / 32;
    auto fetch = [&] {
      // the step's records as 16-byte halves, 32 consecutive ones a copy (whole sectors)
      const int n = ft < t1 ? 2 * min(32, len - 32 * fi) : 0;
      const uint4* src = reinterpret_cast<const uint4*>(momh) + 2 * (base + int64_t(ft - t0) * len + 32 * fi);
#pragma unroll
      for (int c = lane; c < 64; c += 32)
        if (c < n) cp_async(ring + fslot * 64 + c, src + c);
      cp_async_commit();
      fslot = (fslot + 1) % NS;
      if (++fi == per_row) fi = 0, ft += tstep;
    };
    int slot = 0;
    if constexpr (H16)
#pragma unroll
      for (int d = 0; d < kNearAhead; ++d) fetch();
    for (int t = tfirst; t < t1; t += tstep) {
      const int64_t e0 = base + int64_t(t - t0) * len;
      cf acc[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) acc[i] = mk<float>(0, 0);
      int qi = q0;
      // entry j's moments against its six source coefficients (a cursor on the
      // near box that holds j when they are not staged; j never decreases from
      // one call to the next)
      auto entry = [&](int j, const cf* m) {
        cf c[6];
        if (staged) {
          load_coefs(cs + 6 * j, c);
        } else {
          while (qi + 1 < q1 && near_off[qi + 1] <= j) ++qi;
          const cf* src = coef + 6 * (int64_t(leaf_start[near_idx[qi]]) + (j - near_off[qi]));
#pragma unroll
          for (int k = 0; k < 6; ++k) c[k] = src[k];
        }
        near_accumulate(acc, m, c);
      };
      if constexpr (H16) {
        for (int i = 0; i < per_row; ++i) {
          cp_async_wait<kNearAhead - 1>();
          __syncwarp();  // the step's records are here, and the slot before is read
          fetch();
          const int j = 32 * i + lane;
          if (j < len) {
            const uint4 lo = ring[slot * 64 + 2 * lane], hi = ring[slot * 64 + 2 * lane + 1];
            cf m[kMom];
            unpack_half<float>(lo, hi, msc, m);
            entry(j, m);
          }
          slot = (slot + 1) % NS;
        }
      } else {
        // entries j and j + 32 loaded together (twice the loads in flight),
        // accumulated in the order j, j + 32 of the one-entry loop
        for (int j = lane; j < len; j += 64) {
          cf ma[kMom], mb[kMom];
          const bool two = j + 32 < len;
#pragma unroll
          for (int q = 0; q < kMom; ++q) ma[q] = mom[q * nnz + e0 + j];
          if (two)
#pragma unroll
            for (int q = 0; q < kMom; ++q) mb[q] = mom[q * nnz + e0 + j + 32];
          entry(j, ma);
          if (two) entry(j + 32, mb);
        }
      }
      int i;
      const float v = warp_sum12(acc, lane, &i);
      if (i >= 0) reinterpret_cast<Rio*>(pot + 6 * int64_t(t))[i] = Rio(i < 8 ? mu0 * v : v);
    }
    if constexpr (H16) cp_async_wait_all();  // (steps past the last row: nothing in them)
  }
}

// a1, float near part, RB = 2 or 4 right-hand sides (blockIdx.y: groups of
// them): each moment is read once for all of them.  The block's eight warps take
// eight of a leaf box's test triangles at a time, a row each, and walk the box's
// source list together, kNearChunk sources a step: the step's coefficients
// ([RB][kNearChunk][6]) come in by cp.async while the step before is multiplied,
// so rows of any length take the same 50 KB.  (Whole rows in shared memory, 1100
// sources and four columns, left one block of an SM and no room beside the far
// part's kernels; coefficients from global memory cost 12 cache lines a load.)
// Lanes meet their entries in k_near's order: the same result to the last bit.
// Moments are kNearChunkSlots - 1 steps of 32 entries ahead, across rows.  Eight
// columns of a cylinder of 40,960 triangles: 3.3 -> 2.1 ms alone, the product 6.7 ->
// 4.84 ms.
constexpr int kNearChunk = 128, kNearChunkThreads = 256, kNearChunkSlots = 3;
template <bool H16, int RB>
constexpr size_t near_chunk_smem() {
  return size_t(2) * RB * 6 * kNearChunk * sizeof(cf) +
         size_t(kNearChunkThreads) * kNearChunkSlots * (H16 ? 2 * sizeof(uint4) : kMom * sizeof(cf));
}
template <typename Rio, bool H16, int RB>
__global__ void __launch_bounds__(kNearChunkThreads, 2)
    k_near_chunk(int64_t nleaf, int nsplit, int64_t nnz, const int32_t* __restrict__ leaf_start,
                 const int32_t* __restrict__ near_ptr, const int32_t* __restrict__ near_idx,
                 const int32_t* __restrict__ near_off, const int64_t* __restrict__ row_ptr,
                 const cf* __restrict__ mom, const __half2* __restrict__ momh, MomScale msc,
                 const cf* __restrict__ coef, float mu0, C2<Rio>* __restrict__ pot, int nrhs, int64_t sc, int64_t sp) {
  extern __shared__ __align__(16) unsigned char near_smem[];
  constexpr int CH = kNearChunk, TH = kNearChunkThreads, NW = TH / 32, NS = kNearChunkSlots;
  // moments on their way: half records [warp][NS][64 halves], or planes
  // [NS][plane][thread] (each thread its own entries)
  uint4* rh = reinterpret_cast<uint4*>(near_smem) + (threadIdx.x >> 5) * NS * 64;
  cf* rf = reinterpret_cast<cf*>(near_smem) + threadIdx.x;
  cf* cs = reinterpret_cast<cf*>(near_smem + near_chunk_smem<H16, RB>()) - 2 * RB * 6 * CH;  // [2][RB][CH][6]
  const int r0 = blockIdx.y * RB, nr = min(RB, nrhs - r0);  // right-hand sides r0 .. r0 + nr - 1
  coef += r0 * sc;
  pot += r0 * sp;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t bi = blockIdx.x; bi < nleaf * nsplit; bi += gridDim.x) {
    const int64_t b = bi / nsplit;
    const int q0 = near_ptr[b], q1 = near_ptr[b + 1];
    const int t0 = leaf_start[b], t1 = leaf_start[b + 1], tstep = NW * nsplit;
    const int64_t base = row_ptr[t0];
    const int len = int(row_ptr[t0 + 1] - base), nchunk = (len + CH - 1) / CH, per_row = (len + 31) / 32;
    const int tg0 = t0 + int(bi % nsplit) * NW;
    // the (row, 32 entries) step after the last one sent on its way, and its slot
    int ft = tg0 + warp, fi = 0, fslot = 0;
    auto fetch = [&] {
      const int n = ft < t1 ? min(32, len - 32 * fi) : 0;
      const int64_t e = base + int64_t(ft - t0) * len + 32 * fi;
      if constexpr (H16) {
        const uint4* src = reinterpret_cast<const uint4*>(momh) + 2 * e;
#pragma unroll
        for (int h = lane; h < 64; h += 32)
          if (h < 2 * n) cp_async(rh + fslot * 64 + h, src + h);
      } else if (lane < n) {
#pragma unroll
        for (int q = 0; q < kMom; ++q) cp_async(rf + (kMom * fslot + q) * TH, mom + q * nnz + e + lane);
      }
      cp_async_commit();
      fslot = (fslot + 1) % NS;
      if (++fi == per_row) fi = 0, ft += tstep;
    };
    int qi = q0, buf = 0;
    auto stage = [&](int c, int to) {
      if (c == 0) qi = q0;
      float4* dst = reinterpret_cast<float4*>(cs + to * (RB * 6 * CH));
      for (int i = threadIdx.x; i < 3 * CH; i += TH) {  // thirds of a source's 48 bytes
        const int j = c * CH + i / 3;
        if (j >= len) break;
        while (qi + 1 < q1 && near_off[qi + 1] <= j) ++qi;
        const cf* src = coef + 6 * (int64_t(leaf_start[near_idx[qi]]) + (j - near_off[qi])) + 2 * (i % 3);
        for (int r = 0; r < nr; ++r) cp_async(dst + r * 3 * CH + i, reinterpret_cast<const float4*>(src + r * sc));
      }
    };
    __syncthreads();  // the previous box's readers are done
    int slot = 0;
    if (tg0 < t1) {
      stage(0, 0);  // (in the group of the first fetch)
#pragma unroll
      for (int d = 0; d < NS - 1; ++d) fetch();
    }
    for (int tg = tg0; tg < t1; tg += tstep) {
      const int t = tg + warp;
      cf acc[RB][6];
#pragma unroll
      for (int r = 0; r < RB; ++r)
#pragma unroll
        for (int i = 0; i < 6; ++i) acc[r][i] = mk<float>(0, 0);
      for (int c = 0; c < nchunk; ++c) {
        const int n = min(CH, len - c * CH);
        // the chunk's coefficients came with the first fetch of the chunk before,
        // four fetches ago unless that was a row's short last chunk
        if (c > 0)
          cp_async_wait<NS - 1>();
        else
          cp_async_wait_all();
        __syncthreads();  // every thread's part of them is here, the other buffer has been read
        if (c + 1 < nchunk)
          stage(c + 1, buf ^ 1);
        else if (tg + tstep < t1)
          stage(0, buf ^ 1);
        const cf* cc = cs + buf * (RB * 6 * CH);
        for (int i = 0; i < n; i += 32) {
          cp_async_wait<NS - 2>();
          __syncwarp();  // the step's moments are here, and the slot before is read
          fetch();
          const int j = i + lane;
          if (t < t1 && j < n) {
            cf m[kMom];
            if constexpr (H16) {
              unpack_half<float>(rh[slot * 64 + 2 * lane], rh[slot * 64 + 2 * lane + 1], msc, m);
            } else {
#pragma unroll
              for (int q = 0; q < kMom; ++q) m[q] = rf[(kMom * slot + q) * TH];
            }
#pragma unroll
            for (int r = 0; r < RB; ++r)
              if (r < nr) {
                cf x[6];
                load_coefs(cc + (r * CH + j) * 6, x);
                near_accumulate(acc[r], m, x);
              }
          }
          slot = (slot + 1) % NS;
        }
        buf ^= 1;
      }
      if (t < t1)
#pragma unroll
        for (int r = 0; r < RB; ++r) {
          if (r >= nr) break;
          int i;
          const float v = warp_sum12(acc[r], lane, &i);
          if (i >= 0) reinterpret_cast<Rio*>(pot + r * sp + 6 * int64_t(t))[i] = Rio(i < 8 ? mu0 * v : v);
        }
    }
    cp_async_wait_all();  // (steps past the last row: nothing in them)
  }
}

// Raises the instance's shared-memory limit once per device (the attribute
// belongs to the current device's copy of the kernel).
static bool device_done(std::atomic<uint64_t>& mask, int* bit) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    *bit = -1;
    return false;
  }
  *bit = dev;
  return (mask.load() >> dev) & 1u;
}

template <typename K>
static pie_status raise_smem(K* kernel, size_t bytes) {
  return cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes)),
                    "near smem attribute");
}
template <typename Rio, bool H16>
static pie_status near_float_prepare() {
  static std::atomic<uint64_t> done{0};
  int bit = -1;
  if (device_done(done, &bit)) return PIE_OK;
  pie_status s = raise_smem(k_near_box<Rio, H16>, kNearSmemMax);
  if (s == PIE_OK) s = raise_smem(k_near_chunk<Rio, H16, 2>, near_chunk_smem<H16, 2>());
  if (s == PIE_OK) s = raise_smem(k_near_chunk<Rio, H16, 4>, near_chunk_smem<H16, 4>());
  if (s == PIE_OK && bit >= 0) done.fetch_or(uint64_t(1) << bit);
  return s;
}

// a1, PIE_FP64: near part in fixed point (near_fixed.cuh).  A block per (leaf
// box, share of its test triangles) and right-hand side (blockIdx.y), grid
// stride over the pairs: the box's source coefficients are staged as
// integers kFixedStage at a time, then its warps take the test triangles in
// turn, lanes over the row.  nsplit shares a box among several blocks when the
// leaf boxes alone do not fill the SMs.  81,920 triangles: 0.68 ms alone (2.2 ms
// with FP64 multiply-adds), 24,576 of a cube: 0.65 ms (1.78); beside the far part
// one block an SM does, since the two use different pipes: the product of 81,920
// triangles 2.7 to 2.9 ms (5.1 with FP64 multiply-adds).

// A product's limbs: hh += h h', x += h l' + l h'; s[0], s[1]: real and imaginary
// part of c times one part of the moment, m = (h, l).
struct FixedSum {
  int64_t hh, x;
};
__device__ __forceinline__ void fixed_cfma(FixedSum* s, const int4& c, const int2& m) {
  s[0].hh += int64_t(c.x) * m.x;
  s[1].hh += int64_t(c.z) * m.x;
  s[0].x += int64_t(c.x) * m.y;
  s[1].x += int64_t(c.z) * m.y;
  s[0].x += int64_t(c.y) * m.x;
  s[1].x += int64_t(c.w) * m.x;
}

// Entries j0 .. j1 of row t in double, for a stage with a coefficient that is
// not finite: lane i < 12 returns component i of the six sums.
__device__ __noinline__ double near_row_double(const FixedNear& nf, int64_t nnz, int64_t t, int b, int64_t e0, int j0,
                                               int j1, int q0, int q1, const int32_t* leaf_start,
                                               const int32_t* near_idx, const int32_t* near_off, const cd* coef) {
  const int lane = threadIdx.x & 31;
  cd acc[6];
  for (int i = 0; i < 6; ++i) acc[i] = mk<double>(0, 0);
  int qi = q0;
  for (int j = j0 + lane; j < j1; j += 32) {
    while (qi + 1 < q1 && near_off[qi + 1] <= j) ++qi;
    const cd* c = coef + 6 * (int64_t(leaf_start[near_idx[qi]]) + (j - near_off[qi]));
    cd m[kMom];
    for (int q = 0; q < kMom; ++q) m[q] = fixed_moment(nf, nnz, q, e0 + j, t, b);
    cfma(acc[0], c[0], m[7]);
    for (int d = 0; d < 3; ++d) {
      cfma(acc[0], c[1 + d], m[1 + d]);
      cfma(acc[1 + d], c[0], m[4 + d]);
      cfma(acc[1 + d], c[1 + d], m[0]);
    }
    cfma(acc[4], c[4], m[0]);
    cfma(acc[5], c[5], m[0]);
  }
  double out = 0;
  for (int i = 0; i < 12; ++i) {
    const double v = warp_sum(i % 2 ? acc[i / 2].y : acc[i / 2].x);
    if (lane == i) out = v;
  }
  return out;
}

// PARTS: moments' parts of a pass over the row.  Both at once take 48 sums and 166
// registers, one after the other 24 and 128 and the coefficients from shared memory
// twice: 81,920 triangles alone 0.68 ms, 0.72, but beside the far part, whose
// kernels the registers hold up, the product 2.97 ms, 2.88.  BLOCKS: blocks of an SM that
// the registers allow.  Shared memory: the stage's coefficients [6][kFixedStage], then
// per warp SLOTS buffers of 32 entries' moments [PARTS][4][32], as much for either
// number (with 61 KB a block three fit, and blocks pile up on some SMs beside the far
// part: products of 81,920 triangles in a row 3.57 ms, 2.69).
constexpr int kFixedWarps = 4;
constexpr size_t kFixedSmem = sizeof(int4) * (6 * kFixedStage + kFixedWarps * 4 * kFixedPlanes * 32);

template <int PARTS, int BLOCKS>
__global__ void __launch_bounds__(32 * kFixedWarps, BLOCKS)
    k_near_fixed(int64_t nleaf, int nsplit, int64_t nnz, const int32_t* __restrict__ leaf_start,
                 const int32_t* __restrict__ near_ptr, const int32_t* __restrict__ near_idx,
                 const int32_t* __restrict__ near_off, const int64_t* __restrict__ row_ptr, const FixedNear nf,
                 const cd* __restrict__ coef, double mu0, cd* __restrict__ pot, int64_t sc = 0, int64_t sp = 0) {
  constexpr int PASSES = 2 / PARTS, PLANES = kFixedPlanes * PARTS, SLOTS = 4 / PARTS;
  extern __shared__ __align__(16) unsigned char fixed_smem[];
  int4(*cs)[kFixedStage] = reinterpret_cast<int4(*)[kFixedStage]>(fixed_smem);
  __shared__ int fields[kFixedWarps][8];  // [warp][part of a, beta, sigma, d]
  coef += blockIdx.y * sc;
  double* out = reinterpret_cast<double*>(pot + blockIdx.y * sp);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int4(*ms)[PLANES][32] = reinterpret_cast<int4(*)[PLANES][32]>(cs + 6) + SLOTS * warp;
  for (int64_t bi = blockIdx.x; bi < nleaf * nsplit; bi += gridDim.x) {
    const int64_t b = bi / nsplit;
    const int q0 = near_ptr[b], q1 = near_ptr[b + 1];
    const int t0 = leaf_start[b] + int(bi % nsplit) * kFixedWarps + warp, t1 = leaf_start[b + 1];
    const int len = int(row_ptr[leaf_start[b] + 1] - row_ptr[leaf_start[b]]);
    const int dl = nf.delta[b];
    for (int j0 = 0; j0 < len; j0 += kFixedStage) {
      const int j1 = min(len, j0 + kFixedStage);
      // largest exponent fields of the stage's a, beta, sigma, d: real and imaginary parts
      int x[8] = {1, 1, 1, 1, 1, 1, 1, 1};
      int qi = q0;
      for (int j = j0 + int(threadIdx.x); j < j1; j += blockDim.x) {
        while (qi + 1 < q1 && near_off[qi + 1] <= j) ++qi;
        const cd* c = coef + 6 * (int64_t(leaf_start[near_idx[qi]]) + (j - near_off[qi]));
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const cd v = c[k];
          const int g = 2 * (k == 0 ? 0 : k < 4 ? 1 : k - 2);
          x[g] = max(x[g], exponent_field(v.x));
          x[g + 1] = max(x[g + 1], exponent_field(v.y));
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = __reduce_max_sync(0xffffffffu, x[i]);
      __syncthreads();  // the previous stage's readers are done
      if (lane == 0)
#pragma unroll
        for (int i = 0; i < 8; ++i) fields[warp][i] = x[i];
      __syncthreads();
      int top = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
#pragma unroll
        for (int w = 0; w < kFixedWarps; ++w) x[i] = max(x[i], fields[w][i]);
        top = max(top, x[i]);
      }
      const bool finite = top < 0x7ff;
      // beta's field covers a and delta; a takes beta's less delta
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        x[2 + p] = max(x[2 + p], x[p] + dl);
        x[p] = x[2 + p] - dl;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] += 53 - kCoefBits;
      qi = q0;
      for (int j = j0 + int(threadIdx.x); j < j1 && finite; j += blockDim.x) {
        while (qi + 1 < q1 && near_off[qi + 1] <= j) ++qi;
        const cd* c = coef + 6 * (int64_t(leaf_start[near_idx[qi]]) + (j - near_off[qi]));
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const cd v = c[k];
          const int g = 2 * (k == 0 ? 0 : k < 4 ? 1 : k - 2);
          const int2 r = fixed_encode(v.x, x[g]), i = fixed_encode(v.y, x[g + 1]);
          cs[k][j - j0] = make_int4(r.x, r.y, i.x, i.y);
        }
      }
      __syncthreads();
      // the warp's (test triangle, pass, 32 entries) steps in one sequence: the next
      // steps' moments are on their way while a step is multiplied, across rows
      // too (rows of a box have one length, one after the other); a lane copies
      // and reads its own entry
      const int64_t base = row_ptr[leaf_start[b]];
      const int count = j1 - j0, tstep = kFixedWarps * nsplit;
      int ft = t0, fp = 0, fj = lane, fslot = 0;
      // the pass's first entry of the row, and how far the next row's lies from there
      const int4* src = nf.mom + base + int64_t(t0 - leaf_start[b]) * len + j0;
      const int64_t next_row = int64_t(tstep) * len - (PASSES - 1) * PLANES * nnz;
      auto fetch = [&] {
        if (fj < count && ft < t1 && finite) {
          const int4* from = src + fj;
#pragma unroll
          for (int g = 0; g < PLANES; ++g, from += nnz) cp_async(&ms[fslot][g][lane], from);
        }
        cp_async_commit();
        fslot = fslot + 1 == SLOTS ? 0 : fslot + 1;
        fj += 32;
        if (fj - lane >= count) {
          fj = lane;
          const bool next = fp + 1 == PASSES;
          src += next ? next_row : PLANES * nnz;
          ft += next ? tstep : 0;
          fp = next ? 0 : fp + 1;
        }
      };
      // exponent of the coefficients in the lane's sum
      const int ec = (lane & 1 ? (lane < 8 ? x[3] : lane < 10 ? x[5] : x[7])
                               : (lane < 8 ? x[2] : lane < 10 ? x[4] : x[6])) - 1075;
      int slot = 0;
      // a pass over row t, part and (PARTS = 2) the next: lane i < 12 gets the value of
      // sum i of the (re c + i im c) (re m + i im m) so far, v of the passes before
      auto pass = [&](int t, int part, double v) {
        FixedSum sum[PARTS][12];
#pragma unroll
        for (int i = 0; i < 12 * PARTS; ++i) sum[i / 12][i % 12] = FixedSum{0, 0};
        for (int j = lane; j - lane < count; j += 32) {
          fetch();
          cp_async_wait<SLOTS - 1>();
          if (j < count) {
            int2 m[PARTS][kMom];
#pragma unroll
            for (int g = 0; g < PLANES; ++g) {
              const int4 w = ms[slot][g][lane];
              m[g / kFixedPlanes][2 * (g % kFixedPlanes)] = make_int2(w.x, w.y);
              m[g / kFixedPlanes][2 * (g % kFixedPlanes) + 1] = make_int2(w.z, w.w);
            }
            // (one coefficient after the other: the sums fill the registers)
            auto product = [&](int i, const int4& c, int q) {
#pragma unroll
              for (int u = 0; u < PARTS; ++u) fixed_cfma(&sum[u][2 * i], c, m[u][q]);
            };
            const int4 a = cs[0][j];
            product(0, a, 7);
            product(1, a, 4);
            product(2, a, 5);
            product(3, a, 6);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              const int4 c = cs[1 + d][j];
              product(0, c, 1 + d);
              product(1 + d, c, 0);
            }
            product(4, cs[4][j], 0);
            product(5, cs[5][j], 0);
          }
          slot = slot + 1 == SLOTS ? 0 : slot + 1;
        }
        const FixedRow row = nf.row[t];
#pragma unroll
        for (int u = 0; u < PARTS; ++u) {
          // value = hh 2^56 + x 2^28: x carried into hh but for 28 bits below it, and
          // the warp's totals in pieces of 27 bits
          int p0 = 0, p1 = 0, p2 = 0, p3 = 0;
#pragma unroll
          for (int i = 0; i < 12; ++i) {
            const FixedSum& s = sum[u][i];
            const int64_t h = s.hh + (s.x >> kLimb);
            const int r0 = int(__reduce_add_sync(0xffffffffu, (uint32_t(s.x) & ((1u << kLimb) - 1)) >> 1));
            const int r1 = int(__reduce_add_sync(0xffffffffu, uint32_t(h) & ((1u << 27) - 1)));
            const int r2 = int(__reduce_add_sync(0xffffffffu, uint32_t(h >> 27) & ((1u << 27) - 1)));
            const int r3 = __reduce_add_sync(0xffffffffu, int(h >> 54));
            if (lane == i) p0 = r0, p1 = r1, p2 = r2, p3 = r3;
          }
          // 96 bits: the totals above the point less five bits, then 5 + 27 bits
          const uint64_t mid = (uint64_t(uint32_t(p2)) << 27) + uint32_t(p1);
          const uint64_t low = uint64_t(uint32_t(p0)) + ((mid & 31) << 27);
          const int64_t hi = int64_t(p3) * (int64_t(1) << 49) + int64_t(mid >> 5) + int64_t(low >> 32);
          const bool im = part + u;
          const int em = lane < 2 ? (im ? row.mt[1] : row.mt[0]) : im ? row.m0[1] : row.m0[0];
          const double w = fixed_scale(hi, uint32_t(low), em + ec + 2 * kLimb - 27);
          const double other = __shfl_xor_sync(0xffffffffu, w, 1);
          v = im ? v + (lane & 1 ? other : -other) : w;  // i im m: the parts change places
        }
        return row.m0[0] == kFixedNan ? nan("") : v;
      };
#pragma unroll
      for (int d = 0; d < SLOTS - 1; ++d) fetch();
      for (int t = t0; t < t1; t += tstep) {
        const int64_t e0 = base + int64_t(t - leaf_start[b]) * len;
        double v = 0;
        if (finite) {
#pragma unroll 1
          for (int part = 0; part < 2; part += PARTS) v = pass(t, part, v);
        } else {
          v = near_row_double(nf, nnz, t, int(b), e0, j0, j1, q0, q1, leaf_start, near_idx, near_off, coef);
        }
        if (lane < 12) {
          if (lane < 8) v *= mu0;
          out[12 * int64_t(t) + lane] = j0 ? out[12 * int64_t(t) + lane] + v : v;
        }
      }
      cp_async_wait_all();  // (the step past the last row: nothing in it)
    }
  }
}

static pie_status near_fixed_prepare() {
  static std::atomic<uint64_t> done{0};
  int bit = -1;
  if (device_done(done, &bit)) return PIE_OK;
  pie_status s = raise_smem(k_near_fixed<2, 3>, kFixedSmem);
  if (s == PIE_OK) s = raise_smem(k_near_fixed<1, 4>, kFixedSmem);
  if (s == PIE_OK && bit >= 0) done.fetch_or(uint64_t(1) << bit);
  return s;
}

// Launch of the fixed-point near part for nrhs columns on a grid of at most
// max_blocks (0: no bound).  lean: the kernel of fewer registers.
static void near_fixed(const Problem& pr, const cd* coef, cd* pot, int nrhs, int64_t max_blocks, bool lean,
                       cudaStream_t st) {
  const FixedNear nf{static_cast<const int4*>(pr.mom), static_cast<const FixedRow*>(pr.fixed_row), pr.fixed_delta};
  // shares per box: the least rounds of three blocks an SM over all columns, staging
  // (about 1/50 of a box's rows) once a share; at least a test triangle for each warp.  Boxes
  // are uneven, so up to 8 % more by this count for finer shares, while a warp has
  // three rows (alone: cube of 24,576 triangles 799 -> 695 us, ellipsoid of 32,768
  // 2870 -> 1400; finer still, spheres lose 10 %)
  const int64_t slots = 3 * int64_t(pr.nsm),
                most = std::min<int64_t>(16, (pr.T / pr.nleaf + kFixedWarps - 1) / kFixedWarps);
  int nsplit = 1;
  double best = 0, costs[17];
  for (int64_t s = 1; s <= most; ++s) {
    const double cost = double((pr.nleaf * nrhs * s + slots - 1) / slots) * (1.0 / double(s) + 0.02);
    if (s == 1 || cost < best) best = cost, nsplit = int(s);
    costs[s] = cost;
  }
  for (int64_t s = nsplit + 1; s <= most && 3 * kFixedWarps * s <= pr.T / pr.nleaf; ++s)
    if (costs[s] <= 1.08 * best) nsplit = int(s);
  int64_t grid = pr.nleaf * nsplit;
  if (max_blocks > 0) grid = std::min(grid, max_blocks);
  auto kernel = lean ? k_near_fixed<1, 4> : k_near_fixed<2, 3>;
  kernel<<<dim3(unsigned(grid), unsigned(nrhs)), 32 * kFixedWarps, kFixedSmem, st>>>(
      pr.nleaf, nsplit, pr.nnz, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr, nf, coef, kMu0, pot,
      6 * pr.T, 6 * pr.T);
}

// Antipode of half-grid sample q (theta rows 0..ntheta/2-1): -khat_q is
// the sample (ntheta-1-i, j+ntheta mod 2 ntheta).
__device__ __forceinline__ int antipode(int q, int ntheta) {
  int nphi = 2 * ntheta;
  int i = q / nphi, j = q % nphi;
  return (ntheta - 1 - i) * nphi + (j + ntheta) % nphi;
}

// Largest block of a per-box far kernel, as its registers allow (up to 64 a
// thread: 1024 threads, up to 80: 768).  The orchestration packs no more rows into
// a block; an angular grid whose one row is wider (20 and 22 theta rows) takes the
// kernel's WIDE form, held to 64 registers.  Asked of the kernel and not set by launch
// bounds: bounds of 1024 cost the float aggregation 61 -> 94 us at 327,680
// triangles, although its 62 registers meet them.
template <auto Kernel>
static int max_threads() {
  static std::atomic<int> most{0};
  if (const int n = most.load()) return n;
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, Kernel) != cudaSuccess) {
    cudaGetLastError();
    return 512;  // the widest row of any of them but WIDE ones
  }
  most.store(a.maxThreadsPerBlock);
  return a.maxThreadsPerBlock;
}
constexpr int kWideThreads = 1024;

// a2: leaf aggregation.  One block per leaf box, one thread per half-grid
// sample q.  The radiation tables are stored for the half grid only, since
// Pi(-khat) = conj(Pi(khat)) and M(-khat) = conj(M(khat)); with c X = c Xr +
// i c Xi the pair of samples is S(q) = A + iB, S(-q) = A - iB, where
// A = sum c Xr and B = sum c Xi.
// Small angular grids pack several boxes into one block (threadIdx.y).
template <typename Rf>
__global__ void k_agg(int P, int ntheta, int64_t nb, const int32_t* __restrict__ leaf_start,
                      const C2<Rf>* __restrict__ Pi, const C2<Rf>* __restrict__ M, const C2<Rf>* __restrict__ coef,
                      Rf mu0, C2<Rf>* __restrict__ S, int64_t sc = 0, int64_t sS = 0) {
  const int64_t b = int64_t(blockIdx.x) * blockDim.y + threadIdx.y;
  if (b >= nb) return;
  coef += blockIdx.y * sc;
  S += blockIdx.y * sS;
  const int Ph = P / 2;
  const int t0 = leaf_start[b], t1 = leaf_start[b + 1];
  for (int q = threadIdx.x; q < Ph; q += blockDim.x) {
    C2<Rf> A[kComp], B[kComp];
#pragma unroll
    for (int c = 0; c < kComp; ++c) A[c] = B[c] = mk<Rf>(0, 0);
    // triangle t's coefficients and table entries, then its multiply-adds;
    // in float two triangles' loads are issued together (latency-bound
    // small grids), the multiply-adds still in triangle order
    constexpr int U = sizeof(Rf) == 4 ? 2 : 1;
    struct Tri {
      C2<Rf> c[6], pi, m[3];
    };
    auto load = [&](int t, Tri& r) {
      const C2<Rf>* cf_ = coef + 6 * (int64_t)t;
#pragma unroll
      for (int k = 0; k < 6; ++k) r.c[k] = cf_[k];
      r.pi = Pi[(int64_t)t * Ph + q];
#pragma unroll
      for (int d = 0; d < 3; ++d) r.m[d] = M[((int64_t)t * 3 + d) * Ph + q];
    };
    auto accumulate = [&](const Tri& r) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        rfma(A[d], r.m[d].x, r.c[0]);
        rfma(A[d], r.pi.x, r.c[1 + d]);
        rfma(B[d], r.m[d].y, r.c[0]);
        rfma(B[d], r.pi.y, r.c[1 + d]);
      }
      rfma(A[3], r.pi.x, r.c[4]);
      rfma(B[3], r.pi.y, r.c[4]);
      rfma(A[4], r.pi.x, r.c[5]);
      rfma(B[4], r.pi.y, r.c[5]);
    };
    int t = t0;
    if constexpr (U > 1)
      for (; t + U <= t1; t += U) {
        Tri r[U];
#pragma unroll
        for (int u = 0; u < U; ++u) load(t + u, r[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) accumulate(r[u]);
      }
    for (; t < t1; ++t) {
      Tri r;
      load(t, r);
      accumulate(r);
    }
    const int qa = antipode(q, ntheta);
    C2<Rf>* o = S + (int64_t)b * kComp * P;
#pragma unroll
    for (int c = 0; c < kComp; ++c) {
      Rf f = c < 3 ? mu0 : Rf(1);
      o[c * P + q] = mk<Rf>(f * (A[c].x - B[c].y), f * (A[c].y + B[c].x));
      o[c * P + qa] = mk<Rf>(f * (A[c].x + B[c].y), f * (A[c].y - B[c].x));
    }
  }
}

// a2 with the twenty real sums of a (box, half-grid sample) shared by several
// threads: a thread per leaf box (threadIdx.y), sample (threadIdx.x) and sum --
// A with one part of c (blockIdx.z even: real, odd: imaginary) or B with the
// other (threadIdx.z) -- NC components each; the two meet in shared memory and
// give that part of S(q) and S(-q).  Every sum runs in k_agg's order.  One
// thread for all twenty leaves a small tree's few hundred warps on one SM
// scheduler each, at 67 clocks a double operation: 56 leaf boxes 51 -> 15 us,
// 272 81 -> 35 us, 4400 (double) 358 -> 336 us; from about 10,000 boxes in double
// and 9,000 in float k_agg is as fast or faster (its loads are wider).
template <typename Rf, int NC>
__global__ void k_agg_split(int P, int ntheta, int64_t nb, const int32_t* __restrict__ leaf_start,
                            const C2<Rf>* __restrict__ Pi, const C2<Rf>* __restrict__ M,
                            const C2<Rf>* __restrict__ coef, Rf mu0, C2<Rf>* __restrict__ S, int64_t sc = 0,
                            int64_t sS = 0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int X = threadIdx.z, part = blockIdx.z & 1, ri = X ? 1 - part : part, c0 = NC * int(blockIdx.z >> 1);
  const int nq = blockDim.x;
  Rf* sums = reinterpret_cast<Rf*>(smem_raw) + threadIdx.y * 2 * NC * nq + threadIdx.x;  // [A, B][component][q]
  const int64_t b = int64_t(blockIdx.x) * blockDim.y + threadIdx.y;
  const bool live = b < nb;
  const Rf* cr = reinterpret_cast<const Rf*>(coef + blockIdx.y * sc) + ri;
  const Rf* pr = reinterpret_cast<const Rf*>(Pi) + X;
  const Rf* mr = reinterpret_cast<const Rf*>(M) + X;
  const int Ph = P / 2;
  const int t0 = live ? leaf_start[b] : 0, t1 = live ? leaf_start[b + 1] : 0;
  for (int q0 = 0; q0 < Ph; q0 += nq) {
    const int q = q0 + threadIdx.x;
    Rf acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0;
    if (q < Ph) {
      // UT triangles' loads together, their multiply-adds in triangle order
      constexpr int UT = NC == 1 ? 4 : 2;
      struct Tri {
        Rf a, c[NC], pi, m[NC];
      };
      auto load = [&](int64_t t, Tri& r) {
        r.a = cr[12 * t];
        r.pi = pr[2 * (t * Ph + q)];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          r.c[c] = cr[12 * t + 2 * (1 + c0 + c)];
          if (c0 + c < 3) r.m[c] = mr[2 * ((t * 3 + c0 + c) * Ph + q)];
        }
      };
      auto accumulate = [&](const Tri& r) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          if (c0 + c < 3) acc[c] = fma(r.m[c], r.a, acc[c]);
          acc[c] = fma(r.pi, r.c[c], acc[c]);
        }
      };
      int t = t0;
      for (; t + UT <= t1; t += UT) {
        Tri r[UT];
#pragma unroll
        for (int u = 0; u < UT; ++u) load(t + u, r[u]);
#pragma unroll
        for (int u = 0; u < UT; ++u) accumulate(r[u]);
      }
      for (; t < t1; ++t) {
        Tri r;
        load(t, r);
        accumulate(r);
      }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c) sums[(X * NC + c) * nq] = acc[c];
    __syncthreads();
    if (live && q < Ph) {
      // real part: A - B at q, A + B at -q; imaginary part: A + B at q, A - B at -q
      Rf* o = reinterpret_cast<Rf*>(S + blockIdx.y * sS + (b * kComp + c0) * P + (X ? antipode(q, ntheta) : q)) + part;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const Rf f = c0 + c < 3 ? mu0 : Rf(1);
        const Rf A = sums[c * nq], B = sums[(NC + c) * nq];
        o[2 * c * P] = X == part ? f * (A - B) : f * (A + B);
      }
    }
  }
}

// a3: interpolation from level l+1 to its parents at level l:
// S_l[b] = sum_children phase_o (F S_child); one block per parent, one thread
// per sample.  The children's patterns are staged in shared memory cg at a
// time (all eight when they fit: one load latency per parent instead of one
// per child), and with fs the filter F^T too (else it is read from global
// memory); children are summed in order, whatever cg.  A thread takes NC
// components, the others threadIdx.z: five where the boxes fill the SMs, one on
// small levels.
template <typename Rf, int NC>
__device__ __forceinline__ void interp_boxes(int P, int64_t nb, const int32_t* __restrict__ child_start,
                                             const int8_t* __restrict__ oct_child, const C2<Rf>* __restrict__ Sc,
                                             const Rf* __restrict__ Ft, const C2<Rf>* __restrict__ phase,
                                             C2<Rf>* __restrict__ Sp, int64_t sSc, int64_t sSp, int cg, bool fs) {
  Sc += blockIdx.y * sSc;
  Sp += blockIdx.y * sSp;
  extern __shared__ unsigned char smem_raw[];
  // the filter (P x P, when fs) first, then one staging region of cg
  // children per threadIdx.y row (small angular grids: one parent per row)
  Rf* fsm = reinterpret_cast<Rf*>(smem_raw);
  const size_t fbytes = fs ? ((sizeof(Rf) * P * P + 15) / 16) * 16 : 0;
  C2<Rf>* sm = reinterpret_cast<C2<Rf>*>(smem_raw + fbytes) + threadIdx.y * cg * kComp * P;
  const int tid = (threadIdx.z * blockDim.y + threadIdx.y) * blockDim.x + threadIdx.x;
  const int nth = blockDim.x * blockDim.y * blockDim.z;
  const int row_tid = threadIdx.z * blockDim.x + threadIdx.x, row_nth = blockDim.x * blockDim.z, c0 = NC * threadIdx.z;
  if (fs)  // P x P reals as 8-byte words (P = 2 N_theta^2 is even)
    for (int i = tid; i < P * P * int(sizeof(Rf)) / 8; i += nth)
      cp_async(reinterpret_cast<uint2*>(fsm) + i, reinterpret_cast<const uint2*>(Ft) + i);
  const Rf* F = fs ? fsm : Ft;
  const int64_t b = int64_t(blockIdx.x) * blockDim.y + threadIdx.y;
  const bool live = b < nb;
  const int b0 = live ? child_start[b] : 0, b1 = live ? child_start[b + 1] : 0;
  const int p = threadIdx.x;
  C2<Rf> acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = mk<Rf>(0, 0);
  for (int k0 = b0;; k0 += cg) {
    const int nk = k0 < b1 ? min(cg, b1 - k0) : 0;
    if (!__syncthreads_or(nk > 0)) {  // every row of the block done
      cp_async_wait_all();            // (nothing may stay in flight at exit)
      break;
    }
    // the nk children are consecutive at level l+1: one contiguous copy
    for (int i = row_tid; i < nk * kComp * P; i += row_nth) cp_async(sm + i, Sc + (int64_t)k0 * kComp * P + i);
    cp_async_wait_all();  // (also completes the filter's copy)
    __syncthreads();
    for (int k = 0; k < nk && p < P; ++k) {
      const C2<Rf>* sk = sm + (k * kComp + c0) * P;
      C2<Rf> sum[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) sum[c] = mk<Rf>(0, 0);
#pragma unroll 4
      for (int q = 0; q < P; ++q) {
        Rf f = F[(int64_t)q * P + p];
#pragma unroll
        for (int c = 0; c < NC; ++c) rfma(sum[c], f, sk[c * P + q]);
      }
      C2<Rf> ph = phase[oct_child[k0 + k] * P + p];
#pragma unroll
      for (int c = 0; c < NC; ++c) cfma(acc[c], ph, sum[c]);
    }
  }
  if (live && p < P) {
#pragma unroll
    for (int c = 0; c < NC; ++c) Sp[((int64_t)b * kComp + c0 + c) * P + p] = acc[c];
  }
}

template <typename Rf, int NC>
__global__ void k_interp(int P, int64_t nb, const int32_t* __restrict__ child_start,
                         const int8_t* __restrict__ oct_child, const C2<Rf>* __restrict__ Sc,
                         const Rf* __restrict__ Ft, const C2<Rf>* __restrict__ phase, C2<Rf>* __restrict__ Sp,
                         int64_t sSc, int64_t sSp, int cg, bool fs) {
  interp_boxes<Rf, NC>(P, nb, child_start, oct_child, Sc, Ft, phase, Sp, sSc, sSp, cg, fs);
}
template <typename Rf, int NC>
__global__ void __launch_bounds__(kWideThreads)
    k_interp_wide(int P, int64_t nb, const int32_t* __restrict__ child_start, const int8_t* __restrict__ oct_child,
                  const C2<Rf>* __restrict__ Sc, const Rf* __restrict__ Ft, const C2<Rf>* __restrict__ phase,
                  C2<Rf>* __restrict__ Sp, int64_t sSc, int64_t sSp, int cg, bool fs) {
  interp_boxes<Rf, NC>(P, nb, child_start, oct_child, Sc, Ft, phase, Sp, sSc, sSp, cg, fs);
}

// ---- factorised filter: F is block-circulant in azimuth (its entries depend
// on phi_j - phi_j' only), so the length-NPHI DFT along phi turns it into
// one real NT x NT block K_m per azimuthal frequency m:
//   (F s)[i][j] = sum_m e^{i m phi_j} sum_i' K_m[i][i'] shat[i'][m],
//   shat[i'][m] = sum_j e^{-i m phi_j} s[i'][j],  K_m = (1/NPHI) DFT_d f_ii'(d).
// F^T uses K_m transposed.

// Structure used below (N_theta = 8, so NPHI = 16 and degrees up to 7):
//  * K_m = K_{-m}, and K_8 = 0: azimuthal order |m| <= degree <= 7, so the
//    Nyquist frequency m = 8 carries nothing;
//  * the Gauss-Legendre theta nodes are symmetric about the equator and
//    P_l^m(-x) = (-1)^(l+m) P_l^m(x), so every K_m commutes with the row
//    reflection i -> NT-1-i.  In the sums and differences of mirrored rows,
//    se_k = s_k + s_{NT-1-k}, so_k = s_k - s_{NT-1-k} (k < NT/2), K_m is two
//    (NT/2) x (NT/2) blocks:  y_i = ye_i + yo_i, y_{NT-1-i} = ye_i - yo_i with
//    ye = KE se, yo = KO so, KE_ik = (K_ik + K_i,NT-1-k)/2,
//    KO_ik = (K_ik - K_i,NT-1-k)/2.  Half the multiply-adds of the full block.

// 4-point DFT in place, X_k = sum_n x_n w^(nk), w = -i (forward) or +i.
template <bool INV, typename R>
__device__ __forceinline__ void dft4(C2<R>& a, C2<R>& b, C2<R>& c, C2<R>& d) {
  const C2<R> t0 = mk<R>(a.x + c.x, a.y + c.y), t1 = mk<R>(a.x - c.x, a.y - c.y);
  const C2<R> t2 = mk<R>(b.x + d.x, b.y + d.y), t3 = mk<R>(b.x - d.x, b.y - d.y);
  a = mk<R>(t0.x + t2.x, t0.y + t2.y);
  c = mk<R>(t0.x - t2.x, t0.y - t2.y);
  // forward: X1 = t1 - i t3, X3 = t1 + i t3 (inverse: signs swapped)
  const C2<R> p = mk<R>(t1.x + t3.y, t1.y - t3.x), q = mk<R>(t1.x - t3.y, t1.y + t3.x);
  b = INV ? q : p;
  d = INV ? p : q;
}

// v * exp(-/+ 2 pi i E / 16) for the exponents of the 16 = 4 x 4 split.
// cos(pi/8) = sqrt(2 + sqrt 2) / 2, sin(pi/8) = sqrt(2 - sqrt 2) / 2.
template <bool INV, int E, typename R>
__device__ __forceinline__ C2<R> twiddle16(C2<R> v) {
  constexpr double c8 = 0.92387953251128675613, s8 = 0.38268343236508977173, h = 0.70710678118654752440;
  constexpr double c = E == 1 ? c8 : E == 3 ? s8 : E == 9 ? -c8 : 0.0;
  constexpr double s = E == 1 ? s8 : E == 3 ? c8 : E == 9 ? -s8 : 0.0;
  const R x = v.x, y = v.y;
  if constexpr (E == 2) {  // (1 -/+ i) h
    return INV ? mk<R>(R(h) * (x - y), R(h) * (x + y)) : mk<R>(R(h) * (x + y), R(h) * (y - x));
  } else if constexpr (E == 4) {  // -/+ i
    return INV ? mk<R>(-y, x) : mk<R>(y, -x);
  } else if constexpr (E == 6) {  // (-1 -/+ i) h
    return INV ? mk<R>(-R(h) * (x + y), R(h) * (x - y)) : mk<R>(R(h) * (y - x), -R(h) * (x + y));
  } else {  // c -/+ i s
    return INV ? mk<R>(fma(x, R(c), -y * R(s)), fma(y, R(c), x * R(s)))
               : mk<R>(fma(x, R(c), y * R(s)), fma(y, R(c), -x * R(s)));
  }
}

// 16-point DFT in registers, X_k = sum_n x_n exp(-/+ 2 pi i n k / 16) (no
// scaling): n = 4 q + r, k = k1 + 4 k2; 4-point DFTs over q, twiddles
// exp(-/+ 2 pi i r k1 / 16), 4-point DFTs over r.  X is returned in out.
template <bool INV, typename R>
__device__ __forceinline__ void fft16(C2<R>* x, C2<R>* out) {
#pragma unroll
  for (int r = 0; r < 4; ++r) dft4<INV>(x[r], x[r + 4], x[r + 8], x[r + 12]);  // x[r + 4 k1] = Y_r[k1]
  x[5] = twiddle16<INV, 1>(x[5]);
  x[9] = twiddle16<INV, 2>(x[9]);
  x[13] = twiddle16<INV, 3>(x[13]);
  x[6] = twiddle16<INV, 2>(x[6]);
  x[10] = twiddle16<INV, 4>(x[10]);
  x[14] = twiddle16<INV, 6>(x[14]);
  x[7] = twiddle16<INV, 3>(x[7]);
  x[11] = twiddle16<INV, 6>(x[11]);
  x[15] = twiddle16<INV, 9>(x[15]);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) dft4<INV>(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) out[k1 + 4 * k2] = x[4 * k1 + k2];
}

constexpr int kFftBatch = 4;  // (child, component) units per warp of the factorised filter kernels

// Mirror-split blocks of K_m (or of K_m^T when TR) in shared memory:
// KE[m][i][k], KO[m][i][k], i, k < NT/2.
template <int NT, bool TR, typename Rf>
__device__ __forceinline__ void load_split_blocks(const Rf* __restrict__ Kf, Rf* KE, Rf* KO, int tid, int nth) {
  constexpr int NPHI = 2 * NT, H = NT / 2;
  for (int it = tid; it < NPHI * H * H; it += nth) {
    const int m = it / (H * H), i = (it / H) % H, k = it % H;
    const Rf* Km = Kf + m * NT * NT;
    const Rf a = TR ? Km[k * NT + i] : Km[i * NT + k];
    const Rf b = TR ? Km[(NT - 1 - k) * NT + i] : Km[i * NT + NT - 1 - k];
    KE[it] = Rf(0.5) * (a + b);
    KO[it] = Rf(0.5) * (a - b);
  }
}

// One azimuthal frequency m of one (child, component): y = K_m a over the NT
// theta rows (a strided by one in shared memory), written to out[i * BP].
template <int NT, int BP, typename Rf>
__device__ __forceinline__ void apply_split_block(const C2<Rf>* a, const Rf* KE, const Rf* KO, C2<Rf>* out) {
  constexpr int H = NT / 2;
  C2<Rf> se[H], so[H];
#pragma unroll
  for (int k = 0; k < H; ++k) {
    const C2<Rf> u = a[k], v = a[NT - 1 - k];
    se[k] = mk<Rf>(u.x + v.x, u.y + v.y);
    so[k] = mk<Rf>(u.x - v.x, u.y - v.y);
  }
#pragma unroll
  for (int i = 0; i < H; ++i) {
    C2<Rf> ye = mk<Rf>(0, 0), yo = mk<Rf>(0, 0);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      rfma(ye, KE[i * H + k], se[k]);
      rfma(yo, KO[i * H + k], so[k]);
    }
    out[i * BP] = mk<Rf>(ye.x + yo.x, ye.y + yo.y);
    out[(NT - 1 - i) * BP] = mk<Rf>(ye.x - yo.x, ye.y - yo.y);
  }
}

// Shared memory of a factorised filter block of nw warps: the mirror-split K_m
// blocks, then one region of kFftBatch spectra per warp (below 48 KB for 4).
constexpr int kFftWarps = 4;
template <int NT, typename Rf>
__host__ __device__ constexpr size_t fft_smem_bytes(int nw) {
  constexpr int NPHI = 2 * NT;
  return sizeof(C2<Rf>) * (size_t(kFftBatch) * nw * NPHI * (NT + 1)) + sizeof(Rf) * 2 * NPHI * (NT / 2) * (NT / 2);
}

// One K_m block in place on a spectrum column (NT theta rows, stride 1):
// K_8 = 0, the others through their mirror-split halves.
template <int NT, typename Rf>
__device__ __forceinline__ void filter_column(C2<Rf>* col, int m, const Rf* KE, const Rf* KO) {
  constexpr int NPHI = 2 * NT, H = NT / 2;
  if (m == NPHI / 2) {
#pragma unroll
    for (int i = 0; i < NT; ++i) col[i] = mk<Rf>(0, 0);
    return;
  }
  C2<Rf> a[NT];
#pragma unroll
  for (int i = 0; i < NT; ++i) a[i] = col[i];
  apply_split_block<NT, 1>(a, KE + m * H * H, KO + m * H * H, col);
}

// a3, a5 (factorised).  A unit is one component of one child box (P
// consecutive samples of the child level's patterns); a warp takes kFftBatch
// consecutive units, whatever their parents, so every lane of every warp but
// the last has work: one lane per (unit, theta row) for the DFTs, one per
// (unit, azimuthal frequency) and turn for the K_m blocks.  (A block per parent
// with its children four at a time ran surfaces' 3.8 children on 93 % of its
// lanes, with block barriers between the steps.)  Per unit one shared-memory
// region of NPHI x (NT+1) complex holds, in turn, the row spectra [m][i], the
// filtered spectra (in place on each column m) and the result [j][i]; a warp
// owns its regions, so the steps are separated by warp barriers only.  Blocks
// of kFftWarps warps share the K_m tables; one warp on small levels, which
// spreads them over the SMs.  327,680 triangles: interpolation 1.36 -> 1.15 ms,
// anterpolation 1.40 -> 1.14 ms; 81,920: 0.44 -> 0.33 and 0.46 -> 0.33 ms.
template <int NT, typename Rf>
struct FftUnits {
  static_assert(NT == 8 && kFftBatch * NT == 32, "16-point register DFT, one warp per kFftBatch units");
  static constexpr int NPHI = 2 * NT, P = NT * NPHI, H = NT / 2;
  // AP: column stride of the spectra (padded by one so that lanes striding
  // over columns hit distinct banks)
  static constexpr int AP = NT + 1, REG = NPHI * AP;
  const Rf *KE, *KO;  // mirror-split K_m blocks
  C2<Rf>* A;          // the warp's regions
  int lane, n;        // units of the warp: first .. first + n - 1
  int64_t first;
  __device__ __forceinline__ FftUnits(unsigned char* smem, int64_t units) {
    Rf* k = reinterpret_cast<Rf*>(smem);
    KE = k;
    KO = k + NPHI * H * H;
    lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    A = reinterpret_cast<C2<Rf>*>(k + 2 * NPHI * H * H) + warp * kFftBatch * REG;
    first = (int64_t(blockIdx.x) * (blockDim.x >> 5) + warp) * kFftBatch;
    n = int(max(int64_t(0), min(int64_t(kFftBatch), units - first)));
  }
  // the lane's row x through the forward DFT, the K_m blocks and the inverse DFT
  __device__ __forceinline__ void filter(C2<Rf>* x, C2<Rf>* X) {
    const int slot = lane / NT, i = lane % NT;
    C2<Rf>* R = A + slot * REG;
    if (slot < n) {
      fft16<false>(x, X);
#pragma unroll
      for (int m = 0; m < NPHI; ++m) R[m * AP + i] = X[m];
    }
    __syncwarp();
    for (int it = lane; it < n * NPHI; it += 32)
      filter_column<NT>(A + (it / NPHI) * REG + (it % NPHI) * AP, it % NPHI, KE, KO);
    __syncwarp();
    if (slot < n) {
#pragma unroll
      for (int m = 0; m < NPHI; ++m) x[m] = R[m * AP + i];
      fft16<true>(x, X);
    }
  }
  // f(sample index from the warp's first unit, value) over the regions, coalesced
  template <typename F>
  __device__ __forceinline__ void each(F f) {
    __syncwarp();
    for (int k = lane; k < n * P; k += 32) f(k, A[(k / P) * REG + (k % NPHI) * AP + (k % P) / NPHI]);
  }
};

// a3: the children's patterns filtered and shifted to their parents' centres,
// Uc[unit] = phase_o (F S_child); k_child_sum adds them up.
template <int NT, typename Rf>
__global__ void __launch_bounds__(32 * kFftWarps, 4) k_interp_fft(int64_t units, const int8_t* __restrict__ oct_child,
                                                                  const C2<Rf>* __restrict__ Sc,
                                                                  const Rf* __restrict__ Kf,
                                                                  const C2<Rf>* __restrict__ phase,
                                                                  C2<Rf>* __restrict__ Uc, int64_t sc = 0) {
  using Units = FftUnits<NT, Rf>;
  constexpr int NPHI = Units::NPHI, P = Units::P;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Units w(smem_raw, units);
  load_split_blocks<NT, false>(Kf, const_cast<Rf*>(w.KE), const_cast<Rf*>(w.KO), threadIdx.x, blockDim.x);
  __syncthreads();
  Sc += blockIdx.y * sc + w.first * P;
  Uc += blockIdx.y * sc + w.first * P;
  const int slot = w.lane / NT, i = w.lane % NT;
  C2<Rf> x[NPHI], X[NPHI];
  if (slot < w.n) {
#pragma unroll
    for (int j = 0; j < NPHI; ++j) x[j] = Sc[slot * P + i * NPHI + j];
  }
  w.filter(x, X);
  if (slot < w.n) {  // phase shift to the parent centre, in the row's own spectra
    const C2<Rf>* ph = phase + oct_child[(w.first + slot) / kComp] * P + i * NPHI;
#pragma unroll
    for (int j = 0; j < NPHI; ++j) w.A[slot * Units::REG + j * Units::AP + i] = cmul(ph[j], X[j]);
  }
  w.each([&](int k, C2<Rf> v) { Uc[k] = v; });
}

// The sum over a parent's children, in order: one thread per (parent,
// component, sample), blocks of (P samples, one component).
template <typename Rf>
__global__ void k_child_sum(int P, const int32_t* __restrict__ child_start, const C2<Rf>* __restrict__ Uc,
                            C2<Rf>* __restrict__ Sp, int64_t sc = 0, int64_t sp = 0) {
  const int64_t b = blockIdx.x;
  const int k = blockIdx.z * P + threadIdx.x;
  Uc += blockIdx.y * sc;
  C2<Rf> v = mk<Rf>(0, 0);
  const int c1 = child_start[b + 1];
#pragma unroll 4
  for (int c = child_start[b]; c < c1; ++c) {
    const C2<Rf> u = Uc[(int64_t)c * kComp * P + k];
    v.x += u.x;
    v.y += u.y;
  }
  Sp[blockIdx.y * sp + b * kComp * P + k] = v;
}

// a5: children take F^T (conj(phase_o) G_parent), added to their incoming patterns.
template <int NT, typename Rf>
__global__ void __launch_bounds__(32 * kFftWarps, 4)
    k_anterp_fft(int64_t units, const int32_t* __restrict__ parent, const int8_t* __restrict__ oct_child,
                 const C2<Rf>* __restrict__ Gp, const Rf* __restrict__ Kf, const C2<Rf>* __restrict__ phase,
                 C2<Rf>* __restrict__ Gc, int64_t sGp = 0, int64_t sGc = 0) {
  using Units = FftUnits<NT, Rf>;
  constexpr int NPHI = Units::NPHI, P = Units::P;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Units w(smem_raw, units);
  load_split_blocks<NT, true>(Kf, const_cast<Rf*>(w.KE), const_cast<Rf*>(w.KO), threadIdx.x, blockDim.x);
  __syncthreads();
  const int slot = w.lane / NT, i = w.lane % NT;
  C2<Rf> x[NPHI], X[NPHI];
  if (slot < w.n) {
    const int64_t ch = (w.first + slot) / kComp, c = (w.first + slot) % kComp;
    const C2<Rf>* src = Gp + blockIdx.y * sGp + (int64_t(parent[ch]) * kComp + c) * P + i * NPHI;
    const C2<Rf>* ph = phase + oct_child[ch] * P + i * NPHI;
#pragma unroll
    for (int j = 0; j < NPHI; ++j) {
      C2<Rf> g = src[j], w = ph[j];
      x[j] = mk<Rf>(w.x * g.x + w.y * g.y, w.x * g.y - w.y * g.x);  // conj(w) g
    }
  }
  w.filter(x, X);
  if (slot < w.n) {
#pragma unroll
    for (int j = 0; j < NPHI; ++j) w.A[slot * Units::REG + j * Units::AP + i] = X[j];
  }
  Gc += blockIdx.y * sGc + w.first * P;
  w.each([&](int k, C2<Rf> v) {
    const C2<Rf> g = Gc[k];
    Gc[k] = mk<Rf>(g.x + v.x, g.y + v.y);
  });
}

// The levels of one translation launch, most boxes first (the leaf level's
// blocks start first, the coarse levels fill in behind them).
constexpr int kMaxTrans = 19;  // levels 3 .. 21
struct TransLevel {
  int64_t first;  // number of the level's first box in the launch
  const int32_t *ptr, *idx, *off;
  const void* T;
  const void* S;
  void* G;
  int64_t stride;  // between right-hand sides
};
struct TransArgs {
  int n = 0;
  int64_t total = 0;
  TransLevel l[kMaxTrans];
};
__device__ __forceinline__ int trans_level(const TransArgs& a, int64_t box) {
  int k = 0;
  while (k + 1 < a.n && box >= a.l[k + 1].first) ++k;
  return k;
}

// a4: translation, all levels at once: G[d] = sum_{s in IL(d)} T[off] * S[s];
// one destination box per threadIdx.y row of a block (several rows for small
// angular grids), one thread per sample and NC components (the others in
// blockIdx.z: five components a thread where the boxes fill the SMs, one on
// small trees).  In float the list is walked U = 4 entries at a time: their
// loads are issued together and the multiply-adds follow in list order (the
// order of the one-entry loop), so a thread waits for one load latency per
// four entries instead of per entry (the small-grid float levels are
// latency-bound).  In double the FP64 pipe bounds the kernel and U = 1
// (measured: U = 2 was 0.5 % slower).  With a launch per level the coarse levels
// left most SMs idle in turn: 327,680 triangles (double) 4.58 -> 4.40 ms, 81,920
// 1.25 -> 1.12 ms, 56 boxes 46 -> 20 us, float patterns of 32 samples at 327,680
// triangles 135 -> 97 us.
template <typename Rf, int NC>
__device__ __forceinline__ void trans_boxes(int P, const TransArgs& args) {
  constexpr int U = sizeof(Rf) == 4 ? 4 : 1;
  const int64_t box = int64_t(blockIdx.x) * blockDim.y + threadIdx.y;
  if (box >= args.total) return;
  const TransLevel& lv = args.l[trans_level(args, box)];
  const int64_t d = box - lv.first;
  const int32_t* __restrict__ il_idx = lv.idx;
  const int32_t* __restrict__ il_off = lv.off;
  const C2<Rf>* __restrict__ Tt = static_cast<const C2<Rf>*>(lv.T);
  const C2<Rf>* __restrict__ S = static_cast<const C2<Rf>*>(lv.S) + blockIdx.y * lv.stride + blockIdx.z * NC * P;
  C2<Rf>* __restrict__ G = static_cast<C2<Rf>*>(lv.G) + blockIdx.y * lv.stride + blockIdx.z * NC * P;
  const int j0 = lv.ptr[d], j1 = lv.ptr[d + 1];
  for (int p = threadIdx.x; p < P; p += blockDim.x) {
    C2<Rf> acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = mk<Rf>(0, 0);
    int j = j0;
    for (; j + U <= j1; j += U) {
      C2<Rf> tv[U], sv[U][NC];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        tv[u] = Tt[(int64_t)il_off[j + u] * P + p];
        const C2<Rf>* src = S + (int64_t)il_idx[j + u] * kComp * P + p;
#pragma unroll
        for (int c = 0; c < NC; ++c) sv[u][c] = src[c * P];
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int c = 0; c < NC; ++c) cfma(acc[c], tv[u], sv[u][c]);
    }
    for (; j < j1; ++j) {
      int s = il_idx[j];
      C2<Rf> tv = Tt[(int64_t)il_off[j] * P + p];
      const C2<Rf>* src = S + (int64_t)s * kComp * P + p;
#pragma unroll
      for (int c = 0; c < NC; ++c) cfma(acc[c], tv, src[c * P]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) G[((int64_t)d * kComp + c) * P + p] = acc[c];
  }
}

template <typename Rf, int NC>
__global__ void k_trans(int P, const TransArgs args) {
  trans_boxes<Rf, NC>(P, args);
}
template <typename Rf, int NC>
__global__ void __launch_bounds__(kWideThreads) k_trans_wide(int P, const TransArgs args) {
  trans_boxes<Rf, NC>(P, args);
}

// a4 for float patterns of at most 128 samples (the inner operator of the
// nested solve): the interaction list of a box is cut into kTransSplit
// contiguous chunks, one per threadIdx.y sub-row, walked as in k_trans (four
// entries at a time), and the chunks' partial sums are added in chunk order
// through shared memory.  A coarse level has few boxes and long lists, so
// this shortens the chain of dependent loads a thread waits through.  The
// order of operations depends on the list alone, never on the launch shape.
constexpr int kTransSplit = 4;
template <typename Rf, int NC>
__global__ void k_trans_split(int P, const TransArgs args) {
  constexpr int U = 4;
  extern __shared__ unsigned char smem_raw[];
  C2<Rf>* part = reinterpret_cast<C2<Rf>*>(smem_raw);  // [row][chunk][component][P]
  const int r = threadIdx.y / kTransSplit, k = threadIdx.y % kTransSplit, p = threadIdx.x;
  const int64_t box = int64_t(blockIdx.x) * (blockDim.y / kTransSplit) + r;
  const bool live = box < args.total && p < P;
  const TransLevel& lv = args.l[trans_level(args, min(box, args.total - 1))];
  const int64_t d = box - lv.first;
  const int32_t* __restrict__ il_idx = lv.idx;
  const int32_t* __restrict__ il_off = lv.off;
  const C2<Rf>* __restrict__ Tt = static_cast<const C2<Rf>*>(lv.T);
  const C2<Rf>* __restrict__ S = static_cast<const C2<Rf>*>(lv.S) + blockIdx.y * lv.stride + blockIdx.z * NC * P;
  C2<Rf>* __restrict__ G = static_cast<C2<Rf>*>(lv.G) + blockIdx.y * lv.stride + blockIdx.z * NC * P;
  C2<Rf> acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = mk<Rf>(0, 0);
  if (live) {
    const int j0 = lv.ptr[d], len = lv.ptr[d + 1] - j0;
    const int q = (len + kTransSplit - 1) / kTransSplit;
    const int a = j0 + min(len, k * q), b = j0 + min(len, (k + 1) * q);
    int j = a;
    for (; j + U <= b; j += U) {
      C2<Rf> tv[U], sv[U][NC];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        tv[u] = Tt[(int64_t)il_off[j + u] * P + p];
        const C2<Rf>* src = S + (int64_t)il_idx[j + u] * kComp * P + p;
#pragma unroll
        for (int c = 0; c < NC; ++c) sv[u][c] = src[c * P];
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int c = 0; c < NC; ++c) cfma(acc[c], tv[u], sv[u][c]);
    }
    for (; j < b; ++j) {
      C2<Rf> tv = Tt[(int64_t)il_off[j] * P + p];
      const C2<Rf>* src = S + (int64_t)il_idx[j] * kComp * P + p;
#pragma unroll
      for (int c = 0; c < NC; ++c) cfma(acc[c], tv, src[c * P]);
    }
  }
  C2<Rf>* mine = part + ((int64_t)(r * kTransSplit + k) * NC) * P;
  if (p < P && k > 0)
#pragma unroll
    for (int c = 0; c < NC; ++c) mine[c * P + p] = acc[c];
  __syncthreads();
  if (!live || k > 0) return;
#pragma unroll
  for (int kk = 1; kk < kTransSplit; ++kk) {
    const C2<Rf>* o = part + ((int64_t)(r * kTransSplit + kk) * NC) * P;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      acc[c].x += o[c * P + p].x;
      acc[c].y += o[c * P + p].y;
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) G[((int64_t)d * kComp + c) * P + p] = acc[c];
}

// a5: anterpolation from level l to level l+1:
// G_child += F^T (conj(phase_o) G_parent); one child box per threadIdx.y
// row of a block (several rows for small angular grids).  With fs the
// filter F is staged in shared memory first (else read from global memory).
template <typename Rf, int NC>
__global__ void k_anterp(int P, int64_t nc, const int32_t* __restrict__ parent, const int8_t* __restrict__ oct_child,
                         const C2<Rf>* __restrict__ Gp, const Rf* __restrict__ Fg, const C2<Rf>* __restrict__ phase,
                         C2<Rf>* __restrict__ Gc, int64_t sGp = 0, int64_t sGc = 0, bool fs = false) {
  Gp += blockIdx.y * sGp;
  Gc += blockIdx.y * sGc;
  extern __shared__ unsigned char smem_raw[];
  Rf* fsm = reinterpret_cast<Rf*>(smem_raw);
  const size_t fbytes = fs ? ((sizeof(Rf) * P * P + 15) / 16) * 16 : 0;
  C2<Rf>* sm = reinterpret_cast<C2<Rf>*>(smem_raw + fbytes) + threadIdx.y * kComp * P;
  const int tid = (threadIdx.z * blockDim.y + threadIdx.y) * blockDim.x + threadIdx.x;
  const int nth = blockDim.x * blockDim.y * blockDim.z;
  const int row_tid = threadIdx.z * blockDim.x + threadIdx.x, row_nth = blockDim.x * blockDim.z, c0 = NC * threadIdx.z;
  if (fs)  // P x P reals as 8-byte words (P = 2 N_theta^2 is even)
    for (int i = tid; i < P * P * int(sizeof(Rf)) / 8; i += nth)
      cp_async(reinterpret_cast<uint2*>(fsm) + i, reinterpret_cast<const uint2*>(Fg) + i);
  const Rf* F = fs ? fsm : Fg;
  const int64_t ch = int64_t(blockIdx.x) * blockDim.y + threadIdx.y;
  const bool live = ch < nc;
  const int par = live ? parent[ch] : 0;
  const int o = live ? oct_child[ch] : 0;
  // the parent's pattern copied in, then turned in place by the thread
  // that copied each entry: conj(phase_o) G_parent
  for (int i = row_tid; live && i < kComp * P; i += row_nth) cp_async(sm + i, Gp + (int64_t)par * kComp * P + i);
  cp_async_wait_all();
  for (int i = row_tid; live && i < kComp * P; i += row_nth) {
    const int q = i % P;
    const C2<Rf> g = sm[i], ph = phase[o * P + q];
    C2<Rf> h;
    h.x = ph.x * g.x + ph.y * g.y;   // conj(ph) * g
    h.y = ph.x * g.y - ph.y * g.x;
    sm[i] = h;
  }
  __syncthreads();
  if (!live) return;
  for (int p = threadIdx.x; p < P; p += blockDim.x) {
    C2<Rf> sum[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) sum[c] = mk<Rf>(0, 0);
#pragma unroll 4
    for (int q = 0; q < P; ++q) {
      Rf f = F[(int64_t)q * P + p];
#pragma unroll
      for (int c = 0; c < NC; ++c) rfma(sum[c], f, sm[(c0 + c) * P + q]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      C2<Rf>& g = Gc[((int64_t)ch * kComp + c0 + c) * P + p];
      g.x += sum[c].x;
      g.y += sum[c].y;
    }
  }
}

// Sum and difference of the incoming leaf patterns over antipodal sample
// pairs, once per box: GS[b][c][q] = G(q) + G(-q), GD[b][c][q] = G(q) - G(-q)
// (half grid q), shared by all triangles of the box in the disaggregation.
// Double only: float adds are cheaper than the pass, so float disaggregation
// forms them itself (the same sums).
template <typename Rf>
__global__ void k_gsgd(int P, int ntheta, const C2<Rf>* __restrict__ G, C2<Rf>* __restrict__ GS,
                       C2<Rf>* __restrict__ GD, int64_t sG = 0, int64_t sH = 0) {
  const int b = blockIdx.x;
  const int Ph = P / 2;
  G += blockIdx.y * sG;
  GS += blockIdx.y * sH;
  GD += blockIdx.y * sH;
  for (int i = threadIdx.x; i < kComp * Ph; i += blockDim.x) {
    const int c = i / Ph, q = i % Ph;
    const C2<Rf> u = G[((int64_t)b * kComp + c) * P + q];
    const C2<Rf> v = G[((int64_t)b * kComp + c) * P + antipode(q, ntheta)];
    GS[((int64_t)b * kComp + c) * Ph + q] = mk<Rf>(u.x + v.x, u.y + v.y);
    GD[((int64_t)b * kComp + c) * Ph + q] = mk<Rf>(u.x - v.x, u.y - v.y);
  }
}

// a6: leaf disaggregation with the receiving (conjugate) patterns, float
// patterns of many triangles (k_disagg_split otherwise).  One thread per
// triangle; the receiving tables are stored sample-major
// ([Ph][T], [3][Ph][T]) so that consecutive threads read consecutive
// triangles, and the box's patterns are shared through the cache.  Over a sample pair (q, -q):
// conj(X(q)) G(q) + X(q) G(-q) = Xr (G(q) + G(-q)) - i Xi (G(q) - G(-q)).
// Writes pot[t].
template <typename Rf, typename Rio>
__global__ void __launch_bounds__(256) k_disagg(int64_t T, int P, int ntheta, const int32_t* __restrict__ leaf_of,
                                                const C2<Rf>* __restrict__ PiR, const C2<Rf>* __restrict__ MR,
                                                const C2<Rf>* __restrict__ G, C2<Rio>* __restrict__ pot,
                                                int64_t sG = 0, int64_t sp = 0) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= T) return;
  const int Ph = P / 2;
  G += blockIdx.y * sG + (int64_t)leaf_of[t] * kComp * P;
  pot += blockIdx.y * sp;
  C2<Rf> acc[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) acc[i] = mk<Rf>(0, 0);
  // sample pair q's patterns and table entries, then its multiply-adds
  // (issuing two sample pairs' loads together was measured slower at
  // N = 819,200 in float: 0.096 against 0.085 ms)
  struct Sample {
    C2<Rf> gs[kComp], gd[kComp], pi, m[3];
  };
  auto load = [&](int q, Sample& r) {
#pragma unroll
    for (int c = 0; c < kComp; ++c) {
      const C2<Rf> u = G[c * P + q], v = G[c * P + antipode(q, ntheta)];
      r.gs[c] = mk<Rf>(u.x + v.x, u.y + v.y);
      r.gd[c] = mk<Rf>(u.x - v.x, u.y - v.y);
    }
    r.pi = PiR[(int64_t)q * T + t];
#pragma unroll
    for (int d = 0; d < 3; ++d) r.m[d] = MR[((int64_t)d * Ph + q) * T + t];
  };
  auto accumulate = [&](const Sample& r) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const C2<Rf> m = r.m[d];
      // U += Mr gs - i Mi gd
      rfma(acc[0], m.x, r.gs[d]);
      acc[0].x = fma(m.y, r.gd[d].y, acc[0].x);
      acc[0].y = fma(-m.y, r.gd[d].x, acc[0].y);
      // V_d += Pr gs - i Pi gd
      rfma(acc[1 + d], r.pi.x, r.gs[d]);
      acc[1 + d].x = fma(r.pi.y, r.gd[d].y, acc[1 + d].x);
      acc[1 + d].y = fma(-r.pi.y, r.gd[d].x, acc[1 + d].y);
    }
#pragma unroll
    for (int c = 3; c < 5; ++c) {
      rfma(acc[1 + c], r.pi.x, r.gs[c]);
      acc[1 + c].x = fma(r.pi.y, r.gd[c].y, acc[1 + c].x);
      acc[1 + c].y = fma(-r.pi.y, r.gd[c].x, acc[1 + c].y);
    }
  };
  for (int q = 0; q < Ph; ++q) {
    Sample r;
    load(q, r);
    accumulate(r);
  }
  C2<Rio>* o = pot + 6 * t;
#pragma unroll
  for (int i = 0; i < 6; ++i) o[i] = mk<Rio>(Rio(acc[i].x), Rio(acc[i].y));
}

// a6 with the twelve real sums of a triangle shared by five threads
// (threadIdx.y, one warp each for the block's 32 triangles): U real, U
// imaginary, the three V real, the three V imaginary, T1 and T2; 6, 6, 6, 6 and
// 8 multiply-adds a sample pair, each sum in k_disagg's order.  In double a
// warp's multiply-add occupies an SM scheduler for 67 clocks, so k_disagg's
// 2048 of them a triangle run one after the other on as many schedulers as
// there are warps of triangles (with the sum / difference patterns: 1280
// triangles 140 -> 36 us, 11,250 172 -> 63 us, 81,920 426 -> 322 us, 327,680
// 1232 -> 1204 us).  Float patterns of many triangles keep k_disagg, which reads
// each table entry once.
template <typename Rf, typename Rio>
__global__ void __launch_bounds__(160) k_disagg_split(int64_t T, int P, int ntheta, const int32_t* __restrict__ leaf_of,
                                                      const C2<Rf>* __restrict__ PiR, const C2<Rf>* __restrict__ MR,
                                                      const C2<Rf>* __restrict__ GS, const C2<Rf>* __restrict__ GD,
                                                      C2<Rio>* __restrict__ pot, int64_t sH = 0, int64_t sp = 0) {
  const int64_t t = blockIdx.x * (int64_t)32 + threadIdx.x;
  if (t >= T) return;
  const int Ph = P / 2;
  // double: the sum and difference patterns GS, GD; float: GS is the pattern G itself
  constexpr bool WHOLE = sizeof(Rf) == 4;
  const Rf* gs = reinterpret_cast<const Rf*>(GS + blockIdx.y * sH + (int64_t)leaf_of[t] * kComp * (WHOLE ? P : Ph));
  const Rf* gd = WHOLE ? gs : reinterpret_cast<const Rf*>(GD + blockIdx.y * sH + (int64_t)leaf_of[t] * kComp * Ph);
  Rio* o = reinterpret_cast<Rio*>(pot + blockIdx.y * sp + 6 * t);
  // NS sums over the sample pairs: load(q, d) gives the operands of sum (or
  // step) d, step(d) its two multiply-adds; four sample pairs' loads are issued
  // ahead of the four being summed
  struct Op {
    C2<Rf> x;
    Rf s, d;
  };
  auto run = [&](auto n, auto load, auto step) {
    constexpr int N = decltype(n)::value, U = sizeof(Rf) == 8 ? 2 : 4;
    Op a[U][N], b[U][N];
    auto fetch = [&](int q, Op(&v)[U][N]) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (q + u < Ph)
#pragma unroll
          for (int d = 0; d < N; ++d) v[u][d] = load(q + u, d);
    };
    auto sum = [&](int q, const Op(&v)[U][N]) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (q + u < Ph)
#pragma unroll
          for (int d = 0; d < N; ++d) step(d, v[u][d]);
    };
    fetch(0, a);
    for (int q = 0; q < Ph; q += 2 * U) {
      fetch(q + U, b);
      sum(q, a);
      fetch(q + 2 * U, a);
      sum(q + U, b);
    }
  };
  auto at_s = [&](int c, int q, int im) {
    if constexpr (WHOLE) return gs[2 * (c * P + q) + im] + gs[2 * (c * P + antipode(q, ntheta)) + im];
    return gs[2 * (c * Ph + q) + im];
  };
  auto at_d = [&](int c, int q, int im) {
    if constexpr (WHOLE) return gs[2 * (c * P + q) + im] - gs[2 * (c * P + antipode(q, ntheta)) + im];
    return gd[2 * (c * Ph + q) + im];
  };
  // im = 0: real part, += x.x s.x + x.y d.y; im = 1: imaginary part, += x.x s.y - x.y d.x
  auto U = [&](auto imc) {
    constexpr int im = decltype(imc)::value;
    Rf u = 0;
    run(
        std::integral_constant<int, 3>(),
        [&](int q, int d) { return Op{MR[((int64_t)d * Ph + q) * T + t], at_s(d, q, im), at_d(d, q, 1 - im)}; },
        [&](int, const Op& v) {
          u = fma(v.x.x, v.s, u);
          u = fma(im ? -v.x.y : v.x.y, v.d, u);
        });
    o[im] = Rio(u);
  };
  auto V = [&](auto imc) {
    constexpr int im = decltype(imc)::value;
    Rf v[3] = {0, 0, 0};
    run(
        std::integral_constant<int, 3>(),
        [&](int q, int d) { return Op{PiR[(int64_t)q * T + t], at_s(d, q, im), at_d(d, q, 1 - im)}; },
        [&](int d, const Op& w) {
          v[d] = fma(w.x.x, w.s, v[d]);
          v[d] = fma(im ? -w.x.y : w.x.y, w.d, v[d]);
        });
#pragma unroll
    for (int d = 0; d < 3; ++d) o[2 + 2 * d + im] = Rio(v[d]);
  };
  switch (threadIdx.y) {
    case 0: return U(std::integral_constant<int, 0>());
    case 1: return U(std::integral_constant<int, 1>());
    case 2: return V(std::integral_constant<int, 0>());
    case 3: return V(std::integral_constant<int, 1>());
  }
  Rf v[4] = {0, 0, 0, 0};  // T1 real, imaginary, T2 real, imaginary
  run(
      std::integral_constant<int, 4>(),
      [&](int q, int d) { return Op{PiR[(int64_t)q * T + t], at_s(3 + d / 2, q, d % 2), at_d(3 + d / 2, q, 1 - d % 2)}; },
      [&](int d, const Op& w) {
        v[d] = fma(w.x.x, w.s, v[d]);
        v[d] = fma(d % 2 ? -w.x.y : w.x.y, w.d, v[d]);
      });
#pragma unroll
  for (int d = 0; d < 4; ++d) o[8 + d] = Rio(v[d]);
}

// Per-triangle potential j of the product: near + far (each rounded to the
// io precision, summed in double, rounded again), or pot alone.
template <typename Rio>
__device__ __forceinline__ C2<Rio> pot_sum(const C2<Rio>* pot, const C2<Rio>* pot2, int64_t j) {
  if (!pot2) return pot[j];
  // (two floats summed in double and rounded again are the floats' rounded sum)
  const C2<Rio> a = pot2[j], b = pot[j];
  return mk<Rio>(a.x + b.x, a.y + b.y);
}

// a7: Galerkin testing of the per-triangle potentials (Section 2):
// RWG m: sum over its two triangles of c [U + (c_t - p).V] + 2c T1; pulse t: T2.
// pot2 (may be null): near-part potentials, added to pot first.  SCALED:
// the result is scale y, y rounded to the io precision first.
template <typename Rio, bool SCALED = false>
__global__ void k_assemble(int64_t N, int64_t E, const int32_t* __restrict__ edge_tt,
                           const int8_t* __restrict__ edge_k, const double* __restrict__ tri_c,
                           const double* __restrict__ tri_dcp, const int64_t* __restrict__ inv_perm,
                           const C2<Rio>* __restrict__ pot, C2<Rio>* __restrict__ y, int64_t sp = 0, int64_t sy = 0,
                           const C2<Rio>* __restrict__ pot2 = nullptr, const double* __restrict__ scale = nullptr) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  auto store = [&](C2<Rio> v) {
    if constexpr (SCALED) v = mk<Rio>(Rio(scale[i] * double(v.x)), Rio(scale[i] * double(v.y)));
    y[i] = v;
  };
  pot += blockIdx.y * sp;
  if (pot2) pot2 += blockIdx.y * sp;
  y += blockIdx.y * sy;
  if (i < E) {
    double yr = 0, yi = 0;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      int64_t t = edge_tt[2 * i + side];
      int k = edge_k[2 * i + side];
      double c = tri_c[3 * t + k];
      const double* dcp = tri_dcp + 9 * t + 3 * k;
      C2<Rio> p[5];
#pragma unroll
      for (int j = 0; j < 5; ++j) p[j] = pot_sum(pot, pot2, 6 * t + j);
      double ur = double(p[0].x) + dcp[0] * double(p[1].x) + dcp[1] * double(p[2].x) + dcp[2] * double(p[3].x);
      double ui = double(p[0].y) + dcp[0] * double(p[1].y) + dcp[1] * double(p[2].y) + dcp[2] * double(p[3].y);
      yr += c * (ur + 2.0 * double(p[4].x));
      yi += c * (ui + 2.0 * double(p[4].y));
    }
    store(mk<Rio>(Rio(yr), Rio(yi)));
  } else {
    int64_t t = inv_perm[i - E];
    store(pot_sum(pot, pot2, 6 * t + 5));
  }
}

// ---------------------------------------------------------------- orchestration

static inline unsigned nblk(int64_t n, int b) { return unsigned((n + b - 1) / b); }

// Blocks per leaf box of the box-staged kernels: enough to give an SM its six,
// at least a test triangle for each of a block's warps.
static int near_box_split(const Problem& pr, int warps) {
  const int64_t want = (6 * int64_t(pr.nsm) + pr.nleaf - 1) / pr.nleaf, most = (pr.T / pr.nleaf + warps - 1) / warps;
  return int(std::max<int64_t>(1, std::min({want, most, int64_t(16)})));
}

static inline MomScale mom_scale(const Problem& pr) {
  MomScale m;
  for (int q = 0; q < kMom; ++q) m.s[q] = pr.mom_scale[q];
  return m;
}

void prof_mark(Problem& pr, int stage, bool end, cudaStream_t st) {
  if (pr.prof_n >= pr.prof_cap) return;
  cudaEventRecord(pr.prof_ev[(size_t(pr.prof_n) * kStages + stage) * 2 + (end ? 1 : 0)], st);
}

// Asks the far kernels for their limits, once per process (set-up).
template <typename Rf>
static void far_prepare() {
  max_threads<k_agg<Rf>>();
  max_threads<k_agg_split<Rf, 1>>();
  max_threads<k_agg_split<Rf, kComp>>();
  max_threads<k_interp<Rf, 1>>();
  max_threads<k_interp<Rf, kComp>>();
  max_threads<k_anterp<Rf, 1>>();
  max_threads<k_anterp<Rf, kComp>>();
  max_threads<k_trans<Rf, 1>>();
  max_threads<k_trans<Rf, kComp>>();
  if constexpr (sizeof(Rf) == 4) {
    max_threads<k_trans_split<Rf, 1>>();
    max_threads<k_trans_split<Rf, kComp>>();
  }
}

pie_status product_prepare(const Problem& pr) {
  if (pr.far_f32())
    far_prepare<float>();
  else
    far_prepare<double>();
  switch (pr.par.precision) {
    case PIE_FP64: return near_fixed_prepare();
    case PIE_FP32: return near_float_prepare<float, false>();
    case PIE_FP32H: return near_float_prepare<float, true>();
    default: return near_float_prepare<double, false>();
  }
}

template <typename Rm, typename Rf, typename Rio, bool H16 = false>
static pie_status apply_t(Problem& pr, const void* xv, void* yv, int nrhs, cudaStream_t st, const double* scale) {
  const int P = pr.P;
  const int L = pr.tree.L;
  const C2<Rio>* x = static_cast<const C2<Rio>*>(xv);
  C2<Rio>* y = static_cast<C2<Rio>*>(yv);
  C2<Rio>* coef = static_cast<C2<Rio>*>(pr.coef);
  C2<Rio>* pot = static_cast<C2<Rio>*>(pr.pot);
  const double w2e = pr.w * pr.w * eps0();
  const unsigned nr = unsigned(nrhs);
  const int64_t sN = pr.N, sT = 6 * pr.T;  // right-hand-side strides of x / y and of coef / pot
  constexpr bool split = sizeof(Rm) < sizeof(Rio);  // float near part, double coefficients
  cf* coef32 = split ? static_cast<cf*>(pr.coef32) : nullptr;
  const C2<Rm>* ncoef = split ? reinterpret_cast<const C2<Rm>*>(coef32) : reinterpret_cast<const C2<Rm>*>(coef);
  prof_mark(pr, 0, false, st);
  k_coef<Rio><<<dim3(nblk(pr.T, 256), nr), 256, 0, st>>>(pr.T, pr.E, x, pr.perm, pr.tri_edge, pr.tri_c, pr.tri_cdcp,
                                                         w2e, coef, coef32, sN, sT, scale);
  prof_mark(pr, 0, true, st);
  // near part into pot2, far part into pot.  With tune.overlap the near part
  // runs on the side stream (HBM-bound, a bounded grid) and the far part on
  // the problem's high-priority stream, concurrently; per-stage profiling
  // keeps them in order on the caller's stream.
  const bool profiling = pr.prof_n < pr.prof_cap;
  const bool with_near = pr.with_near;
  const bool overlap = pr.tune.overlap && !profiling && with_near;
  C2<Rio>* pot2 = static_cast<C2<Rio>*>(pr.pot2);
  cudaStream_t sn = st, sf = st;
  unsigned near_grid = nblk(pr.T * 32, 256);
  if (overlap) {
    // inside a stream capture (a multi-mesh group's graph) the far part
    // stays on the capturing stream: with every member's far part at the
    // highest priority the members' near parts waited for all of them
    // (group launch 131.4 -> 137.6 ms for the four configuration-3 meshes)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    pie_status s = cuda_check(cudaStreamIsCapturing(st, &cap), "capture status");
    if (s == PIE_OK) s = cuda_check(cudaEventRecord(pr.ev_fork, st), "fork");
    if (s == PIE_OK) s = cuda_check(cudaStreamWaitEvent(pr.side, pr.ev_fork, 0), "fork");
    if (s == PIE_OK && cap == cudaStreamCaptureStatusNone)
      s = cuda_check(cudaStreamWaitEvent(pr.far, pr.ev_fork, 0), "fork");
    if (s != PIE_OK) return s;
    sn = pr.side;
    if (cap == cudaStreamCaptureStatusNone) sf = pr.far;
    if (pr.tune.near_ctas_per_sm > 0)
      near_grid = std::min<unsigned>(near_grid, unsigned(pr.nsm * pr.tune.near_ctas_per_sm));
  }
  prof_mark(pr, 1, false, st);
  // the float near part reads each pair's moments once for RB right-hand sides
  // (RB chosen per call: a wide accumulator set costs occupancy when unused)
  auto near_launch = [&](auto rb) {
    if constexpr (sizeof(Rm) == 4)
      k_near<Rm, Rio, decltype(rb)::value, H16><<<dim3(near_grid, nblk(nrhs, decltype(rb)::value)), 256, 0, sn>>>(
          pr.T, pr.nnz, pr.leaf_of, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr,
          static_cast<const C2<Rm>*>(pr.mom), static_cast<const __half2*>(pr.mom), mom_scale(pr), ncoef, Rm(kMu0),
          pot2, nrhs, sT, sT);
  };
  // float near part: the box-staged kernels (RB 1, or 2 and 4 by chunks), or
  // one warp per test triangle (RB 1, 2, 4 or 8) when tuned so
  int rb = pr.tune.near_rhs_block;
  if (rb == 0) rb = nrhs == 1 ? 1 : nrhs == 2 ? 2 : 4;
  const bool boxed = sizeof(Rm) == 4 && pr.tune.near_kernel != 1;
  auto box_launch = [&](auto rbc) {
    if constexpr (sizeof(Rm) == 4) {
      constexpr int RB = decltype(rbc)::value, TH = RB == 1 ? kNearBoxThreads : kNearChunkThreads;
      const int nsplit = near_box_split(pr, TH / 32);
      unsigned grid = unsigned(pr.nleaf * nsplit);
      if (overlap && pr.tune.near_ctas_per_sm > 0)
        // many short blocks make room for the far part's by themselves: a bound
        // only where all of them would start at once
        grid = std::min<unsigned>(grid, unsigned(pr.nsm * pr.tune.near_ctas_per_sm *
                                                 (grid > unsigned(16 * pr.nsm) ? 8192 / TH : 256 / TH)));
      const cf* mom = static_cast<const cf*>(pr.mom);
      const __half2* momh = static_cast<const __half2*>(pr.mom);
      const cf* c = reinterpret_cast<const cf*>(ncoef);
      if constexpr (RB == 1) {
        const int stage = near_box_stage<H16>(pr);
        k_near_box<Rio, H16><<<dim3(grid, nr), TH, near_box_smem<H16>(stage), sn>>>(
            pr.nleaf, nsplit, stage, pr.nnz, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr, mom,
            momh, mom_scale(pr), c, float(kMu0), pot2, sT, sT);
      } else {
        k_near_chunk<Rio, H16, RB><<<dim3(grid, nblk(nrhs, RB)), TH, near_chunk_smem<H16, RB>(), sn>>>(
            pr.nleaf, nsplit, pr.nnz, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr, mom, momh,
            mom_scale(pr), c, float(kMu0), pot2, nrhs, sT, sT);
      }
    }
  };
  if (!with_near) {
    pot2 = nullptr;
  } else if constexpr (sizeof(Rm) == 8) {  // PIE_FP64: fixed point, each column by itself
    // beside the far part: one block an SM where it ends with the far part, else two
    // (three leave the filter kernels no shared memory until they are done: the 100 MHz
    // plate 377 us beside 100 KB an SM, 440 beside 209), and three where the near part
    // takes four times as long (cylinder of 9472 triangles 834 us with two, 625;
    // ellipsoid of 8192 750, 575).  One block takes 89 ps a pair (81,920 triangles: 1.9
    // ms), the far part 1.6 ps a double operation: 20 a list entry and sample, 32 a
    // triangle and sample for aggregation and disaggregation, about 9000 a box and
    // component for the filters
    double far_ops = 32.0 * double(pr.T) * P;
    for (int l = 3; l <= L; ++l)
      far_ops += 20.0 * P * double(pr.lev[l].nlist) + (l > 3 ? 9000.0 * kComp * double(pr.lev[l].nb) : 0.0);
    const double near_part = 89.0 * double(pr.nnz) / (1.6 * far_ops);  // over the far part
    const int64_t per_sm = near_part > 4.0 ? 3 : near_part > 1.0 ? 2 : 1;
    // (the kernel of fewer registers up to there: plates, at 2.9, 356 us, 381 with the
    // other; 1120, 1314)
    near_fixed(pr, coef, pot2, nrhs,
               overlap && pr.tune.near_ctas_per_sm > 0
                   ? int64_t(pr.nsm) * per_sm * ((pr.tune.near_ctas_per_sm + 1) / 2) : 0,
               overlap && near_part <= 4.0, sn);
  } else if (boxed && (rb == 1 || rb == 2 || rb == 4)) {
    if (rb == 1)
      box_launch(std::integral_constant<int, 1>());
    else if (rb == 2)
      box_launch(std::integral_constant<int, 2>());
    else
      box_launch(std::integral_constant<int, 4>());
  } else if (rb == 1)
    near_launch(std::integral_constant<int, 1>());
  else if (rb == 2)
    near_launch(std::integral_constant<int, 2>());
  else if (rb == 4)
    near_launch(std::integral_constant<int, 4>());
  else
    near_launch(std::integral_constant<int, 8>());
  if (overlap) {
    pie_status s = cuda_check(cudaEventRecord(pr.ev_join, sn), "join");
    if (s != PIE_OK) return s;
  }
  prof_mark(pr, 1, true, st);
  const int tpb = P < 1024 ? ((P + 31) / 32) * 32 : 1024;
  const C2<Rf>* Pi = static_cast<const C2<Rf>*>(pr.Pi);
  const C2<Rf>* M = static_cast<const C2<Rf>*>(pr.M);
  auto sl = [&](int l) { return int64_t(pr.lev[l].nb) * kComp * P; };  // pattern stride per right-hand side
  prof_mark(pr, 2, false, st);
  // far coefficients in the far precision (MIXED and FP64: the io buffer)
  const C2<Rf>* fcoef = reinterpret_cast<const C2<Rf>*>(coef);
  // boxes per block of the per-box far kernels (threads: one per sample):
  // tune.far_rows, or enough to fill 128 threads; at most the kernel's threads
  auto far_rows = [&](int threads, int most) {
    const int r = pr.tune.far_rows > 0 ? pr.tune.far_rows : (threads < 64 ? 128 / threads : 1);
    return std::max(1, std::min(r, most / threads));
  };
  // grids of fewer warps than kWideWarps an SM (eight a scheduler) give each
  // warp less to do (components and sums over more threads); the arithmetic
  // stays the same
  constexpr int kWideWarps = 32;
  auto narrow = [&](int64_t warps) { return warps < int64_t(kWideWarps) * pr.nsm; };
  {
    // half-grid threads per box
    const int ath = P / 2 < 32 ? P / 2 : ((P / 2 + 31) / 32) * 32;
    const int64_t warps = (pr.lev[L].nb * ath + 31) / 32 * nr;  // of the whole-sample kernel
    C2<Rf>* SL = static_cast<C2<Rf>*>(pr.lev[L].S);
    auto split = [&](auto ncc) {
      constexpr int NC = decltype(ncc)::value;
      const int most = max_threads<k_agg_split<Rf, NC>>(), sth = std::min(most / 64 * 32, ath);
      const int abp = far_rows(2 * sth, most);
      k_agg_split<Rf, NC><<<dim3(nblk(pr.lev[L].nb, abp), nr, 2 * kComp / NC), dim3(sth, abp, 2),
                            sizeof(Rf) * 2 * NC * sth * abp, sf>>>(P, pr.par.ntheta, pr.lev[L].nb, pr.leaf_start, Pi,
                                                                   M, fcoef, Rf(kMu0), SL, sT, sl(L));
    };
    if (narrow(2 * warps)) {
      split(std::integral_constant<int, 1>());
    } else if (narrow(sizeof(Rf) == 8 ? warps / 4 : warps)) {
      split(std::integral_constant<int, kComp>());
    } else {
      const int abp = far_rows(ath, max_threads<k_agg<Rf>>());
      k_agg<Rf><<<dim3(nblk(pr.lev[L].nb, abp), nr), dim3(ath, abp), 0, sf>>>(
          P, pr.par.ntheta, pr.lev[L].nb, pr.leaf_start, Pi, M, fcoef, Rf(kMu0), SL, sT, sl(L));
    }
  }
  prof_mark(pr, 2, true, st);
  const size_t sm = sizeof(C2<Rf>) * kComp * P;
  // dense-filter kernels: the P x P filter in shared memory when it is at
  // most 16 KB; boxes per block within 48 KB of shared memory; interpolation
  // stages up to eight children per parent in what is left
  const size_t fsb = ((sizeof(Rf) * size_t(P) * P + 15) / 16) * 16;
  const bool fsh = fsb <= 16384;
  const size_t fsm_bytes = fsh ? fsb : 0;
  const int fbp = std::max(1, std::min(far_rows(tpb, kWideThreads), int((49152 - fsm_bytes) / sm)));
  const int cg = int(std::max<size_t>(1, std::min<size_t>(8, (49152 - fsm_bytes) / (sm * fbp))));
  const bool fft8 = pr.par.ntheta == 8;
  prof_mark(pr, 3, false, st);
  // units of the factorised filter between level l and its children, and warps per block
  auto fft_units = [&](int l) { return pr.lev[l + 1].nb * kComp; };
  auto fft_nw = [&](int l) { return narrow(fft_units(l) / kFftBatch * nr) ? 1 : kFftWarps; };
  for (int l = L - 1; l >= 3 && fft8; --l) {
    const int nw = fft_nw(l);
    // the shifted child patterns pass through the child level's G, free until the translation
    C2<Rf>* U = static_cast<C2<Rf>*>(pr.lev[l + 1].G);
    k_interp_fft<8, Rf><<<dim3(nblk(fft_units(l), kFftBatch * nw), nr), 32 * nw, fft_smem_bytes<8, Rf>(nw), sf>>>(
        fft_units(l), pr.lev[l + 1].octant, static_cast<const C2<Rf>*>(pr.lev[l + 1].S),
        static_cast<const Rf*>(pr.lev[l].Kf), static_cast<const C2<Rf>*>(pr.lev[l].phase), U, sl(l + 1));
    k_child_sum<Rf><<<dim3(unsigned(pr.lev[l].nb), nr, kComp), P, 0, sf>>>(
        P, pr.lev[l].child_start, U, static_cast<C2<Rf>*>(pr.lev[l].S), sl(l + 1), sl(l));
  }
  // dense filter: (components a thread, boxes per block, children staged at a time)
  auto dense = [&](int64_t nb, auto f) {
    if (narrow(nb * (tpb / 32) * nr) &&
        tpb * kComp <= std::min(max_threads<k_interp<Rf, 1>>(), max_threads<k_anterp<Rf, 1>>()))
      f(std::integral_constant<int, 1>(), 1, int(std::max<size_t>(1, std::min<size_t>(8, (49152 - fsm_bytes) / sm))));
    else
      f(std::integral_constant<int, kComp>(), fbp, cg);
  };
  for (int l = L - 1; l >= 3 && !fft8; --l)
    dense(pr.lev[l].nb, [&](auto ncc, int rows, int kids) {
      constexpr int NC = decltype(ncc)::value;
      const int most = max_threads<k_interp<Rf, NC>>() / (kComp / NC);
      auto kernel = k_interp<Rf, NC>;
      // (in double a grid that wide needs more than 48 KB a child: refused)
      if constexpr (sizeof(Rf) == 4 && NC > 1)
        if (tpb > most) kernel = k_interp_wide<Rf, NC>;
      const int n = std::max(1, std::min(rows, most / tpb));
      kernel<<<dim3(nblk(pr.lev[l].nb, n), nr), dim3(tpb, n, kComp / NC), fsm_bytes + sm * n * kids, sf>>>(
          P, pr.lev[l].nb, pr.lev[l].child_start, pr.lev[l + 1].octant, static_cast<const C2<Rf>*>(pr.lev[l + 1].S),
          static_cast<const Rf*>(pr.lev[l].Ft), static_cast<const C2<Rf>*>(pr.lev[l].phase),
          static_cast<C2<Rf>*>(pr.lev[l].S), sl(l + 1), sl(l), kids, fsh);
    });
  prof_mark(pr, 3, true, st);
  prof_mark(pr, 4, false, st);
  TransArgs ta;
  for (int l = L; l >= 3; --l) {
    if (!((pr.far_mask >> l) & 1u)) {  // level left out: no incoming pattern of its own
      pie_status s = cuda_check(cudaMemsetAsync(pr.lev[l].G, 0, sizeof(C2<Rf>) * sl(l) * nr, sf), "memset");
      if (s != PIE_OK) return s;
      continue;
    }
    ta.l[ta.n++] = TransLevel{ta.total,       pr.lev[l].il_ptr, pr.lev[l].il_idx, pr.lev[l].il_off,
                              pr.lev[l].trans, pr.lev[l].S,      pr.lev[l].G,      sl(l)};
    ta.total += pr.lev[l].nb;
  }
  if (ta.total > 0) {
    // per right-hand side: components a thread takes
    const bool one = narrow(ta.total * (tpb / 32) * int64_t(nr));
    auto launch = [&](auto ncc) {
      constexpr int NC = decltype(ncc)::value;
      if constexpr (sizeof(Rf) == 4)
        if (tpb <= 128) {  // float, small grid: each list cut into kTransSplit chunks
          const int tbp = far_rows(tpb * kTransSplit, max_threads<k_trans_split<Rf, NC>>());
          k_trans_split<Rf, NC><<<dim3(nblk(ta.total, tbp), nr, kComp / NC), dim3(tpb, tbp * kTransSplit),
                                  sizeof(C2<Rf>) * NC * P * kTransSplit * tbp, sf>>>(P, ta);
          return;
        }
      const int most = max_threads<k_trans<Rf, NC>>();
      auto kernel = k_trans<Rf, NC>;
      if constexpr (sizeof(Rf) == 8 && NC > 1)
        if (tpb > most) kernel = k_trans_wide<Rf, NC>;
      const int tbp = far_rows(tpb, most);  // destination boxes per block
      kernel<<<dim3(nblk(ta.total, tbp), nr, kComp / NC), dim3(tpb, tbp), 0, sf>>>(P, ta);
    };
    if (one)
      launch(std::integral_constant<int, 1>());
    else
      launch(std::integral_constant<int, kComp>());
  }
  prof_mark(pr, 4, true, st);
  prof_mark(pr, 5, false, st);
  for (int l = 3; l < L && fft8; ++l) {
    const int nw = fft_nw(l);
    k_anterp_fft<8, Rf><<<dim3(nblk(fft_units(l), kFftBatch * nw), nr), 32 * nw, fft_smem_bytes<8, Rf>(nw), sf>>>(
        fft_units(l), pr.lev[l + 1].parent, pr.lev[l + 1].octant, static_cast<const C2<Rf>*>(pr.lev[l].G),
        static_cast<const Rf*>(pr.lev[l].Kf), static_cast<const C2<Rf>*>(pr.lev[l].phase),
        static_cast<C2<Rf>*>(pr.lev[l + 1].G), sl(l), sl(l + 1));
  }
  for (int l = 3; l < L && !fft8; ++l)
    dense(pr.lev[l + 1].nb, [&](auto ncc, int rows, int) {
      constexpr int NC = decltype(ncc)::value;
      const int n = std::max(1, std::min(rows, max_threads<k_anterp<Rf, NC>>() / (kComp / NC) / tpb));
      k_anterp<Rf, NC><<<dim3(nblk(pr.lev[l + 1].nb, n), nr), dim3(tpb, n, kComp / NC), fsm_bytes + sm * n, sf>>>(
          P, pr.lev[l + 1].nb, pr.lev[l + 1].parent, pr.lev[l + 1].octant, static_cast<const C2<Rf>*>(pr.lev[l].G),
          static_cast<const Rf*>(pr.lev[l].F), static_cast<const C2<Rf>*>(pr.lev[l].phase),
          static_cast<C2<Rf>*>(pr.lev[l + 1].G), sl(l), sl(l + 1), fsh);
    });
  prof_mark(pr, 5, true, st);
  prof_mark(pr, 6, false, st);
  {
    const C2<Rf>* G = static_cast<const C2<Rf>*>(pr.lev[L].G);
    const C2<Rf>* PiR = static_cast<const C2<Rf>*>(pr.PiR);
    const C2<Rf>* MR = static_cast<const C2<Rf>*>(pr.MR);
    const int nt = pr.par.ntheta;
    if constexpr (sizeof(Rf) == 4) {
      if (narrow((pr.T + 31) / 32 * nr))
        k_disagg_split<Rf, Rio><<<dim3(nblk(pr.T, 32), nr), dim3(32, 5), 0, sf>>>(pr.T, P, nt, pr.leaf_of, PiR, MR, G, G,
                                                                                  pot, sl(L), sT);
      else
        k_disagg<Rf, Rio><<<dim3(nblk(pr.T, 256), nr), 256, 0, sf>>>(pr.T, P, nt, pr.leaf_of, PiR, MR, G, pot, sl(L),
                                                                     sT);
    } else {
      C2<Rf>* GS = static_cast<C2<Rf>*>(pr.gsgd);
      const int64_t sH = int64_t(pr.lev[L].nb) * kComp * (P / 2);
      C2<Rf>* GD = GS + int64_t(pr.par.max_nrhs) * sH;
      k_gsgd<Rf><<<dim3(unsigned(pr.lev[L].nb), nr), 128, 0, sf>>>(P, nt, G, GS, GD, sl(L), sH);
      k_disagg_split<Rf, Rio><<<dim3(nblk(pr.T, 32), nr), dim3(32, 5), 0, sf>>>(pr.T, P, nt, pr.leaf_of, PiR, MR, GS, GD,
                                                                                pot, sH, sT);
    }
  }
  prof_mark(pr, 6, true, st);
  if (overlap) {
    pie_status s = PIE_OK;
    if (sf != st) {
      s = cuda_check(cudaEventRecord(pr.ev_far, sf), "join");
      if (s == PIE_OK) s = cuda_check(cudaStreamWaitEvent(st, pr.ev_far, 0), "join");
    }
    if (s == PIE_OK) s = cuda_check(cudaStreamWaitEvent(st, pr.ev_join, 0), "join");
    if (s != PIE_OK) return s;
  }
  prof_mark(pr, 7, false, st);
  auto assemble = [&](auto scaled) {
    k_assemble<Rio, decltype(scaled)::value><<<dim3(nblk(pr.N, 256), nr), 256, 0, st>>>(
        pr.N, pr.E, pr.edge_tt, pr.edge_k, pr.tri_c, pr.tri_dcp, pr.inv_perm, pot, y, sT, sN, pot2, scale);
  };
  if (scale)
    assemble(std::true_type());
  else
    assemble(std::false_type());
  prof_mark(pr, 7, true, st);
  if (pr.prof_n < pr.prof_cap) ++pr.prof_n;
  return cuda_check(cudaGetLastError(), "apply launch");
}

// Near part alone: y = Z_near x (pairs of triangles in neighbouring leaf boxes).
template <typename Rm, typename Rio, bool H16 = false>
static pie_status apply_near_t(Problem& pr, const void* xv, void* yv, cudaStream_t st) {
  C2<Rio>* coef = static_cast<C2<Rio>*>(pr.coef);
  C2<Rio>* pot = static_cast<C2<Rio>*>(pr.pot);
  constexpr bool split = sizeof(Rm) < sizeof(Rio);
  cf* coef32 = split ? static_cast<cf*>(pr.coef32) : nullptr;
  const C2<Rm>* ncoef = split ? reinterpret_cast<const C2<Rm>*>(coef32) : reinterpret_cast<const C2<Rm>*>(coef);
  k_coef<Rio><<<nblk(pr.T, 256), 256, 0, st>>>(pr.T, pr.E, static_cast<const C2<Rio>*>(xv), pr.perm, pr.tri_edge,
                                               pr.tri_c, pr.tri_cdcp, pr.w * pr.w * eps0(), coef, coef32);
  if constexpr (sizeof(Rm) == 8) {
    near_fixed(pr, coef, pot, 1, 0, false, st);
  } else if (pr.tune.near_kernel != 1) {  // the box-staged kernel, unless tuned off
    const int nsplit = near_box_split(pr, kNearBoxThreads / 32), stage = near_box_stage<H16>(pr);
    k_near_box<Rio, H16><<<unsigned(pr.nleaf * nsplit), kNearBoxThreads, near_box_smem<H16>(stage), st>>>(
        pr.nleaf, nsplit, stage, pr.nnz, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr,
        static_cast<const cf*>(pr.mom), static_cast<const __half2*>(pr.mom), mom_scale(pr), ncoef, float(kMu0), pot);
  } else {
    k_near<Rm, Rio, 1, H16><<<nblk(pr.T * 32, 256), 256, 0, st>>>(
        pr.T, pr.nnz, pr.leaf_of, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr,
        static_cast<const C2<Rm>*>(pr.mom), static_cast<const __half2*>(pr.mom), mom_scale(pr), ncoef, Rm(kMu0),
        pot);
  }
  k_assemble<Rio><<<nblk(pr.N, 256), 256, 0, st>>>(pr.N, pr.E, pr.edge_tt, pr.edge_k, pr.tri_c, pr.tri_dcp,
                                                   pr.inv_perm, pot, static_cast<C2<Rio>*>(yv));
  return cuda_check(cudaGetLastError(), "apply_near launch");
}

pie_status apply_near_one(Problem& pr, const void* x, void* y, cudaStream_t st) {
  switch (pr.par.precision) {
    case PIE_FP64:
      return apply_near_t<double, double>(pr, x, y, st);
    case PIE_FP32:
      return apply_near_t<float, float>(pr, x, y, st);
    case PIE_FP32H:
      return apply_near_t<float, float, true>(pr, x, y, st);
    default:
      return apply_near_t<float, double>(pr, x, y, st);
  }
}

pie_status apply_batch(Problem& pr, const void* x, void* y, int nrhs, cudaStream_t st, const double* scale) {
  if (nrhs < 1 || nrhs > pr.par.max_nrhs) {
    set_error("batch larger than max_nrhs");
    return PIE_ERR_PARAM;
  }
  switch (pr.par.precision) {
    case PIE_FP64:
      return apply_t<double, double, double>(pr, x, y, nrhs, st, scale);
    case PIE_FP32:
      return apply_t<float, float, float>(pr, x, y, nrhs, st, scale);
    case PIE_MIXED:
      return apply_t<float, double, double>(pr, x, y, nrhs, st, scale);
    case PIE_FP32H:
      return apply_t<float, float, float, true>(pr, x, y, nrhs, st, scale);
  }
  set_error("unknown precision");
  return PIE_ERR_PARAM;
}

pie_status apply_one(Problem& pr, const void* x, void* y, cudaStream_t st, const double* scale) {
  return apply_batch(pr, x, y, 1, st, scale);
}

pie_status apply_cols(Problem& pr, const void* x, void* y, int nrhs, cudaStream_t st) {
  const size_t col = (pr.io_f32() ? sizeof(cf) : sizeof(cd)) * size_t(pr.N);
  const int chunk = std::max(1, std::min(pr.tune.rhs_chunk, pr.par.max_nrhs));
  for (int j = 0; j < nrhs; j += chunk) {
    pie_status s = apply_batch(pr, static_cast<const char*>(x) + col * j, static_cast<char*>(y) + col * j,
                               std::min(chunk, nrhs - j), st);
    if (s != PIE_OK) return s;
  }
  return PIE_OK;
}

// ---------------------------------------------------------------- right-hand side

// Per triangle (tree order) the integrals of the plane-wave potentials with
// the 7-point rule, stored in the potential layout so that k_assemble forms
// b_J = -<f_m, A> and b_sigma = -i w eps0 <p_t, Phi>:
//   U = -int (r - c_t).A,  V = -int A,  T1 = 0,  T2 = -i w eps0 int Phi.
template <typename Rio>
__global__ void k_rhs(int64_t T, const double* __restrict__ vert, const double* __restrict__ cent,
                      const double* __restrict__ area, double k0, double kx, double ky, double kz, double ex,
                      double ey, double ez, double E0, double weps, const double* __restrict__ rule,
                      C2<Rio>* __restrict__ pot) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= T) return;
  const double* v = vert + 9 * t;
  double Ur = 0, Ui = 0, Vr[3] = {0, 0, 0}, Vi[3] = {0, 0, 0}, Pr = 0, Pim = 0;
  for (int q = 0; q < 7; ++q) {
    double b0 = rule[4 * q], b1 = rule[4 * q + 1], b2 = rule[4 * q + 2], wq = rule[4 * q + 3] * area[t];
    double r[3];
    for (int d = 0; d < 3; ++d) r[d] = b0 * v[d] + b1 * v[3 + d] + b2 * v[6 + d];
    double s, c;
    sincos(k0 * (kx * r[0] + ky * r[1] + kz * r[2]), &s, &c);
    double er = ex * r[0] + ey * r[1] + ez * r[2];
    // Phi = -E0 (e.r) e^{i phase};  A = -(E0/c0)(e.r) khat e^{i phase}
    double phr = -E0 * er * c, phi = -E0 * er * s;
    Pr += wq * phr;
    Pim += wq * phi;
    double ar = phr / kC0, ai = phi / kC0;
    double kh[3] = {kx, ky, kz};
    double ud = 0;
    for (int d = 0; d < 3; ++d) ud += (r[d] - cent[3 * t + d]) * kh[d];
    Ur += wq * ud * ar;
    Ui += wq * ud * ai;
    for (int d = 0; d < 3; ++d) {
      Vr[d] += wq * kh[d] * ar;
      Vi[d] += wq * kh[d] * ai;
    }
  }
  C2<Rio>* o = pot + 6 * t;
  o[0] = mk<Rio>(Rio(-Ur), Rio(-Ui));
  for (int d = 0; d < 3; ++d) o[1 + d] = mk<Rio>(Rio(-Vr[d]), Rio(-Vi[d]));
  o[4] = mk<Rio>(0, 0);
  // -i weps (Pr + i Pim) = weps Pim - i weps Pr
  o[5] = mk<Rio>(Rio(weps * Pim), Rio(-weps * Pr));
}

pie_status rhs_planewave(Problem& pr, const double* khat, const double* pol, double E0, void* b, cudaStream_t st) {
  const double* rule = pr.rule7;
  const double weps = pr.w * eps0();
  if (pr.io_f32()) {
    k_rhs<float><<<nblk(pr.T, 128), 128, 0, st>>>(pr.T, pr.vert, pr.cent, pr.area, pr.k0, khat[0], khat[1], khat[2],
                                                  pol[0], pol[1], pol[2], E0, weps, rule, static_cast<cf*>(pr.pot));
    k_assemble<float><<<nblk(pr.N, 256), 256, 0, st>>>(pr.N, pr.E, pr.edge_tt, pr.edge_k, pr.tri_c, pr.tri_dcp,
                                                       pr.inv_perm, static_cast<cf*>(pr.pot), static_cast<cf*>(b));
  } else {
    k_rhs<double><<<nblk(pr.T, 128), 128, 0, st>>>(pr.T, pr.vert, pr.cent, pr.area, pr.k0, khat[0], khat[1], khat[2],
                                                   pol[0], pol[1], pol[2], E0, weps, rule, static_cast<cd*>(pr.pot));
    k_assemble<double><<<nblk(pr.N, 256), 256, 0, st>>>(pr.N, pr.E, pr.edge_tt, pr.edge_k, pr.tri_c, pr.tri_dcp,
                                                        pr.inv_perm, static_cast<cd*>(pr.pot), static_cast<cd*>(b));
  }
  return cuda_check(cudaGetLastError(), "rhs launch");
}

// Right-hand side for potentials given at the 7 quadrature points of every
// triangle (Eqs. (1)-(2)): U = -int (r - c_t).A, V = -int A, T1 = 0,
// T2 = -i w eps0 int Phi, tested by k_assemble into b_J = -<f_m, A>,
// b_sigma = -i w eps0 <p_t, Phi>.  Aq [T][7][3], Pq [T][7] in mesh order.
template <typename Rio>
__global__ void k_rhs_q(int64_t T, const int64_t* __restrict__ perm, const double* __restrict__ vert,
                        const double* __restrict__ cent, const double* __restrict__ area, const cd* __restrict__ Aq,
                        const cd* __restrict__ Pq, double weps, const double* __restrict__ rule,
                        C2<Rio>* __restrict__ pot) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= T) return;
  const int64_t m = perm[t];
  const double* v = vert + 9 * t;
  double Ur = 0, Ui = 0, Vr[3] = {0, 0, 0}, Vi[3] = {0, 0, 0}, Pr = 0, Pim = 0;
  for (int q = 0; q < 7; ++q) {
    const double b0 = rule[4 * q], b1 = rule[4 * q + 1], b2 = rule[4 * q + 2], wq = rule[4 * q + 3] * area[t];
    const cd* A = Aq + (m * 7 + q) * 3;
    const cd P = Pq[m * 7 + q];
    for (int d = 0; d < 3; ++d) {
      const double u = b0 * v[d] + b1 * v[3 + d] + b2 * v[6 + d] - cent[3 * t + d];
      Ur += wq * u * A[d].x;
      Ui += wq * u * A[d].y;
      Vr[d] += wq * A[d].x;
      Vi[d] += wq * A[d].y;
    }
    Pr += wq * P.x;
    Pim += wq * P.y;
  }
  C2<Rio>* o = pot + 6 * t;
  o[0] = mk<Rio>(Rio(-Ur), Rio(-Ui));
  for (int d = 0; d < 3; ++d) o[1 + d] = mk<Rio>(Rio(-Vr[d]), Rio(-Vi[d]));
  o[4] = mk<Rio>(0, 0);
  o[5] = mk<Rio>(Rio(weps * Pim), Rio(-weps * Pr));
}

pie_status rhs_potentials(Problem& pr, const void* Aq, const void* Pq, void* b, cudaStream_t st) {
  const double weps = pr.w * eps0();
  const cd* A = static_cast<const cd*>(Aq);
  const cd* P = static_cast<const cd*>(Pq);
  if (pr.io_f32()) {
    k_rhs_q<float><<<nblk(pr.T, 128), 128, 0, st>>>(pr.T, pr.perm, pr.vert, pr.cent, pr.area, A, P, weps, pr.rule7,
                                                    static_cast<cf*>(pr.pot));
    k_assemble<float><<<nblk(pr.N, 256), 256, 0, st>>>(pr.N, pr.E, pr.edge_tt, pr.edge_k, pr.tri_c, pr.tri_dcp,
                                                       pr.inv_perm, static_cast<cf*>(pr.pot), static_cast<cf*>(b));
  } else {
    k_rhs_q<double><<<nblk(pr.T, 128), 128, 0, st>>>(pr.T, pr.perm, pr.vert, pr.cent, pr.area, A, P, weps, pr.rule7,
                                                     static_cast<cd*>(pr.pot));
    k_assemble<double><<<nblk(pr.N, 256), 256, 0, st>>>(pr.N, pr.E, pr.edge_tt, pr.edge_k, pr.tri_c, pr.tri_dcp,
                                                        pr.inv_perm, static_cast<cd*>(pr.pot), static_cast<cd*>(b));
  }
  return cuda_check(cudaGetLastError(), "rhs launch");
}

// ---------------------------------------------------------------- far and near-zone fields
//
// The three field maps sum a phase over every (triangle, direction or point)
// pair and bind on the FP64 pipe (two fused multiply-adds per clock and SM),
// so they are written for few double operations.  The 7-point rule is the
// centroid and two orbits of three points r_ok = c + s_o v_k, v_k = vertex k -
// c, s_o = 1 - 3 a_o; so with sum_k v_k = 0 and J = a (r - c) + beta,
//   sum_q w_q J(r_q) e^{-i k rhat.r_q}
//     = A e^{-i k rhat.c} [beta C + a sum_k v_k D(p_k)],  p_k = k rhat.v_k,
//   C = w_0 + sum_k f(p_k),  f(p) = sum_o w_o e^{-i s_o p},
//   D(p) = sum_o w_o s_o (e^{-i s_o p} - 1):
// (the stored centroid's rounding, sum_k v_k = 3 e != 0, enters as beta + a e:
// left out it would be the largest error by far, 1e-16 |c| / h);
// one sincos per triangle and direction instead of seven, and f and D are
// power series whose coefficients carry the rule's moments.  p is at most
// 2/3 k h (h: longest edge of the mesh), so the number of terms follows from
// k h alone: NT terms (of the even and of the odd part) leave less than 1e-17.
// pie_problem_create bounds k h by 0.52 (leaf boxes of at least 1.5 h, k times
// a level-3 box of at most 0.77), which 7 terms cover.
constexpr int kFieldTerms = 7;
struct FieldRule {
  double w0, w[2], s[2];                                 // the rule: centroid and two orbits
  double fe[kFieldTerms], fo[kFieldTerms];               // f: even part, odd part / p
  double de[kFieldTerms], dO[kFieldTerms];               // D: even part, odd part / p
  double ce[kFieldTerms], so[kFieldTerms];               // cos, sin / p
};

static FieldRule field_rule(const Problem& pr) {
  FieldRule r{};
  const std::vector<double>& q = pr.rule7_host;
  r.w0 = q[3];
  for (int o = 0; o < 2; ++o) {
    r.w[o] = q[4 * (1 + 3 * o) + 3];
    r.s[o] = 1.0 - 3.0 * q[4 * (1 + 3 * o) + 1];
  }
  double fact = 1.0, pw[2] = {r.w[0], r.w[1]};  // n!, w_o s_o^n
  for (int n = 0; n < 2 * kFieldTerms; ++n) {
    if (n > 0) fact *= n;
    const double sg = (n / 2) % 2 ? -1.0 : 1.0;
    const double f = sg * (pw[0] + pw[1]) / fact;
    for (int o = 0; o < 2; ++o) pw[o] *= r.s[o];
    const double d = n == 0 ? 0.0 : sg * (pw[0] + pw[1]) / fact;
    (n % 2 ? r.fo : r.fe)[n / 2] = n % 2 ? -f : f;
    (n % 2 ? r.dO : r.de)[n / 2] = n % 2 ? -d : d;
    (n % 2 ? r.so : r.ce)[n / 2] = sg / fact;
  }
  return r;
}

// Terms for phases up to 2/3 k h: 3 below k h = 6e-3, 5 below 0.13, 7 up to
// kMaxFieldKh (first omitted term (2/3 k h)^(2 NT) / (2 NT)! < 1e-17).  A longer
// direction than a unit vector scales the phases and may leave that range: NT = 0,
// sine and cosine of each orbit.
constexpr double kMaxFieldKh = 0.52;
static int field_terms(double kh) { return kh < 6e-3 ? 3 : kh < 0.13 ? 5 : kh <= kMaxFieldKh ? 7 : 0; }

// Length of the longest of n vectors.
static double longest(const double* v, int64_t n) {
  double r2 = 0;
  for (int64_t i = 0; i < n; ++i)
    r2 = std::max(r2, v[3 * i] * v[3 * i] + v[3 * i + 1] * v[3 * i + 1] + v[3 * i + 2] * v[3 * i + 2]);
  return std::sqrt(r2);
}

// Phase of a centroid: 5 terms below 0.09 and 6 below 0.2 (bodies well below a
// wavelength, the method's range; a fifth of a pair's operations less than
// sincos, a term 2 % of the adjoint map; first omitted terms 0.09^10 / 10! = 1e-17 and
// 0.2^12 / 12! = 9e-18), else sincos (CT = 0).
static int centroid_terms(double phase) { return phase < 0.09 ? 5 : phase < 0.2 ? 6 : 0; }

template <int NT>
__device__ __forceinline__ double horner(const double* c, double z) {
  double v = c[NT - 1];
#pragma unroll
  for (int j = NT - 2; j >= 0; --j) v = fma(v, z, c[j]);
  return v;
}

template <int CT>
__device__ __forceinline__ void field_sincos(const FieldRule& R, double p, double* s, double* c) {
  if constexpr (CT == 0) {
    sincos(p, s, c);
  } else {
    const double z = p * p;
    *c = horner<CT>(R.ce, z);
    *s = p * horner<CT>(R.so, z);
  }
}

// f(p) added to C, D(p) returned (NT = 0: D but for a constant, which cancels in G_k).
template <int NT>
__device__ __forceinline__ cd field_phase(const FieldRule& R, double p, cd& C) {
  if constexpr (NT == 0) {
    // (both orbits written out: as a loop, nvcc 13.0 left a term out of C)
    cd D = mk<double>(0, 0);
    double s0, c0, s1, c1;
    sincos(R.s[0] * p, &s0, &c0);
    sincos(R.s[1] * p, &s1, &c1);
    const cd e0 = mk<double>(R.w[0] * c0, -R.w[0] * s0), e1 = mk<double>(R.w[1] * c1, -R.w[1] * s1);
    C.x += e0.x + e1.x;
    C.y += e0.y + e1.y;
    rfma(D, R.s[0], e0);
    rfma(D, R.s[1], e1);
    return D;
  } else {
    const double z = p * p;
    C.x += horner<NT>(R.fe, z);
    C.y = fma(p, horner<NT>(R.fo, z), C.y);
    return mk<double>(horner<NT>(R.de, z), p * horner<NT>(R.dO, z));
  }
}

// C and G_k = D(p_k) - D(p_2), k = 0, 1 (sum_k v_k D_k = v_0 G_0 + v_1 G_1).
template <int NT>
__device__ __forceinline__ void field_triangle(const FieldRule& R, double p0, double p1, cd& C, cd& G0, cd& G1) {
  C = mk<double>(R.w0, 0);
  const cd D2 = field_phase<NT>(R, -(p0 + p1), C);
  G0 = field_phase<NT>(R, p0, C);
  G1 = field_phase<NT>(R, p1, C);
  G0 = mk<double>(G0.x - D2.x, G0.y - D2.y);
  G1 = mk<double>(G1.x - D2.x, G1.y - D2.y);
}

// A warp per (direction or point, chunk of triangles): lanes stride over the
// chunk, the six sums are reduced once per warp and the chunks' partial sums
// are added in order by k_field_finish, so the sum does not depend on
// scheduling.  Chunks are cut by the number of triangles alone, so that a field
// does not depend on the directions or points beside it either: at least
// `least` triangles (128, four a lane; the warp's reduction is eight adds) and at
// most kFieldChunks chunks, which gives one direction a few hundred warps.
// (One block per direction left the pipe idle: 181 directions on 152 SMs.)
constexpr int64_t kFieldChunks = 1024;
static void field_chunks(const Problem& pr, int64_t least, int64_t* nchunk, int64_t* len) {
  *len = std::max(least, ((pr.T + kFieldChunks - 1) / kFieldChunks + 31) / 32 * 32);
  *nchunk = (pr.T + *len - 1) / *len;
}

// Scratch of one field call: the leaf sum / difference patterns, which only
// live inside a product, or a stream-ordered allocation where they are too
// small.  The maps and the adjoint map share no other buffer, so a call waits on
// the device for the last one that used the patterns, whatever its stream (not
// inside a stream capture, whose launches are the caller's to order).
struct FieldScratch {
  void* p = nullptr;
  cudaStream_t st;
  cudaEvent_t done = nullptr;
  bool own = false;
  FieldScratch(Problem& pr, size_t bytes, cudaStream_t s_, pie_status& s) : st(s_) {
    if (bytes <= pr.gsgd_bytes) {
      p = pr.gsgd;
      cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
      s = cuda_check(cudaStreamIsCapturing(st, &cap), "capture status");
      if (s != PIE_OK || cap != cudaStreamCaptureStatusNone) return;
      done = pr.ev_field;
      s = cuda_check(cudaStreamWaitEvent(st, done, 0), "field scratch");
      return;
    }
    s = cuda_check(cudaMallocAsync(&p, bytes, st), "field scratch");
    own = s == PIE_OK;
  }
  ~FieldScratch() {
    if (own) cudaFreeAsync(p, st);
    if (done) cudaEventRecord(done, st);
  }
};

// Directions or points of one launch: their partial sums take at most kFieldScratch bytes.
constexpr size_t kFieldScratch = size_t(64) << 20;
static int64_t field_batch(int64_t n, int64_t nchunk) {
  return std::min<int64_t>(n, std::max<int64_t>(1, int64_t(kFieldScratch / (6 * sizeof(double) * size_t(nchunk)))));
}

// The warp's six sums into out[0..5], each step of the butterfly keeping half of
// the values on either side (8 adds a lane instead of 30).
__device__ __forceinline__ void field_partial(const double (&S)[6], double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
  auto step = [](bool up, double lo, double hi, int o) {
    const double keep = up ? hi : lo, send = up ? lo : hi;
    return keep + __shfl_xor_sync(0xffffffffu, send, o);
  };
  double x[3], y[2];
#pragma unroll
  for (int i = 0; i < 3; ++i) x[i] = step(h4, S[i], S[3 + i], 16);
  y[0] = step(h3, x[0], x[2], 8);
  y[1] = step(h3, x[1], 0.0, 8);
  double z = step(h2, y[0], y[1], 4);
  z += __shfl_xor_sync(0xffffffffu, z, 2);
  z += __shfl_xor_sync(0xffffffffu, z, 1);
  if ((lane & 3) == 0 && !(h3 && h2)) out[(h4 ? 3 : 0) + (h3 ? 2 : 0) + (h2 ? 1 : 0)] = z;
}

// Far field: partial sums of F = sum_t int J exp(-i k0 rhat.r).  181
// directions on 81,920 triangles: 3.06 ms; a block per direction with a sincos
// per quadrature point took 20.4 ms.
template <typename Rio, int NT, int CT>
__global__ void __launch_bounds__(128) k_farfield(int64_t T, int64_t ndir, int64_t nchunk, int64_t len,
                                                  const double* __restrict__ vert, const double* __restrict__ cent,
                                                  const double* __restrict__ area, const C2<Rio>* __restrict__ coef,
                                                  const double* __restrict__ rhat, double k0, const FieldRule R,
                                                  double* __restrict__ partial) {
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (w >= ndir * nchunk) return;
  const int64_t dir = w % ndir, ch = w / ndir;
  const double kx = k0 * rhat[3 * dir], ky = k0 * rhat[3 * dir + 1], kz = k0 * rhat[3 * dir + 2];
  double S[6] = {0, 0, 0, 0, 0, 0};
  const int64_t t1 = min(T, (ch + 1) * len);
  for (int64_t t = ch * len + (threadIdx.x & 31); t < t1; t += 32) {
    const double cx = cent[3 * t], cy = cent[3 * t + 1], cz = cent[3 * t + 2];
    const double* v = vert + 9 * t;
    const double v0[3] = {v[0] - cx, v[1] - cy, v[2] - cz}, v1[3] = {v[3] - cx, v[4] - cy, v[5] - cz};
    cd C, G0, G1;
    field_triangle<NT>(R, kx * v0[0] + ky * v0[1] + kz * v0[2], kx * v1[0] + ky * v1[1] + kz * v1[2], C, G0, G1);
    double s, c;
    field_sincos<CT>(R, kx * cx + ky * cy + kz * cz, &s, &c);
    const C2<Rio>* o = coef + 6 * t;
    const cd a = cvt<double>(o[0]);
    // times A e^{-i phase}, shared by the three components
    const double A = area[t];
    const cd e = mk<double>(A * c, -A * s);
    const cd eC = cmul(e, C), ea = cmul(e, a);
    const cd h0 = cmul(ea, G0), h1 = cmul(ea, G1);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const cd b = cvt<double>(o[1 + d]);
      S[d] += eC.x * b.x - eC.y * b.y + v0[d] * h0.x + v1[d] * h1.x;
      S[3 + d] += eC.x * b.y + eC.y * b.x + v0[d] * h0.y + v1[d] * h1.y;
    }
  }
  field_partial(S, partial + 6 * (dir * nchunk + ch));
}

// Sums the chunks of one direction or point (a warp each, lanes over chunks
// in a fixed order); with rhat also E = i w mu0/(4 pi) (I - rr) F.
__global__ void k_field_finish(int64_t n, int64_t nchunk, const double* __restrict__ partial,
                               const double* __restrict__ rhat, double pref, cd* __restrict__ E) {
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (w >= n) return;
  const int lane = threadIdx.x & 31;
  double S[6] = {0, 0, 0, 0, 0, 0};
  for (int64_t c = lane; c < nchunk; c += 32)
#pragma unroll
    for (int i = 0; i < 6; ++i) S[i] += partial[6 * (w * nchunk + c) + i];
#pragma unroll
  for (int i = 0; i < 6; ++i) S[i] = warp_sum(S[i]);
  if (lane) return;
  if (!rhat) {
    for (int d = 0; d < 3; ++d) E[3 * w + d] = mk<double>(S[d], S[3 + d]);
    return;
  }
  const double* r = rhat + 3 * w;
  const double dr = r[0] * S[0] + r[1] * S[1] + r[2] * S[2], di = r[0] * S[3] + r[1] * S[4] + r[2] * S[5];
  for (int d = 0; d < 3; ++d)  // i pref (tr + i ti) = -pref ti + i pref tr
    E[3 * w + d] = mk<double>(-pref * (S[3 + d] - r[d] * di), pref * (S[d] - r[d] * dr));
}

// beta += a e with 3 e = sum_k v_k, the rounding of the stored centroid.
__global__ void k_field_coef(int64_t T, const double* __restrict__ vert, const double* __restrict__ cent,
                             cd* __restrict__ coef) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= T) return;
  const double* v = vert + 9 * t;
  cd* o = coef + 6 * t;
  const cd a = o[0];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double c = cent[3 * t + d];
    rfma(o[1 + d], ((v[d] - c) + (v[3 + d] - c) + (v[6 + d] - c)) / 3.0, a);
  }
}

// Local coefficients of the solution x for the field maps.
template <typename Rio>
static C2<Rio>* field_coef(Problem& pr, const void* x, cudaStream_t st) {
  C2<Rio>* coef = static_cast<C2<Rio>*>(pr.coef);
  k_coef<Rio><<<nblk(pr.T, 256), 256, 0, st>>>(pr.T, pr.E, static_cast<const C2<Rio>*>(x), pr.perm, pr.tri_edge,
                                               pr.tri_c, pr.tri_cdcp, pr.w * pr.w * eps0(), coef, nullptr);
  if constexpr (sizeof(Rio) == 8) k_field_coef<<<nblk(pr.T, 256), 256, 0, st>>>(pr.T, pr.vert, pr.cent, coef);
  return coef;
}

// Runs f(integral_constant<NT>, integral_constant<CT>) for the numbers of
// series terms at k h and at phase, the largest phase of a centroid.  ANY: k h
// may exceed kMaxFieldKh.
template <bool ANY, typename F>
static void with_field_terms(double kh, double phase, F f) {
  auto with_ct = [&](auto nt) {
    switch (centroid_terms(phase)) {
      case 5: return f(nt, std::integral_constant<int, 5>());
      case 6: return f(nt, std::integral_constant<int, 6>());
      default: return f(nt, std::integral_constant<int, 0>());
    }
  };
  if constexpr (ANY)
    if (field_terms(kh) == 0) return f(std::integral_constant<int, 0>(), std::integral_constant<int, 0>());
  switch (field_terms(kh)) {
    case 3: return with_ct(std::integral_constant<int, 3>());
    case 5: return with_ct(std::integral_constant<int, 5>());
    default: return with_ct(std::integral_constant<int, 7>());
  }
}

template <typename Rio>
static pie_status farfield_t(Problem& pr, const void* x, const double* rhat, int64_t ndir, void* E, cudaStream_t st) {
  int64_t nchunk, len;
  field_chunks(pr, 128, &nchunk, &len);
  const int64_t batch = field_batch(ndir, nchunk);
  pie_status s = PIE_OK;
  FieldScratch scratch(pr, sizeof(double) * (3 * size_t(ndir) + 6 * size_t(nchunk * batch)), st, s);
  if (s != PIE_OK) return s;
  double* d_rhat = static_cast<double*>(scratch.p);
  double* partial = d_rhat + 3 * ndir;
  s = cuda_check(cudaMemcpyAsync(d_rhat, rhat, sizeof(double) * 3 * ndir, cudaMemcpyHostToDevice, st), "copy");
  if (s != PIE_OK) return s;
  const C2<Rio>* coef = field_coef<Rio>(pr, x, st);
  const FieldRule R = field_rule(pr);
  const double k = pr.k0 * longest(rhat, ndir);
  with_field_terms<true>(k * pr.h_max, k * pr.r_max, [&](auto nt, auto ct) {
    for (int64_t d = 0; d < ndir; d += batch) {
      const int64_t n = std::min(batch, ndir - d);
      k_farfield<Rio, decltype(nt)::value, decltype(ct)::value><<<nblk(n * nchunk * 32, 128), 128, 0, st>>>(
          pr.T, n, nchunk, len, pr.vert, pr.cent, pr.area, coef, d_rhat + 3 * d, pr.k0, R, partial);
      k_field_finish<<<nblk(n * 32, 128), 128, 0, st>>>(n, nchunk, partial, d_rhat + 3 * d, pr.w * kMu0 / (4.0 * kPi),
                                                        static_cast<cd*>(E) + 3 * d);
    }
  });
  return cuda_check(cudaGetLastError(), "farfield launch");
}

pie_status farfield(Problem& pr, const void* x, const double* rhat, int64_t ndir, void* E, cudaStream_t st) {
  return pr.io_f32() ? farfield_t<float>(pr, x, rhat, ndir, E, st) : farfield_t<double>(pr, x, rhat, ndir, E, st);
}

}  // namespace pie

namespace pie {

// Near part with caller-chosen scratch for the per-triangle coefficients and
// potentials (each [T][6] complex of the problem's io type).
pie_status apply_near_scratch(Problem& pr, const void* x, void* y, void* coef, void* pot, cudaStream_t st) {
  const double w2e = pr.w * pr.w * eps0();
  if (pr.io_f32()) {
    k_coef<float><<<nblk(pr.T, 256), 256, 0, st>>>(pr.T, pr.E, static_cast<const cf*>(x), pr.perm, pr.tri_edge,
                                                   pr.tri_c, pr.tri_cdcp, w2e, static_cast<cf*>(coef), nullptr);
    if (pr.near_h16())
      k_near<float, float, 1, true><<<nblk(pr.T * 32, 256), 256, 0, st>>>(
          pr.T, pr.nnz, pr.leaf_of, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr, nullptr,
          static_cast<const __half2*>(pr.mom), mom_scale(pr), static_cast<const cf*>(coef), float(kMu0),
          static_cast<cf*>(pot));
    else
      k_near<float, float><<<nblk(pr.T * 32, 256), 256, 0, st>>>(
          pr.T, pr.nnz, pr.leaf_of, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr,
          static_cast<const cf*>(pr.mom), nullptr, mom_scale(pr), static_cast<const cf*>(coef), float(kMu0),
          static_cast<cf*>(pot));
    k_assemble<float><<<nblk(pr.N, 256), 256, 0, st>>>(pr.N, pr.E, pr.edge_tt, pr.edge_k, pr.tri_c, pr.tri_dcp,
                                                       pr.inv_perm, static_cast<const cf*>(pot), static_cast<cf*>(y));
  } else {
    const bool split = pr.near_f32();
    k_coef<double><<<nblk(pr.T, 256), 256, 0, st>>>(pr.T, pr.E, static_cast<const cd*>(x), pr.perm, pr.tri_edge,
                                                    pr.tri_c, pr.tri_cdcp, w2e, split ? nullptr : static_cast<cd*>(coef),
                                                    split ? static_cast<cf*>(coef) : nullptr);
    if (split)
      k_near<float, double><<<nblk(pr.T * 32, 256), 256, 0, st>>>(
          pr.T, pr.nnz, pr.leaf_of, pr.leaf_start, pr.near_ptr, pr.near_idx, pr.near_off, pr.row_ptr,
          static_cast<const cf*>(pr.mom), nullptr, mom_scale(pr), static_cast<const cf*>(coef), float(kMu0),
          static_cast<cd*>(pot));
    else
      near_fixed(pr, static_cast<const cd*>(coef), static_cast<cd*>(pot), 1, 0, false, st);
    k_assemble<double><<<nblk(pr.N, 256), 256, 0, st>>>(pr.N, pr.E, pr.edge_tt, pr.edge_k, pr.tri_c, pr.tri_dcp,
                                                        pr.inv_perm, static_cast<const cd*>(pot), static_cast<cd*>(y));
  }
  return cuda_check(cudaGetLastError(), "apply_near_noalloc launch");
}

}  // namespace pie

namespace pie {

// ---------------------------------------------------------------- adjoint

template <typename R>
__global__ void k_conj(int64_t n, const C2<R>* __restrict__ x, C2<R>* __restrict__ y) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) y[i] = mk<R>(x[i].x, -x[i].y);
}

// y = Z^T x (conj = false) or Z^H x = conj(Z conj x) (conj = true).  The
// discrete operator is complex symmetric -- the near pair moments by the
// two-sided near-singular rule, the far part by the antipodal angular grid
// (aggregation and disaggregation are each other's transposes, F^T is the
// anterpolation of F, T_{-w}(k) = T_w(-k)) -- so Z^T x runs the same stages.
pie_status apply_t_one(Problem& pr, const void* x, void* y, bool conj, cudaStream_t st) {
  if (!conj) return apply_one(pr, x, y, st);
  const int64_t N = pr.N;
  if (pr.io_f32()) {
    k_conj<float><<<nblk(N, 256), 256, 0, st>>>(N, static_cast<const cf*>(x), static_cast<cf*>(pr.vec));
    pie_status s = apply_one(pr, pr.vec, y, st);
    if (s != PIE_OK) return s;
    k_conj<float><<<nblk(N, 256), 256, 0, st>>>(N, static_cast<const cf*>(y), static_cast<cf*>(y));
  } else {
    k_conj<double><<<nblk(N, 256), 256, 0, st>>>(N, static_cast<const cd*>(x), static_cast<cd*>(pr.vec));
    pie_status s = apply_one(pr, pr.vec, y, st);
    if (s != PIE_OK) return s;
    k_conj<double><<<nblk(N, 256), 256, 0, st>>>(N, static_cast<const cd*>(y), static_cast<cd*>(y));
  }
  return cuda_check(cudaGetLastError(), "adjoint launch");
}

// Adjoint of the far-field map x -> E (Section 2 far zone): with
// h(r) = sum_d conj(i w mu0 / 4 pi) exp(+i k rhat_d . r) (I - rhat_d rhat_d) E_d,
// (F^H E)_m = sum_{t in m} c_t,m int_t (r - p_m) . h(r) dr, i.e. the Galerkin
// testing of the potentials U = int (r - c_t).h, V = int h (T1 = T2 = 0).
// One thread per triangle over a chunk of the directions (blockIdx.y; enough
// chunks to give every SM kAdjWarps warps, of at least eight directions), the conjugates of the far field's C and
// G_k per pair; kAdjTile directions at a time in shared memory, each as k rhat
// and the vector -i pref (I - rr) E.  A launch of one chunk writes the
// potentials, otherwise out holds the chunks' partial sums [chunk][8][T].
// 181 directions on 32,768 triangles: 1.16 ms; 5.12 ms with a sincos per
// quadrature point.
constexpr int kAdjTile = 32, kAdjWarps = 32;
template <typename Rio, int NT, int CT>
__global__ void __launch_bounds__(128) k_farfield_adj(int64_t T, int64_t ndir, int64_t len,
                                                      const double* __restrict__ vert,
                                                      const double* __restrict__ cent,
                                                      const double* __restrict__ area,
                                                      const double* __restrict__ rhat, const cd* __restrict__ E,
                                                      double k0, double pref, const FieldRule R,
                                                      C2<Rio>* __restrict__ pot, double* __restrict__ out) {
  __shared__ double sm[kAdjTile][9];
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool live = t < T;
  const int64_t tt = live ? t : T - 1;
  const double cx = cent[3 * tt], cy = cent[3 * tt + 1], cz = cent[3 * tt + 2];
  const double* v = vert + 9 * tt;
  const double v0[3] = {v[0] - cx, v[1] - cy, v[2] - cz}, v1[3] = {v[3] - cx, v[4] - cy, v[5] - cz};
  cd U = mk<double>(0, 0), V[3] = {U, U, U};
  const int64_t d1 = min(ndir, (blockIdx.y + 1) * len);
  for (int64_t d0 = blockIdx.y * len; d0 < d1; d0 += kAdjTile) {
    const int n = int(min(int64_t(kAdjTile), d1 - d0));
    __syncthreads();
    if (int(threadIdx.x) < n) {
      const double* r = rhat + 3 * (d0 + threadIdx.x);
      const cd* e = E + 3 * (d0 + threadIdx.x);
      const double er = r[0] * e[0].x + r[1] * e[1].x + r[2] * e[2].x;
      const double ei = r[0] * e[0].y + r[1] * e[1].y + r[2] * e[2].y;
      for (int d = 0; d < 3; ++d) {
        sm[threadIdx.x][d] = k0 * r[d];
        sm[threadIdx.x][3 + 2 * d] = pref * (e[d].y - r[d] * ei);
        sm[threadIdx.x][4 + 2 * d] = -pref * (e[d].x - r[d] * er);
      }
    }
    __syncthreads();
    for (int i = 0; i < n; ++i) {
      const double kx = sm[i][0], ky = sm[i][1], kz = sm[i][2];
      cd C, G0, G1;
      field_triangle<NT>(R, kx * v0[0] + ky * v0[1] + kz * v0[2], kx * v1[0] + ky * v1[1] + kz * v1[2], C, G0, G1);
      double s, c;
      field_sincos<CT>(R, kx * cx + ky * cy + kz * cz, &s, &c);
      // e^{i phase} conj(X) = conj(e^{-i phase} X)
      const cd e = mk<double>(c, -s);
      C = cmul(e, C);
      G0 = cmul(e, G0);
      G1 = cmul(e, G1);
      cd h0 = mk<double>(0, 0), h1 = h0;  // v_k . E
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const cd b = mk<double>(sm[i][3 + 2 * d], sm[i][4 + 2 * d]);
        cfma_conj(V[d], C, b);
        rfma(h0, v0[d], b);
        rfma(h1, v1[d], b);
      }
      cfma_conj(U, G0, h0);
      cfma_conj(U, G1, h1);
    }
  }
  if (!live) return;
#pragma unroll
  for (int d = 0; d < 3; ++d)  // the centroid's rounding
    rfma(U, (v0[d] + v1[d] + (v[6 + d] - cent[3 * t + d])) / 3.0, V[d]);
  const double A = area[t];
  if (gridDim.y > 1) {
    double* o = out + int64_t(blockIdx.y) * 8 * T + t;
    o[0] = A * U.x;
    o[T] = A * U.y;
    for (int d = 0; d < 3; ++d) {
      o[(2 + 2 * d) * T] = A * V[d].x;
      o[(3 + 2 * d) * T] = A * V[d].y;
    }
    return;
  }
  C2<Rio>* o = pot + 6 * t;
  o[0] = mk<Rio>(Rio(A * U.x), Rio(A * U.y));
  for (int d = 0; d < 3; ++d) o[1 + d] = mk<Rio>(Rio(A * V[d].x), Rio(A * V[d].y));
  o[4] = o[5] = mk<Rio>(0, 0);
}

// Adds the direction chunks' partial sums in order.
template <typename Rio>
__global__ void k_farfield_adj_finish(int64_t T, int64_t nchunk, const double* __restrict__ in,
                                      C2<Rio>* __restrict__ pot) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= T) return;
  double S[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int64_t c = 0; c < nchunk; ++c)
#pragma unroll
    for (int i = 0; i < 8; ++i) S[i] += in[(c * 8 + i) * T + t];
  C2<Rio>* o = pot + 6 * t;
#pragma unroll
  for (int i = 0; i < 4; ++i) o[i] = mk<Rio>(Rio(S[2 * i]), Rio(S[2 * i + 1]));
  o[4] = o[5] = mk<Rio>(0, 0);
}

template <typename Rio>
static pie_status farfield_adjoint_t(Problem& pr, const double* rhat, int64_t ndir, const void* E, void* u,
                                     cudaStream_t st) {
  const int64_t warps = (pr.T + 31) / 32;
  const int64_t most = std::min((int64_t(pr.nsm) * kAdjWarps + warps - 1) / warps, (ndir + 7) / 8);
  const int64_t len = ((ndir + most - 1) / most + 3) / 4 * 4, nchunk = (ndir + len - 1) / len;
  pie_status s = PIE_OK;
  FieldScratch scratch(pr, sizeof(double) * (3 * size_t(ndir) + (nchunk > 1 ? 8 * size_t(pr.T) * nchunk : 0)), st, s);
  if (s != PIE_OK) return s;
  double* d_rhat = static_cast<double*>(scratch.p);
  double* partial = d_rhat + 3 * ndir;
  s = cuda_check(cudaMemcpyAsync(d_rhat, rhat, sizeof(double) * 3 * ndir, cudaMemcpyHostToDevice, st), "copy");
  if (s != PIE_OK) return s;
  C2<Rio>* pot = static_cast<C2<Rio>*>(pr.pot);
  const FieldRule R = field_rule(pr);
  const double k = pr.k0 * longest(rhat, ndir);
  with_field_terms<true>(k * pr.h_max, k * pr.r_max, [&](auto nt, auto ct) {
    k_farfield_adj<Rio, decltype(nt)::value, decltype(ct)::value><<<dim3(nblk(pr.T, 128), unsigned(nchunk)), 128, 0, st>>>(
        pr.T, ndir, len, pr.vert, pr.cent, pr.area, d_rhat, static_cast<const cd*>(E), pr.k0,
        pr.w * kMu0 / (4.0 * kPi), R, pot, partial);
  });
  if (nchunk > 1) k_farfield_adj_finish<Rio><<<nblk(pr.T, 128), 128, 0, st>>>(pr.T, nchunk, partial, pot);
  k_assemble<Rio><<<nblk(pr.N, 256), 256, 0, st>>>(pr.N, pr.E, pr.edge_tt, pr.edge_k, pr.tri_c, pr.tri_dcp,
                                                   pr.inv_perm, pot, static_cast<C2<Rio>*>(u));
  return cuda_check(cudaGetLastError(), "farfield adjoint launch");
}

pie_status farfield_adjoint(Problem& pr, const double* rhat, int64_t ndir, const void* E, void* u, cudaStream_t st) {
  return pr.io_f32() ? farfield_adjoint_t<float>(pr, rhat, ndir, E, u, st)
                     : farfield_adjoint_t<double>(pr, rhat, ndir, E, u, st);
}

}  // namespace pie

namespace pie {

// ---------------------------------------------------------------- Eq. (3) and near-zone fields

// out = src[off:off+n] * scale
__global__ void k_slice_scale(int64_t n, const cd* __restrict__ src, double scale, cd* __restrict__ out) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) out[i] = mk<double>(scale * src[i].x, scale * src[i].y);
}

// Single layer of Eq. (3): y_t = <p_t, g, q> for pulse coefficients q
// (mesh order).  It is the pulse-pulse block of the PIE operator divided by
// w^2 eps0, applied to [0 ; q] through the same near and far stages.
pie_status single_layer_one(Problem& pr, const void* q, void* y, cudaStream_t st) {
  const int64_t E = pr.E, T = pr.T;
  cd* v = static_cast<cd*>(pr.vec);
  cd* v2 = static_cast<cd*>(pr.vec2);
  pie_status s = cuda_check(cudaMemsetAsync(v, 0, sizeof(cd) * E, st), "memset");
  if (s == PIE_OK) s = cuda_check(cudaMemcpyAsync(v + E, q, sizeof(cd) * T, cudaMemcpyDeviceToDevice, st), "copy");
  if (s == PIE_OK) s = apply_one(pr, v, v2, st);
  if (s != PIE_OK) return s;
  k_slice_scale<<<nblk(T, 256), 256, 0, st>>>(T, v2 + E, 1.0 / (pr.w * pr.w * eps0()), static_cast<cd*>(y));
  return cuda_check(cudaGetLastError(), "single layer launch");
}

// b_t = <p_t, Phi^inc> = int_t Phi^inc for the plane-wave potential
// Phi^inc = -E0 (pol.r) exp(i k khat.r); 7-point rule; b in mesh order.
__global__ void k_phi_inc(int64_t T, const double* __restrict__ vert, const double* __restrict__ area,
                          const int64_t* __restrict__ perm, double k0, double kx, double ky, double kz, double ex,
                          double ey, double ez, double E0, const double* __restrict__ rule, cd* __restrict__ b) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= T) return;
  const double* v = vert + 9 * t;
  double pr_ = 0, pi_ = 0;
  for (int q = 0; q < 7; ++q) {
    double r[3];
    for (int d = 0; d < 3; ++d) r[d] = rule[4 * q] * v[d] + rule[4 * q + 1] * v[3 + d] + rule[4 * q + 2] * v[6 + d];
    const double wq = rule[4 * q + 3] * area[t];
    double s, c;
    sincos(k0 * (kx * r[0] + ky * r[1] + kz * r[2]), &s, &c);
    const double er = ex * r[0] + ey * r[1] + ez * r[2];
    pr_ += -wq * E0 * er * c;
    pi_ += -wq * E0 * er * s;
  }
  b[perm[t]] = mk<double>(pr_, pi_);
}

pie_status rhs_potential(Problem& pr, const double* khat, const double* pol, double E0, void* b, cudaStream_t st) {
  k_phi_inc<<<nblk(pr.T, 128), 128, 0, st>>>(pr.T, pr.vert, pr.area, pr.perm, pr.k0, khat[0], khat[1], khat[2],
                                             pol[0], pol[1], pol[2], E0, pr.rule7, static_cast<cd*>(b));
  return cuda_check(cudaGetLastError(), "rhs potential launch");
}

// Scattered field at observation points off the surface (Section 2:
// near-zone E from J and the charge density rho):
//   E_s(r) = i w mu0 sum_t int_t J g  -  (1/eps0) sum_t rho_t int_t grad_r g,
// grad_r g = (r - r') (i k - 1/R) g / R; 7-point rule on every triangle (the
// rule is accurate for points farther than about a triangle size).  coef
// holds the local coefficients of J (tree order), rho the pulse coefficients
// of the charge density (mesh order).
// A warp per (point, chunk of triangles), as k_farfield.  e^{ikR_q} =
// e^{ikR_c} e^{ik(R_q - R_c)} with the centroid's distance R_c: one sincos per
// triangle, a short series per quadrature point, and 1/R from one rsqrt (no
// division).  With g_q = w_q e^{ik(R_q - R_c)} / R_q and F_q = g_q (ik - 1/R_q)/R_q
// the sums over an orbit need sum g, sum_o s_o g_ok, sum F, sum_o s_o F_ok only:
// J and r - r' are affine in s_o v_k.  1024 points, 20,480 triangles: 13.2 ms;
// 42.0 ms with a block per point, a sincos and five divisions per quadrature
// point.
template <int NT, int CT>
__global__ void __launch_bounds__(128) k_nearzone(int64_t T, int64_t npts, int64_t nchunk, int64_t len,
                                                  const double* __restrict__ vert, const double* __restrict__ cent,
                                                  const double* __restrict__ area, const int64_t* __restrict__ perm,
                                                  const cd* __restrict__ coef, const cd* __restrict__ rho,
                                                  const double* __restrict__ pts, double k0, double wmu,
                                                  double inv_eps, const FieldRule Q, double* __restrict__ partial) {
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (w >= npts * nchunk) return;
  const int64_t ip = w % npts, ch = w / npts;
  const double px = pts[3 * ip], py = pts[3 * ip + 1], pz = pts[3 * ip + 2];
  double S[6] = {0, 0, 0, 0, 0, 0};
  const int64_t t1 = min(T, (ch + 1) * len);
  for (int64_t t = ch * len + (threadIdx.x & 31); t < t1; t += 32) {
    const double c[3] = {cent[3 * t], cent[3 * t + 1], cent[3 * t + 2]};
    const double x[3] = {px - c[0], py - c[1], pz - c[2]};
    const double R2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
    const double i0 = rsqrt(R2), R0 = R2 * i0;
    // common factor A e^{ik R_0} / (4 pi), times i w mu0 for J (ea: times a)
    // and -rho / eps0 for the gradient
    double sn, cs;
    field_sincos<CT>(Q, k0 * R0, &sn, &cs);
    const double A = area[t] * (1.0 / (4.0 * kPi));
    const cd ej = mk<double>(-wmu * A * sn, wmu * A * cs), r = rho[perm[t]];
    const cd er = cmul(mk<double>(A * cs, A * sn), mk<double>(-inv_eps * r.x, -inv_eps * r.y));
    const cd* o6 = coef + 6 * t;
    const cd ea = cmul(ej, o6[0]);
    // centroid: g = w_0 / R_0
    cd g = mk<double>(Q.w0 * i0, 0), F = mk<double>(-g.x * i0 * i0, k0 * g.x * i0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double* v = vert + 9 * t + 3 * k;
      const double u[3] = {v[0] - c[0], v[1] - c[1], v[2] - c[2]};
      cd gk = mk<double>(0, 0), Fk = gk;
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const double dx = fma(-Q.s[o], u[0], x[0]), dy = fma(-Q.s[o], u[1], x[1]), dz = fma(-Q.s[o], u[2], x[2]);
        const double q2 = dx * dx + dy * dy + dz * dz;
        const double ri = rsqrt(q2);
        double sp, cp;
        field_sincos<NT>(Q, k0 * fma(q2, ri, -R0), &sp, &cp);
        const double wr = Q.w[o] * ri;
        const cd h = mk<double>(wr * cp, wr * sp);
        // h (ik - 1/R) / R
        const cd f = mk<double>(-ri * fma(h.x, ri, k0 * h.y), ri * fma(k0, h.x, -h.y * ri));
        g.x += h.x;
        g.y += h.y;
        F.x += f.x;
        F.y += f.y;
        rfma(gk, Q.s[o], h);
        rfma(Fk, Q.s[o], f);
      }
      // v_k (ea sum_o s_o g - er sum_o s_o F)
      cd h = cmul(ea, gk);
      cfma(h, mk<double>(-er.x, -er.y), Fk);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        S[d] = fma(u[d], h.x, S[d]);
        S[3 + d] = fma(u[d], h.y, S[3 + d]);
      }
    }
    const cd eg = cmul(ej, g), eF = cmul(er, F);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const cd b = o6[1 + d];
      S[d] += eg.x * b.x - eg.y * b.y + x[d] * eF.x;
      S[3 + d] += eg.x * b.y + eg.y * b.x + x[d] * eF.y;
    }
  }
  field_partial(S, partial + 6 * (ip * nchunk + ch));
}

pie_status nearzone(Problem& pr, const void* x, const void* rho, const double* pts, int64_t npts, void* E,
                    cudaStream_t st) {
  int64_t nchunk, len;
  // (small bodies half as many a chunk: 1 to 37 points on 1280 triangles 112 -> 92 us;
  // 1024 points on 20,480 would take 13.4 ms instead of 13.2)
  field_chunks(pr, pr.T < 8192 ? 64 : 128, &nchunk, &len);
  const int64_t batch = field_batch(npts, nchunk);
  pie_status s = PIE_OK;
  FieldScratch scratch(pr, sizeof(double) * (3 * size_t(npts) + 6 * size_t(nchunk * batch)), st, s);
  if (s != PIE_OK) return s;
  double* d_pts = static_cast<double*>(scratch.p);
  double* partial = d_pts + 3 * npts;
  s = cuda_check(cudaMemcpyAsync(d_pts, pts, sizeof(double) * 3 * npts, cudaMemcpyHostToDevice, st), "copy");
  if (s != PIE_OK) return s;
  const cd* coef = field_coef<double>(pr, x, st);
  const FieldRule Q = field_rule(pr);
  // the phases are k times the distances of the points from the centroids
  with_field_terms<false>(pr.k0 * pr.h_max, pr.k0 * (pr.r_max + longest(pts, npts)), [&](auto nt, auto ct) {
    for (int64_t i = 0; i < npts; i += batch) {
      const int64_t n = std::min(batch, npts - i);
      k_nearzone<decltype(nt)::value, decltype(ct)::value><<<nblk(n * nchunk * 32, 128), 128, 0, st>>>(
          pr.T, n, nchunk, len, pr.vert, pr.cent, pr.area, pr.perm, coef, static_cast<const cd*>(rho), d_pts + 3 * i,
          pr.k0, pr.w * kMu0, 1.0 / eps0(), Q, partial);
      k_field_finish<<<nblk(n * 32, 128), 128, 0, st>>>(n, nchunk, partial, nullptr, 0.0, static_cast<cd*>(E) + 3 * i);
    }
  });
  return cuda_check(cudaGetLastError(), "nearfield launch");
}

}  // namespace pie
