// k_quality.cu -- the mesh quality measures of the experiments section
// (Sec. 4): smallest interior angles and slivers (< 5 degrees), areas and
// their variance, the equilateral ratio by an edge-length test, the aspect
// ratio AR = longest edge / shortest altitude (median, 95th percentile,
// maximum) and the 2-degree histogram of the smallest angles.
//
// This GPU runs FP64 at about 1.6 instructions per clock and SM, against 114
// for FP32, so three double-precision atan2 and a division per triangle set
// the time of a pass that reads 215 MB on a 10.7e6-triangle mesh.  The pass
// therefore computes in double only what is summed in double (the cross
// product, the area's sum and its square's sum: eight instructions) and
// decides the rest from single precision with an error bound, evaluating the
// double formulas only for a triangle within the bound of a decision, so that
// every count and every stored AR is the one the double formulas give:
//  - the side vectors and their squared lengths as two floats each (about 46
//    bits): the equilateral test, and AR rounded to single precision;
//  - the smallest angle as a float (asin of the sine opposite the shortest
//    side): its histogram bin and the sliver test;
//  - the smallest angle and the largest AR over the mesh as per-block float
//    extremes; a second kernel evaluates the doubles of the triangles within
//    the bound of the mesh's extremes, in the blocks that hold any.
// Measured on that mesh (4096^2 Voronoi labels, h = 2): 3.74 ms for the pass
// in doubles throughout, 0.42 ms for this one.
//
// AR is stored as a float per triangle.  Percentiles are nearest-rank (the
// k-th smallest value) and exact on those floats: a radix select over the
// float's bits in three levels (bits 31-20, 19-10, 9-0), each a histogram for
// both ranks at once; one block then finds the bin that holds each rank, so
// the host waits once.  Most triangles are uncut lattice cells of one AR: each
// thread counts a run of equal bins in a register before it adds to the
// shared histogram (40 us a level with an atomic per value, 18 us with runs).
#include <algorithm>

#include "sbmt_cell.cuh"
#include "sbmt_launch.h"

namespace sbmt {

namespace {

constexpr int QHIST = 30;  // 2-degree bins of the smallest angle

// positive doubles order as their bit patterns
SBMT_DEV void atomic_min_pos(unsigned long long* a, double v) { atomicMin(a, (unsigned long long)__double_as_longlong(v)); }
SBMT_DEV void atomic_max_pos(unsigned long long* a, double v) { atomicMax(a, (unsigned long long)__double_as_longlong(v)); }

SBMT_DEV double angle_at(double ox, double oy, double ux, double uy, double vx, double vy) {
  const double d1x = ux - ox, d1y = uy - oy, d2x = vx - ox, d2y = vy - oy;
  return atan2(fabs(d1x * d2y - d1y * d2x), d1x * d2x + d1y * d2y);
}

// the smallest angle in degrees and AR by the double formulas
__device__ __noinline__ double q_angle(double2 a, double2 b, double2 c) {
  return fmin(fmin(angle_at(a.x, a.y, b.x, b.y, c.x, c.y), angle_at(b.x, b.y, c.x, c.y, a.x, a.y)),
              angle_at(c.x, c.y, a.x, a.y, b.x, b.y)) *
         57.295779513082320876798;
}
struct QLen {
  double ar;
  bool equi;
};
__device__ __noinline__ QLen q_lengths(double2 a, double2 b, double2 c) {
  const double abx = b.x - a.x, aby = b.y - a.y, bcx = c.x - b.x, bcy = c.y - b.y, cax = a.x - c.x, cay = a.y - c.y;
  const double l0 = abx * abx + aby * aby, l1 = bcx * bcx + bcy * bcy, l2 = cax * cax + cay * cay;
  const double area = 0.5 * fabs(abx * (c.y - a.y) - aby * (c.x - a.x));
  const double lmax = fmax(fmax(l0, l1), l2), lmin = fmin(fmin(l0, l1), l2);
  return QLen{lmax / (2.0 * area), (lmax - lmin) <= 1e-9 * lmax};
}

// A number as two floats, by integer instructions (a conversion from double
// runs at the FP64 rate): h the upper 24 bits of the double, l the next 29
// rounded to 24, so that |d - (h + l)| <= 2^-48 |d|.  Below 2^-60 it is taken
// as 0 and the caller leaves such sizes to the double formulas.
struct F2 {
  float h, l;
};
SBMT_DEV F2 f2_of(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned sign = hi & 0x80000000u, mag = hi & 0x7FFFFFFFu, e = mag >> 20;
  if (e < 1023 - 60 || e > 1023 + 60) return F2{0.0f, 0.0f};
  F2 r;
  r.h = __uint_as_float(sign | ((mag - (896u << 20)) << 3) | (lo >> 29));
  // the 29 lower bits in units of 2^(e - 1075)
  r.l = __uint_as_float(__float_as_uint((float)(lo & 0x1FFFFFFFu) * __uint_as_float((e - 948u) << 23)) | sign);
  return r;
}
SBMT_DEV F2 f2_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return F2{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
SBMT_DEV F2 f2_sub(F2 a, F2 b) {
  const F2 s = f2_two_sum(a.h, -b.h);
  const float l = __fadd_rn(s.l, __fsub_rn(a.l, b.l));
  const float h = __fadd_rn(s.h, l);
  return F2{h, __fsub_rn(l, __fsub_rn(h, s.h))};
}
// x^2 + y^2, within 2^-44 of it
SBMT_DEV F2 f2_len2(F2 x, F2 y) {
  const float p = __fmul_rn(x.h, x.h), q = __fmul_rn(y.h, y.h);
  const float pe = __fmaf_rn(__fadd_rn(x.h, x.h), x.l, __fmaf_rn(x.h, x.h, -p));
  const float qe = __fmaf_rn(__fadd_rn(y.h, y.h), y.l, __fmaf_rn(y.h, y.h, -q));
  const F2 s = f2_two_sum(p, q);
  const float l = __fadd_rn(s.l, __fadd_rn(pe, qe));
  const float h = __fadd_rn(s.h, l);
  return F2{h, __fsub_rn(l, __fsub_rn(h, s.h))};
}

// the float measures of a triangle whose doubled area (double) is X >= 0
struct QFast {
  float ang;  // the smallest angle in degrees, within QANG_TOL
  float ar;   // AR rounded to single precision, as the double formula gives it
  int equi;
  bool ang_ok, len_ok;  // whether ang, and ar and equi, are within the bounds
};
// The angle's sine squared is (X / lmax)(X / lmid) with X and the lengths
// within 3 2^-24 relatively, 2^-20 with the divisions; the angle (at most 60
// degrees) is off by tan / 2 of that, below 1e-6 rad, and asinf's error is
// smaller: below 1e-4 degrees.
constexpr float QANG_TOL = 2e-4f;
SBMT_DEV QFast q_fast(double ux, double uy, double vx, double vy, double X) {
  const F2 fux = f2_of(ux), fuy = f2_of(uy), fvx = f2_of(vx), fvy = f2_of(vy), x = f2_of(X);
  const F2 l0 = f2_len2(fux, fuy), l2 = f2_len2(fvx, fvy), l1 = f2_len2(f2_sub(fvx, fux), f2_sub(fvy, fuy));
  // longest and shortest by the upper floats; equal ones differ by 2^-24 at
  // most, and then either's two floats give the same answers within the bounds
  F2 lmax = l0.h > l1.h || (l0.h == l1.h && l0.l > l1.l) ? l0 : l1;
  if (l2.h > lmax.h || (l2.h == lmax.h && l2.l > lmax.l)) lmax = l2;
  F2 lmin = l0.h < l1.h || (l0.h == l1.h && l0.l < l1.l) ? l0 : l1;
  if (l2.h < lmin.h || (l2.h == lmin.h && l2.l < lmin.l)) lmin = l2;
  const float lmid = fmaxf(fminf(l0.h, l1.h), fminf(fmaxf(l0.h, l1.h), l2.h));
  QFast r;
  // sizes and shapes outside the bounds' reach: the doubles (the third side
  // is a difference of the others, good to 2^-46 of them)
  const bool safe = lmax.h < 1.0e15f && lmin.h > 1.0e-10f && lmin.h > 1.0e-5f * lmax.h && x.h > 1.0e-5f * lmax.h;
  r.ang_ok = safe;
  const float s2 = (x.h / lmax.h) * (x.h / lmid);
  r.ang = asinf(fminf(sqrtf(s2), 1.0f)) * 57.29578f;
  const float d = __fadd_rn(__fsub_rn(lmax.h, lmin.h), __fsub_rn(lmax.l, lmin.l)), t = 1e-9f * lmax.h;
  r.equi = d <= t;
  // AR = lmax / X as two floats, then rounded; a quotient within 2^-38 of
  // the middle between two floats is left to the double formula
  const float q = lmax.h / x.h;
  const float rem = __fmaf_rn(-q, x.l, __fadd_rn(__fmaf_rn(-q, x.h, lmax.h), lmax.l));
  const float ql = rem / x.h;
  r.ar = __fadd_rn(q, ql);
  const float e = __fadd_rn(__fsub_rn(q, r.ar), ql);
  const unsigned bits = __float_as_uint(r.ar);
  const float half = __uint_as_float((bits & 0x7F800000u) - (24u << 23));
  r.len_ok = safe && fabsf(d - t) > 1e-11f * lmax.h && (bits & 0x7FFFFFu) != 0u &&
             fabsf(fabsf(e) - half) > 3.7e-12f * r.ar;
  return r;
}

// mm: [1] min doubled area (double bits); cnt: [0] slivers, [1] equilateral;
// part: per block (sum of doubled areas, of their squares); ext: per block
// the smallest angle and the largest AR as floats; h0: the select's first level.
// The triangles that need a double formula are queued in shared memory and
// taken by the whole block when 256 are there: a boundary along a pixel
// column cuts lattice corners into 30-60-90 triangles, on the edge of a bin,
// and a few lanes of most boundary warps in the formulas cost as much as all
// 32 (1.34 ms for the pass, against 0.42 ms).
constexpr int QL0 = 4096;  // bins of the first level: bits 31-20
constexpr int QT = 256;    // threads per block
__global__ void __launch_bounds__(QT) k_quality(const double* xy, const int* tri, u64 T, float* ar_out,
                                                unsigned long long* mm, unsigned long long* cnt, double* part,
                                                u32* hist, float2* ext, u32* h0) {
  __shared__ u32 s_hist[QHIST];
  __shared__ u32 s_l0[QL0];
  __shared__ double s_red[2][8];
  __shared__ float s_ext[2][8];
  __shared__ unsigned long long s_cnt[2];
  __shared__ u32 s_queue[2 * QT];  // triangle << 1 | lengths too (triangles stay below 2^31)
  __shared__ u32 s_nq;
  if (threadIdx.x < QHIST) s_hist[threadIdx.x] = 0;
  if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0;
  if (threadIdx.x == 0) s_nq = 0;
  for (int k = threadIdx.x; k < QL0; k += blockDim.x) s_l0[k] = 0;
  __syncthreads();
  unsigned long long amin = 0x7FF0000000000000ull;
  double sa = 0.0, sa2 = 0.0;
  float angmin = 1e30f, armax = 0.0f;
  u32 slv = 0, equ = 0, top = 0;  // top: triangles of the histogram's last bin
  u32 run_bin = 0, run = 0;
  const double2* pt = reinterpret_cast<const double2*>(xy);
  auto queued = [&](u32 e) {
    const u64 t = e >> 1;
    const double2 a = pt[tri[3 * t]], b = pt[tri[3 * t + 1]], c = pt[tri[3 * t + 2]];
    const double ang = q_angle(a, b, c);
    atomicAdd(&s_hist[min((int)(ang * 0.5), QHIST - 1)], 1u);
    slv += ang < 5.0 ? 1u : 0u;
    angmin = fminf(angmin, (float)ang);
    if (e & 1u) {
      const QLen l = q_lengths(a, b, c);
      const float ar = (float)l.ar;
      ar_out[t] = ar, armax = fmaxf(armax, ar), equ += l.equi ? 1u : 0u;
      atomicAdd(&s_l0[__float_as_uint(ar) >> 20], 1u);
    }
  };
  for (u64 t0 = (u64)blockIdx.x * QT; t0 < T; t0 += (u64)gridDim.x * QT) {
    const u64 t = t0 + threadIdx.x;
    if (t < T) {
      const double2 a = pt[tri[3 * t]], b = pt[tri[3 * t + 1]], c = pt[tri[3 * t + 2]];
      const double abx = b.x - a.x, aby = b.y - a.y, acx = c.x - a.x, acy = c.y - a.y;
      const double X = fabs(abx * acy - aby * acx);
      amin = min(amin, (unsigned long long)__double_as_longlong(X));
      sa += X, sa2 += X * X;
      const QFast f = q_fast(abx, aby, acx, acy, X);
      if (f.len_ok) {
        ar_out[t] = f.ar;
        armax = fmaxf(armax, f.ar);
        equ += (u32)f.equi;
        const u32 bin0 = __float_as_uint(f.ar) >> 20;
        if (bin0 != run_bin) {
          if (run) atomicAdd(&s_l0[run_bin], run);
          run_bin = bin0, run = 0;
        }
        ++run;
      }
      // the bin floor(angle / 2) and angle < 5, unless the float angle is
      // within its bound of an edge
      const float h = f.ang * 0.5f;
      const int bin = (int)h;
      const float fr = h - (float)bin;
      const bool last = h > (float)(QHIST - 1) + QANG_TOL;
      if (!f.len_ok || !f.ang_ok ||
          !(last || (fr > QANG_TOL && fr < 1.0f - QANG_TOL && fabsf(f.ang - 5.0f) > QANG_TOL))) {
        s_queue[atomicAdd(&s_nq, 1u)] = (u32)(t << 1) | (f.len_ok ? 0u : 1u);
      } else {
        if (last) ++top;
        else atomicAdd(&s_hist[bin], 1u);
        slv += f.ang < 5.0f ? 1u : 0u;
        angmin = fminf(angmin, f.ang);
      }
    }
    __syncthreads();
    const u32 nq = s_nq;
    __syncthreads();
    if (nq >= QT) {
      queued(s_queue[nq - QT + threadIdx.x]);
      __syncthreads();
      if (threadIdx.x == 0) s_nq = nq - QT;
      __syncthreads();
    }
  }
  if (threadIdx.x < s_nq) queued(s_queue[threadIdx.x]);
  if (run) atomicAdd(&s_l0[run_bin], run);
  // block reductions
  for (int o = 16; o > 0; o >>= 1) {
    angmin = fminf(angmin, __shfl_xor_sync(0xffffffffu, angmin, o));
    armax = fmaxf(armax, __shfl_xor_sync(0xffffffffu, armax, o));
    amin = min(amin, __shfl_xor_sync(0xffffffffu, amin, o));
    sa += __shfl_xor_sync(0xffffffffu, sa, o);
    sa2 += __shfl_xor_sync(0xffffffffu, sa2, o);
  }
  slv = __reduce_add_sync(0xffffffffu, slv), equ = __reduce_add_sync(0xffffffffu, equ);
  top = __reduce_add_sync(0xffffffffu, top);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) {
    if (amin < 0x7FF0000000000000ull) atomicMin(&mm[1], amin);
    s_red[0][w] = sa, s_red[1][w] = sa2;
    s_ext[0][w] = angmin, s_ext[1][w] = armax;
    atomicAdd(&s_cnt[0], (unsigned long long)slv);
    atomicAdd(&s_cnt[1], (unsigned long long)equ);
    if (top) atomicAdd(&s_hist[QHIST - 1], top);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double x = 0.0, y = 0.0;
    float lo = 1e30f, hi = 0.0f;
    for (int k = 0; k < 8; ++k) {
      x += s_red[0][k], y += s_red[1][k];
      lo = fminf(lo, s_ext[0][k]), hi = fmaxf(hi, s_ext[1][k]);
    }
    part[2 * blockIdx.x] = x, part[2 * blockIdx.x + 1] = y;
    ext[blockIdx.x] = make_float2(lo, hi);
    atomicAdd(&cnt[0], s_cnt[0]);
    atomicAdd(&cnt[1], s_cnt[1]);
  }
  if (threadIdx.x < QHIST && s_hist[threadIdx.x]) atomicAdd(&hist[threadIdx.x], s_hist[threadIdx.x]);
  for (int k = threadIdx.x; k < QL0; k += blockDim.x)
    if (s_l0[k]) atomicAdd(&h0[k], s_l0[k]);
}

// mm: [0] the smallest angle, [2] the largest AR (double bits).  Launched with
// k_quality's grid (at most QEXT_BLOCKS blocks), in its turns of QT triangles.
// The turns of those blocks of k_quality whose float extremes are within the
// bounds of the mesh's are shared out over this grid's blocks, and the double
// formulas evaluated for their triangles within the bounds.
constexpr int QEXT_BLOCKS = 152 * 8;
__global__ void __launch_bounds__(QT) k_quality_ext(const double* xy, const int* tri, u64 T, const float* ar,
                                                    const float2* ext, unsigned long long* mm) {
  __shared__ float s_lo[8], s_hi[8];
  __shared__ unsigned short s_near[QEXT_BLOCKS];
  __shared__ u32 s_w[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float lo = 1e30f, hi = 0.0f;
  for (u32 k = threadIdx.x; k < gridDim.x; k += QT) lo = fminf(lo, ext[k].x), hi = fmaxf(hi, ext[k].y);
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) s_lo[w] = lo, s_hi[w] = hi;
  __syncthreads();
  for (int k = 0; k < 8; ++k) lo = fminf(lo, s_lo[k]), hi = fmaxf(hi, s_hi[k]);
  const float alim = lo + 2.0f * QANG_TOL, rlim = hi * (1.0f - 2.4e-7f);
  // the blocks within the bounds, in order (the same list in every block)
  u32 n = 0;
  for (u32 k0 = 0; k0 < gridDim.x; k0 += QT) {
    const u32 k = k0 + threadIdx.x;
    const bool near = k < gridDim.x && (ext[k].x <= alim || ext[k].y >= rlim);
    const unsigned m = __ballot_sync(0xffffffffu, near);
    if (lane == 0) s_w[w] = (u32)__popc(m);
    __syncthreads();
    u32 before = n;
    for (int q = 0; q < 8; ++q) {
      if (q < w) before += s_w[q];
      n += s_w[q];
    }
    if (near) s_near[before + __popc(m & ((1u << lane) - 1u))] = (unsigned short)k;
    __syncthreads();
  }
  const u64 span = (u64)gridDim.x * QT, turns = (T + span - 1) / span;
  double angmin = 1e300, armax = 0.0;
  for (u64 item = blockIdx.x; item < n * turns; item += gridDim.x) {
    const u32 k = s_near[item / turns];
    const u64 t = (item % turns) * span + (u64)k * QT + threadIdx.x;
    if (t >= T) continue;
    const double2* pt = reinterpret_cast<const double2*>(xy);
    const double2 a = pt[tri[3 * t]], b = pt[tri[3 * t + 1]], c = pt[tri[3 * t + 2]];
    if (ar[t] >= rlim) armax = fmax(armax, q_lengths(a, b, c).ar);
    const double abx = b.x - a.x, aby = b.y - a.y, acx = c.x - a.x, acy = c.y - a.y;
    const QFast f = q_fast(abx, aby, acx, acy, fabs(abx * acy - aby * acx));
    if (!f.ang_ok || f.ang <= alim) angmin = fmin(angmin, q_angle(a, b, c));
  }
  for (int o = 16; o > 0; o >>= 1) {
    angmin = fmin(angmin, __shfl_xor_sync(0xffffffffu, angmin, o));
    armax = fmax(armax, __shfl_xor_sync(0xffffffffu, armax, o));
  }
  if (lane == 0) {
    if (angmin < 1e300) atomic_min_pos(&mm[0], angmin);
    if (armax > 0.0) atomic_max_pos(&mm[2], armax);
  }
}

// the radix select's state: per rank the bits above the current level, and
// the rank among the values that have them
struct QSel {
  u32 pre[2];
  u64 rank[2];
};

// one level of the radix select: histogram of the bits [lo, lo + width) of
// the values whose bits above lo + width equal prefix[r], for the two ranks
// (once when the prefixes are equal: the pick reads it for both)
__global__ void __launch_bounds__(256) k_select_hist(const float* v, u64 T, int lo, int width, const QSel* sel,
                                                     u32* h) {
  extern __shared__ u32 s_h[];  // 2 << width counters
  const int nb = 1 << width;
  for (int k = threadIdx.x; k < 2 * nb; k += blockDim.x) s_h[k] = 0;
  const u32 p0 = sel->pre[0], p1 = sel->pre[1];
  __syncthreads();
  const int above = lo + width;
  u32 run_bin = 0, run = 0;
  auto take = [&](u32 bits) {
    const u32 top = bits >> above;
    if (top != p0 && top != p1) return;
    const u32 bin = ((bits >> lo) & (u32)(nb - 1)) + (top == p0 ? 0u : (u32)nb);
    if (bin != run_bin) {
      if (run) atomicAdd(&s_h[run_bin], run);
      run_bin = bin, run = 0;
    }
    ++run;
  };
  const u64 T4 = T >> 2;  // v is 256-byte aligned
  const uint4* v4 = reinterpret_cast<const uint4*>(v);
  for (u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x; t < T4; t += (u64)gridDim.x * blockDim.x) {
    const uint4 x = v4[t];
    take(x.x), take(x.y), take(x.z), take(x.w);
  }
  if (blockIdx.x == 0 && threadIdx.x < (u32)(T & 3)) take(__float_as_uint(v[4 * T4 + threadIdx.x]));
  if (run) atomicAdd(&s_h[run_bin], run);
  __syncthreads();
  for (int k = threadIdx.x; k < 2 * nb; k += blockDim.x)
    if (s_h[k]) atomicAdd(&h[k], s_h[k]);
}

// the bin that holds each rank (one block): both ranks read the first nb
// counters when `shared` or their prefixes are equal, else the second its own
__global__ void __launch_bounds__(1024) k_select_pick(const u32* h, int width, int shared, QSel* sel) {
  __shared__ u32 s_sum[32];
  __shared__ u32 s_bin[2];
  __shared__ u64 s_cum[2];
  const int nb = 1 << width, per = nb / 1024, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const bool one = shared || sel->pre[0] == sel->pre[1];
  for (int r = 0; r < 2; ++r) {
    const u32* hr = h + (r && !one ? nb : 0);
    u32 own = 0;
    for (int k = 0; k < per; ++k) own += hr[per * threadIdx.x + k];
    u32 inc = own;
    for (int o = 1; o < 32; o <<= 1) {
      const u32 y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) s_sum[w] = inc;
    if (threadIdx.x == 0) s_bin[r] = (u32)nb - 1u, s_cum[r] = 0;
    __syncthreads();
    u64 cum = inc - own;
    for (int k = 0; k < w; ++k) cum += s_sum[k];
    const u64 rank = sel->rank[r];
    // the first bin whose running count reaches the rank
    for (int k = 0; k < per; ++k) {
      const u32 c = hr[per * threadIdx.x + k];
      if (cum < rank && cum + c >= rank) s_bin[r] = per * threadIdx.x + (u32)k, s_cum[r] = cum;
      cum += c;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int r = 0; r < 2; ++r) sel->rank[r] -= s_cum[r], sel->pre[r] = (sel->pre[r] << width) | s_bin[r];
}

}  // namespace

size_t quality_select_words() { return 8 + QL0 + 2 * 2048; }

int launch_quality(const double* xy, const int* tri, u64 T, float* ar, unsigned long long* mm,
                   unsigned long long* cnt, double* part, int nblocks, u32* hist, float2* ext, u32* select,
                   cudaStream_t st) {
  QSel* sel = reinterpret_cast<QSel*>(select);
  u32* h0 = select + 8;
  u32* h1 = h0 + QL0;  // 2 x 1024 counters per level
  u32* h2 = h1 + 2048;
  k_quality<<<nblocks, 256, 0, st>>>(xy, tri, T, ar, mm, cnt, part, hist, ext, h0);
  k_quality_ext<<<nblocks, 256, 0, st>>>(xy, tri, T, ar, ext, mm);
  k_select_pick<<<1, 1024, 0, st>>>(h0, 12, 1, sel);
  k_select_hist<<<152 * 4, 256, 8192, st>>>(ar, T, 10, 10, sel, h1);
  k_select_pick<<<1, 1024, 0, st>>>(h1, 10, 0, sel);
  k_select_hist<<<152 * 4, 256, 8192, st>>>(ar, T, 0, 10, sel, h2);
  k_select_pick<<<1, 1024, 0, st>>>(h2, 10, 0, sel);
  return 7;
}

}  // namespace sbmt
