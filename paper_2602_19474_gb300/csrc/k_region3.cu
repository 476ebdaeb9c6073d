// k_region3.cu -- Region III of Alg. 3's schedule (the corollary on
// pipelined parallel scheduling: Regions I and II, a barrier, then Region
// III): Alg. 2, the template retriangulation, run on the preprocessed mesh T,
// one cell at a time from its local intersection class (the corollary on
// lookup-driven parallel retriangulation: patches out of place, then one
// deterministic stitching by scan offsets).
//
// T's vertices are doubles (Steps 1-2 move them off the lattice), so every
// quantity is a double computed by one fixed formula, each operation rounded
// once (explicit round-to-nearest intrinsics: no contraction into FMAs).
// Degenerate incidences are exact: a pixel line is k - 1/2, and a vertex
// snapped onto a pixel corner sits on it exactly.
//
//  - An event of a mesh edge e is a point of the open edge where the
//    boundary meets it: the crossing of a boundary pixel edge, or a pixel
//    corner on e with a boundary pixel edge not collinear with e (Alg. 1's
//    endpoint on the edge; a run of boundary along e is embedded by e
//    itself: Alg. 1's overlap).  An end of e on the boundary (Alg. 1's
//    vertex on the segment) is not an event of e.  An edge's events are
//    computed from its lower-id end P: on the horizontal pixel line y0 the
//    crossing is x = P.x + ((y0 - P.y)(Q.x - P.x)) / (Q.y - P.y), on a
//    vertical line likewise; the two cells beside the edge see the same
//    points.
//  - The boundary vertices inside a cell are the PSLG vertices strictly
//    inside its chord on their horizontal pixel line.
//  - The boundary pieces of a cell are the boundary runs of each pixel line
//    strictly between the cell's extreme corners, cut at the cell's nodes on
//    the line.
//  - Tier-T (the table's regime, as on the lattice): no piece ends at a
//    corner of the cell and every event ends one piece; no inside vertex
//    and one or two chords, or one inside vertex every piece ends at.  The
//    patch is the App. G template of the cell's key.  Every other cut cell
//    (Tier-G) takes the greedy rule: vertex pairs in order of squared length
//    rounded to single precision (ties by local index pair), kept when the
//    open segment holds no vertex and crosses no kept edge.
//
// Kernels: k_r3_screen
// (every cell: a cell whose pixel box carries one label is uncut and takes
// that label, with no double-precision work; the others are listed);
// k_r3_link (the listed cells around each vertex); k_r3_count (the listed cells: triangles, events on the edges each owns --
// the smaller of the two cells beside an edge -- and inside vertices; a
// record of what it found for each cut cell); a scan; k_r3_emit_uncut;
// k_r3_cells (the cut cells of at most 32 nodes: Tier-T patches and the
// greedy rule, a group of lanes a cell, from the records); k_r3_tierg (one
// warp per larger cell).
//
// One thread per cut cell rebuilt the cell's graph in double formulas, twice
// for a Tier-G cell, with 3 of 32 lanes active: 1.20 + 0.71 ms for the 1.9e5 cut
// cells of a 4096^2 label image at h = 2.  With the records, and one event,
// line, candidate or triangle per lane, 0.40 ms (0.38 ms for the count
// that writes them).
#include "sbmt_cell.cuh"
#include "sbmt_greedy.cuh"
#include "sbmt_keys.cuh"
#include "sbmt_launch.h"

namespace sbmt {

namespace {

constexpr int R3_MAXE = 16;  // events on one edge
constexpr int R3_MAXI = 16;  // boundary vertices inside one cell
constexpr int R3_MAXN = 48;  // nodes of one cell: 3 corners, events, inside vertices
constexpr int R3_MAXP = 48;  // boundary pieces of one cell
constexpr int R3_OUTSIDE = 0x10000;

SBMT_DEV double dad(double a, double b) { return __dadd_rn(a, b); }
SBMT_DEV double dsb(double a, double b) { return __dsub_rn(a, b); }
SBMT_DEV double dml(double a, double b) { return __dmul_rn(a, b); }
SBMT_DEV double ddv(double a, double b) { return __ddiv_rn(a, b); }

SBMT_DEV int r3_px(const R3Args& a, i64 x, i64 y) {
  if (x < 0 || y < 0 || x >= a.W || y >= a.H) return R3_OUTSIDE;
  const unsigned char* row = a.img + y * a.pitch;
  return a.dtype == 1 ? (int)row[x] : (int)reinterpret_cast<const unsigned short*>(row)[x];
}
// horizontal pixel edge (m, k): from corner (m, k) to (m + 1, k), between
// pixels (m, k - 1) and (m, k); vertical edge (m, k): from corner (m, k) to
// (m, k + 1), between pixels (m - 1, k) and (m, k)
SBMT_DEV bool r3_hb(const R3Args& a, i64 m, i64 k) { return r3_px(a, m, k - 1) != r3_px(a, m, k); }
SBMT_DEV bool r3_vb(const R3Args& a, i64 m, i64 k) { return r3_px(a, m - 1, k) != r3_px(a, m, k); }
enum { R3E = 1, R3N = 2, R3W = 4, R3S = 8 };
SBMT_DEV int r3_cmask(const R3Args& a, i64 cx, i64 cy) {
  return (r3_hb(a, cx, cy) ? R3E : 0) | (r3_vb(a, cx, cy) ? R3N : 0) | (r3_hb(a, cx - 1, cy) ? R3W : 0) |
         (r3_vb(a, cx, cy - 1) ? R3S : 0);
}
SBMT_DEV bool r3_is_vertex(int m) { return m != 0 && m != (R3E | R3W) && m != (R3N | R3S); }

// position t on a pixel line: the pixel edge j holding it (edge j spans
// [j - 1/2, j + 1/2]), or the corner c with t = c - 1/2 (returns true)
SBMT_DEV bool r3_at_corner(double t, i64* idx) {
  const double fl = floor(t), fr = dsb(t, fl);
  if (fr == 0.5) {
    *idx = (i64)fl + 1;
    return true;
  }
  *idx = fr < 0.5 ? (i64)fl : (i64)fl + 1;
  return false;
}
SBMT_DEV double r3_hx(double2 P, double2 Q, double y0) {
  return dad(P.x, ddv(dml(dsb(y0, P.y), dsb(Q.x, P.x)), dsb(Q.y, P.y)));
}
SBMT_DEV double r3_vy(double2 P, double2 Q, double x0) {
  return dad(P.y, ddv(dml(dsb(x0, P.x), dsb(Q.y, P.y)), dsb(Q.x, P.x)));
}
SBMT_DEV double r3_orient(double2 p, double2 q, double2 r) {
  return dsb(dml(dsb(q.x, p.x), dsb(r.y, p.y)), dml(dsb(q.y, p.y), dsb(r.x, p.x)));
}
SBMT_DEV int r3_sgn(double o) { return o > 0.0 ? 1 : (o < 0.0 ? -1 : 0); }
SBMT_DEV i64 r3_lo(double v) { return (i64)floor(dad(v, 0.5)); }
SBMT_DEV i64 r3_hi(double v) { return (i64)ceil(dad(v, 0.5)); }

struct R3Ev {
  double x, y, s;
  int kind;  // 0 on horizontal line k, 1 on vertical line m, 2 at pixel corner (m, k)
  int m, k;
};

// the boundary pixel edges at corner (cx, cy) not collinear with an edge
// that is horizontal (hz) or vertical (vt)
SBMT_DEV bool r3_corner_event(const R3Args& a, i64 cx, i64 cy, bool hz, bool vt) {
  int m = r3_cmask(a, cx, cy);
  if (hz) m &= ~(R3E | R3W);
  if (vt) m &= ~(R3N | R3S);
  return m != 0;
}

// ---------------------------------------------------------------------------
// single-precision filters for the positions on pixel lines.  The double
// formulas above are the definition (the oracle's arithmetic); a float
// computation decides where a proven bound allows, the double formula
// where it does not, so that every decision is the double formula's.
// ---------------------------------------------------------------------------
// This GPU converts from double to float, from 64-bit integers to double
// from float to 64-bit integers and from 64-bit integers to float on its FP64
// pipe (a few per clock per SM, against about a hundred for float arithmetic
// and for 32-bit conversions), so the filters take doubles apart with integer
// instructions, and 64-bit integers to float by their upper 32 bits.
//
// v (|v| <= 2^24) as a 64-bit fixed-point number with 36 fraction bits:
// floor(v 2^36), exactly, and whether v 2^36 was not an integer (*inexact)
SBMT_DEV i64 r3_fix36(double v, bool* inexact) {
  const u64 b = (u64)__double_as_longlong(v);
  const bool neg = (b >> 63) != 0;
  const int e = (int)((b >> 52) & 0x7FF);
  const u64 frac = b & 0xFFFFFFFFFFFFFull;
  i64 f;
  bool lost;
  if (e == 0) {
    lost = frac != 0;  // zero, or a denormal (below one unit)
    f = (neg && lost) ? 1 : 0;
  } else {
    const i64 m = (i64)(frac | (1ull << 52));
    const int sh = e - 1039;  // v = m 2^(e - 1075), so v 2^36 = m 2^(e - 1039); sh <= 8 up to 2^24
    if (sh >= 0) {
      f = m << sh, lost = false;
    } else if (sh > -63) {
      lost = (m & ((1ll << -sh) - 1)) != 0;
      f = (m >> -sh) + ((neg && lost) ? 1 : 0);  // magnitude rounded towards the floor
    } else {
      f = neg ? 1 : 0, lost = true;
    }
  }
  *inexact = lost;
  return neg ? -f : f;
}
// the float of an integer |n| < 2^22, exactly: n in the mantissa of 1.5 2^23 + n.
// (Of larger ones it is wrong by up to millions: used only where the pixel index
// has that range, or an edge long enough to give a larger n has a crossing
// tolerance above 1/2, which leaves the crossing to the double formula.)
SBMT_DEV float r3_i2f(int n) { return __fsub_rn(__int_as_float(0x4B400000 + n), 12582912.0f); }
// the nearest integer to a float |z| < 2^22, and the floor
SBMT_DEV int r3_fint(float z) { return __float_as_int(__fadd_rn(z, 12582912.0f)) - 0x4B400000; }
SBMT_DEV int r3_ffloor(float z) {
  const int n = r3_fint(z);
  return r3_i2f(n) > z ? n - 1 : n;
}
// A coordinate v as an integer i = floor(v) and f: the remainder v - i (in
// [0, 1), exact in double) truncated to a multiple of 2^-23, so that
// v - i - 2^-23 - 2^-36 < f <= v - i.
struct R3Split {
  i64 i, fx;
  float f;
  bool inexact;
};
SBMT_DEV R3Split r3_split(double v) {
  R3Split s;
  s.fx = r3_fix36(v, &s.inexact);
  s.i = s.fx >> 36;
  const int n23 = (int)((s.fx & ((1ll << 36) - 1)) >> 13);
  s.f = __fmul_rn(__fsub_rn(__int_as_float(0x4B000000 | n23), 8388608.0f), 1.1920928955078125e-7f);  // n23 2^-23
  return s;
}
struct R3Corner {  // what the line tests need of it
  i64 fx;
  bool inexact;
};
// v against the pixel line k - 1/2, exactly, from fx = floor(v 2^36):
// below iff fx < (k - 1/2) 2^36; above iff fx is greater, or equal with
// bits dropped
SBMT_DEV i64 r3_line36(i64 k) { return (k << 36) - (1ll << 35); }
template <class V>
SBMT_DEV bool r3_lt(const V& v, i64 k) { return v.fx < r3_line36(k); }
template <class V>
SBMT_DEV bool r3_gt(const V& v, i64 k) {
  const i64 t = r3_line36(k);
  return v.fx > t || (v.fx == t && v.inexact);
}
// the float of a coordinate difference from the fixed-point values (within
// 2^-35 + (2^-24 + 2^-31) |d| of the double difference's real value)
SBMT_DEV float r3_fdiff(const R3Split& q, const R3Split& p) {
  return i64_float(q.fx - p.fx, -36);
}

// The crossing of the edge from P (its lower-id end) with the line at
// coordinate c0 = k - 1/2 across it, as w = (position along the line) - B,
// B the integer part of P's coordinate along the line.  With A = c0 - P (in
// the crossing direction: k - 1/2 - Pi - Pr, the integer part exact) and
// s = the edge's slope in float, w = Pr + A s.  The remainders are within
// 2^-22 of their values, the differences within 2^-35 + 2^-23 |d|, the
// slope within 5 2^-24 |s| relatively, so the float w is within
// 2^-24 (8 + 8|s| + 7 D + |w|) of the real w of the double inputs (D: the
// edge's larger extent; |A| is below the extent across the line, |A s|
// below the extent along it), and the double formula within
// 2^-53 (|position| + 3 D) of that real value.  Where the line, or a pixel
// corner compared with w, is 2^23 or more from P (cells reaching millions of
// pixels outside the image), its distance in float (r3_half) is within 2^-23 of
// it: 2 more of D and of |w|.  T (below) is above the sum at every coordinate up
// to 2^24.
SBMT_DEV float r3_half(i64 n) { return __fsub_rn((float)(int)n, 0.5f); }  // n - 1/2, |n| <= 2^24 + 2^15
SBMT_DEV float r3_cross_tol(float D, float s, float w) {
  return 6.0e-7f * (D + fabsf(s) + 2.0f * fabsf(w) + 3.0f) + 1.5e-8f;
}
// the double formula's crossing with the line c0 (vert: x = c0, giving y):
// its pixel edge or corner index in *j, *corner set
__device__ __noinline__ void r3_cross_exact(double2 P, double2 Q, double c0, bool vert, i64* j, bool* corner) {
  *corner = r3_at_corner(vert ? r3_vy(P, Q, c0) : r3_hx(P, Q, c0), j);
}
// The same in integers for an edge between two pixel corners (snapped vertices:
// the usual reason for a crossing at a corner).  The formula's differences are
// then integers of at most 2^15, its product exact, its quotient exact where it is an
// integer and otherwise at least 2^-15 from one, far above its rounding.
// a, b: across the line and along it, p the edge's first end, q the other.
SBMT_DEV bool r3_corner_ends(const R3Split& px, const R3Split& py, const R3Split& qx, const R3Split& qy, float D) {
  constexpr i64 M = (1ll << 36) - 1, HALF = 1ll << 35;
  return ((px.fx ^ HALF) & M) == 0 && ((py.fx ^ HALF) & M) == 0 && ((qx.fx ^ HALF) & M) == 0 &&
         ((qy.fx ^ HALF) & M) == 0 && !(px.inexact || py.inexact || qx.inexact || qy.inexact) && D <= 32768.0f;
}
SBMT_DEV void r3_cross_corners(const R3Split& pa, const R3Split& pb, const R3Split& qa, const R3Split& qb, int line,
                               i64* j, bool* corner) {
  int num = (line - (int)(pa.i + 1)) * (int)(qb.i - pb.i), den = (int)(qa.i - pa.i);
  if (den < 0) num = -num, den = -den;
  int q = num / den, r = num - q * den;
  if (r < 0) --q;
  *corner = r == 0;
  *j = pb.i + 1 + q;
}

// the pixel lines strictly between two coordinates (closed: or through one of
// them), within [0, most]: the first, and their number
template <class V>
SBMT_DEV int r3_lines(const V& a, const V& b, int most, int* first, bool closed = false) {
  const bool sw = b.fx < a.fx || (b.fx == a.fx && a.inexact);  // the lower of the two first
  const i64 lo = sw ? b.fx : a.fx, hi = sw ? a.fx : b.fx;
  const bool hx = sw ? a.inexact : b.inexact;
  constexpr i64 HALF = 1ll << 35;
  const bool lx = sw ? b.inexact : a.inexact;
  const i64 k0 = max(((lo + HALF - (closed && !lx ? 1 : 0)) >> 36) + 1, (i64)0);
  const i64 k1 = min((hi + HALF - (hx || closed ? 0 : 1)) >> 36, (i64)most);
  *first = (int)k0;
  return k1 < k0 ? 0 : (int)(k1 - k0 + 1);
}
// an event as the count pass records it: pixel indices m, k (at most 32768),
// the cell's edge and the kind; an inside vertex has kind 3, edge 3
SBMT_DEV u64 r3_entry(int edge, int kind, int m, int k) {
  return (u64)(u32)m | (u64)(u32)k << 16 | (u64)(edge << 2 | kind) << 32;
}

SBMT_DEV bool r3_same(double a, double b) {  // a == b without an FP64 compare (finite numbers)
  const i64 p = __double_as_longlong(a), q = __double_as_longlong(b);
  return p == q || ((p | q) << 1) == 0;
}


// the cell's two chord ends on a pixel line (vert: the vertical line x = c0,
// else the horizontal y = c0): (position along the line, source = corner 0..2
// or 3 + edge); the number of ends found (2 for a proper cell)
SBMT_DEV int r3_chord(const double2* K, const int* id, bool vert, double c0, double* pos, int* src) {
  int n = 0;
  for (int c = 0; c < 3; ++c)
    if ((vert ? K[c].x : K[c].y) == c0) {
      if (n == 2) return 3;
      pos[n] = vert ? K[c].y : K[c].x, src[n++] = c;
    }
  for (int j = 0; j < 3; ++j) {
    const int u = j, w = j == 2 ? 0 : j + 1;
    const double2 P = id[u] < id[w] ? K[u] : K[w], Q = id[u] < id[w] ? K[w] : K[u];
    const double pa = vert ? P.x : P.y, pb = vert ? Q.x : Q.y;
    if (!((pa < c0 && c0 < pb) || (pb < c0 && c0 < pa))) continue;
    if (n == 2) return 3;
    pos[n] = vert ? r3_vy(P, Q, c0) : r3_hx(P, Q, c0), src[n++] = 3 + j;
  }
  if (n == 2 && pos[1] < pos[0]) {
    const double t = pos[0];
    pos[0] = pos[1], pos[1] = t;
    const int s = src[0];
    src[0] = src[1], src[1] = s;
  }
  return n;
}

struct R3Cell {
  double2 K[3];
  int id[3];
  double ylo, yhi, xlo, xhi;
};
// the corners alone (the bounding box left unset)
SBMT_DEV R3Cell r3_load_k(const R3Args& a, u32 c) {
  R3Cell C;
  const int* t = a.ttri + 3 * (u64)c;
  for (int q = 0; q < 3; ++q) C.id[q] = t[q], C.K[q] = reinterpret_cast<const double2*>(a.txy)[C.id[q]];
  return C;
}
SBMT_DEV R3Cell r3_load(const R3Args& a, u32 c) {
  R3Cell C;
  const int* t = a.ttri + 3 * (u64)c;
  for (int q = 0; q < 3; ++q) C.id[q] = t[q], C.K[q] = reinterpret_cast<const double2*>(a.txy)[C.id[q]];
  C.ylo = fmin(fmin(C.K[0].y, C.K[1].y), C.K[2].y), C.yhi = fmax(fmax(C.K[0].y, C.K[1].y), C.K[2].y);
  C.xlo = fmin(fmin(C.K[0].x, C.K[1].x), C.K[2].x), C.xhi = fmax(fmax(C.K[0].x, C.K[1].x), C.K[2].x);
  return C;
}

// the label of the pixels x0 .. x0 + w, y0 .. y0 + h (w, h below 4) when they
// carry one, else -1
template <typename T>
SBMT_DEV int r3_box(const R3Args& a, int x0, int y0, int w, int h) {
  const unsigned char* row = a.img + (i64)y0 * a.pitch;
  const T l0 = reinterpret_cast<const T*>(row)[x0];
  T v[4][4];
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int x = 0; x < 4; ++x)
      v[y][x] = y <= h && x <= w ? reinterpret_cast<const T*>(row + y * a.pitch)[x0 + x] : l0;
  bool one = true;
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int x = 0; x < 4; ++x) one &= v[y][x] == l0;
  return one ? (int)l0 : -1;
}

// one label over the pixels touching the cell's bounding box: no boundary
// pixel edge meets the cell, and every pixel the cell covers has that label
// (returned, OUTSIDE as 0xFFFF), or -1.  The box is the double-precision one
// grown by 1e-6 px, or any box holding it: a larger box finds a cell of one
// label at most where the exact one does, and a cell it misses becomes a
// candidate with no event and no inside vertex, emitted as it is with the
// label of the pixel holding its centroid, a pixel of the exact box -- the
// same output.  Here the box comes from the corners' fixed-point values
// (within 2^-36 of the doubles), its ends moved outwards by 2^-36 and
// 2e-6 px, all in integer arithmetic.
SBMT_DEV int r3_uniform(const R3Args& a, const i64* X, const i64* Y) {
  constexpr i64 HALF = 1ll << 35, GROW = 137439 + 1;  // 1/2 and 2e-6 (rounded up) plus 2^-36, in 2^-36 units
  const i64 xlo = min(min(X[0], X[1]), X[2]), xhi = max(max(X[0], X[1]), X[2]);
  const i64 ylo = min(min(Y[0], Y[1]), Y[2]), yhi = max(max(Y[0], Y[1]), Y[2]);
  // ceil(lo - 1/2 - grow) and floor(hi + 1/2 + grow) in pixels
  const i64 x0 = -((-(xlo - HALF - GROW)) >> 36), x1 = (xhi + HALF + GROW) >> 36;
  const i64 y0 = -((-(ylo - HALF - GROW)) >> 36), y1 = (yhi + HALF + GROW) >> 36;
  if (x0 >= 0 && y0 >= 0 && x1 < a.W && y1 < a.H && x1 - x0 < 4 && y1 - y0 < 4) {
    // at most 4 x 4 pixels inside the image: every load issued at once
    return a.dtype == 1 ? r3_box<unsigned char>(a, (int)x0, (int)y0, (int)(x1 - x0), (int)(y1 - y0))
                        : r3_box<unsigned short>(a, (int)x0, (int)y0, (int)(x1 - x0), (int)(y1 - y0));
  }
  const int l0 = r3_px(a, x0, y0);
  // every pixel beyond the image reads OUTSIDE, like those of the one-pixel
  // margin kept: the scan stops there without changing its answer
  for (i64 y = max(y0, (i64)-1), ye = min(y1, (i64)a.H); y <= ye; ++y)
    for (i64 x = max(x0, (i64)-1), xe = min(x1, (i64)a.W); x <= xe; ++x)
      if (r3_px(a, x, y) != l0) return -1;
  return l0 == R3_OUTSIDE ? 0xFFFF : l0;
}

// counter-clockwise (a positive orientation of the doubles), with a
// single-precision filter: the coordinate differences from the fixed-point
// values are within 2^-35 + 2^-24 |d| of the doubles' (D: the largest), so
// the float orientation is within 2^-33 D + 7 2^-24 D^2 of the exact one,
// and the double formula within 2^-50 D^2 of it; beyond twice that the
// float sign decides, else the double formula
SBMT_DEV bool r3_ccw(const double2* K, const i64* X, const i64* Y) {
  constexpr float S36 = 1.4551915228366852e-11f;  // 2^-36
  // (converted on the FP64 pipe: this kernel waits for loads, and the integer
  // form took it from 205 to 238 us)
  const float ax = __fmul_rn((float)(X[1] - X[0]), S36), ay = __fmul_rn((float)(Y[1] - Y[0]), S36);
  const float bx = __fmul_rn((float)(X[2] - X[0]), S36), by = __fmul_rn((float)(Y[2] - Y[0]), S36);
  const float o = __fsub_rn(__fmul_rn(ax, by), __fmul_rn(ay, bx));
  const float D = fmaxf(fmaxf(fabsf(ax), fabsf(ay)), fmaxf(fabsf(bx), fabsf(by))) + 5.9604645e-8f;
  const float T = 4.7e-10f * D + 1.4e-6f * D * D;
  if (o > T) return true;
  if (o < -T) return false;
  return r3_orient(K[0], K[1], K[2]) > 0.0;
}

// the boundary vertices strictly inside the cell (r3_entry), in corner-id
// order; the count, -1 past R3_MAXI, -2 for a row the cell meets in
// other than two points.  Rows strictly inside the cell's y-range; on each,
// the chord's two ends (a corner on the row, or an edge crossing it, as in
// r3_chord): a corner compared with the pixel corners exactly through its
// fixed-point value, a crossing as a float interval around the double
// formula's position (the crossing filter's bound), the double formula
// taken only where the interval holds the pixel corner compared with.
struct R3End {
  i64 b;     // integer base of the position
  float w, T;
  int src;   // corner 0..2, or 3 + edge
};
// the sign of (an edge end's position) - (cx - 1/2), from the double formula
__device__ __noinline__ int r3_end_cmp_exact(const R3Cell& C, int src, i64 cx, int cy) {
  const double c0 = (double)cy - 0.5;
  const int j = src - 3, u = j, v = j == 2 ? 0 : j + 1;
  const bool fwd = C.id[u] < C.id[v];
  const double p = r3_hx(fwd ? C.K[u] : C.K[v], fwd ? C.K[v] : C.K[u], c0);
  const double x0 = dsb((double)cx, 0.5);
  return p < x0 ? -1 : (p > x0 ? 1 : 0);
}
// the end's position below x0 = cx - 1/2: a corner's exactly from its
// fixed-point value, a crossing's from the float interval or the double
// formula
SBMT_DEV bool r3_end_below(const R3Cell& C, const R3Split* sx, const R3End& e, i64 cx, int cy) {
  if (e.src < 3) return r3_lt(sx[e.src], cx);
  const float h = r3_half(cx - e.b);
  if (__fsub_rn(h, e.w) > e.T) return true;
  if (__fsub_rn(e.w, h) > e.T) return false;
  return r3_end_cmp_exact(C, e.src, cx, cy) < 0;
}
SBMT_DEV bool r3_end_above(const R3Cell& C, const R3Split* sx, const R3End& e, i64 cx, int cy) {
  if (e.src < 3) return r3_gt(sx[e.src], cx);
  const float h = r3_half(cx - e.b);
  if (__fsub_rn(e.w, h) > e.T) return true;
  if (__fsub_rn(h, e.w) > e.T) return false;
  return r3_end_cmp_exact(C, e.src, cx, cy) > 0;
}
SBMT_DEV int r3_inside(const R3Args& a, const R3Cell& C, u64* out) {
  R3Split sx[3], sy[3];
  for (int q = 0; q < 3; ++q) sx[q] = r3_split(C.K[q].x), sy[q] = r3_split(C.K[q].y);
  float sl[3], D[3];
  for (int j = 0; j < 3; ++j) {
    const int u = j, v = j == 2 ? 0 : j + 1;
    const int P = C.id[u] < C.id[v] ? u : v, Q = P == u ? v : u;
    const float dxf = r3_fdiff(sx[Q], sx[P]), dyf = r3_fdiff(sy[Q], sy[P]);
    sl[j] = __fdiv_rn(dxf, dyf), D[j] = fmaxf(fabsf(dxf), fabsf(dyf));
  }
  // rows strictly between the extreme corners, columns through or between them
  R3Split xl = sx[0], xh = sx[0], yl = sy[0], yh = sy[0];
  for (int q = 1; q < 3; ++q) {
    if (sx[q].fx < xl.fx) xl = sx[q];
    if (sx[q].fx > xh.fx || (sx[q].fx == xh.fx && sx[q].inexact)) xh = sx[q];
    if (sy[q].fx < yl.fx) yl = sy[q];
    if (sy[q].fx > yh.fx || (sy[q].fx == yh.fx && sy[q].inexact)) yh = sy[q];
  }
  int cy0, cx0;
  const int rows = r3_lines(yl, yh, a.H, &cy0), cols = r3_lines(xl, xh, a.W, &cx0, true);
  int n = 0;
  for (int cy = cy0; cy < cy0 + rows; ++cy) {
    bool lt[3], gt[3];
    for (int q = 0; q < 3; ++q) lt[q] = r3_lt(sy[q], cy), gt[q] = r3_gt(sy[q], cy);
    R3End e[2];
    int ne = 0;
    for (int q = 0; q < 3; ++q)
      if (!lt[q] && !gt[q]) {  // the corner lies on the row
        if (ne == 2) return -2;
        e[ne++] = R3End{sx[q].i, sx[q].f, 0.0f, q};  // compared exactly
      }
    for (int j = 0; j < 3; ++j) {
      const int u = j, v = j == 2 ? 0 : j + 1;
      if (!((lt[u] && gt[v]) || (lt[v] && gt[u]))) continue;
      if (ne == 2) return -2;
      const int P = C.id[u] < C.id[v] ? u : v;
      const float hP = r3_half(cy - sy[P].i);
      const float w = __fadd_rn(sx[P].f, __fmul_rn(__fsub_rn(hP, sy[P].f), sl[j]));
      e[ne++] = R3End{sx[P].i, w, r3_cross_tol(D[j], sl[j], w), 3 + j};
    }
    if (ne != 2) return -2;
    for (int cx = cx0; cx < cx0 + cols; ++cx) {
      const bool inside = (r3_end_below(C, sx, e[0], cx, cy) && r3_end_above(C, sx, e[1], cx, cy)) ||
                          (r3_end_below(C, sx, e[1], cx, cy) && r3_end_above(C, sx, e[0], cx, cy));
      if (!inside) continue;
      if (!r3_is_vertex(r3_cmask(a, cx, cy))) continue;
      if (n == R3_MAXI) return -1;
      out[n] = r3_entry(3, 3, (int)cx, (int)cy);
      ++n;
    }
  }
  return n;
}

// ---------------------------------------------------------------------------
// the same for a cut cell without a record (the count pass ran out of room),
// by a group of G lanes (sbmt_greedy.cuh): the crossings of its edges with the
// pixel lines and the pixel corners of its bounding box are shared out over the
// lanes
// ---------------------------------------------------------------------------
// a bounded list of the events found on the cell's edges, in no order
constexpr int R3_LIST = R3_MAXN;
struct R3Found {
  int2 mk[R3_LIST];              // the pixel indices (m, k)
  unsigned char jk[R3_LIST];     // edge << 2 | kind
  u32 ins[R3_MAXI];              // inside vertices: corner ids, in id order
};
struct R3Geo2 {  // the cell in the filters' numbers
  R3Split x[3], y[3];
};

// the cell's events into F (up to R3_LIST of them) and their number per edge,
// the same in every lane; each through the float filter of r3_cross_tol, with
// the double formula where it does not decide.  n = 0 cells: live false.
template <int G>
SBMT_DEV int r3_events(const R3Args& a, const R3Cell& C, const R3Geo2& S, bool live, const GLane<G>& me, R3Found& F,
                       int (&cnt)[3]) {
  int ne = 0;
  cnt[0] = cnt[1] = cnt[2] = 0;
#pragma unroll
  for (int vert = 0; vert < 2; ++vert) {
    int first[3], num[3], total = 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int w = j == 2 ? 0 : j + 1;
      num[j] = !live ? 0 : vert ? r3_lines(S.x[j], S.x[w], a.W, &first[j]) : r3_lines(S.y[j], S.y[w], a.H, &first[j]);
      total += num[j];
    }
    const int most = warp_max(total);
    const int ne_h = ne;  // vertical lines: the corners found on the horizontal ones count once
    for (int i0 = 0; i0 < most; i0 += G) {
      const int i = i0 + me.l;
      bool found = false;
      int kind = 0, m = 0, k = 0, j = 0;
      if (i < total) {
        j = i < num[0] ? 0 : i < num[0] + num[1] ? 1 : 2;
        const int line = i - (j > 0 ? num[0] : 0) - (j > 1 ? num[1] : 0) + (j == 0 ? first[0] : j == 1 ? first[1] : first[2]);
        const int u = j, w = j == 2 ? 0 : j + 1;
        const bool fwd = (u == 0 ? C.id[0] : u == 1 ? C.id[1] : C.id[2]) < (w == 0 ? C.id[0] : w == 1 ? C.id[1] : C.id[2]);
        const int pi = fwd ? u : w, qi = fwd ? w : u;
        const R3Split px = pi == 0 ? S.x[0] : pi == 1 ? S.x[1] : S.x[2], py = pi == 0 ? S.y[0] : pi == 1 ? S.y[1] : S.y[2];
        const R3Split qx = qi == 0 ? S.x[0] : qi == 1 ? S.x[1] : S.x[2], qy = qi == 0 ? S.y[0] : qi == 1 ? S.y[1] : S.y[2];
        const float dxf = r3_fdiff(qx, px), dyf = r3_fdiff(qy, py), D = fmaxf(fabsf(dxf), fabsf(dyf));
        const float sl = vert ? __fdiv_rn(dyf, dxf) : __fdiv_rn(dxf, dyf);
        const R3Split& pc = vert ? px : py;  // across the line, and along it
        const R3Split& pl = vert ? py : px;
        const float hp = r3_i2f((int)(line - pc.i)) - 0.5f;
        const float z0 = __fadd_rn(pl.f, __fmul_rn(__fsub_rn(hp, pc.f), sl));
        const float z = __fadd_rn(z0, 0.5f);
        const int zi = r3_ffloor(z);
        const float fr = __fsub_rn(z, r3_i2f(zi)), T = r3_cross_tol(D, sl, z0);
        i64 jj;
        bool corner = false;
        if (fr > T && fr < 1.0f - T) {
          jj = pl.i + zi;
        } else if (r3_corner_ends(px, py, qx, qy, D)) {
          r3_cross_corners(pc, pl, vert ? qx : qy, vert ? qy : qx, line, &jj, &corner);
        } else {
          const double2 P = pi == 0 ? C.K[0] : pi == 1 ? C.K[1] : C.K[2], Q = qi == 0 ? C.K[0] : qi == 1 ? C.K[1] : C.K[2];
          r3_cross_exact(P, Q, (double)line - 0.5, vert, &jj, &corner);
        }
        m = vert ? line : (int)jj, k = vert ? (int)jj : line;
        if (corner) {
          const bool hz = py.fx == qy.fx && py.inexact == qy.inexact && (!py.inexact || r3_same(C.K[u].y, C.K[w].y));
          const bool vt = px.fx == qx.fx && px.inexact == qx.inexact && (!px.inexact || r3_same(C.K[u].x, C.K[w].x));
          kind = 2;
          found = r3_corner_event(a, m, k, hz, vt);
          if (vert)
            for (int t = 0; t < min(ne_h, R3_LIST); ++t)
              if (F.jk[t] == (unsigned char)(j << 2 | 2) && F.mk[t].x == m && F.mk[t].y == k) found = false;
        } else {
          kind = vert;
          found = vert ? r3_vb(a, m, k) : r3_hb(a, m, k);
        }
      }
      const u32 bal = me.ballot(found);
      if (found) {
        const int at = ne + __popc(bal & me.below());
        if (at < R3_LIST) F.mk[at] = make_int2(m, k), F.jk[at] = (unsigned char)(j << 2 | kind);
      }
      ne += __popc(bal);
#pragma unroll
      for (int q = 0; q < 3; ++q) cnt[q] += __popc(me.ballot(found && j == q));
    }
    __syncwarp();
  }
  return ne;
}

// the boundary vertices strictly inside the cell, as corner ids y (W+1) + x in
// id order in F.ins (R3_MAXI at most); their number, the same in every lane
template <int G>
SBMT_DEV int r3_inside_g(const R3Args& a, const R3Cell& C, const R3Geo2& S, bool live, const GLane<G>& me, R3Found& F) {
  // rows strictly between the extreme corners, columns through or between them
  int cy0 = 0, cx0 = 0, rows = 0, cols = 0;
  if (live) {
    R3Split lo = S.y[0], hi = S.y[0];
#pragma unroll
    for (int q = 1; q < 3; ++q) {
      if (S.y[q].fx < lo.fx) lo = S.y[q];
      if (S.y[q].fx > hi.fx || (S.y[q].fx == hi.fx && S.y[q].inexact)) hi = S.y[q];
    }
    rows = r3_lines(lo, hi, a.H, &cy0);
    lo = S.x[0], hi = S.x[0];
#pragma unroll
    for (int q = 1; q < 3; ++q) {
      if (S.x[q].fx < lo.fx) lo = S.x[q];
      if (S.x[q].fx > hi.fx || (S.x[q].fx == hi.fx && S.x[q].inexact)) hi = S.x[q];
    }
    cols = r3_lines(lo, hi, a.W, &cx0, true);
  }
  const int total = rows * cols, most = warp_max(total);
  int n = 0;
  for (int i0 = 0; i0 < most; i0 += G) {
    const int i = i0 + me.l;
    bool inside = false;
    int cy = 0, cx = 0;
    if (i < total) {
      cy = cy0 + i / cols, cx = cx0 + i % cols;
      if (r3_is_vertex(r3_cmask(a, cx, cy))) {
        bool lt[3], gt[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) lt[q] = r3_lt(S.y[q], cy), gt[q] = r3_gt(S.y[q], cy);
        // inside when one chord end is below the corner and the other above
        bool some_below = false, some_above = false;
#pragma unroll
        for (int q = 0; q < 3; ++q)
          if (!lt[q] && !gt[q]) some_below |= r3_lt(S.x[q], cx), some_above |= r3_gt(S.x[q], cx);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const int u = j, v = j == 2 ? 0 : j + 1;
          if (!((lt[u] && gt[v]) || (lt[v] && gt[u]))) continue;
          const bool fwd = C.id[u] < C.id[v];
          const R3Split &px = fwd ? S.x[u] : S.x[v], &py = fwd ? S.y[u] : S.y[v];
          const R3Split &qx = fwd ? S.x[v] : S.x[u], &qy = fwd ? S.y[v] : S.y[u];
          const float dxf = r3_fdiff(qx, px), dyf = r3_fdiff(qy, py), sl = __fdiv_rn(dxf, dyf);
          const float hP = r3_half(cy - py.i);
          const float w = __fadd_rn(px.f, __fmul_rn(__fsub_rn(hP, py.f), sl));
          const float T = r3_cross_tol(fmaxf(fabsf(dxf), fabsf(dyf)), sl, w), h = r3_half(cx - px.i);
          if (__fsub_rn(h, w) > T) some_below = true;
          else if (__fsub_rn(w, h) > T) some_above = true;
          else {
            const int o = r3_end_cmp_exact(C, 3 + j, cx, cy);
            some_below |= o < 0, some_above |= o > 0;
          }
        }
        inside = some_below && some_above;
      }
    }
    const u32 bal = me.ballot(inside);
    if (inside) {
      const int at = n + __popc(bal & me.below());
      if (at < R3_MAXI) F.ins[at] = (u32)cy * (u32)(a.W + 1) + (u32)cx;
    }
    n += __popc(bal);
  }
  __syncwarp();
  return n;
}

// events of the edge from P (its lower-id end) to Q, in order from P, with
// their coordinates, all in the double formulas (the emission's form: every
// event's position is needed there); the count, or -1 past R3_MAXE
SBMT_DEV int r3_edge_events_d(const R3Args& a, double2 P, double2 Q, R3Ev* ev) {
  int n = 0;
  const double dx = dsb(Q.x, P.x), dy = dsb(Q.y, P.y);
  const bool hz = dy == 0.0, vt = dx == 0.0;
  const double ylo = fmin(P.y, Q.y), yhi = fmax(P.y, Q.y), xlo = fmin(P.x, Q.x), xhi = fmax(P.x, Q.x);
  const i64 k0 = max((i64)0, r3_lo(ylo)), k1 = min((i64)a.H, r3_hi(yhi));
  for (i64 k = k0; k <= k1; ++k) {
    const double y0 = (double)k - 0.5;
    if (!(ylo < y0 && y0 < yhi)) continue;
    const double x = r3_hx(P, Q, y0);
    i64 j;
    const bool corner = r3_at_corner(x, &j);
    if (corner ? r3_corner_event(a, j, k, hz, vt) : r3_hb(a, j, k)) {
      if (n == R3_MAXE) return -1;
      ev[n++] = R3Ev{x, y0, 0.0, corner ? 2 : 0, (int)j, (int)k};
    }
  }
  const i64 m0 = max((i64)0, r3_lo(xlo)), m1 = min((i64)a.W, r3_hi(xhi));
  for (i64 m = m0; m <= m1; ++m) {
    const double x0 = (double)m - 0.5;
    if (!(xlo < x0 && x0 < xhi)) continue;
    const double y = r3_vy(P, Q, x0);
    i64 j;
    const bool corner = r3_at_corner(y, &j);
    if (corner) {
      bool dup = false;
      for (int t = 0; t < n; ++t)
        if (ev[t].kind == 2 && ev[t].m == (int)m && ev[t].k == (int)j) dup = true;
      if (dup || !r3_corner_event(a, m, j, hz, vt)) continue;
    } else if (!r3_vb(a, m, j)) {
      continue;
    }
    if (n == R3_MAXE) return -1;
    ev[n++] = R3Ev{x0, y, 0.0, corner ? 2 : 1, (int)m, (int)j};
  }
  const bool alongx = fabs(dx) >= fabs(dy);
  for (int t = 0; t < n; ++t) ev[t].s = alongx ? ddv(dsb(ev[t].x, P.x), dx) : ddv(dsb(ev[t].y, P.y), dy);
  // insertion sort by (s, kind, k, m)
  for (int t = 1; t < n; ++t) {
    const R3Ev e = ev[t];
    int u = t - 1;
    while (u >= 0) {
      const R3Ev& f = ev[u];
      const bool gt = f.s != e.s ? f.s > e.s : f.kind != e.kind ? f.kind > e.kind : f.k != e.k ? f.k > e.k : f.m > e.m;
      if (!gt) break;
      ev[u + 1] = f;
      --u;
    }
    ev[u + 1] = e;
  }
  return n;
}

// the boundary vertices strictly inside the cell, as corner ids y (W+1) + x
// in id order, in the double formulas (the emission's form); the count, or
// -1 past R3_MAXI (ids written when out != null)
SBMT_DEV int r3_inside_d(const R3Args& a, const R3Cell& C, u32* out) {
  int n = 0;
  const i64 cy0 = max((i64)0, r3_lo(C.ylo)), cy1 = min((i64)a.H, r3_hi(C.yhi));
  const i64 cx0 = max((i64)0, r3_lo(C.xlo)), cx1 = min((i64)a.W, r3_hi(C.xhi));
  for (i64 cy = cy0; cy <= cy1; ++cy) {
    const double y0 = (double)cy - 0.5;
    if (!(C.ylo < y0 && y0 < C.yhi)) continue;
    double pos[2];
    int src[2];
    if (r3_chord(C.K, C.id, false, y0, pos, src) != 2) return -2;
    for (i64 cx = cx0; cx <= cx1; ++cx) {
      const double x0 = (double)cx - 0.5;
      if (!(pos[0] < x0 && x0 < pos[1])) continue;
      if (!r3_is_vertex(r3_cmask(a, cx, cy))) continue;
      if (n == R3_MAXI) return -1;
      if (out) out[n] = (u32)(cy * (a.W + 1) + cx);
      ++n;
    }
  }
  return n;
}

// the other cell beside the cell's edge j (-1 on the mesh's outer boundary;
// -2 when more than one other cell has the edge)
SBMT_DEV int r3_neighbour(const R3Args& a, u32 c, const R3Cell& C, int j) {
  const int u = C.id[j], w = C.id[j == 2 ? 0 : j + 1];
  int found = -1;
  for (u32 e = a.head[u]; e != NONE;) {
    const u32 c2 = a.cand[e / 3u];
    e = a.link[e];
    if (c2 == c) continue;
    const int* t = a.ttri + 3 * (u64)c2;
    if (t[0] == w || t[1] == w || t[2] == w) {
      if (found >= 0) return -2;
      found = (int)c2;
    }
  }
  return found;
}

// the local edge of cell c2 running between vertices u and w
SBMT_DEV int r3_edge_in(const R3Args& a, u32 c2, int u, int w) {
  const int* t = a.ttri + 3 * (u64)c2;
  for (int j = 0; j < 3; ++j) {
    const int p = t[j], q = t[j == 2 ? 0 : j + 1];
    if ((p == u && q == w) || (p == w && q == u)) return j;
  }
  return -1;
}

// ---------------------------------------------------------------------------
// The candidate cells around each vertex, for the cell across an edge: an edge
// with events has boundary on both sides of it, so the cells beside it are
// candidates, and only those need listing -- a linked list per vertex, pushed
// by exchanging its head (the counts, scan and lists over every cell took 0.19
// ms for 9.8e6 cells, 0.02 ms for the few percent that are
// candidates).  Entry 3 q + k is candidate q's at its corner k, so that an entry is
// its successor alone.  The order of a list depends on the run; what is looked up
// in it does not.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_r3_link(R3Args a) {
  const u32 n = *a.ncand;
  for (u32 q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const u32 c = a.cand[q];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int v = a.ttri[3 * (u64)c + k];
      if (v < 0 || (u32)v >= a.nv) {
        atomicOr(a.err, R3_GEOMETRY);
        continue;
      }
      const u32 e = 3 * q + (u32)k;
      a.link[e] = atomicExch(a.head + v, e);
    }
  }
}

// ---------------------------------------------------------------------------
// screen: every cell; a cell whose pixel box carries one label is uncut (its
// label is the box's); the others go to the candidate list
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_r3_screen(R3Args a) {
  const int lane = threadIdx.x & 31;
  for (u64 c0 = (u64)blockIdx.x * blockDim.x; c0 < a.nt; c0 += (u64)gridDim.x * blockDim.x) {
    const u64 c = c0 + threadIdx.x;
    bool cand = false;
    if (c < a.nt) {
      const int* t = a.ttri + 3 * c;
      double2 K[3];
      i64 X[3], Y[3];
      for (int q = 0; q < 3; ++q) {
        K[q] = reinterpret_cast<const double2*>(a.txy)[t[q]];
        bool ix, iy;
        X[q] = r3_fix36(K[q].x, &ix), Y[q] = r3_fix36(K[q].y, &iy);
      }
      int l = -1;
      if (!r3_ccw(K, X, Y)) atomicOr(a.err, R3_GEOMETRY);
      else l = r3_uniform(a, X, Y);
      cand = l < 0;
      a.ulab[c] = (unsigned short)(cand ? 0 : l);
    }
    const unsigned m = __ballot_sync(0xFFFFFFFFu, cand);
    // a warp's 32 cells fill one word of the candidate bit-plane
    const u64 w0 = c0 + (threadIdx.x & ~31u);
    if (lane == 0 && w0 < a.nt) a.cmark[w0 >> 5] = m;
    if (m) {
      u32 base = 0;
      if (lane == 0) base = atomicAdd(a.ncand, (u32)__popc(m));
      base = __shfl_sync(0xFFFFFFFFu, base, 0);
      if (cand) a.cand[base + __popc(m & ((1u << lane) - 1u))] = (u32)c;
    }
  }
}

// The lists of the cut cells, by node count: at most 8 and at most 16 from the
// two ends of cutl, at most 32 and above from the two ends of glist, and those
// of at most 32 nodes without a record in ovl; ncls[q] is the length of list q.
// Lists 0 to 2 hold records' places, the others cells.
SBMT_DEV u32* r3_list(const R3Args& a, int q, u32 i) {
  u32* base = q < 2 ? a.cutl : q < 4 ? a.glist : a.ovl;
  return (q & 1) ? base + (a.nt - 1 - i) : base + i;
}
// A cut cell's record, in 64-bit words of rec: {cell, neighbour of edge 0},
// {neighbours of edges 1 and 2} (-1: none), {counts: events per edge and inside
// vertices, a byte each}, then the events' and the inside vertices' entries.
// The room is one word per cell of the mesh (a few percent of them are cut);
// a cell for which it is used up is listed without a record.
constexpr int R3_HEAD = 3;

// the events on the cell's edges, through the filters (the count pass's form:
// positions are not needed there): their number, or -1 past R3_MAXE on an edge; ev
// receives them (r3_entry), cnt their number per edge.  One loop over the lines
// of all three edges: with a loop an edge and direction, a warp ran the longest of
// each (437 us for the candidates of 4096^2 labels, 397 this way, 382 with registers
// for six blocks an SM instead of four).
SBMT_DEV int r3_events_t(const R3Args& a, const R3Cell& C, u64* ev, int (&cnt)[3]) {
  R3Split sx[3], sy[3];
#pragma unroll
  for (int t = 0; t < 3; ++t) sx[t] = r3_split(C.K[t].x), sy[t] = r3_split(C.K[t].y);
  // per edge: its lower-id end first, the differences, whether between two pixel corners
  float dx[3], dy[3], D[3];
  bool fwd[3], grid[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int w = j == 2 ? 0 : j + 1;
    fwd[j] = C.id[j] < C.id[w];
    dx[j] = r3_fdiff(sx[w], sx[j]), dy[j] = r3_fdiff(sy[w], sy[j]);
    D[j] = fmaxf(fabsf(dx[j]), fabsf(dy[j])), grid[j] = r3_corner_ends(sx[j], sy[j], sx[w], sy[w], D[j]);
  }
  int ne = 0;
  cnt[0] = cnt[1] = cnt[2] = 0;
#pragma unroll 1
  for (int vert = 0; vert < 2; ++vert) {
    int first[3], num[3];
    float slope[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int w = j == 2 ? 0 : j + 1;
      num[j] = vert ? r3_lines(sx[j], sx[w], a.W, &first[j]) : r3_lines(sy[j], sy[w], a.H, &first[j]);
      slope[j] = vert ? __fdiv_rn(dy[j], dx[j]) : __fdiv_rn(dx[j], dy[j]);  // (not used without lines)
    }
    const int total = num[0] + num[1] + num[2], ne_h = ne;  // vertical lines: the corners found on the horizontal ones count once
#pragma unroll 1
    for (int i = 0; i < total; ++i) {
      const int j = i < num[0] ? 0 : i < num[0] + num[1] ? 1 : 2;
      const int line = i - (j > 0 ? num[0] : 0) - (j > 1 ? num[1] : 0) + (j == 0 ? first[0] : j == 1 ? first[1] : first[2]);
      const bool fw = j == 0 ? fwd[0] : j == 1 ? fwd[1] : fwd[2];
      const int pi = fw ? j : (j == 2 ? 0 : j + 1), qi = fw ? (j == 2 ? 0 : j + 1) : j;
      const R3Split px = pi == 0 ? sx[0] : pi == 1 ? sx[1] : sx[2], py = pi == 0 ? sy[0] : pi == 1 ? sy[1] : sy[2];
      const R3Split& pc = vert ? px : py;  // across the line, and along it
      const R3Split& pl = vert ? py : px;
      const float sl = j == 0 ? slope[0] : j == 1 ? slope[1] : slope[2], Dj = j == 0 ? D[0] : j == 1 ? D[1] : D[2];
      const float hp = r3_i2f((int)(line - pc.i)) - 0.5f;
      const float w = __fadd_rn(pl.f, __fmul_rn(__fsub_rn(hp, pc.f), sl));
      const float z = __fadd_rn(w, 0.5f);
      const int zi = r3_ffloor(z);
      const float fr = __fsub_rn(z, r3_i2f(zi)), tol = r3_cross_tol(Dj, sl, w);
      i64 at;
      bool corner = false;
      if (fr > tol && fr < 1.0f - tol) {
        at = pl.i + zi;
      } else {
        const R3Split qx = qi == 0 ? sx[0] : qi == 1 ? sx[1] : sx[2], qy = qi == 0 ? sy[0] : qi == 1 ? sy[1] : sy[2];
        if (j == 0 ? grid[0] : j == 1 ? grid[1] : grid[2]) {
          r3_cross_corners(pc, pl, vert ? qx : qy, vert ? qy : qx, line, &at, &corner);
        } else {
          const double2 P = pi == 0 ? C.K[0] : pi == 1 ? C.K[1] : C.K[2], Q = qi == 0 ? C.K[0] : qi == 1 ? C.K[1] : C.K[2];
          r3_cross_exact(P, Q, (double)line - 0.5, vert, &at, &corner);
        }
      }
      const i64 m = vert ? line : at, k = vert ? at : line;
      const u64 entry = r3_entry(j, corner ? 2 : vert, (int)m, (int)k);
      bool found;
      if (corner) {
        const double2 P = pi == 0 ? C.K[0] : pi == 1 ? C.K[1] : C.K[2], Q = qi == 0 ? C.K[0] : qi == 1 ? C.K[1] : C.K[2];
        bool dup = false;
        if (vert)
          for (int t = 0; t < ne_h; ++t) dup |= ev[t] == entry;
        found = !dup && r3_corner_event(a, m, k, r3_same(P.y, Q.y), r3_same(P.x, Q.x));
      } else {
        found = vert ? r3_vb(a, m, k) : r3_hb(a, m, k);
      }
      if (!found) continue;
      if ((j == 0 ? cnt[0] : j == 1 ? cnt[1] : cnt[2]) == R3_MAXE) return -1;
      ev[ne++] = entry;
      cnt[0] += j == 0, cnt[1] += j == 1, cnt[2] += j == 2;
    }
  }
  return ne;
}

// the candidates: events on the edges, inside vertices, the cells beside
// the edges that carry events.  (Eight lanes a candidate, as in k_r3_cells,
// took 0.99 ms against 0.44: here the cells are alike, and what every lane
// needs is computed once.)
__global__ void __launch_bounds__(128, 6) k_r3_count(R3Args a) {
  u64 ev[3 * R3_MAXE + R3_MAXI];
  const u32 n = *a.ncand;
  for (u32 q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const u32 c = a.cand[q];
    const R3Cell C = r3_load_k(a, c);
    int cnt[3];
    const int found = r3_events_t(a, C, ev, cnt);
    const bool bad = found < 0;
    const int ne = bad ? 0 : found;
    const int ni = bad ? 0 : r3_inside(a, C, ev + ne);
    if (bad || ni == -1 || 3 + ne + ni > R3_MAXN) {
      atomicOr(a.err, R3_CAPACITY);
    } else if (ni < 0) {
      atomicOr(a.err, R3_GEOMETRY);
    } else if (ne + ni > 0) {
      const unsigned act = __activemask();
      const int lane = threadIdx.x & 31, lead = __ffs(act) - 1;
      if (lane == lead) atomicAdd(a.ncut, (u32)__popc(act));
      int nb[3] = {-1, -1, -1};
      u32 nown = 0, own3 = 0;
      for (int j = 0; j < 3; ++j) {
        if (cnt[j] == 0) continue;
        nb[j] = r3_neighbour(a, c, C, j);
        if (nb[j] == -2) atomicOr(a.err, R3_GEOMETRY);
        if (nb[j] < 0 || (u32)nb[j] > c) nown += (u32)cnt[j], own3 |= (u32)cnt[j] << (8 * j);
      }
      a.ntri[c] = (u32)(2 * ni + 3 + ne - 2), a.nin[c] = (u32)ni, a.nown[c] = nown, a.own3[c] = own3;
      atomicOr(a.kmark + (c >> 5), 1u << (c & 31));
      atomicAdd(a.wsum[0] + (c >> 5), (u32)(2 * ni + ne));
      if (nown) atomicAdd(a.wsum[1] + (c >> 5), nown);
      if (ni) atomicAdd(a.wsum[2] + (c >> 5), (u32)ni);
      // the record, and the cell's place in its list: one atomic per list and
      // group of lanes
      const int nodes = 3 + ne + ni;
      int cls = nodes <= 8 ? 0 : nodes <= 16 ? 1 : nodes <= 32 ? 2 : 3;
      u32 item = c;
      if (cls < 3) {
        const u32 words = (u32)(R3_HEAD + ne + ni);
        const unsigned long long at = atomicAdd(a.nrec, (unsigned long long)words);
        if (at + words <= a.nt) {
          u64* r = a.rec + at;
          r[0] = (u64)c | (u64)(u32)nb[0] << 32, r[1] = (u64)(u32)nb[1] | (u64)(u32)nb[2] << 32;
          r[2] = (u64)(cnt[0] | cnt[1] << 8 | cnt[2] << 16 | ni << 24);
          for (int t = 0; t < ne + ni; ++t) r[R3_HEAD + t] = ev[t];
          item = (u32)at;
        } else {
          cls = 4;
        }
      }
      const unsigned peers = __match_any_sync(__activemask(), cls);
      const int first = __ffs(peers) - 1;
      u32 base = 0;
      if (lane == first) base = atomicAdd(a.ncls + cls, (u32)__popc(peers));
      base = __shfl_sync(peers, base, first);
      *r3_list(a, cls, base + __popc(peers & ((1u << lane) - 1u))) = item;
    }
  }
}

// ---------------------------------------------------------------------------
// the local boundary graph of a cut cell
// ---------------------------------------------------------------------------
struct R3Local {
  int nev[3], ne, ni, n, np;
  double2 v[R3_MAXN];
  u32 gid[R3_MAXN];
  unsigned char on_edge[R3_MAXN];
  unsigned char pa[R3_MAXP], pb[R3_MAXP];
  int mask, klass;
};

// Offsets.  An uncut cell has one triangle and nothing else, and a few percent
// of the cells are cut, so the counts are summed and scanned per word of 32
// cells, and the cut cells before a cell in its word added on use (dense counts
// and three scans over every cell: 0.36 ms of writes and passes for 9.8e6 cells;
// 0.03 ms this way).  The events owned by the cells before c:
SBMT_DEV u32 r3_before(const R3Args& a, u32 c, int which, const u32* count, u32 one) {
  u32 sum = a.woff[which][c >> 5];
  for (u32 m = a.kmark[c >> 5] & ((1u << (c & 31)) - 1u); m; m &= m - 1)
    sum += count[(c & ~31u) + (u32)__ffs(m) - 1u] - one;
  return sum;
}
SBMT_DEV u32 r3_toff(const R3Args& a, u32 c) { return c + r3_before(a, c, 0, a.ntri, 1u); }
SBMT_DEV u32 r3_ioff(const R3Args& a, u32 c) { return r3_before(a, c, 2, a.nin, 0u); }
// the first event id of cell c's edge j
SBMT_DEV u32 r3_edge_base(const R3Args& a, u32 c, int j) {
  const u32 o = a.own3[c];
  u32 b = a.nv + r3_before(a, c, 1, a.nown, 0u);
  for (int t = 0; t < j; ++t) b += (o >> (8 * t)) & 255u;
  return b;
}

// builds L for cut cell c; writes the coordinates of the events of the edges
// c owns and of its inside vertices when write is set; 0, or an R3_ error
template <typename EvBuf>
SBMT_DEV u32 r3_build(const R3Args& a, u32 c, const R3Cell& C, R3Local& L, EvBuf& ev, bool write) {
  L.ne = 0;
  L.n = 3;
  for (int q = 0; q < 3; ++q) {
    L.v[q] = C.K[q], L.gid[q] = (u32)C.id[q];
    L.on_edge[q] = (unsigned char)((1 << q) | (1 << (q == 0 ? 2 : q - 1)));
  }
  // events per edge, in counter-clockwise order along the cell's edge j
  for (int j = 0; j < 3; ++j) {
    const int u = j, w = j == 2 ? 0 : j + 1;
    const bool fwd = C.id[u] < C.id[w];
    R3Ev* e = ev[j];
    const int n = r3_edge_events_d(a, fwd ? C.K[u] : C.K[w], fwd ? C.K[w] : C.K[u], e);
    if (n < 0 || L.n + n > R3_MAXN) return R3_CAPACITY;
    L.nev[j] = n;
    if (n == 0) continue;
    const int nb = r3_neighbour(a, c, C, j);
    if (nb == -2) return R3_GEOMETRY;
    u32 base;
    if (nb < 0 || (u32)nb > c) {
      base = r3_edge_base(a, c, j);
      if (write)
        for (int t = 0; t < n; ++t) reinterpret_cast<double2*>(a.xy)[base + t] = make_double2(e[t].x, e[t].y);
    } else {
      const int j2 = r3_edge_in(a, (u32)nb, C.id[u], C.id[w]);
      if (j2 < 0) return R3_GEOMETRY;
      base = r3_edge_base(a, (u32)nb, j2);
    }
    if (!fwd)  // counter-clockwise along j runs from the higher-id end
      for (int t = 0; t < n / 2; ++t) {
        const R3Ev x = e[t];
        e[t] = e[n - 1 - t], e[n - 1 - t] = x;
      }
    for (int t = 0; t < n; ++t) {
      L.v[L.n] = make_double2(e[t].x, e[t].y);
      L.gid[L.n] = base + (fwd ? (u32)t : (u32)(n - 1 - t));
      L.on_edge[L.n] = (unsigned char)(1 << j);
      ++L.n;
    }
    L.ne += n;
  }
  // inside vertices
  u32 ins[R3_MAXI];
  const int ni = r3_inside_d(a, C, ins);
  if (ni == -1 || L.n + ni > R3_MAXN) return R3_CAPACITY;
  if (ni < 0) return R3_GEOMETRY;
  L.ni = ni;
  const u32 ibase = a.nv + a.ne_total + r3_ioff(a, c);
  for (int t = 0; t < ni; ++t) {
    const u32 cid = ins[t];
    const double2 p = make_double2((double)(cid % (u32)(a.W + 1)) - 0.5, (double)(cid / (u32)(a.W + 1)) - 0.5);
    L.v[L.n] = p, L.gid[L.n] = ibase + (u32)t, L.on_edge[L.n] = 0;
    if (write) reinterpret_cast<double2*>(a.xy)[ibase + t] = p;
    ++L.n;
  }
  // pieces: horizontal lines by y, then vertical lines by x, each along the
  // line; oriented with the lower label on the left
  L.np = 0;
  for (int vert = 0; vert < 2; ++vert) {
    const double lo = vert ? C.xlo : C.ylo, hi = vert ? C.xhi : C.yhi;
    const i64 L0 = max((i64)0, r3_lo(lo)), L1 = min((i64)(vert ? a.W : a.H), r3_hi(hi));
    for (i64 line = L0; line <= L1; ++line) {
      const double c0 = (double)line - 0.5;
      if (!(lo < c0 && c0 < hi)) continue;
      double pos[2];
      int src[2];
      if (r3_chord(C.K, C.id, vert, c0, pos, src) != 2) return R3_GEOMETRY;
      // nodes on the line: the chord ends that are nodes, the inside vertices
      int nd[R3_MAXI + 2];
      double np_[R3_MAXI + 2];
      int nn = 0;
      for (int end = 0; end < 2; ++end) {
        int node = -1;
        if (src[end] < 3) {
          node = src[end];
        } else {
          const int j = src[end] - 3;
          int b = 3;
          for (int t = 0; t < j; ++t) b += L.nev[t];
          for (int t = 0; t < L.nev[j]; ++t) {
            const R3Ev& e = ev[j][t];
            const bool hit = e.kind == 2 ? (vert ? e.m == line : e.k == line)
                                         : (e.kind == (vert ? 1 : 0) && (vert ? e.m : e.k) == line);
            if (hit) {
              node = b + t;
              break;
            }
          }
        }
        if (end == 1) {
          for (int t = 0; t < ni; ++t) {
            const u32 cid = ins[t];
            const i64 cx = cid % (u32)(a.W + 1), cy = cid / (u32)(a.W + 1);
            if ((vert ? cx : cy) == line)
              nd[nn] = 3 + L.ne + t, np_[nn++] = vert ? (double)cy - 0.5 : (double)cx - 0.5;
          }
        }
        if (node >= 0) nd[nn] = node, np_[nn++] = pos[end];
      }
      for (int t = 0; t + 1 < nn; ++t) {
        const double mid = dml(dad(np_[t], np_[t + 1]), 0.5);
        i64 j;
        r3_at_corner(mid, &j);  // at a corner: the pixel edge starting there
        int l0, l1;
        bool fwd;
        if (!vert) {
          if (!r3_hb(a, j, line)) continue;
          l0 = r3_px(a, j, line - 1), l1 = r3_px(a, j, line);
          fwd = l1 < l0;  // going +x the left side is above
        } else {
          if (!r3_vb(a, line, j)) continue;
          l0 = r3_px(a, line - 1, j), l1 = r3_px(a, line, j);
          fwd = l0 < l1;  // going +y the left side is -x
        }
        if (L.np == R3_MAXP) return R3_CAPACITY;
        L.pa[L.np] = (unsigned char)(fwd ? nd[t] : nd[t + 1]);
        L.pb[L.np] = (unsigned char)(fwd ? nd[t + 1] : nd[t]);
        ++L.np;
      }
    }
  }
  // Alg. 1 mask (a corner on a piece sets both its edges, an event its
  // edge, an edge on a boundary run its own bit, bit 0 an inside vertex) and
  // the (m, n) class of the first two pieces
  auto bits = [&](int w) -> int {
    if (w < 3) return (2 << w) | (2 << (w == 0 ? 2 : w - 1));
    if (w < 3 + L.ne) {
      int k = w - 3;
      for (int j = 0; j < 3; ++j) {
        if (k < L.nev[j]) return 2 << j;
        k -= L.nev[j];
      }
    }
    return 0;
  };
  int mask = L.ni > 0 ? 1 : 0, pc0 = 0, pc1 = 0;
  for (int t = 0; t < L.np; ++t) {
    const int b = bits(L.pa[t]) | bits(L.pb[t]);
    mask |= b;
    if (t == 0) pc0 = __popc(b);
    if (t == 1) pc1 = __popc(b);
  }
  for (int j = 0; j < 3; ++j) {
    const double2 p = C.K[j], q = C.K[j == 2 ? 0 : j + 1];
    for (int vert = 0; vert < 2; ++vert) {
      const double ca = vert ? p.x : p.y, cb = vert ? q.x : q.y;
      i64 line;
      if (ca != cb || !r3_at_corner(ca, &line)) continue;
      const double ta = vert ? p.y : p.x, tb = vert ? q.y : q.x;
      const double t0 = fmin(ta, tb), t1 = fmax(ta, tb);
      for (i64 g = r3_lo(t0) - 1; g <= r3_hi(t1) + 1; ++g) {
        if (!((double)g + 0.5 > t0 && (double)g - 0.5 < t1)) continue;
        if (vert ? r3_vb(a, line, g) : r3_hb(a, g, line)) mask |= 2 << j;
      }
    }
  }
  L.mask = mask;
  L.klass = L.np == 1 ? thm32_class(0, pc0) : L.np == 2 ? thm32_class(pc0, pc1) : 0;
  return 0;
}

// the label of the pixel holding ((x1 + x2) + x3) / 3
SBMT_DEV unsigned short r3_label(const R3Args& a, double2 p, double2 q, double2 r) {
  const double cx = ddv(dad(dad(p.x, q.x), r.x), 3.0), cy = ddv(dad(dad(p.y, q.y), r.y), 3.0);
  const int l = r3_px(a, (i64)floor(dad(cx, 0.5)), (i64)floor(dad(cy, 0.5)));
  return l == R3_OUTSIDE ? (unsigned short)0xFFFF : (unsigned short)l;
}

__device__ __noinline__ unsigned short r3_label_d(const R3Args& a, double2 p, double2 q, double2 r) {
  return r3_label(a, p, q, r);
}
// the same from the coordinates' fixed-point values, sx and sy their sums:
// floor((X1 + X2 + X3) / 3 + 1/2) is the double formula's unless the sum is
// within a bound of a pixel line (three floors, 3 2^-36 below the exact sum at
// most; the double formula's roundings, below 2^-25 px at 2^24).  -1 when it is.
SBMT_DEV int r3_label36(const R3Args& a, i64 sx, i64 sy) {
  constexpr i64 ONE3 = 3ll << 36, BAND = 1ll << 14;  // 3 px; 2^-22 px
  i64 at[2];
  bool near = false;
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    // the quotient by 3 2^36: the upper part first, so that 32 bits divide
    const i64 sum = (d ? sy : sx) + (ONE3 >> 1);
    const int hi = (int)(sum >> 36);
    const int f = (hi >= 0 ? hi : hi - 2) / 3;
    const i64 rem = sum - (i64)f * ONE3;
    at[d] = f;
    near |= rem < BAND || rem > ONE3 - BAND;
  }
  if (near) return -1;
  const int l = r3_px(a, at[0], at[1]);
  return l == R3_OUTSIDE ? 0xFFFF : l;
}

// ---------------------------------------------------------------------------
// the cells left as they are: uncut cells of one label, labelled by their
// pixel box, and candidates the boundary only touches (at a corner or along
// an edge), labelled by the pixel holding the centroid
// ---------------------------------------------------------------------------
// (the kernel took 148 us on 4096^2 labels with the double formula for every
// candidate left as it is, 128 with the fixed-point one: its loads bound it now)
__device__ __noinline__ unsigned short r3_cell_label(const R3Args& a, int u, int v, int w) {
  const double2* K = reinterpret_cast<const double2*>(a.txy);
  const double2 p = K[u], q = K[v], r = K[w];
  bool ix;
  const i64 sx = r3_fix36(p.x, &ix) + r3_fix36(q.x, &ix) + r3_fix36(r.x, &ix);
  const i64 sy = r3_fix36(p.y, &ix) + r3_fix36(q.y, &ix) + r3_fix36(r.y, &ix);
  const int l = r3_label36(a, sx, sy);
  return l >= 0 ? (unsigned short)l : r3_label_d(a, p, q, r);
}
__global__ void __launch_bounds__(256) k_r3_emit_uncut(R3Args a) {
  const u32 lane = threadIdx.x & 31u;
  for (u64 c0 = (u64)blockIdx.x * blockDim.x; c0 < a.nt; c0 += (u64)gridDim.x * blockDim.x) {
    const u64 c = c0 + threadIdx.x;  // a warp has the 32 cells of a word
    const u64 word = c >> 5;
    const u32 cuts = word < (a.nt + 31) / 32 ? a.kmark[word] : 0u;
    const bool cut = (cuts >> lane) & 1u;
    u32 extra = 0;
    if (cuts) {
      const u32 own = cut ? a.ntri[c] - 1u : 0u;
      extra = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const u32 y = __shfl_up_sync(0xFFFFFFFFu, extra, o);
        if (lane >= (u32)o) extra += y;
      }
      extra -= own;
    }
    const u64 w0 = c & ~31ull;
    if (cuts == 0 && w0 + 32 <= a.nt) {
      // 32 uncut cells: their triangles are consecutive on both sides, copied
      // as whole lines
      const u64 o0 = w0 + a.woff[0][word];
      const int* in = a.ttri + 3 * w0 + lane;
      const int v0 = in[0], v1 = in[32], v2 = in[64];
      const u32 cm = a.cmark[word];
      unsigned short lab;
      if ((cm >> lane) & 1u) {
        const int* t = a.ttri + 3 * c;
        lab = r3_cell_label(a, t[0], t[1], t[2]);
      } else {
        lab = a.ulab[c];
      }
      int* out = a.tri + 3 * o0 + lane;
      out[0] = v0, out[32] = v1, out[64] = v2;
      a.label[o0 + lane] = lab;
      a.code[o0 + lane] = 0;
      continue;
    }
    if (c >= a.nt || cut) continue;
    const u64 t0 = c + a.woff[0][word] + extra;
    const int* t = a.ttri + 3 * c;
    const int3 tv = make_int3(t[0], t[1], t[2]);
    unsigned short lab;
    if ((a.cmark[c >> 5] >> (c & 31)) & 1u) {
      lab = r3_cell_label(a, tv.x, tv.y, tv.z);
    } else {
      lab = a.ulab[c];
    }
    reinterpret_cast<int3*>(a.tri)[t0] = tv;
    a.label[t0] = lab;
    a.code[t0] = 0;
  }
}

// ---------------------------------------------------------------------------
// the cut cells of at most 32 nodes: a group of 8, 16 or 32 lanes each builds
// the local boundary graph and takes the template of a Tier-T cell or the
// greedy rule (sbmt_greedy.cuh) of a Tier-G one.  The double formulas run one
// event, candidate or piece per lane; positions on pixel lines, orientations
// and centroid labels are decided in fixed point or single precision where a
// bound allows.
// ---------------------------------------------------------------------------
template <int G>
struct R3State {
  GCell<G> c;
  R3Found F;                  // a cell without a record
  unsigned char ix[3];        // corners: whether x, y are off the fixed-point grid
  unsigned char tj[G];        // the events as found: edge << 2 | kind, pixel indices
  int2 tmk[G];
  double vx[G], vy[G];  // the nodes: corners, events counter-clockwise, inside vertices
  i64 X[G], Y[G];       // floor(v 2^36)
  double s[G];          // while ordering: the events' parameters along their edges
  u32 gid[G];
  int2 mk[G];             // events: pixel indices and kind, in node order
  unsigned char kind[G];
  unsigned char pa[3 * G], pb[3 * G];  // the pieces
};

// The kernel is long: what it needs rarely or in several places is kept out of
// line, and short loops stay loops (inlined and unrolled it waited for
// instructions in 18 of 27 cycles per issue: 595 us against 527, before the barriers below).
__device__ __noinline__ int r3_late(const double* x, const double* y, int u, int v, int w) {
  return r3_sgn(r3_orient(make_double2(x[u], y[u]), make_double2(x[v], y[v]), make_double2(x[w], y[w])));
}
__device__ __noinline__ int r3_pixel(const R3Args& a, int x, int y) { return r3_px(a, x, y); }

// the geometry for the greedy rule: the filter decides outside its band, and
// the double formula of each test, taken as the rule states it, inside.  The
// float coordinates are within 2^-24 M + 2^-35 of the differences from the
// first corner (M: the largest), so a float determinant is within
// 48 2^-24 M^2 + 8 2^-35 M of the doubles' exact one and the double formula
// within 32 2^-53 M^2 of it.
template <int G>
struct R3Geo {
  const R3State<G>* s;
  float T;
  SBMT_DEV float tol() const { return T; }
  SBMT_DEV double2 pt(int k) const { return make_double2(s->vx[k], s->vy[k]); }
  SBMT_DEV bool resolve(int, int, int, int*) const { return false; }
  SBMT_DEV int late(int u, int v, int w) const { return r3_late(s->vx, s->vy, u, v, w); }
  SBMT_DEV bool between(int u, int w, int k) const {
    const double2 pu = pt(u), pw = pt(w), pk = pt(k);
    const double ex = dsb(pw.x, pu.x), ey = dsb(pw.y, pu.y), len2 = dad(dml(ex, ex), dml(ey, ey));
    const double t = dad(dml(dsb(pk.x, pu.x), ex), dml(dsb(pk.y, pu.y), ey));
    return t > 0.0 && t < len2;
  }
  SBMT_DEV float key(int u, int w, int) const {
    const double dx = dsb(s->vx[w], s->vx[u]), dy = dsb(s->vy[w], s->vy[u]);
    return __double2float_rn(dad(dml(dx, dx), dml(dy, dy)));
  }
  SBMT_DEV bool less(float kx, unsigned short x, int, float ky, unsigned short y, int) const {
    return kx < ky || (kx == ky && x < y);
  }
};

// r3_at_corner through the fixed-point value
SBMT_DEV bool r3_at_corner36(double t, i64* idx) {
  bool inexact;
  const i64 f = r3_fix36(t, &inexact), fl = f >> 36, fr = f & ((1ll << 36) - 1);
  constexpr i64 HALF = 1ll << 35;
  *idx = fr < HALF ? fl : fl + 1;
  return fr == HALF && !inexact;
}

template <int G>
__device__ __noinline__ unsigned short r3_node_label(const R3Args& a, const R3State<G>& s, int p, int q, int r) {
  const int l = r3_label36(a, s.X[p] + s.X[q] + s.X[r], s.Y[p] + s.Y[q] + s.Y[r]);
  return l >= 0 ? (unsigned short)l
                : r3_label(a, make_double2(s.vx[p], s.vy[p]), make_double2(s.vx[q], s.vy[q]),
                           make_double2(s.vx[r], s.vy[r]));
}

// Tier-T: the key and rotation of the cell in the table's regime, or key 0
// (-1: a graph outside the table where none can be)
template <int G>
SBMT_DEV int r3_tier_t(const R3State<G>& s, int ni, int ne, int np, int n0, int n1, int n2, int* sigma_out) {
  if (ni > 1 || np > 8) return 0;
  const int P = 3 + ne;
  u32 once = 0, twice = 0;
  for (int t = 0; t < np; ++t) {
    if (s.pa[t] < 3 || s.pb[t] < 3) return 0;
    const u32 x = 1u << s.pa[t], y = 1u << s.pb[t];
    twice |= once & x, once |= x;
    twice |= once & y, once |= y;
  }
  const u32 evs = ((1u << ne) - 1u) << 3;
  if ((once & evs) != evs || (twice & evs)) return 0;
  if (ni == 0 && !(np == 1 || np == 2)) return 0;
  if (ni == 1)
    for (int t = 0; t < np; ++t)
      if (s.pa[t] != P && s.pb[t] != P) return 0;
  auto edge_of = [&](int w) -> int { return w - 3 < n0 ? 0 : w - 3 < n0 + n1 ? 1 : w - 3 < n0 + n1 + n2 ? 2 : -1; };
  int dir = 0;
  if (ni == 0 && np == 2) {
    int X[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int ea = edge_of(s.pa[c]), eb = edge_of(s.pb[c]);
      if (ea == eb) return -1;  // a chord with both ends on one edge
      X[c] = eb == (ea + 1) % 3 ? eb : ea;
    }
    if (X[0] == X[1]) {  // nested chords at corner X
      const int ein = (X[0] + 2) % 3, eout = X[0];
      int near = -1, best = -1;
      for (int c = 0; c < 2; ++c)
        for (int end = 0; end < 2; ++end) {
          const int w = end ? s.pb[c] : s.pa[c];
          if (edge_of(w) == ein && w > best) best = w, near = c;
        }
      dir = (edge_of(s.pa[near]) == ein && edge_of(s.pb[near]) == eout) ? 1 : 0;
    }
  }
  const int st = ni == 1 ? 1 : 0;
  const int cr0 = (st << 10) | (n0 << 7) | (n1 << 4) | (n2 << 1) | dir;
  const int cr1 = (st << 10) | (n1 << 7) | (n2 << 4) | (n0 << 1) | dir;
  const int cr2 = (st << 10) | (n2 << 7) | (n0 << 4) | (n1 << 1) | dir;
  int best = cr0, sigma = 0;
  if (cr1 < best) best = cr1, sigma = 1;
  if (cr2 < best) best = cr2, sigma = 2;
  for (int k = 0; k < NKEYS; ++k)
    if (g_keys.code[k] == best) {
      *sigma_out = sigma;
      return k + 1;
    }
  return -1;
}

// LIST: which list; REC: whether its cells come with the count pass's records.
// The block barriers order nothing (a group's data is its own warp's): they keep the
// warps of a block in the same part of this long kernel, so that they share what
// the instruction caches hold.  With blocks of two warps, each warp at a place of
// its own, 13 of 22 cycles per issue went to waiting for instructions: 527 us for the
// 1.9e5 cut cells of 4096^2 labels, 454 with four warps to a block, 425 with six, 404 with
// seven (the most whose groups fit 48 KB of shared memory; four blocks an SM).
constexpr int CELL_T = 224;
template <int G, int LIST, bool REC, int T>
__global__ void __launch_bounds__(T, 1024 / T) k_r3_cells(R3Args a) {
  constexpr int C_ = T / G;
  __shared__ R3State<G> sm[C_];
  const GLane<G> me;
  R3State<G>& s = sm[threadIdx.x / G];
  const u32 total = a.ncls[LIST];
  u32 ngc = 0, ngt = 0;
  for (u32 q = blockIdx.x * C_ + threadIdx.x / G;; q += gridDim.x * C_) {
    bool live = q < total;
    if (!__syncthreads_or(live)) break;
    u32 err = 0, c = 0;
    int cnt[3] = {0, 0, 0}, nb[3] = {-1, -1, -1}, ne, ni;
    u64 entry = 0;  // this lane's event or inside vertex
    auto put = [&](int v, double x, double y, u32 gid, int em) {
      bool ix, iy;
      s.vx[v] = x, s.vy[v] = y, s.X[v] = r3_fix36(x, &ix), s.Y[v] = r3_fix36(y, &iy);
      s.gid[v] = gid, s.c.em[v] = (unsigned char)em;
      if (v < 3) s.ix[v] = (unsigned char)((ix ? 1 : 0) | (iy ? 2 : 0));
    };
    if (REC) {
      const u64* r = a.rec + (live ? *r3_list(a, LIST, q) : 0u);
      if (live) {
        const u64 h0 = r[0], h1 = r[1], h2 = r[2];
        c = (u32)h0, nb[0] = (int)(u32)(h0 >> 32), nb[1] = (int)(u32)h1, nb[2] = (int)(u32)(h1 >> 32);
        cnt[0] = (int)(h2 & 255u), cnt[1] = (int)((h2 >> 8) & 255u), cnt[2] = (int)((h2 >> 16) & 255u);
        ni = (int)((h2 >> 24) & 255u);
      } else {
        ni = 0;
      }
      ne = cnt[0] + cnt[1] + cnt[2];
      if (live && me.l < ne + ni) entry = r[R3_HEAD + me.l];
    } else {
      c = live ? *r3_list(a, LIST, q) : 0u;
      const R3Cell C = r3_load_k(a, c);
      R3Geo2 S;
#pragma unroll
      for (int t = 0; t < 3; ++t) S.x[t] = r3_split(C.K[t].x), S.y[t] = r3_split(C.K[t].y);
      ne = r3_events<G>(a, C, S, live, me, s.F, cnt);
      ni = r3_inside_g<G>(a, C, S, live, me, s.F);
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (live && cnt[j] > 0) nb[j] = r3_neighbour(a, c, C, j);
      if (me.l < ne) {
        entry = r3_entry(s.F.jk[me.l] >> 2, s.F.jk[me.l] & 3, s.F.mk[me.l].x, s.F.mk[me.l].y);
      } else if (me.l < ne + ni) {
        const u32 cid = s.F.ins[me.l - ne];
        entry = r3_entry(3, 3, (int)(cid % (u32)(a.W + 1)), (int)(cid / (u32)(a.W + 1)));
      }
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (nb[j] == -2) err |= R3_GEOMETRY;
    }
    const int n = live ? 3 + ne + ni : 0;
    const u32 nt = live ? a.ntri[c] : 0u;
    // its offsets: the lanes add up the cut cells before it in its word
    u32 t0 = 0, e0 = 0, i0v = 0;
    if (live) {
      const u32 before = a.kmark[c >> 5] & ((1u << (c & 31)) - 1u);
#pragma unroll
      for (int b = 0; b < 32; b += G) {
        if (!((before >> (b + me.l)) & 1u)) continue;
        const u32 x = (c & ~31u) + (u32)(b + me.l);
        t0 += a.ntri[x] - 1u, e0 += a.nown[x], i0v += a.nin[x];
      }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      t0 += __shfl_xor_sync(0xffffffffu, t0, o), e0 += __shfl_xor_sync(0xffffffffu, e0, o);
      i0v += __shfl_xor_sync(0xffffffffu, i0v, o);
    }
    if (live) t0 += c + a.woff[0][c >> 5], e0 += a.nv + a.woff[1][c >> 5], i0v += a.nv + a.ne_total + a.woff[2][c >> 5];
    if (live && (n > G || (u32)(2 * ni + ne + 1) != nt)) err |= R3_COUNT;  // the count pass found others
    if (err) {
      if (me.l == 0) atomicOr(a.err, err);
      live = false;
    }
    // the corners
    if (live && me.l < 3) {
      const int k = me.l, id = a.ttri[3 * (u64)c + (u32)k];
      const double2 K = reinterpret_cast<const double2*>(a.txy)[id];
      put(k, K.x, K.y, (u32)id, (1 << k) | (1 << (k == 0 ? 2 : k - 1)));
    }
    // the events: one lane each (n <= G), with their position on their edge
    double ex = 0.0, ey = 0.0, es = 0.0;
    const int ej = (int)(entry >> 34), ekind = (int)(entry >> 32) & 3;
    const int2 emk = make_int2((int)(entry & 0xFFFFu), (int)((entry >> 16) & 0xFFFFu));
    bool fwd = true;
    const bool isev = live && me.l < ne;
    if (isev) s.tj[me.l] = (unsigned char)(ej << 2 | ekind), s.tmk[me.l] = emk;
    __syncwarp();
    if (isev) {
      const int w = ej == 2 ? 0 : ej + 1;
      fwd = (int)s.gid[ej] < (int)s.gid[w];
      const int pi = fwd ? ej : w, qi = fwd ? w : ej;
      const double2 P = make_double2(s.vx[pi], s.vy[pi]), Q = make_double2(s.vx[qi], s.vy[qi]);
      const double dx = dsb(Q.x, P.x), dy = dsb(Q.y, P.y);
      ex = (double)emk.x - 0.5, ey = (double)emk.y - 0.5;  // a corner; else one of the two from the other
      if (ekind != 2) {  // one division for either kind
        const bool v = ekind == 1;
        const double t = ddv(dml(v ? dsb(ex, P.x) : dsb(ey, P.y), v ? dy : dx), v ? dx : dy);
        if (v) ey = dad(P.y, t);
        else ex = dad(P.x, t);
      }
      const bool alongx = fabs(dx) >= fabs(dy);
      es = ddv(alongx ? dsb(ex, P.x) : dsb(ey, P.y), alongx ? dx : dy);
      s.s[me.l] = es;
    }
    __syncthreads();
    // rank on the edge by (s, kind, k, m); node order runs counter-clockwise
    int node = -1;
    u32 gid = 0;
    if (isev) {
      int r = 0;
      for (int t = 0; t < ne; ++t) {
        if (t == me.l || (s.tj[t] >> 2) != ej) continue;
        const double f = s.s[t];
        const int tk = s.tj[t] & 3;
        const int2 tm = s.tmk[t];
        r += (f != es ? f < es : tk != ekind ? tk < ekind : tm.y != emk.y ? tm.y < emk.y : tm.x < emk.x) ? 1 : 0;
      }
      const int own = ej == 0 ? cnt[0] : ej == 1 ? cnt[1] : cnt[2], other = ej == 0 ? nb[0] : ej == 1 ? nb[1] : nb[2];
      const int b0 = ej == 0 ? 0 : ej == 1 ? cnt[0] : cnt[0] + cnt[1];
      const int v = 3 + b0 + (fwd ? r : own - 1 - r);
      u32 base;
      if (other < 0 || (u32)other > c) {
        const u32 o3 = a.own3[c];
        base = e0 + (ej > 0 ? o3 & 255u : 0u) + (ej > 1 ? (o3 >> 8) & 255u : 0u) + (u32)r;
        reinterpret_cast<double2*>(a.xy)[base] = make_double2(ex, ey);
      } else {
        const int j2 = r3_edge_in(a, (u32)other, (int)s.gid[ej], (int)s.gid[ej == 2 ? 0 : ej + 1]);
        if (j2 < 0) err |= R3_GEOMETRY;
        base = r3_edge_base(a, (u32)other, max(j2, 0)) + (u32)r;
      }
      node = v, gid = base;
    }
    // inside vertices
    if (live && me.l >= ne && me.l < ne + ni) {
      ex = (double)emk.x - 0.5, ey = (double)emk.y - 0.5;
      node = 3 + me.l, gid = i0v + (u32)(me.l - ne);
      reinterpret_cast<double2*>(a.xy)[gid] = make_double2(ex, ey);
    }
    if (node >= 0) {
      put(node, ex, ey, gid, isev ? 1 << ej : 0);
      s.mk[node] = emk, s.kind[node] = (unsigned char)ekind;
    }
    if (me.ballot(err != 0)) {
      if (err) atomicOr(a.err, err);
      live = false;
    }
    __syncthreads();
    R3Corner Sx[3], Sy[3];
#pragma unroll
    for (int t = 0; t < 3; ++t)
      Sx[t] = R3Corner{s.X[t], (s.ix[t] & 1) != 0}, Sy[t] = R3Corner{s.Y[t], (s.ix[t] & 2) != 0};
    // the filter's frame
    float M = 0.0f;
    if (live && me.l < n) {
      const float fx = i64_float(s.X[me.l] - s.X[0], -36), fy = i64_float(s.Y[me.l] - s.Y[0], -36);
      s.c.f[me.l] = make_float2(fx, fy);
      M = fmaxf(fabsf(fx), fabsf(fy));
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    // pieces: horizontal lines by y, then vertical lines by x, one line per
    // lane: its nodes in order, and a piece between two consecutive ones when
    // the pixel edge at their middle is a boundary; lower label on the left
    int np = 0;
    {
      int f0[2], nl[2];
#pragma unroll
      for (int vert = 0; vert < 2; ++vert) {
        R3Corner lo = vert ? Sx[0] : Sy[0], hi = lo;
#pragma unroll
        for (int t = 1; t < 3; ++t) {
          const R3Corner v = vert ? Sx[t] : Sy[t];
          if (v.fx < lo.fx) lo = v;
          if (v.fx > hi.fx || (v.fx == hi.fx && v.inexact)) hi = v;
        }
        nl[vert] = live ? r3_lines(lo, hi, vert ? a.W : a.H, &f0[vert]) : 0;
      }
      const int lines = nl[0] + nl[1], most = warp_max(lines);
      for (int i0 = 0; i0 < most; i0 += G) {
        const int i = i0 + me.l;
        const bool on = i < lines, vert = on && i >= nl[0];
        const int line = on ? (vert ? f0[1] + i - nl[0] : f0[0] + i) : 0;
        int end[2] = {-1, -1}, nend = 0;
        u32 ins = 0;
        if (on) {
          bool lt[3], gt[3];
#pragma unroll
          for (int t = 0; t < 3; ++t) {
            const R3Corner v{vert ? Sx[t].fx : Sy[t].fx, vert ? Sx[t].inexact : Sy[t].inexact};
            lt[t] = r3_lt(v, line), gt[t] = r3_gt(v, line);
          }
#pragma unroll
          for (int t = 0; t < 3; ++t)
            if (!lt[t] && !gt[t]) {
              if (nend < 2) end[nend] = t;
              ++nend;
            }
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const int w = j == 2 ? 0 : j + 1;
            if (!((lt[j] && gt[w]) || (lt[w] && gt[j]))) continue;
            int node = -1;
            const int b0 = 3 + (j > 0 ? cnt[0] : 0) + (j > 1 ? cnt[1] : 0);
            for (int v = b0 + cnt[j] - 1; v >= b0; --v)  // the first in order
              if ((s.kind[v] == 2 || s.kind[v] == (vert ? 1 : 0)) && (vert ? s.mk[v].x : s.mk[v].y) == line) node = v;
            if (nend < 2) end[nend] = node;
            ++nend;
          }
          for (int v = 3 + ne; v < n; ++v)
            if ((vert ? s.mk[v].x : s.mk[v].y) == line) ins |= 1u << v;
          if (nend != 2) err |= R3_GEOMETRY, ins = 0, end[0] = end[1] = -1;
        }
        auto pos = [&](int v) { return vert ? s.vy[v] : s.vx[v]; };
        // the ends around the inside vertices (which lie strictly between)
        int lo = end[0], hi = end[1];
        if (lo >= 0 && hi >= 0) {
          if (pos(hi) < pos(lo)) lo = end[1], hi = end[0];
        } else if (ins && (lo >= 0 || hi >= 0)) {
          const int v = max(lo, hi);
          const bool before = pos(v) < pos(__ffs(ins) - 1);
          lo = before ? v : -1, hi = before ? -1 : v;
        }
        // counted, then written after the earlier lanes' pieces
        int at = 0, sum = 0;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
          int prev = lo, k = 0;
          u32 rest = ins;
          bool end = on && hi >= 0;
          while (rest || end) {
            int cur;
            if (rest) cur = __ffs(rest) - 1, rest &= rest - 1;
            else cur = hi, end = false;
            if (prev >= 0) {
              i64 j;
              r3_at_corner36(dml(dad(pos(prev), pos(cur)), 0.5), &j);  // at a corner: the pixel edge starting there
              // the pixels below or left of the line, and above or right of it
              const int l0 = r3_pixel(a, vert ? line - 1 : (int)j, vert ? (int)j : line - 1);
              const int l1 = r3_pixel(a, vert ? line : (int)j, vert ? (int)j : line);
              if (l0 != l1) {
                const bool f = vert ? l0 < l1 : l1 < l0;  // going +x the left side is above, going +y it is -x
                if (pass && at + k < 3 * G)
                  s.pa[at + k] = (unsigned char)(f ? prev : cur), s.pb[at + k] = (unsigned char)(f ? cur : prev);
                ++k;
              }
            }
            prev = cur;
          }
          if (pass == 0) {
            int before = k;
#pragma unroll
            for (int o = 1; o < G; o <<= 1) {
              const int t = __shfl_up_sync(0xffffffffu, before, o, G);
              if (me.l >= o) before += t;
            }
            sum = __shfl_sync(0xffffffffu, before, G - 1, G);
            at = np + before - k;
          }
        }
        np += sum;
      }
    }
    if (np + 3 + ne > 3 * G || np > R3_MAXP) err |= R3_CAPACITY;  // (no planar graph on n nodes has as many edges)
    if (me.ballot(err != 0)) {
      if (err) atomicOr(a.err, err);
      live = false;
    }
    __syncthreads();
    // Alg. 1 mask (a corner on a piece sets both its edges, an event its
    // edge, an edge on a boundary run its own bit, bit 0 an inside vertex)
    // and the (m, n) class of the first two pieces
    int mask = 0, klass = 0, key = -1, sigma = 0;
    if (live) {
      mask = ni > 0 ? 1 : 0;
      int pc0 = 0, pc1 = 0;
      for (int t = 0; t < np; ++t) {
        const int b = ((int)s.c.em[s.pa[t]] | (int)s.c.em[s.pb[t]]) << 1;
        mask |= b;
        if (t == 0) pc0 = __popc(b);
        if (t == 1) pc1 = __popc(b);
      }
      klass = np == 1 ? thm32_class(0, pc0) : np == 2 ? thm32_class(pc0, pc1) : 0;
#pragma unroll 1
      for (int e = 0; e < 6; ++e) {
        // edge j on the vertical or horizontal pixel line `line`: the pixel
        // edges (g - 1/2, g + 1/2) it has a stretch of
        const int j = e >> 1, vert = e & 1, w = j == 2 ? 0 : j + 1;
        const i64 *ac = vert ? s.X : s.Y, *al = vert ? s.Y : s.X;  // across the line, along it
        constexpr i64 HALF = 1ll << 35, ONE = 1ll << 36;
        if (((s.ix[j] | s.ix[w]) >> (vert ? 0 : 1)) & 1) continue;
        const i64 ca = ac[j];
        if (ca != ac[w] || (ca & (ONE - 1)) != HALF) continue;
        const int line = (int)(ca >> 36) + 1;
        const bool sw = al[w] < al[j];
        const i64 e0 = al[sw ? w : j], e1 = al[sw ? j : w];
        const int x1 = (s.ix[sw ? j : w] >> (vert ? 1 : 0)) & 1;
        // g + 1/2 > e0 and g - 1/2 < e1
        for (int g = (int)((e0 + HALF) >> 36); ((i64)g << 36) - HALF < e1 + x1; ++g)
          if (r3_pixel(a, vert ? line - 1 : g, vert ? g : line - 1) != r3_pixel(a, vert ? line : g, vert ? g : line))
            mask |= 2 << j;
      }
      key = r3_tier_t<G>(s, ni, ne, np, cnt[0], cnt[1], cnt[2], &sigma);
      if (key < 0) {
        if (me.l == 0) atomicOr(a.err, R3_GEOMETRY);
        live = false;
      }
    }
    int3* tri = reinterpret_cast<int3*>(a.tri);
    if (live && key > 0) {
      const unsigned long long w = g_keys.tris[(key - 1) * 3 + sigma];
      const unsigned short code = (unsigned short)((mask & 15) | (sigma << 4) | (key << 6) | (klass << 12));
      for (int k = me.l; k < (int)nt; k += G) {
        int q3[3];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int l = tri_label(w, k, u);
          q3[u] = l == 7 ? 3 + ne : l;
        }
        tri[t0 + k] = make_int3((int)s.gid[q3[0]], (int)s.gid[q3[1]], (int)s.gid[q3[2]]);
        a.label[t0 + k] = r3_node_label<G>(a, s, q3[0], q3[1], q3[2]);
        a.code[t0 + k] = code;
      }
    }
    // Tier-G
    const bool tg = live && key == 0;
    __syncthreads();
    if (!__any_sync(0xffffffffu, tg)) continue;
    // constraints: the pieces and the boundary cycle, each an edge as the
    // rule's list has it (above 12 nodes the smaller node first)
    if (tg) {
      const int v = me.l;
      if (v < n) {
        // the cycle's edge from node v to the next, and the one before
        int next = -1, prev = -1;
        if (v < 3) {
          const int own = v == 0 ? cnt[0] : v == 1 ? cnt[1] : cnt[2], b0 = 3 + (v > 0 ? cnt[0] : 0) + (v > 1 ? cnt[1] : 0);
          const int pk = v == 0 ? cnt[2] : v == 1 ? cnt[0] : cnt[1];
          next = own ? b0 : (v == 2 ? 0 : v + 1);
          prev = pk ? (v == 0 ? 2 + ne : b0 - 1) : (v == 0 ? 2 : v - 1);
        } else if (v < 3 + ne) {
          const int e = v - 3, k = e < cnt[0] ? 0 : e < cnt[0] + cnt[1] ? 1 : 2;
          const int b0 = k == 0 ? 0 : k == 1 ? cnt[0] : cnt[0] + cnt[1], own = k == 0 ? cnt[0] : k == 1 ? cnt[1] : cnt[2];
          next = e + 1 == b0 + own ? (k == 2 ? 0 : k + 1) : v + 1;
          prev = e == b0 ? k : v - 1;
        }
        s.c.adj[v] = next >= 0 ? (1u << next) | (1u << prev) : 0u;
        if (next >= 0) {
          const bool sw = n > 12 && next < v;
          s.c.ce[np + v] = (unsigned short)(sw ? (next << 8) | v : (v << 8) | next);
        }
      }
      if (me.l == 0) s.c.nce = np + 3 + ne;
    }
    __syncwarp();
    if (tg)
      for (int t = me.l; t < np; t += G) {
        const int p = s.pa[t], r = s.pb[t];
        const bool sw = n > 12 && r < p;
        s.c.ce[t] = (unsigned short)(sw ? (r << 8) | p : (p << 8) | r);
        atomicOr(&s.c.adj[p], 1u << r);
        atomicOr(&s.c.adj[r], 1u << p);
      }
    __syncwarp();
    const R3Geo<G> geo{&s, 80.0f * 5.9604645e-8f * M * M * 1.0001f + 16.0f * 2.910383e-11f * M};
    g_greedy<G, true>(s.c, geo, tg ? n : 0);
    if (tg) {
      const int nf = (int)s.c.nface;
      if ((u32)nf != nt) {
        if (me.l == 0) atomicOr(a.err, R3_COUNT);
      } else {
        const unsigned short code = (unsigned short)((mask & 15) | (63 << 6) | (klass << 12));
        if (me.l == 0) ++ngc, ngt += (u32)nf;
        for (int k = me.l; k < nf; k += G) {
          const u32 f = s.c.face[k];
          u32 r = 0;
          for (int j = 0; j < nf; ++j) r += s.c.face[j] < f ? 1u : 0u;
          const int p = (int)(f >> 16), u = (int)((f >> 8) & 255u), w = (int)(f & 255u);
          tri[t0 + r] = make_int3((int)s.gid[p], (int)s.gid[u], (int)s.gid[w]);
          a.label[t0 + r] = r3_node_label<G>(a, s, p, u, w);
          a.code[t0 + r] = code;
        }
      }
    }
    __syncwarp();
  }
  // the counts, one atomic per warp
  ngc = __reduce_add_sync(0xffffffffu, ngc), ngt = __reduce_add_sync(0xffffffffu, ngt);
  if (me.lane == 0 && ngc) atomicAdd(a.ng, ngc), atomicAdd(a.ngtri, ngt);
}

// ---------------------------------------------------------------------------
// Cells of more than 32 nodes (all Tier-G): one warp each.  Lane 0 builds the
// cell's boundary graph in shared memory; the warp ranks the candidate pairs, runs the greedy pass
// (each candidate tested by the lanes against the nodes and the kept
// edges), lists the faces and writes them in sorted order.
// ---------------------------------------------------------------------------
constexpr int R3G_WARPS = 2;
constexpr int R3G_MAXC = R3_MAXN * (R3_MAXN - 1) / 2;
constexpr int R3G_MAXE = 3 * R3_MAXN;  // kept edges of a triangulation of n points
constexpr int R3G_MAXF = 2 * R3_MAXN;

struct R3GShared {
  R3Local L;
  R3Ev ev[3][R3_MAXE];
  float key[R3G_MAXC];
  unsigned short cand[R3G_MAXC], sorted[R3G_MAXC];
  unsigned long long adj[R3_MAXN];
  unsigned char ea[R3G_MAXE], eb[R3G_MAXE];
  int face[R3G_MAXF];
  int ncand, nedge, nface;
  u32 err;
};
struct R3SharedEv {
  R3Ev (*e)[R3_MAXE];
  SBMT_DEV R3Ev* operator[](int j) { return e[j]; }
};

__global__ void __launch_bounds__(32 * R3G_WARPS) k_r3_tierg(R3Args a) {
  __shared__ R3GShared sh[R3G_WARPS];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  R3GShared& S = sh[wid];
  const u32 ng = a.ncls[3];
  for (u32 g = blockIdx.x * R3G_WARPS + wid; g < ng; g += gridDim.x * R3G_WARPS) {
    const u32 c = *r3_list(a, 3, g);
    if (lane == 0) {
      const R3Cell C = r3_load(a, c);
      R3SharedEv ev{S.ev};
      S.err = r3_build(a, c, C, S.L, ev, true);
    }
    __syncwarp();
    if (S.err) {
      if (lane == 0) atomicOr(a.err, S.err);
      __syncwarp();
      continue;
    }
    const R3Local& L = S.L;
    const int n = L.n;
    // constraints: the cell's boundary cycle and the pieces
    if (lane == 0) {
      for (int w = 0; w < n; ++w) S.adj[w] = 0;
      S.nedge = 0;
      auto add = [&](int p, int q) {
        if ((S.adj[p] >> q) & 1ull) return;
        S.adj[p] |= 1ull << q, S.adj[q] |= 1ull << p;
        const int lo = p < q ? p : q, hi = p < q ? q : p;
        S.ea[S.nedge] = (unsigned char)lo, S.eb[S.nedge] = (unsigned char)hi;
        ++S.nedge;
      };
      for (int t = 0; t < L.np; ++t) add(L.pa[t], L.pb[t]);
      int cyc[R3_MAXN], nc = 0, b = 3;
      for (int j = 0; j < 3; ++j) {
        cyc[nc++] = j;
        for (int t = 0; t < L.nev[j]; ++t) cyc[nc++] = b + t;
        b += L.nev[j];
      }
      for (int t = 0; t < nc; ++t) add(cyc[t], cyc[t + 1 == nc ? 0 : t + 1]);
      S.ncand = 0;
    }
    __syncwarp();
    // candidate pairs, keyed by squared length rounded to single precision
    for (int p0 = 0; p0 < n * n; p0 += 32) {
      const int p = p0 + lane, u = p / n, w = p % n;
      bool ok = p < n * n && u < w && !((S.adj[u] >> w) & 1ull) && (L.on_edge[u] & L.on_edge[w]) == 0;
      const unsigned m = __ballot_sync(0xFFFFFFFFu, ok);
      int base = 0;
      if (lane == 0) base = S.ncand, S.ncand += __popc(m);
      base = __shfl_sync(0xFFFFFFFFu, base, 0);
      if (ok) {
        const int slot = base + __popc(m & ((1u << lane) - 1u));
        const double dx = dsb(L.v[w].x, L.v[u].x), dy = dsb(L.v[w].y, L.v[u].y);
        S.key[slot] = __double2float_rn(dad(dml(dx, dx), dml(dy, dy)));
        S.cand[slot] = (unsigned short)(u * R3_MAXN + w);
      }
      __syncwarp();
    }
    const int ncand = S.ncand;
    // rank each candidate among all by (key, u, w)
    for (int i = lane; i < ncand; i += 32) {
      const float ki = S.key[i];
      const unsigned short ci = S.cand[i];
      int r = 0;
      for (int k = 0; k < ncand; ++k) {
        const float kk = S.key[k];
        r += (kk < ki || (kk == ki && S.cand[k] < ci)) ? 1 : 0;
      }
      S.sorted[r] = ci;
    }
    __syncwarp();
    // greedy pass
    for (int r = 0; r < ncand; ++r) {
      const int u = S.sorted[r] / R3_MAXN, w = S.sorted[r] % R3_MAXN;
      const double2 pu = L.v[u], pw = L.v[w];
      const double ex = dsb(pw.x, pu.x), ey = dsb(pw.y, pu.y), len2 = dad(dml(ex, ex), dml(ey, ey));
      bool bad = false;
      for (int k = lane; k < n; k += 32) {
        if (k == u || k == w || r3_orient(pu, pw, L.v[k]) != 0.0) continue;
        const double t = dad(dml(dsb(L.v[k].x, pu.x), ex), dml(dsb(L.v[k].y, pu.y), ey));
        if (t > 0.0 && t < len2) bad = true;
      }
      const int ne = min(S.nedge, R3G_MAXE);
      for (int t = lane; t < ne && !bad; t += 32) {
        const int p = S.ea[t], q = S.eb[t];
        if (p == u || p == w || q == u || q == w) continue;
        const int o1 = r3_sgn(r3_orient(pu, pw, L.v[p])), o2 = r3_sgn(r3_orient(pu, pw, L.v[q]));
        const int o3 = r3_sgn(r3_orient(L.v[p], L.v[q], pu)), o4 = r3_sgn(r3_orient(L.v[p], L.v[q], pw));
        if (o1 * o2 < 0 && o3 * o4 < 0) bad = true;
      }
      if (__any_sync(0xFFFFFFFFu, bad)) continue;
      if (lane == 0) {
        if (S.nedge < R3G_MAXE) {
          S.adj[u] |= 1ull << w, S.adj[w] |= 1ull << u;
          S.ea[S.nedge] = (unsigned char)u, S.eb[S.nedge] = (unsigned char)w;
        }
        ++S.nedge;
      }
      __syncwarp();
    }
    if (S.nedge > R3G_MAXE) {
      if (lane == 0) atomicOr(a.err, R3_CAPACITY);
      __syncwarp();
      continue;
    }
    // faces: 3-cycles with no node inside, smallest index first, CCW
    if (lane == 0) S.nface = 0;
    __syncwarp();
    for (int p = lane; p < n; p += 32) {
      unsigned long long mb = S.adj[p] & ~((2ull << p) - 1ull);
      while (mb) {
        const int q = __ffsll((long long)mb) - 1;
        mb &= mb - 1;
        unsigned long long mc = S.adj[p] & S.adj[q] & ~((2ull << q) - 1ull);
        while (mc) {
          const int r = __ffsll((long long)mc) - 1;
          mc &= mc - 1;
          const int o = r3_sgn(r3_orient(L.v[p], L.v[q], L.v[r]));
          if (o == 0) continue;
          bool empty = true;
          for (int k = 0; k < n && empty; ++k) {
            if (k == p || k == q || k == r) continue;
            if (r3_sgn(r3_orient(L.v[p], L.v[q], L.v[k])) == o && r3_sgn(r3_orient(L.v[q], L.v[r], L.v[k])) == o &&
                r3_sgn(r3_orient(L.v[r], L.v[p], L.v[k])) == o)
              empty = false;
          }
          if (!empty) continue;
          const int f = o > 0 ? (p << 12 | q << 6 | r) : (p << 12 | r << 6 | q);
          const int slot = atomicAdd(&S.nface, 1);
          if (slot < R3G_MAXF) S.face[slot] = f;
        }
      }
    }
    __syncwarp();
    const int nf = S.nface;
    const u32 t0 = r3_toff(a, c);
    if (nf != (int)a.ntri[c]) {
      if (lane == 0) atomicOr(a.err, R3_COUNT);
      __syncwarp();
      continue;
    }
    const unsigned short code = (unsigned short)((L.mask & 15) | (63 << 6) | (L.klass << 12));
    if (lane == 0) atomicAdd(a.ngtri, (u32)nf), atomicAdd(a.ng, 1u);
    int3* tri = reinterpret_cast<int3*>(a.tri);
    for (int i = lane; i < nf; i += 32) {
      const int f = S.face[i];
      int r = 0;
      for (int k = 0; k < nf; ++k) r += S.face[k] < f ? 1 : 0;
      const int p = f >> 12, q = (f >> 6) & 63, s = f & 63;
      tri[t0 + r] = make_int3((int)L.gid[p], (int)L.gid[q], (int)L.gid[s]);
      a.label[t0 + r] = r3_label(a, L.v[p], L.v[q], L.v[s]);
      a.code[t0 + r] = code;
    }
    __syncwarp();
  }
}

}  // namespace

int launch_r3_count(const R3Args& a, cudaStream_t st) {
  const unsigned g = (unsigned)std::min<u64>((a.nt + 255) / 256, 152 * 16);
  k_r3_screen<<<std::max(g, 1u), 256, 0, st>>>(a);
  k_r3_link<<<152 * 8, 256, 0, st>>>(a);
  k_r3_count<<<152 * 16, 128, 0, st>>>(a);
  return 3;
}

int launch_r3_emit(const R3Args& a, cudaStream_t st) {
  const unsigned g = (unsigned)std::min<u64>((a.nt + 255) / 256, 152 * 16);
  k_r3_emit_uncut<<<std::max(g, 1u), 256, 0, st>>>(a);
  k_r3_tierg<<<152 * 8, 32 * R3G_WARPS, 0, st>>>(a);
  k_r3_cells<32, 4, false, 64><<<152 * 5, 64, 0, st>>>(a);
  k_r3_cells<32, 2, true, 64><<<152 * 5, 64, 0, st>>>(a);
  k_r3_cells<16, 1, true, 64><<<152 * 10, 64, 0, st>>>(a);
  k_r3_cells<8, 0, true, CELL_T><<<152 * (1024 / CELL_T), CELL_T, 0, st>>>(a);
  return 6;
}

}  // namespace sbmt
