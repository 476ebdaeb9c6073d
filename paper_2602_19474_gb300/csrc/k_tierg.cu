// k_tierg.cu -- K4-G: cells outside the regime of Lemma 3.1 ("Tier-G").
//
// At grid edges h of a few pixels the pixel staircase puts several boundary
// vertices, or several chords, into one base triangle, outside the paper's
// finite table (Lemma 3.1 needs segments longer than the grid edge,
// Sec. 3.2).  Such a cell is triangulated by a deterministic Steiner-free
// rule: its local boundary graph (the cell's boundary split at the crossing
// events, plus the pieces of boundary segments inside it) is completed
// greedily -- every other vertex pair in order of exact squared length, ties
// by local index pair, kept when its open segment holds no vertex and crosses
// no kept edge.  A maximal plane straight-line graph on a point set
// triangulates its convex hull, so the result tiles the cell and embeds every
// boundary piece.  The faces are the 3-cycles with no vertex inside, listed
// with the smallest local index first, counter-clockwise, in sorted order.
//
// The cells are first ordered by vertex count, largest first.  A cell of at
// most 32 vertices is taken by a group of 8, 16 or 32 lanes, the least that
// has a lane per vertex (sbmt_greedy.cuh); the lanes gather its pairs and
// events side by side too, and write its triangles.  Larger cells (up to 64
// vertices) run one warp each on vertex lists.  A thread per cell (up to 9
// vertices), and a warp whose first lane gathers (above that), were bound by
// the latency of one lane's chain of loads, exact tests and local memory.
// Measured before and now, kernels alone: one 64^2 bitmap, a few cells, 81 and
// 24 us; 2.3e5 cells of at most 9 vertices (8192^2 labels, h = 2) 345 and 335
// us; ten noise bitmaps of 256 to 4096 px at h = 2, 4 and 8, by size 307 and
// 247, 1313 and 272, 239 and 82 us.
#include "sbmt_cell.cuh"
#include "sbmt_greedy.cuh"
#include "sbmt_launch.h"

namespace sbmt {

namespace {

constexpr int TN = TIERG_TN;  // up to this many vertices: 8 lanes a cell
constexpr int TM = TIERG_WN;  // up to this many: 16 lanes
constexpr int TL = 32;        // up to this many: a warp with a lane per vertex
constexpr int WN = 64;        // a warp on vertex lists
constexpr int NSIZE = TIERG_SIZES;  // sizes 0 .. TM, then TM + 1 .. TL pooled, then above TL
constexpr int WWARPS = 4;
constexpr int TG_OCC = 12;  // blocks of 64 threads an SM (80 registers): 8 took 452 us where 12 took 391
constexpr int GORDER_W = 8;  // ordering kernel: cell buckets (warps) per block

SBMT_DEV constexpr int pow2_at_least(int x) {
  int m = 1;
  while (m < x) m <<= 1;
  return m;
}

// The state of one Tier-G cell above TL vertices, in shared memory, with the
// kept edges listed.  Cell-local coordinates keep full 32-bit components: a
// value near the cell can have components of order the image size (a point on
// a slanted grid edge has x = a + b sqrt3 with both large).
template <int N>
struct GStore {
  static constexpr int NCAND = N * (N - 1) / 2;
  static constexpr int NCANDP = pow2_at_least(NCAND);
  int xa[N], xb[N], ya[N], yb[N];  // cell-local exact coordinates (a + b sqrt3)
  u32 gid[N];
  u32 ref[N];  // event index (events) or pixel-corner id (inside vertices) while building
  u64 adj[N];
  unsigned short edge[3 * N];   // kept edges
  unsigned short cand[NCANDP];  // candidate order
  u32 tri[2 * N];
  float fx[N], fy[N];  // the values rounded once from double, for the fast filters
  unsigned char em[N];  // the cell edges a vertex lies on (bit k: edge k)
  int n, nev, nedge, ntri, ok;
};
template <int N>
SBMT_DEV float sfx(const GStore<N>& s, int k) {
  return s.fx[k];
}
template <int N>
SBMT_DEV float sfy(const GStore<N>& s, int k) {
  return s.fy[k];
}

template <int N>
SBMT_DEV Pq lpt(const GStore<N>& s, int k) {
  return Pq{zq(s.xa[k], s.xb[k]), zq(s.ya[k], s.yb[k])};
}
template <int N>
SBMT_DEV Zq len2(const GStore<N>& s, int u, int v) {
  const Zq dx = zq((i64)s.xa[v] - s.xa[u], (i64)s.xb[v] - s.xb[u]);
  const Zq dy = zq((i64)s.ya[v] - s.ya[u], (i64)s.yb[v] - s.yb[u]);
  return dx * dx + dy * dy;
}
// candidate order: exact squared length, then the packed pair (u << 8 | v)
template <int N>
SBMT_DEV bool cand_less(const GStore<N>& s, unsigned short x, unsigned short y) {
  if (x == 0xFFFFu) return false;
  if (y == 0xFFFFu) return true;
  const int c = zcmp(len2(s, x >> 8, x & 255), len2(s, y >> 8, y & 255));
  if (c != 0) return c < 0;
  return x < y;
}
SBMT_DEV Zq dot3(const Pq& o, const Pq& p, const Pq& q) {
  return (p.x - o.x) * (q.x - o.x) + (p.y - o.y) * (q.y - o.y);
}

// Same order as cand_less, decided in single precision when the two lengths
// are far apart and exactly otherwise.  Coordinates are rounded from their
// exact values (error below |coordinate| 2^-24), so a key's error stays far
// below tol for cells of extent E (scaled units).
template <int N>
SBMT_DEV bool cand_less_fast(const GStore<N>& s, unsigned short x, unsigned short y, float tolc) {
  const int xu = x >> 8, xv = x & 255, yu = y >> 8, yv = y & 255;
  const float dx0 = sfx(s, xv) - sfx(s, xu), dy0 = sfy(s, xv) - sfy(s, xu);
  const float dx1 = sfx(s, yv) - sfx(s, yu), dy1 = sfy(s, yv) - sfy(s, yu);
  const float kx = dx0 * dx0 + dy0 * dy0, ky = dx1 * dx1 + dy1 * dy1;
  const float tol = 1e-5f * (kx + ky) + tolc;
  if (kx < ky - tol) return true;
  if (kx > ky + tol) return false;
  return cand_less(s, x, y);
}

// cand_less_fast with the sort's padding entries (0xFFFF) last
template <int N>
SBMT_DEV bool cand_less_sent(const GStore<N>& s, unsigned short x, unsigned short y, float tolc) {
  if (x == 0xFFFFu) return false;
  if (y == 0xFFFFu) return true;
  return cand_less_fast(s, x, y, tolc);
}

SBMT_DEV void prefetch_l1(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// Build the local boundary graph (one thread): corners A, B, C; the events
// on AB, BC, CA in counter-clockwise order; the inside vertices by pixel-
// corner id; constraint edges = boundary cycle + one piece per pair.
template <int N>
SBMT_DEV void build_local(const GridP& g, const CellGeo& cg, const CutRec& rec, const Pair* P, const Seg* segs,
                          const Event* ev, GStore<N>& s) {
  s.ok = 0;
  s.nedge = 0;
  const Pq A = lattice_pt(g, cg.ci[0], cg.cj[0]);
  for (int k = 0; k < 3; ++k) {
    const Pq p = lattice_pt(g, cg.ci[k], cg.cj[k]);
    s.xa[k] = (int)(p.x.a - A.x.a), s.xb[k] = (int)(p.x.b - A.x.b);
    s.ya[k] = (int)(p.y.a - A.y.a), s.yb[k] = (int)(p.y.b - A.y.b);
    s.gid[k] = vid(g, cg.ci[k], cg.cj[k]);
    s.ref[k] = NONE;
  }
  // events: gather once, keyed by (local edge, counter-clockwise position)
  int ne = 0;
  int ek[N];
  for (u32 k = 0; k < rec.npairs; ++k) {
    const Pair pr = P[k];
    for (int end = 0; end < 2; ++end) {
      const u32 e = end == 0 ? pr.ev_in : pr.ev_out;
      if (e == NONE) continue;
      if (3 + ne >= N) return;
      const Event x = ev[e];
      const int le = local_edge(cg, x.edge);
      if (le < 0) return;
      const int t = 3 + ne;
      s.ref[t] = e, ek[t] = le, s.gid[t] = x.gid;
      s.xa[t] = (int)(x.xa - A.x.a), s.xb[t] = (int)(x.xb - A.x.b);
      s.ya[t] = (int)(x.ya - A.y.a), s.yb[t] = (int)(x.yb - A.y.b);
      ++ne;
    }
  }
  for (int a = 4; a < 3 + ne; ++a)
    for (int b = a; b > 3; --b) {
      const Zq pb = ccw_pos_xy(cg.down, ek[b], zq(s.xa[b], s.xb[b]), zq(s.ya[b], s.yb[b]));
      const Zq pa = ccw_pos_xy(cg.down, ek[b - 1], zq(s.xa[b - 1], s.xb[b - 1]), zq(s.ya[b - 1], s.yb[b - 1]));
      if (!(ek[b] < ek[b - 1] || (ek[b] == ek[b - 1] && zcmp(pb, pa) < 0))) break;
      int ti = ek[b];
      ek[b] = ek[b - 1], ek[b - 1] = ti;
      u32 tu = s.ref[b];
      s.ref[b] = s.ref[b - 1], s.ref[b - 1] = tu;
      tu = s.gid[b], s.gid[b] = s.gid[b - 1], s.gid[b - 1] = tu;
      ti = s.xa[b], s.xa[b] = s.xa[b - 1], s.xa[b - 1] = ti;
      ti = s.xb[b], s.xb[b] = s.xb[b - 1], s.xb[b - 1] = ti;
      ti = s.ya[b], s.ya[b] = s.ya[b - 1], s.ya[b - 1] = ti;
      ti = s.yb[b], s.yb[b] = s.yb[b - 1], s.yb[b - 1] = ti;
    }
  int nev[3] = {0, 0, 0};
  for (int t = 3; t < 3 + ne; ++t) nev[ek[t]]++;
  // inside vertices: distinct pixel-corner ids, ascending
  int n = 3 + ne;
  for (u32 k = 0; k < rec.npairs; ++k) {
    const Pair pr = P[k];
    if (pr.ev_in != NONE && pr.ev_out != NONE) continue;
    const Seg sg = segs[pr.seg];
    for (int end = 0; end < 2; ++end) {
      if ((end == 0 ? pr.ev_in : pr.ev_out) != NONE) continue;
      const u32 id = corner_id(g, sg, end);
      int pos = 3 + ne;
      while (pos < n && s.ref[pos] < id) ++pos;
      if (pos < n && s.ref[pos] == id) continue;
      if (n >= N) return;
      for (int t = n; t > pos; --t) s.ref[t] = s.ref[t - 1];
      s.ref[pos] = id;
      ++n;
    }
  }
  if ((u32)(n - 3 - ne) != rec.nchain) return;
  for (int k = 3 + ne; k < n; ++k) {
    const Pq p = corner_of_id(g, s.ref[k]);
    s.xa[k] = (int)(p.x.a - A.x.a), s.xb[k] = (int)(p.x.b - A.x.b);
    s.ya[k] = (int)(p.y.a - A.y.a), s.yb[k] = (int)(p.y.b - A.y.b);
    s.gid[k] = rec.chain_base + (u32)(k - 3 - ne);
  }
  s.n = n, s.nev = ne;
  for (int k = 0; k < n; ++k) {
    s.em[k] = k < 3 ? (unsigned char)((1 << k) | (1 << (k == 0 ? 2 : k - 1))) : k < 3 + ne ? (unsigned char)(1 << ek[k]) : 0;
    s.adj[k] = 0;
    s.fx[k] = (float)zdouble(zq(s.xa[k], s.xb[k]));
    s.fy[k] = (float)zdouble(zq(s.ya[k], s.yb[k]));
  }
  bool room = true;
  auto add_edge = [&](int u, int v) {
    if (u > v) {
      const int t = u;
      u = v, v = t;
    }
    if ((s.adj[u] >> v) & 1ull) return;
    if (s.nedge >= 3 * N) {
      room = false;
      return;
    }
    s.adj[u] |= 1ull << v, s.adj[v] |= 1ull << u;
    s.edge[s.nedge] = (unsigned short)((u << 8) | v);
    ++s.nedge;
  };
  {  // boundary cycle A, events on AB, B, events on BC, C, events on CA
    int prev = 0, e = 3, first = 0;
    for (int k = 0; k < 3; ++k) {
      if (k) add_edge(prev, k), prev = k;
      for (int t = 0; t < nev[k]; ++t) add_edge(prev, e), prev = e++;
    }
    add_edge(prev, first);
  }
  for (u32 k = 0; k < rec.npairs; ++k) {  // boundary pieces
    const Pair pr = P[k];
    int loc[2] = {-1, -1};
    for (int end = 0; end < 2; ++end) {
      const u32 e = end == 0 ? pr.ev_in : pr.ev_out;
      if (e != NONE) {
        for (int t = 3; t < 3 + ne; ++t)
          if (s.ref[t] == e) loc[end] = t;
      } else {
        const u32 id = corner_id(g, segs[pr.seg], end);
        for (int t = 3 + ne; t < n; ++t)
          if (s.ref[t] == id) loc[end] = t;
      }
    }
    if (loc[0] < 0 || loc[1] < 0) return;
    add_edge(loc[0], loc[1]);
  }
  s.ok = room ? 1 : 0;
}

// The greedy completion and face listing by a warp.
template <int N, class O>
SBMT_DEV void greedy_faces(GStore<N>& s, int lane, int nb, const O& ori, float tolc) {
  const int n = s.n;
  // candidate pairs not joined by a constraint edge
  int m = 0;
    for (int u = 0; u < n; ++u)
      for (int vb = u + 1; vb < n; vb += 32) {
        const int v = vb + lane;
        // a pair on one cell edge that is not a cycle edge has a vertex
        // between its ends and is always rejected: left out
        const bool ok = v < n && !((s.adj[u] >> v) & 1ull) && !(s.em[u] & s.em[v]);
        const u32 bal = __ballot_sync(0xffffffffu, ok);
        if (ok) s.cand[m + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)((u << 8) | v);
        m += __popc(bal);
      }
    int M = 1;
    while (M < m) M <<= 1;
    for (int k = m + lane; k < M; k += 32) s.cand[k] = 0xFFFFu;
    __syncwarp();
    for (int kk = 2; kk <= M; kk <<= 1)
      for (int jj = kk >> 1; jj > 0; jj >>= 1) {
        for (int i = lane; i < M; i += 32) {
          const int l = i ^ jj;
          if (l > i) {
            const unsigned short x = s.cand[i], y = s.cand[l];
            const bool up = (i & kk) == 0;
            if (up ? cand_less_sent(s, y, x, tolc) : cand_less_sent(s, x, y, tolc)) s.cand[i] = y, s.cand[l] = x;
          }
        }
        __syncwarp();
      }
  // keep a pair when its open segment holds no vertex and crosses no kept edge
  const int max_edges = 3 * n - nb - 3;
  for (int ci = 0; ci < m && s.nedge < max_edges; ++ci) {
    const int u = s.cand[ci] >> 8, v = s.cand[ci] & 255;
    bool bad = false;
    for (int k = lane; k < n && !bad; k += 32) {
      if (k == u || k == v || ori(u, v, k) != 0) continue;
      const Pq pu = lpt(s, u), pv = lpt(s, v), pk = lpt(s, k);
      if (zsign(dot3(pu, pv, pk)) > 0 && zsign(dot3(pv, pu, pk)) > 0) bad = true;
    }
    const int ned = s.nedge;
    for (int k = lane; k < ned && !bad; k += 32) {
      const int a = s.edge[k] >> 8, b = s.edge[k] & 255;
      if (a == u || a == v || b == u || b == v) continue;
      const int o1 = ori(u, v, a), o2 = ori(u, v, b);
      if (o1 * o2 >= 0) continue;
      const int o3 = ori(a, b, u), o4 = ori(a, b, v);
      if (o3 * o4 < 0) bad = true;
    }
    if (!__any_sync(0xffffffffu, bad) && lane == 0) {
      s.adj[u] |= 1ull << v, s.adj[v] |= 1ull << u;
      s.edge[s.nedge] = (unsigned short)((u << 8) | v);
      s.nedge = s.nedge + 1;
    }
    __syncwarp();
  }
  // faces: 3-cycles with no vertex strictly inside
  if (lane == 0) s.ntri = 0;
  __syncwarp();
  for (int u = lane; u < n; u += 32) {
    for (u64 vs = s.adj[u] & ~((2ull << u) - 1ull); vs; vs &= vs - 1) {
      const int v = __ffsll((long long)vs) - 1;
      for (u64 ws = s.adj[u] & s.adj[v] & ~((2ull << v) - 1ull); ws; ws &= ws - 1) {
        const int x = __ffsll((long long)ws) - 1;
        const int o = ori(u, v, x);
        if (o == 0) continue;
        bool empty = true;
        for (int k = 0; k < n && empty; ++k) {
          if (k == u || k == v || k == x) continue;
          if (ori(u, v, k) == o && ori(v, x, k) == o && ori(x, u, k) == o) empty = false;
        }
        if (!empty) continue;
        const int slot = atomicAdd(&s.ntri, 1);
        if (slot < 2 * N)
          s.tri[slot] = o > 0 ? ((u32)u << 16 | (u32)v << 8 | (u32)x) : ((u32)u << 16 | (u32)x << 8 | (u32)v);
      }
    }
  }
  __syncwarp();
  const int nt = min(s.ntri, 2 * N);
    // by rank, the lanes together: the keys are distinct (each face once)
    constexpr int R = (2 * N + 31) / 32;
    u32 key[R];
    int rank[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int k = lane + q * 32;
      key[q] = k < nt ? s.tri[k] : 0u;
      rank[q] = 0;
      if (k < nt)
        for (int j = 0; j < nt; ++j) rank[q] += s.tri[j] < key[q] ? 1 : 0;
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < R; ++q)
      if (lane + q * 32 < nt) s.tri[rank[q]] = key[q];
  __syncwarp();
}

template <int N>
SBMT_DEV int ori_filtered(const GStore<N>& s, int a, int b, int c, float tol) {
  const float fxa = sfx(s, a), fya = sfy(s, a);
  const float dx1 = sfx(s, b) - fxa, dy1 = sfy(s, b) - fya;
  const float dx2 = sfx(s, c) - fxa, dy2 = sfy(s, c) - fya;
  const float d = dx1 * dy2 - dy1 * dx2;
  if (d > tol) return 1;
  if (d < -tol) return -1;
  // three points of one cell edge (an exact line) need no exact test
  if (s.em[a] & s.em[b] & s.em[c]) return 0;
  return orient3(lpt(s, a), lpt(s, b), lpt(s, c));
}

// orientation decided in single precision when clear, exactly otherwise
template <int N>
struct OriFiltered {
  const GStore<N>* s;
  float tol;
  SBMT_DEV int operator()(int u, int v, int w) const { return ori_filtered(*s, u, v, w, tol); }
};

template <int N>
SBMT_DEV void write_patch(const GridP& g, const unsigned char* img, i64 pitch, int dtype, const CellGeo& cg,
                          const CutRec& rec, const GStore<N>& s, int lane, int* tri, unsigned short* label,
                          unsigned short* code, double* xy, u32 xy0, u32* err) {
  const Pq A = lattice_pt(g, cg.ci[0], cg.cj[0]);
  const int nt = min(s.ntri, 2 * N);
  if (lane == 0 && (u32)s.ntri != rec.ntri) atomicOr(err, ERR_COUNT);
  const unsigned short cd = (unsigned short)(rec.code & 0xFFFFu);
  for (int k = lane; k < nt && k < (int)rec.ntri; k += 32) {
    const int a = (int)(s.tri[k] >> 16), b = (int)((s.tri[k] >> 8) & 255u), c = (int)(s.tri[k] & 255u);
    const u32 o = rec.tri_off + (u32)k;
    tri[3 * (i64)o] = (int)s.gid[a];
    tri[3 * (i64)o + 1] = (int)s.gid[b];
    tri[3 * (i64)o + 2] = (int)s.gid[c];
    const Pq pa = lpt(s, a), pb = lpt(s, b), pc = lpt(s, c);
    label[o] = label_of(g, img, pitch, dtype, Pq{pa.x + A.x, pa.y + A.y}, Pq{pb.x + A.x, pb.y + A.y},
                        Pq{pc.x + A.x, pc.y + A.y});
    code[o] = cd;
  }
  // coordinates of the cell's inside vertices
  const int nin = (int)rec.nchain;
  const double invS = g.invS;
  for (int k = lane; k < nin; k += 32) {
    const int loc = s.n - nin + k;
    double2 v;
    v.x = zdouble(zq((i64)s.xa[loc] + A.x.a, (i64)s.xb[loc] + A.x.b)) * invS;
    v.y = zdouble(zq((i64)s.ya[loc] + A.y.a, (i64)s.yb[loc] + A.y.b)) * invS;
    reinterpret_cast<double2*>(xy)[s.gid[loc] - xy0] = v;
  }
}

// the number of local vertices of a Tier-G cell: ntri = 2 n_in + n_b - 2
SBMT_DEV int local_count(const CutRec& rec) { return (int)(rec.ntri + 2 - rec.nchain); }
SBMT_DEV int boundary_count(const CutRec& rec) { return (int)(rec.ntri + 2 - 2 * rec.nchain); }

// Tier-G cells of the whole batch ordered by local vertex count, largest
// first within each list, so that the groups of a warp run cells of one size.
// bd->gcnt[n] holds the batch's number of Tier-G cells with n vertices (those
// above TM pooled: TM + 1 .. TL, then above TL).  The cells of at most TM vertices
// form one order: those above TN run 16 lanes each (slist), the others 8
// (olist).  Cells of TM + 1 .. TL vertices go to wlist from its front, those
// above TL from its back.  One warp per
// cell bucket scans the bucket's records (in cell order) and gives each
// Tier-G cell its output range from the scans the emission kernel uses: its
// triangles follow those of the bucket's earlier cells (one each when uncut,
// ntri each when cut) and its inside vertices those of the bucket's earlier
// cut cells.  In the compact format only the cut cells' triangles are listed.
// The lists hold (job, record) pairs.
template <bool ONE>
__global__ void __launch_bounds__(32 * GORDER_W) k_gorder_b(const __grid_constant__ Job one,
                                                            const Job* __restrict__ jobs, const u32* __restrict__ bpre,
                                                            int njobs, BatchDev* bd, uint2* olist, uint2* slist,
                                                            uint2* wlist, uint2* wlast) {
  __shared__ u32 s_base[TM + 1];
  __shared__ u32 s_kw;
  __shared__ u32 s_wc[GORDER_W][NSIZE];  // per warp: its cells per size, then its first place among the block's
  __shared__ u32 s_blk[NSIZE];           // the block's first place per size (one atomic per size and block)
  if (threadIdx.x == 0) {
    u32 run = 0, big = 0;
    for (int n = TM; n >= 0; --n) {
      s_base[n] = run, run += bd->gcnt[n];
      if (n == TN + 1) big = run;  // the cells above TN
    }
    s_kw = big;
    if (blockIdx.x == 0) bd->nolist = run - big, bd->nslist = big;
  }
  for (int i = threadIdx.x; i < GORDER_W * NSIZE; i += blockDim.x) (&s_wc[0][0])[i] = 0u;
  __syncthreads();
  SBMT_BLOCK_JOB(ONE, one, jobs, bpre, njobs)
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const u32 b = lb * GORDER_W + (u32)w;
  const bool live = b < J.nbc;  // a warp past the job's buckets still meets the block's barriers
  CutRec* recs = J.recs;
  const u32 n = live ? J.bcut[b] : 0u, rec0 = live ? J.bbase[b] : 0u;
  // the warp's Tier-G cells per size
  for (u32 base = 0; base < n; base += 32) {
    const u32 r = base + (u32)lane;
    CutRec rec{};
    if (r < n) rec = recs[rec0 + r];
    const bool tg = r < n && (rec.code & (1u << 16));
    const unsigned tmask = __ballot_sync(0xffffffffu, tg);
    if (tg) {
      const int key = tierg_size(local_count(rec));
      const unsigned peers = __match_any_sync(tmask, key);
      if (lane == __ffs(peers) - 1) s_wc[w][key] += (u32)__popc(peers);
    }
    __syncwarp();
  }
  __syncthreads();
  // per size: the warps' places within the block, and one atomic for the block
  if (threadIdx.x < NSIZE) {
    const int key = (int)threadIdx.x;
    u32 tot = 0;
    for (int q = 0; q < GORDER_W; ++q) {
      const u32 c = s_wc[q][key];
      s_wc[q][key] = tot, tot += c;
    }
    s_blk[key] = tot ? atomicAdd(&bd->gcur[key], tot) : 0u;
  }
  __syncthreads();
  if (!live) return;
  const u32* extra_scan = J.extra_scan;
  const u32* cut_scan = J.cp.on ? J.cp.cut_scan : nullptr;
  const u32 CB0 = J.NVg + J.NE;
  const u32 kw = s_kw;
  u32 ct = 0, cc = 0;  // the bucket's earlier records: sum of (ntri - 1), of nchain
  for (u32 base = 0; base < n; base += 32) {
    const u32 r = base + (u32)lane;
    const bool valid = r < n;
    CutRec rec{};
    if (valid) rec = recs[rec0 + r];
    const u32 vt = valid ? rec.ntri - 1u : 0u, vc = valid ? rec.nchain : 0u;
    u32 it = vt, ic = vc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u32 t = __shfl_up_sync(0xffffffffu, it, o), c = __shfl_up_sync(0xffffffffu, ic, o);
      if (lane >= o) it += t, ic += c;
    }
    const u32 pt = ct + it - vt, pc = cc + ic - vc;
    ct += __shfl_sync(0xffffffffu, it, 31), cc += __shfl_sync(0xffffffffu, ic, 31);
    const bool tg = valid && (rec.code & (1u << 16));
    const unsigned tmask = __ballot_sync(0xffffffffu, tg);
    if (tg) {
      recs[rec0 + r].tri_off = cut_scan ? extra_scan[b] + cut_scan[b] + r + pt : rec.cell + extra_scan[b] + pt;
      recs[rec0 + r].chain_base = CB0 + J.chain_scan[b] + pc;
      const int key = tierg_size(local_count(rec));
      // the cells of one size take consecutive places, in the warp's order
      const unsigned peers = __match_any_sync(tmask, key);
      const int leader = __ffs(peers) - 1;
      u32 at = 0;
      if (lane == leader) at = s_blk[key] + s_wc[w][key], s_wc[w][key] += (u32)__popc(peers);
      at = __shfl_sync(peers, at, leader) + (u32)__popc(peers & ((1u << lane) - 1u));
      const uint2 e = make_uint2((u32)jk, rec0 + r);
      if (key == TM + 2) {
        *(wlast - at) = e;
      } else if (key == TM + 1) {
        wlist[at] = e;
      } else {
        const u32 pos = s_base[key] + at;  // place in the order, largest first
        if (pos < kw) slist[pos] = e;
        else olist[pos - kw] = e;
      }
    }
    __syncwarp();
  }
}

SBMT_DEV void tierg_over(const Job& J, u32 cell) {
  atomicOr(jc(J, JC_ERR), ERR_CAPACITY);
  const u32 slot = atomicAdd(jc(J, JC_NOVER), 1u);
  if (slot < OVER_CAP) J.over[slot] = cell;
}

// ---------------------------------------------------------------------------
// cells of at most 32 vertices: a group of G lanes each
// ---------------------------------------------------------------------------
template <int G>
struct TState {
  GCell<G> c;
  int xa[G], xb[G], ya[G], yb[G];  // cell-local exact coordinates (a + b sqrt3)
  u32 gid[G];
  union {
    // while gathering: the events as found (their (edge, position) keys,
    // cell-local coordinates, vertex ids) and the pieces' ends at pixel
    // corners, with the local vertex each becomes
    struct {
      u64 ekey[G];
      int4 exy[G];
      u32 egid[G];
      u32 cid[4 * G];
      unsigned char cfirst[4 * G];  // whether an end is its corner's first in the list
      unsigned char eloc[G], cloc[4 * G];
    } t;
    // afterwards: the candidates' exact squared lengths la + lb sqrt3
    struct {
      i64 a[G * (G - 1) / 2], b[G * (G - 1) / 2];
    } len;
  };
};

// (a + b sqrt3) / 1 of a point near the cell as a float, by integers (this
// GPU's FP64 runs at a small fraction of its FP32 rate): the value with 32
// fraction bits modulo 2^64 -- exact but for b times what sqrt3 is beyond 2^-64
// and one unit of 2^-32 -- then rounded once.  The components may be of the order
// of the image, the sum is below 2^31.
SBMT_DEV float zq_float(int a, int b) {
  const u64 v = ((u64)(i64)a << 32) + (u64)(i64)b * 7439101573ull + (u64)(((i64)b * 2227873595ll) >> 32);
  return i64_float((i64)v, -32);
}

// zsign with a single-precision estimate in front: its error is below 2.4e-7
// (|a| + |b| sqrt3) (three roundings of 2^-24 a term and one of the sum)
SBMT_DEV int zsign_fast(Zq v) {
  const float fa = i64_float(v.a), fb = i64_float(v.b) * 1.7320508f, t = fa + fb;
  if (fabsf(t) > 4e-7f * (fabsf(fa) + fabsf(fb))) return t > 0.0f ? 1 : -1;
  return zsign(v);
}

// the lattice path's geometry: exact numbers behind single-precision filters.
// M, the grid edge in scaled units, bounds the cell's extent, and a float
// coordinate is off by 2^-24 M + 2^-32: the filters' bands are several times
// the resulting errors (a determinant 1.2e-6 M^2, a squared length or a dot
// product 1.1e-6 M^2).
template <int G>
struct LatGeo {
  TState<G>* s;
  float M2;
  SBMT_DEV float tol() const { return 8e-6f * M2; }
  SBMT_DEV Pq pt(int k) const { return Pq{zq(s->xa[k], s->xb[k]), zq(s->ya[k], s->yb[k])}; }
  SBMT_DEV bool resolve(int u, int v, int w, int* o) const {
    // three points of one cell edge, pixel column or pixel row need no test
    if (s->c.em[u] & s->c.em[v] & s->c.em[w]) *o = 0;
    else if (s->xa[u] == s->xa[v] && s->xa[v] == s->xa[w] && s->xb[u] == s->xb[v] && s->xb[v] == s->xb[w]) *o = 0;
    else if (s->ya[u] == s->ya[v] && s->ya[v] == s->ya[w] && s->yb[u] == s->yb[v] && s->yb[v] == s->yb[w]) *o = 0;
    else {
      const int x1a = s->xa[v] - s->xa[u], x1b = s->xb[v] - s->xb[u], y1a = s->ya[v] - s->ya[u], y1b = s->yb[v] - s->yb[u];
      const int x2a = s->xa[w] - s->xa[u], x2b = s->xb[w] - s->xb[u], y2a = s->ya[w] - s->ya[u], y2b = s->yb[w] - s->yb[u];
      *o = zsign_fast(Zq{(i64)x1a * y2a - (i64)y1a * x2a + 3 * ((i64)x1b * y2b - (i64)y1b * x2b),
                         (i64)x1a * y2b + (i64)x1b * y2a - (i64)y1a * x2b - (i64)y1b * x2a});
    }
    return true;
  }
  SBMT_DEV int late(int, int, int) const { return 0; }
  SBMT_DEV bool ahead(int o, int p, int q) const {  // (p - o) . (q - o) > 0
    const float2 a = s->c.f[o], b = s->c.f[p], c = s->c.f[q];
    const float t = (b.x - a.x) * (c.x - a.x) + (b.y - a.y) * (c.y - a.y);
    if (fabsf(t) > 8e-6f * M2) return t > 0.0f;
    return zsign(dot3(pt(o), pt(p), pt(q))) > 0;
  }
  SBMT_DEV bool between(int u, int v, int k) const { return ahead(u, v, k) && ahead(v, u, k); }
  SBMT_DEV float key(int u, int v, int i) const {
    // the exact squared length beside the float one: equal lengths are common
    // (steps of the pixel grid), and then only the two components are compared
    const int xa = s->xa[v] - s->xa[u], xb = s->xb[v] - s->xb[u], ya = s->ya[v] - s->ya[u], yb = s->yb[v] - s->yb[u];
    s->len.a[i] = (i64)xa * xa + (i64)ya * ya + 3 * ((i64)xb * xb + (i64)yb * yb);
    s->len.b[i] = 2 * ((i64)xa * xb + (i64)ya * yb);
    const float2 a = s->c.f[u], b = s->c.f[v];
    const float dx = b.x - a.x, dy = b.y - a.y;
    return dx * dx + dy * dy;
  }
  // by exact squared length, then the packed pair
  SBMT_DEV bool less(float kx, unsigned short x, int i, float ky, unsigned short y, int j) const {
    if (kx < ky - 5e-6f * M2) return true;
    if (kx > ky + 5e-6f * M2) return false;
    const i64 a = s->len.a[i] - s->len.a[j], b = s->len.b[i] - s->len.b[j];
    if ((a | b) == 0) return x < y;
    return zsign_fast(Zq{a, b}) < 0;  // a + b sqrt3 is 0 only for a = b = 0
  }
};

// The group's cell into its state: corners A, B, C; the events on AB, BC, CA
// in counter-clockwise order (the registry numbers an edge's events along it,
// so their vertex ids order them); the inside vertices by pixel-corner id; the
// boundary cycle and the pieces.  Lane l takes pairs l and l + G (a cell of n
// vertices has at most 2 (n - 3) pieces: an event ends one, a corner four at
// most).  Returns n, or -1 for a record that does not fit its counts.
template <int G>
SBMT_DEV int tg_gather(const GridP& g, const CellGeo& cg, const CutRec& rec, bool live, const Pair* P, const Seg* segs,
                       const Event* ev, TState<G>& s, const GLane<G>& me, Pq* A_out) {
  const int n = live ? (int)(rec.ntri + 2 - rec.nchain) : 0, np = live ? (int)rec.npairs : 0;
  bool bad = n > G || np > 2 * G;
  Pq A{zq(0), zq(0)};
  if (live) A = lattice_pt(g, cg.ci[0], cg.cj[0]);
  *A_out = A;
  auto put = [&](int v, int xa, int xb, int ya, int yb, u32 gid, int em) {
    s.xa[v] = xa, s.xb[v] = xb, s.ya[v] = ya, s.yb[v] = yb;
    s.c.f[v] = make_float2(zq_float(xa, xb), zq_float(ya, yb));
    s.gid[v] = gid, s.c.em[v] = (unsigned char)em;
  };
  // the pieces' ends: events and pixel corners, listed in any order; a lane
  // keeps the list places of its own pieces' ends (corners from 128)
  int ne = 0, nc = 0;
  const int slots = __any_sync(0xffffffffu, np > G) ? 2 : 1;  // few cells have more pieces than lanes
  int at[4] = {0, 0, 0, 0};
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    if (t >= slots) break;
    const int k = me.l + t * G;
    Pair pr{0, 0, NONE, NONE};
    const bool has = !bad && k < np;
    if (has) pr = P[k];
    Seg sg{0, 0, 0, 0};
    if (has && (pr.ev_in == NONE || pr.ev_out == NONE)) sg = segs[pr.seg];
#pragma unroll
    for (int end = 0; end < 2; ++end) {
      const u32 e = end == 0 ? pr.ev_in : pr.ev_out;
      const bool isev = has && e != NONE, isc = has && e == NONE;
      const u32 be = me.ballot(isev), bc = me.ballot(isc);
      if (isev) {
        const Event x = ev[e];
        int le = local_edge(cg, x.edge);
        if (le < 0) bad = true, le = 0;
        // AB runs with its edge; BC with it in an up cell; CA against it
        const bool fwd = le == 0 || (le == 1 && !cg.down);
        const int i = ne + __popc(be & me.below());
        at[2 * t + end] = i;
        if (i < G) {
          s.t.ekey[i] = (u64)le << 32 | (fwd ? x.gid : ~x.gid);
          s.t.exy[i] = make_int4((int)(x.xa - A.x.a), (int)(x.xb - A.x.b), (int)(x.ya - A.y.a), (int)(x.yb - A.y.b));
          s.t.egid[i] = x.gid;
        }
      } else if (isc) {
        const int i = nc + __popc(bc & me.below());
        at[2 * t + end] = 128 + i;
        if (i < 4 * G) s.t.cid[i] = corner_id(g, sg, end);
      }
      ne += __popc(be), nc += __popc(bc);
    }
  }
  const int nin = live ? (int)rec.nchain : 0;
  if (live && ne != n - 3 - nin) bad = true;
  bad = me.ballot(bad) != 0;
  if (bad) ne = nc = 0;
  __syncwarp();
  if (me.l < ne) {
    const u64 key = s.t.ekey[me.l];
    int r = 0;
    for (int j = 0; j < ne; ++j) r += s.t.ekey[j] < key ? 1 : 0;
    const int4 p = s.t.exy[me.l];
    s.t.eloc[me.l] = (unsigned char)(3 + r);
    put(3 + r, p.x, p.y, p.z, p.w, s.t.egid[me.l], 1 << (int)(key >> 32));
  }
  const int cmax = warp_max(nc);
  int nfirst = 0;
  for (int i0 = 0; i0 < cmax; i0 += G) {
    const int i = i0 + me.l;
    bool first = i < nc;
    if (first) {
      const u32 id = s.t.cid[i];
      for (int j = 0; j < i; ++j) first = first && s.t.cid[j] != id;
      s.t.cfirst[i] = first;
    }
    nfirst += __popc(me.ballot(first));
  }
  if (live && nfirst != nin) bad = true;  // the same in every lane of the group
  __syncwarp();
  for (int i = me.l; i < nc && !bad; i += G) {
    const u32 id = s.t.cid[i];
    int r = 0;
    for (int j = 0; j < nc; ++j) r += (s.t.cfirst[j] && s.t.cid[j] < id) ? 1 : 0;
    s.t.cloc[i] = (unsigned char)(3 + ne + r);
    if (s.t.cfirst[i]) {
      const Pq p = corner_of_id(g, id);
      put(3 + ne + r, (int)(p.x.a - A.x.a), (int)(p.x.b - A.x.b), (int)(p.y.a - A.y.a), (int)(p.y.b - A.y.b),
          rec.chain_base + (u32)r, 0);
    }
  }
  if (live && !bad && me.l < 3) {
    const int k = me.l;
    const i64 ci = k == 0 ? cg.ci[0] : k == 1 ? cg.ci[1] : cg.ci[2], cj = k == 0 ? cg.cj[0] : k == 1 ? cg.cj[1] : cg.cj[2];
    const Pq p = lattice_pt(g, ci, cj);
    put(k, (int)(p.x.a - A.x.a), (int)(p.x.b - A.x.b), (int)(p.y.a - A.y.a), (int)(p.y.b - A.y.b), vid(g, ci, cj),
        (1 << k) | (1 << (k == 0 ? 2 : k - 1)));
  }
  __syncwarp();
  // the boundary cycle: A, events on AB, B, events on BC, C, events on CA
  const int em = live && !bad && me.l >= 3 && me.l < 3 + ne ? (int)s.c.em[me.l] : 0;
  const int n0 = __popc(me.ballot(em == 1)), n1 = __popc(me.ballot(em == 2)), n2 = __popc(me.ballot(em == 4));
  if (live && !bad) {
    u32 adj = 0;
    if (me.l < 3) {
      const int k = me.l;
      const int own = k == 0 ? n0 : k == 1 ? n1 : n2, b0 = k == 0 ? 3 : k == 1 ? 3 + n0 : 3 + n0 + n1;
      const int pk = k == 0 ? n2 : k == 1 ? n0 : n1;  // the events of the edge ending here
      adj = 1u << (own ? b0 : (k == 2 ? 0 : k + 1));
      adj |= 1u << (pk ? (k == 0 ? 2 + n0 + n1 + n2 : b0 - 1) : (k == 0 ? 2 : k - 1));
    } else if (me.l < 3 + ne) {
      const int e = me.l - 3, k = e < n0 ? 0 : e < n0 + n1 ? 1 : 2;
      const int b0 = k == 0 ? 0 : k == 1 ? n0 : n0 + n1, own = k == 0 ? n0 : k == 1 ? n1 : n2;
      adj = 1u << (e == b0 ? k : me.l - 1);
      adj |= 1u << (e + 1 == b0 + own ? (k == 2 ? 0 : k + 1) : me.l + 1);
    }
    if (me.l < n) s.c.adj[me.l] = adj;
  }
  __syncwarp();
  // the pieces
  int nce = 0;
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    if (t >= slots) break;
    const bool has = live && !bad && me.l + t * G < np;
    const u32 b = me.ballot(has);
    if (has) {
      const int x = at[2 * t], y = at[2 * t + 1];
      const int lx = x < 128 ? s.t.eloc[x] : s.t.cloc[x - 128], ly = y < 128 ? s.t.eloc[y] : s.t.cloc[y - 128];
      const int p = min(lx, ly), q = max(lx, ly);
      s.c.ce[nce + __popc(b & me.below())] = (unsigned short)((p << 8) | q);
      atomicOr(&s.c.adj[p], 1u << q);
      atomicOr(&s.c.adj[q], 1u << p);
    }
    nce += __popc(b);
  }
  if (me.l == 0) s.c.nce = nce;
  __syncwarp();
  return bad ? -1 : n;
}

template <bool ONE, int G>
__global__ void __launch_bounds__(64, TG_OCC) k_tierg_group_b(const __grid_constant__ Job one, const Job* __restrict__ jobs,
                                                      const u32* count, const uint2* list) {
  constexpr int C = 64 / G;  // cells per block and turn
  __shared__ TState<G> sm[C];
  const GLane<G> me;
  TState<G>& s = sm[threadIdx.x / G];
  const u32 total = *count;
  for (u32 item = blockIdx.x * C + threadIdx.x / G;; item += gridDim.x * C) {
    const bool live = item < total;
    if (!__any_sync(0xffffffffu, live)) break;
    uint2 e = make_uint2(0u, 0u);
    if (live) e = list[item];
    const Job& J = ONE ? one : jobs[e.x];
    const GridP& g = J.g;
    CutRec rec{};
    CellGeo cg{};
    if (live) rec = J.recs[e.y], cg = cell_geo(g, rec.cell, cell_row_near(g, rec.cell));
    Pq A;
    const int n = tg_gather<G>(g, cg, rec, live, J.raw + rec.pair_lo, J.segs, J.ev, s, me, &A);
    if (live && n < 0 && me.l == 0) tierg_over(J, rec.cell);
    // every point of a cell lies within M = 6p scaled units of its corner A
    const float M = (float)(6 * (int)g.p);
    const LatGeo<G> geo{&s, M * M};
    g_greedy<G, false>(s.c, geo, max(n, 0));
    if (n > 0) {
      const int nt = min((int)s.c.nface, 2 * G);
      if (me.l == 0 && s.c.nface != rec.ntri) atomicOr(jc(J, JC_ERR), ERR_COUNT);
      const unsigned short cd = (unsigned short)(rec.code & 0xFFFFu);
      const Zq Sx = zq(3 * A.x.a, 3 * A.x.b), Sy = zq(3 * A.y.a, 3 * A.y.b);
      for (int k = me.l; k < nt; k += G) {
        const u32 f = s.c.face[k];
        u32 r = 0;
        for (int j = 0; j < nt; ++j) r += s.c.face[j] < f ? 1u : 0u;
        if (r >= rec.ntri) continue;
        const int a = (int)(f >> 16), b = (int)((f >> 8) & 255u), c = (int)(f & 255u);
        const u32 o = rec.tri_off + r;
        J.tri[3 * (i64)o] = (int)s.gid[a], J.tri[3 * (i64)o + 1] = (int)s.gid[b], J.tri[3 * (i64)o + 2] = (int)s.gid[c];
        J.label[o] = label_at_sum(g, J.img, J.pitch, J.dtype,
                                  Sx + zq((i64)s.xa[a] + s.xa[b] + s.xa[c], (i64)s.xb[a] + s.xb[b] + s.xb[c]),
                                  Sy + zq((i64)s.ya[a] + s.ya[b] + s.ya[c], (i64)s.yb[a] + s.yb[b] + s.yb[c]));
        J.code[o] = cd;
      }
      // coordinates of the cell's inside vertices
      const int nin = (int)rec.nchain, loc = n - nin + me.l;
      if (me.l < nin) {
        const double invS = g.invS;
        double2 v;
        v.x = zdouble(zq((i64)s.xa[loc] + A.x.a, (i64)s.xb[loc] + A.x.b)) * invS;
        v.y = zdouble(zq((i64)s.ya[loc] + A.y.a, (i64)s.yb[loc] + A.y.b)) * invS;
        reinterpret_cast<double2*>(J.xy)[s.gid[loc] - J.cp.xy0] = v;
      }
    }
    __syncwarp();
  }
}

// one warp per Tier-G cell above TL vertices, the state in shared memory
template <bool ONE>
__global__ void __launch_bounds__(32 * WWARPS) k_tierg_warp_b(const __grid_constant__ Job one,
                                                              const Job* __restrict__ jobs, const u32* count,
                                                              const uint2* last) {
  constexpr int N = WN;
  __shared__ GStore<N> sm[WWARPS];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  GStore<N>& s = sm[w];
  const u32 total = *count;
  for (u32 item = blockIdx.x * WWARPS + w; item < total; item += gridDim.x * WWARPS) {
    const uint2 e = *(last - item);
    const Job& J = ONE ? one : jobs[e.x];
    const GridP g = J.g;
    const CutRec rec = J.recs[e.y];
    const CellGeo cg = cell_geo(g, rec.cell, cell_row_near(g, rec.cell));
    // the lanes request the cell's pair records, events and segments into
    // L1 together, so that the one lane building the local graph finds them
    // there instead of waiting on each in turn
    const Pair* P = J.raw + rec.pair_lo;
    for (u32 k = (u32)lane; k < rec.npairs; k += 32) {
      const Pair pr = P[k];
      if (pr.ev_in != NONE) prefetch_l1(J.ev + pr.ev_in);
      if (pr.ev_out != NONE) prefetch_l1(J.ev + pr.ev_out);
      prefetch_l1(J.segs + pr.seg);
    }
    __syncwarp();
    if (lane == 0) build_local(g, cg, rec, P, J.segs, J.ev, s);
    __syncwarp();
    if (!s.ok) {
      if (lane == 0) tierg_over(J, rec.cell);
      __syncwarp();
      continue;
    }
    // cell-local coordinates are bounded by the cell extent M = 6p scaled units
    const float M = (float)(6 * (int)g.p);
    greedy_faces<N>(s, lane, boundary_count(rec), OriFiltered<N>{&s, 8e-6f * M * M}, 1e-4f * M * M);
    write_patch<N>(g, J.img, J.pitch, J.dtype, cg, rec, s, lane, J.tri, J.label, J.code, J.xy, J.cp.xy0,
                   jc(J, JC_ERR));
    __syncwarp();
  }
}

// the status words of every job (error bits, cut cells, Tier-G cells, Tier-G
// triangles, cells over the Tier-G limit) into its mapped host slot
__global__ void k_status_b(const Job* __restrict__ jobs, int njobs, const BatchDev* bd) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < njobs; k += gridDim.x * blockDim.x) {
    const Job& J = jobs[k];
    for (int w = 0; w < 5; ++w) J.hinfo[w] = *jc(J, JC_ERR + w);
  }
  __threadfence_system();
}

}  // namespace

namespace {

template <bool ONE>
int launch_tierg(const Job& oj, const Job* jobs, const u32* bpre, int njobs, u32 nblocks, const BatchPtrs& bp,
                 int blocks_per_sm, cudaStream_t st, cudaStream_t st2, cudaEvent_t ev_order, cudaEvent_t ev_warp) {
  k_gorder_b<ONE><<<nblocks, 32 * GORDER_W, 0, st>>>(oj, jobs, bpre, njobs, bp.bd, bp.olist, bp.slist, bp.wlist,
                                                     bp.wlast);
  k_tierg_group_b<ONE, 8><<<152 * blocks_per_sm, 64, 0, st>>>(oj, jobs, &bp.bd->nolist, bp.olist);
  // the larger cells on their own stream when given one, after the 8-lane
  // groups and beside the emission, the largest first.  (Beside the groups too, from the
  // order alone: 1 to 2% faster with few cells, but 2.06 against 2.04 ms on
  // 8192^2 labels, where they take room from both.)
  if (st2) {
    if (cudaEventRecord(ev_order, st) != cudaSuccess || cudaStreamWaitEvent(st2, ev_order, 0) != cudaSuccess) return -1;
  }
  cudaStream_t ws = st2 ? st2 : st;
  k_tierg_warp_b<ONE><<<152 * 2, 32 * WWARPS, 0, ws>>>(oj, jobs, &bp.bd->gcur[TM + 2], bp.wlast);
  k_tierg_group_b<ONE, 32><<<152 * 6, 64, 0, ws>>>(oj, jobs, &bp.bd->gcur[TM + 1], bp.wlist);
  k_tierg_group_b<ONE, 16><<<152 * 12, 64, 0, ws>>>(oj, jobs, &bp.bd->nslist, bp.slist);
  if (st2) {
    if (cudaEventRecord(ev_warp, st2) != cudaSuccess || cudaStreamWaitEvent(st, ev_warp, 0) != cudaSuccess) return -1;
  }
  return 5;
}

}  // namespace

int launch_tierg_b(const Job* one, const Job* jobs, const u32* bpre, int njobs, u32 nblocks, const BatchPtrs& bp,
                   int blocks_per_sm, cudaStream_t st, cudaStream_t st2, cudaEvent_t ev_order, cudaEvent_t ev_warp) {
  if (nblocks == 0) return 0;
  const Job none{};
  if (one) return launch_tierg<true>(*one, jobs, bpre, njobs, nblocks, bp, blocks_per_sm, st, st2, ev_order, ev_warp);
  return launch_tierg<false>(none, jobs, bpre, njobs, nblocks, bp, blocks_per_sm, st, st2, ev_order, ev_warp);
}

int launch_status_b(const Job* jobs, int njobs, const BatchPtrs& bp, cudaStream_t st) {
  k_status_b<<<(njobs + 255) / 256, 256, 0, st>>>(jobs, njobs, bp.bd);
  return 1;
}

}  // namespace sbmt
