// sbmt_greedy.cuh -- the greedy completion of a cell's local boundary graph
// by a group of G lanes (G = 8, 16 or 32; 32 / G cells to a warp), shared by
// the lattice path (k_tierg.cu) and the retriangulation of a preprocessed mesh
// (k_region3.cu).
//
// The rule: every vertex pair not joined by a constraint edge and not on one
// cell edge, in the geometry's order (length, then the pair), is kept when its
// open segment holds no vertex and crosses no kept edge; the faces are the
// 3-cycles with no vertex inside, listed smallest index first,
// counter-clockwise, in sorted order.
//
// The cell has at most G vertices, so that sets of vertices are masks of G
// bits and a lane owns a vertex:
//  - per directed pair (u, v) the vertices left of it, and those the float
//    filter leaves undecided (the geometry resolves them, at once or on use);
//  - each lane lists its own candidates (pairs u, u + d), those blocked by a
//    vertex or a constraint edge left out, and ranks them by counting;
//  - the greedy pass goes through the ranks, the lanes testing one kept edge
//    each against the candidate, one ballot per candidate.
// One thread per cell needs as many steps as the cell has pairs times
// vertices, with its state in local memory; here the pairs, the candidates and
// the kept edges of a cell are tested side by side, and the state (0.8 KB for
// G = 8) is in shared memory.
//
// The groups of a warp run the same number of turns of every loop (the
// largest of theirs), so that the ballots meet; a group without a cell has n = 0.
#pragma once
#include "sbmt_dev.cuh"

namespace sbmt {

template <int G>
struct GMask;
template <>
struct GMask<8> {
  typedef unsigned char T;
};
template <>
struct GMask<16> {
  typedef unsigned short T;
};
template <>
struct GMask<32> {
  typedef u32 T;
};

// one cell's state in shared memory
template <int G>
struct GCell {
  typedef typename GMask<G>::T M;
  float2 f[G];        // the vertices in the filter's frame
  M L[G][G];          // L[u][v]: the vertices left of u -> v
  M Z[G][G];          // Z[u][v]: those within the filter's band of its line (both ways round)
  unsigned char em[G];  // the cell edges a vertex lies on (bit k: edge k)
  u32 adj[G];
  unsigned short ce[3 * G];  // constraint edges tested against the candidates (u << 8 | v)
  unsigned short ke[3 * G];  // kept edges
  float key[G * (G - 1) / 2];
  unsigned short cand[G * (G - 1) / 2], ord[G * (G - 1) / 2];
  u32 face[2 * G];
  u32 nface;
  int nce;
};

// a lane's place in its group
template <int G>
struct GLane {
  int lane, l, base;
  SBMT_DEV GLane() : lane((int)(threadIdx.x & 31u)), l(lane & (G - 1)), base(lane & ~(G - 1)) {}
  SBMT_DEV u32 ballot(bool p) const {
    const u32 b = __ballot_sync(0xffffffffu, p);
    return G == 32 ? b : (b >> base) & ((1u << (G & 31)) - 1u);
  }
  SBMT_DEV u32 below() const { return (1u << l) - 1u; }
};
SBMT_DEV int warp_max(int x) { return __reduce_max_sync(0xffffffffu, x); }

// The geometry Geo gives
//   tol()          the filter's bound on a float determinant;
//   resolve(u,v,w) true when an undecided triple is decided at once: *s its sign;
//   late(u,v,w)    the sign of a triple left in Z, on use;
//   between(u,v,k) whether vertex k, on the line u v, lies strictly between;
//   key(u,v,i)     the pair's single-precision key (the pair is candidate i);
//   less(ki,pi,i,kj,pj,j) the order of candidates i and j (keys, pairs u << 8 | v).
// LATE: whether triples can stay in Z undecided (then every sign read from
// the sets is checked for it).
template <int G, bool LATE, class Geo>
SBMT_DEV int g_sign(const GCell<G>& s, const Geo& geo, int u, int v, int w) {
  if ((s.Z[u][v] >> w) & 1u) return LATE ? geo.late(u, v, w) : 0;
  return ((s.L[u][v] >> w) & 1u) ? 1 : -1;
}
// edge (a, b) and pair (u, v), no end in common, cross properly; l and r are
// the vertices left and right of u -> v (an end in common is neither, so most
// edges leave at the first test)
template <int G, bool LATE, class Geo>
SBMT_DEV bool g_cross(const GCell<G>& s, const Geo& geo, int u, int v, u32 l, u32 r, int a, int b) {
  if (LATE) {
    if (a == u || a == v || b == u || b == v) return false;
    const u32 und = ((u32)s.Z[u][v] >> a) | ((u32)s.Z[u][v] >> b) | ((u32)s.Z[a][b] >> u) | ((u32)s.Z[a][b] >> v);
    if (und & 1u) {
      const int o1 = g_sign<G, LATE>(s, geo, u, v, a), o2 = g_sign<G, LATE>(s, geo, u, v, b);
      if (o1 * o2 >= 0) return false;
      return g_sign<G, LATE>(s, geo, a, b, u) * g_sign<G, LATE>(s, geo, a, b, v) < 0;
    }
  }
  if (!((((l >> a) & (r >> b)) | ((l >> b) & (r >> a))) & 1u)) return false;
  const u32 x = s.L[a][b], y = s.L[b][a];
  return ((((x >> u) & (y >> v)) | ((x >> v) & (y >> u))) & 1u) != 0;
}

// the sets, candidates, greedy pass and faces of the group's cell of n
// vertices (0: none); s.f, s.em, s.adj (constraints and boundary cycle) and
// s.ce are filled in and visible to the warp.  On return s.face[0 .. nface)
// holds the faces (p << 16 | q << 8 | r) unsorted, visible to the warp.
template <int G, bool LATE, class Geo>
SBMT_DEV void g_greedy(GCell<G>& s, const Geo& geo, int n) {
  typedef typename GMask<G>::T M;
  const GLane<G> me;
  const int u = me.l;
  const u32 valid = n >= 32 ? 0xffffffffu : (1u << n) - 1u;
  const int half = n >> 1;
  const float tol = geo.tol();
  const int nmax = warp_max(n), hmax = nmax >> 1;
  // sets of the pairs (u, u + d), d up to n / 2; when n is even, the pairs half the
  // cycle apart by their lower vertex's lane alone.  A pair's L and Z must come
  // from one lane: the float determinants taken from its two ends round
  // differently, and at the edge of the band one decides a vertex that the other
  // leaves undecided.
  auto mine = [&](int d) { return u < n && d <= half && !(2 * d == n && u >= d); };
  for (int d = 1; d <= hmax; ++d) {
    if (mine(d)) {
      int v = u + d;
      if (v >= n) v -= n;
      const float2 pu = s.f[u], pv = s.f[v];
      const float dx = pv.x - pu.x, dy = pv.y - pu.y;
      u32 lm = 0, rm = 0;
      for (int w0 = 0; w0 < n; w0 += 8) {
        u32 l8 = 0, r8 = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {  // past n: masked off
          const float2 pw = s.f[w0 + w];
          const float o = __fmaf_rn(dx, pw.y - pu.y, -__fmul_rn(dy, pw.x - pu.x));
          l8 |= o > tol ? 1u << w : 0u;
          r8 |= o < -tol ? 1u << w : 0u;
        }
        lm |= l8 << w0, rm |= r8 << w0;
      }
      const u32 ends = (1u << u) | (1u << v), in = valid & ~ends;
      lm &= in, rm &= in;
      u32 zm = valid & ~(lm | rm | ends);
      for (u32 und = zm; und; und &= und - 1) {
        const int w = __ffs(und) - 1;
        int o;
        if (!geo.resolve(u, v, w, &o)) continue;
        if (o > 0) lm |= 1u << w, zm &= ~(1u << w);
        else if (o < 0) rm |= 1u << w, zm &= ~(1u << w);
      }
      s.L[u][v] = (M)lm, s.L[v][u] = (M)rm, s.Z[u][v] = s.Z[v][u] = (M)zm;
    }
  }
  __syncwarp();
  // candidates: pairs joined by no constraint, not on one cell edge (another
  // vertex lies between such a pair), blocked by no vertex and no constraint
  int m = 0;
  const u32 au = u < n ? s.adj[u] : 0u;
  const u32 eu = u < n ? s.em[u] : 0u;
  const int nce = n ? s.nce : 0;
  for (int d = 1; d <= hmax; ++d) {
    bool ok = mine(d);
    int p = 0, q = 0;
    if (ok) {
      int v = u + d;
      if (v >= n) v -= n;
      p = min(u, v), q = max(u, v);
      ok = !((au >> v) & 1u) && !(eu & s.em[v]);
      if (ok)
        for (u32 z = s.Z[p][q]; z && ok; z &= z - 1) {
          const int k = __ffs(z) - 1;
          if (LATE && geo.late(p, q, k) != 0) continue;
          if (geo.between(p, q, k)) ok = false;
        }
    }
    if (ok) {
      const u32 l = s.L[p][q], r = s.L[q][p];
      for (int c = 0; c < nce && ok; ++c) {
        const unsigned e = s.ce[c];
        if (g_cross<G, LATE>(s, geo, p, q, l, r, (int)(e >> 8), (int)(e & 255u))) ok = false;
      }
    }
    const u32 bal = me.ballot(ok);
    if (ok) {
      const int at = m + __popc(bal & me.below());
      s.cand[at] = (unsigned short)((p << 8) | q), s.key[at] = geo.key(p, q, at);
    }
    m += __popc(bal);
  }
  __syncwarp();
  // ranks
  const int mmax = warp_max(m);
  for (int i0 = 0; i0 < mmax; i0 += G) {
    const int i = i0 + me.l;
    if (i < m) {
      const unsigned short ci = s.cand[i];
      const float ki = s.key[i];
      int r = 0;
      for (int j = 0; j < m; ++j)
        if (j != i && geo.less(s.key[j], s.cand[j], j, ki, ci, i)) ++r;
      s.ord[r] = ci;
    }
  }
  __syncwarp();
  // the greedy pass
  int nk = 0;
  for (int r = 0; r < mmax; ++r) {
    bool bad = false;
    int p = 0, q = 0;
    if (r < m) {
      p = s.ord[r] >> 8, q = s.ord[r] & 255;
      if (me.l < nk) {
        const u32 l = s.L[p][q], rr = s.L[q][p];
        for (int k = me.l; k < nk; k += G) {
          const unsigned e = s.ke[k];
          bad |= g_cross<G, LATE>(s, geo, p, q, l, rr, (int)(e >> 8), (int)(e & 255u));
        }
      }
    }
    const u32 bal = me.ballot(bad);
    if (r < m && bal == 0) {
      if (me.l == 0) {
        if (nk < 3 * G) s.ke[nk] = (unsigned short)((p << 8) | q);
        s.adj[p] |= 1u << q, s.adj[q] |= 1u << p;
      }
      nk = min(nk + 1, 3 * G);
    }
    __syncwarp();
  }
  // faces, from their smallest vertex
  if (me.l == 0) s.nface = 0;
  __syncwarp();
  if (u < n) {
    const u32 a = s.adj[u];
    for (u32 vs = a & ~((2u << u) - 1u); vs; vs &= vs - 1) {
      const int v = __ffs(vs) - 1;
      for (u32 ws = a & s.adj[v] & ~((2u << v) - 1u); ws; ws &= ws - 1) {
        const int w = __ffs(ws) - 1;
        const int o = g_sign<G, LATE>(s, geo, u, v, w);
        if (o == 0) continue;
        const u32 self = (1u << u) | (1u << v) | (1u << w);
        u32 in = o > 0 ? (u32)(s.L[u][v] & s.L[v][w] & s.L[w][u]) : (u32)(s.L[v][u] & s.L[w][v] & s.L[u][w]);
        if (LATE && !(in & ~self)) {
          // a vertex undecided at some side and not clearly outside another
          u32 und = (s.Z[u][v] | s.Z[v][w] | s.Z[w][u]) & ~self;
          for (; und && !(in & ~self); und &= und - 1) {
            const int k = __ffs(und) - 1;
            if (g_sign<G, LATE>(s, geo, u, v, k) == o && g_sign<G, LATE>(s, geo, v, w, k) == o &&
                g_sign<G, LATE>(s, geo, w, u, k) == o)
              in |= 1u << k;
          }
        }
        if (in & ~self) continue;
        const u32 at = atomicAdd(&s.nface, 1u);
        if (at < 2u * G)
          s.face[at] = o > 0 ? ((u32)u << 16 | (u32)v << 8 | (u32)w) : ((u32)u << 16 | (u32)w << 8 | (u32)v);
      }
    }
  }
  __syncwarp();
}

}  // namespace sbmt
