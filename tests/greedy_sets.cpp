// sbmt_greedy.cuh on the host: the 32 lanes of a warp as coroutines that run
// from one warp-wide operation to the next, in ascending or in descending
// order of the lanes.  What a step leaves in shared memory may not depend on
// the order.  Cells of n vertices whose vertex w lies at the edge of the
// filter's band of the pair (u, u + n / 2): the determinant taken from u
// decides w, the one from the other end does not, or the other way round.
// Prints, per group size, the cells tried and those of each kind of failure.
#include <ucontext.h>

#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

struct Idx { unsigned x; } threadIdx;

namespace warp {
ucontext_t lane_ctx[32], main_ctx;
char stack[32][1 << 16];
bool done[32];
unsigned arg[32];  // a lane's operand of the operation it waits at
int cur;
void wait() { swapcontext(&lane_ctx[cur], &main_ctx); }
unsigned ballot(unsigned v) {
  arg[cur] = v, wait();
  unsigned m = 0;
  for (int l = 0; l < 32; ++l) m |= (arg[l] ? 1u : 0u) << l;
  wait();
  return m;
}
int reduce_max(int v) {
  arg[cur] = (unsigned)v, wait();
  int m = (int)arg[0];
  for (int l = 1; l < 32; ++l) m = (int)arg[l] > m ? (int)arg[l] : m;
  wait();
  return m;
}
void (*body)();
void entry() {
  body();
  done[cur] = true;
  swapcontext(&lane_ctx[cur], &main_ctx);
}
void run(void (*f)(), bool descending) {
  body = f;
  for (int l = 0; l < 32; ++l) {
    done[l] = false;
    getcontext(&lane_ctx[l]);
    lane_ctx[l].uc_stack.ss_sp = stack[l], lane_ctx[l].uc_stack.ss_size = sizeof stack[l], lane_ctx[l].uc_link = nullptr;
    makecontext(&lane_ctx[l], entry, 0);
  }
  for (bool any = true; any;) {
    any = false;
    for (int k = 0; k < 32; ++k) {
      const int l = descending ? 31 - k : k;
      if (done[l]) continue;
      any = true, cur = l, threadIdx.x = (unsigned)l;
      swapcontext(&main_ctx, &lane_ctx[l]);
    }
  }
}
}  // namespace warp

inline unsigned __ballot_sync(unsigned, bool p) { return warp::ballot(p); }
inline int __reduce_max_sync(unsigned, int x) { return warp::reduce_max(x); }
inline void __syncwarp() { warp::wait(); }
inline unsigned atomicAdd(unsigned* p, unsigned v) {
  const unsigned o = *p;
  *p = o + v;
  return o;
}
inline int __popc(unsigned x) { return __builtin_popcount(x); }
inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
inline float __int_as_float(int x) {
  float f;
  std::memcpy(&f, &x, 4);
  return f;
}
inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
inline float __fmul_rn(float a, float b) { return a * b; }
using std::max;
using std::min;

#include "sbmt_greedy.cuh"

using namespace sbmt;

// the retriangulation's geometry: triples in the band stay undecided and are
// decided by the doubles on use
struct Geo {
  const double *x, *y;
  float T;
  float tol() const { return T; }
  bool resolve(int, int, int, int*) const { return false; }
  int late(int u, int v, int w) const {
    const double o = (x[v] - x[u]) * (y[w] - y[u]) - (y[v] - y[u]) * (x[w] - x[u]);
    return (o > 0) - (o < 0);
  }
  bool between(int, int, int) const { return false; }
  float key(int u, int w, int) const { return (float)((x[w] - x[u]) * (x[w] - x[u]) + (y[w] - y[u]) * (y[w] - y[u])); }
  bool less(float kx, unsigned short a, int, float ky, unsigned short b, int) const {
    return kx < ky || (kx == ky && a < b);
  }
};

template <int G>
struct Run {
  static GCell<G> cell[32 / G];
  static double x[G], y[G];
  static Geo geo;
  static int n;
  static void lane() {  // the first group has the cell, the others none
    const int g = (int)threadIdx.x / G;
    g_greedy<G, true>(cell[g], geo, g == 0 ? n : 0);
  }
  static float det(int u, int v, int w) {  // the filter's determinant
    const float2* f = cell[0].f;
    return __fmaf_rn(f[v].x - f[u].x, f[w].y - f[u].y, -__fmul_rn(f[v].y - f[u].y, f[w].x - f[u].x));
  }
  static int decided(float o) { return o > geo.T ? 1 : o < -geo.T ? -1 : 0; }
  static int test() {
    std::mt19937 rng(7 * G);
    std::uniform_real_distribution<double> U(0.0, 2.0);
    int cells = 0, order = 0, sign = 0;
    for (long t = 0; t < 4000000 && cells < 200; ++t) {
      n = 6 + 2 * (int)(rng() % (G / 2 - 2));
      if (n > G) n = G;
      float M = 0.0f;
      for (int k = 0; k < n; ++k) {
        const double a = 6.283185307179586 * k / n;
        x[k] = 1.0 + 0.9 * std::cos(a) + 0.1 * (U(rng) - 1.0), y[k] = 1.0 + 0.9 * std::sin(a) + 0.1 * (U(rng) - 1.0);
        cell[0].f[k] = float2{(float)x[k], (float)y[k]};
        M = std::fmax(M, std::fmax(cell[0].f[k].x, cell[0].f[k].y));
      }
      geo = Geo{x, y, 80.0f * 5.9604645e-8f * M * M * 1.0001f + 16.0f * 2.910383e-11f * M};
      const int u = (int)(rng() % (unsigned)(n / 2)), v = u + n / 2;
      int w = (int)(rng() % (unsigned)n);
      while (w == u || w == v) w = (w + 1) % n;
      // w beside the line u v, the band's width away
      const double s = 0.2 + 0.3 * U(rng), dx = x[v] - x[u], dy = y[v] - y[u], d = (rng() & 1 ? 1.0 : -1.0) * geo.T / (dx * dx + dy * dy);
      x[w] = x[u] + s * dx - d * dy, y[w] = y[u] + s * dy + d * dx;
      cell[0].f[w] = float2{(float)x[w], (float)y[w]};
      if (decided(det(u, v, w)) == -decided(det(v, u, w))) continue;
      ++cells;
      // the cycle 0 .. n - 1 as the constraints
      for (int k = 0; k < n; ++k) cell[0].adj[k] = (1u << ((k + 1) % n)) | (1u << ((k + n - 1) % n)), cell[0].em[k] = 0;
      cell[0].nce = 0;
      GCell<G> got[2];
      for (int o = 0; o < 2; ++o) {
        const GCell<G> before = cell[0];
        warp::run(&lane, o == 1);
        got[o] = cell[0];
        cell[0] = before;
      }
      bool same = true, right = true;
      for (int a = 0; a < n; ++a)
        for (int b = 0; b < n; ++b) {
          if (a == b) continue;
          same = same && got[0].L[a][b] == got[1].L[a][b] && got[0].Z[a][b] == got[1].Z[a][b];
          for (int c = 0; c < n; ++c)
            if (c != a && c != b) right = right && g_sign<G, true>(got[0], geo, a, b, c) == geo.late(a, b, c);
        }
      order += !same, sign += !right;
    }
    std::printf("%d %d %d %d\n", G, cells, order, sign);
    return 0;
  }
};
template <int G> GCell<G> Run<G>::cell[32 / G];
template <int G> double Run<G>::x[G];
template <int G> double Run<G>::y[G];
template <int G> Geo Run<G>::geo;
template <int G> int Run<G>::n;

int main() { return Run<8>::test() || Run<16>::test() || Run<32>::test(); }
