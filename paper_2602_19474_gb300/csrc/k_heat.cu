// k_heat.cu -- transient heat diffusion on a label region of a finished mesh
// (App. H): du/dt = alpha Lap u on the triangles of one label, u = 0 on the
// region's boundary, from a Gaussian pulse.
//
// Linear finite elements: the cotangent stiffness K (a triangle with angle
// theta_k at corner k couples the ends i, j of the opposite edge with
// -cot(theta_k) / 2 and adds cot(theta_k) / 2 to both diagonals), the lumped
// mass M (a third of each incident triangle's area), backward Euler in time:
// (M + alpha dt K) u_{n+1} = M u_n on the free vertices (those of the region
// not on a triangle of another label).  Each step is solved by conjugate
// gradients with the diagonal as preconditioner.  The operator is assembled
// once per call into sparse rows over the free vertices (from one record per
// region triangle), so that each product is a gather with no atomics.
// Double precision throughout.  The result does not depend on the order in
// which threads run: records are placed by a scan, each free vertex's mass
// and diagonal are gathered over its incident records in record order, the
// rows' entries are sorted by column, and every sum over the grid adds the
// blocks' partial sums in one fixed order.
#include <algorithm>
#include <cstring>
#include <vector>

#include "sbmt_dev.cuh"
#include "sbmt_launch.h"

namespace sbmt {

namespace {

constexpr int HB = 256;  // threads per block

// one region triangle: its corners and the weights cot(theta_k) / 2 of the
// edges opposite each corner
struct HeatTri {
  int v[3];
  int pad;
  double w[3];
  double third;  // a third of the triangle's area
};

__global__ void __launch_bounds__(HB) k_heat_flags(const int* tri, const unsigned short* label, u64 T, int L,
                                                   u32* flag) {
  for (u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += (u64)gridDim.x * blockDim.x) {
    const u32 f = label[t] == (unsigned short)L ? 1u : 2u;
#pragma unroll
    for (int k = 0; k < 3; ++k) atomicOr(flag + tri[3 * t + k], f);
  }
}

// free vertices (flag 1) as 0/1 for the scan that numbers them
__global__ void __launch_bounds__(HB) k_heat_free(u64 V, u32* flag) {
  for (u64 v = (u64)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (u64)gridDim.x * blockDim.x)
    flag[v] = flag[v] == 1u ? 1u : 0u;
}

// the free vertices in id order (fidx: exclusive scan of the 0/1 flags)
__global__ void __launch_bounds__(HB) k_heat_list(u64 V, const u32* free01, const u32* fidx, u32* list) {
  for (u64 v = (u64)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (u64)gridDim.x * blockDim.x)
    if (free01[v]) list[fidx[v]] = (u32)v;
}

// region triangles as 0/1 flags, for the scan that places their records
__global__ void __launch_bounds__(HB) k_heat_tflag(const unsigned short* label, u64 T, int L, u32* tf) {
  for (u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += (u64)gridDim.x * blockDim.x)
    tf[t] = label[t] == (unsigned short)L ? 1u : 0u;
}

// the region's triangles: records (corners as free indices, -1 for
// boundary vertices) at their scan positions, in triangle order, and the
// number of records at each free vertex
__global__ void __launch_bounds__(HB) k_heat_setup(const double* xy, const int* tri, const unsigned short* label,
                                                   u64 T, int L, const u32* free01, const u32* fidx, const u32* tpos,
                                                   HeatTri* rec, u32* vcnt) {
  const double2* p = reinterpret_cast<const double2*>(xy);
  for (u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += (u64)gridDim.x * blockDim.x) {
    if (label[t] != (unsigned short)L) continue;
    HeatTri h;
    double2 c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int v = tri[3 * t + k];
      c[k] = p[v];
      h.v[k] = free01[v] ? (int)fidx[v] : -1;
    }
    h.pad = 0;
    const double cross = fabs((c[1].x - c[0].x) * (c[2].y - c[0].y) - (c[1].y - c[0].y) * (c[2].x - c[0].x));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double2 a = c[k], b = c[(k + 1) % 3], d = c[(k + 2) % 3];
      const double dot = (b.x - a.x) * (d.x - a.x) + (b.y - a.y) * (d.y - a.y);
      h.w[k] = 0.5 * dot / cross;  // cot(theta_k) / 2 = (u . v) / (2 |u x v|)
    }
    h.third = cross / 6.0;  // a third of the area |u x v| / 2
    rec[tpos[t]] = h;
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (h.v[k] >= 0) atomicAdd(vcnt + h.v[k], 1u);
  }
}

// each free vertex's incident records (record index * 4 + corner), placed
// at cursors from the scan of the counts; sorted afterwards
__global__ void __launch_bounds__(HB) k_heat_inc(const HeatTri* rec, u32 nr, u32* cur, u32* inc) {
  for (u32 t = blockIdx.x * blockDim.x + threadIdx.x; t < nr; t += gridDim.x * blockDim.x) {
    const HeatTri h = rec[t];
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (h.v[k] >= 0) inc[atomicAdd(cur + h.v[k], 1u)] = 4 * t + (u32)k;
  }
}

// per free vertex, in record order: the lumped mass (a third of each
// incident triangle's area |u x v| / 2) and the stiffness diagonal (the
// weights of the two edges at the vertex)
__global__ void __launch_bounds__(HB) k_heat_gather(const HeatTri* rec, u32 n, const u32* vptr, u32* inc,
                                                    double* mass, double* kdiag) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const u32 e0 = vptr[i], e1 = vptr[i + 1];
    for (u32 a = e0 + 1; a < e1; ++a)  // insertion sort: a vertex has few records
      for (u32 b = a; b > e0 && inc[b] < inc[b - 1]; --b) {
        const u32 t = inc[b];
        inc[b] = inc[b - 1], inc[b - 1] = t;
      }
    double m = 0.0, d = 0.0;
    for (u32 e = e0; e < e1; ++e) {
      const HeatTri h = rec[inc[e] >> 2];
      const int c = (int)(inc[e] & 3u);
      m += h.third;
      // the edges at corner c are those opposite corners c + 1 and c + 2
      d += h.w[(c + 1) % 3];
      d += h.w[(c + 2) % 3];
    }
    mass[i] = m;
    kdiag[i] = d;
  }
}

// the free vertices: the pulse, the operator's inverse diagonal
__global__ void __launch_bounds__(HB) k_heat_init(const double* xy, u32 n, const u32* list, const double* mass,
                                                  const double* kdiag, double tau, double x0, double y0,
                                                  double s2, double amp, double* x, double* dg, double* dinv) {
  const double2* p = reinterpret_cast<const double2*>(xy);
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double2 c = p[list[i]];
    const double dx = c.x - x0, dy = c.y - y0;
    x[i] = amp * exp(-(dx * dx + dy * dy) / (2.0 * s2));
    dg[i] = mass[i] + tau * kdiag[i];
    dinv[i] = 1.0 / dg[i];
  }
}

// the operator as sparse rows over the free vertices: two entries per
// region-triangle edge with both ends free, -tau cot/2 each (an edge shared
// by two region triangles gives two entries for the same neighbour, merged
// afterwards); the diagonal is kept apart
__global__ void __launch_bounds__(HB) k_heat_rowcount(const HeatTri* rec, u32 n, u32* cnt) {
  for (u32 t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const HeatTri h = rec[t];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int i = h.v[(k + 1) % 3], j = h.v[(k + 2) % 3];
      if (i >= 0 && j >= 0) atomicAdd(cnt + i, 1u), atomicAdd(cnt + j, 1u);
    }
  }
}
__global__ void __launch_bounds__(HB) k_heat_fill(const HeatTri* rec, u32 n, double tau, u32* cur, u32* col,
                                                  double* val) {
  for (u32 t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const HeatTri h = rec[t];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int i = h.v[(k + 1) % 3], j = h.v[(k + 2) % 3];
      if (i < 0 || j < 0) continue;
      const double w = -tau * h.w[k];
      const u32 a = atomicAdd(cur + i, 1u), b = atomicAdd(cur + j, 1u);
      col[a] = (u32)j, val[a] = w;
      col[b] = (u32)i, val[b] = w;
    }
  }
}

// each row's entries of one column summed, in place at the row's start;
// mcnt: the merged counts.  A row of at most MR entries (two per neighbour) is
// merged and ordered in a column of shared memory of its thread's own: in
// place, each step waited for the one before through the cache (128 us for
// 0.38e6 rows, 47 this way).
constexpr int MR = 16, MT = 192;
SBMT_DEV u32 merge_row(u32 n, u32* col, double* val, u32 step) {
  u32 m = 0;
  for (u32 e = 0; e < n; ++e) {
    const u32 c = col[e * step];
    const double v = val[e * step];
    u32 k = 0;
    while (k < m && col[k * step] != c) ++k;
    if (k < m) {
      val[k * step] += v;
    } else {
      col[m * step] = c, val[m * step] = v;
      ++m;
    }
  }
  // the row's entries by column, so that each product sums them in one order
  for (u32 a = 1; a < m; ++a) {
    const u32 c = col[a * step];
    const double v = val[a * step];
    u32 b = a;
    for (; b > 0 && c < col[(b - 1) * step]; --b)
      col[b * step] = col[(b - 1) * step], val[b * step] = val[(b - 1) * step];
    col[b * step] = c, val[b * step] = v;
  }
  return m;
}
__global__ void __launch_bounds__(MT) k_heat_merge(u32 n, const u32* rowptr, u32* col, double* val, u32* mcnt) {
  __shared__ double s_val[MR][MT];
  __shared__ u32 s_col[MR][MT];
  u32* sc = &s_col[0][threadIdx.x];
  double* sv = &s_val[0][threadIdx.x];
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const u32 e0 = rowptr[i], cnt = rowptr[i + 1] - e0;
    if (cnt > MR) {
      mcnt[i] = merge_row(cnt, col + e0, val + e0, 1);
      continue;
    }
#pragma unroll 4
    for (u32 e = 0; e < cnt; ++e) sc[e * MT] = col[e0 + e], sv[e * MT] = val[e0 + e];
    const u32 m = merge_row(cnt, sc, sv, MT);
    for (u32 e = 0; e < m; ++e) col[e0 + e] = sc[e * MT], val[e0 + e] = sv[e * MT];
    mcnt[i] = m;
  }
}

// The merged rows again for the solver, in slices of 32 rows (one warp):
// entry k < SW of row i at slice (i / 32), place 32 k + i % 32, so that a
// warp reads its rows' k-th entries as one contiguous piece.  The first SF
// are there for every row (absent ones name the row itself), so that the
// solver loads them without waiting for the row's count.  Entries from SW on
// (rows of more than SW neighbours, few on these meshes) stay in the rows.
constexpr int SW = 8, SF = 6;
__global__ void __launch_bounds__(HB) k_heat_slices(u32 n, const u32* rowptr, const u32* mcnt, const u32* col,
                                                    const double* val, double* sval, u32* scol) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const u32 e0 = rowptr[i], m = min(mcnt[i], (u32)SW);
    const size_t at = (size_t)(i >> 5) * (32 * SW) + (i & 31u);
    for (u32 k = 0; k < max(m, (u32)SF); ++k) {
      scol[at + 32 * k] = k < m ? col[e0 + k] : i;
      sval[at + 32 * k] = k < m ? val[e0 + k] : 0.0;
    }
  }
}

// u over the mesh: 0, then the free values at their vertices
__global__ void __launch_bounds__(HB) k_heat_zero(u64 V, double* u) {
  for (u64 v = (u64)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (u64)gridDim.x * blockDim.x) u[v] = 0.0;
}
__global__ void __launch_bounds__(HB) k_heat_put(u32 n, const u32* list, const double* x, double* u) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) u[list[i]] = x[i];
}

// ---------------------------------------------------------------------------
// The time steps: one cooperative launch for the whole call, one block of 512
// threads on each SM (fewer for small regions), all resident, so that a phase
// of the solver ends in a barrier across the grid instead of a launch, and the
// host reads nothing until the last step.  Each block keeps the same rows
// throughout, their vectors in shared memory.  Per iteration:
//   q = A z + beta q, p = z + beta p; p.q        | barrier
//   r, z; r.z (and r.r every eighth time)        | barrier, x meanwhile
// What an iteration costs is this GPU's FP64 rate, about 1.6 instructions per
// clock and SM (13 per row of 6 entries), and the two barriers.  So: the product
// is taken of z, which is final before beta is known, and p and q follow by
// recurrence, which saves the barrier that a new p would need before the next
// product; no work that only sometimes counts (r.r); a block's sums through shared
// memory in halves (a dependent FP64 add is some 100 clocks); the blocks' sums
// published and awaited in one step, which is the barrier (below), and
// added in one fixed order; one division per block.
// Measured on 0.38e6 free vertices (4096^2 Voronoi labels, h = 2), clocks of an
// iteration: products 14e3 and residuals 4.5e3 (both the FP64 rate), barriers
// 9e3 and 11e3.  The call took 8.4 ms with three barriers and the vectors in L2 and
// 5.8 ms now on the same GPU (5.9 and 4.2 ms on another).  Sums by integer limbs
// instead of FP64 trees, every block waiting for all slots, and a smaller share of rows
// for block 0 gained nothing.
// ---------------------------------------------------------------------------
constexpr int CT = 512;         // threads per block
constexpr int CG_BLOCKS = 152;  // the most blocks: one per SM of this GPU
constexpr int CG_SUMS = 3;      // the most sums a barrier carries
constexpr int SLOT_WORDS = 4 * CG_SUMS * CG_BLOCKS + 16 * CG_BLOCKS;
struct HeatCg {
  u32 n, nsteps;
  u32 block_rows;  // the most rows a block has, in whole slices
  int maxit, sliced;
  u32 stall;  // test of the wait's bound: the last block publishes nothing at this barrier (1, 2, ...)
  double tol;
  const u32* rowptr;
  const u32* mcnt;
  const u32* col;
  const double* val;
  const u32* scol;
  const double* sval;
  const double* mass;
  const double* dg;
  const double* dinv;
  double *x, *r, *z, *p, *q, *b;
  unsigned long long* slot;  // SLOT_WORDS published sums, all bits set at first
  u32* fail;                 // a wait ran out
  unsigned long long* peak;  // per step: the maximum of x (double bits), 0 at least
  int* iters;                // per step
  int* done;                 // [0] steps finished, [1] the last one converged
};
constexpr unsigned long long CG_EMPTY = ~0ull;  // no sum has these bits

SBMT_DEV unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
SBMT_DEV void st_relaxed(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// orders this thread's accesses (and those it has seen through a block
// barrier) across the grid
SBMT_DEV void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// waits until K words are no longer empty; bounded by the global timer (two
// seconds), after which the failure word is set and every wait ends
template <int K>
SBMT_DEV bool wait_words(const HeatCg& h, const unsigned long long* p, size_t step, unsigned long long (&w)[K]) {
  unsigned long long t0 = 0;
  u32 spins = 0;
  while (true) {
    bool wait = false;
#pragma unroll
    for (int k = 0; k < K; ++k) w[k] = ld_acquire(p + k * step);
#pragma unroll
    for (int k = 0; k < K; ++k) wait |= w[k] == CG_EMPTY;
    if (!wait) return true;
    if ((++spins & 1023u) == 0) {
      unsigned long long clk;
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(clk));
      if (t0 == 0) t0 = clk;
      if (clk - t0 > 2000000000ull) atomicExch(h.fail, 1u);
      if (atomicAdd(h.fail, 0u)) return false;
    }
  }
}

// The grid's sums of K values per thread into s_out, and a barrier across the
// grid: what a block's threads wrote before it is seen by every block after
// it.  (TREE false: the barrier alone.)  A block publishes its sums in its
// slots once its writes are fenced; block 0's thread b waits for block b's,
// block 0 adds them (lane l takes blocks l, l + 32, ..., then a fixed tree)
// and hands them to each block in a slot of its own, so that nobody but block
// 0 reads more than one place (every block waiting for all 152 slots took 5 us
// a barrier, 3 us this way).  Four buffers by turns: entering barrier g, a
// block empties its slots of buffer (g + 2) % 4.  Those held barrier g - 2,
// which it has left (and block 0 had read its sums before that), and they are
// not written before it publishes barrier g + 2.  mid() runs between publishing
// and waiting, end(sums) on one thread before the block goes on.  False when a wait ran out.
template <int K, bool TREE, class Mid, class End>
SBMT_DEV bool grid_sums(const HeatCg& h, const double (&v)[K], u32& gen, double (*s)[CT], double* s_out, int* s_fail,
                        const Mid& mid, const End& end) {
  const u32 tid = threadIdx.x;
  double t[K];
#pragma unroll
  for (int k = 0; k < K; ++k) t[k] = 0.0;
  if (tid == 0) *s_fail = 0;
  if (TREE) {
#pragma unroll
    for (int k = 0; k < K; ++k) s[k][tid] = v[k];
    __syncthreads();
    if (tid < CT / 4) {
#pragma unroll
      for (int k = 0; k < K; ++k)
        s[k][tid] = (s[k][tid] + s[k][tid + CT / 4]) + (s[k][tid + CT / 2] + s[k][tid + 3 * CT / 4]);
    }
    __syncthreads();
    if (tid < 32) {
      static_assert(CT == 512, "the second step adds four values per lane");
#pragma unroll
      for (int k = 0; k < K; ++k) t[k] = (s[k][tid] + s[k][tid + 32]) + (s[k][tid + 64] + s[k][tid + 96]);
      for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < K; ++k) t[k] += __shfl_xor_sync(0xFFFFFFFFu, t[k], o);
      }
    }
  } else {
    __syncthreads();
  }
  if (gridDim.x > 1) {
    // in: [buffer][sum][block]; out: [buffer][block][4], a sector per block
    unsigned long long* in = h.slot + (size_t)(gen & 3u) * CG_SUMS * CG_BLOCKS;
    unsigned long long* in2 = h.slot + (size_t)((gen + 2) & 3u) * CG_SUMS * CG_BLOCKS;
    unsigned long long* out = h.slot + 4 * CG_SUMS * CG_BLOCKS + (size_t)(gen & 3u) * 4 * CG_BLOCKS;
    unsigned long long* out2 = h.slot + 4 * CG_SUMS * CG_BLOCKS + (size_t)((gen + 2) & 3u) * 4 * CG_BLOCKS;
    if (tid == 0) {
#pragma unroll
      for (int k = 0; k < CG_SUMS; ++k)
        st_relaxed(in2 + k * CG_BLOCKS + blockIdx.x, CG_EMPTY), st_relaxed(out2 + 4 * blockIdx.x + k, CG_EMPTY);
      fence_gpu();
      if (gen + 1 != h.stall || blockIdx.x != gridDim.x - 1) {
#pragma unroll
        for (int k = 0; k < K; ++k)
          st_relaxed(in + k * CG_BLOCKS + blockIdx.x, (unsigned long long)__double_as_longlong(t[k]));
      }
    }
    mid();
    if (blockIdx.x == 0) {
      __syncthreads();  // the tree's last reads of s
      if (tid < gridDim.x) {
        unsigned long long w[K];
        if (!wait_words<K>(h, in + tid, CG_BLOCKS, w)) *s_fail = 1;
#pragma unroll
        for (int k = 0; k < K; ++k) s[k][tid] = __longlong_as_double((long long)w[k]);
      }
      __syncthreads();
      if (TREE && tid < 32) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
          t[k] = 0.0;
          for (u32 b = tid; b < gridDim.x; b += 32) t[k] += s[k][b];
        }
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
          for (int k = 0; k < K; ++k) t[k] += __shfl_xor_sync(0xFFFFFFFFu, t[k], o);
        }
        if (tid == 0) {
#pragma unroll
          for (int k = 0; k < K; ++k) s_out[k] = t[k];
        }
      }
      if (TREE) __syncthreads();
      if (tid > 0 && tid < gridDim.x) {
        fence_gpu();
#pragma unroll
        for (int k = 0; k < K; ++k)
          st_relaxed(out + 4 * tid + k, TREE ? (unsigned long long)__double_as_longlong(s_out[k]) : 0ull);
      }
    } else if (tid == 0) {
      unsigned long long w[K];
      if (!wait_words<K>(h, out + 4 * blockIdx.x, 1, w)) *s_fail = 1;
#pragma unroll
      for (int k = 0; k < K; ++k) t[k] = __longlong_as_double((long long)w[k]);
    }
  }
  if (gridDim.x == 1) mid();
  if (TREE && tid == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) s_out[k] = t[k];
    end(t);
  }
  ++gen;
  __syncthreads();
  return *s_fail == 0;
}

// Row i of A = M + tau K times v (v read from L2: other SMs write it); dd: the
// diagonal's part.  A warp's lanes hold the 32 rows of one slice.  (Two or
// three rows in flight per thread were no faster: 16 warps hide the loads behind
// the FP64 pipe's 19 clocks an instruction.)
SBMT_DEV double row_times(const HeatCg& h, u32 i, const double* v, double dd) {
  const u32 m = h.mcnt[i];
  double a = dd;
  u32 k0 = 0;
  if (h.sliced) {
    double w[SF], g[SF];
    const size_t at = (size_t)(i >> 5) * (32 * SW) + (i & 31u);
#pragma unroll
    for (int k = 0; k < SF; ++k) w[k] = h.sval[at + 32 * k], g[k] = __ldcg(v + h.scol[at + 32 * k]);
#pragma unroll
    for (int k = 0; k < SF; ++k)
      if ((u32)k < m) a += w[k] * g[k];
    for (u32 k = SF; k < min(m, (u32)SW); ++k) a += h.sval[at + 32 * k] * __ldcg(v + h.scol[at + 32 * k]);
    k0 = SW;
  }
  if (k0 < m)
    for (u32 e = h.rowptr[i] + k0, e1 = h.rowptr[i] + m; e < e1; ++e) a += h.val[e] * __ldcg(v + h.col[e]);
  return a;
}

// Rows of a block: whole slices of 32, the same number (or one less) in every
// block, so that the FP64 pipes of all SMs finish together (rows dealt out in
// rounds of CT left most SMs idle in the last round).
SBMT_HD u32 cg_slice(u32 n, u32 block, u32 blocks) { return (u32)((u64)((n + 31) / 32) * block / blocks); }
constexpr int CG_VECS = 6;  // vectors of a block's rows held on chip
constexpr size_t CG_SMEM = 227 * 1024 - 13 * 1024;  // what a block has for them, beside its sums

// ONCHIP: the block's rows of x, r, z, p, q and the diagonals stay in shared
// memory for the whole solve (48 B a row: up to 0.69e6 free vertices); only z, which the
// product gathers, is also written through to L2.  Otherwise they stay in L2.
//
// Two barriers an iteration: the product is taken of z, which is final
// before beta is known, and q = A z + beta q, p = z + beta p follow from it, so that
// the new p needs no barrier of its own before the next product.
//
// These recurrences drift from the true residual b - A x sooner than a product
// taken of p itself: over regions of 5e3 to 5e4 vertices of a label image the
// residual a step can reach was the same at alpha dt = 5 (a step of some 50
// iterations), and at 5e4 and 5e6 (300 to 800 iterations) 1.3 to 1.6 times as
// large.  So a long step takes r = b - A x anew after ANEW iterations, 4 ANEW,
// and so on: what drifted until then is gone, and the reachable residual is
// 0.3 to 0.6 times the product form's at alpha dt = 500 and below 0.1 times at 5e4
// and above.  It costs a product and two barriers each time, none in a step of
// fewer iterations.
constexpr int ANEW = 96;  // a multiple of 8: where the residual is looked at
template <bool ONCHIP>
__global__ void __launch_bounds__(CT, 1) k_heat_cg(const __grid_constant__ HeatCg h) {
  extern __shared__ double s_vec[];
  __shared__ double s[CG_SUMS][CT];
  __shared__ double s_sum[CG_SUMS], s_k;
  __shared__ int s_fail;
  const u32 row0 = 32 * cg_slice(h.n, blockIdx.x, gridDim.x);
  const u32 rows = min(32 * cg_slice(h.n, blockIdx.x + 1, gridDim.x), h.n) - row0;
  const u32 R = h.block_rows, tid = threadIdx.x;
  double* x = ONCHIP ? s_vec : h.x + row0;
  double* r = ONCHIP ? s_vec + R : h.r + row0;
  double* z = ONCHIP ? s_vec + 2 * R : h.z + row0;
  double* p = ONCHIP ? s_vec + 3 * R : h.p + row0;
  double* q = ONCHIP ? s_vec + 4 * R : h.q + row0;
  double* dinv = ONCHIP ? s_vec + 5 * R : nullptr;
  // (a thread touches only its own rows of these: no block barrier)
  if (ONCHIP)
    for (u32 l = tid; l < rows; l += CT) x[l] = h.x[row0 + l], dinv[l] = h.dinv[row0 + l];
  auto dinv_at = [&](u32 l) { return ONCHIP ? dinv[l] : h.dinv[row0 + l]; };
  u32 gen = 0;
  for (u32 step = 0; step < h.nsteps; ++step) {
    double rz = 0.0, rr = 0.0, be = 0.0, stop = 0.0;
    int it = 0, anew = ANEW;
    bool first = true;
    while (true) {
      // b = M x; r = b - A x, z = D^-1 r; r.z, r.r, b.b.  Later in the step, r anew in
      // the place of the recurrence's: the direction goes on
      if (!first) {
        if (ONCHIP)
          for (u32 l = tid; l < rows; l += CT) h.x[row0 + l] = x[l];
        const double none[1] = {0.0};  // (x of all blocks is there after the barrier)
        if (!grid_sums<1, false>(h, none, gen, s, s_sum, &s_fail, [] {}, [](const double*) {})) return;
      }
      double a3[3] = {0.0, 0.0, 0.0};
      for (u32 l = tid; l < rows; l += CT) {
        const u32 i = row0 + l;
        const double xi = x[l], bi = first ? h.mass[i] * xi : h.b[i], dd = h.dg[i] * xi;
        const double qi = row_times(h, i, h.x, dd);
        const double di = dinv_at(l), rv = di != 0.0 ? bi - qi : 0.0, zv = rv * di;
        r[l] = rv, z[l] = zv;
        if (first) p[l] = 0.0, q[l] = 0.0, h.b[i] = bi;
        if (ONCHIP) h.z[i] = zv;
        a3[0] += rv * zv, a3[1] += rv * rv, a3[2] += bi * bi;
      }
      if (!grid_sums<3, true>(h, a3, gen, s, s_sum, &s_fail, [] {},
                              [&](const double* t) { s_k = rz != 0.0 ? be * (t[0] / rz) : 0.0; }))
        return;
      rz = s_sum[0], rr = s_sum[1], be = s_k;
      if (first) stop = h.tol * h.tol * s_sum[2];
      first = false;
      while (rr > stop && it < h.maxit && it != anew) {
        bool look = false;
        while (!look) {
          double a1[1] = {0.0};
          for (u32 l = tid; l < rows; l += CT) {
            // (the diagonal times z is r, up to z's rounding)
            const double qv = row_times(h, row0 + l, h.z, r[l]) + be * q[l], pv = z[l] + be * p[l];
            q[l] = qv, p[l] = pv;
            a1[0] += pv * qv;
          }
          if (!grid_sums<1, true>(h, a1, gen, s, s_sum, &s_fail, [] {},
                                  [&](const double* t) { s_k = t[0] != 0.0 ? rz / t[0] : 0.0; }))
            return;
          const double al = s_k;
          ++it;
          look = (it & 7) == 0 || it == h.maxit;  // the residual is looked at (and summed) every eighth iteration
          double a2[2] = {0.0, 0.0};
          for (u32 l0 = tid; l0 < rows; l0 += 3 * CT) {
            double rv[3], qv[3], dv[3];
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              const u32 l = l0 + u * CT;
              if (l < rows) rv[u] = r[l], qv[u] = q[l], dv[u] = dinv_at(l);
            }
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              const u32 l = l0 + u * CT;
              if (l >= rows) continue;
              const double rn = rv[u] - al * qv[u], zn = rn * dv[u];
              r[l] = rn, z[l] = zn;
              if (ONCHIP) h.z[row0 + l] = zn;
              a2[0] += rn * zn;
              if (look) a2[1] += rn * rn;
            }
          }
          // (x is not needed before the next step: updated while the sums travel)
          auto update_x = [&] {
#pragma unroll 4
            for (u32 l = tid; l < rows; l += CT) x[l] += al * p[l];
          };
          const auto beta = [&](const double* t) { s_k = rz != 0.0 ? t[0] / rz : 0.0; };
          if (look) {
            if (!grid_sums<2, true>(h, a2, gen, s, s_sum, &s_fail, update_x, beta)) return;
          } else {
            const double only[1] = {a2[0]};
            if (!grid_sums<1, true>(h, only, gen, s, s_sum, &s_fail, update_x, beta)) return;
          }
          rz = s_sum[0], be = s_k;
          if (look) rr = s_sum[1];
        }
      }
      if (!(rr > stop) || it >= h.maxit) break;
      anew *= 4;
    }
    // the step's peak (positive doubles order as their bits, infinity above all;
    // NaNs are left out, as fmax leaves them), and x for the next step's product
    unsigned long long top = 0;
    for (u32 l = tid; l < rows; l += CT) {
      const double xv = x[l];
      if (ONCHIP) h.x[row0 + l] = xv;
      const long long bits = __double_as_longlong(xv);
      if (bits > 0 && bits <= 0x7FF0000000000000ll) top = max(top, (unsigned long long)bits);
    }
    for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
    if ((threadIdx.x & 31) == 0 && top) atomicMax(h.peak + step, top);
    if (blockIdx.x == 0 && threadIdx.x == 0)
      h.iters[step] = it, h.done[0] = (int)step + 1, h.done[1] = rr > stop ? 0 : 1;
    if (rr > stop) return;
    if (step + 1 == h.nsteps) return;
    const double none[1] = {0.0};
    if (!grid_sums<1, false>(h, none, gen, s, s_sum, &s_fail, [] {}, [](const double*) {})) return;
  }
}

unsigned grid_v(u64 n) { return (unsigned)std::max<u64>(1, std::min<u64>((n + HB - 1) / HB, 152 * 8)); }

}  // namespace

size_t heat_scratch_bytes(u64 T, u64 V, int nsteps) {
  return 256 * 32 + T * (sizeof(HeatTri) + 6 * (4 + 8) + 4 + 4 + 12) + V * (4 + 4 + 4 + 4 + 4 + 4 + 4 + 8 * 10) +
         8 * SLOT_WORDS + 12 * (size_t)std::max(nsteps, 1) + 64 +
         4 * scan_scratch_words((u32)std::min<u64>(std::max(T, V), 0xFFFFFFFFu));
}

int heat_solve(const double* xy, const int* tri, const unsigned short* label, u64 T, u64 V, int L, double alpha,
               double dt, int nsteps, double x0, double y0, double sigma, double amp, double tol, int maxit,
               double* u, double* peaks, int* iters, int max_blocks, int stall, void* scratch, cudaStream_t st) {
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  char* s = (char*)scratch;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = s + off;
    off = up(off + bytes);
    return p;
  };
  HeatTri* rec = (HeatTri*)take(T * sizeof(HeatTri));
  u32* flag = (u32*)take(4 * V);
  u32* fidx = (u32*)take(4 * (V + 1));
  u32* list = (u32*)take(4 * V);
  u32* tf = (u32*)take(4 * T);          // region triangles as 0/1
  u32* tpos = (u32*)take(4 * (T + 1));  // their scan: record positions
  u32* vcnt = (u32*)take(4 * V);        // records per free vertex
  u32* vptr = (u32*)take(4 * (V + 1));  // their scan
  u32* inc = (u32*)take(4 * 3 * T);     // incident records per free vertex
  double* mass = (double*)take(8 * V);
  double* kdiag = (double*)take(8 * V);
  double* dinv = (double*)take(8 * V);
  double* dg = (double*)take(8 * V);
  u32* rowptr = (u32*)take(4 * (V + 1));
  u32* mcnt = (u32*)take(4 * V);
  u32* col = (u32*)take(4 * 6 * T);
  double* val = (double*)take(8 * 6 * T);
  double* x = (double*)take(8 * V);
  double* q = (double*)take(8 * V);
  double* r = (double*)take(8 * V);
  double* z = (double*)take(8 * V);
  double* p = (double*)take(8 * V);
  double* b = (double*)take(8 * V);
  unsigned long long* slot = (unsigned long long*)take(8 * SLOT_WORDS);
  // the solver's results: a failed wait, 0, steps done, convergence, then per
  // step the peak and the iterations
  const size_t res_bytes = 16 + 12 * (size_t)std::max(nsteps, 1);
  char* res = take(res_bytes);
  u32* sscr = (u32*)take(4 * scan_scratch_words((u32)std::max(T, V)) + 4);
  const unsigned gt = grid_v(T);
  const double tau = alpha * dt;
  int launches = 0;
  if (cudaMemsetAsync(flag, 0, 4 * V, st) || cudaMemsetAsync(res, 0, res_bytes, st) ||
      cudaMemsetAsync(slot, 0xFF, 8 * SLOT_WORDS, st))
    return -1;
  k_heat_flags<<<gt, HB, 0, st>>>(tri, label, T, L, flag);
  k_heat_free<<<grid_v(V), HB, 0, st>>>(V, flag);
  launches += 2 + launch_scan(flag, fidx, (u32)V, sscr, st);
  k_heat_list<<<grid_v(V), HB, 0, st>>>(V, flag, fidx, list);
  k_heat_tflag<<<gt, HB, 0, st>>>(label, T, L, tf);
  launches += 2 + launch_scan(tf, tpos, (u32)T, sscr, st);
  u32 n = 0, nr = 0;
  if (cudaMemcpyAsync(&n, fidx + V, 4, cudaMemcpyDeviceToHost, st) ||
      cudaMemcpyAsync(&nr, tpos + T, 4, cudaMemcpyDeviceToHost, st) || cudaStreamSynchronize(st))
    return -1;
  if (cudaMemsetAsync(vcnt, 0, 4 * (size_t)std::max<u32>(n, 1), st)) return -1;
  k_heat_setup<<<gt, HB, 0, st>>>(xy, tri, label, T, L, flag, fidx, tpos, rec, vcnt);
  const unsigned gv = grid_v(n);
  const unsigned gr = grid_v(nr);
  launches += 1;
  if (n > 0) {
    // the free vertices' incident records, sorted, then their mass and diagonal
    launches += launch_scan(vcnt, vptr, n, sscr, st);
    if (cudaMemcpyAsync(mcnt, vptr, 4 * (size_t)n, cudaMemcpyDeviceToDevice, st)) return -1;
    k_heat_inc<<<gr, HB, 0, st>>>(rec, nr, mcnt, inc);
    k_heat_gather<<<gv, HB, 0, st>>>(rec, n, vptr, inc, mass, kdiag);
    k_heat_init<<<gv, HB, 0, st>>>(xy, n, list, mass, kdiag, tau, x0, y0, sigma * sigma, amp, x, dg, dinv);
    launches += 3;
  }
  // the rows: counts (in flag, free now), their scan, then the entries at
  // cursors starting from the row offsets
  if (n > 0) {
    if (cudaMemsetAsync(flag, 0, 4 * (size_t)n, st)) return -1;
    k_heat_rowcount<<<gr, HB, 0, st>>>(rec, nr, flag);
    launches += 1 + launch_scan(flag, rowptr, n, sscr, st);
    if (cudaMemcpyAsync(flag, rowptr, 4 * (size_t)n, cudaMemcpyDeviceToDevice, st)) return -1;
    k_heat_fill<<<gr, HB, 0, st>>>(rec, nr, tau, flag, col, val);
    k_heat_merge<<<(unsigned)std::min<u64>((n + MT - 1) / MT, 152 * 6), MT, 0, st>>>(n, rowptr, col, val, mcnt);
    launches += 2;
  }
  bool converged = true;
  if (n == 0)
    for (int step = 0; step < nsteps; ++step) {
      if (iters) iters[step] = 0;
      if (peaks) peaks[step] = 0.0;
    }
  if (n > 0 && nsteps > 0) {
    // the slices take the place of the triangle records, which are done with
    const size_t sval_bytes = (size_t)((n + 31) / 32) * 32 * SW * 8;
    const bool sliced = sval_bytes + sval_bytes / 2 <= T * sizeof(HeatTri);
    double* sval = (double*)rec;
    u32* scol = (u32*)((char*)rec + sval_bytes);
    if (sliced) {
      k_heat_slices<<<gv, HB, 0, st>>>(n, rowptr, mcnt, col, val, sval, scol);
      ++launches;
    }
    unsigned long long* peak = (unsigned long long*)(res + 16);
    int* its = (int*)(peak + nsteps);
    HeatCg h{};
    h.n = n, h.nsteps = (u32)nsteps, h.maxit = maxit, h.sliced = sliced ? 1 : 0, h.tol = tol;
    h.stall = (u32)stall;
    h.rowptr = rowptr, h.mcnt = mcnt, h.col = col, h.val = val, h.scol = scol, h.sval = sval;
    h.mass = mass, h.dg = dg, h.dinv = dinv, h.x = x, h.r = r, h.z = z, h.p = p, h.q = q, h.b = b;
    h.slot = slot, h.fail = (u32*)res, h.peak = peak, h.iters = its, h.done = (int*)res + 2;
    void* args[] = {&h};
    // One block per SM, as many as the process may use at once: a launch whose
    // blocks cannot all be resident is refused, and is tried with half of them.
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) return -1;
    unsigned grid = (unsigned)std::min<u64>(std::min(CG_BLOCKS, std::max(sms, 1)), (n + CT - 1) / CT);
    if (max_blocks > 0) grid = std::min(grid, (unsigned)max_blocks);
    while (true) {
      h.block_rows = 32 * (((n + 31) / 32 + grid - 1) / grid);
      const size_t vec_bytes = (size_t)CG_VECS * 8 * h.block_rows;
      const bool onchip = vec_bytes <= CG_SMEM;
      const void* cg = onchip ? (const void*)k_heat_cg<true> : (const void*)k_heat_cg<false>;
      if (onchip && cudaFuncSetAttribute(cg, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CG_SMEM) != cudaSuccess)
        return -1;
      const cudaError_t e = cudaLaunchCooperativeKernel(cg, dim3(grid), dim3(CT), args, onchip ? vec_bytes : 0, st);
      if (e == cudaSuccess) break;
      if (e != cudaErrorCooperativeLaunchTooLarge || grid == 1) return -1;
      cudaGetLastError();
      grid /= 2;
    }
    ++launches;
    std::vector<char> hres(res_bytes);
    if (cudaMemcpyAsync(hres.data(), res, res_bytes, cudaMemcpyDeviceToHost, st) || cudaStreamSynchronize(st))
      return -1;
    const u32* words = (const u32*)hres.data();
    if (words[0]) return -3;  // a wait across the grid ran out
    const int done = (int)words[2];
    for (int step = 0; step < done; ++step) {
      if (peaks) std::memcpy(peaks + step, hres.data() + 16 + 8 * (size_t)step, 8);
      if (iters) std::memcpy(iters + step, hres.data() + 16 + 8 * (size_t)nsteps + 4 * (size_t)step, 4);
    }
    converged = words[3] != 0;
  }
  k_heat_zero<<<grid_v(V), HB, 0, st>>>(V, u);
  k_heat_put<<<std::max(gv, 1u), HB, 0, st>>>(n, list, x, u);
  launches += 2;
  if (!converged) return -2;
  return launches;
}

}  // namespace sbmt
