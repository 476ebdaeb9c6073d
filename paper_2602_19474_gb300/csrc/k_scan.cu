// k_scan.cu -- exclusive prefix sums of u32 counts (offsets of the output
// patches, of the (cell, segment) pairs and crossing events per segment, of
// the bucket ranges).  The meshing path scans every array of a batch in one
// single-pass launch (k_mscan); the preprocessing, retriangulation and heat
// paths use the two-kernel scan (one block for small inputs).
#include "sbmt_cell.cuh"
#include "sbmt_launch.h"

namespace sbmt {

namespace {

constexpr int TILE = 2048;  // elements per tile (256 threads x 8)

// one block of 1024 threads: exclusive scan of n values, total at out[n]
__global__ void __launch_bounds__(1024) k_scan_small(const u32* in, u32* out, u32 n) {
  __shared__ u32 sh[1024];
  const u32 t = threadIdx.x;
  const u32 chunk = (n + 1023) / 1024;
  const u32 a = min(n, t * chunk), e = min(n, a + chunk);
  u32 s = 0;
  for (u32 i = a; i < e; ++i) s += in[i];
  sh[t] = s;
  __syncthreads();
  for (u32 o = 1; o < 1024; o <<= 1) {
    const u32 v = t >= o ? sh[t - o] : 0u;
    __syncthreads();
    sh[t] += v;
    __syncthreads();
  }
  u32 run = sh[t] - s;
  for (u32 i = a; i < e; ++i) {
    const u32 v = in[i];
    out[i] = run;
    run += v;
  }
  if (t == 1023) out[n] = sh[1023];
}

// Up to three arrays of one length at once (blockIdx.y: which), as two kernels:
// the tiles' sums, then the tiles, every block adding the sums before its tile
// itself.  Up to SELF_TILES tiles that costs less than a launch of one block that
// scans the sums in between (one array, caches flushed: 1.0e6 values 19 and 23 us,
// 8.0e6 59 and 64, 1.67e7 -- 8155 tiles -- 109 and 117); above, where the sums
// read grow with the square of the tiles, they are scanned (equal near 4e7 values;
// 5.0e7: 322 and 312 us).
// A value is the word itself or, with BITS, the number of its bits (of a
// bit-plane with rows of wpr words, those of columns 0 .. W; wpr 0: all).
struct Scan3 {
  const u32* in[3];
  u32* out[3];
  u32* part[3];
  int wpr, W;
};
template <bool BITS>
SBMT_DEV u32 scan_value(const Scan3& s, const u32* in, u64 i) {
  u32 v = in[i];
  if (BITS) {
    if (s.wpr > 0) {
      const int c0 = 32 * (int)((u32)i % (u32)s.wpr);
      if (s.W - c0 < 31) v &= (2u << (s.W - c0)) - 1u;
    }
    v = __popc(v);
  }
  return v;
}
template <bool BITS>
__global__ void __launch_bounds__(256) k_tile_sums(Scan3 s, u32 n) {
  __shared__ u32 s_sh[8];
  const u32* in = s.in[blockIdx.y];
  const u64 i0 = (u64)blockIdx.x * TILE + threadIdx.x;
  u32 sum = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (i0 + 256 * u < n) sum += scan_value<BITS>(s, in, i0 + 256 * u);
  u32 tot;
  block_exscan256(sum, &tot, s_sh);
  if (threadIdx.x == 0) s.part[blockIdx.y][blockIdx.x] = tot;
}
template <bool BITS, bool SCANNED>
__global__ void __launch_bounds__(256) k_tile_scan(Scan3 s, u32 n) {
  __shared__ u32 s_sh[8];
  const u32* in = s.in[blockIdx.y];
  const u32* part = s.part[blockIdx.y];
  u32* out = s.out[blockIdx.y];
  const u64 i0 = (u64)blockIdx.x * TILE + 8 * threadIdx.x;
  u32 v[8], sum = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    v[u] = i0 + u < n ? scan_value<BITS>(s, in, i0 + u) : 0u;
    sum += v[u];
  }
  u32 prefix;
  if (SCANNED) {
    prefix = part[blockIdx.x];
  } else {
    u32 before = 0;
    for (u32 k = threadIdx.x; k < blockIdx.x; k += 256) before += part[k];
    block_exscan256(before, &prefix, s_sh);
  }
  u32 tot;
  u32 run = block_exscan256(sum, &tot, s_sh) + prefix;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    if (i0 + u < n) out[i0 + u] = run;
    run += v[u];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 255) out[n] = run;
}

constexpr u32 SELF_TILES = 8192;  // up to this many tiles a block adds the sums before it itself

template <bool BITS>
int run_scan(const Scan3& s, int arrays, u32 n, cudaStream_t st) {
  const u32 tiles = n / TILE + 1;
  k_tile_sums<BITS><<<dim3(tiles, arrays), 256, 0, st>>>(s, n);
  if (tiles <= SELF_TILES) {
    k_tile_scan<BITS, false><<<dim3(tiles, arrays), 256, 0, st>>>(s, n);
    return 2;
  }
  for (int k = 0; k < arrays; ++k) k_scan_small<<<1, 1024, 0, st>>>(s.part[k], s.part[k], tiles);
  k_tile_scan<BITS, true><<<dim3(tiles, arrays), 256, 0, st>>>(s, n);
  return 2 + arrays;
}

// ---------------------------------------------------------------------------
// Batched single-pass scan: every tile of every scan job in one launch.
// Tiles take their order from a ticket counter (so a tile's predecessors
// were started before it), publish their sum, and look back over their
// predecessors' published sums (decoupled look-back): a tile's flag word is
// status << 32 | value, status 1 = the tile's own sum, 2 = the inclusive
// prefix through the tile, 3 = an error upstream.  Every wait is bounded by
// the global timer; a wait that runs out records ERR_TIMEOUT in the job's
// error word and publishes status 3, so that the tiles after it stop at once.
// ---------------------------------------------------------------------------
constexpr unsigned long long FLAG_AGG = 1ull << 32, FLAG_INC = 2ull << 32, FLAG_ERR = 3ull << 32;
constexpr unsigned long long WAIT_LIMIT_NS = 1000000000ull;  // one second

SBMT_DEV unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__global__ void __launch_bounds__(256) k_mscan(const ScanJob* __restrict__ sj, const u32* __restrict__ tpre,
                                               int nsj, unsigned long long* flags, u32* ticket, u32 stall_tile) {
  __shared__ u32 s_sh[8];
  __shared__ u32 s_tile, s_prefix;
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
  __syncthreads();
  const u32 tile = s_tile;
  const int k = job_of(tpre, nsj, tile);
  const ScanJob J = sj[k];
  const u32 t = tile - tpre[k];
  const u64 base = (u64)t * MSCAN_TILE;
  const u32 n = J.n_dev ? min(*J.n_dev, J.n) : J.n;
  if (base > n) {
    // past the end of a scan whose length is known on the device only: no
    // output, and nothing after it waits for a value from here
    if (threadIdx.x == 0) atomicExch(flags + tile, FLAG_INC);
    return;
  }
  u32 v[8], s = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const u64 i = base + (u64)threadIdx.x * 8 + u;
    v[u] = i < n ? J.in[i] : 0u;
    s += v[u];
  }
  u32 tot;
  const u32 ex = block_exscan256(s, &tot, s_sh);
  if (threadIdx.x == 0) {
    const bool stall = tile == stall_tile;
    volatile unsigned long long* vf = flags;
    u32 prefix = 0;
    bool bad = false;
    if (t > 0) {
      if (!stall) atomicExch(flags + tile, FLAG_AGG | tot);
      unsigned long long t0 = 0;
      for (u32 p = tile - 1;;) {
        const unsigned long long f = vf[p];
        const unsigned long long st = f & (3ull << 32);
        if (st == 0) {
          const unsigned long long now = global_ns();
          if (t0 == 0) t0 = now;
          if (now - t0 > WAIT_LIMIT_NS) {
            bad = true;
            atomicOr(J.err, ERR_TIMEOUT);
            break;
          }
          __nanosleep(128);
          continue;
        }
        if (st == FLAG_ERR) {
          bad = true;
          break;
        }
        prefix += (u32)f;
        if (st == FLAG_INC) break;
        --p;  // an aggregate: keep looking back (tile 0 of a job always publishes its prefix)
        t0 = 0;
      }
    }
    if (!stall) atomicExch(flags + tile, bad ? FLAG_ERR : (FLAG_INC | (u32)(prefix + tot)));
    s_prefix = prefix;
  }
  __syncthreads();
  u32 run = s_prefix + ex;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const u64 i = base + (u64)threadIdx.x * 8 + u;
    if (i <= n) {
      J.out[i] = run;
      if (J.out2) J.out2[i] = run;
      if (J.big && i < n && v[u] > J.big_thr) J.big[atomicAdd(J.nbig, 1u)] = make_uint2((u32)J.img, (u32)i);
    }
    run += v[u];
  }
}

}  // namespace

size_t scan_scratch_words(u32 n) { return (size_t)n / TILE + 2; }

int launch_scan(const u32* in, u32* out, u32 n, u32* scratch, cudaStream_t st) {
  if (n <= 4096) {
    k_scan_small<<<1, 1024, 0, st>>>(in, out, n);
    return 1;
  }
  Scan3 s{};
  s.in[0] = in, s.out[0] = out, s.part[0] = scratch;
  return run_scan<false>(s, 1, n, st);
}

int launch_scan_bits(const u32* in, int wpr, int W, u32* out, u32 n, u32* scratch, cudaStream_t st) {
  Scan3 s{};
  s.in[0] = in, s.out[0] = out, s.part[0] = scratch, s.wpr = wpr, s.W = W;
  return run_scan<true>(s, 1, n, st);
}

size_t scan3_scratch_words(u32 n) { return 3 * scan_scratch_words(n); }

int launch_scan3(const u32* const in[3], u32* const out[3], u32 n, u32* scratch, cudaStream_t st) {
  Scan3 s{};
  for (int k = 0; k < 3; ++k) s.in[k] = in[k], s.out[k] = out[k], s.part[k] = scratch + k * scan_scratch_words(n);
  return run_scan<false>(s, 3, n, st);
}

int launch_mscan(const ScanJob* sj, const u32* tpre, int nsj, u32 ntiles, unsigned long long* flags, u32* ticket,
                 u32 stall_tile, cudaStream_t st) {
  if (ntiles == 0) return 0;
  k_mscan<<<ntiles, 256, 0, st>>>(sj, tpre, nsj, flags, ticket, stall_tile);
  return 1;
}

}  // namespace sbmt
