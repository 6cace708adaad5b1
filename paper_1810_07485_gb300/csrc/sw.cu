// Swendsen-Wang update of the two-dimensional Ising model: the benchmark on
// which the paper measures its union-find (Sec. 4.1).  Kernels, a small
// engine and the lcqmc_sw_* entry points of include/lcqmc.h.
//
// One update (L x L periodic lattice, site i = y L + x, spin s in {0, 1}):
//   bonds R(i) = (i, right) and D(i) = (i, below); the draws of site i are
//   Philox(ctr = (TAG_SWBOND << 24, i, 0, sweep), key = seed), word 0 for
//   R(i), word 1 for D(i); a bond is active iff its spins are equal and its
//   draw is below T = round(2^32 (1 - e^{-2K}));
//   clusters of active bonds, each named by its smallest site index r;
//   every cluster flips with the coin bit (r mod 128) of
//   Philox(ctr = (TAG_SWFLIP << 24, r / 128, 0, sweep)).
//
// GPU layout: 64 x 32 site tiles, one 256-thread block each; spins one bit per
// site, a 64-bit word per tile row (bytes only at the C interface).  Inside a
// row the active right bonds form runs of consecutive sites; everything a
// cluster needs is kept per run, and rows are handled as words.
//   k_sw_local  bond draws, union-find of the tile's runs in shared memory
//               (min-root hooking, one CAS), flattened: the local root of every
//               run start (its cluster's smallest site in the tile); tile-boundary
//               bonds kept as bit masks
//   k_sw_merge  boundary bonds united in the global forest (same min-root rule,
//               path halving), one warp per tile: the paper's two-step
//               local/global union-find (Sec. 3.2) inside one GPU
//   k_sw_find   global root of every open component's local root (path
//               halving) and its coin, one warp per tile
//   k_sw_flip   one coin per local root, spins flipped; sizes of clusters
//               closed in the tile squared here, sizes of open ones added at
//               their global root
//   k_sw_sizes  open clusters' sizes squared, cleared for the next update; the
//               update's record and running sums
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "dev.cuh"
#include "engine.h"
#include "uf.cuh"

namespace lcq {
namespace {

constexpr int SW_TX = 64, SW_TY = 32, SW_TS = SW_TX * SW_TY;  // tile of 64 x 32 sites
// Threads of a tile's block: SW_TPB, or SW_TPB_WIDE for lattices of up to two
// tiles per SM, whose update lasts as long as one tile's steps (us per update,
// 256 / 1024 threads: L=48 29 / 24, L=333 43 / 34, L=700, 242 tiles, 48 / 43,
// L=800, 325 tiles, 50 / 52, L=1500 75 / 90).
constexpr int SW_TPB = 256, SW_TPB_WIDE = 1024, SW_WIDE_TILES = 152 * 2;
constexpr int SW_WORDS = SW_TS / 32;    // bitmap words per tile
constexpr int SW_SIZE_BLOCKS = 1216;    // blocks of the open-cluster pass: 8 per SM
// An open cluster's root is the smallest site of a tile component that holds
// a site on the tile's border: at most 2 (64 + 32) of them per tile.
constexpr int SW_OPEN_PER_TILE = 2 * (SW_TX + SW_TY);
constexpr int SW_RING = 4096;
constexpr uint32_t TAG_SWBOND = 5u, TAG_SWFLIP = 6u;
constexpr int64_t SW_MAX_SITES = 2147483647;  // site ids are int32

struct SwDev {
  int32_t L, ntx, nty, ntile;
  int64_t N;
  uint64_t T;  // a bond is active iff its draw is below T
  uint64_t seed;
  uint32_t sweep, ring_cap;
  int64_t n_updates;
  double sum[LCQMC_SW_NOBS], sumsq[LCQMC_SW_NOBS];
};

typedef unsigned long long u64;

struct SwScratch {
  SwDev *dev;
  int *status;
  uint8_t *bytes;               // N: spins as bytes, for the C interface only
  u64 *spin;                    // per tile, SW_TY rows: spins of its sites (0 past its edges)
  u64 *starts;                  // per tile, SW_TY rows: first sites of the runs of active right bonds
  unsigned short *lroot;        // per tile, SW_TS: local root, at run starts
  int32_t *par;                 // N: global forest, at the local roots of open components
  uint32_t *openb;              // per tile, SW_WORDS words: local roots of open components
  uint32_t *edge_r;             // per tile: right-edge bond of row j active (bit j)
  u64 *edge_d;                  // per tile: bottom-edge bond of column j active (bit j)
  unsigned short *olocal;       // per tile, SW_OPEN_PER_TILE: local roots of open components
  int32_t *oroot;               // the same: their global roots, the top bit their cluster's coin
  int *onum;                    // per tile: their number
  int32_t *csize;               // N: size of an open cluster at its root; 0 between updates
  int32_t *olist;               // per tile, SW_OPEN_PER_TILE: roots of open clusters in the tile
  int *rnum;                    // per tile: their number
  long long *tile_part;         // per tile: n_eq, n_act, closed clusters, mag, largest closed
  unsigned long long *tile_c2;  // per tile: sum of the closed clusters' size^2
  // per block of k_sw_sizes, over its tiles and its open clusters: n_eq, n_act,
  // clusters, mag, largest
  long long *size_part;
  unsigned long long *size_c2;  // per block of k_sw_sizes: sum of size^2
  unsigned *done;               // blocks of k_sw_sizes done; 0 between updates
  lcqmc_sw_record *ring;
  int32_t *roots;               // lcqmc_sw_get_roots output (N), allocated on demand
};

__device__ __forceinline__ void sw_tile(const SwDev &D, int t, int &x0, int &y0, int &w, int &h) {
  const int ty = t / D.ntx, tx = t - ty * D.ntx;
  x0 = tx * SW_TX;
  y0 = ty * SW_TY;
  w = min(SW_TX, D.L - x0);
  h = min(SW_TY, D.L - y0);
}

// Shared-memory union-find of one tile (local ids, lp[x] <= x, one CAS on the
// larger root).  Walks are bounded by the tile size.
__device__ __forceinline__ int sw_find(volatile int *lp, int x, int *status) {
  for (int it = 0; it <= SW_TS; ++it) {
    const int p = lp[x];
    if (p == x) return x;
    const int g = lp[p];
    if (g != p) lp[x] = g;  // path halving
    x = g;
  }
  atomicOr(status, ST_TIMEOUT);
  return x;
}

__device__ __forceinline__ void sw_union(int *lp, int a, int b, int *status) {
  for (int it = 0; it <= SW_TS; ++it) {
    a = sw_find(lp, a, status);
    b = sw_find(lp, b, status);
    if (a == b) return;
    if (a > b) {
      const int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(lp + b, b, a) == b) return;
  }
  atomicOr(status, ST_TIMEOUT);
}

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ unsigned long long warp_sum_ull(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ long long warp_max_ll(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, (long long)__shfl_down_sync(0xffffffffu, v, o));
  return v;
}

// Block-wide sums of NS int64 values, the max of one more, and one uint64 sum;
// valid in thread 0.  One barrier pair per call.
template <int NS>
__device__ void block_reduce(long long (&v)[NS], long long &mx, unsigned long long &u) {
  __shared__ long long ps[NS][32], pm[32];
  __shared__ unsigned long long pu[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < NS; ++k) v[k] = warp_sum_ll(v[k]);
  mx = warp_max_ll(mx);
  u = warp_sum_ull(u);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NS; ++k) ps[k][wid] = v[k];
    pm[wid] = mx;
    pu[wid] = u;
  }
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int k = 0; k < NS; ++k) v[k] = warp_sum_ll(lane < nw ? ps[k][lane] : 0);
    mx = warp_max_ll(lane < nw ? pm[lane] : 0);
    u = warp_sum_ull(lane < nw ? pu[lane] : 0ull);
  }
  __syncthreads();
}

// ---- rows as 64-bit words -----------------------------------------------------------
// The word of the first n columns.
__device__ __forceinline__ u64 low_bits(int n) { return n >= 64 ? ~0ull : ((1ull << n) - 1ull); }

// Half row k of rows in shared memory (32 columns).
__device__ __forceinline__ uint32_t half_row(const u64 *rows, int k) { return reinterpret_cast<const uint32_t *>(rows)[k]; }

// First column of the run that holds column x, given the row's run starts.
__device__ __forceinline__ int run_start(u64 starts, int x) { return 63 - __clzll((long long)(starts & (~0ull >> (63 - x)))); }

// Columns of the run that starts at column x.
__device__ __forceinline__ u64 run_bits(u64 starts, int x, int w) {
  const u64 above = starts & (~1ull << x);  // later starts
  return (above ? ((above & (0ull - above)) - 1ull) : low_bits(w)) & (~0ull << x);
}

// Starts of the runs that hold a bit of x.
__device__ __forceinline__ u64 runs_with(u64 starts, u64 x) {
  u64 go = ~starts;  // columns a bit may move down from, o places at a time
#pragma unroll
  for (int o = 1; o < 64; o <<= 1) {
    x |= (x & go) >> o;
    go &= go << o;
  }
  return x & starts;
}

// Site id of tile-local index l.
__device__ __forceinline__ int32_t site_of(int x0, int y0, int L, int l) {
  return (int32_t)((int64_t)(y0 + (l >> 6)) * L + x0 + (l & 63));
}

// Philox4x32-10 of the counter (TAG_SWBOND << 24, site, 0, sweep), words 0 and
// 1: the rounds whose inputs do not depend on the site are taken once (15 of
// the 20 products are left), with the round keys.
struct SiteDraw {
  uint32_t k0, k1, b1, d0, e1, f;

  __device__ __forceinline__ SiteDraw(uint32_t key0, uint32_t key1, uint32_t sweep) : k0(key0), k1(key1) {
    const u64 p0 = (u64)M0 * (TAG_SWBOND << 24);           // round 0: second product zero
    const uint32_t a = (uint32_t)(p0 >> 32) ^ sweep ^ k1;  // c2 of round 1
    const u64 p1 = (u64)M1 * a;                            // round 1: c1 = 0
    const uint32_t c = (uint32_t)(p1 >> 32) ^ (k0 + W0);   // c0 of round 2
    const u64 p2 = (u64)M0 * c;
    b1 = (uint32_t)p0 ^ (k1 + W1);
    d0 = (uint32_t)p1 ^ (k0 + 2 * W0);
    e1 = (uint32_t)(p2 >> 32) ^ (k1 + 2 * W1);
    f = (uint32_t)p2;
  }

  __device__ __forceinline__ void operator()(uint32_t site, uint32_t &x, uint32_t &y) const {
    const u64 p = (u64)M0 * (site ^ k0);                 // round 1
    const u64 q = (u64)M1 * ((uint32_t)(p >> 32) ^ b1);  // round 2
    uint32_t c0 = (uint32_t)(q >> 32) ^ d0, c1 = (uint32_t)q, c2 = e1 ^ (uint32_t)p, c3 = f;
#pragma unroll
    for (uint32_t r = 3; r < 10; ++r) {
      const u64 u = (u64)M0 * c0, v = (u64)M1 * c2;
      c0 = (uint32_t)(v >> 32) ^ c1 ^ (k0 + r * W0);
      c1 = (uint32_t)v;
      c2 = (uint32_t)(u >> 32) ^ c3 ^ (k1 + r * W1);
      c3 = (uint32_t)u;
    }
    x = c0;
    y = c1;
  }

  static constexpr uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
};

__device__ __forceinline__ uint32_t same_on_all(uint32_t x) { return __reduce_max_sync(0xffffffffu, x); }

// ---- bonds and tile union-find --------------------------------------------------
// The draws of a half row are two ballots of a warp; one thread per row then
// takes the row's bonds as words: active right and down bonds, run starts, and
// the down bonds that need a union (one whose left neighbour is also active,
// with both right bonds between them active, joins runs already joined).  Those
// bonds are listed, about 650 of 2048 sites at K_c, and taken by whole warps, run
// start to run start.  A run's first bond to the row above hangs the run below
// the upper one by a plain store: every run has one such bond at most and hangs
// below a lower index, so the stores make a forest whose roots are their trees'
// lowest sites.  Only a run's further bonds need find and compare-and-swap.  A
// run's root is stored when found, so that the rows below walk from there.
//
// Bound by instruction issue (82 % at L=8192): the draws are a fifth of it, the
// unions a tenth, hanging the runs and finding their roots a fifth, listing and
// row words the rest.  L=8192: 530 us with a union for every listed bond, 483
// with the runs hung, 471 with their roots stored, 449 with the list made from
// half rows in 32 bits.
template <int NT>
__global__ void __launch_bounds__(NT, 2048 / NT) k_sw_local(SwScratch s) {
  constexpr int PER = SW_TS / NT, ROWS = NT / SW_TX;  // sites per thread, rows per step
  __shared__ int lp[SW_TS];               // forest of the run starts
  __shared__ unsigned short vlist[SW_TS]; // upper ends of the down bonds to unite
  __shared__ uint32_t drawR[SW_WORDS], drawD[SW_WORDS];  // draws below T, per half row
  __shared__ u64 start_s[SW_TY];
  __shared__ uint32_t vert_s[SW_WORDS], more_s[SW_WORDS];
  __shared__ u64 open_run[SW_TY];         // run starts of open sites
  __shared__ uint32_t open_s[SW_WORDS];   // sites on active tile-boundary bonds
  __shared__ uint32_t ob[SW_WORDS];       // local roots of open components
  __shared__ int vbase[SW_WORDS];
  __shared__ int nvert, nopen;
  const bool stop = __ldcg(s.status) != 0;
  const SwDev &D = *s.dev;
  const int t = blockIdx.x, L = D.L;
  int x0, y0, w, h;
  sw_tile(D, t, x0, y0, w, h);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const SiteDraw draw(same_on_all((uint32_t)D.seed), same_on_all((uint32_t)(D.seed >> 32)), same_on_all(D.sweep));
  const bool some = D.T > 0;  // a draw is below T iff T > 0 and it is at most T - 1
  const uint32_t top = (uint32_t)(D.T - 1);
  if (threadIdx.x < SW_WORDS) {
    ob[threadIdx.x] = 0u;
    open_s[threadIdx.x] = 0u;
    if (threadIdx.x == 0) nopen = 0;
  }
  {
    const int lx = 32 * (wid & 1) + lane;
    const uint32_t g0 = (uint32_t)((int64_t)y0 * L + x0 + lx);
#pragma unroll 2
    for (int k = 0; k < PER; ++k) {
      const int ly = ROWS * k + (wid >> 1), l = ly * SW_TX + lx;
      uint32_t x, y;
      draw(g0 + (uint32_t)ly * (uint32_t)L, x, y);
      const bool in = some && lx < w && ly < h;
      const uint32_t mr = __ballot_sync(0xffffffffu, in && x <= top);
      const uint32_t md = __ballot_sync(0xffffffffu, in && y <= top);
      if (lane == 0) {
        drawR[l >> 5] = mr;
        drawD[l >> 5] = md;
      }
      lp[l] = l;
    }
  }
  // One answer for the block: a walk that runs out in another block sets the status
  // word while this one starts, and what follows shares what every warp wrote.
  if (__syncthreads_or(stop)) return;
  const int tx = t % D.ntx, ty = t / D.ntx;
  const int left = ty * D.ntx + (tx ? tx - 1 : D.ntx - 1), right = ty * D.ntx + (tx + 1 < D.ntx ? tx + 1 : 0);
  const int up = (ty ? ty - 1 : D.nty - 1) * D.ntx + tx, down = (ty + 1 < D.nty ? ty + 1 : 0) * D.ntx + tx;
  if (wid == 0) {  // a thread per row
    const int j = lane;
    const u64 *own = s.spin + (int64_t)t * SW_TY;
    u64 r = 0, d = 0, eq_r = 0, eq_d = 0;
    if (j < h) {
      const u64 me = own[j], cols = low_bits(w);
      const u64 next = (me >> 1) | ((s.spin[(int64_t)right * SW_TY + j] & 1ull) << (w - 1));
      const u64 below = j + 1 < h ? own[j + 1] : s.spin[(int64_t)down * SW_TY];
      eq_r = ~(me ^ next) & cols;
      eq_d = ~(me ^ below) & cols;
      r = eq_r & (((u64)drawR[2 * j + 1] << 32) | drawR[2 * j]);
      d = eq_d & (((u64)drawD[2 * j + 1] << 32) | drawD[2 * j]);
    }
    const u64 last = 1ull << (w - 1);
    const uint32_t er = __ballot_sync(0xffffffffu, (r & last) != 0);
    const u64 open = (r & last) | (j == h - 1 ? d : 0ull);
    const u64 ri = r & ~last;                  // right bonds inside the tile
    const u64 di = j < h - 1 ? d : 0ull;       // down bonds inside the tile
    const u64 r1 = __shfl_down_sync(0xffffffffu, ri, 1);
    const u64 vert = di & ~((di & ri & r1) << 1);
    const u64 starts = ~(ri << 1) & (j < h ? low_bits(w) : 0ull);
    start_s[j] = starts;
    // the bonds whose lower run has one further left already
    u64 go = ~__shfl_down_sync(0xffffffffu, starts, 1), more = (vert << 1) & go;
#pragma unroll
    for (int o = 1; o < 64; o <<= 1) {
      more |= go & (more << o);
      go &= go << o;
    }
    more &= vert;
    vert_s[2 * j] = (uint32_t)vert;
    vert_s[2 * j + 1] = (uint32_t)(vert >> 32);
    more_s[2 * j] = (uint32_t)more;
    more_s[2 * j + 1] = (uint32_t)(more >> 32);
    if ((uint32_t)open) atomicOr(&open_s[2 * j], (uint32_t)open);
    if (open >> 32) atomicOr(&open_s[2 * j + 1], (uint32_t)(open >> 32));
    const int nlo = __popc((uint32_t)vert) | __popc((uint32_t)more) << 16;  // at most 2048 each in a tile
    const int nv = nlo + (__popc((uint32_t)(vert >> 32)) | __popc((uint32_t)(more >> 32)) << 16);
    int inc = nv;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    vbase[2 * j] = inc - nv;
    vbase[2 * j + 1] = inc - nv + nlo;
    int n_eq = __popcll(eq_r) + __popcll(eq_d), n_act = __popcll(r) + __popcll(d);
    n_eq = __reduce_add_sync(0xffffffffu, n_eq);
    n_act = __reduce_add_sync(0xffffffffu, n_act);
    s.starts[(int64_t)t * SW_TY + j] = starts;
    if (j == h - 1) s.edge_d[t] = d;
    if (lane == 31) nvert = inc;
    if (lane == 0) {
      s.edge_r[t] = er;
      s.tile_part[5 * (int64_t)t] = n_eq;
      s.tile_part[5 * (int64_t)t + 1] = n_act;
    }
  } else if (wid == 1) {
    // bonds of the neighbouring tiles that end in this one: R of the column to
    // the left
    const int j = lane, wl = min(SW_TX, L - (left % D.ntx) * SW_TX);
    if (j < h) {
      const uint32_t g = (uint32_t)((int64_t)(y0 + j) * L + (x0 == 0 ? L - 1 : x0 - 1));
      uint32_t x, y;
      draw(g, x, y);
      const u64 a = s.spin[(int64_t)left * SW_TY + j] >> (wl - 1), b = s.spin[(int64_t)t * SW_TY + j];
      if (some && x <= top && !((a ^ b) & 1ull)) atomicOr(&open_s[2 * j], 1u);
    }
  } else if (wid < 4) {  // D of the row above
    const int c = threadIdx.x - 64, hu = min(SW_TY, L - (up / D.ntx) * SW_TY);
    bool on = false;
    if (c < w) {
      const uint32_t g = (uint32_t)((int64_t)(y0 == 0 ? L - 1 : y0 - 1) * L + x0 + c);
      uint32_t x, y;
      draw(g, x, y);
      const u64 a = s.spin[(int64_t)up * SW_TY + hu - 1], b = s.spin[(int64_t)t * SW_TY];
      on = some && y <= top && !(((a ^ b) >> c) & 1ull);
    }
    const uint32_t m = __ballot_sync(0xffffffffu, on);
    if (lane == 0 && m) atomicOr(&open_s[wid - 2], m);
  }
  __syncthreads();
  // the open sites' runs, a thread per row
  if (wid == NT / 32 - 1) {
    const u64 open = ((u64)open_s[2 * lane + 1] << 32) | open_s[2 * lane];
    open_run[lane] = runs_with(start_s[lane], open);
  }
  const int nall = nvert & 0xffff, nfirst = nall - (nvert >> 16);
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int word = k * (NT / 32) + wid;  // half row
    const uint32_t v = vert_s[word], m = more_s[word], low = (1u << lane) - 1u;
    if ((v >> lane) & 1u) {
      const int b = vbase[word], i = (b >> 16) + __popc(m & low);
      vlist[(m >> lane) & 1u ? nfirst + i : (b & 0xffff) + __popc(v & low) - i] = (unsigned short)(32 * word + lane);
    }
  }
  __syncthreads();
  auto ends = [&](int i, int &a, int &b) {
    const int l = vlist[i], lx = l & (SW_TX - 1), ly = l / SW_TX;
    a = ly * SW_TX + run_start(start_s[ly], lx);
    b = (ly + 1) * SW_TX + run_start(start_s[ly + 1], lx);
  };
  for (int i = threadIdx.x; i < nfirst; i += NT) {
    int a, b;
    ends(i, a, b);
    lp[b] = a;  // a run's only one of these bonds, and a < b
  }
  __syncthreads();
  for (int i = nfirst + threadIdx.x; i < nall; i += NT) {
    int a, b;
    ends(i, a, b);
    sw_union(lp, a, b, s.status);
  }
  __syncthreads();
  // every run's local root (read-only walks: no union is running any more)
#pragma unroll 2
  for (int k = 0; k < PER; ++k) {
    const int word = k * (NT / 32) + wid, l = 32 * word + lane;
    if ((half_row(start_s, word) >> lane) & 1u) {
      volatile int *f = lp;
      int r = f[l];
      for (int it = 0, g; it <= SW_TS && (g = f[r]) != r; ++it) r = g;
      f[l] = r;
      s.lroot[(int64_t)t * SW_TS + l] = (unsigned short)r;
      if ((half_row(open_run, word) >> lane) & 1u) atomicOr(&ob[r >> 5], 1u << (r & 31));
    }
  }
  __syncthreads();
  if (threadIdx.x < SW_WORDS) {
    uint32_t m = ob[threadIdx.x];
    s.openb[(int64_t)t * SW_WORDS + threadIdx.x] = m;
    int at = m ? atomicAdd(&nopen, __popc(m)) : 0;
    while (m) {  // open components are listed, and enter the global forest as their own roots
      const int l = 32 * threadIdx.x + __ffs(m) - 1;
      const int32_t g = site_of(x0, y0, L, l);
      m &= m - 1;
      s.par[g] = g;
      s.olocal[(int64_t)t * SW_OPEN_PER_TILE + at++] = (unsigned short)l;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) s.onum[t] = nopen;
}

// ---- tile-boundary bonds in the global forest ------------------------------------
// Site of the local root of tile t's column x, row y.
__device__ __forceinline__ int32_t local_root(const SwScratch &s, const SwDev &D, int t, int x, int y) {
  const int l = y * SW_TX + run_start(s.starts[(int64_t)t * SW_TY + y], x);
  int x0, y0, w, h;
  sw_tile(D, t, x0, y0, w, h);
  return site_of(x0, y0, D.L, s.lroot[(int64_t)t * SW_TS + l]);
}

// One thread per edge bond.  Most find the larger local root still its own parent
// and hang it below the smaller one (L=3000 update 165 -> 154 us, L=8192 899 -> 895,
// against a search for both global roots first).  Between SW_WALK_MIN and
// SW_WALK_TILES tiles every thread walks once more after its union: the time there
// is the longest chain of dependent accesses, and all threads' walks halve the same
// paths for the waiting unions and for k_sw_find.  One update, us, without / with the
// walk, at K_c: L=48 24.0 / 24.6, L=250 31.4 / 31.6, L=333, 66 tiles, 34.5 / 34.6,
// L=500, 128 tiles, 35.7 / 35.6, L=700, 242 tiles, 42.4 / 41.6, L=1000 50.6 / 49.2,
// L=1500, 1128 tiles, 69.4 / 67.5, L=2000 93.1 / 92.3, L=3000, 4418 tiles, 153.8 /
// 154.0.  The lines are K_c's, where the paths are longest; away from it the walk
// costs: L=1000, 1500, 2000 at K = 0.3 40.1 / 40.8, 54.9 / 55.6, 75.0 / 75.7, at K =
// 0.7 40.0 / 41.5, 57.5 / 61.0, 81.8 / 89.0.
constexpr int SW_WALK_MIN = 152, SW_WALK_TILES = 2048;
constexpr int SW_EDGE = SW_TX + SW_TY;

__global__ void __launch_bounds__(SW_EDGE) k_sw_merge(SwScratch s) {
  if (__ldcg(s.status)) return;
  const SwDev &D = *s.dev;
  const int t = blockIdx.x, j = threadIdx.x;
  int x0, y0, w, h;
  sw_tile(D, t, x0, y0, w, h);
  const uint32_t er = s.edge_r[t];
  const u64 ed = s.edge_d[t];
  const int tx = t % D.ntx, ty = t / D.ntx;
  const int right = ty * D.ntx + (tx + 1 < D.ntx ? tx + 1 : 0), down = (ty + 1 < D.nty ? ty + 1 : 0) * D.ntx + tx;
  int32_t a, b;
  if (j < SW_TY) {
    if (!((er >> j) & 1u)) return;
    a = local_root(s, D, t, w - 1, j);
    b = local_root(s, D, right, 0, j);
  } else {
    const int c = j - SW_TY;
    if (!((ed >> c) & 1ull)) return;
    a = local_root(s, D, t, c, h - 1);
    b = local_root(s, D, down, c, 0);
  }
  if (a != b) {  // one try on the two local roots before the search for global ones
    const int lo = min(a, b), hi = max(a, b), old = atomicCAS(s.par + hi, hi, lo);
    if (old != hi && old != lo) uf_union(s.par, lo, old, s.status);
  }
  if (D.ntile <= SW_WALK_MIN || D.ntile > SW_WALK_TILES) return;
  const int r = uf_find(s.par, a, s.status);
  if (r != a) s.par[a] = r;
}

// ---- global roots of the open components --------------------------------------------
// Chains of dependent loads, about 50 per tile at K_c: a kernel of their own
// keeps every warp slot of the chip on them (inside k_sw_flip a block's other
// work waited for them: 0.53 ms there).
__global__ void __launch_bounds__(256) k_sw_find(SwScratch s) {
  if (__ldcg(s.status)) return;
  const SwDev &D = *s.dev;
  const int t = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (t >= D.ntile) return;
  int x0, y0, w, h;
  sw_tile(D, t, x0, y0, w, h);
  const uint32_t k0 = (uint32_t)D.seed, k1 = (uint32_t)(D.seed >> 32);
  const int n = s.onum[t];
  for (int i = lane; i < n; i += 32) {
    const int64_t k = (int64_t)t * SW_OPEN_PER_TILE + i;
    const int32_t g = site_of(x0, y0, D.L, s.olocal[k]);
    // path halving on the way and the root stored at the start: every entry
    // still points to an ancestor
    const int gr = uf_find(s.par, g, s.status);
    if (gr != g) s.par[g] = gr;
    const int coin = coin_from(philox(TAG_SWFLIP << 24, (uint32_t)gr >> 7, 0u, D.sweep, k0, k1), (uint32_t)gr);
    s.oroot[k] = (int32_t)((uint32_t)gr | ((uint32_t)coin << 31));
  }
}

// ---- roots, coins, flips, cluster sizes ---------------------------------------------
// A site's coin as a root of its own is one bit of at most two Philox blocks per
// row; the local roots of open components take their global root's coin
// instead.  A run then flips as its local root's bit says: the coins of the run
// starts are ballots, spread over the runs by word operations, one thread per
// row.  Sizes are added once per run.
template <int NT>
__global__ void __launch_bounds__(NT, 2048 / NT) k_sw_flip(SwScratch s) {
  constexpr int PER = SW_TS / NT, ROWS = NT / SW_TX;  // sites per thread, rows per step
  __shared__ int cnt[SW_TS];
  __shared__ uint32_t coin_s[SW_WORDS];               // per half row: coins of its sites as roots
  __shared__ uint32_t flip_s[SW_WORDS];               // per half row: run starts that flip
  __shared__ int32_t groot[SW_OPEN_PER_TILE];         // global roots of the open components
  __shared__ u64 start_s[SW_TY];
  __shared__ int nroot;
  __shared__ uint32_t closed[3];
  if (__ldcg(s.status)) return;
  const SwDev &D = *s.dev;
  const int t = blockIdx.x, L = D.L;
  int x0, y0, w, h;
  sw_tile(D, t, x0, y0, w, h);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nopen = s.onum[t];
  const unsigned short *olocal = s.olocal + (int64_t)t * SW_OPEN_PER_TILE;
  const int32_t *oroot = s.oroot + (int64_t)t * SW_OPEN_PER_TILE;
  const uint32_t k0 = same_on_all((uint32_t)D.seed), k1 = same_on_all((uint32_t)(D.seed >> 32)),
                 sweep = same_on_all(D.sweep);
  const unsigned short *lroot = s.lroot + (int64_t)t * SW_TS;
  for (int l = threadIdx.x; l < SW_TS; l += NT) cnt[l] = 0;
  if (threadIdx.x < SW_TY) start_s[threadIdx.x] = s.starts[(int64_t)t * SW_TY + threadIdx.x];
  if (threadIdx.x == 0) nroot = 0;
  if (threadIdx.x < 3) closed[threadIdx.x] = 0u;
  __syncthreads();
  // local roots of the thread's run starts (0xffff: no start)
  unsigned short lr[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int ly = ROWS * k + (wid >> 1), lx = 32 * (wid & 1) + lane;
    lr[k] = (half_row(start_s, 2 * ly + (wid & 1)) >> lane) & 1u ? lroot[ly * SW_TX + lx] : (unsigned short)0xffff;
  }
  if (threadIdx.x < SW_WORDS) {
    // half row: 32 sites from g on, in one or two blocks of 128 coins
    const int ly = threadIdx.x >> 1, lx = 32 * (threadIdx.x & 1);
    uint32_t c = 0u;
    if (ly < h && lx < w) {
      const uint32_t g = (uint32_t)site_of(x0, y0, L, ly * SW_TX + lx);
      const U4 o = philox(TAG_SWFLIP << 24, g >> 7, 0u, sweep, k0, k1);
      const int i = (g >> 5) & 3;
      const uint32_t lo = i == 0 ? o.x : i == 1 ? o.y : i == 2 ? o.z : o.w;
      uint32_t hi = i == 0 ? o.y : i == 1 ? o.z : o.w;
      if (i == 3 && (g & 31u)) hi = philox(TAG_SWFLIP << 24, (g >> 7) + 1u, 0u, sweep, k0, k1).x;
      c = __funnelshift_r(lo, hi, g & 31u);
    }
    coin_s[threadIdx.x] = c;
  }
  // sizes of the local components, a run at a time
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int ly = ROWS * k + (wid >> 1), lx = 32 * (wid & 1) + lane;
    if (lr[k] != 0xffff) atomicAdd(&cnt[lr[k]], __popcll(run_bits(start_s[ly], lx, w)));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nopen; i += NT) {
    const int l = olocal[i];
    const uint32_t bit = 1u << (l & 31);
    const int32_t r = oroot[i];
    groot[i] = r & 0x7fffffff;
    if (r < 0)
      atomicOr(&coin_s[l >> 5], bit);
    else
      atomicAnd(&coin_s[l >> 5], ~bit);
  }
  __syncthreads();
  // clusters closed in the tile: their number, sum of squares (at most 2^22) and
  // largest, in 32 bits
  uint32_t nc = 0, c2 = 0, mx = 0;
  const uint32_t *openb = s.openb + (int64_t)t * SW_WORDS;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int ly = ROWS * k + (wid >> 1), lx = 32 * (wid & 1) + lane, l = ly * SW_TX + lx;
    bool f = false;
    if (lr[k] != 0xffff) {
      const int r = lr[k];
      f = (coin_s[r >> 5] >> (r & 31)) & 1u;
      if (r == l && !((openb[l >> 5] >> (l & 31)) & 1u)) {  // a cluster closed in the tile
        const uint32_t c = (uint32_t)cnt[l];
        nc += 1;
        c2 += c * c;
        mx = max(mx, c);
      }
    }
    const uint32_t m = __ballot_sync(0xffffffffu, f);
    if (lane == 0) flip_s[l >> 5] = m;
  }
  nc = __reduce_add_sync(0xffffffffu, nc);
  c2 = __reduce_add_sync(0xffffffffu, c2);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) {
    atomicAdd(&closed[0], nc);
    atomicAdd(&closed[1], c2);
    atomicMax(&closed[2], mx);
  }
  // Open components of one cluster are added up in the tile first (about half of
  // them belong to the largest cluster at K_c: an atomic for each took 0.35 ms).
  for (int i = threadIdx.x; i < nopen; i += NT) {
    const int32_t gr = groot[i];
    int size = 0, lead = i;
    bool root = false;
    for (int j = 0; j < nopen; ++j)
      if (groot[j] == gr) {
        const int l = olocal[j];
        lead = min(lead, j);
        size += cnt[l];
        root |= gr == site_of(x0, y0, L, l);
      }
    if (lead == i) {
      atomicAdd(s.csize + gr, size);
      if (root) {  // the cluster's root is in this tile: listed once
        s.olist[(int64_t)t * SW_OPEN_PER_TILE + atomicAdd(&nroot, 1)] = gr;
      }
    }
  }
  __syncthreads();
  if (wid) return;
  int mag = 0;
  if (lane < h) {  // a thread per row: the starts' flips spread over their runs
    u64 f = ((u64)flip_s[2 * lane + 1] << 32) | flip_s[2 * lane], go = ~start_s[lane] & low_bits(w);
#pragma unroll
    for (int o = 1; o < 64; o <<= 1) {
      f |= go & (f << o);
      go &= go << o;
    }
    u64 *row = s.spin + (int64_t)t * SW_TY + lane;
    const u64 ns = *row ^ f;
    *row = ns;
    mag = w - 2 * __popcll(ns);
  }
  mag = __reduce_add_sync(0xffffffffu, mag);
  if (lane == 0) {
    s.rnum[t] = nroot;
    s.tile_part[5 * (int64_t)t + 2] = closed[0];
    s.tile_part[5 * (int64_t)t + 3] = mag;
    s.tile_part[5 * (int64_t)t + 4] = closed[2];
    s.tile_c2[t] = closed[1];
  }
}

// ---- open clusters: sizes squared and cleared; the tiles' sums; the record --------------
// A size is taken and cleared by one exchange (a load followed by a store to the
// same word waits for the load at L2: 0.2 ms).  The block that finishes last
// adds up the blocks' sums and writes the record, its fp64 values one per lane.
__global__ void __launch_bounds__(256) k_sw_sizes(SwScratch s) {
  __shared__ int last;
  if (__ldcg(s.status)) return;
  SwDev &D = *s.dev;
  long long v[4] = {0, 0, 0, 0};  // n_eq, n_act, clusters, magnetization
  long long mx = 0;
  unsigned long long c2 = 0;
  const int lane = threadIdx.x & 31, nwarp = gridDim.x * (blockDim.x / 32);
  for (int t = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); t < D.ntile; t += nwarp) {  // a warp per tile
    const int n = s.rnum[t];
    for (int i = lane; i < n; i += 32) {
      const int r = s.olist[(int64_t)t * SW_OPEN_PER_TILE + i];
      const long long c = atomicExch(s.csize + r, 0);
      v[2] += 1;
      c2 += (unsigned long long)c * (unsigned long long)c;
      mx = max(mx, c);
    }
  }
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < D.ntile; t += gridDim.x * blockDim.x) {
    const long long *p = s.tile_part + 5 * (int64_t)t;
    v[0] += p[0];
    v[1] += p[1];
    v[2] += p[2];
    v[3] += p[3];
    mx = max(mx, p[4]);
    c2 += s.tile_c2[t];
  }
  block_reduce<4>(v, mx, c2);
  if (gridDim.x > 1) {
    if (threadIdx.x == 0) {
      long long *p = s.size_part + 5 * (int64_t)blockIdx.x;
      p[0] = v[0];
      p[1] = v[1];
      p[2] = v[2];
      p[3] = v[3];
      p[4] = mx;
      s.size_c2[blockIdx.x] = c2;
      __threadfence();
      last = atomicAdd(s.done, 1u) == gridDim.x - 1;
      __threadfence();
    }
    __syncthreads();
    if (!last) return;
    v[0] = v[1] = v[2] = v[3] = mx = 0;
    c2 = 0;
    for (int b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
      const long long *p = s.size_part + 5 * (int64_t)b;
      v[0] += __ldcg(p);
      v[1] += __ldcg(p + 1);
      v[2] += __ldcg(p + 2);
      v[3] += __ldcg(p + 3);
      mx = max(mx, __ldcg(p + 4));
      c2 += __ldcg(s.size_c2 + b);
    }
    block_reduce<4>(v, mx, c2);
  }
  if (threadIdx.x >= 32) return;
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = __shfl_sync(0xffffffffu, v[k], 0);
  c2 = __shfl_sync(0xffffffffu, c2, 0);
  const int64_t N = D.N;
  // lane 0: energy = -(1/N) sum_bonds sigma sigma; 1: chi = sum_c |c|^2 / N;
  // 2: M^2 / N; 3: |M| / N
  const double m = (double)v[3];
  const double num = lane == 0 ? (double)(2 * N - 2 * v[0]) : lane == 1 ? (double)c2 : lane == 2 ? m * m : fabs(m);
  const double x = num / (double)N;
  lcqmc_sw_record &r = s.ring[D.n_updates % D.ring_cap];
  if (lane < LCQMC_SW_NOBS) {
    D.sum[lane] += x;
    D.sumsq[lane] += x * x;
  }
  if (lane == 0) r.energy = x;
  if (lane == 1) r.chi = x;
  __syncwarp();
  if (lane == 0) {
    r.sweep = D.sweep;
    r.n_eq = v[0];
    r.n_act = v[1];
    r.n_clusters = v[2];
    r.max_cluster = mx;
    r.sum_c2 = c2;
    r.mag = v[3];
    D.n_updates += 1;
    D.sweep += 1u;
    *s.done = 0u;
  }
}

// Tile and tile-local index of site g.
__device__ __forceinline__ void tile_site(const SwDev &D, int64_t g, int &t, int &x, int &y) {
  const int gy = (int)(g / D.L), gx = (int)(g - (int64_t)gy * D.L);
  t = (gy / SW_TY) * D.ntx + gx / SW_TX;
  x = gx % SW_TX;
  y = gy % SW_TY;
}

__global__ void k_sw_roots(SwScratch s) {
  if (__ldcg(s.status)) return;
  const SwDev &D = *s.dev;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < D.N; g += (int64_t)gridDim.x * blockDim.x) {
    int t, x, y, x0, y0, w, h;
    tile_site(D, g, t, x, y);
    sw_tile(D, t, x0, y0, w, h);
    const int l = s.lroot[(int64_t)t * SW_TS + y * SW_TX + run_start(s.starts[(int64_t)t * SW_TY + y], x)];
    const int32_t r = site_of(x0, y0, D.L, l);
    const bool open = (s.openb[(int64_t)t * SW_WORDS + (l >> 5)] >> (l & 31)) & 1u;
    s.roots[g] = open ? uf_root(s.par, r, s.status) : r;
  }
}

// Spins between bytes (row-major) and tile rows, a warp per tile row.
__global__ void k_sw_pack(SwScratch s) {
  const SwDev &D = *s.dev;
  const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (i >= (int64_t)D.ntile * SW_TY) return;
  int x0, y0, w, h;
  sw_tile(D, (int)(i / SW_TY), x0, y0, w, h);
  const int y = (int)(i % SW_TY), lane = threadIdx.x & 31;
  const uint8_t *p = s.bytes + (int64_t)(y0 + y) * D.L + x0;
  const uint32_t lo = __ballot_sync(0xffffffffu, y < h && lane < w && (p[lane] & 1));
  const uint32_t hi = __ballot_sync(0xffffffffu, y < h && lane + 32 < w && (p[lane + 32] & 1));
  if (lane == 0) s.spin[i] = ((u64)hi << 32) | lo;
}

__global__ void k_sw_unpack(SwScratch s) {
  const SwDev &D = *s.dev;
  const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (i >= (int64_t)D.ntile * SW_TY) return;
  int x0, y0, w, h;
  sw_tile(D, (int)(i / SW_TY), x0, y0, w, h);
  const int y = (int)(i % SW_TY), lane = threadIdx.x & 31;
  if (y >= h) return;
  uint8_t *p = s.bytes + (int64_t)(y0 + y) * D.L + x0;
  const u64 row = s.spin[i];
  if (lane < w) p[lane] = (uint8_t)((row >> lane) & 1ull);
  if (lane + 32 < w) p[lane + 32] = (uint8_t)((row >> (lane + 32)) & 1ull);
}

#define SWCK(call)                                                                   \
  do {                                                                               \
    cudaError_t e_ = (call);                                                         \
    if (e_ != cudaSuccess) {                                                         \
      set_error(std::string("CUDA error: ") + cudaGetErrorString(e_) + " at " #call); \
      return LCQMC_E_CUDA;                                                           \
    }                                                                                \
  } while (0)

uint64_t sw_threshold(double K) {
  const double x = std::floor(std::ldexp(-std::expm1(-2.0 * K), 32) + 0.5);
  if (x <= 0.0) return 0;
  if (x >= 4294967296.0) return (uint64_t)1 << 32;
  return (uint64_t)x;
}

}  // namespace

class SwEngine {
 public:
  ~SwEngine() { release(); }

  int init(int64_t L, double K, uint64_t seed, void *stream) {
    if (L < 2 || L > 46340 || L * L > SW_MAX_SITES) {
      set_error("L must be >= 2 with L^2 < 2^31");
      return LCQMC_E_INVAL;
    }
    if (!(K >= 0.0) || !std::isfinite(K)) {
      set_error("K must be finite and >= 0");
      return LCQMC_E_INVAL;
    }
    if (stream) {
      st_ = (cudaStream_t)stream;
    } else {
      SWCK(cudaStreamCreateWithFlags(&st_, cudaStreamNonBlocking));
      own_stream_ = true;
    }
    h_ = SwDev{};
    h_.L = (int32_t)L;
    h_.N = L * L;
    h_.ntx = (int32_t)((L + SW_TX - 1) / SW_TX);
    h_.nty = (int32_t)((L + SW_TY - 1) / SW_TY);
    h_.ntile = h_.ntx * h_.nty;
    h_.T = sw_threshold(K);
    h_.seed = seed;
    h_.ring_cap = SW_RING;
    const int64_t N = h_.N, nt = h_.ntile;
    int rc = 0;
    rc |= dalloc((void **)&s_.dev, sizeof(SwDev));
    rc |= dalloc((void **)&s_.status, sizeof(int));
    rc |= dalloc((void **)&s_.bytes, (size_t)N);
    rc |= dalloc((void **)&s_.spin, 8 * (size_t)nt * SW_TY);
    rc |= dalloc((void **)&s_.starts, 8 * (size_t)nt * SW_TY);
    rc |= dalloc((void **)&s_.lroot, 2 * (size_t)nt * SW_TS);
    rc |= dalloc((void **)&s_.par, 4 * (size_t)N);
    rc |= dalloc((void **)&s_.openb, 4 * (size_t)nt * SW_WORDS);
    rc |= dalloc((void **)&s_.edge_r, 4 * (size_t)nt);
    rc |= dalloc((void **)&s_.edge_d, 8 * (size_t)nt);
    rc |= dalloc((void **)&s_.olocal, 2 * (size_t)nt * SW_OPEN_PER_TILE);
    rc |= dalloc((void **)&s_.oroot, 4 * (size_t)nt * SW_OPEN_PER_TILE);
    rc |= dalloc((void **)&s_.onum, 4 * (size_t)nt);
    rc |= dalloc((void **)&s_.csize, 4 * (size_t)N);
    rc |= dalloc((void **)&s_.olist, 4 * (size_t)nt * SW_OPEN_PER_TILE);
    rc |= dalloc((void **)&s_.rnum, 4 * (size_t)nt);
    rc |= dalloc((void **)&s_.tile_part, 5 * 8 * (size_t)nt);
    rc |= dalloc((void **)&s_.tile_c2, 8 * (size_t)nt);
    rc |= dalloc((void **)&s_.size_part, 5 * 8 * (size_t)SW_SIZE_BLOCKS);
    rc |= dalloc((void **)&s_.size_c2, 8 * (size_t)SW_SIZE_BLOCKS);
    rc |= dalloc((void **)&s_.done, sizeof(unsigned));
    rc |= dalloc((void **)&s_.ring, sizeof(lcqmc_sw_record) * SW_RING);
    if (rc) return LCQMC_E_NOMEM;
    SWCK(cudaMemsetAsync(s_.status, 0, sizeof(int), st_));
    SWCK(cudaMemsetAsync(s_.done, 0, sizeof(unsigned), st_));
    SWCK(cudaMemsetAsync(s_.spin, 0, 8 * (size_t)nt * SW_TY, st_));  // ordered start: every sigma = +1
    SWCK(cudaMemsetAsync(s_.csize, 0, 4 * (size_t)N, st_));
    SWCK(cudaMemcpyAsync(s_.dev, &h_, sizeof(SwDev), cudaMemcpyHostToDevice, st_));
    for (int i = 0; i <= 4; ++i) SWCK(cudaEventCreate(&ev_[i]));
    SWCK(cudaStreamSynchronize(st_));
    return LCQMC_OK;
  }

  int update(int64_t n) {
    if (n < 0) {
      set_error("n must be >= 0");
      return LCQMC_E_INVAL;
    }
    nvtxRangePushA("lcqmc_sw_update");  // profiler range (no-op without a tool)
    const int rc = update_n(n);
    nvtxRangePop();
    return rc;
  }

  int update_n(int64_t n) {
    if (timing_) {
      for (int64_t i = 0; i < n; ++i) {
        int rc = enqueue(true);
        if (rc) return rc;
        ++enq_;
      }
      return LCQMC_OK;
    }
    // graphs of kGraphBlock updates, then of one (a launch per update left gaps
    // between the few microseconds of a small lattice's updates)
    const int64_t nblk = n / kGraphBlock, rest = n % kGraphBlock;
    int rc = nblk ? capture(kGraphBlock, &gexec_blk_) : LCQMC_OK;
    if (!rc && rest) rc = capture(1, &gexec_);
    if (rc) return rc;
    for (int64_t i = 0; i < nblk; ++i) {
      SWCK(cudaGraphLaunch(gexec_blk_, st_));
      enq_ += kGraphBlock;
    }
    for (int64_t i = 0; i < rest; ++i) {
      SWCK(cudaGraphLaunch(gexec_, st_));
      ++enq_;
    }
    return LCQMC_OK;
  }

  int sync() {
    SWCK(cudaStreamSynchronize(st_));
    int st = 0;
    SWCK(cudaMemcpy(&st, s_.status, sizeof(int), cudaMemcpyDeviceToHost));
    if (st) {
      set_error("a bounded union-find walk ran out (status " + std::to_string(st) + ")");
      return LCQMC_E_DEVICE_TIMEOUT;
    }
    return LCQMC_OK;
  }

  int records(lcqmc_sw_record *out, int64_t max_n, int64_t *n_out) {
    if (!n_out || (max_n > 0 && !out)) {
      set_error("null output");
      return LCQMC_E_INVAL;
    }
    int rc = sync();
    if (rc) return rc;
    if (enq_ - read_ > SW_RING) read_ = enq_ - SW_RING;  // older records were overwritten
    const int64_t n = std::min<int64_t>(max_n, enq_ - read_);
    for (int64_t k = 0; k < n;) {
      const int64_t pos = (read_ + k) % SW_RING;
      const int64_t run = std::min<int64_t>(n - k, SW_RING - pos);
      SWCK(cudaMemcpy(out + k, s_.ring + pos, sizeof(lcqmc_sw_record) * run, cudaMemcpyDeviceToHost));
      k += run;
    }
    read_ += n;
    *n_out = n;
    return LCQMC_OK;
  }

  int measure(lcqmc_sw_obs *out) {
    if (!out) {
      set_error("null output");
      return LCQMC_E_INVAL;
    }
    int rc = sync();
    if (rc) return rc;
    SwDev d;
    SWCK(cudaMemcpy(&d, s_.dev, sizeof(SwDev), cudaMemcpyDeviceToHost));
    std::memset(out, 0, sizeof(*out));
    out->n_updates = d.n_updates;
    for (int k = 0; k < LCQMC_SW_NOBS; ++k) {
      out->sum[k] = d.sum[k];
      out->sumsq[k] = d.sumsq[k];
    }
    return LCQMC_OK;
  }

  int set_spins(const uint8_t *spins, uint32_t sweep) {
    if (!spins) {
      set_error("null spins");
      return LCQMC_E_INVAL;
    }
    for (int64_t i = 0; i < h_.N; ++i)
      if (spins[i] > 1) {
        set_error("spins must be 0 or 1");
        return LCQMC_E_STATE;
      }
    int rc = sync();
    if (rc) return rc;
    // On the handle's stream: a plain copy from pageable memory may return before its
    // last bytes have arrived, and the handle's own stream does not wait for it.
    SWCK(cudaMemcpyAsync(s_.bytes, spins, (size_t)h_.N, cudaMemcpyHostToDevice, st_));
    k_sw_pack<<<h_.ntile * SW_TY / 8, 256, 0, st_>>>(s_);  // a warp per tile row
    SWCK(cudaGetLastError());
    SWCK(cudaMemcpyAsync((char *)s_.dev + offsetof(SwDev, sweep), &sweep, sizeof(uint32_t),
                         cudaMemcpyHostToDevice, st_));
    SWCK(cudaStreamSynchronize(st_));  // the caller's memory is its own again
    return LCQMC_OK;
  }

  int get_spins(uint8_t *spins) {
    if (!spins) {
      set_error("null spins");
      return LCQMC_E_INVAL;
    }
    int rc = sync();
    if (rc) return rc;
    k_sw_unpack<<<h_.ntile * SW_TY / 8, 256, 0, st_>>>(s_);  // a warp per tile row
    SWCK(cudaGetLastError());
    SWCK(cudaMemcpyAsync(spins, s_.bytes, (size_t)h_.N, cudaMemcpyDeviceToHost, st_));
    SWCK(cudaStreamSynchronize(st_));
    return LCQMC_OK;
  }

  int get_roots(int32_t *roots) {
    if (!roots) {
      set_error("null roots");
      return LCQMC_E_INVAL;
    }
    if (enq_ == 0) {
      set_error("no update has run yet");
      return LCQMC_E_STATE;
    }
    int rc = sync();
    if (rc) return rc;
    if (!s_.roots && dalloc((void **)&s_.roots, 4 * (size_t)h_.N)) return LCQMC_E_NOMEM;
    const int64_t blocks = std::min<int64_t>((h_.N + 255) / 256, 4096);
    k_sw_roots<<<(int)blocks, 256, 0, st_>>>(s_);
    SWCK(cudaGetLastError());
    rc = sync();
    if (rc) return rc;
    SWCK(cudaMemcpy(roots, s_.roots, 4 * (size_t)h_.N, cudaMemcpyDeviceToHost));
    return LCQMC_OK;
  }

  int set_phase_timing(int on) {
    int rc = sync();
    if (rc) return rc;
    timing_ = on != 0;
    for (double &x : ph_) x = 0.0;
    return LCQMC_OK;
  }

  int phase_times(double *ms, int nphase) {
    if (!ms || nphase < 0) {
      set_error("null output");
      return LCQMC_E_INVAL;
    }
    int rc = sync();
    if (rc) return rc;
    if (pending_) {
      accumulate();
      pending_ = false;
    }
    for (int k = 0; k < nphase; ++k) ms[k] = k < LCQMC_SW_NPHASE ? ph_[k] : 0.0;
    return LCQMC_OK;
  }

  cudaStream_t stream() const { return st_; }
  int64_t sites() const { return h_.N; }

 private:
  int dalloc(void **p, size_t bytes) {
    if (cudaMalloc(p, std::max<size_t>(bytes, 16)) != cudaSuccess) {
      (void)cudaGetLastError();
      set_error("device allocation of " + std::to_string(bytes) + " bytes failed");
      *p = nullptr;
      return 1;
    }
    allocs_.push_back(*p);
    return 0;
  }

  void release() {
    if (st_) cudaStreamSynchronize(st_);
    if (gexec_) cudaGraphExecDestroy(gexec_);
    if (gexec_blk_) cudaGraphExecDestroy(gexec_blk_);
    gexec_ = gexec_blk_ = nullptr;
    for (cudaEvent_t &e : ev_)
      if (e) cudaEventDestroy(e);
    for (void *p : allocs_) cudaFree(p);
    allocs_.clear();
    if (own_stream_ && st_) cudaStreamDestroy(st_);
    st_ = nullptr;
  }

  void accumulate() {
    for (int k = 0; k < LCQMC_SW_NPHASE; ++k) {
      float t = 0.f;
      if (cudaEventElapsedTime(&t, ev_[k], ev_[k + 1]) == cudaSuccess) ph_[k] += t;
    }
  }

  int capture(int count, cudaGraphExec_t *out) {
    if (*out) return LCQMC_OK;
    SWCK(cudaStreamBeginCapture(st_, cudaStreamCaptureModeThreadLocal));
    int rc = LCQMC_OK;
    for (int i = 0; i < count && !rc; ++i) rc = enqueue(false);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(st_, &g);
    if (rc) {
      if (e == cudaSuccess) cudaGraphDestroy(g);
      return rc;
    }
    SWCK(e);
    e = cudaGraphInstantiate(out, g, 0);
    cudaGraphDestroy(g);
    SWCK(e);
    return LCQMC_OK;
  }

  int enqueue(bool timed) {
    if (timed && pending_) {  // the previous timed update's events are complete once it is
      SWCK(cudaEventSynchronize(ev_[LCQMC_SW_NPHASE]));
      accumulate();
      pending_ = false;
    }
    auto mark = [&](int k) -> cudaError_t { return timed ? cudaEventRecord(ev_[k], st_) : cudaSuccess; };
    const int nt = h_.ntile;
    const int nsize = (int)std::min<int64_t>(SW_SIZE_BLOCKS, ((int64_t)nt + 7) / 8);
    SWCK(mark(0));  // [0] bond draws, tile union-find
    if (nt <= SW_WIDE_TILES)
      k_sw_local<SW_TPB_WIDE><<<nt, SW_TPB_WIDE, 0, st_>>>(s_);
    else
      k_sw_local<SW_TPB><<<nt, SW_TPB, 0, st_>>>(s_);
    SWCK(mark(1));  // [1] tile-boundary bonds, global union-find
    k_sw_merge<<<nt, SW_EDGE, 0, st_>>>(s_);
    SWCK(mark(2));  // [2] roots, coins, flips
    k_sw_find<<<(nt * 32 + 255) / 256, 256, 0, st_>>>(s_);
    if (nt <= SW_WIDE_TILES)
      k_sw_flip<SW_TPB_WIDE><<<nt, SW_TPB_WIDE, 0, st_>>>(s_);
    else
      k_sw_flip<SW_TPB><<<nt, SW_TPB, 0, st_>>>(s_);
    SWCK(mark(3));  // [3] open clusters' sizes, record
    k_sw_sizes<<<nsize, 256, 0, st_>>>(s_);
    SWCK(mark(4));
    SWCK(cudaGetLastError());
    if (timed) pending_ = true;
    return LCQMC_OK;
  }

  SwDev h_{};
  SwScratch s_{};
  cudaStream_t st_ = nullptr;
  bool own_stream_ = false;
  static constexpr int kGraphBlock = 8;
  cudaGraphExec_t gexec_ = nullptr, gexec_blk_ = nullptr;
  cudaEvent_t ev_[LCQMC_SW_NPHASE + 1] = {};
  bool timing_ = false, pending_ = false;
  double ph_[LCQMC_SW_NPHASE] = {};
  std::vector<void *> allocs_;
  int64_t enq_ = 0, read_ = 0;
};

}  // namespace lcq

struct lcqmc_sw {
  lcq::SwEngine eng;
};

#define SWNEED(h)                         \
  do {                                    \
    if (!(h)) {                           \
      lcq::set_error("null handle");      \
      return LCQMC_E_INVAL;               \
    }                                     \
  } while (0)

extern "C" {

int lcqmc_sw_create(int64_t L, double K, uint64_t seed, void *cuda_stream, lcqmc_sw_t *out) {
  if (!out) {
    lcq::set_error("null output handle");
    return LCQMC_E_INVAL;
  }
  *out = nullptr;
  auto *h = new (std::nothrow) lcqmc_sw;
  if (!h) {
    lcq::set_error("host allocation failed");
    return LCQMC_E_NOMEM;
  }
  int rc = h->eng.init(L, K, seed, cuda_stream);
  if (rc) {
    delete h;
    return rc;
  }
  *out = h;
  return LCQMC_OK;
}

int lcqmc_sw_update(lcqmc_sw_t h, int64_t n) {
  SWNEED(h);
  return h->eng.update(n);
}

int lcqmc_sw_sync(lcqmc_sw_t h) {
  SWNEED(h);
  return h->eng.sync();
}

int lcqmc_sw_get_records(lcqmc_sw_t h, lcqmc_sw_record *out, int64_t max_n, int64_t *n_out) {
  SWNEED(h);
  return h->eng.records(out, max_n, n_out);
}

int lcqmc_sw_measure(lcqmc_sw_t h, lcqmc_sw_obs *out) {
  SWNEED(h);
  return h->eng.measure(out);
}

int lcqmc_sw_set_spins(lcqmc_sw_t h, const uint8_t *spins, uint32_t sweep) {
  SWNEED(h);
  return h->eng.set_spins(spins, sweep);
}

int lcqmc_sw_get_spins(lcqmc_sw_t h, uint8_t *spins) {
  SWNEED(h);
  return h->eng.get_spins(spins);
}

int lcqmc_sw_get_roots(lcqmc_sw_t h, int32_t *roots) {
  SWNEED(h);
  return h->eng.get_roots(roots);
}

int lcqmc_sw_set_phase_timing(lcqmc_sw_t h, int enable) {
  SWNEED(h);
  return h->eng.set_phase_timing(enable);
}

int lcqmc_sw_get_phase_times(lcqmc_sw_t h, double *ms, int nphase) {
  SWNEED(h);
  return h->eng.phase_times(ms, nphase);
}

void *lcqmc_sw_stream(lcqmc_sw_t h) { return h ? (void *)h->eng.stream() : nullptr; }

int lcqmc_sw_destroy(lcqmc_sw_t h) {
  delete h;
  return LCQMC_OK;
}

}  // extern "C"
